"""Several callers on one device: streams that defer block transpositions beside one another."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
import paper_2511_20564_b200 as E  # noqa: E402
import synth_inputs as S  # noqa: E402
from helpers import assert_blocks_equal  # noqa: E402

pytestmark = pytest.mark.gpu


def test_scratch_is_reused_after_an_unrelated_stream_has_joined():
    """Stream A samples with the transposition deferred, an unrelated stream B joins, A samples again with the same scratch
    and blocks: the second sample must not begin before the first one's transposition has ended."""
    w = S.WORKLOADS["medium_small"]
    indptr, indices, _ = S.build_graph(w)
    ip, ix = torch.from_numpy(indptr).cuda(), torch.from_numpy(indices).cuda()
    blocks = E.Blocks(w.n_nodes, w.batch, w.fanouts)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for step in range(0, 6, 2):
        seeds = [S.seed_batch(w.n_nodes, w.batch, w.seed, s) for s in (step, step + 1)]
        dev = [torch.from_numpy(s).cuda() for s in seeds]
        torch.cuda.synchronize()
        E.sample_khop(ip, ix, dev[0], blocks, w.seed, step, stream=a, defer_transpose=True)
        E.sample_join(stream=b)
        E.sample_khop(ip, ix, dev[1], blocks, w.seed, step + 1, stream=a, defer_transpose=True)
        E.sample_join(stream=a)
        a.synchronize()
        assert_blocks_equal(blocks.to_host(), oracle.sample_khop(indptr, indices, seeds[1], w.fanouts, w.seed, step + 1))


def test_two_callers_step_beside_one_another_with_deferral():
    """Two callers, each with its stream, blocks and weights; the steps of one are issued between the calls of the other, so
    that each finds the other's deferred work.  Same bits as the same steps one after the other."""
    w = S.WORKLOADS["medium_small"]
    indptr, indices, _ = S.build_graph(w)
    X_h, Ws_h = S.build_model(w)
    ip, ix = torch.from_numpy(indptr).cuda(), torch.from_numpy(indices).cuda()
    X = torch.from_numpy(X_h).cuda().to(torch.bfloat16)
    Ws = [torch.from_numpy(W).cuda().to(torch.bfloat16) for W in Ws_h]
    blocks = [E.Blocks(w.n_nodes, w.batch, w.fanouts) for _ in range(2)]
    dH = torch.randn(blocks[0].caps[0][0], w.hidden, device="cuda").to(torch.bfloat16)
    seeds = [[torch.from_numpy(S.seed_batch(w.n_nodes, w.batch, w.seed, 10 * who + i)).cuda() for i in range(3)] for who in range(2)]

    def sample(who, i, st):
        E.sample_khop(ip, ix, seeds[who][i], blocks[who], w.seed, i, stream=st, defer_transpose=True)

    def train(who, st):
        with torch.cuda.stream(st):
            H, ctx = E.sage_forward(blocks[who], X, Ws)
            dWs, dX = E.sage_backward(blocks[who], X, Ws, ctx, dH)
            return [t.clone() for t in [H, dX, blocks[who].counts] + dWs]

    want = {}
    for who in range(2):
        for i in range(3):
            sample(who, i, torch.cuda.default_stream())
            want[who, i] = train(who, torch.cuda.default_stream())
            torch.cuda.synchronize()
    st = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    got = {}
    for i in range(3):
        sample(0, i, st[0])
        sample(1, i, st[1])
        got[1, i] = train(1, st[1])
        got[0, i] = train(0, st[0])
    torch.cuda.synchronize()
    for key, tensors in want.items():
        n_src = int(tensors[2][-1, 1])
        for k, (p, q) in enumerate(zip(got[key], tensors)):
            assert torch.equal(p[:n_src], q[:n_src]) if k == 1 else torch.equal(p, q), (key, k)
        assert int(tensors[2][:, 3].sum()) == 0


def _joint_case(fanouts, n_pairs, dtype):
    rng = np.random.default_rng(len(fanouts))
    n, d, dense_dim = 4000, 64, 64
    deg = rng.integers(0, 12, n)
    deg[:4] = (900, 300, 0, 40)
    indptr = np.r_[0, np.cumsum(deg)].astype(np.int64)
    indices = rng.integers(0, n, indptr[-1]).astype(np.int32)
    norm = lambda *s: rng.standard_normal(s).astype(np.float32)
    z = 2 * d + dense_dim
    arrays = dict(X=norm(n, d), W_gnn=[norm(d, 2 * d) * 0.1 for _ in fanouts], W_t=[norm(128, z) * 0.1, norm(64, 128) * 0.1, norm(1, 64)],
                  b_t=[norm(128), norm(64), norm(1)])
    if dtype == torch.bfloat16:
        r = S.to_bf16_values
        arrays.update(X=r(arrays["X"]), W_gnn=[r(W) for W in arrays["W_gnn"]], W_t=[r(W) for W in arrays["W_t"]])
    pu, pi = (rng.integers(0, n, n_pairs).astype(np.int32) for _ in range(2))
    return indptr, indices, arrays, pu, pi, norm(n_pairs, dense_dim), (rng.random(n_pairs) < 0.3).astype(np.float32)


def _joint_run(case, fanouts, dtype, phases=(0,)):
    indptr, indices, a, pu, pi, dense, labels = case
    cu = lambda x, t=None: torch.from_numpy(np.ascontiguousarray(x)).cuda().to(t or torch.from_numpy(np.ascontiguousarray(x)).dtype)
    js = E.JointStep(cu(indptr), cu(indices), cu(a["X"], dtype), pu.size, dense.shape[1], fanouts, [cu(W, dtype) for W in a["W_gnn"]],
                     [cu(W, dtype) for W in a["W_t"]], [cu(b) for b in a["b_t"]])
    for step in (4, 5):                                      # the second step finds the first one's scratch
        for phase in phases:
            js.run(cu(pu), cu(pi), cu(dense), cu(labels), 21, step, phase=phase)
    torch.cuda.synchronize()
    n_rows = js.n_rows.tolist()[0]
    return js, [js.n_rows, js.loss, js.logits, js.dX_ids[:n_rows], js.dX_rows[:n_rows]] + js.dW_gnn + js.dW_tower + js.db_tower


@pytest.mark.parametrize("phases", [(0,), (1, 2)])
@pytest.mark.parametrize("fanouts", [[4], [3, 3, 2], [3, 2, 2, 2]])
def test_joint_step_over_one_three_and_four_hops(fanouts, phases):
    """With four hops no sort lane is free for the grouping of the pairs, which then shares the first hop's."""
    case = _joint_case(fanouts, 200, torch.float32)
    indptr, indices, a, pu, pi, dense, labels = case
    js, _ = _joint_run(case, fanouts, torch.float32, phases)
    want = oracle.joint_step(indptr, indices, a["X"], pu, pi, dense, labels, fanouts, a["W_gnn"], a["W_t"], a["b_t"], 21, 5, bf16=False,
                             acts_gnn=[1] * len(fanouts), acts_tower=(1, 1), gate=None)
    n_rows, status = js.n_rows.tolist()
    assert status == 0 and np.array_equal(js.dX_ids[:n_rows].cpu().numpy(), want["dX_ids"])
    pairs = [(js.logits, want["logits"]), (js.dX_rows[:n_rows], want["dX"])] + list(zip(js.dW_gnn, want["dW_gnn"])) + \
        list(zip(js.dW_tower, want["dW_tower"])) + list(zip(js.db_tower, want["db_tower"]))
    for k, (got, ref) in enumerate(pairs):
        ref = np.asarray(ref, np.float64).reshape(got.shape)
        assert np.linalg.norm(got.double().cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref), k


NO_HELPER = """
import sys, pickle, torch
sys.path[:0] = {path!r}
import test_gpu_callers as T
out = [[t.cpu() for t in T._joint_run(T._joint_case(f, 200, torch.bfloat16), f, torch.bfloat16)[1]] for f in ([5, 3], [3, 2, 2, 2])]
out.append([t.cpu() for t in T._sage_run()])
torch.save(out, {out!r})
"""


def _sage_run():
    """Two steps with the transposition deferred, one with it in a call of its own."""
    w = S.WORKLOADS["tiny"]
    indptr, indices, _ = S.build_graph(w)
    X, Ws = S.build_model(w)
    ip, ix, X = torch.from_numpy(indptr).cuda(), torch.from_numpy(indices).cuda(), torch.from_numpy(X).cuda()
    Ws = [torch.from_numpy(W).cuda() for W in Ws]
    blocks = E.Blocks(w.n_nodes, w.batch, w.fanouts)
    dH = torch.from_numpy(np.random.default_rng(1).standard_normal((blocks.caps[0][0], w.hidden)).astype(np.float32)).cuda()
    out = []
    for step in range(3):
        seeds = torch.from_numpy(S.seed_batch(w.n_nodes, w.batch, w.seed, step)).cuda()
        E.sample_khop(ip, ix, seeds, blocks, w.seed, step, defer_transpose=step < 2, transpose=step < 2)
        if step == 2:
            E.blocks_transpose(blocks)
        H, ctx = E.sage_forward(blocks, X, Ws)
        dWs, dX = E.sage_backward(blocks, X, Ws, ctx, dH)
        out += [t.clone() for t in [H, blocks.counts, dX[: int(blocks.counts[-1, 1])]] + dWs]
    return out


def test_without_helper_streams_the_results_are_the_same(tmp_path):
    """E2EGREC_NO_HELPER_STREAM keeps all work on the caller's stream: joint steps of two and four hops and encoder steps
    with every form of the transposition give the same bits."""
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    out = str(tmp_path / "out.pt")
    code = NO_HELPER.format(path=[here, os.path.dirname(here)], out=out)
    subprocess.check_call([sys.executable, "-c", code], env=dict(os.environ, E2EGREC_NO_HELPER_STREAM="1"), timeout=300)
    got = torch.load(out)
    want = [_joint_run(_joint_case(f, 200, torch.bfloat16), f, torch.bfloat16)[1] for f in ([5, 3], [3, 2, 2, 2])] + [_sage_run()]
    for a, b in zip(got, want):
        assert len(a) == len(b) and all(torch.equal(x, y.cpu()) for x, y in zip(a, b))


@pytest.mark.parametrize("dtype,d", [(torch.bfloat16, 256), (torch.float32, 128)])
def test_weight_gradients_on_two_streams_share_one_buffer_of_partial_sums(dtype, d):
    """The bottom layer's product would move more than 256 MB by its block's capacity and stays on the caller's stream, the top
    layer's runs on the helper stream behind the deferred transposition, and few rows are live: the bottom layer is soon there."""
    n, batch, hidden = 250_000, 8192, 2 * d if dtype == torch.float32 else d
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    ip, ix, _ = E.graph_from_coo(n, *(torch.randint(0, n, (n,), device="cuda", generator=g, dtype=torch.int32) for _ in range(2)))
    X = torch.randn(n, d, device="cuda", generator=g).to(dtype)
    Ws = [(0.1 * torch.randn(hidden, 2 * k, device="cuda", generator=g)).to(dtype) for k in (d, hidden)]
    b = E.Blocks(n, batch, [25, 15], "cuda")
    dH = torch.randn(batch, hidden, device="cuda", generator=g).to(dtype)
    rows, es = b.caps[-1][0], X.element_size()
    assert rows * (hidden + 2 * d) * es >= 256 << 20 > batch * 3 * hidden * es
    H, ctx = E.sage_forward(_sampled(b, ip, ix, g, 0), X, Ws)
    scratch = torch.empty(E.binding.sage_backward_scratch_bytes(b, X, Ws), dtype=torch.uint8, device="cuda")
    dWs, dX = E.sage_backward(b, X, Ws, ctx, dH, scratch=scratch)
    for step in range(1, 9):
        _sampled(b, ip, ix, g, step)
        E.sage_forward(b, X, Ws, ctx=ctx, H_out=H)
        E.sage_backward(b, X, Ws, ctx, dH, dWs=dWs, dX_rows=dX, scratch=scratch)
        torch.cuda.synchronize()
        cat = E.binding.sage_ctx_views(b, X, Ws, ctx)[1][0][:batch].double()
        dZ = dH.double() * (H > 0)
        # no chain of additions is longer than the rows of a split and the splits: 8192 / 148 + 148, doubled for the tensor core's
        # sums, which may truncate
        bound = 512 * 2.0 ** -24 * (dZ.abs().T @ cat.abs())
        assert bool(((dWs[1].double() - dZ.T @ cat).abs() <= bound).all()), step


def _sampled(b, ip, ix, g, step):
    seeds = torch.randperm(ip.numel() - 1, device="cuda", generator=g)[: b.caps[0][0]].to(torch.int32)
    E.sample_khop(ip, ix, seeds, b, 77, step, defer_transpose=True)
    return b
