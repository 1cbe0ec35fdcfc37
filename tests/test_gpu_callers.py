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
