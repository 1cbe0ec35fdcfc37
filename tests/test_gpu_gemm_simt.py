"""The fp32-FMA product in its three operand layouts (through the gated fusion, which uses all of them) at the edges of its
tiles: sizes around 32 and 64, rows that are no multiple of 16 bytes, one row, one column, more rows than one split takes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2511_20564_b200 as E  # noqa: E402

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24


@pytest.mark.parametrize("d", [1, 3, 20, 31, 32, 33, 63, 64, 65, 130])
@pytest.mark.parametrize("rows", [1, 63, 64, 65, 300, 1500])
def test_gate_in_fp32(rows, d):
    rng = np.random.default_rng(rows * 1000 + d)
    alloc = (rows + 127) // 128 * 128
    mk = lambda r: torch.from_numpy(rng.standard_normal((r, d)).astype(np.float32)).cuda()
    F, dFused, Wg, bg = mk(alloc), mk(alloc), mk(d) / d ** 0.5, mk(1)[0]
    fused, gate, ws = E.gate_fusion_forward(F, rows, Wg, bg)
    f, df, w, b = (t.double().cpu().numpy() for t in (F[:rows], dFused[:rows], Wg, bg))
    g = 1 / (1 + np.exp(-(f @ w.T + b)))
    # d products and additions, one more for the bias; the sigmoid's slope is at most 1/4, its own error a few units
    err_g = 0.25 * (d + 2) * EPS * (np.abs(f) @ np.abs(w.T) + np.abs(b)) + 8 * EPS
    assert (np.abs(gate[:rows].double().cpu().numpy() - g) <= err_g).all()
    assert (np.abs(fused[:rows].double().cpu().numpy() - g * f) <= (err_g + 2 * EPS) * np.abs(f)).all()

    gate = torch.sigmoid(mk(alloc))
    dF, dWg, dbg = E.gate_fusion_backward(dFused, F, rows, gate, Wg, ws)
    g = gate[:rows].double().cpu().numpy()
    dpre = df * f * g * (1 - g)                          # five fp32 roundings
    mass = np.abs(dpre)
    assert (np.abs(dWg.double().cpu().numpy() - dpre.T @ f) <= (rows + 8) * EPS * (mass.T @ np.abs(f)) + 1e-30).all()
    assert (np.abs(dbg.double().cpu().numpy() - dpre.sum(0)) <= (rows + 8) * EPS * mass.sum(0) + 1e-30).all()
    bound = (d + 10) * EPS * (mass @ np.abs(w)) + 4 * EPS * np.abs(df * g)
    assert (np.abs(dF[:rows].double().cpu().numpy() - (dpre @ w + df * g)) <= bound + 1e-30).all()


@pytest.mark.parametrize("rows,d,hidden", [(50_000, 256, 256), (12_000, 256, 256), (6_000, 1024, 1024), (35_000, 256, 64), (4_096, 160, 320),
                                           (150, 64, 64)])
def test_weight_gradients_over_many_rows(rows, d, hidden):
    """Weight gradients contract over all rows of a batch.  The error of a sum of independent terms, relative to the sums'
    norm, is below half a unit times the square root of the longest chain of additions, which is that of 148 splits of
    the rows at most: 148 + rows / 148.  A chain over a tenth of 50 k rows misses it by a factor of two."""
    g = torch.Generator(device="cuda").manual_seed(rows + d)
    mk = lambda *s: torch.randn(*s, device="cuda", generator=g)
    ptr = torch.arange(rows + 1, device="cuda", dtype=torch.int64)
    idx = torch.randint(0, rows, (rows,), device="cuda", generator=g, dtype=torch.int32)
    blocks = E.Blocks(rows, rows, [1], "cuda")
    E.sample_khop(ptr, idx, torch.arange(rows, dtype=torch.int32, device="cuda"), blocks, 1, 1)
    X, W, dH = mk(rows, d), mk(hidden, 2 * d) * 0.05, mk(rows, hidden)
    _, ctx = E.sage_forward(blocks, X, [W], acts=[0])
    dWs, _ = E.sage_backward(blocks, X, [W], ctx, dH, acts=[0])
    cat = E.sage_ctx_views(blocks, X, [W], ctx)[0][0][:rows]
    want = dH.double().T @ cat.double()
    err = float((dWs[0].double() - want).norm() / want.norm())
    assert err <= 0.5 * EPS * (148 + rows / 148) ** 0.5 + EPS, err


@pytest.mark.parametrize("rows,d", [(65_536, 256), (65_536, 257), (65_537, 33), (70_000, 4)])
def test_gate_in_fp32_where_the_kernels_change(rows, d):
    """The last products of the asynchronous kernel and the first of the other one, by rows and by tiles."""
    test_gate_in_fp32(rows, d)


@pytest.mark.parametrize("rows,d,hidden", [(65_536, 64, 128), (65_537, 64, 128), (90_000, 100, 72)])
def test_weight_gradients_where_the_kernels_change(rows, d, hidden):
    test_weight_gradients_over_many_rows(rows, d, hidden)
