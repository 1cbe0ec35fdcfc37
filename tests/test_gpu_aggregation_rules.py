"""Rules of the aggregation's dispatch that other tests do not reach: inputs whose windows are shared by four warps, rows four
gigabytes apart, blocks with more windows than the grid has blocks, upstream gradients that lie on no 16-byte boundary."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2511_20564_b200 as E  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 8), ("bf16", 64), ("f32", 20), ("f32", 32), ("f32", 64)])
def test_windows_of_large_inputs(dtype, d):
    """2^24 entries and a ragged rest: runs of 256 entries, two stretches per warp for rows of up to 128 bytes."""
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    n, n_rows = 40_000, 1000
    lens = torch.randint(0, 12, (n,), device="cuda", generator=g)
    lens[::97] = 0
    lens[[3, 77, n // 2, n - 1]] = torch.tensor([5_000_000, 8191, 12_000_000, 1025], device="cuda")
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(lens, 0)
    m = int(ptr[-1])
    assert m >= 1 << 24
    idx = torch.randint(0, n_rows, (m,), device="cuda", generator=g, dtype=torch.int32)
    X = torch.randint(-8, 9, (n_rows, d), device="cuda", generator=g).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    w = torch.randint(1, 3, (n_rows,), device="cuda", generator=g).float()
    # sums of whole numbers below 2^24 in size: exact in any order, then rounded to the storage type
    seg = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)

    def sums(rows):
        out = torch.zeros(n, d, dtype=torch.float64, device="cuda")
        for s in range(0, m, 1 << 22):
            out.index_add_(0, seg[s:s + (1 << 22)], rows[idx[s:s + (1 << 22)].long()])
        return out

    plain, weighted = sums(X.double()), sums(X.double() * w.double()[:, None])
    assert float(plain.abs().max()) < 2 ** 24 and float(weighted.abs().max()) < 2 ** 24
    out, _ = E.aggregate_forward(ptr, idx, X, sum_only=True)
    assert torch.equal(out.double(), plain.to(out.dtype).double())
    out, _ = E.aggregate_backward(ptr, idx, w, X)
    assert torch.equal(out.double(), weighted.to(out.dtype).double())


def test_rows_four_gigabytes_apart():
    if torch.cuda.mem_get_info()[0] < 16 << 30:
        pytest.skip("needs 16 GB of device memory")
    d, stride = 64, (1 << 30) + 4                            # fp32 values: 16 bytes more than 4 GB
    store = torch.empty(2 * stride + d, device="cuda")
    X = store.as_strided((3, d), (stride, 1))
    small = torch.randint(-8, 9, (3, d), device="cuda").float()
    X.copy_(small)
    ptr = torch.tensor([0, 3, 3, 5, 105], dtype=torch.int64, device="cuda")
    idx = torch.arange(105, dtype=torch.int32, device="cuda") % 3
    assert torch.equal(E.aggregate_forward(ptr, idx, X, sum_only=True)[0], E.aggregate_forward(ptr, idx, small, sum_only=True)[0])
    b = E.Blocks(3, 3, [2], "cuda")
    gi = torch.tensor([1, 2, 0, 2, 0, 1], dtype=torch.int32, device="cuda")
    E.sample_khop(torch.tensor([0, 2, 4, 6], dtype=torch.int64, device="cuda"), gi, torch.arange(3, dtype=torch.int32, device="cuda"), b, 1, 0)
    W = torch.randn(16, 2 * d, device="cuda")
    assert torch.equal(E.sage_forward(b, X, [W])[0], E.sage_forward(b, small, [W])[0])


def _one_layer(dtype, d, hidden, seeds, fanout, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    m = 30 * n
    ids = [(n * torch.rand(m, device="cuda", generator=g) ** p).to(torch.int32) for p in (1, 3)]
    ptr, idx, _ = E.graph_from_coo(n, *ids)
    b = E.Blocks(n, seeds, [fanout], "cuda")
    E.sample_khop(ptr, idx, torch.randperm(n, device="cuda", generator=g)[:seeds].to(torch.int32), b, 5, 1)
    X = torch.randn(n, d, device="cuda", generator=g).to(dtype)
    W = (0.1 * torch.randn(hidden, 2 * d, device="cuda", generator=g)).to(dtype)
    H, ctx = E.sage_forward(b, X, [W], acts=[0])[:2]
    return b, X, W, ctx, g


@pytest.mark.parametrize("d", [32, 100, 128])
def test_blocks_with_more_windows_than_the_grid_has_blocks(d):
    """One identity layer in fp32: dX = dH W_self for the destinations plus the transposed mean of dH W_agg."""
    hidden, seeds = 16, 20_000
    b, X, W, ctx, g = _one_layer(torch.float32, d, hidden, seeds, 30, 60_000)
    n_dst, n_src, n_edges, status = b.counts[0].tolist()
    assert status == 0 and n_edges > 148 * 4 * 512 and n_src > n_dst
    dH = torch.randn(seeds, hidden, device="cuda", generator=g)
    _, dX = E.sage_backward(b, X, [W], ctx, dH, acts=[0])
    ip = b.t[0]["indptr"][: n_dst + 1].long()
    cnt = ip[1:] - ip[:-1]
    row, col = torch.repeat_interleave(torch.arange(n_dst, device="cuda"), cnt), b.t[0]["col"][:n_edges].long()
    inv = 1.0 / cnt.clamp(min=1).double()

    def adjoint(dh, w):
        out = torch.zeros(n_src, d, dtype=torch.float64, device="cuda")
        out[:n_dst] = dh @ w[:, :d]
        return out.index_add_(0, col, ((dh @ w[:, d:]) * inv[:, None])[row])

    want, mass = adjoint(dH.double(), W.double()), adjoint(dH.double().abs(), W.double().abs())
    terms = torch.bincount(col, minlength=n_src).double()[:, None] + hidden + 4      # additions on the way to an element
    err = (dX[:n_src].double() - want).abs()
    assert bool((err <= terms * 2.0 ** -24 * mass + 1e-300).all()), float((err - terms * 2.0 ** -24 * mass).max())


@pytest.mark.parametrize("dtype,hidden", [("bf16", 64), ("bf16", 24), ("f32", 20), ("f32", 64)])
def test_upstream_gradients_on_no_boundary(dtype, hidden):
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    b, X, W, ctx, g = _one_layer(dt, 64, hidden, 300, 6, 5_000)
    wide = torch.randn(2, 300, hidden + 3, device="cuda", generator=g).to(dt)
    dHs = [wide[r, :, 3:] for r in range(2)]
    (dW1,), dX1 = E.sage_backward(b, X, [W], ctx, dHs[0])
    (dW2,), dX2 = E.sage_backward(b, X, [W], ctx, dHs[0].contiguous())
    assert torch.equal(dW1, dW2) and torch.equal(dX1, dX2)
    (dW1,), dX1 = E.sage_backward_multi(b, X, [W], ctx, dHs)
    (dW2,), dX2 = E.sage_backward_multi(b, X, [W], ctx, [h.contiguous() for h in dHs])
    assert torch.equal(dW1, dW2) and all(torch.equal(p, q) for p, q in zip(dX1, dX2))
    assert not np.array_equal(dX1[0].float().cpu().numpy(), dX1[1].float().cpu().numpy())


@pytest.mark.parametrize("dtype,d,m", [("bf16", 64, 48_000_000), ("bf16", 40, 50_000_001), ("f32", 20, 48_000_001), ("f32", 32, 47_999_000)])
def test_windows_that_four_warps_share(dtype, d, m):
    """As many entries as take two stretches per warp, and one window less: hubs, short and empty segments, exact sums."""
    g = torch.Generator(device="cuda")
    g.manual_seed(d)
    n, n_rows = 1_200_000, 3000
    lens = torch.randint(0, 30, (n,), device="cuda", generator=g)
    lens[::7] = 0
    lens[5::1000] = 4000
    lens[[3, 77, n // 2]] = torch.tensor([2_000_000, 8191, 1025], device="cuda")
    lens[n - 1] = 0
    lens[n - 1] = m - lens.sum()
    assert int(lens[n - 1]) > 1_000_000
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(lens, 0)
    idx = torch.randint(0, n_rows, (m,), device="cuda", generator=g, dtype=torch.int32)
    X = torch.randint(-4, 5, (n_rows, d), device="cuda", generator=g).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    w = torch.randint(1, 3, (n_rows,), device="cuda", generator=g).float()
    # prefix sums of whole numbers of up to 8 are exact in 64 bits; sums below 2^24 are exact in 32, in any order
    ids, run = idx.long(), torch.zeros(m + 1, dtype=torch.float64, device="cuda")
    for scale, out in ((None, E.aggregate_forward(ptr, idx, X, sum_only=True)[0]), (w, E.aggregate_backward(ptr, idx, w, X)[0])):
        for c in range(d):
            column = X[:, c].double() if scale is None else X[:, c].double() * scale.double()
            torch.cumsum(column[ids], 0, out=run[1:])
            want = run[ptr[1:]] - run[ptr[:-1]]
            assert float(want.abs().max()) < 2 ** 24
            assert torch.equal(out[:, c].double(), want.to(out.dtype).double()), c
