"""Whole-graph segment reduction (one warp per stretch of entries) at the shapes where its walk can go wrong: segments that
end on stretch and window boundaries, one segment over everything, runs of empty segments longer than the walk steps
through, lengths around the limit between the short and the long form, every row width class."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2511_20564_b200 as E  # noqa: E402

pytestmark = pytest.mark.gpu

LENGTHS = {
    "one_entry": [1],
    "one_segment": [5000],
    "empty_ends": [0, 0, 3, 0, 700, 0, 0],
    "short_and_long": [1, 8, 9, 7, 16, 17, 31, 32, 33, 63, 64, 65, 2, 0, 128, 1, 1, 1] * 9,
    "stretch_sized": [32, 64, 128, 256, 96, 32, 512, 1024, 1, 31, 480],
    "long_gaps": [5] + [0] * 1000 + [40] + [0] * 129 + [2] + [0] * 127 + [9] + [0] * 31 + [1] + [0] * 64 + [300],
}


@pytest.mark.parametrize("lengths", sorted(LENGTHS))
@pytest.mark.parametrize("dtype,d", [("bf16", 8), ("bf16", 40), ("bf16", 64), ("bf16", 104), ("bf16", 256), ("bf16", 512),
                                     ("f32", 4), ("f32", 20), ("f32", 32), ("f32", 100), ("f32", 128), ("f32", 1024)])
def test_walk(lengths, dtype, d):
    rng = np.random.default_rng(len(lengths) * 1000 + d)
    lens = np.asarray(LENGTHS[lengths], np.int64)
    ptr = np.zeros(lens.size + 1, np.int64)
    np.cumsum(lens, out=ptr[1:])
    m, n_rows = int(ptr[-1]), 50
    idx = rng.integers(0, n_rows, m).astype(np.int32)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    X = torch.from_numpy(rng.standard_normal((n_rows, d)).astype(np.float32)).to(dt)
    w = rng.uniform(-2, 2, n_rows).astype(np.float32)
    pd, ix, Xd = torch.from_numpy(ptr).cuda(), torch.from_numpy(idx).cuda(), X.cuda()
    rows = X.to(torch.float64).numpy()[idx]
    seg = np.repeat(np.arange(lens.size), lens)

    def sums(values):
        out = np.zeros((lens.size, d))
        np.add.at(out, seg, values)
        return out

    def check(got, want, mass):
        # n additions and two roundings of factors in fp32, then the rounding to the storage type
        bound = (lens[:, None] + 3) * 2.0 ** -24 * mass + (2.0 ** -8 if dtype == "bf16" else 2.0 ** -23) * np.abs(want)
        err = np.abs(got.double().cpu().numpy() - want)
        assert (err <= bound + 1e-300).all(), (err - bound).max()

    out, _ = E.aggregate_forward(pd, ix, Xd)
    inv = (1.0 / np.maximum(lens, 1))[:, None]
    check(out, sums(rows) * inv, sums(np.abs(rows)) * inv)
    out, _ = E.aggregate_forward(pd, ix, Xd, sum_only=True)
    check(out, sums(rows), sums(np.abs(rows)))
    dX, _ = E.aggregate_backward(pd, ix, torch.from_numpy(w).cuda(), Xd)
    wr = rows * w.astype(np.float64)[idx][:, None]
    check(dX, sums(wr), sums(np.abs(wr)))


def test_as_many_segments_as_the_entry_point_takes():
    """2^31 - 1 segments, with entries in the first and the last ones: windows of 32 segments that begin among the last and
    reach beyond 2^31.  52 GB of offsets and rows."""
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 70 << 30:
        pytest.skip("needs 70 GB of device memory")
    n, d = (1 << 31) - 1, 4
    tail = torch.tensor([3, 0, 40, 1, 300, 0, 10_000], dtype=torch.int64)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = 2                                              # segment 0: two entries
    ptr[n + 1 - tail.numel():] += torch.cumsum(tail, 0).cuda()
    m = 2 + int(tail.sum())
    rng = np.random.default_rng(9)
    X = torch.from_numpy(rng.integers(-8, 9, (50, d)).astype(np.float32))       # sums of whole numbers: exact in any order
    idx = torch.from_numpy(rng.integers(0, 50, m).astype(np.int32))
    out = torch.empty(n, d, device="cuda")
    E.aggregate_forward(ptr, idx.cuda(), X.cuda(), out=out, sum_only=True)
    rows = X[idx.long()]
    cuts = [0, 2] + (2 + torch.cumsum(tail, 0)).tolist()
    want = torch.stack([rows[a:b].sum(0) for a, b in zip(cuts, cuts[1:])])
    assert torch.equal(out[0].cpu(), want[0]) and torch.equal(out[n - tail.numel():].cpu(), want[1:])
    for a in range(1, n - tail.numel(), 1 << 28):            # everything between is empty
        assert not bool(out[a:min(a + (1 << 28), n - tail.numel())].any())
