"""The radix sort behind graph ingest and block transposition at its edges: one element, tiles that are full, one short and
one over, both tile sizes, every number of digits and passes, one key for all elements, keys out of range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2511_20564_b200 as E  # noqa: E402

pytestmark = pytest.mark.gpu


def check_ingest(n, row, col):
    ptr, idx, bad = E.graph_from_coo(n, torch.from_numpy(row).cuda(), torch.from_numpy(col).cuda())
    order = np.lexsort((col, row))
    want_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(row, minlength=n), out=want_ptr[1:])
    assert int(bad) == 0
    assert np.array_equal(ptr.cpu().numpy(), want_ptr) and np.array_equal(idx.cpu().numpy(), col[order])
    cptr, crow, ceid, bad = E.csr_transpose(ptr, idx, n)
    back = np.argsort(col[order], kind="stable")
    np.cumsum(np.bincount(col, minlength=n), out=want_ptr[1:])
    assert int(bad) == 0
    assert np.array_equal(cptr.cpu().numpy(), want_ptr) and np.array_equal(ceid.cpu().numpy(), back)
    assert np.array_equal(crow.cpu().numpy(), row[order][back])


@pytest.mark.parametrize("m", [1, 31, 4095, 4096, 4097, 8193, 70_001])
@pytest.mark.parametrize("n", [1, 200, 1024, 60_000, 1_000_000, 9_000_000, 20_000_000])
def test_sizes(m, n):
    rng = np.random.default_rng(m + n)
    check_ingest(n, rng.integers(0, n, m).astype(np.int32), (n * rng.random(m) ** 4).astype(np.int32))


@pytest.mark.parametrize("m", [2 * 148 * 8192 - 1, 2 * 148 * 8192 + 8191])
def test_line_between_the_tile_sizes(m):
    rng = np.random.default_rng(m)
    row, col = rng.integers(0, 300_000, m).astype(np.int32), (300_000 * rng.random(m) ** 6).astype(np.int32)
    check_ingest(300_000, row, col)
    check_ingest(300_000, np.full(m, 299_999, np.int32), col)


def test_ids_out_of_range_are_flagged_and_count_as_zero():
    row, col = np.array([5, -1, 2, 7], np.int32), np.array([1, 2, 9, 3], np.int32)
    ptr, idx, bad = E.graph_from_coo(8, torch.from_numpy(row).cuda(), torch.from_numpy(col).cuda())
    assert int(bad) != 0
    assert ptr.cpu().tolist() == [0, 1, 1, 2, 2, 2, 3, 3, 4] and idx.cpu().tolist() == [2, 0, 1, 3]


def test_blocks_can_be_transposed_again():
    rng = np.random.default_rng(3)
    n, m = 50_000, 400_000
    ids = [torch.from_numpy((n * rng.random(m) ** 3).astype(np.int32)).cuda() for _ in range(2)]
    ptr, idx, _ = E.graph_from_coo(n, *ids)
    seeds = torch.arange(0, 3000, dtype=torch.int32, device="cuda")
    got = []
    for again in (0, 1, 2):
        b = E.Blocks(n, 3000, [12, 7], "cuda")
        E.sample_khop(ptr, idx, seeds, b, 11, 4, transpose=again == 0)
        for _ in range(again):
            E.blocks_transpose(b)
        torch.cuda.synchronize()
        c = b.counts.cpu().numpy()
        got.append([t[k][:e].cpu().numpy() for t, row in zip(b.t, c)
                    for k, e in (("csc_ptr", row[1] + 1), ("csc_row", row[2]), ("csc_eid", row[2]), ("csc_col", row[2]))])
    for other in got[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(got[0], other))


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    """The sorting entry points compiled so that a look-back of the sort ends at its first round without progress."""
    import ctypes
    import os
    import subprocess
    from paper_2511_20564_b200 import build
    csrc = os.path.join(build.HERE, "csrc")
    so = str(tmp_path_factory.mktemp("sort") / "impatient.so")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-shared"] + build.NVCC_FLAGS +
                          ["-DE2EGREC_SORT_SPIN_LIMIT=0", "-o", so] + [os.path.join(csrc, f) for f in ("ingest.cu", "sampler.cu", "api.cu")])
    L, real = ctypes.CDLL(so), E.binding.lib()
    for fn in ("graph_from_coo", "csr_transpose", "sample_khop", "sample_khop_workspace", "sampler_scratch_init"):
        getattr(L, "e2egrec_" + fn).argtypes, getattr(L, "e2egrec_" + fn).restype = getattr(real, "e2egrec_" + fn).argtypes, getattr(real, "e2egrec_" + fn).restype
    return L


@pytest.mark.parametrize("n,m", [(200, 60_000), (9_000_000, 300_000), (300_000, 2 * 148 * 8192)])
def test_ingest_whose_waits_run_out(impatient, n, m, monkeypatch):
    """The status says so and no entry is reachable through the offsets; rows are those of entries that exist."""
    rng = np.random.default_rng(m)
    row, col = (torch.from_numpy((n * rng.random(m) ** 4).astype(np.int32)).cuda() for _ in range(2))
    good_ptr, good_idx, _ = E.graph_from_coo(n, row, col)
    want_ptr, want_row, want_eid, _ = E.csr_transpose(good_ptr, good_idx, n)
    monkeypatch.setattr(E.binding, "lib", lambda: impatient)
    poison = torch.full((8 * m,), 0x7F7F7F7F, dtype=torch.int32, device="cuda")      # what the buffers below are cut from
    del poison
    ptr, idx, bad = E.graph_from_coo(n, row, col)
    assert int(bad) in (0, 4) and (m < 1_000_000 or int(bad) == 4)
    assert not bool(ptr.any()) if int(bad) else torch.equal(ptr, good_ptr) and torch.equal(idx, good_idx)
    ptr, rows, eid, bad = E.csr_transpose(good_ptr, good_idx, n)
    assert int(bad) in (0, 4) and (m < 1_000_000 or int(bad) == 4)
    assert not bool(ptr.any()) if int(bad) else torch.equal(ptr, want_ptr) and torch.equal(rows, want_row) and torch.equal(eid, want_eid)
    assert 0 <= int(rows.min()) and int(rows.max()) < n


def test_sample_whose_transposition_waits_run_out(impatient, monkeypatch):
    rng = np.random.default_rng(5)
    n, m = 400_000, 4_000_000
    ptr, idx, _ = E.graph_from_coo(n, *(torch.from_numpy(rng.integers(0, n, m).astype(np.int32)).cuda() for _ in range(2)))
    seeds = torch.arange(0, 8000, dtype=torch.int32, device="cuda")
    want = E.Blocks(n, 8000, [9, 8], "cuda")
    E.sample_khop(ptr, idx, seeds, want, 3, 1)
    monkeypatch.setattr(E.binding, "lib", lambda: impatient)
    b = E.Blocks(n, 8000, [9, 8], "cuda")
    for t in b.t:
        for k in ("csc_row", "csc_eid", "csc_col"):
            t[k].fill_(0x7F7F7F7F)
    E.sample_khop(ptr, idx, seeds, b, 3, 1)
    torch.cuda.synchronize()
    assert torch.equal(b.counts[:, :3], want.counts[:, :3]) and int(b.counts[1, 3]) == 4
    for h, (got, ref) in enumerate(zip(b.t, want.t)):
        n_src, n_edges = int(b.counts[h, 1]), int(b.counts[h, 2])
        assert torch.equal(got["col"][:n_edges], ref["col"][:n_edges])
        if int(b.counts[h, 3]):
            assert not bool(got["csc_ptr"][: n_src + 1].any())
        else:
            for k in ("csc_row", "csc_eid", "csc_col"):
                assert torch.equal(got[k][:n_edges], ref[k][:n_edges])


@pytest.mark.parametrize("m", [5000, 2 * 148 * 8192 + 100])
def test_keys_that_neighbours_share(m):
    """Warps that see one key, two keys in turn, and a hub in between others: what the ranking does with lanes of one digit."""
    n, at = 70_000, np.arange(m)
    rng = np.random.default_rng(m)
    spread = rng.integers(0, n, m)
    for row in (at // 40 % n, np.where(at % 2, 5, 66_000), np.where(rng.random(m) < 0.3, 1234, spread)):
        check_ingest(n, row.astype(np.int32), spread.astype(np.int32))
        check_ingest(n, spread.astype(np.int32), row.astype(np.int32))
