"""Sampling over every tile of destinations that the fanout and the batch choose, with uniform and weighted draws: rows of
one and two entries beyond the fanout, hubs, rows without weight, batches that fill no tile, many more tiles than a look-back
round reads; and the local ids are idle again afterwards, also when no transposition releases them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import oracle  # noqa: E402
import paper_2511_20564_b200 as E  # noqa: E402
from helpers import assert_blocks_equal  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    rng = np.random.default_rng(5)
    n = 30_000
    deg = rng.integers(0, 9, n)
    deg[:200] = rng.integers(90, 135, 200)
    deg[200:204] = (5000, 70_000, 101, 102)
    indptr = np.zeros(n + 1, np.int64)
    np.cumsum(deg, out=indptr[1:])
    indices = rng.integers(0, n, indptr[-1]).astype(np.int32)
    q = rng.integers(0, 4, indices.size).astype(np.uint32) * rng.integers(1, 1 << 16, indices.size).astype(np.uint32)
    q[indptr[150]:indptr[160]] = 0
    return n, indptr, indices, q


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("batch,fanouts", [(1, [1]), (3, [128]), (257, [100]), (20_000, [100]), (20_000, [1, 2]), (4097, [15, 10]),
                                           (700, [25, 15]), (500, [7, 5, 3, 2])])
def test_blocks(graph, batch, fanouts, weighted):
    n, indptr, indices, q = graph
    rng = np.random.default_rng(batch)
    seeds = rng.permutation(np.r_[0:204, rng.permutation(np.arange(204, n))[: max(batch - 204, 0)]])[:batch].astype(np.int32)
    ip, ix = torch.from_numpy(indptr).cuda(), torch.from_numpy(indices).cuda()
    cum = E.edge_cumulate(ip, torch.from_numpy(q.view(np.int32)).cuda()) if weighted else None
    want_cum = oracle.edge_cumulate(indptr, q) if weighted else None
    blocks = E.Blocks(n, batch, fanouts, "cuda")
    for step, transpose in ((0, True), (1, False), (2, True)):
        E.sample_khop(ip, ix, torch.from_numpy(seeds).cuda(), blocks, 77, step, edge_cum=cum, transpose=transpose)
        if not transpose:
            E.blocks_transpose(blocks)
        want = oracle.sample_khop(indptr, indices, seeds, fanouts, 77, step, edge_cum=want_cum)
        torch.cuda.synchronize()
        assert_blocks_equal(blocks.to_host(), want)


@pytest.mark.parametrize("batch,fanouts", [(3000, [4, 3]), (40, [5, 100, 2])])
def test_ids_out_of_range_are_flagged_at_the_hop_that_meets_them(graph, batch, fanouts):
    """One entry of one node beyond the graph: the status of the hops that draw from that node's row has the bit in every
    sample, whichever tile of the hop flags it and however early, and no other hop's has; the entry becomes its row's node."""
    n, _, _, _ = graph
    rng = np.random.default_rng(batch)
    deg = np.full(n, 2)
    indptr = np.r_[0, np.cumsum(deg)].astype(np.int64)
    indices = rng.integers(0, n, 2 * n).astype(np.int32)
    seeds = rng.permutation(n)[:batch].astype(np.int32)
    clean = oracle.sample_khop(indptr, indices, seeds, fanouts, 3, 0)
    new = clean[1]["src_nodes"][clean[0]["n_src"]:]          # met by the second hop first: the third one draws from it
    late = clean[0]["src_nodes"][-1]                         # the second hop's last destination
    ip = torch.from_numpy(indptr).cuda()
    blocks = E.Blocks(n, batch, fanouts, "cuda")
    sd = torch.from_numpy(seeds).cuda()
    for node, first_hop in ((late, 1), (new[len(new) // 2], 2)):
        if first_hop >= len(fanouts):
            continue
        bad = indices.copy()
        bad[indptr[node]] = n + 7
        ix = torch.from_numpy(bad).cuda()
        for step in range(20):
            E.sample_khop(ip, ix, sd, blocks, 3, step)
            assert [int(s) & 1 for s in blocks.counts[:, 3].tolist()] == [int(h >= first_hop) for h in range(len(fanouts))]
        b = blocks.to_host()[first_hop]
        at = b["indptr"][np.flatnonzero(b["src_nodes"][: b["n_dst"]] == node)[0]]
        assert b["nbr_global"][at] == node
    E.sample_khop(ip, torch.from_numpy(indices).cuda(), sd, blocks, 3, 0)
    assert_blocks_equal(blocks.to_host(), clean)
