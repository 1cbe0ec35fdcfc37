"""What a user of this library has it do: the workloads that its speed is judged by.

Every case goes through the public entry points of the package, on inputs drawn on the GPU from a seed: bipartite
user-item graphs with bounded-Zipf popularity (both directions stored, parallel edges kept), N(0, 1) features, Glorot
weights, seed batches drawn in proportion to a node's activity.  A case is one of these kinds:

  serve           embeddings of a few users: k-hop sample and encoder forward, nothing kept for a backward pass
  step            one training step of the GNN branch: sample, forward, backward (weight and feature gradients)
  multitask       the two-task step: SSL loss, both gradients through one backward pass, their norms, one GradNorm update
  lightgcn        sample, LightGCN propagation over the sampled blocks, its adjoint (importance-weighted sampling)
  joint           the joint step of encoder and ranking tower on user-item pairs (with or without the gated fusion)
  whole_mean      mean aggregation over a whole directed graph and its transpose
  whole_lightgcn  LightGCN over a whole graph, forward and adjoint
  ingest          edge list -> canonical CSR -> CSC
"""
import numpy as np
import torch

import paper_2511_20564_b200 as E

DEV = "cuda"
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


# ------------------------------------------------------------------------------------------------- the cases

# Graphs of this repository's benchmark: 5 k, 500 k and 6.25 M nodes with 40 k, 10 M and 125 M interactions.
TINY = dict(users=2_000, items=3_000, interactions=40_000, alpha=1.2, q=0.0)
MEDIUM = dict(users=200_000, items=300_000, interactions=10_000_000, alpha=1.2, q=0.0)
LARGE = dict(users=2_500_000, items=3_750_000, interactions=125_000_000, alpha=1.05, q=10.0)
NO_GRAPH = dict(users=0, items=0, interactions=0, alpha=0.0, q=0.0)


def _sampled(name, kind, graph, dtype, dim, hidden, fanouts, batch, **more):
    return dict(graph, name=name, kind=kind, dtype=dtype, dim=dim, hidden=hidden, fanouts=fanouts, batch=batch, **more)


def listed():
    return [
        # online inference for the users of one request: the smallest call, bound by latency and launches
        _sampled("serve_64_bf16", "serve", MEDIUM, "bf16", 128, 128, "15-10", 64, bias=False),
        # a small experiment in fp32: the tiny configuration
        _sampled("step_tiny_f32", "step", TINY, "f32", 64, 64, "10-5", 256, bias=False),
        # the ordinary training step: the medium configuration
        _sampled("step_medium_bf16", "step", MEDIUM, "bf16", 128, 128, "15-10", 4096, bias=False),
        # the two-hop shape 25, 15 with a last, incomplete batch, widths that divide into no tile, fp32 and biases
        _sampled("step_ragged_f32", "step", MEDIUM, "f32", 100, 72, "25-15", 777, bias=True),
        # the largest training step: model, fanouts and batch of the large configuration, its graph at one eighth (the
        # feature table, 3.2 GB, is far larger than the L2 cache)
        _sampled("step_large_bf16", "step", LARGE, "bf16", 256, 256, "20-10-5", 8192, bias=False),
        # recommendation and self-supervised gradient through the encoder together, task weights updated
        _sampled("multitask_bf16", "multitask", MEDIUM, "bf16", 128, 128, "15-10", 4096, bias=False),
        # the default backbone and sampler of the method: LightGCN on one hop of 100 weighted neighbours
        _sampled("lightgcn_1hop100_bf16", "lightgcn", MEDIUM, "bf16", 128, 128, "100", 4096, weighted=True),
        # encoder and ranking tower trained together on 4096 user-item pairs
        _sampled("joint_bf16", "joint", MEDIUM, "bf16", 128, 128, "15-10", 4096, dense=64, h1=512, h2=256, gate=False),
        # the same with the gated fusion and a batch that is no multiple of the tile
        _sampled("joint_gate_ragged_bf16", "joint", MEDIUM, "bf16", 128, 128, "15-10", 1000, dense=64, h1=512, h2=256, gate=True),
        # aggregation without sampling: the full-graph configuration (5 M nodes, 10^8 entries)
        dict(NO_GRAPH, name="whole_mean_bf16", kind="whole_mean", dtype="bf16", dim=64, nodes=5_000_000, entries=100_000_000, alpha=1.1),
        # three LightGCN layers over the whole medium graph in fp32
        dict(MEDIUM, name="whole_lightgcn_f32", kind="whole_lightgcn", dtype="f32", dim=64, layers=3),
        # a day's interactions into a graph: set-up of the medium configuration
        dict(MEDIUM, name="ingest_20m", kind="ingest"),
    ]


KINDS = ["serve"] * 2 + ["step"] * 4 + ["multitask"] + ["lightgcn"] * 2 + ["joint"] * 2 + ["whole_mean"] * 2 + ["whole_lightgcn", "ingest"]


def _log(rng, lo, hi):
    return int(round(float(lo) * (float(hi) / lo) ** rng.random()))


def draw(rng):
    largest = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= largest:
            return c


def _draw(rng):
    kind = rng.choice(KINDS)
    if kind == "whole_mean":
        n = _log(rng, 10_000, 5_000_000)
        dtype = rng.choice(["bf16", "bf16", "f32"])
        return dict(NO_GRAPH, kind=kind, dtype=dtype, dim=rng.choice([32, 64, 64, 100, 128, 256]) if dtype == "f32" else rng.choice([64, 64, 104, 128, 256]),
                    nodes=n, entries=min(100_000_000, int(n * rng.uniform(4, 20))), alpha=rng.choice([1.05, 1.1, 1.2]))
    nodes = _log(rng, 5_000, 2_000_000 if kind in ("whole_lightgcn", "ingest") else 6_250_000)
    users = int(nodes * rng.uniform(0.2, 0.8))
    g = dict(users=users, items=nodes - users, interactions=int(nodes * rng.uniform(4, 20)), alpha=rng.choice([1.05, 1.2]), q=rng.choice([0.0, 10.0]))
    if kind == "ingest":
        return dict(g, kind=kind)
    if kind == "whole_lightgcn":
        return dict(g, kind=kind, dtype=rng.choice(["bf16", "f32"]), dim=rng.choice([32, 64, 104, 128]), layers=rng.randint(1, 4))
    dtype = "bf16" if rng.random() < 0.75 else "f32"
    dim = rng.choice([64, 128, 128, 256, 256, 104] if dtype == "bf16" else [32, 64, 100, 128, 256])
    hidden = dim if kind in ("multitask", "lightgcn") or rng.random() < 0.7 else rng.choice([64, 128, 256])
    top = nodes // 4
    if kind == "serve":
        batch, hops = _log(rng, 8, 512), rng.choice(["15-10", "25-15", "100", "20-10-5"])
    elif dtype == "f32":         # fp32 is for small models and for checks
        batch, hops = _log(rng, 64, 2048), rng.choice(["10-5", "15-10", "25-15", "100"])
    else:
        batch, hops = _log(rng, 128, 8192), rng.choice(["15-10", "25-15", "100", "20-10-5"])
    batch = min(batch, top)
    if kind == "lightgcn":
        return _pick(g, kind, dtype, dim, dim, hops, batch, weighted=rng.random() < 0.5)
    if kind == "joint":
        h1 = rng.choice([256, 512])
        return _pick(g, kind, dtype, dim, hidden, "15-10" if hops == "20-10-5" else hops, max(64, min(batch, 4096, top // 2)), dense=rng.choice([32, 64]),
                     h1=h1, h2=h1 // 2, gate=rng.random() < 0.5)
    return _pick(g, kind, dtype, dim, hidden, hops, batch, bias=rng.random() < 0.3)


def _pick(graph, kind, dtype, dim, hidden, fanouts, batch, **more):
    c = _sampled("", kind, graph, dtype, dim, hidden, fanouts, batch, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------- inputs

def _zipf(gen, size, n, alpha, q=0.0):
    """Ranks in [0, n) with P(rank r) ~ (r + 1 + q)^-alpha, by inversion of the continuous law."""
    u = torch.rand(size, dtype=torch.float64, device=DEV, generator=gen)
    e = 1.0 - alpha
    lo, hi = (1.0 + q) ** e, (n + 1.0 + q) ** e
    r = (lo + u.mul_(hi - lo)).pow_(1.0 / e).sub_(q)
    return r.floor_().to(torch.int64).sub_(1).clamp_(0, n - 1)


def _ids(gen, size, n, alpha, q=0.0):
    """`size` ids of [0, n), popular ones scattered over the range."""
    perm = torch.randperm(n, device=DEV, generator=gen).to(torch.int32)
    out = torch.empty(size, dtype=torch.int32, device=DEV)
    for s in range(0, size, 1 << 25):
        t = min(size, s + (1 << 25))
        out[s:t] = perm[_zipf(gen, t - s, n, alpha, q)]
    return out


def _interactions(c, gen):
    users = _ids(gen, c["interactions"], c["users"], c["alpha"], c["q"])
    items = _ids(gen, c["interactions"], c["items"], c["alpha"], c["q"]).add_(c["users"])
    return users, items


def _coo(users, items):
    return torch.cat([users, items]), torch.cat([items, users])


def _normal(gen, rows, cols, dtype):
    out = torch.empty(rows, cols, dtype=dtype, device=DEV)
    for s in range(0, rows, 1 << 21):
        t = min(rows, s + (1 << 21))
        out[s:t] = torch.randn(t - s, cols, device=DEV, generator=gen)
    return out


def _glorot(gen, rows, cols, dtype):
    lim = (6.0 / (rows + cols)) ** 0.5
    return torch.empty(rows, cols, device=DEV).uniform_(-lim, lim, generator=gen).to(dtype)


def _seed_batch(users, items, batch, n_nodes, gen, rng):
    """`batch` distinct nodes met as endpoints of uniformly drawn interactions, in the order in which they are met."""
    got = np.zeros(0, np.int32)
    for _ in range(8):
        idx = torch.randint(0, users.numel(), (4 * batch,), device=DEV, generator=gen)
        cand = np.concatenate([got, torch.stack([users[idx], items[idx]], 1).reshape(-1).cpu().numpy()])
        got = cand[np.sort(np.unique(cand, return_index=True)[1])][:batch]
        if got.size == batch:
            break
    else:                                                   # a few hubs hold nearly all interactions: fill up with others
        rest = np.setdiff1d(rng.permutation(n_nodes)[: 2 * batch].astype(np.int32), got)
        got = np.concatenate([got, rng.permutation(rest)])[:batch]
    return torch.from_numpy(np.ascontiguousarray(got)).to(DEV)


def _edge_weights(indptr, gen):
    """Integer sampling weights, round(2^16 omega / (largest omega of the row)) with log-normal omega, at least 1."""
    deg = indptr[1:] - indptr[:-1]
    n, m = deg.numel(), int(indptr[-1])
    omega = torch.randn(m, device=DEV, generator=gen).exp_()
    row = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    top = torch.zeros(n, device=DEV).scatter_reduce_(0, row, omega, "amax")
    return (omega / top[row] * 65536.0).round_().clamp_(1, 65536).to(torch.int32)


def _inv_sqrt(deg):
    return torch.where(deg > 0, deg.clamp(min=1).to(torch.float64).rsqrt(), 0.0).to(torch.float32)


def prepare(case, seed):
    c = dict(case)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    rng = np.random.Generator(np.random.Philox(int(seed)))
    s = {"kind": c["kind"], "seed": int(seed) * 2654435761 % (1 << 63), "step": int(seed) % 100_000}
    if c["kind"] == "whole_mean":
        n, m = c["nodes"], c["entries"]
        dst, src = _ids(gen, m, n, c["alpha"]), _ids(gen, m, n, c["alpha"])
        s["indptr"], s["indices"], _ = E.graph_from_coo(n, dst, src)
        del dst, src
        s["csc_ptr"], s["csc_row"] = E.csr_transpose(s["indptr"], s["indices"], n)[:2]
        deg = s["indptr"][1:] - s["indptr"][:-1]
        s["inv_deg"] = torch.where(deg > 0, 1.0 / deg.clamp(min=1).to(torch.float32), 0.0)
        s["X"], s["G"] = (_normal(gen, n, c["dim"], DTYPES[c["dtype"]]) for _ in range(2))
        s["out"], s["dX"] = torch.zeros_like(s["X"]), torch.zeros_like(s["X"])
        s["ws"] = E.aggregate_forward(s["indptr"], s["indices"], s["X"], out=s["out"])[1]
        s["ws_b"] = E.aggregate_backward(s["csc_ptr"], s["csc_row"], s["inv_deg"], s["G"], dX=s["dX"])[1]
        return s
    users, items = _interactions(c, gen)
    n = c["users"] + c["items"]
    if c["kind"] == "ingest":
        s["n"] = n
        s["row"], s["col"] = _coo(users, items)
        return s
    s["indptr"], s["indices"], _ = E.graph_from_coo(n, *_coo(users, items))
    dt, d = DTYPES[c["dtype"]], c["dim"]
    s["X"] = _normal(gen, n, d, dt)
    if c["kind"] == "whole_lightgcn":
        s["layers"] = c["layers"]
        s["csc_ptr"], s["csc_row"] = E.csr_transpose(s["indptr"], s["indices"], n)[:2]
        s["inv_sqrt"] = _inv_sqrt(s["indptr"][1:] - s["indptr"][:-1])
        s["dY"] = _normal(gen, n, d, dt)
        s["Y"], s["ws"] = E.lightgcn_forward(s["indptr"], s["indices"], s["inv_sqrt"], s["layers"], s["X"])
        s["dH"] = torch.zeros_like(s["Y"])
        return s
    fanouts = [int(f) for f in c["fanouts"].split("-")]
    L, batch, hidden = len(fanouts), c["batch"], c["hidden"]
    Ws = [_glorot(gen, hidden, 2 * (d if l == 0 else hidden), dt) for l in range(L)]
    if c["kind"] == "joint":
        P, zdim = batch, 2 * hidden + c["dense"]
        idx = torch.randint(0, users.numel(), (P,), device=DEV, generator=gen)
        s["user"], s["item"] = users[idx].contiguous(), items[idx].contiguous()
        s["dense"] = torch.randn(P, c["dense"], device=DEV, generator=gen)
        s["labels"] = (torch.rand(P, device=DEV, generator=gen) < 0.1).to(torch.float32)
        Wt = [_glorot(gen, a, b, dt) for a, b in ((c["h1"], zdim), (c["h2"], c["h1"]), (1, c["h2"]))]
        bt = [torch.zeros(W.shape[0], device=DEV) for W in Wt]
        gate = dict(W_gate=_glorot(gen, zdim, zdim, dt), b_gate=torch.zeros(zdim, device=DEV)) if c["gate"] else {}
        s["joint"] = E.JointStep(s["indptr"], s["indices"], s["X"], P, c["dense"], fanouts, Ws, Wt, bt, **gate)
        s["joint"].ws.zero_()                               # node ids beyond the step's own are then zeros in every run
        E.sampler_scratch_init(n, s["joint"].ws)
        return s
    s["seeds"] = _seed_batch(users, items, batch, n, gen, rng)
    s["blocks"] = b = E.Blocks(n, batch, fanouts, DEV)
    s["edge_cum"] = E.edge_cumulate(s["indptr"], _edge_weights(s["indptr"], gen)) if c.get("weighted") else None
    if c["kind"] == "lightgcn":
        s["inv_sqrt"] = _inv_sqrt(s["indptr"][1:] - s["indptr"][:-1])
        s["dY"] = _normal(gen, b.caps[0][0], d, dt)
        E.sample_khop(s["indptr"], s["indices"], s["seeds"], b, s["seed"], s["step"], edge_cum=s["edge_cum"])
        s["Y"], s["ctx"] = E.lightgcn_sampled_forward(b, s["X"], s["inv_sqrt"])
        s["dX"], s["scratch"] = E.lightgcn_sampled_backward(b, s["ctx"], s["dY"])
        return s
    s["Ws"] = Ws
    s["biases"] = [torch.randn(hidden, device=DEV, generator=gen) * 0.1 for _ in Ws] if c["bias"] else None
    s["ctx"] = torch.empty(E.binding.sage_forward_ctx_bytes(b, s["X"], Ws), dtype=torch.uint8, device=DEV)
    s["H"] = torch.zeros(batch, hidden, dtype=dt, device=DEV)
    if c["kind"] == "serve":
        return s
    f32 = dict(dtype=torch.float32, device=DEV)
    rhs = 2 if c["kind"] == "multitask" else 1
    s["dH"] = _normal(gen, batch, hidden, dt)
    s["dWs"] = [torch.zeros(W.shape, **f32) for W in Ws]
    s["dbs"] = [torch.zeros(hidden, **f32) for _ in Ws] if c["bias"] else None
    s["dX"] = [torch.zeros(b.caps[-1][1], d, dtype=dt, device=DEV) for _ in range(rhs)]
    if rhs == 1:
        s["scratch"] = torch.empty(E.binding.sage_backward_scratch_bytes(b, s["X"], Ws), dtype=torch.uint8, device=DEV)
    else:
        s["scratch"] = torch.empty(E.binding.sage_backward_multi_scratch_bytes(b, s["X"], Ws, 2), dtype=torch.uint8, device=DEV)
        s["dH_ssl"] = torch.zeros(batch, hidden, dtype=dt, device=DEV)
        s["w0"], s["w"], s["L"], s["g"] = torch.tensor([0.8, 1.2], **f32), torch.ones(2, **f32), torch.zeros(2, **f32), torch.zeros(2, **f32)
        s["L"][1] = 0.6                                     # the recommendation loss of the step, as the ranking model reports it
        s["L0"] = torch.tensor([4.0 * batch * hidden, 0.7], **f32)
    return s


# ------------------------------------------------------------------------------------------------- one pass

def run(state):
    s, kind = state, state["kind"]
    if kind == "whole_mean":
        E.aggregate_forward(s["indptr"], s["indices"], s["X"], out=s["out"], ws=s["ws"])
        E.aggregate_backward(s["csc_ptr"], s["csc_row"], s["inv_deg"], s["G"], dX=s["dX"], ws=s["ws_b"])
        return s["out"], s["dX"]
    if kind == "whole_lightgcn":
        E.lightgcn_forward(s["indptr"], s["indices"], s["inv_sqrt"], s["layers"], s["X"], Y=s["Y"], ws=s["ws"])
        E.lightgcn_backward(s["csc_ptr"], s["csc_row"], s["inv_sqrt"], s["layers"], s["dY"], dH0=s["dH"], ws=s["ws"])
        return s["Y"], s["dH"]
    if kind == "ingest":
        indptr, indices, bad = E.graph_from_coo(s["n"], s["row"], s["col"])
        return indptr, indices, bad, E.csr_transpose(indptr, indices, s["n"])
    if kind == "joint":
        j = s["joint"].run(s["user"], s["item"], s["dense"], s["labels"], s["seed"], s["step"])
        return j.loss, j.logits, j.dW_gnn, j.dW_tower, j.db_tower, j.dX_rows, j.dX_ids, j.n_rows
    b = s["blocks"]
    if kind == "serve":
        E.sample_khop(s["indptr"], s["indices"], s["seeds"], b, s["seed"], s["step"], transpose=False)
        return E.sage_forward(b, s["X"], s["Ws"], s["biases"], ctx=s["ctx"], H_out=s["H"])[0], b.counts
    E.sample_khop(s["indptr"], s["indices"], s["seeds"], b, s["seed"], s["step"], defer_transpose=True, edge_cum=s["edge_cum"])
    ids, counts = b.t[-1]["src_nodes"], b.counts            # the node of every gradient row, and how many there are
    if kind == "lightgcn":
        E.lightgcn_sampled_forward(b, s["X"], s["inv_sqrt"], ctx=s["ctx"], Y=s["Y"])
        E.lightgcn_sampled_backward(b, s["ctx"], s["dY"], dX_rows=s["dX"], scratch=s["scratch"])
        return s["Y"], s["dX"], ids, counts
    E.sage_forward(b, s["X"], s["Ws"], s["biases"], ctx=s["ctx"], H_out=s["H"])
    if kind == "step":
        E.sage_backward(b, s["X"], s["Ws"], s["ctx"], s["dH"], dWs=s["dWs"], dbs=s["dbs"], dX_rows=s["dX"][0], scratch=s["scratch"])
        return s["H"], s["dWs"], s["dbs"], s["dX"], ids, counts
    s["w"].copy_(s["w0"])                                   # the task weights as the step finds them
    E.ssl_loss(s["H"], s["X"], s["seeds"], None, s["w"][:1], loss=s["L"][:1], dH=s["dH_ssl"])
    E.sage_backward_multi(b, s["X"], s["Ws"], s["ctx"], [s["dH_ssl"], s["dH"]], dWs=s["dWs"], dbs=s["dbs"], dX_rows=s["dX"], scratch=s["scratch"])
    E.gradient_norms(s["dX"], counts[-1, 1:2], out=s["g"])
    E.gradnorm_update(s["w"], s["L"], s["L0"], s["g"], 1.0, 0.025)
    return s["H"], s["L"], s["dWs"], s["dbs"], s["dX"], s["g"], s["w"], ids, counts


# ------------------------------------------------------------------------------------------------- work and tolerance

def _hops(c):
    """Expected (destinations, sources, entries) of every hop.  Rows shorter than the fanout and nodes met twice make
    blocks smaller than their capacities; the shares are those seen on the listed graphs and batches."""
    n = c["users"] + c["items"]
    dst, out = float(c["batch"] * (0.7 if c["kind"] == "joint" else 1.0)), []
    for h, f in enumerate(int(f) for f in c["fanouts"].split("-")):
        entries = dst * f * (0.88 if f <= 25 else 0.67)
        src = min(float(n), dst + (0.2, 0.15, 0.2, 0.2)[h] * entries)
        out.append((dst, src, entries))
        dst = src
    return out


def work(case):
    c = case
    if c["kind"] == "ingest":
        n, m = c["users"] + c["items"], 2 * c["interactions"]
        return {"bytes": m * (8 + 4) + n * 8 + m * (4 + 4 + 8) + n * 16, "flops": 0}
    es = 2 if c["dtype"] == "bf16" else 4
    row = c["dim"] * es
    if c["kind"] == "whole_mean":                           # every feature and gradient row once in and once out
        return {"bytes": 4 * c["nodes"] * row + 2 * c["entries"] * 4 + c["nodes"] * 20, "flops": 2 * c["entries"] * c["dim"]}
    if c["kind"] == "whole_lightgcn":
        n, m = c["users"] + c["items"], 2 * c["interactions"]
        return {"bytes": 4 * n * row + 2 * m * 4 + n * 20, "flops": 2 * c["layers"] * m * c["dim"] * 2}
    hops = _hops(c)
    L, d, hid = len(hops), c["dim"], c["hidden"]
    outer_src = hops[-1][1]
    by = sum(e * 12 + s * 4 + t * 12 for t, s, e in hops) + outer_src * row
    fl = sum(e * d for _, _, e in hops)
    if c["kind"] == "lightgcn":
        return {"bytes": by + outer_src * row + 2 * c["batch"] * row, "flops": 2 * fl}
    for l in range(L):
        fl += 2.0 * hops[L - 1 - l][0] * 2 * (d if l == 0 else hid) * hid * (1 if c["kind"] == "serve" else 3)
    by += c["batch"] * hid * es
    if c["kind"] == "serve":
        return {"bytes": by, "flops": fl}
    rhs = 2 if c["kind"] == "multitask" else 1
    by += rhs * (outer_src * row + c["batch"] * hid * es)
    if c["kind"] == "joint":
        z = 2 * hid + c["dense"]
        fl += 6.0 * c["batch"] * (z * c["h1"] + c["h1"] * c["h2"] + (z * z if c["gate"] else 0))
        by += c["batch"] * (c["dense"] * 4 + 16)
    return {"bytes": by, "flops": fl}


def _cost(c):
    """Seconds that a pass takes at least, roughly: gathered rows, dense products, sorts."""
    if c["kind"] == "ingest":
        return 2 * c["interactions"] * 80 / 4e12
    row = c["dim"] * (2 if c["dtype"] == "bf16" else 4)
    if c["kind"] == "whole_mean":
        return 2 * c["entries"] * (row + 4) / 5e12
    if c["kind"] == "whole_lightgcn":
        return 4 * c["layers"] * c["interactions"] * (row + 4) / 5e12
    w, hops = work(c), _hops(c)
    passes = 1 if c["kind"] == "serve" else 3 if c["kind"] == "multitask" else 2
    on_tensor_cores = c["dtype"] == "bf16" and c["dim"] % 64 == 0
    return passes * sum(e * (row + 30) for _, _, e in hops) / 4e12 + w["flops"] / (4e14 if on_tensor_cores else 1e13)


def tolerance(case):
    # Whole numbers (graphs, blocks, node ids, counts) are fixed by the inputs.  Sums are formed in fp32 and stored in the
    # feature type: against the same path with float64 sums and the same storage points the fp32 step is off by 3e-7 and
    # the bf16 step by 7e-5 (single elements 8e-6 and 8e-3), more where a hub adds up a million rows.  In bf16 a mean that
    # rounds the other way can turn the sign of a ReLU input that is zero to within rounding; one such sign moves the
    # gradients of a small batch, with some ten thousand active elements, by 1e-2.
    if case["kind"] == "ingest":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1e-2, "max": 0.5}
