"""The workloads on which the speed of the library is followed.

Every case is what a user's program does through `binding.Context`: the whole method on device-resident
inputs (partition, induced subgraphs, local steps of all trainers, aggregation), one aggregation round on
subgraphs that the program keeps, the whole path from host buffers, link prediction, neighbour sampling, and
the averaging of large models.  Shapes are those of the named workloads in `inputs.py` (at full size or
scaled), of the tests and of `bench.py`, plus ragged ones; the graphs are drawn on the GPU with torch from the same
families (uniform, Chung-Lu power law, planted communities).
"""
import math

import torch

from paper_2305_09887_b200 import binding

LR = 0.01


def _training(name, kind, graph, n, degree, F, hidden, layers, classes, M, K, **options):
    """A case that trains.  graph: 'uniform', 'powerlaw' (exponent `gamma`) or 'communities' (super-nodes of 100
    nodes, `degree` inside and half of it between them)."""
    case = dict(name=name, kind=kind, graph=graph, n=n, degree=degree, gamma=2.1, F=F, hidden=hidden, layers=layers,
                classes=classes, M=M, K=K, super_nodes=False, bf16=False, gcn=False, prelu=False, layernorm=False,
                streams=False, stragglers=False, pairs=0)
    case.update(options)
    return case


def listed():
    return [
        # the smallest use: the Tiny workload start to end, where launches and host work are all there is
        _training("tiny_method", "method", "uniform", 2_000, 10, 64, 64, 2, 8, M=4, K=5),
        # nothing is a multiple of anything: a small social graph with odd widths and three trainers
        _training("ragged_method", "method", "powerlaw", 30_011, 17, 71, 90, 3, 13, M=3, K=7),
        # one aggregation round of the Medium workload on subgraphs that are kept between rounds
        _training("medium_round", "round", "powerlaw", 200_000, 25, 128, 256, 3, 47, M=8, K=20),
        # time-based aggregation (trainers that finish different numbers of steps, one that failed), every trainer
        # on a stream of its own, on a tenth of the SuperTMA graph
        _training("stragglers_round", "round", "communities", 200_000, 20, 100, 256, 3, 47, M=5, K=10, super_nodes=True,
                  streams=True, stragglers=True),
        # the SuperTMA workload at full size: grouped partition, subgraphs, one round
        _training("supertma_method", "method", "communities", 2_000_000, 20, 100, 256, 3, 47, M=16, K=10, super_nodes=True),
        # the Large workload at a fifth of its nodes (2 classes, 64-bit row offsets), start to end
        _training("large_method", "method", "powerlaw", 5_000_000, 52, 128, 256, 2, 2, M=32, K=5, gamma=2.0),
        # the trainer-count and width sweep: width 512, bf16 operands, nodes assigned one by one
        _training("sweep_bf16", "round", "communities", 500_000, 20, 512, 512, 3, 47, M=8, K=5, bf16=True),
        # the paper's encoder with Layer Normalization and PReLU, GCN layers
        _training("gcn_layernorm", "round", "powerlaw", 200_000, 25, 128, 256, 3, 47, M=8, K=10, gcn=True, prelu=True, layernorm=True),
        # the paper's task: link prediction on each part's edges and as many random-tail negatives
        _training("link_round", "link", "powerlaw", 200_000, 25, 128, 256, 3, 256, M=8, K=5, prelu=True, layernorm=True, pairs=65_536),
        # three hops of the neighbour sampler from a mini-batch of training edges' end points
        dict(name="sample_hops", kind="sample", n=800_000, degree=30, gamma=2.1, batch=8_192, fanouts="15,10,5"),
        # the averaging of large replicas, with the last SGD step folded in
        dict(name="average_large", kind="average", M=64, P=4_194_304, sgd=True),
        # host buffers in, parameters out: a quarter of the Medium workload from pinned memory
        _training("host_method", "host", "powerlaw", 50_000, 25, 128, 256, 3, 47, M=8, K=10),
    ]


def _log(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _estimate(case):
    """Seconds a case takes on the GPU, roughly; only to keep drawn cases no costlier than the largest listed one."""
    if case["kind"] in ("sample", "average"):
        return work(case)["bytes"] / 1e12
    w = work(case)
    n, K, dims = case["n"], case["K"], _dims(case)
    gathered = _kept(case) * K * 4.0 * (2 * sum(dims[1:-1]) + 2 * dims[-1])
    rows = n * K * 4.0 * (10 * sum(dims[1:-1]) + 2 * dims[0])
    return w["bytes"] / 1e12 + w["flops"] / 150e12 + gathered / 3e12 + rows / 3e12


def draw(rng):
    limit = _estimate(next(c for c in listed() if c["name"] == "supertma_method"))
    while True:
        kind = rng.choice(("method", "method", "round", "round", "round", "host", "link", "sample", "average"))
        if kind == "sample":
            fanouts = [rng.choice((5, 10, 15, 25)) for _ in range(rng.choice((2, 3)))]
            case = dict(kind=kind, n=_log(rng, 2_000, 2_000_000), degree=rng.randint(8, 50), gamma=rng.choice((2.0, 2.1, 2.5)),
                        batch=_log(rng, 64, 16_384), fanouts=",".join(str(f) for f in fanouts))
            if case["batch"] * 4 > case["n"]:
                continue
        elif kind == "average":
            case = dict(kind=kind, M=rng.choice((2, 3, 4, 8, 16, 23, 32, 64)), P=_log(rng, 9_000, 8_000_000), sgd=rng.random() < 0.5)
        else:
            graph = rng.choice(("uniform", "powerlaw", "powerlaw", "communities", "communities"))
            n = _log(rng, 2_000, 2_000_000 if kind in ("method", "round") else 200_000)
            if graph == "communities":
                n = max(2_000, n // 100 * 100)
            layers = rng.choice((2, 2, 3, 3))
            variant = rng.random()
            hidden = rng.choice((64, 90, 128, 200, 256, 256, 384, 512))
            case = _training(
                "", kind, graph, n, rng.randint(8, 52), rng.choice((33, 64, 71, 100, 128, 128, 256, 512)), hidden,
                layers, hidden if kind == "link" else rng.choice((2, 2, 7, 13, 40, 47, 47)),
                M=rng.choice((2, 3, 4, 5, 8, 8, 16, 23, 32)), K=rng.choice((3, 5, 7, 10, 20)), gamma=rng.choice((2.0, 2.1, 2.5)),
                super_nodes=graph == "communities" and rng.random() < 0.7, bf16=rng.random() < 0.2,
                gcn=0.7 < variant < 0.9, prelu=variant > 0.8, layernorm=variant > 0.8,
                pairs=_log(rng, 500, 65_536) if kind == "link" else 0)
            del case["name"]
            if kind == "round" and rng.random() < 0.3:
                case["streams"] = case["M"] <= 8
                case["stragglers"] = True
        if _estimate(case) <= 0.8 * limit:
            return case


# ---- shapes ---------------------------------------------------------------------------------------------

def _dims(case):
    return (case["F"],) + (case["hidden"],) * (case["layers"] - 1) + (case["classes"],)


def _variant(case):
    return (int(case["gcn"]), int(case["prelu"]), int(case["layernorm"]))


def _decoder(case):
    return (case["classes"], case["hidden"], 1)


def _entries(case):
    return case["n"] * case["degree"] * (1.5 if case.get("graph") == "communities" else 1.0)


def _kept(case):
    """Expected entries inside the parts: 1/M of those between super-nodes (or of all), and all inside them."""
    e = _entries(case)
    if case["super_nodes"]:
        inside = case["n"] * case["degree"]
        return inside + (e - inside) / case["M"]
    return e / case["M"]


def work(case):
    if case["kind"] == "average":
        M, P = case["M"], case["P"]
        return {"bytes": 4.0 * P * M * (3 if case["sgd"] else 2), "flops": P * M * (3.0 if case["sgd"] else 1.0)}
    if case["kind"] == "sample":
        size, touched = float(case["batch"]), 0.0
        for f in (int(v) for v in case["fanouts"].split(",")):
            drawn = size * min(f, case["degree"])
            touched += size * (4.0 + 16.0 + 4.0 * case["degree"]) + 8.0 * size + 4.0 * drawn
            size = min(float(case["n"]), size + drawn)
            touched += 4.0 * size
        return {"bytes": touched, "flops": 0.0}
    n, M, K, dims = float(case["n"]), case["M"], case["K"], _dims(case)
    e, kept = _entries(case), _kept(case)
    nsrc = 1 if case["gcn"] else 2
    layers = list(zip(dims[:-1], dims[1:]))
    P = sum((nsrc * a + 1) * b for a, b in layers)
    moved = 4.0 * n * dims[0] + 4.0 * n + 8.0 * M * P                       # features, labels, parameters in and out
    if case["kind"] in ("method", "host"):
        moved += 4.0 * e + 8.0 * n + 12.0 * n + (4.0 * n if case["super_nodes"] else 0.0) + 8.0 * n + 4.0 * kept
    else:
        moved += 8.0 * n + 4.0 * kept
    dense = sum(2.0 * n * nsrc * a * b for a, b in layers)
    flops = 2 * dense + sum(2.0 * n * nsrc * a * b for a, b in layers[1:])      # forward, weights, inputs of layers 1..
    flops += 2.0 * kept * (sum(min(a, b) for a, b in layers[1:]) + sum(b for _, b in layers[1:]))
    flops *= K
    flops += 2.0 * kept * dims[0]
    if case["kind"] == "link":
        pairs, dd = 2.0 * M * case["pairs"], _decoder(case)
        flops += K * pairs * sum(6.0 * a * b for a, b in zip(dd[:-1], dd[1:]))
        moved += 12.0 * pairs
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # Trained parameters and losses after the case's steps; partitions, subgraphs and samples are whole numbers and
    # have to be the same.  Measured against the same steps in 64 bits on 40 cases of these ranges, then about four
    # times the worst.  fp32-accurate products: 3e-6 of a tensor (2e-6 where a ReLU branch at zero flips), 4e-5 at a single
    # value.  Operands rounded to bf16 (2^-9 each): 3e-5 of the parameters, 2e-4 to 9e-4 of the losses, 2e-3 at a single value.
    # Averaging: 1.5e-7 and 1.1e-6.
    if case["kind"] == "sample":
        return "exact"
    if case["kind"] == "average":
        return {"rel": 6e-7, "max": 5e-6}
    return {"rel": 1e-3, "max": 1e-2} if case["bf16"] else {"rel": 1e-5, "max": 2e-4}


# ---- inputs, drawn on the GPU ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _csr(n, u, v, wide):
    """Both directions of every pair, no loops, no duplicates, columns sorted."""
    keep = u != v
    u, v = u[keep], v[keep]
    keys = torch.cat([u * n + v, v * n + u])
    del u, v, keep
    keys = torch.unique(keys)
    bounds = torch.arange(n + 1, device="cuda", dtype=torch.int64) * n
    rowptr = torch.searchsorted(keys, bounds)
    col = (keys % n).to(torch.int32)
    return rowptr if wide else rowptr.to(torch.int32), col


def _power_law_pairs(n, pairs, gamma, g):
    """Chung-Lu by endpoint sampling: both ends from w(x) ~ (x + i0)^(-1/(gamma-1)), the top expected degree capped
    at the square root of the entries; ids are a random permutation of the ranks."""
    expo = -1.0 / (gamma - 1.0)
    e1 = expo + 1.0

    def integral(b, i0):
        if abs(e1) < 1e-12:
            return math.log((b + i0) / i0)
        return ((b + i0) ** e1 - i0 ** e1) / e1

    cap, lo, hi = math.sqrt(2.0 * pairs), 1e-3, float(n)
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        if 2.0 * pairs * integral(1.0, mid) / integral(float(n), mid) > cap:
            lo = mid
        else:
            hi = mid
    i0 = hi
    ids = torch.randperm(n, device="cuda", generator=g)

    def ends():
        u = torch.rand(pairs, device="cuda", generator=g, dtype=torch.float64)
        if abs(e1) < 1e-12:
            x = i0 * torch.exp(u * math.log((n + i0) / i0)) - i0
        else:
            a, b = i0 ** e1, (n + i0) ** e1
            x = (a + u * (b - a)).pow(1.0 / e1) - i0
        return ids[x.to(torch.int64).clamp_(0, n - 1)]

    return ends(), ends()


def _graph(case, g):
    """(rowptr, col, group_id or None) on the GPU."""
    n, degree = case["n"], case["degree"]
    if case.get("graph", "powerlaw") == "powerlaw":
        return (*_csr(n, *_power_law_pairs(n, n * degree // 2, case["gamma"], g), wide=case["gamma"] == 2.0), None)
    if case["graph"] == "uniform":
        u = torch.randint(n, (n * degree // 2,), device="cuda", generator=g)
        v = torch.randint(n, (n * degree // 2,), device="cuda", generator=g)
        return (*_csr(n, u, v, wide=False), None)
    size = 100
    clusters = n // size
    at = torch.randperm(n, device="cuda", generator=g)              # members of a cluster are scattered over the ids
    group_id = torch.empty(n, dtype=torch.int32, device="cuda")
    group_id[at] = (torch.arange(n, device="cuda") // size).to(torch.int32)
    inside = torch.triu_indices(size, size, 1, device="cuda")
    us, vs = [], []
    for c0 in range(0, clusters, 4_000):
        c1 = min(clusters, c0 + 4_000)
        hit = torch.rand((c1 - c0) * inside.shape[1], device="cuda", generator=g) < degree / (size - 1)
        hit = torch.nonzero(hit).squeeze(1)
        first = (hit // inside.shape[1] + c0) * size
        k = hit % inside.shape[1]
        us.append(at[first + inside[0][k]])
        vs.append(at[first + inside[1][k]])
    a, b = _power_law_pairs(n, n * degree // 4, case["gamma"], g)
    differ = group_id[a] != group_id[b]
    us.append(a[differ])
    vs.append(b[differ])
    return (*_csr(n, torch.cat(us), torch.cat(vs), wide=False), group_id)


def _weights(dims, variant, g, decoder=None):
    """Initial parameters in the library's order: per layer the Xavier-uniform weight matrices and zero biases, then
    (hidden layers) scale 1 and shift 0 of the normalisation and the PReLU slope 0.25; the decoder's after them."""
    gcn, prelu, layernorm = variant
    out = []

    def uniform(a, b, count):
        r = math.sqrt(6.0 / (a + b))
        out.append((torch.rand(count * a * b, device="cuda", generator=g) * 2 - 1) * r)

    for l, (a, b) in enumerate(zip(dims[:-1], dims[1:])):
        uniform(a, b, 1 if gcn else 2)
        out.append(torch.zeros(b, device="cuda"))
        if l < len(dims) - 2:
            if layernorm:
                out.append(torch.ones(b, device="cuda"))
                out.append(torch.zeros(b, device="cuda"))
            if prelu:
                out.append(torch.full((1,), 0.25, device="cuda"))
    for k, (a, b) in enumerate(zip((decoder or ())[:-1], (decoder or ())[1:])):
        uniform(a, b, 1)
        if k < len(decoder) - 2:
            out.append(torch.full((1,), 0.25, device="cuda"))
    return torch.cat(out)


_contexts = []


def _context():
    """One context per program, as a user's program keeps it."""
    if not _contexts:
        _contexts.append(binding.Context(0))
    return _contexts[0]


def _subgraphs(case, s):
    """Partition and induced subgraphs: what the method starts with, or what a program keeps between rounds."""
    ctx, M = s["ctx"], case["M"]
    part_id, part_offsets, perm, local_id = ctx.partition(case["n"], s["group_id"], s["seed"], M, grouped=s["group_id"] is not None)
    rowptr_out, col_out, edge_offsets, kept_cut, edge_host = ctx.build_induced_csr(
        s["rowptr"], s["col"], M, part_id, part_offsets, perm, local_id)
    return dict(part_id=part_id, part_offsets=part_offsets, perm=perm, local_id=local_id, rowptr_out=rowptr_out, col_out=col_out,
                edge_offsets=edge_offsets, kept_cut=kept_cut, part_host=part_offsets.cpu().tolist(), edge_host=edge_host)


def _link_pairs(case, s, g):
    """Per part up to `pairs` of its undirected edges as positives and one random-tail negative for each."""
    us, vs, labels, offsets = [], [], [], [0]
    for p in range(case["M"]):
        lo, hi = s["part_host"][p], s["part_host"][p + 1]
        rp = s["rowptr_out"][lo + p: hi + p + 1]
        cols = s["col_out"][s["edge_host"][p]: s["edge_host"][p + 1]]
        rows = torch.repeat_interleave(torch.arange(hi - lo, device="cuda", dtype=torch.int32), rp[1:] - rp[:-1])
        up = torch.nonzero(rows < cols).squeeze(1)
        up = up[torch.randperm(up.numel(), device="cuda", generator=g)[:case["pairs"]]]
        tails = torch.randint(max(hi - lo, 1), (up.numel(),), device="cuda", generator=g, dtype=torch.int32)
        us += [rows[up], rows[up]]
        vs += [cols[up], tails]
        labels += [torch.ones_like(tails), torch.zeros_like(tails)]
        offsets.append(offsets[-1] + 2 * up.numel())
    return torch.cat(us).contiguous(), torch.cat(vs).contiguous(), torch.cat(labels), offsets


def prepare(case, seed):
    g = _generator(seed)
    s = dict(case=case, ctx=_context(), seed=seed & 0x7FFFFFFF)
    if case["kind"] == "average":
        s["params"] = torch.randn(case["M"], case["P"], device="cuda", generator=g) * 0.05
        s["grads"] = torch.randn(case["M"], case["P"], device="cuda", generator=g) * 1e-3 if case["sgd"] else None
        return s
    if case["kind"] == "sample":
        rowptr, s["col"], _ = _graph(case, g)
        s["rowptr"] = rowptr.to(torch.int64)
        s["frontier"] = torch.sort(torch.randperm(case["n"], device="cuda", generator=g)[:case["batch"]])[0].to(torch.int32)
        size, s["blocks"] = case["batch"], []                               # the program's own buffers for the blocks of a mini-batch
        for f in (int(v) for v in case["fanouts"].split(",")):
            drawn, size_next = size * f, min(case["n"], size * (f + 1))
            s["blocks"].append((torch.zeros(size + 1, dtype=torch.int64, device="cuda"), torch.zeros(drawn, dtype=torch.int32, device="cuda"),
                                torch.zeros(size_next, dtype=torch.int32, device="cuda")))
            size = size_next
        return s
    n, M, dims, variant = case["n"], case["M"], _dims(case), _variant(case)
    s["rowptr"], s["col"], group_id = _graph(case, g)
    s["group_id"] = group_id if case["super_nodes"] else None
    C = case["classes"]
    if C == 2:                                                              # rare positives
        y = (torch.rand(n, device="cuda", generator=g) < 0.01).to(torch.int64)
    elif group_id is not None:                                              # constant inside a community
        y = torch.randint(C, (n // 100,), device="cuda", generator=g)[group_id.to(torch.int64)]
    else:
        y = torch.randint(C, (n,), device="cuda", generator=g)
    X = torch.randn(n, case["F"], device="cuda", generator=g)
    X += 0.5 * torch.randn(C, case["F"], device="cuda", generator=g)[y]
    y = y.to(torch.int32)
    decoder = _decoder(case) if case["kind"] == "link" else None
    params0 = _weights(dims, variant, g, decoder)
    if case["kind"] == "host":
        pinned = lambda t: None if t is None else t.cpu().pin_memory().numpy()  # noqa: E731
        return dict(case=case, ctx=s["ctx"], seed=s["seed"], rowptr=pinned(s["rowptr"]), col=pinned(s["col"]), X=pinned(X), y=pinned(y),
                    group_id=pinned(s["group_id"]), params0=pinned(params0))
    s.update(X=X, y=y, params0=params0, loss=torch.zeros(M, case["K"], device="cuda"))
    if case["kind"] == "method":                                            # the program's own buffer for the subgraphs' columns
        most = min(1.1 * _entries(case), 1.3 * _kept(case)) + n
        s["columns"] = torch.zeros(int(most), dtype=torch.int32, device="cuda")
    if case["kind"] in ("round", "link"):
        s.update(_subgraphs(case, s))
        s["Xp"], s["yp"] = s["ctx"].gather_rows(X, s["perm"]), s["ctx"].gather_rows(y, s["perm"])
        for k in ("X", "y", "rowptr", "col", "part_id", "part_offsets", "perm", "local_id"):
            del s[k]
    if case["kind"] == "link":
        s["pair_u"], s["pair_v"], s["pair_label"], s["pair_offsets"] = _link_pairs(case, s, g)
    if case["stragglers"]:                                                  # the slowest third as fast, the last one failed
        s["steps"] = [max(1, case["K"] * (3 * M - 2 * p) // (3 * M)) for p in range(M)]
        s["steps"][-1] = 0
    if case["streams"]:
        s["streams"] = [torch.cuda.Stream() for _ in range(M)]
    return s


# ---- one pass -------------------------------------------------------------------------------------------

def _run_sample(case, s):
    frontier, out = s["frontier"], []
    for hop, fanout in enumerate(int(v) for v in case["fanouts"].split(",")):
        block = s["ctx"].sample_hop(s["rowptr"], s["col"], frontier, fanout, s["seed"], hop)
        for kept, new in zip(s["blocks"][hop], block):
            kept[:new.numel()].copy_(new)
        frontier = block[2]
        out.append(frontier.numel())
    return s["blocks"], out


def _run_average(case, s):
    if case["sgd"]:
        s["ctx"].sgd_aggregate(s["params"], s["grads"], LR)
    else:
        s["ctx"].aggregate(s["params"])
    return s["params"]


def _run_host(case, s):
    params, losses, kept, cut = s["ctx"].train_host(
        s["rowptr"], s["col"], s["X"], s["y"], _dims(case), case["M"], case["K"], 1, LR, s["seed"], s["params0"],
        group_id=s["group_id"], gemm_dtype=int(case["bf16"]), variant=_variant(case))
    return params, losses, kept, cut


def _run_method(case, s):
    ctx, M = s["ctx"], case["M"]
    sub = _subgraphs(case, s)
    yp = ctx.gather_rows(s["y"], sub["perm"])
    params = s["params0"].expand(M, -1).contiguous()
    ctx.local_steps(_dims(case), LR, M, sub["part_host"], sub["edge_host"], sub["rowptr_out"], sub["col_out"], s["X"], yp, params, case["K"],
                    loss_out=s["loss"], gemm_dtype=int(case["bf16"]), variant=_variant(case), perm=sub["perm"])
    ctx.aggregate(params)
    s["columns"][:sub["col_out"].numel()].copy_(sub["col_out"])
    out = {k: sub[k] for k in ("part_id", "part_offsets", "perm", "local_id", "rowptr_out", "edge_offsets", "kept_cut")}
    return dict(out, columns=s["columns"], params=params, loss=s["loss"])


def _run_round(case, s):
    ctx, M = s["ctx"], case["M"]
    params = s["params0"].expand(M, -1).contiguous()
    streams = s.get("streams")
    if streams:
        for stream in streams:
            stream.wait_stream(torch.cuda.current_stream())
    if case["kind"] == "link":
        ctx.link_steps(_dims(case), _decoder(case), LR, M, s["part_host"], s["edge_host"], s["rowptr_out"], s["col_out"], s["Xp"],
                       s["pair_offsets"], s["pair_u"], s["pair_v"], s["pair_label"], params, case["K"], loss_out=s["loss"],
                       gemm_dtype=int(case["bf16"]), variant=_variant(case))
    else:
        ctx.local_steps(_dims(case), LR, M, s["part_host"], s["edge_host"], s["rowptr_out"], s["col_out"], s["Xp"], s["yp"], params,
                        s.get("steps", case["K"]), loss_out=s["loss"], streams=streams, gemm_dtype=int(case["bf16"]), variant=_variant(case))
    if streams:
        for stream in streams:
            torch.cuda.current_stream().wait_stream(stream)
    if case["stragglers"]:
        ctx.aggregate_masked(params, [k > 0 for k in s["steps"]])
    else:
        ctx.aggregate(params)
    return params, s["loss"]


_RUN = dict(sample=_run_sample, average=_run_average, host=_run_host, method=_run_method, round=_run_round, link=_run_round)


def run(state):
    return _RUN[state["case"]["kind"]](state["case"], state)
