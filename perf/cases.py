"""What a user of the library has it do, as measurable cases.

Every case but the static builds is one step of a sliding-window stream on a
resident graph: newly arrived edges are inserted, the oldest ones expire and
some weights change; then the caller reads which vertices changed community
and updates its own copy of the labels.  The window slides round a ring of
edge chunks, so a state can take any number of steps and each one is a valid
batch of the same size.  A static-build case takes a CSR snapshot to labels.

    form    apply    one graph, one batch per step (LDL.apply)
            batched  many graphs, one batch each per step (apply_batches)
            served   many graphs, one request each per step (Server)
            create   CSR snapshot -> hierarchy and labels (LDL.from arrays)
    graph   planted  equal blocks, 5 of 6 partners inside the block (the
                     SBM-style streams), blocks of 100 vertices
            rmat     R-MAT (0.57, 0.19, 0.19, 0.05): skewed social streams
            power    power-law degrees (exponent 2.5) and community sizes,
                     a fifth of the edges leaving the community; updates
                     fall into one region of the graph
    n, deg  vertices (per graph) and mean neighbours per vertex
    batch   updates per step (per graph)
"""
import math

import numpy as np
import torch

from paper_2502_18497_gb300 import DELETE, INSERT, LDL, REWEIGHT, Server, apply_batches

K = 6       # chunks of the ring
WINDOW = 3  # chunks present at any time
BLOCK = 100  # vertices per planted block


def _case(name, form, graph, n, deg, batch, directed=False, wmax=1, **more):
    c = dict(form=form, graph=graph, n=n, deg=deg, batch=batch, directed=directed, wmax=wmax, gamma_num=1,
             gamma_den=1, atomic=True, on_device=False, graphs=1)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # an interactive service: one edge arrives and one expires, the answer is awaited
        _case("one_edge_planted_10k", "apply", "planted", 10_000, 12, 2, wmax=4),
        # the test-suite's C1 stream: small batches on a small community graph
        _case("batch100_planted_10k", "apply", "planted", 10_000, 12, 100, wmax=4),
        # the SBM-style rewiring sequences: 500-edge batches, unit weights
        _case("batch500_planted_131k", "apply", "planted", 131_000, 16, 500),
        # a tenant of the served form: directed stream of middling size
        _case("batch1k_rmat_131k", "apply", "rmat", 1 << 17, 16, 1_000, directed=True, wmax=16),
        # the benchmark's stream: directed R-MAT, 2^20 vertices, 16M arcs, batches of 10^4
        _case("batch10k_rmat_1m", "apply", "rmat", 1 << 20, 16, 10_000, directed=True, wmax=16),
        # a small batch on a large graph: what locality is for
        _case("batch100_power_2m", "apply", "power", 2_000_003, 32, 100),
        # bulk ingest: 10^5 updates at once on the same graph
        _case("batch100k_power_2m", "apply", "power", 2_000_003, 32, 100_000),
        # an undirected skewed graph of odd size, batches handed over on the device
        _case("batch30k_rmat_836k_dev", "apply", "rmat", 835_937, 24, 30_000, wmax=4, on_device=True),
        # weights so large that gains need 128 bits, rational resolution, no undo log
        _case("batch777_rmat_60k_wide", "apply", "rmat", 60_001, 12, 777, directed=True, wmax=1 << 28,
              gamma_num=3, gamma_den=2, atomic=False),
        # many small graphs updated together, 0.1% of each one's edges
        _case("batched_32_graphs", "batched", "planted", 12_000, 12, 72, wmax=8, graphs=32),
        # tenants of a request server, one request each in flight
        _case("served_6_tenants", "served", "rmat", 30_000, 16, 400, directed=True, wmax=16, graphs=6),
        # loading a graph: the static hierarchy from a CSR snapshot
        _case("create_rmat_1m", "create", "rmat", 1 << 20, 16, 0, directed=True, wmax=16),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    form = rng.choice(["apply"] * 7 + ["batched", "served", "create"])
    graph = rng.choice(["planted", "rmat", "power"])
    directed = graph == "rmat" and rng.random() < 0.6
    wmax = 1 if graph == "power" else rng.choice([1, 4, 16, 1000])
    deg = rng.choice([6, 8, 12, 16, 24, 32])
    if form in ("batched", "served"):
        n = log(1_500, 40_000)
        graphs = rng.randint(2, 24 if form == "batched" else 8)
        return _case("", form, graph, n, deg, max(2, log(0.0002 * n * deg, 0.005 * n * deg)), directed, wmax,
                     graphs=graphs)
    n = log(3_000, 16_000_000 // max(16, deg))
    if form == "create":
        return _case("", form, graph, n, deg, 0, directed, wmax)
    batch = log(2, max(3, min(30_000, n * deg // 100)))
    gn, gd = rng.choice([(1, 1), (1, 1), (1, 1), (3, 2), (1, 2)])
    return _case("", form, graph, n, deg, batch, directed, wmax, gamma_num=gn, gamma_den=gd,
                 atomic=rng.random() < 0.8, on_device=rng.random() < 0.3)


# ---------------------------------------------------------------- inputs (drawn on the GPU)
def _rand(g, n):
    return torch.rand(n, generator=g, device="cuda")


def _randint(g, lo, hi, n):
    return torch.randint(lo, hi, (n,), generator=g, device="cuda")


def _rmat_keys(g, n, edges, directed):
    scale = max(1, (n - 1).bit_length())
    over = (1 << scale) / n
    draws = int(edges * 1.25 * over * over) + 64
    src = torch.zeros(draws, dtype=torch.int64, device="cuda")
    dst = torch.zeros_like(src)
    for _ in range(scale):
        u = _rand(g, draws)
        src = 2 * src + (u >= 0.76).long()
        dst = 2 * dst + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95)).long()
    ok = (src < n) & (dst < n) & (src != dst)
    src, dst = src[ok], dst[ok]
    if not directed:
        src, dst = torch.minimum(src, dst), torch.maximum(src, dst)
    return src * n + dst


def _planted_keys(g, n, edges):
    v = _randint(g, 0, n, edges)
    b0 = v // BLOCK * BLOCK
    size = torch.clamp(n - b0, max=BLOCK)
    inner = b0 + (_rand(g, edges) * size).long()
    other = torch.where(_rand(g, edges) < 5 / 6, inner, _randint(g, 0, n, edges))
    ok = other != v
    v, other = v[ok], other[ok]
    return torch.minimum(v, other) * n + torch.maximum(v, other)


def _power_keys(g, n, deg):
    d = torch.clamp(deg / 3 * (1 - _rand(g, n)).pow(-2 / 3), 1, min(20_000, n // 4)).long()
    sizes = (50 ** -0.5 + _rand(g, n // 50 + 1) * (min(50_000, n // 2) ** -0.5 - 50 ** -0.5)).pow(-2).long()
    comm = torch.searchsorted(torch.cumsum(sizes, 0), torch.arange(n, device="cuda"), right=True)
    stub = torch.repeat_interleave(torch.arange(n, device="cuda"), d)
    out = _rand(g, stub.numel()) < 0.2
    pairs = []
    for part, order in ((stub[~out], None), (stub[out], 0)):
        at = _rand(g, part.numel()).double()
        part = part[torch.argsort(at + comm[part] if order is None else at)]
        part = part[: part.numel() // 2 * 2].view(-1, 2)
        pairs.append(part)
    e = torch.cat(pairs)
    e = e[e[:, 0] != e[:, 1]]
    return torch.minimum(e[:, 0], e[:, 1]) * n + torch.maximum(e[:, 0], e[:, 1])


def _csr(n, keys, w, directed):
    """Host CSR arrays of the arcs (keys sorted, or both directions of edges)."""
    if not directed:
        keys = torch.cat([keys, keys % n * n + keys // n])
        w = torch.cat([w, w])
        keys, order = torch.sort(keys)
        w = w[order]
    src = keys // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rp.cpu().numpy(), (keys % n).int().cpu().numpy(), w.int().cpu().numpy()


def _stream(case, seed):
    """(CSR arrays of the first window, batches of the ring) of one graph."""
    n, deg, directed, batch = case["n"], case["deg"], case["directed"], case["batch"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    edges = n * deg if directed else n * deg // 2
    if case["graph"] == "rmat":
        keys = _rmat_keys(g, n, edges, directed)
    elif case["graph"] == "planted":
        keys = _planted_keys(g, n, edges)
    else:
        keys = _power_keys(g, n, deg)
    keys = torch.unique(keys)
    w = _randint(g, 1, case["wmax"] + 1, keys.numel())
    if not batch:
        return _csr(n, keys, w, directed), []
    # a batch: `move` arrivals, as many expiries, the rest weight changes
    move = max(1, batch * 9 // 20)
    rew = max(0, batch - 2 * move)
    want = K * (move + rew)
    if case["graph"] == "power":  # edges of one region: consecutive ids share communities
        v0 = int(_randint(g, 0, n, 1))
        pool = torch.argsort((keys // n - v0).abs())[: min(keys.numel(), 4 * want + 64)]
    else:
        pool = torch.arange(keys.numel(), device="cuda")
    pick = pool[torch.randperm(pool.numel(), generator=g, device="cuda")[:want]]
    move = min(move, pick.numel() // K)
    ring, spare = pick[: K * move].view(K, move), pick[K * move :]
    rew = min(rew, spare.numel() // K)
    present = torch.ones(keys.numel(), dtype=torch.bool, device="cuda")
    present[ring[WINDOW:].reshape(-1)] = False
    csr = _csr(n, keys[present], w[present], directed)
    batches = []
    for lap in range(2):
        for p in range(K):
            parts = [(ring[(p + WINDOW) % K], INSERT), (ring[p], DELETE), (spare[p * rew : (p + 1) * rew], REWEIGHT)]
            rows = []
            for at, op in parts:
                k = keys[at]
                wt = torch.zeros_like(k) if op == DELETE else _randint(g, 1, case["wmax"] + 1 + lap, k.numel())
                rows.append(torch.stack([k // n, k % n, torch.full_like(k, op), wt], 1))
            b = torch.cat(rows)
            b = b[torch.randperm(b.shape[0], generator=g, device="cuda")].int().contiguous()
            batches.append(b if case["on_device"] else b.cpu().numpy())
    return csr, batches


def prepare(case, seed):
    graphs = case["graphs"]
    args = dict(directed=case["directed"], gamma_num=case["gamma_num"], gamma_den=case["gamma_den"],
                no_rollback=0 if case["atomic"] else 1)
    made = []
    for i in range(graphs):
        one = dict(case)
        if graphs > 1:  # graphs of one host are alike, not equal: a third to five thirds of n
            one["n"] = max(1_000, case["n"] * (graphs + 2 * (i + 1)) // (2 * graphs + 1))
            one["batch"] = max(2, case["batch"] * one["n"] // case["n"])
        made.append((one["n"], *_stream(one, seed * 1009 + i)))
    state = {"case": case, "step": 0}
    if case["form"] == "create":
        n, csr, _ = made[0]
        state.update(n=n, csr=csr, args=args)
        return state
    streams = [torch.cuda.Stream() for _ in made] if graphs > 1 else []
    if case["form"] == "served":
        state["server"] = Server(workers=4)
        args["server"] = state["server"]
    state["ldl"] = [LDL(n, *csr, stream=streams[i].cuda_stream if streams else None, **args)
                    for i, (n, csr, _) in enumerate(made)]
    state["streams"] = streams
    state["ring"] = [b for _, _, b in made]
    state["labels"] = [d.labels() for d in state["ldl"]]
    return state


def _take_changes(state):
    """What a caller does after a batch: its own labels take the changed ones."""
    for mine, d in zip(state["labels"], state["ldl"]):
        ids, lab = d.changed()
        mine[ids] = lab


def run(state):
    case = state["case"]
    if case["form"] == "create":
        d = LDL(state["n"], *state["csr"], **state["args"])
        out = {"labels": d.labels(), "modularity": d.modularity(), "levels": d.levels}
        d.close()
        return out
    ldl, now = state["ldl"], state["step"] % (2 * K)
    state["step"] += 1
    batches = [ring[now] for ring in state["ring"]]
    if case["form"] == "apply":
        ldl[0].apply(batches[0], on_device=case["on_device"])
        _take_changes(state)
    elif case["form"] == "batched":
        apply_batches(ldl, batches)
        _take_changes(state)
    else:
        server = state["server"]
        tickets = [server.submit(d, b) for d, b in zip(ldl, batches)]
        if any(server.wait(t)[0] for t in tickets):
            raise RuntimeError("a request failed")
        for mine, d in zip(state["labels"], ldl):
            mine[:] = d.labels()
    labels = state["labels"][0] if len(ldl) == 1 else np.concatenate(state["labels"])
    return {"labels": labels, "modularity": np.array([d.modularity() for d in ldl]),
            "levels": np.array([d.levels for d in ldl])}


def work(case):
    """Static build: the CSR in, one sweep over its entries with their labels,
    the labels out.  Batch: its updates (16 bytes), the rows of the endpoints
    and of their neighbours (the first candidate set) once, at 12 bytes an
    entry (id, weight, label), bounded by the whole graph, and 8 bytes for
    each relabelled endpoint."""
    total = 0
    for i in range(case["graphs"]):
        n = case["n"] if case["graphs"] == 1 else case["n"] * (case["graphs"] + 2 * (i + 1)) // (2 * case["graphs"] + 1)
        entries = n * case["deg"] * (2 if case["directed"] else 1)
        if case["form"] == "create":
            total += n * 8 + n * case["deg"] * 8 + entries * 12 + n * 4
            continue
        b = max(2, case["batch"] * n // case["n"])
        swept = min(entries, 2 * b * (1 + case["deg"]) * case["deg"])
        total += 16 * b + 12 * swept + 16 * b
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    # labels are whole numbers and compared as such; the modularity follows from
    # them by integer arithmetic, and there is no other way to it than the
    # method itself, which plain array code does not do in reasonable time
    return None
