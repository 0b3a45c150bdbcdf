"""What a user of this framework has it do, as timed cases.

Every case is a dynamic graph held by a handle and one call sequence on it:
a Dynamic Frontier step (`dfl_step`), a batch apply followed by an ND, DS or
DF update, a static Louvain run, or the same for a group of graphs, with the
membership (and, where it is the caller's state too, K and Sigma) read back.
Graphs are the shapes the method is evaluated on: a stochastic block model,
R-MAT graphs with 8 edges per vertex, a temporal preferential-attachment
stream with a sliding window, and weighted planted partitions, alone and as a
group.  They are made on the GPU from the seed alone.

A pass applies the next batch of a stream.  A stream plays its batches
forward and then undoes them in reverse order (every deleted edge comes back
with its weight, every insertion is removed), so that it never runs out and
the graph keeps its size.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2404_19634_gb300 as dfl

FORWARD = 4  # batches of a stream before it turns back

MODES = {"nd": dfl.ND, "ds": dfl.DS, "df": dfl.DF}


def listed():
    return [
        # the smallest call: a 10,000-vertex block model kept up to date
        # after every 100 changes, batch and results on the host
        {"name": "sbm10k_df_100", "graph": "planted", "n": 10_000, "blocks": 50, "mu": 0.33, "degree": 5.9,
         "w_max": 1, "call": "step", "mode": "df", "batch": 100, "host": True},
        # ... and its communities from scratch (a user's first call)
        {"name": "sbm10k_static", "graph": "planted", "n": 10_000, "blocks": 50, "mu": 0.33, "degree": 5.9,
         "w_max": 1, "call": "static", "host": True},
        # a few dozen changes on a large skewed graph: latency of a step that
        # touches almost nothing
        {"name": "rmat22_df_1e-6", "graph": "rmat", "scale": 22, "call": "step", "mode": "df", "batch": 34,
         "host": False},
        # the method's headline: batches of 1e-3 of the edges of an R-MAT
        # graph of 2^22 vertices
        {"name": "rmat22_df_1e-3", "graph": "rmat", "scale": 22, "call": "step", "mode": "df", "batch": 33_554,
         "host": False},
        # the largest request of the served stream: a million changes from
        # pinned host memory
        {"name": "rmat21_df_1e6_host", "graph": "rmat", "scale": 21, "call": "step", "mode": "df",
         "batch": 1_000_000, "host": True},
        # a temporal stream of 2 million vertices: 3,000 interactions arrive
        # and the 3,000 oldest expire
        {"name": "temporal_df_1e-4", "graph": "temporal", "n": 2_000_000, "steps": 30_000_000, "call": "update",
         "mode": "df", "batch": 3_000, "host": False},
        # the other two dynamic methods a user may choose
        {"name": "rmat22_nd_1e-3", "graph": "rmat", "scale": 22, "call": "update", "mode": "nd", "batch": 33_554,
         "host": False},
        {"name": "rmat20_ds_1e-4", "graph": "rmat", "scale": 20, "call": "update", "mode": "ds", "batch": 839,
         "host": False},
        # communities from scratch: the skewed graph, and a weighted graph of
        # even degrees and an odd size
        {"name": "rmat22_static", "graph": "rmat", "scale": 22, "call": "static", "host": False},
        {"name": "planted400k_static", "graph": "planted", "n": 400_003, "blocks": 613, "mu": 0.3, "degree": 16.0,
         "w_max": 16, "call": "static", "host": False},
        # many independent graphs of uneven size in one handle
        {"name": "group32_df_1e-4", "graph": "group", "graphs": 32, "n_lo": 10_000, "n_hi": 200_000, "call": "update",
         "mode": "df", "frac": 1e-4, "host": True},
        {"name": "group32_static", "graph": "group", "graphs": 32, "n_lo": 10_000, "n_hi": 200_000, "call": "static",
         "host": True},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["planted", "rmat", "rmat", "temporal", "group"])
    call = rng.choice(["step", "step", "update", "static"])
    c = {"graph": kind, "call": call, "host": rng.random() < 0.4}
    if kind == "planted":
        n = log(5_000, 400_000) | 1
        c.update(n=n, blocks=max(2, min(log(20, 2000), n // 32)), mu=round(rng.uniform(0.1, 0.5), 3),
                 degree=round(rng.uniform(6.0, 16.0), 2), w_max=rng.choice([1, 16]))
        edges = n * c["degree"] / 2
    elif kind == "rmat":
        c.update(scale=rng.randint(14, 21))
        edges = 8 << c["scale"]
    elif kind == "temporal":
        n = log(50_000, 1_000_000)
        c.update(n=n, steps=15 * n)
        edges = 13 * n
    else:
        g = rng.randint(4, 32)
        c.update(graphs=g, n_lo=5_000, n_hi=log(20_000, 150_000), host=True)
        if call == "step":
            c["call"] = "update"
        if call != "static":
            c.update(frac=math.exp(rng.uniform(math.log(1e-5), math.log(1e-3))))
    if c["call"] != "static":
        c["mode"] = "df" if c["call"] == "step" else rng.choice(["df", "df", "nd", "ds"])
        if kind != "group":
            c["batch"] = log(8, min(edges * 0.02, 500_000))
    return c


# ---------------------------------------------------------------------------
# Graphs, on the GPU
# ---------------------------------------------------------------------------
def _rand_int(gen, high, k):
    return (torch.rand(k, generator=gen, device="cuda", dtype=torch.float64) * high).long()


def _rmat_pairs(gen, scale, edges, a=0.57, b=0.19, c=0.19):
    u = torch.zeros(edges, dtype=torch.int64, device="cuda")
    v = torch.zeros(edges, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = torch.rand(edges, generator=gen, device="cuda")
        u = u * 2 + (r >= a + b)
        v = v * 2 + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    perm = torch.randperm(1 << scale, generator=gen, device="cuda")
    return perm[u], perm[v]


def _planted_pairs(gen, n, blocks, mu, degree):
    size = n // blocks  # the last block takes the remainder
    k_in, k_out = int(n * (1 - mu) * degree / 2), int(n * mu * degree / 2)
    u = _rand_int(gen, n, k_in)
    blk = torch.clamp(u // size, max=blocks - 1)
    width = torch.where(blk == blocks - 1, n - size * (blocks - 1), size)
    v = blk * size + (torch.rand(k_in, generator=gen, device="cuda", dtype=torch.float64) * width).long()
    return torch.cat([u, _rand_int(gen, n, k_out)]), torch.cat([v, _rand_int(gen, n, k_out)])


def _temporal_pairs(gen, n, steps, p_repeat=0.3):
    """Preferential attachment with repeats: a step repeats an earlier
    interaction, or joins the newcomer (or a uniform arrived vertex) to a
    target drawn in proportion to its interactions so far plus the mean."""
    gap = max(1, steps // n)
    delta = max(1, 2 * steps // n)
    t = torch.arange(steps, device="cuda")
    arrived = torch.clamp(t // gap + 2, max=n)
    newest = t // gap + 1
    arrival = (t % gap == 0) & (newest < n)
    unit = lambda: torch.rand(steps, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    src = torch.where(arrival, newest, (unit() * arrived).long())
    repeat = (unit() < p_repeat) & ~arrival & (t > 0)
    earlier = (unit() * t).long()
    urn = (unit() * (delta * arrived + 2 * t)).long()
    on_vertex = urn < delta * arrived
    ptr = torch.full((2 * steps,), -1, dtype=torch.int64, device="cuda")
    val = torch.zeros(2 * steps, dtype=torch.int64, device="cuda")
    val[0::2] = src
    ptr[0::2] = torch.where(repeat, 2 * earlier, torch.full_like(t, -1))
    ptr[1::2] = torch.where(repeat, 2 * earlier + 1, torch.where(on_vertex, torch.full_like(t, -1), urn - delta * arrived))
    val[1::2] = torch.where(on_vertex, urn // delta, torch.zeros_like(t))
    todo = torch.nonzero(ptr >= 0).flatten()
    while todo.numel():  # pointers lead to earlier slots
        p = ptr[todo]
        pp = ptr[p]
        ready = pp < 0
        val[todo[ready]] = val[p[ready]]
        ptr[todo[ready]] = -1
        ptr[todo[~ready]] = pp[~ready]
        todo = todo[~ready]
    return val[0::2].clone(), val[1::2].clone()


def _keys(u, v):
    """Undirected pairs as lo << 32 | hi, self pairs dropped."""
    keep = u != v
    u, v = u[keep], v[keep]
    return (torch.minimum(u, v) << 32) | torch.maximum(u, v)


def _csr(n, key, w):
    """Symmetric CSR of distinct undirected pairs: offsets int64, indices and
    weights int32, rows sorted by neighbour."""
    u, v = key >> 32, key & 0xFFFFFFFF
    arcs, order = torch.sort(torch.cat([(u << 32) | v, (v << 32) | u]))
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(arcs >> 32, minlength=n), 0)
    return off, (arcs & 0xFFFFFFFF).int(), torch.cat([w, w])[order].int()


def _edges(key, w):
    return torch.stack([key >> 32, key & 0xFFFFFFFF, w], 1).int()


def _random_stream(gen, n, key, w, size, w_max):
    """Batches of 80% insertions between uniform pairs and 20% deletions of
    whole existing edges, forward and then undone."""
    n_del = max(1, round(size * 0.2))
    n_ins = max(1, size - n_del)
    pick = torch.randperm(key.numel(), generator=gen, device="cuda")[: FORWARD * n_del]
    forward, back = [], []
    for k in range(FORWARD):
        p = pick[k * n_del:(k + 1) * n_del]
        new = torch.unique(_keys(_rand_int(gen, n, n_ins), _rand_int(gen, n, n_ins)))
        new = new[~torch.isin(new, key[pick])]  # a whole-edge deletion takes the base weight alone
        new = new[torch.randperm(new.numel(), generator=gen, device="cuda")]
        nw = _rand_int(gen, w_max, new.numel()) + 1
        forward.append((_edges(key[p], torch.zeros_like(p)), _edges(new, nw)))
        back.append((_edges(new, nw), _edges(key[p], w[p])))
    return forward + back[::-1]


def _window_stream(src, dst, start, end, size):
    """Sliding-window batches: `size` interactions arrive, the oldest expire."""
    forward, back = [], []
    for k in range(FORWARD):
        a, b = end + k * size, start + k * size
        ins, ic = torch.unique(_keys(src[a:a + size], dst[a:a + size]), return_counts=True)
        dels, dc = torch.unique(_keys(src[b:b + size], dst[b:b + size]), return_counts=True)
        forward.append((_edges(dels, dc), _edges(ins, ic)))
        back.append((_edges(ins, ic), _edges(dels, dc)))
    return forward + back[::-1]


def _graph(case, gen):
    """(n, pair keys, weights, batch stream or None) of a single-graph case."""
    size = case.get("batch")
    if case["graph"] == "temporal":
        n, steps = case["n"], case["steps"]
        src, dst = _temporal_pairs(gen, n, steps)
        end = steps * 9 // 10
        key, w = torch.unique(_keys(src[:end], dst[:end]), return_counts=True)
        size = min(size, (steps - end) // FORWARD) if size else None
        return n, key, w, _window_stream(src, dst, 0, end, size) if size else None
    if case["graph"] == "rmat":
        n, w_max = 1 << case["scale"], 1
        u, v = _rmat_pairs(gen, case["scale"], 8 * n)
    else:
        n, w_max = case["n"], case["w_max"]
        u, v = _planted_pairs(gen, n, case["blocks"], case["mu"], case["degree"])
    key = torch.unique(_keys(u, v))
    w = _rand_int(gen, w_max, key.numel()) + 1
    return n, key, w, _random_stream(gen, n, key, w, size, w_max) if size else None


def _group_sizes(case):
    g = case["graphs"]  # log-spaced over the range, so that the work is the same for every seed
    return [round(math.exp(math.log(case["n_lo"]) + (math.log(case["n_hi"]) - math.log(case["n_lo"])) * (k + 0.5) / g))
            for k in range(g)]


def _options(case):
    # the paper's aggregation tolerance: 1 for temporal streams, 0.8 otherwise
    return dfl.default_options(tau_agg=1.0 if case["graph"] == "temporal" else 0.8)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    st = {"case": case, "pos": 0}
    stream = torch.cuda.Stream()
    if case["graph"] == "group":
        graphs, streams = [], []
        for n in _group_sizes(case):
            blocks = max(2, min(20 + int(_rand_int(gen, 1980, 1)), n // 32))
            mu = 0.1 + 0.4 * float(torch.rand(1, generator=gen, device="cuda"))
            key = torch.unique(_keys(*_planted_pairs(gen, n, blocks, mu, 16.0)))
            w = _rand_int(gen, 16, key.numel()) + 1
            off, idx, ws = _csr(n, key, w)
            graphs.append((n, off.cpu().numpy().view(np.uint64), idx.cpu().numpy().view(np.uint32),
                           ws.cpu().numpy().view(np.uint32)))
            if case["call"] != "static":
                size = max(2, round(case["frac"] * key.numel()))
                streams.append(_random_stream(gen, n, key, w, size, 16))
        h = dfl.DflGroup(graphs, options=_options(case), stream=stream)
        st["batches"] = [tuple([s[k][side].cpu().numpy().view(np.uint32) for s in streams] for side in (0, 1))
                         for k in range(2 * FORWARD)] if streams else None
    else:
        n, key, w, batches = _graph(case, gen)
        csr = _csr(n, key, w)
        torch.cuda.synchronize()  # the handle's stream reads what this one made
        h = dfl.Dfl(n, *csr, options=_options(case), stream=stream)
        if batches and case["host"]:
            batches = [tuple(x.cpu().pin_memory() for x in b) for b in batches]
        st["batches"] = batches
    if case["call"] != "static":
        h.static()
    st["h"] = h
    if case["host"]:
        st["C"] = torch.empty(h.n, dtype=torch.int32).pin_memory()
    else:
        st["C"] = torch.empty(h.n, dtype=torch.int32, device="cuda")
        st["K"] = torch.empty(h.n, dtype=torch.int64, device="cuda")
        st["Sigma"] = torch.empty(h.n, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    return st


def run(state):
    case, h = state["case"], state["h"]
    if case["call"] == "static":
        h.static()
    else:
        dels, ins = state["batches"][state["pos"]]
        state["pos"] = (state["pos"] + 1) % len(state["batches"])
        if case["graph"] == "group":
            h.apply_batches(dels, ins)
            h.update(MODES[case["mode"]])
        elif case["call"] == "step":
            h.step(dels, ins, MODES[case["mode"]])
        else:
            h.apply_batch(dels, ins)
            h.update(MODES[case["mode"]])
    out = {"membership": h.membership(state["C"])}
    if case["host"]:
        if case["graph"] != "group":
            out["modularity"] = h.modularity()[0]
        return out
    two_m = ctypes.c_int64()
    rc = dfl.dfl_weights(h.handle, state["K"].data_ptr(), state["Sigma"].data_ptr(), ctypes.byref(two_m),
                         dfl.MEM_DEVICE)
    if rc:
        raise dfl.DflError(rc, "dfl_weights")
    out.update(K=state["K"], Sigma=state["Sigma"], two_m=two_m.value)
    return out


def work(case):
    """A static run and an ND or DS update read the graph, its membership, K
    and Sigma once; a DF update reads the rows that the batch touches.  The
    batch is read once and the results are written once."""
    kind = case["graph"]
    if kind == "rmat":
        n, m = 1 << case["scale"], 8 << case["scale"]
    elif kind == "temporal":
        n, m = case["n"], 0.65 * case["steps"]
    elif kind == "group":
        n = sum(_group_sizes(case))
        m = 8 * n
    else:
        n, m = case["n"], case["n"] * case["degree"] / 2
    edges = 0
    if case["call"] != "static":
        edges = case["frac"] * m if kind == "group" else case["batch"] * (2 if kind == "temporal" else 1)
    arcs = min(2 * m, 2 * edges * 2 * m / n) if case.get("mode") == "df" else 2 * m
    rows = min(n, 2 * edges) if case.get("mode") == "df" else n
    results = 4 * n if case["host"] else 20 * n
    return {"bytes": 12 * edges + 16 * edges + 8 * arcs + 24 * rows + results, "flops": 2 * arcs}


def exact(case, seed):
    """None: memberships, K, Sigma and 2m are whole numbers, which stay equal,
    and the modularity's one division is of whole numbers that follow from the
    membership of a whole Louvain run."""
    return None
