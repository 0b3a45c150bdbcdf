"""Edges of the kernels' tiles and dispatch limits, bit for bit against the
CPU oracle (every compared value is an integer, so nothing has a tolerance).
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dfl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2404_19634_gb300 as mod
    mod.build()
    mod.load()
    return mod


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


_STREAMS = []


def pair(dfl, orc, g, **kw):
    import torch
    off, idx, w = synth.to_csr(g)
    s = torch.cuda.Stream()
    _STREAMS.append(s)
    a = dfl.Dfl(g.n, off, idx, w, options=dfl.default_options(**kw), stream=s)
    b = orc.Oracle(g.n, off, idx, w)
    b.set_options(**{k: v for k, v in kw.items() if k != "flags"})
    return a, b


def same(a, b):
    assert np.array_equal(a.membership(), b.membership())
    for x, y in zip(a.weights(), b.weights()):
        assert np.array_equal(x, y)
    assert a.modularity()[1:] == b.modularity()[1:]


def random_graph(n, m, seed, w_max=9):
    """n vertices and about m random weighted edges."""
    rng = np.random.default_rng(seed)
    if n < 2:
        return synth.EdgeList(n, *(np.zeros(0, np.uint32),) * 3)
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    key = np.unique(np.minimum(u, v)[u != v] * np.int64(n) + np.maximum(u, v)[u != v])
    return synth.EdgeList(n, (key // n).astype(np.uint32), (key % n).astype(np.uint32),
                          rng.integers(1, w_max + 1, key.size).astype(np.uint32))


def stars(degrees, leaves, seed):
    """One centre per degree, joined to the first `degree` of a shared pool of
    leaves, which are also joined in a ring (so that centres meet many
    communities and leaves have choices)."""
    rng = np.random.default_rng(seed)
    c = len(degrees)
    u = np.concatenate([np.full(d, k) for k, d in enumerate(degrees)] + [c + np.arange(leaves)])
    v = np.concatenate([c + rng.permutation(leaves)[:d] for d in degrees] + [c + (np.arange(leaves) + 1) % leaves])
    return synth.EdgeList(c + leaves, np.minimum(u, v).astype(np.uint32), np.maximum(u, v).astype(np.uint32),
                          rng.integers(1, 20, u.size).astype(np.uint32))


@pytest.mark.parametrize("n", [1, 31, 2047, 2049, 8191, 8200, 20_011])
@pytest.mark.parametrize("density", [0.002, 0.2, 1.0])
def test_frontier_lists_at_tile_edges(dfl, orc, n, density):
    """A frontier given as a bitmap (sparse: its tiles compacted together;
    dense: tile by tile) reaches exactly the vertices it names."""
    g = random_graph(n, 3 * n, n)
    rng = np.random.default_rng(7)
    F = (rng.random(n) < density).astype(np.uint8)
    F[-1] = 1
    R = np.ones(n, np.uint8)
    a, b = pair(dfl, orc, g)
    C = rng.integers(0, max(1, n // 3), n).astype(np.uint32)
    a.set_membership(C)
    b.set_membership(C)
    Fa, ma, Sa = a.move_iteration(F, R)
    Fb, mb, Sb = b.move_iteration(F, R)
    assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb
    a.static()
    b.static()
    same(a, b)


@pytest.mark.parametrize("degrees", [(64, 65), (1023, 1024, 1025), (2048, 4097, 1), (1030,) * 40])
def test_row_sums_of_hubs(dfl, orc, degrees):
    """K, 2m and the modularity at the row lengths where a row takes the
    whole warp, and where it is queued and cut into pieces."""
    g = stars(degrees, 4100, 3)
    a, b = pair(dfl, orc, g)
    C = np.random.default_rng(1).integers(0, 50, g.n).astype(np.uint32)
    a.set_membership(C)
    b.set_membership(C)
    same(a, b)


@pytest.mark.parametrize("degrees", [(512, 513), (1024, 1025, 3), (4000, 600, 511)])
def test_delta_screening_marks_hub_neighbours(dfl, orc, degrees):
    g = stars(degrees, 4100, 5)
    a, b = pair(dfl, orc, g)
    a.static()
    b.static()
    c = len(degrees)
    C = a.membership()
    # each centre loses an edge inside its community and gains one across
    dels, ins = [], []
    for k in range(c):
        row = np.concatenate([g.v[g.u == k], g.u[g.v == k]])
        inside = row[C[row] == C[k]]
        if inside.size:
            dels.append((k, inside[0], 0))
        other = np.flatnonzero(C != C[k])
        if other.size:
            ins.append((k, other[-1 - k], 2))
    dels, ins = np.array(dels, np.uint32).reshape(-1, 3), np.array(ins, np.uint32).reshape(-1, 3)
    assert dels.size + ins.size
    assert a.apply_batch(dels, ins) == 0 and b.apply_batch(dels, ins) == 0
    for x, y in zip(a.mark(1), b.mark(1)):
        assert np.array_equal(x, y)
    a.update(1)
    b.update(1)
    same(a, b)


@pytest.mark.parametrize("mean_degree,n,flags", [
    (16, 12_000, 4),    # a list above the lane bin's limit, host launches
    (16, 33_000, 32),   # ... graph replay
    (4, 33_000, 4),     # bin 0's long lists
    (4, 33_000, 32),
])
def test_lane_per_vertex_lists(dfl, orc, mean_degree, n, flags):
    """Long lists of vertices of up to 8, 16 and 32 arcs (a lane each), with
    weights, deleted arcs and re-inserted ones in the rows."""
    g = random_graph(n, n * mean_degree // 2, mean_degree)
    a, b = pair(dfl, orc, g, substeps=1, flags=flags, max_iterations=3)
    a.static()
    b.static()
    same(a, b)
    stream = synth.BatchStream(g, 5)
    for _ in range(2):
        dels, ins = stream.next(2000, w_max=9)
        assert a.apply_batch(dels, ins) == 0 and b.apply_batch(dels, ins) == 0
        a.update(0)
        b.update(0)
        same(a, b)


@pytest.mark.parametrize("flags", [4, 32])
def test_lane_per_vertex_scores_beyond_64_bits(dfl, orc, flags):
    """A community holding nearly all of 2m becomes a super-vertex (a
    self-loop and a few arcs) whose K times 2m is above 2^63, in a second pass
    over a long list of small super-vertices."""
    n, heavy = 80_000, 105_000_000
    g = random_graph(n - 21, (n - 21) * 5 // 4, 3, w_max=3)
    hub = n - 21  # a star of 20 heavy edges, three of its leaves joined to the rest
    u = np.concatenate([g.u, np.full(20, hub), np.array([5, 70, 900])]).astype(np.uint32)
    v = np.concatenate([g.v, hub + 1 + np.arange(20), hub + 1 + np.arange(3)]).astype(np.uint32)
    w = np.concatenate([g.w, np.full(20, heavy), np.ones(3)]).astype(np.uint32)
    a, b = pair(dfl, orc, synth.EdgeList(n, u, v, w), substeps=1, flags=flags, max_iterations=3, tau_agg=1.0)
    a.set_tuning(bin_warp=0)  # every vertex of up to 32 arcs in one list
    a.static()
    b.static()
    same(a, b)
    two_m = a.weights()[2]
    assert two_m < 2**32 and (40 * heavy) * two_m > 2**63
    assert a.stats()["num_communities"] > 12_000 and a.stats()["passes"] > 1


@pytest.mark.parametrize("flags", [4, 16, 32])  # host launches, persistent kernel, graph replay
@pytest.mark.parametrize("degrees", [(8, 9, 64, 65), (511, 512, 513), (1024, 1025, 2600), (520,) * 300])
def test_movers_mark_their_neighbours(dfl, orc, degrees, flags):
    """The next frontier around movers whose rows are marked by eight lanes,
    a warp, or in queued pieces."""
    g = stars(degrees, 2700, 9)
    a, b = pair(dfl, orc, g, flags=flags)
    rng = np.random.default_rng(2)
    for _ in range(3):
        C = rng.integers(0, g.n, g.n).astype(np.uint32)
        a.set_membership(C)
        b.set_membership(C)
        F, R = (rng.random(g.n) < 0.7).astype(np.uint8), (rng.random(g.n) < 0.9).astype(np.uint8)
        F[: len(degrees)] = 1
        Fa, ma, Sa = a.move_iteration(F, R)
        Fb, mb, Sb = b.move_iteration(F, R)
        assert ma[: len(degrees)].any()
        assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb


def hub_graph(degree, leaves, seed):
    """A hub of the given degree among weighted leaves joined in a ring."""
    return stars((degree, 300, 40, 12, 3), leaves, seed)


@pytest.mark.parametrize("substeps", [1, 4, 8])
@pytest.mark.parametrize("degree,leaves", [(4097, 4100), (5000, 6000), (60_000, 70_000), (131_072, 131_100),
                                           (131_073, 131_100)])  # (the last one is left to the per-bin kernels)
def test_small_frontier_with_a_hub(dfl, orc, degree, leaves, substeps):
    """A frontier of a few vertices around a hub decided by the whole cluster:
    a community of its own for every leaf, and a few communities."""
    g = hub_graph(degree, leaves, 4)
    a, b = pair(dfl, orc, g, flags=4, substeps=substeps)
    rng = np.random.default_rng(8)
    R = np.ones(g.n, np.uint8)
    for communities in (g.n, 50, 3):
        C = (np.arange(g.n) if communities == g.n else rng.integers(0, communities, g.n)).astype(np.uint32)
        a.set_membership(C)
        b.set_membership(C)
        F = np.zeros(g.n, np.uint8)
        F[:5] = 1
        F[rng.integers(5, g.n, 200)] = 1
        Fa, ma, Sa = a.move_iteration(F, R)
        Fb, mb, Sb = b.move_iteration(F, R)
        assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb
        same(a, b)


@pytest.mark.parametrize("n,m", [(40, 90), (700, 9000), (3000, 9000), (5000, 60_000)])
@pytest.mark.parametrize("max_iterations", [1, 2, 20, 47])
def test_small_frontier_runs_whole_passes(dfl, orc, n, m, max_iterations):
    """Passes of several iterations in one launch: iteration counts, trace,
    memberships; also when they take more than one launch's iterations, and
    sub-steps without a vertex."""
    g = random_graph(n, m, n + 1)
    a, b = pair(dfl, orc, g, flags=4, substeps=8, max_iterations=max_iterations, tau_num=1, tau_den=10**12)
    a.static()
    b.static()
    same(a, b)
    assert a.stats()["iterations"] == b.stats()["iterations"] and a.trace() == b.trace()
    stream = synth.BatchStream(g, 5)
    for size in (1, 5, 100):
        dels, ins = stream.next(size, w_max=9)
        if size == 5:
            assert a.apply_batch(dels, ins) == 0
            a.update(2)
        else:
            assert a.step(dels, ins) == 0
        assert b.apply_batch(dels, ins) == 0
        b.update(2)
        same(a, b)
        assert a.stats()["affected_ever"] == b.stats()["affected_ever"] and a.trace() == b.trace()


@pytest.mark.parametrize("two_calls", [True, False])
def test_row_search_at_window_and_tail_edges(dfl, orc, two_calls):
    """Batches that look up the first, last and middle arcs of rows of every
    length around the search's windows and splits, then arcs of unsorted tails
    of every length, tombstones among them; absent edges are refused."""
    degrees = list(range(1, 40)) + [143, 144, 145, 146, 152, 153, 154, 161, 162, 1000, 1459, 4095, 4096]
    g = stars(degrees, 4200, 6)
    a, b = pair(dfl, orc, g)
    a.static()
    b.static()
    c = len(degrees)
    rows = [np.sort(np.concatenate([g.v[g.u == k], g.u[g.v == k]])) for k in range(c)]
    rng = np.random.default_rng(3)

    def both(dels, ins):
        dels, ins = np.array(dels, np.uint32).reshape(-1, 3), np.array(ins, np.uint32).reshape(-1, 3)
        if two_calls:
            ra = a.apply_batch(dels, ins, check=False)
            if ra == 0:
                a.update(2)
        else:
            ra = a.step(dels, ins, check=False)
        rb = b.apply_batch(dels, ins)
        assert ra == rb
        if rb == 0:
            b.update(2)
        return rb

    added = [[] for _ in range(c)]
    for t in range(6):
        dels, ins = [], []
        for k in range(c):
            r = rows[k]
            if t % 2 == 0 and r.size > 2:  # some arcs leave, some gain weight
                for at in {0, r.size - 1, r.size // 2, int(rng.integers(r.size))}:
                    (dels if rng.random() < 0.5 else ins).append((k, int(r[at]), 0 if len(dels) % 2 else 1))
                ins = [(u, v, max(1, w)) for u, v, w in ins]
            if added[k]:
                v = added[k][int(rng.integers(len(added[k])))]
                ins.append((k, v, 3))
            free = np.setdiff1d(c + np.arange(4200), np.concatenate([r, np.array(added[k], np.int64)]))
            if free.size:
                new = rng.choice(free, min(1 + k % 7, free.size), replace=False)
                ins += [(k, int(v), 2) for v in new]
                added[k] += [int(v) for v in new]
        assert both(dels, ins) in (0, -2)
        for x, y in zip(a.graph(), b.graph()):
            assert np.array_equal(x, y)
        same(a, b)
    absent = next(v for v in c + np.arange(4200) if v not in set(rows[20]) | set(added[20]))
    assert both([(20, int(absent), 0)], []) == -2
    same(a, b)


def test_batch_touching_most_vertices(dfl, orc):
    """A batch whose arcs outnumber an eighth of the vertices: marked through
    the bitmap, and every row's record and pair's slot used and reset."""
    g = random_graph(50_000, 150_000, 2)
    a, b = pair(dfl, orc, g)
    a.static()
    b.static()
    stream = synth.BatchStream(g, 6)
    for t in range(3):
        dels, ins = stream.next(60_000, w_max=5)
        if t == 1:
            assert a.apply_batch(dels, ins) == 0
            a.update(2)
        else:
            assert a.step(dels, ins) == 0
        assert b.apply_batch(dels, ins) == 0
        b.update(2)
        for x, y in zip(a.graph(), b.graph()):
            assert np.array_equal(x, y)
        same(a, b)
        assert a.stats()["affected_initial"] == b.stats()["affected_initial"] and a.trace() == b.trace()


@pytest.mark.parametrize("members", [1, 31, 33, 255, 257, 700])
@pytest.mark.parametrize("degree", [0, 1, 3, 128, 129, 600])
def test_aggregation_of_flattened_rows(dfl, orc, members, degree):
    """One community of `members` vertices with `degree` arcs each outside it
    (bins by total degree, rows queued from 129 arcs on), among communities of
    one vertex, isolated vertices included."""
    rng = np.random.default_rng(members * 1000 + degree)
    n = 3000 + members
    u = np.repeat(np.arange(members), degree)
    v = np.concatenate([members + rng.permutation(2900)[:degree] for _ in range(members)]) if degree else u
    ring = np.arange(members - 1)  # arcs inside, so that the community has a self-loop
    u, v = np.concatenate([u, ring]), np.concatenate([v, ring + 1])
    g = synth.EdgeList(n, u.astype(np.uint32), v.astype(np.uint32), rng.integers(1, 9, u.size).astype(np.uint32))
    a, b = pair(dfl, orc, g)
    C = np.arange(n, dtype=np.uint32)
    C[:members] = 7 if members > 7 else 0
    a.set_membership(C)
    b.set_membership(C)
    for x, y in zip(a.aggregate(), b.aggregate()):
        assert np.array_equal(x, y)


def test_aggregation_of_several_giants(dfl, orc):
    """Giant communities side by side, with rows longer than one block's share."""
    g = stars((3000, 2500, 200, 130, 5000), 6000, 12)
    a, b = pair(dfl, orc, g)
    rng = np.random.default_rng(0)
    for k in (2, 3, 40):
        C = rng.integers(0, k, g.n).astype(np.uint32)
        a.set_membership(C)
        b.set_membership(C)
        for x, y in zip(a.aggregate(), b.aggregate()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("flags", [16, 32])  # persistent kernel, graph replay
@pytest.mark.parametrize("degrees", [(4097, 6143, 6145), (8191, 8192, 8193), (12_287, 12_289, 4500), (16_400,)])
def test_huge_vertices_in_chunks(dfl, orc, degrees, flags):
    """Vertices of one chunk and of several, with few communities (the chunk
    table is decided as it is, or flushed once) and with one per leaf (flushed
    every round)."""
    g = stars(degrees, 16_500, 21)
    a, b = pair(dfl, orc, g, flags=flags)
    rng = np.random.default_rng(2)
    R = np.ones(g.n, np.uint8)
    for communities in (g.n, 2000, 5):
        C = (np.arange(g.n) if communities == g.n else rng.integers(0, communities, g.n)).astype(np.uint32)
        a.set_membership(C)
        b.set_membership(C)
        for _ in range(2):  # (the second round finds every table empty again)
            F = np.zeros(g.n, np.uint8)
            F[: len(degrees)] = 1
            F[rng.integers(0, g.n, 300)] = 1
            Fa, ma, Sa = a.move_iteration(F, R)
            Fb, mb, Sb = b.move_iteration(F, R)
            assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb
        same(a, b)


@pytest.mark.parametrize("sizes", [(1,), (255, 1, 256, 257, 2, 31, 33, 700), (1,) * 300, (513, 3, 767), (5000,)])
def test_group_weights_at_slice_borders(dfl, orc, sizes):
    """Each graph's 2m (and so the exact modularity) where graphs begin and
    end at, next to and inside a 256-vertex slice, before and after a batch."""
    import torch
    gs = [random_graph(n, 3 * n, 60 + k) for k, n in enumerate(sizes)]
    csrs = [(g.n, *synth.to_csr(g)) for g in gs]
    s = torch.cuda.Stream()
    _STREAMS.append(s)
    grp = dfl.DflGroup(csrs, stream=s)
    orcs = [orc.Oracle(n, off, idx, w) for n, off, idx, w in csrs]

    def check():
        K = grp.weights()[0]
        start = 0
        for k, o in enumerate(orcs):
            assert np.array_equal(grp.graph_membership(k), o.membership())
            assert np.array_equal(K[start:start + sizes[k]], o.weights()[0])
            assert grp.graph_modularity(k)[1:] == o.modularity()[1:]
            start += sizes[k]

    grp.static()
    for o in orcs:
        o.static()
    check()
    none = np.zeros((0, 3), np.uint32)
    ins = [np.array([[0, n - 1, 3 + k]], np.uint32) if n > 1 else none for k, n in enumerate(sizes)]
    grp.apply_batches([none] * len(sizes), ins)
    grp.update(2)
    for o, i in zip(orcs, ins):
        assert o.apply_batch(none, i) == 0
        o.update(2)
    check()
