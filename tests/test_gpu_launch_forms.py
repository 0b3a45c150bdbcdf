"""The forms a local-moving iteration takes that small inputs no longer reach
by themselves, bit for bit against the CPU oracle (every compared value is an
integer, so nothing has a tolerance): host launches of the per-bin kernels with
the list lengths known (the serial flag and the decide-phase profile keep the
small-frontier kernel from taking the iteration), one after another and on
concurrent streams; scores of 128 bits in every table; and the small-frontier
kernel's list of moves near its largest size.
"""
import numpy as np
import pytest

import synth
from test_gpu_kernel_edges import dfl, orc, pair, random_graph, same, stars  # noqa: F401 (dfl, orc: fixtures)

pytestmark = pytest.mark.gpu

NO_GRAPH, SERIAL, PERSISTENT, PROFILE_MOVE = 4, 8, 16, 64
HOST_FORMS = [NO_GRAPH | SERIAL, NO_GRAPH | PROFILE_MOVE]


def launches(h, call):
    before = h.stats()["kernel_launches"]
    out = call()
    return out, h.stats()["kernel_launches"] - before


@pytest.mark.parametrize("flags", HOST_FORMS)
@pytest.mark.parametrize("degrees", [(8, 9, 64, 65), (511, 512, 513), (1024, 1025, 2600), (257, 900, 4097, 9000), (520,) * 300])
def test_host_launched_iteration(dfl, orc, degrees, flags):  # noqa: F811
    """One iteration around movers of every bin, each sub-step class with some
    bins empty; more kernels than the small-frontier form has."""
    g = stars(degrees, max(2700, max(degrees)), 9)
    a, b = pair(dfl, orc, g, flags=flags)
    small, _ = pair(dfl, orc, g, flags=NO_GRAPH)
    rng = np.random.default_rng(2)
    for density in (0.7, 0.01):
        C = rng.integers(0, g.n, g.n).astype(np.uint32)
        for x in (a, b, small):
            x.set_membership(C)
        F, R = (rng.random(g.n) < density).astype(np.uint8), (rng.random(g.n) < 0.9).astype(np.uint8)
        F[: len(degrees)] = 1
        (Fa, ma, Sa), count = launches(a, lambda: a.move_iteration(F, R))
        Fb, mb, Sb = b.move_iteration(F, R)
        assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb
        if density < 0.1:
            assert count > launches(small, lambda: small.move_iteration(F, R))[1]
        same(a, b)


@pytest.mark.parametrize("flags", HOST_FORMS)
@pytest.mark.parametrize("n,m", [(40, 90), (3000, 9000), (5000, 60_000)])
def test_host_launched_passes(dfl, orc, n, m, flags):  # noqa: F811
    """Whole runs: static, then updates of every mode and a fused step."""
    g = random_graph(n, m, n + 1)
    a, b = pair(dfl, orc, g, flags=flags, substeps=8, tau_num=1, tau_den=10**9)
    a.static()
    b.static()
    same(a, b)
    assert a.stats()["iterations"] == b.stats()["iterations"] and a.trace() == b.trace()
    stream = synth.BatchStream(g, 5)
    for mode in (2, 1, 0, 2):
        dels, ins = stream.next(max(4, m // 100), w_max=9)
        if mode == 2:
            assert a.step(dels, ins) == 0
        else:
            assert a.apply_batch(dels, ins) == 0
            a.update(mode)
        assert b.apply_batch(dels, ins) == 0
        b.update(mode)
        same(a, b)
        assert a.stats()["affected_ever"] == b.stats()["affected_ever"] and a.trace() == b.trace()


@pytest.mark.parametrize("flags", HOST_FORMS)
def test_host_launched_group(dfl, orc, flags):  # noqa: F811
    import torch
    gs = [random_graph(n, 4 * n, 80 + n) for n in (30, 900, 257, 1500)]
    csrs = [(g.n, *synth.to_csr(g)) for g in gs]
    grp = dfl.DflGroup(csrs, options=dfl.default_options(flags=flags), stream=torch.cuda.Stream())
    orcs = [orc.Oracle(*c) for c in csrs]
    grp.static()
    streams = [synth.BatchStream(g, 3) for g in gs]
    for o in orcs:
        o.static()
    for mode in (2, 1, 0):
        batches = [s.next(6, w_max=5) for s in streams]
        grp.apply_batches([d for d, _ in batches], [i for _, i in batches])
        grp.update(mode)
        for k, o in enumerate(orcs):
            assert o.apply_batch(*batches[k]) == 0
            o.update(mode)
            assert np.array_equal(grp.graph_membership(k), o.membership())
            assert grp.graph_modularity(k)[1:] == o.modularity()[1:]


# ---------------------------------------------------------------------------
# Scores of 128 bits.  Only a community holding more than half of 2m has
# 2m * K >= 2^63, so it is a super-vertex of a later pass (a self-loop of nearly
# all of its weight).
# ---------------------------------------------------------------------------
def heavy_graph(pairs, hubs, links, degree, seed):
    """`pairs` pairs of vertices, the first `hubs` of them joined to `links`
    others each; a ballast pair; loose vertices, which make the first pass run
    more than one iteration; and at the end a star of 0.55 of the whole weight,
    joined to both vertices of `degree` pairs so that each pair is better off
    as it is, but the two communities better off together.  Returns the graph
    and the membership: a community per pair, ballast and star."""
    rng = np.random.default_rng(seed)
    x = 2 * np.arange(pairs)
    e = [(x, x + 1, np.full(pairs, 2000))]
    u = np.repeat(np.arange(hubs), links)
    v = np.concatenate([rng.permutation(pairs)[:links] for _ in range(hubs)])
    e.append((x[u[u != v]], x[v[u != v]], np.ones(int((u != v).sum()))))
    at = 2 * pairs
    e.append((np.array([at]), np.array([at + 1]), np.array([930_000_000])))
    loose = at + 2 + np.arange(40)
    e.append((loose[:-1], loose[1:], rng.integers(1, 9, 39)))
    hub = int(loose[-1]) + 1
    leaves = hub + 1 + np.arange(20)
    e.append((np.full(20, hub), leaves, np.full(20, 58_000_000)))
    joined = rng.permutation(pairs)[:degree]
    for side in (0, 1):
        e.append((x[joined] + side, leaves[rng.integers(0, 20, degree)], 4000 + rng.integers(0, 200, degree)))
    n = hub + 21
    a, b, w = (np.concatenate([t[k] for t in e]).astype(np.int64) for k in range(3))
    lo, hi = np.minimum(a, b), np.maximum(a, b)
    _, first = np.unique(lo * n + hi, return_index=True)
    C = np.arange(n, dtype=np.uint32)
    C[x + 1] = x
    C[at + 1] = at
    C[leaves] = hub
    g = synth.EdgeList(n, lo[first].astype(np.uint32), hi[first].astype(np.uint32), w[first].astype(np.uint32))
    return g, C, hub


# per form: pairs, hubs, links of a hub, degree of the heavy super-vertex; the
# host launches have more vertices of its bin than warps or blocks
HEAVY = {"table": (8000, 8000, 24, 100), "mid": (1500, 1400, 300, 600), "whole": (3200, 500, 1100, 3000),
         "small table": (1500, 1500, 24, 100), "small mid": (700, 90, 300, 600), "small whole": (3050, 40, 1100, 3000)}


@pytest.mark.parametrize("form,flags,substeps", [
    ("table", NO_GRAPH | SERIAL, 1), ("mid", NO_GRAPH | SERIAL, 1), ("whole", NO_GRAPH | SERIAL, 1),
    ("table", PERSISTENT, 4), ("mid", PERSISTENT, 4), ("whole", PERSISTENT, 4),
    ("small table", NO_GRAPH, 4), ("small mid", NO_GRAPH, 4), ("small whole", NO_GRAPH, 4),
])
def test_scores_beyond_64_bits_in_tables(dfl, orc, form, flags, substeps):  # noqa: F811
    """The heavy super-vertex moves, and the vertices after it find the warp's
    or block's table empty."""
    g, C, hub = heavy_graph(*HEAVY[form], seed=4)
    kw = dict(substeps=substeps, tau_num=1, tau_den=10**15, tau_agg=1.0, max_iterations=6)
    a, b = pair(dfl, orc, g, flags=flags, **kw)
    first = orc.Oracle(g.n, *synth.to_csr(g))
    first.set_options(max_passes=1, **kw)
    for h in (a, b, first):
        h.set_membership(C)
        h.update(0)
    # the first pass leaves the pairs and the star as they were
    F = first.membership()
    assert np.array_equal(F == F[hub], C == C[hub]) and np.array_equal(F[0:2 * HEAVY[form][0]:2], F[1:2 * HEAVY[form][0]:2])
    K, _, two_m = b.weights()
    K = [int(K[C == C[hub]].sum()), int(two_m)]
    assert K[1] < 2**32 and K[0] * K[1] >= 2**63
    assert b.stats()["passes"] > 1
    same(a, b)
    assert a.stats()["iterations"] == b.stats()["iterations"]
    assert (b.membership() == b.membership()[hub]).sum() > 21  # it joined another community, or was joined


@pytest.mark.parametrize("n", [11_900, 12_000, 12_001])  # (the last is left to the per-bin kernels)
@pytest.mark.parametrize("cycles,bin_warp", [(4, 8), (2, 4)])
def test_small_frontier_where_nearly_every_vertex_moves(dfl, orc, n, cycles, bin_warp):  # noqa: F811
    """The largest sub-step class the small-frontier kernel takes, of vertices
    that nearly all move: its lists of moves are as full as they get."""
    rng = np.random.default_rng(n + cycles)
    u = np.concatenate([rng.permutation(n) for _ in range(cycles)])
    v = np.concatenate([np.roll(u[k * n:(k + 1) * n], 1) for k in range(cycles)])
    key = np.unique(np.minimum(u, v) * np.int64(n) + np.maximum(u, v))
    g = synth.EdgeList(n, (key // n).astype(np.uint32), (key % n).astype(np.uint32),
                       rng.integers(1, 9, key.size).astype(np.uint32))
    a, b = pair(dfl, orc, g, flags=NO_GRAPH, substeps=1, max_iterations=4)
    a.set_tuning(bin_warp=bin_warp)
    C = rng.integers(0, n // 3, n).astype(np.uint32)
    a.set_membership(C)
    b.set_membership(C)
    ones = np.ones(n, np.uint8)
    Fa, ma, Sa = a.move_iteration(ones, ones)
    Fb, mb, Sb = b.move_iteration(ones, ones)
    assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb
    assert ma.mean() > 0.9
    a.static()
    b.static()
    same(a, b)
    assert a.trace() == b.trace()


@pytest.mark.parametrize("flags", [NO_GRAPH | SERIAL, PERSISTENT, 32])  # (32: graph replay)
@pytest.mark.parametrize("degrees", [(4097, 5120, 5121), (8191, 8192, 8193), (12_289, 16_400), (4100,) * 75, (4100,) * 76,
                                     (4150,) * 77])
def test_hubs_of_a_run_from_singletons(dfl, orc, degrees, flags):  # noqa: F811
    """Static runs over few hub arcs (chunks of 1,024) and over more than the
    line between the chunk sizes, every class in one sub-step."""
    g = stars(degrees, max(4200, max(degrees)), 17)
    a, b = pair(dfl, orc, g, flags=flags, substeps=1, max_iterations=3)
    a.static()
    b.static()
    same(a, b)
    assert a.trace() == b.trace() and a.stats()["iterations"] == b.stats()["iterations"]
    a.update(0)  # from communities: chunks of 4,096
    b.update(0)
    same(a, b)
    # ... and from the many communities that one iteration leaves
    kw = dict(max_passes=1, max_iterations=1, substeps=1)
    a.set_options(dfl.default_options(flags=flags, **kw))
    b.set_options(**kw)
    a.static()
    b.static()
    F = R = np.ones(g.n, np.uint8)
    Fa, ma, Sa = a.move_iteration(F, R)
    Fb, mb, Sb = b.move_iteration(F, R)
    assert np.array_equal(Fa, Fb) and np.array_equal(ma, mb) and Sa == Sb
    same(a, b)


@pytest.mark.parametrize("n,degrees", [
    (3000, (64, 65, 128, 129, 2900)),            # four rows a warp
    (155_648, (127, 128, 129, 257)), (155_649, (255, 256, 257, 1000)),  # ... eight
    (311_297, (256, 257, 700)),                  # ... sixteen
    (622_592, (256, 257, 513)), (622_593, (511, 512, 513, 40_000)),     # ... thirty-two
])
def test_row_sums_at_the_lines_between_their_forms(dfl, orc, n, degrees):  # noqa: F811
    """K, 2m and the modularity where a warp takes more rows, with rows at the
    lengths that are queued, side by side at the first ids."""
    c = len(degrees)
    hubs = stars(degrees, n - c, 5)
    rng = np.random.default_rng(n)
    keep = (np.arange(hubs.u.size) < sum(degrees)) | (rng.random(hubs.u.size) < 0.5)  # half of the leaves' ring
    g = synth.EdgeList(n, hubs.u[keep], hubs.v[keep], hubs.w[keep])
    a, b = pair(dfl, orc, g)
    C = rng.integers(0, 40, n).astype(np.uint32)
    a.set_membership(C)
    b.set_membership(C)
    same(a, b)


@pytest.mark.parametrize("flags", [0, NO_GRAPH, PERSISTENT, 32])
@pytest.mark.parametrize("degrees,leaves", [((30, 5), 600), ((3000, 700, 300) * 20, 3000), ((5000, 4200) * 6, 9000)])
def test_delta_screening_frontier_counted_on_the_host(dfl, orc, degrees, leaves, flags):  # noqa: F811
    """DS updates whose frontier is small, refused by the small-frontier kernel,
    or replayed: the marked vertices' count and the whole run, also after a
    marking that no update followed."""
    g = stars(degrees, leaves, 11)
    a, b = pair(dfl, orc, g, flags=flags)
    a.static()
    b.static()
    stream = synth.BatchStream(g, 5)
    for size in (8, 900, 40):
        dels, ins = stream.next(size, w_max=9)
        assert a.apply_batch(dels, ins) == 0 and b.apply_batch(dels, ins) == 0
        for x, y in zip(a.mark(1), b.mark(1)):
            assert np.array_equal(x, y)
        a.update(1)
        b.update(1)
        same(a, b)
        assert a.stats()["affected_initial"] == b.stats()["affected_initial"] and a.trace() == b.trace()
