"""The routes a call can take by size, degree, memory and option give the same integers.

Sizes sit at the edges where a route changes: rounds small and large enough for one cluster of
blocks, for helper clusters and for one launch per phase; rows at the lengths where the row
sort changes; ball sets by search and by ORs; path keys by ranks and by binary search; batch
graphs whose state fits shared memory and not.  Every comparison is exact equality.
"""

import threading

import numpy as np
import pytest

from synth import erdos_renyi_gnm, rmat

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def htd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2411_06405_gb300 import build

    build.build()
    import paper_2411_06405_gb300 as mod

    mod._lib.load()
    torch.cuda.set_device(0)
    return mod


def gpu_graph(htd, n, s, d):
    return htd.htd_build_csr(n, torch.from_numpy(np.asarray(s, dtype=np.int32)).cuda(),
                             torch.from_numpy(np.asarray(d, dtype=np.int32)).cuda())


def host(t):
    return t.cpu().numpy()


# (vertices, edge list, h): small rounds only; hubs (rows of more than 64 slots, detection
# items split over warps); first rounds of more than 16,384 items at h = 1 and 2 (launches per
# phase) and the rounds after them (helper clusters, then one cluster)
ROUNDS = [
    (64, erdos_renyi_gnm(64, 200, 1), 2),
    (1 << 11, rmat(11, 12, 0.57, 0.19, 0.19, 2), 2),
    (1 << 10, rmat(10, 8, 0.57, 0.19, 0.19, 3), 3),
    (30000, erdos_renyi_gnm(30000, 120000, 4), 1),
    (30000, erdos_renyi_gnm(30000, 120000, 4), 2),
    (3000, erdos_renyi_gnm(3000, 12000, 5), 3),
]


@pytest.mark.parametrize("case", range(len(ROUNDS)))
def test_round_routes_agree(htd, case):
    n, (s, d), h = ROUNDS[case]
    g = gpu_graph(htd, n, s, d)
    t, stamp, st = htd.htd_truss_decompose(g, h, stamps=True)
    flags = [htd.HTD_OPT_NO_GRAPH, htd.HTD_OPT_TIMING, htd.HTD_OPT_COMPACT_BALLS, htd.HTD_OPT_PERSISTENT_ROUNDS,
             htd.HTD_OPT_REBUILD]
    if g.m < 30000:
        flags.append(htd.HTD_OPT_TINY_LOSS_TABLE)
    for f in flags:
        t2, stamp2, st2 = htd.htd_truss_decompose(g, h, stamps=True, flags=f)
        assert torch.equal(t, t2) and torch.equal(stamp, stamp2), f"flags {f}"
        assert st2["rounds"] == st["rounds"]
    # nor do the counts of an incremental peel depend on who ran its rounds
    _, _, sc = htd.htd_truss_decompose(g, h, flags=htd.HTD_OPT_PERSISTENT_ROUNDS)
    for key in ("frontier_edges", "hsup_evals", "member_tests", "levels"):
        assert sc[key] == st[key], key


def test_peels_side_by_side(htd):
    """Cluster rounds of several threads and streams at once, each on its own handle."""
    graphs = [ROUNDS[i] for i in (1, 2, 4, 5)] * 2
    ref = [host(htd.htd_truss_decompose(gpu_graph(htd, n, s, d), h)[0]) for n, (s, d), h in graphs]
    out = [None] * len(graphs)

    def run(i):
        n, (s, d), h = graphs[i]
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            out[i] = host(htd.htd_truss_decompose(gpu_graph(htd, n, s, d), h)[0])

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(graphs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(out, ref):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("h", [1, 2, 3])
def test_support_then_peel_on_one_handle(htd, oracle_mod, h):
    # an h-support lays the balls out by need, a peel densely: alternating on one handle
    n = 600
    s, d = erdos_renyi_gnm(n, 2400, 12)
    og = oracle_mod.OracleGraph.from_raw(n, s, d)
    sup, truss = og.h_support(h), og.truss_decompose(h)[0]
    g = gpu_graph(htd, n, s, d)
    for _ in range(2):
        np.testing.assert_array_equal(host(htd.htd_h_support(g, h)), sup)
        np.testing.assert_array_equal(host(htd.htd_truss_decompose(g, h)[0]), truss)
        other = 1 + h % 3
        np.testing.assert_array_equal(host(htd.htd_h_support(g, other)), og.h_support(other))


@pytest.mark.parametrize("deg", [63, 64, 65, 255, 256, 257, 700])
@pytest.mark.parametrize("h", [2, 3])
def test_support_around_hubs(htd, oracle_mod, h, deg):
    # three hubs of `deg` neighbours (64 and more are ORed as n-bit rows at h = 2) over a
    # sparse random graph: at h = 3 its balls come from ORs
    n = 900
    rng = np.random.default_rng(deg)
    s, d = erdos_renyi_gnm(n, 700, deg)
    for hub in (0, 31, 899):
        nb = rng.choice(n, size=deg, replace=False)
        s, d = np.concatenate([s, np.full(deg, hub)]), np.concatenate([d, nb])
    og = oracle_mod.OracleGraph.from_raw(n, s, d)
    np.testing.assert_array_equal(host(htd.htd_h_support(gpu_graph(htd, n, s, d), h)), og.h_support(h))


@pytest.mark.parametrize("n", [257, 6001, 20000])
def test_support_of_long_cycles(htd, n):
    # radius 3 by ORs on the short cycle, by search on the long ones: two balls of seven
    # consecutive vertices, one step apart, share six
    x = np.arange(n)
    g = gpu_graph(htd, n, x, (x + 1) % n)
    assert (host(htd.htd_h_support(g, 3)) == 4).all()


@pytest.mark.parametrize("n", [368639, 368641])
def test_hindex_on_either_side_of_the_rank_index(htd, n):
    # the rank index of a ball needs 8 bytes per 32 vertices of shared memory: it ends at
    # 368,640 vertices.  Isolated vertices change no key
    s, d = rmat(9, 6, 0.57, 0.19, 0.19, 21)
    small, big = gpu_graph(htd, 512, s, d), gpu_graph(htd, n, s, d)
    a = htd.htd_hindex_decompose(small, 2)
    b = htd.htd_hindex_decompose(big, 2)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert torch.equal(a[0], htd.htd_truss_decompose(small, 2)[0])


def test_batch_blocks_at_the_layout_edges(htd):
    # state in shared memory up to 220 KiB, else in global scratch; 32 and more words per ball
    graphs = []
    for i, n in enumerate([33, 500, 800, 1000, 1023, 1024, 1025, 1100, 1300, 2100]):
        s, d = erdos_renyi_gnm(n, 2 * n, 40 + i)
        graphs.append((n, s, d, 1 + i % 3))
        s, d = erdos_renyi_gnm(n, 3 * n, 60 + i)
        graphs.append((n, s, d, 2))
    res, _ = htd.htd_truss_decompose_batched(graphs, flags=htd.HTD_OPT_BATCH_BLOCKS)
    for i, (n, s, d, h) in enumerate(graphs):
        assert torch.equal(htd.htd_truss_decompose(gpu_graph(htd, n, s, d), h)[0], res[i]), f"graph {i}"


def test_csr_rows_at_the_sort_edges(htd, oracle_mod):
    # rows of the lengths where the sort takes another form, with duplicates in both directions
    lengths = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 4095, 4096, 4097]
    n = 5000 + len(lengths)
    rng = np.random.default_rng(8)
    s = np.concatenate([np.full(k, 5000 + i) for i, k in enumerate(lengths)])
    d = np.concatenate([rng.choice(5000, size=k, replace=False) for k in lengths])
    dup = rng.random(s.size) < 0.02
    for extra in (0, 1):
        src = np.concatenate([s, d[dup]]) if extra else s
        dst = np.concatenate([d, s[dup]]) if extra else d
        g = gpu_graph(htd, n, src, dst)
        eu, ev = (host(t) for t in htd.htd_edges(g))
        eu_ref, ev_ref = oracle_mod.normalise(n, src, dst)
        np.testing.assert_array_equal(eu, eu_ref)
        np.testing.assert_array_equal(ev, ev_ref)
        row_ptr, col, slot_eid = (host(t) for t in htd.htd_csr(g))
        xs = np.repeat(np.arange(n), np.diff(row_ptr))
        np.testing.assert_array_equal(eu_ref[slot_eid], np.minimum(xs, col))
        np.testing.assert_array_equal(ev_ref[slot_eid], np.maximum(xs, col))
        assert all((np.diff(col[row_ptr[x]:row_ptr[x + 1]]) > 0).all() for x in range(n))


@pytest.mark.parametrize("h", [1, 2])
def test_window_of_many_levels(htd, h):
    # disjoint cliques of 4 to 12 vertices, 1,100 of each: a level has 6,600 to 72,600 edges, so
    # that the window of the cluster rounds (32,768 edges) holds one level, several or not one
    src, dst, ref, base = [], [], [], 0
    for size in range(4, 13):
        u, v = np.triu_indices(size, 1)
        off = base + size * np.arange(1100)[:, None]
        src.append((u + off).ravel())
        dst.append((v + off).ravel())
        ref.append(np.full(1100 * u.size, size))
        base += 1100 * size
    src, dst, ref = (np.concatenate(x) for x in (src, dst, ref))
    # other vertex ids, so that the levels are mixed in the scan
    perm = np.random.default_rng(9).permutation(base)
    a, b = np.minimum(perm[src], perm[dst]), np.maximum(perm[src], perm[dst])
    order = np.lexsort((b, a))
    g = gpu_graph(htd, base, a, b)
    t, _, st = htd.htd_truss_decompose(g, h)
    np.testing.assert_array_equal(host(t), ref[order])
    assert st["rounds"] == 9


def test_peels_join_a_long_one(htd):
    """A peel that begins alone has most of the room for clusters and makes room for the peels
    that start beside it: its launches hold fewer and fewer clusters, then more again."""
    long_case = (1 << 13, rmat(13, 8, 0.57, 0.19, 0.19, 6), 2)
    short = [(2000 + 100 * i, erdos_renyi_gnm(2000 + 100 * i, 8000, 70 + i), 2 + i % 2) for i in range(6)]

    def peel(case):
        n, (s, d), h = case
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            t, stamp, _ = htd.htd_truss_decompose(gpu_graph(htd, n, s, d), h, stamps=True)
            return host(t), host(stamp)

    ref = [peel(c) for c in [long_case] + short]
    out = {}
    done = threading.Event()

    def run_long():
        for _ in range(3):
            out[0] = peel(long_case)
        done.set()

    def run_short(i):
        while True:
            out[i] = peel(short[i - 1])
            if done.wait(0.002 * i):
                return

    threads = [threading.Thread(target=run_long)]
    threads += [threading.Thread(target=run_short, args=(i,)) for i in range(1, 7)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i, (t, stamp) in enumerate(ref):
        np.testing.assert_array_equal(out[i][0], t)
        np.testing.assert_array_equal(out[i][1], stamp)


@pytest.mark.parametrize("scale,factor,h", [(14, 60, 1), (13, 8, 2), (11, 8, 3)])
def test_rounds_that_no_helper_joins(htd, scale, factor, h):
    """Where helper clusters do not start (a busy device), rounds too large for one cluster go to
    the phase launches instead of running on its 16 SMs."""
    s, d = rmat(scale, factor, 0.57, 0.19, 0.19, 8)
    g = gpu_graph(htd, 1 << scale, s, d)
    t, stamp, st = htd.htd_truss_decompose(g, h, stamps=True)
    lib = htd._lib.load()
    lib.htd_test_no_helpers(1)
    try:
        t2, stamp2, st2 = htd.htd_truss_decompose(g, h, stamps=True)
    finally:
        lib.htd_test_no_helpers(0)
    assert torch.equal(t, t2) and torch.equal(stamp, stamp2)
    assert st2["rounds"] == st["rounds"]
    if h == 1:  # (rounds of up to a million update items)
        assert st2["kernel_launches"] > st["kernel_launches"] + 40


def test_clique_of_more_items_than_an_int_holds(htd):
    # all 12.5 M edges of a clique go in one round: 25 M edge sides of 157 detection items each are
    # 3.9e9 items, of which the list takes its 2^22
    n = 5000
    u, v = (torch.from_numpy(x.astype(np.int32)).cuda() for x in np.triu_indices(n, 1))
    g = htd.htd_build_csr(n, u, v)
    for flags in (0, htd.HTD_OPT_PERSISTENT_ROUNDS, htd.HTD_OPT_COMPACT_BALLS):
        t, _, st = htd.htd_truss_decompose(g, 2, flags=flags)
        assert bool((t == n).all()) and st["rounds"] == 1
    t, _, _ = htd.htd_truss_decompose(g, 3)
    assert bool((t == n).all())
    g.free()


def test_batches_of_a_round_move_on(htd):
    # a dense graph: one round has three times the detection items that a batch holds.  The sides
    # that fit a batch are its first ones, so that a handful of batches finish the round
    n = 3000
    s, d = erdos_renyi_gnm(n, 200000, 30)
    g = gpu_graph(htd, n, s, d)
    ref = None
    for flags in (0, htd.HTD_OPT_PERSISTENT_ROUNDS, htd.HTD_OPT_COMPACT_BALLS) * 4:
        t, stamp, st = htd.htd_truss_decompose(g, 2, stamps=True, flags=flags)
        assert st["slots"] < st["rounds"] + 20, flags
        ref = ref or (t, stamp)
        assert torch.equal(t, ref[0]) and torch.equal(stamp, ref[1])
