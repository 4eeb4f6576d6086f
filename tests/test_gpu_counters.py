"""The counters of htd_stats agree with what the calls did."""

import numpy as np
import pytest

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


def test_update_bytes_of_batches_with_many_items(htd):
    # 30 M edges at 200,000 vertices, h = 1: batches of up to 36 M update items.  Every removed
    # edge brings an item per 32 slots of both its endpoints' rows; an item counts 144 bytes, a
    # test 4 more and one that lowers a support 8 more
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    n, m = 200000, 30_000_000
    src, dst = (torch.randint(0, n, (m,), generator=gen, device="cuda", dtype=torch.int32) for _ in range(2))
    g = htd.htd_build_csr(n, src, dst)
    deg = np.diff(htd.htd_csr(g)[0].cpu().numpy().astype(np.int64))
    _, _, st = htd.htd_truss_decompose(g, 1)
    g.free()
    least = 144 * int((deg * ((deg + 31) // 32)).sum()) + 4 * st["member_tests"]
    assert least <= st["alg_bytes_update"] <= least + 8 * st["member_tests"]


def test_detection_bytes_of_a_clique(htd):
    # h = 1, compact balls: a removed edge is one pair, and its one look-up reads two words of
    # metadata and, in a clique's dense ball, one of the ball
    n = 40
    u, v = np.triu_indices(n, 1)
    g = htd.htd_build_csr(n, u.astype(np.int32), v.astype(np.int32))
    _, _, st = htd.htd_truss_decompose(g, 1, flags=htd.HTD_OPT_COMPACT_BALLS)
    assert st["pairs_tested"] == g.m
    assert st["alg_bytes_detect"] == 12 * g.m


@pytest.mark.parametrize("n,ors", [(257, True), (20000, False)])
def test_ball_bytes_at_radius_3(htd, n, ors):
    # cycles: radius 3 by ORs of radius-2 rows on the short one (three rows of 9 words a
    # vertex), by search on the long one (five vertices within two hops, 8 bytes and two slots
    # each).  All edges go in one round; where that is finished by rebuilds, each ball is built
    # once more, of a vertex without edges (8 bytes)
    x = np.arange(n, dtype=np.int32)
    g = htd.htd_build_csr(n, x, ((x + 1) % n).astype(np.int32))
    _, _, st = htd.htd_truss_decompose(g, 3)
    assert st["rounds"] == 1
    assert st["alg_bytes_ball"] == n * ((3 * 4 * 9 if ors else 5 * 16) + 8 * st["rounds_rebuilt"])


def test_rounds_of_many_batches_are_left_to_the_phase_launches(htd):
    # 128-slot tables: nearly every round takes a dozen batches.  A batch is four launches; the
    # cluster round kernel before each of them would be a fifth that has nothing to do
    from synth import erdos_renyi_gnm

    n = 2000
    s, d = erdos_renyi_gnm(n, 8000, 3)
    g = htd.htd_build_csr(n, s.astype(np.int32), d.astype(np.int32))
    t, stamp, _ = htd.htd_truss_decompose(g, 2, stamps=True)
    t2, stamp2, st = htd.htd_truss_decompose(g, 2, stamps=True, flags=htd.HTD_OPT_TINY_LOSS_TABLE)
    assert torch.equal(t, t2) and torch.equal(stamp, stamp2)
    assert st["slots"] > 5 * st["rounds"]
    assert st["kernel_launches"] < 4.4 * st["slots"]
