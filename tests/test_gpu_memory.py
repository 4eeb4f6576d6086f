"""Device memory the library holds: what it keeps between handles can be given back."""

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


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_is_given_back(htd):
    n = 20000
    s, d = erdos_renyi_gnm(n, 80000, 3)
    src, dst = torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()

    def peel():
        g = htd.htd_build_csr(n, src, dst)
        t = htd.htd_truss_decompose(g, 2)[0].cpu().numpy()
        g.free()
        return t

    ref = peel()
    htd.htd_trim_memory()
    before = free_bytes()
    np.testing.assert_array_equal(peel(), ref)  # (on the host: PyTorch's kernels take memory at first use)
    kept = before - free_bytes()
    assert 0 < kept <= 600 << 20
    live = htd.htd_build_csr(n, src, dst)
    htd.htd_trim_memory()
    np.testing.assert_array_equal(htd.htd_truss_decompose(live, 2)[0].cpu().numpy(), ref)
    live.free()
    htd.htd_trim_memory()
    assert free_bytes() >= before - (2 << 20)


@pytest.mark.parametrize("h", [1, 2, 3, 4])
def test_support_holds_what_its_balls_need(htd, h):
    # 512 vertices with edges among 368,641: n bits for every vertex would be 17 GB
    s, d = rmat(9, 6, 0.57, 0.19, 0.19, 21)
    small = htd.htd_build_csr(512, s, d)
    ref = htd.htd_h_support(small, h).cpu().numpy()
    big = htd.htd_build_csr(368641, s, d)
    before = free_bytes()
    for _ in range(2):
        np.testing.assert_array_equal(htd.htd_h_support(big, h).cpu().numpy(), ref)
        # (h >= 3: the level lists of the search, 2n int32 a resident block, are scratch too)
        assert before - free_bytes() < (256 << 20 if h < 3 else 5 << 30)
    big.free()


def test_support_gives_large_rows_back(htd):
    # a star of 12,000 leaves among 300,001 vertices, h = 3: its balls come from ORs of radius-2
    # rows of all vertices, 11 GB, more than stays with a handle
    n, k = 300001, 12000
    v = 25 * np.arange(k + 1)
    g = htd.htd_build_csr(n, np.zeros(k, np.int32), v[1:].astype(np.int32))
    before = free_bytes()
    for _ in range(2):
        sup = htd.htd_h_support(g, 3)
        held = before - free_bytes()
        assert (sup.cpu().numpy() == k - 1).all()
        assert held < 6 << 30
    hx = htd.htd_hindex_decompose(g, 3, max_iter=1)[0]
    assert hx.numel() == k
    assert before - free_bytes() < 6 << 30
    g.free()


@pytest.mark.parametrize("h", [1, 2, 3, 4])
@pytest.mark.parametrize("family", ["er", "rmat"])
def test_support_in_room_by_the_bound(htd, family, h):
    # n-bit sets of 32,768 vertices take 128 MiB: room for the balls comes from their bound, then
    # from what they took.  Compared with the entry point that needs no storage for balls
    n = 1 << 15
    s, d = erdos_renyi_gnm(n, 60000, 17) if family == "er" else rmat(15, 4, 0.57, 0.19, 0.19, 18)
    g = htd.htd_build_csr(n, s.astype(np.int32), d.astype(np.int32))
    row_ptr, col, _ = htd.htd_csr(g)
    eu, ev = htd.htd_edges(g)
    ref = htd.htd_h_support_static(n, row_ptr, col, eu, ev, h, torch.empty_like(eu))
    for _ in range(3):
        assert torch.equal(htd.htd_h_support(g, h), ref)
