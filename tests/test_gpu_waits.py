"""Waits between the clusters of a round kernel end by themselves: a peel whose wait runs out fails
with HTD_ETIMEOUT, whatever form its rounds take, and the handle works afterwards."""

import pytest

from synth import rmat

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

HTD_ETIMEOUT = 4


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


@pytest.mark.parametrize("scale,factor,h", [(14, 60, 1), (13, 8, 2), (11, 8, 3)])
def test_wait_that_runs_out(htd, scale, factor, h):
    s, d = rmat(scale, factor, 0.57, 0.19, 0.19, 8)
    g = htd.htd_build_csr(1 << scale, torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda())
    ref, stamp, _ = htd.htd_truss_decompose(g, h, stamps=True)
    lib = htd._lib.load()
    for _ in range(2):
        lib.htd_test_wait_polls(1)  # a helper gives up before the leader has a job for it
        try:
            with pytest.raises(htd.HtdError) as e:
                htd.htd_truss_decompose(g, h)
        finally:
            lib.htd_test_wait_polls(0)
        assert e.value.status == HTD_ETIMEOUT
        again, stamp2, _ = htd.htd_truss_decompose(g, h, stamps=True)
        assert torch.equal(again, ref) and torch.equal(stamp2, stamp)
