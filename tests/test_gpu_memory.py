"""Device memory the library holds: what it keeps between handles can be given back."""

import numpy as np
import pytest

from synth import erdos_renyi_gnm

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
