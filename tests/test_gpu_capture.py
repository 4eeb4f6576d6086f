"""Calls whose stream is being captured into a CUDA graph are refused with HTD_ECUDA before they
touch the capture or the handle: the capture goes on, and the handle works afterwards."""

import gc

import numpy as np
import pytest

from synth import erdos_renyi_gnm

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

HTD_ECUDA = 3


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


def status_of(call):
    try:
        call()
    except Exception as e:
        return e.status  # not the exception: its frames would keep a test's graph alive
    return 0


@pytest.mark.parametrize("h", [1, 2, 3, 4])
def test_refused_under_capture(htd, oracle_mod, h):
    n = 200
    s, d = erdos_renyi_gnm(n, 700, 5)
    og = oracle_mod.OracleGraph.from_raw(n, s, d)
    sup, truss = og.h_support(h), og.truss_decompose(h)[0]
    src, dst = torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()
    # freed handles leave pooled memory and a pinned status block for the next one
    warm = htd.htd_build_csr(n, src, dst)
    htd.htd_truss_decompose(warm, h)
    warm.free()
    g = htd.htd_build_csr(n, src, dst)
    batch = htd.BatchInput([(n, s, d, h)])
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    calls = (lambda: htd.htd_build_csr(n, src, dst), lambda: htd.htd_edges(g), lambda: htd.htd_csr(g),
             lambda: htd.htd_h_support(g, h), lambda: htd.htd_truss_decompose(g, h),
             lambda: htd.htd_hindex_decompose(g, h), lambda: htd.htd_truss_decompose_batched(batch))
    # a collection during the capture could end an earlier CUDAGraph, which ends the capture
    gc.collect()
    gc.disable()
    try:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            got = [status_of(call) for call in calls]
            x += 1
    finally:
        gc.enable()
    assert got == [HTD_ECUDA] * len(calls)
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 1).all()
    np.testing.assert_array_equal(htd.htd_truss_decompose(g, h)[0].cpu().numpy(), truss)
    np.testing.assert_array_equal(htd.htd_h_support(g, h).cpu().numpy(), sup)
    res, _ = htd.htd_truss_decompose_batched(batch)
    np.testing.assert_array_equal(res[0].cpu().numpy(), truss)
