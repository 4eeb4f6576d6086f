"""A call whose device memory runs out at any one of its allocations either still gives the
right integers (it has another way) or fails with HTD_ENOMEM, and the next call on the same
handle gives the right ones."""

import ctypes

import numpy as np
import pytest

from synth import erdos_renyi_gnm, rmat

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

HTD_ENOMEM = 2


@pytest.fixture(scope="module")
def htd():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2411_06405_gb300 import build

    build.build()
    import paper_2411_06405_gb300 as mod

    lib = mod._lib.load()
    lib.htd_test_fail_alloc.argtypes = [ctypes.c_int64]
    lib.htd_test_fail_alloc.restype = ctypes.c_int64
    torch.cuda.set_device(0)
    return mod


# hubs: at h = 3 the h-support takes its balls from ORs of radius-2 rows
N, (SRC, DST) = 256, rmat(8, 8, 0.57, 0.19, 0.19, 31)


def build(htd):
    return htd.htd_build_csr(N, torch.from_numpy(SRC).cuda(), torch.from_numpy(DST).cuda())


def failing_each(htd, op, fresh):
    """Runs op(fresh()) with its k-th allocation failing, k = 1, 2, ... until all of its
    allocations succeed; yields (that run's result or None, the argument)."""
    lib = htd._lib.load()
    for k in range(1, 500):
        arg = fresh()
        lib.htd_test_fail_alloc(k)
        got = None
        try:
            got = op(arg)
        except htd._lib.HtdError as e:
            assert e.status == HTD_ENOMEM, f"allocation {k}: {e}"
        finally:
            left = lib.htd_test_fail_alloc(0)
        if left > 0:
            assert k > 1  # the hook was reached
            return
        yield got, arg
    raise AssertionError("more than 500 allocations")


@pytest.mark.parametrize("h", [1, 2, 3, 4])
def test_support(htd, oracle_mod, h):
    og = oracle_mod.OracleGraph.from_raw(N, SRC, DST)
    sup, truss = og.h_support(h), og.truss_decompose(h)[0]
    for got, g in failing_each(htd, lambda g: htd.htd_h_support(g, h), lambda: build(htd)):
        if got is not None:
            np.testing.assert_array_equal(got.cpu().numpy(), sup)
        np.testing.assert_array_equal(htd.htd_h_support(g, h).cpu().numpy(), sup)
        np.testing.assert_array_equal(htd.htd_truss_decompose(g, h)[0].cpu().numpy(), truss)
        g.free()


@pytest.mark.parametrize("h", [1, 2, 3, 4])
def test_decompose(htd, oracle_mod, h):
    og = oracle_mod.OracleGraph.from_raw(N, SRC, DST)
    sup, truss = og.h_support(h), og.truss_decompose(h)[0]
    for got, g in failing_each(htd, lambda g: htd.htd_truss_decompose(g, h)[0], lambda: build(htd)):
        if got is not None:
            np.testing.assert_array_equal(got.cpu().numpy(), truss)
        np.testing.assert_array_equal(htd.htd_truss_decompose(g, h)[0].cpu().numpy(), truss)
        np.testing.assert_array_equal(htd.htd_h_support(g, h).cpu().numpy(), sup)
        g.free()


def test_hindex(htd, oracle_mod):
    truss = oracle_mod.OracleGraph.from_raw(N, SRC, DST).truss_decompose(3)[0]
    run = lambda g: htd.htd_hindex_decompose(g, 3, prune=True)[0]
    for got, g in failing_each(htd, run, lambda: build(htd)):
        if got is not None:
            np.testing.assert_array_equal(got.cpu().numpy(), truss)
        np.testing.assert_array_equal(run(g).cpu().numpy(), truss)
        g.free()


@pytest.mark.parametrize("blocks", [False, True])
def test_batch(htd, blocks):
    graphs = [(120, *erdos_renyi_gnm(120, 400, 21), 2), (128, *rmat(7, 6, 0.57, 0.19, 0.19, 22), 2)]
    flags = htd.HTD_OPT_BATCH_BLOCKS if blocks else 0
    ref = htd.htd_truss_decompose_batched(graphs, flags=flags)[0]
    run = lambda b: htd.htd_truss_decompose_batched(b, flags=flags)[0]
    for got, b in failing_each(htd, run, lambda: htd.BatchInput(graphs)):
        for res in ([got] if got is not None else []) + [run(b)]:
            assert all(torch.equal(x, y) for x, y in zip(res, ref))


def test_build(htd):
    ref = [t.clone() for t in htd.htd_csr(build(htd))]
    for got, _ in failing_each(htd, lambda _: build(htd), lambda: None):
        for g in ([got] if got is not None else []) + [build(htd)]:
            assert all(torch.equal(x, y) for x, y in zip(htd.htd_csr(g), ref))


def test_failure_is_reported_once(htd):
    # the error of a failed allocation stays out of the next call's launch checks
    lib = htd._lib.load()
    g = build(htd)
    for _ in range(3):
        lib.htd_test_fail_alloc(1)
        with pytest.raises(htd._lib.HtdError):
            build(htd)
        assert lib.htd_test_fail_alloc(0) == 0
        htd.htd_h_support(g, 2)
        build(htd)
