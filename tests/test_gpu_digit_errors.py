"""A tensor-core wait that gives up inside an FP64 product from digits: every call that waits for
the product reports ADC_ERR_TIMEOUT (-5), and none is left for a later call on the context.

The wait limit is lowered to 1 ns through the test hook, so a wait gives up long before the
copies and MMAs it waits for finish; the kernels drain what they have in flight and return
(as in test_gpu_parity.py for the split and sliced products). Results after it are compared
with those before it: the same products in the same order, 1e-14 of the norm.
"""
import contextlib

import numpy as np
import pytest

from synthetic import make_problem, random_vectors

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TIMEOUT = -5


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from conftest import build_library
    build_library()
    import paper_2511_21640_gb300 as m
    return m


@contextlib.contextmanager
def short_waits(gpu):
    assert gpu.lib.adc_diag_set_wait_ns(1) == 0
    try:
        yield
    finally:
        assert gpu.lib.adc_diag_set_wait_ns(0) == 0


def _context(gpu, kind="EA"):
    # large enough for the satellite ladder of 32 vectors to run from digits
    p = make_problem(*((12, 40, 60) if kind == "EA" else (36, 20, 60)), seed=61, sigma=0.08)
    return gpu.Context(p.B, p.eps_occ, p.eps_vir, kind=kind, order=3, x=0.5)


def _same(a, b):
    return np.linalg.norm(a - b) <= 1e-14 * np.linalg.norm(b)


@pytest.mark.parametrize("kind", ["EA", "IP"])
def test_sigma(gpu, kind):
    with _context(gpu, kind) as ctx:
        X = random_vectors(ctx.N, 32, seed=62)
        first = ctx.sigma(X, "fp64")
        with short_waits(gpu), pytest.raises(gpu.AdcError) as ei:
            ctx.sigma(X, "fp64")
        assert ei.value.code == TIMEOUT
        assert _same(ctx.sigma(X, "fp64"), first)


def test_batch_sigma(gpu):
    with _context(gpu) as a, _context(gpu, "IP") as b:
        X = [torch.from_numpy(random_vectors(c.N, 32, seed=63)).cuda() for c in (a, b)]
        with gpu.Batch([a, b]) as batch:
            first = [s.cpu().numpy() for s in batch.sigma(X, "fp64")]
            with short_waits(gpu), pytest.raises(gpu.AdcError) as ei:
                batch.sigma(X, "fp64")
            assert ei.value.code == TIMEOUT
            again = [s.cpu().numpy() for s in batch.sigma(X, "fp64")]
        for c, s, f, x in zip((a, b), again, first, X):
            assert _same(s, f)
            assert _same(c.sigma(x, "fp64").cpu().numpy(), f)


@pytest.mark.parametrize("batched", [False, True])
def test_davidson(gpu, batched):
    with _context(gpu) as ctx:
        X = random_vectors(ctx.N, 32, seed=64)
        first = ctx.sigma(X, "fp64")
        if batched:
            with gpu.Batch([ctx]) as batch, short_waits(gpu), pytest.raises(gpu.AdcError) as ei:
                batch.davidson(24, tol=1e-8, precision="fp64")
        else:
            with short_waits(gpu), pytest.raises(gpu.AdcError) as ei:
                ctx.davidson(24, tol=1e-8, precision="fp64")
        assert ei.value.code == TIMEOUT
        assert _same(ctx.sigma(X, "fp64"), first)


def test_a_later_failure_reports_it(gpu):
    """An asynchronous product (device operands) whose wait gave up, then a call that fails for
    another reason before it waits: that call reports the wait, and the next one succeeds."""
    with _context(gpu) as ctx:
        X = torch.from_numpy(random_vectors(ctx.N, 32, seed=65)).cuda()
        first = ctx.sigma(X, "fp64").cpu().numpy()
        S = torch.empty_like(X)
        with short_waits(gpu):
            assert gpu.lib.adc_sigma(ctx._h, X.data_ptr(), S.data_ptr(), 32, 0) == 0
            g = np.array([float("nan")])  # refused inside the call
            w = np.zeros(8)
            rc = gpu.lib.adc_sigma_adjoint(ctx._h, X.data_ptr(), g.ctypes.data, 1, S.data_ptr(), w.ctypes.data,
                                           w.ctypes.data, (gpu.ctypes.c_double * 1)())
            assert rc == TIMEOUT
        assert gpu.lib.adc_sigma(ctx._h, X.data_ptr(), S.data_ptr(), 32, 0) == 0
        assert gpu.lib.adc_sync(ctx._h) == 0
        assert _same(S.cpu().numpy(), first)
