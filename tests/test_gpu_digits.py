"""The digit products on the tensor cores (tc_slice.cu) at the edges of their tiles.

Seeded uniform operands against the FP64 units (``adc_diag_gemm``): 5 the
sliced product (42 bits), 6 the setup's (48 bits, digits whose width follows
the inner size), 7 the FP64 product (56 bits).

Tolerances, relative to the Frobenius norm. Rounding an operand to `bits` bits
below its row maximum leaves an error uniform in +-2^(-bits-1), that is
2^(-bits) of the operands' RMS for uniform values (max = sqrt(3) RMS), sqrt(2)
of that for both operands; the dropped digit classes add less than as much
again: 2^(1.5 - bits), and a factor of two in hand. The FP64 reference
(three products per complex multiply-add) carries at most 2^-50 sqrt(K) of its own.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BITS = {5: 42, 6: 48, 7: 56}


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from conftest import build_library
    build_library()
    import paper_2511_21640_gb300 as m
    return m


# tile widths 32, 64 and 128 real columns with one column more and less; row
# tiles of 128; inner sizes around a block of 64, around the exact runs of both
# passes, split over the SMs, and (48 bits) of every digit width
@pytest.mark.parametrize("M,N,K", [
    (1, 1, 1), (127, 16, 63), (128, 17, 64), (129, 32, 65), (257, 33, 193), (130, 64, 320), (128, 65, 384),
    (300, 129, 385), (64, 5, 30000), (1100, 140, 700), (90, 70, 2100), (40, 33, 9000),
    # the FP64 units' tiles (strips of 4 and 8 rows or columns, 8, 16, 32 and 64 square), whole and split
    (3, 300, 50), (300, 3, 50), (7, 90, 1000), (90, 7, 1000), (9, 9, 20), (20, 20, 400), (70, 50, 40), (700, 650, 33)])
@pytest.mark.parametrize("which", [5, 6, 7])
def test_digit_product_edges(gpu, which, M, N, K):
    err, _ = gpu.diag_gemm(which, M, N, K, seed=3 + M, reps=1)
    assert err < 2.0 ** (2.5 - BITS[which]) + 2.0 ** -50 * math.sqrt(K), err


@pytest.mark.parametrize("which,M,N,K", [(2, 6000, 1300, 3300), (3, 6000, 1300, 3300)])
def test_wide_grouped_launch(gpu, which, M, N, K):
    """A grouped BF16x3 launch large enough for the wide loop, one job and three (one of them
    narrow, its inner sums split inside a block's three products). Each operand keeps 16 bits
    (2^-17 relative, 2^-16.5 for both) and the FP32 sums of K random terms lose at most 2^-24
    sqrt(2 K) of the largest: 2^-14 covers both."""
    err, _ = gpu.diag_gemm(which, M, N, K, seed=21, reps=1)
    assert err < 2.0 ** -14, err


@pytest.mark.parametrize("kind,nocc,nvir", [("EA", 12, 40), ("IP", 36, 20)])
def test_kept_digits_go_back_when_memory_runs_short(gpu, kind, nocc, nvir):
    """A memory limit that fits a long block of FP64 products only without the digits kept by an
    earlier one: the block runs, and equals the unlimited context's to the rounding of either
    route (56 bits or FP64 sums of K terms: 1e-13 of the largest output)."""
    from synthetic import make_problem
    p = make_problem(nocc=nocc, nvir=nvir, naux=60, seed=5)
    rng = np.random.default_rng(6)

    def context(limit):
        return gpu.Context(p.B, p.eps_occ, p.eps_vir, kind=kind, order=3, x=0.5, mem_limit=limit)

    with context(0) as c:
        X = rng.standard_normal((1500, c.N)) + 1j * rng.standard_normal((1500, c.N))
        held = c.memory()["in_use"]
        c.sigma(X[:32], "fp64")
        kept = c.memory()["in_use"] - held
        setup_peak = c.memory()["peak"]
        want = c.sigma(X, "fp64")
        peak = c.memory()["peak"]
    assert kept > 0 and peak > setup_peak
    limit = max(peak - kept // 4, setup_peak)
    with context(limit) as c:
        c.sigma(X[:32], "fp64")
        got = c.sigma(X, "fp64")
        assert c.memory()["peak"] <= limit
    assert np.abs(got - want).max() < 1e-13 * np.abs(want).max()
