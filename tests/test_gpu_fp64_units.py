"""opts.fp64_units: every FP64 contraction by multiply-adds, whatever its size.

Element-wise bound of a product on the FP64 units: three real multiply-add chains of K terms
(T1 = sum ar br, T2 = sum ai bi, T3 = sum (ar + ai)(br + bi)) and four roundings, so at most
(K + 8) 2^-52 sum (|ar| + |ai|)(|br| + |bi|) per component, whatever the row and column maxima.
Whole results of both routes agree to 1e-13 of the largest element (56 bits or FP64 sums).
"""
import numpy as np
import pytest

from synthetic import make_problem
from test_gpu_digit_forms import _mag, _ops, exact

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from conftest import build_library
    build_library()
    import paper_2511_21640_gb300 as m
    return m


def _close(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return np.abs(a - b).max() <= 1e-13 * np.abs(b).max()


def _digits(stats):
    return [k for k in stats if k.startswith(("tc_digits", "sl_pack"))]


def test_graded_operands_keep_their_digits(gpu):
    """Large elements of the rows against small ones of the columns: every element of the product is
    small against the row and column maxima, and right to the FP64 units' own bound; from digits it
    is right to 56 bits of those maxima only."""
    M, N, K = 24, 10, 90
    A, B = _ops(M, N, K, seed=3)
    g = 10.0 ** -np.linspace(0.0, 12.0, K)
    A, B = (A * g)[0], (B * g[::-1, None])[0]
    want = exact(A, B)
    out = [gpu.diag_zgemm(d, (M, N, K, 1), A.ravel(), (0, K, 1), B.ravel(), (0, N, 1), np.zeros(M * N),
                          (0, N, 1)).reshape(M, N) for d in (0, 1)]
    err = [np.maximum(np.abs((o - want).real), np.abs((o - want).imag)) for o in out]
    assert (err[0] <= (K + 8) * 2.0 ** -52 * (_mag(A) @ _mag(B))).all()
    top = np.abs(A).max(axis=1)[:, None] * np.abs(B).max(axis=0)[None, :]
    assert (err[1] <= 2.0 ** -51 * K * top).all()


@pytest.mark.parametrize("kind,nocc,nvir", [("EA", 12, 40), ("IP", 36, 20), ("EE", 6, 30)])
def test_every_contraction_stays_on_the_units(gpu, kind, nocc, nvir):
    p = make_problem(nocc, nvir, 60, seed=71, sigma=0.08)

    def run(units):
        with gpu.Context(p.B, p.eps_occ, p.eps_vir, kind=kind, order=3, x=0.5, profile=True, fp64_units=units) as c:
            setup = _digits(c.profile_read())
            c.profile(True)
            rng = np.random.default_rng(72)
            X = rng.standard_normal((32, c.N)) + 1j * rng.standard_normal((32, c.N))
            S = c.sigma(X, "fp64")
            g = c.sigma_adjoint(X[:2], np.array([1.0, -0.5]))
            ran = _digits(c.profile_read())
            return setup, ran, c.kept_digits()["own"], S, c.diagonal(), g[0]

    with_digits, units = run(False), run(True)
    assert with_digits[0] and with_digits[1]
    assert not units[0] and not units[1] and units[2] == 0
    for a, b in zip(with_digits[3:], units[3:]):
        assert _close(a, b)


def test_solves_and_batches_take_the_option(gpu):
    probs = [make_problem(6, 20, 30, seed=73 + i, sigma=0.08) for i in range(2)]
    for q in probs:
        q.kind, q.order, q.x = "EA", 3, 0.5
    om = [gpu.batch_solve(probs, 2, tol=1e-8, precision="fp64", fp64_units=u)[0] for u in (False, True)]
    assert np.abs(om[0] - om[1]).max() < 1e-9
    q = probs[0]
    r = [gpu.ssfns(q.B, q.eps_occ, q.eps_vir, kind="EA", nroots=1, tol=1e-8, fp64_units=u)[0]["omega_corrected"]
         for u in (False, True)]
    assert abs(r[0] - r[1]) < 1e-9


def test_other_values_are_refused(gpu):
    p = make_problem(4, 6, 8, seed=1)
    o = gpu.adc_opts()
    gpu.lib.adc_opts_default(gpu.ctypes.byref(o))
    assert o.fp64_units == 0
    o.fp64_units = 2
    h = gpu.ctypes.c_void_p()
    rc = gpu.lib.adc_init(gpu.ctypes.byref(h), p.B.ctypes.data, 8, p.eps_occ.ctypes.data, 4, p.eps_vir.ctypes.data, 6,
                          0, 3, 1.0, gpu.ctypes.byref(o))
    assert rc == -1 and not h.value
