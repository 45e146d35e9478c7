"""The FP64 product from 56-bit digits (tc_slice.cu) over the forms zgemm takes: strides, orders,
conjugation, factors, batches with a shared operand, operand chunks, graded, zero, extreme and
non-finite rows, and a stream under capture. Every element is compared with the exact sum
(error-free products and math.fsum) within the bound of the method:

with 2^Ea, 2^Eb the powers of two above the largest component of the element's row of A and
column of B, and Sa, Sb the sums of their components' magnitudes over the inner index,
* operand rounding to 56 bits: 2^-57 (2^Ea Sb + 2^Eb Sa) (and their product, 1% covers it);
* dropped digit classes: digits are at most 64 in magnitude after the first, class c = i + j
  weighs 2^(-7 c), so the classes 10..16 hold at most 7/4 2^-56 (1 + 1/128 ...) < 1.8 2^-56 of
  2^(Ea + Eb) for each of the 2 K real terms of a component;
* rounding of the result, the factors, and of partial sums where the inner index is split:
  2^-51 (|alpha| sum|A||B| + |beta C|).
"""
import math

import numpy as np
import pytest

from synthetic import make_problem, random_vectors

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


# ---------------------------------------------------------------- the exact product
def _split(x):
    c = 134217729.0 * x  # 2^27 + 1
    hi = c - (c - x)
    return hi, x - hi


def _terms(a, b):
    """a b as the unevaluated sums p + e, exactly (a [M][1][K], b [1][N][K])."""
    p = a * b
    (ah, al), (bh, bl) = _split(a), _split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def exact(A, B):
    """A [M][K] times B [K][N]: the components' exact sums rounded once."""
    ar, ai = A.real[:, None, :], A.imag[:, None, :]
    br, bi = B.real.T[None], B.imag.T[None]
    out = np.empty((A.shape[0], B.shape[1]), np.complex128)
    re = np.concatenate(_terms(ar, br) + _terms(-ai, bi), axis=2)
    im = np.concatenate(_terms(ar, bi) + _terms(ai, br), axis=2)
    for m in range(out.shape[0]):
        for n in range(out.shape[1]):
            out[m, n] = complex(math.fsum(re[m, n].tolist()), math.fsum(im[m, n].tolist()))
    return out


def _mag(x):
    return np.abs(x.real) + np.abs(x.imag)


def bound(A, B, alpha, beta, C0):
    """Largest error of a component of alpha A B + beta C0."""
    top = lambda x, ax: np.ldexp(1.0, np.frexp(np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis=ax))[1])
    ea, eb = top(A, 1)[:, None], top(B, 0)[None, :]
    sa, sb = _mag(A).sum(axis=1)[:, None], _mag(B).sum(axis=0)[None, :]
    t = 1.01 * 2.0 ** -57 * (ea * sb + eb * sa) + 1.8 * 2.0 ** -56 * 2 * A.shape[1] * (ea * eb)
    fa = abs(complex(alpha).real) + abs(complex(alpha).imag)
    fb = abs(complex(beta).real) + abs(complex(beta).imag)
    return fa * t + 2.0 ** -51 * (fa * (_mag(A) @ _mag(B)) + fb * _mag(C0)) + 5e-324


def check(gpu, A, B, order_a="k", order_b="n", pad=0, conjA=False, conjB=False, alpha=1.0, beta=0.0, order_c="n",
          share=None, batch=1, seed=0):
    """One product of A [batch][M][K] and B [batch][K][N] (share: 'A' or 'B' used by the whole batch)
    laid out with the named index contiguous and rows padded, against the exact one."""
    rng = np.random.default_rng(seed)
    M, K, N = A.shape[1], A.shape[2], B.shape[2]

    def lay(x, fast_last):
        nb, r, c = x.shape
        inner, outer = (c, r) if fast_last else (r, c)
        ld = inner + pad
        flat = np.full(nb * outer * ld, np.nan + 0j)  # padding is never read
        v = flat.reshape(nb, outer, ld)
        v[:, :, :inner] = x if fast_last else x.transpose(0, 2, 1)
        return flat, ((outer * ld,) + ((ld, 1) if fast_last else (1, ld))), v

    a, sA, _ = lay(A, order_a == "k")
    b, sB, _ = lay(B, order_b == "n")
    C0 = rng.standard_normal((batch, M, N)) + 1j * rng.standard_normal((batch, M, N))
    c, sC, _ = lay(C0, order_c == "n")
    if share == "A":
        sA = (0,) + sA[1:]
    if share == "B":
        sB = (0,) + sB[1:]
    got = gpu.diag_zgemm(1, (M, N, K, batch), a, sA, b, sB, c, sC, alpha, beta, conjA, conjB)
    outer, inner = (M, N) if order_c == "n" else (N, M)
    g = got.reshape(batch, outer, inner + pad)
    assert np.isnan(g[:, :, inner:].real).all()  # nor written
    g = g[:, :, :inner] if order_c == "n" else g[:, :, :inner].transpose(0, 2, 1)
    worst = 0.0
    for z in range(batch):
        x = A[0 if share == "A" else z]
        y = B[0 if share == "B" else z]
        x, y = (x.conj() if conjA else x), (y.conj() if conjB else y)
        want = alpha * exact(x, y) + beta * C0[z]
        tol = bound(x, y, alpha, beta, C0[z])
        err = np.maximum(np.abs((g[z] - want).real), np.abs((g[z] - want).imag))
        assert (err <= tol).all(), float((err / tol).max())
        worst = max(worst, float((err / tol).max()))
    return worst


def _ops(M, N, K, batch=1, seed=1):
    rng = np.random.default_rng(seed)
    gauss = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    return gauss(batch, M, K), gauss(batch, K, N)


@pytest.mark.parametrize("M,N", [(33, 7), (7, 33), (130, 3)])  # the larger side becomes the row operand
@pytest.mark.parametrize("order_a,order_b,order_c", [("k", "n", "n"), ("m", "n", "n"), ("k", "k", "m"), ("m", "k", "n")])
@pytest.mark.parametrize("conjA,conjB", [(False, False), (True, False), (False, True)])
def test_orders_and_conjugation(gpu, M, N, order_a, order_b, order_c, conjA, conjB):
    A, B = _ops(M, N, 70)
    check(gpu, A, B, order_a, order_b, 3, conjA, conjB, order_c=order_c)


@pytest.mark.parametrize("alpha,beta", [(0.7, 0.0), (1.0, 1.0), (-0.3, 0.4), (0.2 + 0.9j, 0.0), (1.0, 0.5 - 2j),
                                        (1j, -1.0), (0.0, 1.0)])
@pytest.mark.parametrize("M,N", [(20, 9), (9, 40)])
def test_factors(gpu, M, N, alpha, beta):
    A, B = _ops(M, N, 65)
    check(gpu, A, B, alpha=alpha, beta=beta, pad=1)


@pytest.mark.parametrize("share", [None, "A", "B"])
@pytest.mark.parametrize("M,N", [(17, 5), (5, 17)])
def test_batches(gpu, M, N, share):
    A, B = _ops(M, N, 66, batch=4)
    check(gpu, A, B, order_a="m", share=share, batch=4, alpha=0.5, beta=0.25j, conjB=True)


@pytest.mark.parametrize("M,N,K,share,batch", [(150, 5, 600, None, 1), (140, 3, 1100, "A", 3), (5, 150, 70, None, 1)])
def test_operand_chunks(gpu, M, N, K, share, batch):
    """A cap of one row tile and 512 inner elements: rows, columns and the inner index in chunks."""
    A, B = _ops(M, N, K, batch)
    assert gpu.lib.adc_diag_set_sliced_cap(1 << 16) == 0
    try:
        check(gpu, A, B, share=share, batch=batch, beta=0.5)
    finally:
        gpu.lib.adc_diag_set_sliced_cap(0)


def test_few_rows_are_one_chunk(gpu):
    """Operands of less than a row tile whose memory there is room for: sliced and multiplied at once
    (two launches per operand, the product, and the sum of its inner splits)."""
    A, B = _ops(20, 10, 5000)
    n0 = gpu.launch_count()
    gpu.diag_zgemm(1, (20, 10, 5000, 1), A.ravel(), (0, 5000, 1), B.ravel(), (0, 10, 1), np.zeros(200), (0, 10, 1))
    assert gpu.launch_count() - n0 <= 6


@pytest.mark.parametrize("what", ["spikes", "tails", "opposed", "zero rows", "huge and tiny", "subnormal", "one term"])
@pytest.mark.parametrize("M,N,K", [(31, 9, 80), (9, 31, 80)])
@pytest.mark.parametrize("order", ["k", "m"])
def test_graded_rows(gpu, M, N, K, what, order):
    """Rows whose elements differ by many orders of magnitude, maxima at different inner indices."""
    A, B = _ops(M, N, K)
    if what == "spikes":
        for m in range(M):
            A[0, m, (5 * m) % K] *= 10.0 ** (m % 13)
        for n in range(N):
            B[0, (7 * n + 3) % K, n] *= 10.0 ** (n % 11)
    elif what == "tails":
        A[0, :, 1:] *= 1e-9
        B[0, :-1, :] *= 1e-9
    elif what == "opposed":
        g = 10.0 ** -np.linspace(0.0, 14.0, K)
        A, B = A * g, B * g[::-1, None]
    elif what == "zero rows":
        A[0, ::3] = 0.0
        B[0, :, 1::4] = 0.0
    elif what == "huge and tiny":
        A *= 1e290
        B *= 1e-300
    elif what == "subnormal":
        A = np.ldexp(A.real, -1050) + 1j * np.ldexp(A.imag, -1050)
        B = B * 2.0 ** 900
    else:
        A[0, :, 1:] = 0.0
    check(gpu, A, B, order_a=order, order_b="k" if order == "k" else "n")


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_rows(gpu, bad):
    """A row (column) with an infinity or a NaN gives a row (column) that is not finite, as on the
    FP64 units, and leaves the others as they are."""
    A, B = _ops(20, 12, 70)
    A[0, 4, 11] = bad
    B[0, 30, 7] = complex(0.0, bad)
    size, sA, sB, sC = (20, 12, 70, 1), (0, 70, 1), (0, 12, 1), (0, 12, 1)
    out = [gpu.diag_zgemm(d, size, A.ravel(), sA, B.ravel(), sB, np.zeros(240), sC).reshape(20, 12) for d in (0, 1)]
    fin = [np.isfinite(o.real) & np.isfinite(o.imag) for o in out]
    assert not fin[1][4].any() and not fin[1][:, 7].any()
    assert np.array_equal(fin[0], fin[1])
    rows, cols = np.arange(20) != 4, np.arange(12) != 7
    a, b = A[:, rows], B[:, :, cols]
    want, tol = exact(a[0], b[0]), bound(a[0], b[0], 1.0, 0.0, np.zeros((19, 11), complex))
    assert (np.abs(out[1][np.ix_(rows, cols)] - want) <= 2 * tol).all()


def test_under_capture(gpu):
    """An FP64 product large enough for digits, captured on the context's stream: it runs on the FP64
    units there, and the replayed graph gives the direct product's result (56 bits or FP64 sums: 1e-13
    of the largest output)."""
    p = make_problem(12, 40, 60, seed=61, sigma=0.08)
    s = torch.cuda.Stream()
    B, eo, ev = (torch.from_numpy(v).cuda() for v in (p.B, p.eps_occ, p.eps_vir))
    torch.cuda.synchronize()
    with gpu.Context(B, eo, ev, kind="EA", order=3, x=0.5, stream=s.cuda_stream) as ctx:
        X = torch.from_numpy(random_vectors(ctx.N, 32, seed=62)).cuda()
        S = torch.empty_like(X)
        torch.cuda.synchronize()
        want = ctx.sigma(X, "fp64")
        ctx.sync()
        assert ctx.kept_digits()["own"] > 0
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.sigma(X, "fp64", out=S)
        S.zero_()
        torch.cuda.synchronize()
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        assert (S - want).abs().max() < 1e-13 * want.abs().max()
        X2 = ctx.sigma(X, "fp64")
        ctx.sync()
        assert torch.equal(X2, want)
        del g
