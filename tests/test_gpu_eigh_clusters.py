"""The refined Hermitian eigensolver on spectra whose close eigenvalues form clusters of
every size that its exact cluster step takes (2 to 8), several at once and next to
separate eigenvalues, against LAPACK (numpy.linalg.eigh). Tolerance 1e-13 of the norm:
the solver accepts vectors orthonormal to 1e-13, and its FP64 products round to
n eps <= 1.5e-14."""

import numpy as np
import pytest

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


@pytest.mark.parametrize("gap", [0.0, 1e-12])
@pytest.mark.parametrize("sizes", [(2,), (3, 1), (4, 2, 1), (5, 7, 3), (6, 8, 1, 2), (8,) * 4, (8,) * 16, (2,) * 63])
def test_clusters_of_every_size(gpu, sizes, gap):
    n = sum(sizes)
    rng = np.random.default_rng(n)
    lam = np.concatenate([1.0 + 0.05 * k + gap * np.arange(s) for k, s in enumerate(sizes)])
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)) + 1j * rng.normal(size=(n, n)))
    A = (Q * lam) @ Q.conj().T
    A = 0.5 * (A + A.conj().T)
    w, V, _, steps = gpu.diag_eigh(1, A)
    nrm = np.abs(lam).max()
    assert steps >= 3, steps
    assert np.abs(w - np.linalg.eigvalsh(A)).max() < 1e-13 * nrm
    assert np.linalg.norm(A @ V - V * w, axis=0).max() < 1e-13 * nrm
    assert np.abs(V.conj().T @ V - np.eye(n)).max() < 1e-13
