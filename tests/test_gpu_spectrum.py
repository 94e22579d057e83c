"""The corner spectrum (reduction to tridiagonal form, bisection, sort) on its own: ctm_set_env computes
it for any corner, real (one CTA up to chi = 96, a thread-block cluster beyond) and Hermitian (one CTA up
to chi = 112, the cluster on the real embedding beyond), against numpy's eigenvalues.

Tolerance: both sides are backward stable, so an eigenvalue of a corner of unit norm is off by a small
multiple of chi u (u = 2^-53); 8 chi u covers both, plus the bisection's final bracket of 4e-16."""
import numpy as np
import pytest

from paper_2509_05090_gb300 import inputs as I

pytestmark = pytest.mark.gpu

KINDS = ("random", "diagonal", "identity", "graded", "pairs", "rank_one", "arrow")


def _corner(chi, kind, cplx, rng):
    R = rng.standard_normal((chi, chi))
    if cplx:
        R = R + 1j * rng.standard_normal((chi, chi))
    H = R + R.conj().T
    if kind == "random":
        return H
    if kind == "diagonal":
        return np.diag(np.sort(rng.uniform(-1, 1, chi))[::-1]).astype(H.dtype)
    if kind == "identity":
        return np.eye(chi, dtype=H.dtype)
    if kind == "graded":      # a converged near-product corner: magnitudes over twelve decades
        g = 10.0 ** (-12.0 * np.arange(chi) / max(1, chi - 1))
        return H * g[:, None] * g[None, :]
    if kind == "pairs":       # nearly degenerate pairs of both signs
        Q = np.linalg.qr(R)[0]
        w = np.repeat(rng.uniform(-1, 1, (chi + 1) // 2), 2)[:chi]
        w[1::2] += 1e-13
        return (Q * w) @ Q.conj().T
    if kind == "rank_one":
        return np.outer(R[0], R[0].conj())
    A = np.diag(np.arange(1.0, chi + 1)).astype(H.dtype)   # arrow: the first column already reduced but one entry
    A[0, 1:2] = A[1:2, 0] = 0.5
    return A


def _expected(C):
    w = np.sort(np.abs(np.linalg.eigvalsh(0.5 * (C + C.conj().T))))[::-1]
    return w / np.linalg.norm(w)


@pytest.mark.parametrize("chi", [1, 2, 3, 4, 5, 9, 31, 32, 33, 65, 72, 73, 96, 97, 98, 128, 130, 161, 257, 512])
def test_real_corner_spectrum(ctm_lib, chi):
    from paper_2509_05090_gb300 import binding
    rng = np.random.default_rng(chi)
    g = binding.CTM(I.random_site_tensor(2, 1, 3), chi)
    C0, T, Q = (x.cpu().numpy() for x in g.ctm_get_env())
    for kind in KINDS:
        C = _corner(chi, kind, False, rng)
        g.ctm_set_env(C / np.linalg.norm(C), T, Q)
        s = g.ctm_get_intermediate("s").cpu().numpy()
        assert np.max(np.abs(s - _expected(C))) <= 8 * chi * 2.0 ** -53 + 4e-16, kind
    g.close()


@pytest.mark.parametrize("chi", [1, 2, 3, 5, 9, 32, 33, 72, 111, 112, 113])
def test_hermitian_corner_spectrum(ctm_lib, chi):
    from paper_2509_05090_gb300 import binding
    rng = np.random.default_rng(chi)
    A = I.random_complex_site_tensor(2, 1, 3)
    g = binding.CTMComplex(A, chi, irrep="E")
    C0, T, Q = (x.cpu().numpy() for x in g.ctm_complex_get_env())
    for kind in KINDS:
        C = _corner(chi, kind, True, rng)
        g.ctm_complex_set_env(C / np.linalg.norm(C), T, Q)
        s = g.ctm_complex_get_intermediate("s").cpu().numpy()
        assert np.max(np.abs(s - _expected(C))) <= 8 * chi * 2.0 ** -53 + 4e-16, kind
    g.close()
