"""The blocked Householder QR (csrc/qr.cu: one panel or 64-column panels, the rest as FP64 slices on the
tensor cores): Y = Q R of a step at panel edges, and with zero and dependent columns."""
import numpy as np
import pytest
import torch

from paper_2509_05090_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _check(g, chi):
    Y, Q, R = (g.ctm_get_intermediate(x) for x in ("Y", "Q", "R"))
    # k reflectors, each applied with a few roundings: k eps in the Frobenius norm, times 4
    tol = 4 * chi * 2.0 ** -53
    eye = torch.eye(chi, dtype=torch.float64, device=Y.device)
    assert float((Y - Q @ R).norm()) <= tol * float(Y.norm())
    assert float((Q.T @ Q - eye).norm()) <= tol * chi ** 0.5
    assert float(torch.tril(R, -1).abs().max()) == 0.0
    assert float(torch.diagonal(R).min()) >= 0.0


@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("D,chi", [(8, 97), (4, 200), (5, 193), (3, 256), (3, 257), (4, 321), (5, 320), (3, 512)])
def test_panels(ctm_lib, D, chi, deterministic):
    from paper_2509_05090_gb300 import binding
    g = binding.CTM(I.random_site_tensor(2, D, 50 + chi), chi, precision="split_bf16", n_split=3,
                    deterministic=deterministic)
    g.ctm_step(2)
    _check(g, chi)
    g.ctm_step(3)   # captured
    _check(g, chi)
    g.close()


@pytest.mark.parametrize("D,chi", [(3, 260), (5, 320)])
def test_zero_and_dependent_columns(ctm_lib, D, chi):
    from paper_2509_05090_gb300 import binding
    g = binding.CTM(I.random_site_tensor(2, D, 77), chi, precision="split_bf16", n_split=3)
    g.ctm_step(2)
    C, T, Q = g.ctm_get_env()
    for c in (0, 63, 64, 130, chi - 1):
        Q[:, c] = 0.0
    Q[:, 90] = Q[:, 89]
    Q[:, 200] = 3.0 * Q[:, 20]
    g.ctm_set_env(C, T, Q)
    g.ctm_step(1)
    _check(g, chi)
    assert np.isfinite(g.ctm_get_intermediate("R").cpu().numpy()).all()
    g.close()


def test_complex_embedding(ctm_lib):
    """The complex step's QR of the real 2n x 2chi embedding: Q stays an isometry."""
    from paper_2509_05090_gb300 import binding
    chi = 72
    g = binding.CTMComplex(I.random_complex_site_tensor(2, 6, 3), chi, precision="split_bf16", n_split=5)
    g.ctm_complex_step(3)
    Q = g.ctm_complex_get_env()[2].reshape(-1, chi)
    eye = torch.eye(chi, dtype=Q.dtype, device=Q.device)
    assert float((Q.conj().T @ Q - eye).abs().pow(2).sum().sqrt()) <= 4 * (2 * chi) ** 1.5 * 2.0 ** -53
    g.close()
