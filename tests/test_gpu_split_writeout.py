"""The split GEMM's write-out over output scales on both sides of its fast path's range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (129, 49, 64), (130, 97, 65), (257, 33, 200), (64, 200, 700)])
@pytest.mark.parametrize("n_split", [2, 5])
def test_scaled_rows_and_columns(ctm_lib, shape, n_split):
    """Power-of-two factors on the rows of A and the columns of B scale the exact integer sums'
    exponents only, so C scales by the same factors.  2^-52 relative: the conversions on the two
    paths may round a tie apart, and each rounds once (2^-53)."""
    from paper_2509_05090_gb300 import binding
    M, N, K = shape
    rng = np.random.default_rng(M * 1000 + N * 10 + K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    r = rng.integers(-475, 476, M)
    c = rng.integers(-475, 476, N)
    r[0], c[0] = 475, 475
    r[-1], c[-1] = (-475, -475) if M > 1 else (475, 475)

    def mul(a, b):
        out = binding.ctm_gemm(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), precision="split_bf16",
                               n_split=n_split)
        return out.cpu().numpy()

    base = mul(A, B)
    got = mul(np.ldexp(A, r[:, None]), np.ldexp(B, c[None, :]))
    want = np.ldexp(base, r[:, None] + c[None, :])
    assert np.all(np.abs(got - want) <= 2.0 ** -52 * np.abs(want))
