"""Digit packs of contiguous-K operands (odd rows, rows of up to 16 warps of 16 K tiles) against the
packs of the same operand transposed."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 63, 65, 129, 641, 1025, 8192, 8193, 8200, 8321, 16383, 16384, 16385])
@pytest.mark.parametrize("M", [1, 5, 130, 2000])
def test_rows_against_columns(ctm_lib, M, K):
    """A B packs A by rows, (B^T A^T)^T by columns.  At four slices every level sum is an exact
    integer, so only the last conversion may round a tie apart: 2^-52 relative."""
    from paper_2509_05090_gb300 import binding
    rng = np.random.default_rng(M + 7 * K)
    A = torch.from_numpy(rng.standard_normal((M, K))).cuda()
    B = torch.from_numpy(rng.standard_normal((K, 17))).cuda()
    C = binding.ctm_gemm(A, B, precision="split_bf16", n_split=4)
    D = binding.ctm_gemm(B.T.contiguous(), A.T.contiguous(), precision="split_bf16", n_split=4).T
    assert bool(((C - D).abs() <= 2.0 ** -52 * D.abs()).all())
