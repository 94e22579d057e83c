"""FP64 contractions on the tensor cores (eight digit slices, csrc/gemm_split.cu): a step at the sizes
where the tiling can go wrong, against the FP64 oracle with the FP64 path's own tolerances
(test_gpu_parity.py), and environments that hold infinities."""
import numpy as np
import pytest

from paper_2509_05090_gb300 import inputs as I
from test_gpu_parity import _step_parity

pytestmark = pytest.mark.gpu

# n = chi D^2 and chi around the 128-row and 64/32-column tiles, the 64-deep K tiles and the
# 128-deep chunks; the smallest ones mix sliced and FP64-pipe contractions in one step
EDGES = [(4, 32, 2), (4, 33, 2), (3, 57, 2), (5, 31, 2), (4, 64, 2), (6, 24, 1), (5, 52, 1), (3, 129, 1), (7, 21, 1)]


@pytest.mark.parametrize("D,chi,pre", EDGES)
def test_step_at_tile_edges(ctm_lib, D, chi, pre):
    _step_parity(I.random_site_tensor(2, D, 900 + 10 * D + chi), chi, pre)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite_environment_is_reported(ctm_lib, bad):
    """A row with an infinity or a NaN has no digit grid; its outputs are the plain FP64 sums, so the
    step reports CTM_ENONFINITE as before."""
    from paper_2509_05090_gb300 import binding
    g = binding.CTM(I.random_site_tensor(2, 4, 31), 40)
    g.ctm_step(2)
    C, T, Q = g.ctm_get_env()
    T[3, 5, 7] = bad
    g.ctm_set_env(C, T, Q)
    with pytest.raises(binding.CtmError) as ei:
        g.ctm_step(1)
    assert ei.value.status == 5
    g.close()
