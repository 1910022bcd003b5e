"""FP64 Lanczos launches take one walk under the automatic schedule, whatever their size, and
give the split's coefficients up to rounding when the split is asked for."""
import pytest
import torch

from paper_2605_26261_gb300 import ftlm, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [1, 4, 8, 16])
def test_automatic_schedule_of_doubles_is_one_walk(cuda_dev, width):
    bonds = inputs.icosidodecahedron()  # 26 bonds inside the high block
    with ftlm.Basis(30, 0, bonds, ftlm.RANK_CR) as b:  # 1.2 GB a vector
        assert ftlm.ftlm_basis_hv_schedule(b.handle, width, torch.float64) == ftlm.HV_ONE_WALK
    M, R = 6, width
    ftlm.ftlm_lanczos_set_block(width)
    try:
        with ftlm.Basis(30, 20, bonds, ftlm.RANK_CR) as b:
            one = ftlm.lanczos(b, R, M, seed=2, dtype=torch.float64, keep_coeffs=True)
            b.set_schedule(ftlm.HV_SPLIT)
            split = ftlm.lanczos(b, R, M, seed=2, dtype=torch.float64, keep_coeffs=True)
            # both sum the same 60 terms per row, in another order, M times
            scale = 0.75 * float(abs(bonds[2]).sum())
            for k in ("alpha", "beta"):
                assert (one[k] - split[k]).abs().max().item() <= 64 * M * 2.0**-53 * scale
    finally:
        ftlm.ftlm_lanczos_set_block(0)
