"""Output of pure-Neumann members: the zero-mean gauge of mrcm_fluxes against
the independent reduction of mrcm_fluxes_static, at cell counts on both sides
of the reduction's block size (2048 cells) and of its largest block count
(256).  Bar: both means sum the same n <= 655,360 values in FP64 in another
order; each is within n eps max|p| of the exact one and far closer on average
(sqrt(n) eps), so 1e-12 max|p| bounds the difference."""
import numpy as np
import pytest

from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(32, 16), (64, 32), (48, 48), (240, 208), (1024, 640)])
def test_zero_mean_output_matches_static(n):
    import torch

    from paper_2404_13811_gb300 import _lib as L
    from paper_2404_13811_gb300.solver import MRCM
    prob = I.lognormal_problem(n, sigma2=1.0, corr_len=0.2, seed=5, bc="noflow", source="q5")
    s = MRCM(prob, I.Partition((16, 16), 2), space=0, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
    s.run(1)
    ph, uh = s.fluxes()
    pd, ud = s.state()
    ps = torch.empty_like(pd)
    us = torch.empty_like(ud)
    L.mrcm_fluxes_static(s.h, 0, us, ps)
    scale = np.abs(ph).max()
    assert np.array_equal(ph, pd.cpu().numpy()) and np.array_equal(uh, ud.cpu().numpy())
    assert np.array_equal(uh, us.cpu().numpy())
    assert np.abs(ph - ps.cpu().numpy()).max() <= 1e-12 * scale
    assert abs(ph.mean()) <= 1e-12 * scale
    s.close()
