"""Rounding of the 3D mixed form's refinement.  With ir_tol met by far (the
refinement runs to its floor) two solutions whose permeabilities differ by a
factor that is no power of two differ by rounding alone.  Residuals in
differences of neighbouring pressures round like the fluxes: a few eps = 2.2e-16
per face, six faces a cell, the errors of eight boxes meeting at random: 20 eps
as a bar.  Residuals that sum rows of pressures of order one round eps |p| T per
face instead, 45 to 90 eps of the fluxes on these fields."""
import numpy as np
import pytest

from oracle import mrcm_oracle as O
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma2,seed", [(1.0, 21), (4.0, 22)])
def test_velocities_agree_across_scales_to_rounding(sigma2, seed):
    from paper_2404_13811_gb300.solver import MRCM
    base = I.lognormal_problem((16, 16, 16), sigma2=sigma2, corr_len=0.2, seed=seed)

    def run(K):
        prob = I.Problem(base.dim, base.n, base.h, K, base.f, base.bc_kind, base.bc_value)
        s = MRCM(prob, I.Partition((8, 8, 8), 1), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
        s.run(2)
        p, u = s.fluxes()
        s.close()
        return p, u

    p0, u0 = run(base.K)
    for c in (3.0, 7.0, 1.0 / 3.0, 0.7):
        p, u = run(base.K * c)
        ep, eu = O.rel_errors(base, p, u / c, p0, u0)
        assert eu <= 20 * np.finfo(float).eps, (c, ep, eu)
