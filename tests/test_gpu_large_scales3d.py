"""3D mixed form at large permeabilities: the pressure does not depend on the
scale and the velocities are proportional to it (bar 1e-8, that of the mixed
parity tests), up to the largest FP64 values the coefficients can take.  The
smoothing solves once started from the pressure times an FP32 reciprocal of the
Jacobi scale, which is infinite from about 1e76 on."""
import numpy as np
import pytest

from oracle import mrcm_oracle as O
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_large_permeabilities_3d():
    from paper_2404_13811_gb300.solver import MRCM
    base = I.lognormal_problem((16, 16, 16), sigma2=1.0, corr_len=0.2, seed=21)

    def run(K):
        prob = I.Problem(base.dim, base.n, base.h, K, base.f, base.bc_kind, base.bc_value)
        s = MRCM(prob, I.Partition((8, 8, 8), 1), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
        s.run(2)
        p, u = s.fluxes()
        s.close()
        return p, u

    p0, u0 = run(base.K)
    for c in (1e40, 1e70, 1e76, 1e90, 1e200):
        p, u = run(base.K * c)
        ep, eu = O.rel_errors(base, p, u / c, p0, u0)
        assert np.all(np.isfinite(u)) and ep <= 1e-8 and eu <= 1e-8, (c, ep, eu)
