"""2D mixed form at permeabilities of any scale: the pressure does not depend on
it and the velocities are proportional to it (bar 1e-8, that of the mixed parity
tests).  Refinements whose FP32 vectors are not scaled by their right-hand
side's exponent end in zeros below about 1e-45 (not converged, or wrong values
at 1e-70 and below) and in infinities from 1e74 on."""
import numpy as np
import pytest

from oracle import mrcm_oracle as O
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sub,overlap", [((64, 48), (16, 16), 4), ((54, 42), (9, 7), 2), ((60, 80), (10, 40), 3)])
def test_permeability_scale_2d(n, sub, overlap):
    from paper_2404_13811_gb300.solver import MRCM
    base = I.lognormal_problem(n, sigma2=1.0, corr_len=0.2, seed=21)

    def run(K):
        prob = I.Problem(base.dim, base.n, base.h, K, base.f, base.bc_kind, base.bc_value)
        s = MRCM(prob, I.Partition(sub, overlap), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
        s.run(2)
        p, u = s.fluxes()
        s.close()
        return p, u

    p0, u0 = run(base.K)
    for c in (1e-150, 1e-80, 1e-70, 1e-60, 1e75, 1e78, 1e150):
        p, u = run(base.K * c)
        ep, eu = O.rel_errors(base, p, u / c, p0, u0)
        assert np.all(np.isfinite(u)) and ep <= 1e-8 and eu <= 1e-8, (c, ep, eu)
