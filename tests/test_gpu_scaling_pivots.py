"""Scale invariance (K -> c K, as in the scaling test) at the scales where pivots
and face coefficients of the FP64 form cross the limits of the FP32 seeds of
its reciprocals (2^126 and 2^127, and 2^-126): lines of 24 cells in 2D and
planes of 81 to 100 cells in 3D, inverted by symmetric tiles.  Bar: that of the
scaling test."""
import numpy as np
import pytest

from oracle import mrcm_oracle as O
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sub,overlap", [((64, 48), (16, 16), 4), ((16, 16, 16), (8, 8, 8), 1)])
@pytest.mark.parametrize("c", [1e-39, 1e-38, 1e-37, 1e36, 1e37, 3e37, 1e38, 3e38, 1e39, 1e40])
def test_fp64_form_at_the_limits_of_fp32(n, sub, overlap, c):
    from paper_2404_13811_gb300.solver import MRCM
    base = I.lognormal_problem(n, sigma2=1.0, corr_len=0.2, seed=21)

    def run(K):
        prob = I.Problem(base.dim, base.n, base.h, K, base.f, base.bc_kind, base.bc_value)
        s = MRCM(prob, I.Partition(sub, overlap), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision="fp64")
        s.run(2)
        p, u = s.fluxes()
        s.close()
        return p, u

    p0, u0 = run(base.K)
    p, u = run(base.K * c)
    ep, eu = O.rel_errors(base, p, u / c, p0, u0)
    assert np.all(np.isfinite(p)) and ep <= 1e-10 and eu <= 1e-10, (c, ep, eu)
