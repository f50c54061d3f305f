"""Mixed-form solves of right-hand sides of any size: 3D problems with
permeabilities scaled down, and gradients from seeds scaled down.  Both are
linear in the scale, so results are compared with those at scale one (bar 1e-8,
that of the mixed parity tests).  A refinement follows its right-hand side down
by twelve digits; where the FP32 vectors ended in zeros on the way, the calls
returned wrong values."""
import numpy as np
import pytest

from oracle import mrcm_oracle as O
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sub,overlap", [((16, 16, 16), (8, 8, 8), 1), ((24, 11, 12), (12, 11, 12), 0)])
def test_small_permeabilities_3d(n, sub, overlap):
    from paper_2404_13811_gb300.solver import MRCM
    base = I.lognormal_problem(n, sigma2=1.0, corr_len=0.2, seed=21)

    def run(K):
        prob = I.Problem(base.dim, base.n, base.h, K, base.f, base.bc_kind, base.bc_value)
        s = MRCM(prob, I.Partition(sub, overlap), space=overlap, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
        s.run(2 if overlap else 0)
        p, u = s.fluxes()
        s.close()
        return p, u

    p0, u0 = run(base.K)
    for c in (1e-40, 1e-50, 1e-60, 1e-77, 1e-150):
        p, u = run(base.K * c)
        ep, eu = O.rel_errors(base, p, u / c, p0, u0)
        assert ep <= 1e-8 and eu <= 1e-8, (c, ep, eu)


@pytest.mark.parametrize("sub,n", [((16, 16), (64, 48)), ((9, 8), (27, 16))])
@pytest.mark.parametrize("steps", [0, 2])
def test_small_seeds(sub, n, steps):
    """Down to 1e-32: below, the interface solve's FP32 factors underflow in either form."""
    from paper_2404_13811_gb300.solver import MRCM
    prob = I.lognormal_problem(n, sigma2=2.0, corr_len=0.15, seed=7)
    rng = np.random.default_rng(3)
    gp, gu = rng.standard_normal(prob.ncells), rng.standard_normal((prob.ncells, 4))
    s = MRCM(prob, I.Partition(sub, 2), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
    s.run(steps)
    g0 = s.adjoint(gp, gu)
    for c in (1e-25, 1e-28, 1e-30, 1e-32, 1e30):
        g = s.adjoint(gp * c, gu * c) / c
        assert np.abs(g - g0).max() <= 1e-8 * np.abs(g0).max(), c
    s.close()
