"""Gradient with boxes near the largest that fit shared memory: the reverse basis
kernel then has the vectors of four, two or one right-hand side at a time (the
factorisation runs on two warps all the same).  Against the oracle's gradient at
the bar of the gradient tests."""
import numpy as np
import pytest

from oracle import mrcm_adjoint as OA
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# the inner boxes sub + 2 l: FP64 24 x 24 four, 26 x 26 two, 26 x 28 one; mixed 32 x 20 four, 32 x 25 two, 32 x 28 one
@pytest.mark.parametrize("precision,sub,ov", [("fp64", (16, 16), 4), ("fp64", (16, 16), 5), ("fp64", (16, 18), 5),
                                              ("mixed", (24, 12), 4), ("mixed", (24, 17), 4), ("mixed", (24, 20), 4)])
def test_gradient_matches_oracle(precision, sub, ov):
    from paper_2404_13811_gb300.solver import MRCM
    n = (3 * sub[0], 3 * sub[1])
    prob = I.lognormal_problem(n, sigma2=2.0, corr_len=0.15, seed=31)
    prob.f = np.random.default_rng(32).standard_normal(prob.f.shape)
    rng = np.random.default_rng(33)
    gp, gu = rng.standard_normal(prob.ncells), rng.standard_normal((prob.ncells, 4))
    _, ref = OA.mrcm_os_adjoint(prob, sub, ov, 1, 1.0, 1.0, 1, gp, gu)
    s = MRCM(prob, I.Partition(sub, ov), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision=precision)
    s.run(1)
    g = s.adjoint(gp, gu)
    s.close()
    assert np.abs(g - np.asarray(ref).reshape(-1)).max() <= 1e-8 * np.abs(ref).max()
