"""3D local solves of the mixed form on a source with a NaN in it (device inputs
are not looked through on the host): the refinement's norms keep the NaN, so
the call ends as not converged instead of returning NaN fields."""
import numpy as np
import pytest

from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,sub", [((16, 12, 10), (8, 6, 5)), ((24, 11, 12), (12, 11, 12))])
def test_nan_source_is_not_converged(n, sub):
    from paper_2404_13811_gb300 import _lib as L
    from paper_2404_13811_gb300.solver import MRCM
    prob = I.lognormal_problem(n, sigma2=1.0, corr_len=0.2, seed=60)
    prob.f = np.zeros_like(prob.f)
    prob.f.flat[5] = np.nan
    s = MRCM(prob, I.Partition(sub, 0), space=0, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed",
             device_inputs=True)
    with pytest.raises(L.MrcmError) as e:
        s.build_basis()
    s.close()
    assert e.value.code == -5, e.value
