"""The autotuner's choice follows a fixed preference among close variants:
handles of one problem take the same variant and agree bit for bit, and the
first solve runs every variant once (the preferred one last, so that its run
is the solve's)."""
import numpy as np
import pytest

from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# subdomains along x and y, space: slabs of 14 (blocked elimination where it takes fewer steps), 30 and 60 unknowns
CASES = [(4, 12, 0), (8, 4, 0), (8, 4, 1)]


@pytest.mark.parametrize("mx,my,space", CASES)
def test_handles_of_one_problem_agree(mx, my, space, monkeypatch):
    monkeypatch.delenv("MRCM_TUNE_CACHE", raising=False)
    from paper_2404_13811_gb300.solver import MRCM
    prob = I.lognormal_problem((12 * mx, 12 * my), sigma2=2.0, corr_len=0.1, seed=11)
    ref = None
    for _ in range(6):
        s = MRCM(prob, I.Partition((12, 12), 2), space=space, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")
        s.run(1)
        st, (p, u) = s.stats(), s.fluxes()
        s.close()
        assert st["slab_inverse_source"] == "measured", st
        if ref is None:
            ref = (st["slab_inverse"], p, u)
        assert st["slab_inverse"] == ref[0] and np.array_equal(p, ref[1]) and np.array_equal(u, ref[2])


def test_first_solve_runs_each_variant_once(monkeypatch):
    monkeypatch.delenv("MRCM_TUNE_CACHE", raising=False)
    from paper_2404_13811_gb300.solver import MRCM
    prob = I.lognormal_problem((96, 48), sigma2=2.0, corr_len=0.1, seed=11)
    s = MRCM(prob, I.Partition((12, 12), 2), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision="mixed")

    def inverses():
        s.profile(True)
        s.build_basis()
        s.solve_interface()
        return s.timings()["interface_lu"][1]

    first, later = inverses(), inverses()
    assert s.stats()["slab_inverse"] == "gauss-jordan-registers"
    s.close()
    assert later > 0 and first == 3 * later, (first, later)
