"""3D local kernels at the sizes where their tiling can go wrong: planes of
1 to 4 register tiles and of 125 to 128 cells (the widest inverted in
registers) and beyond (the shared-memory inverse), planes of one warp's 32,
64 and 128 rows, boxes of 3 to 12 planes along each axis, extents of one cell
in a plane, and rounds of 1 to 4 right-hand sides -- against the oracle at the
bars of the 3D parity tests (relative L2 1e-10 FP64, 1e-8 mixed)."""
import numpy as np
import pytest

from oracle import mrcm_oracle as O
from paper_2404_13811_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "mixed": 1e-8}

# n, sub, overlap, space: the largest box of each is the comment
CASES = [
    ((6, 4, 3), (3, 4, 3), 1, 0),       # 4 x 4 x 3: planes of 12 cells
    ((2, 2, 8), (1, 1, 4), 0, 0),       # 1 x 1 x 4: planes of one cell
    ((1, 6, 14), (1, 3, 7), 0, 0),      # 1 x 3 x 7: one cell thick
    ((16, 5, 5), (8, 5, 5), 1, 0),      # 9 x 5 x 5: planes of 25 along x
    ((8, 18, 4), (8, 9, 4), 1, 1),      # 8 x 10 x 4: planes of 32 along y
    ((16, 8, 11), (8, 8, 11), 1, 1),    # 9 x 8 x 11: planes of 72 along z
    ((20, 12, 10), (10, 12, 10), 0, 0),  # 10 x 12 x 10: planes of 100 along y
    ((16, 14, 14), (8, 14, 14), 1, 0),  # 9 x 14 x 14: planes of 126
    ((16, 32, 8), (8, 16, 8), 0, 0),    # 8 x 16 x 8: planes of 64
    ((24, 11, 12), (12, 11, 12), 0, 0),  # 12 x 11 x 12: planes of 132 (shared memory)
    ((6, 44, 34), (3, 22, 34), 0, 1),   # 3 x 22 x 34: three right-hand sides a round fit (mixed), six are solved
]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_box_shapes_match_oracle(case, precision):
    from paper_2404_13811_gb300 import _lib as L
    from paper_2404_13811_gb300.solver import MRCM
    n, sub, ov, space = CASES[case]
    prob = I.lognormal_problem(n, sigma2=2.0, corr_len=0.2, seed=40 + case)
    prob.f = np.random.default_rng(7 + case).standard_normal(prob.f.shape)
    ns = 2 if ov else 0
    ref = O.mrcm_os(prob, sub, ov, space, 1.0, 1.0, ns)
    try:
        s = MRCM(prob, I.Partition(sub, ov), space=space, alpha_basis=1.0, alpha_smooth=1.0, precision=precision)
    except L.MrcmError as e:
        assert e.code == -7, e   # a box that does not fit shared memory is refused
        pytest.skip(str(e))
    s.run(ns)
    p, u = s.fluxes()
    s.close()
    ep, eu = O.rel_errors(prob, p, u, ref.p, ref.u)
    assert ep <= TOL[precision] and eu <= TOL[precision], (ep, eu)
