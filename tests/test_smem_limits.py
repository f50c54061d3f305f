"""Shared memory of the box kernels: what a box needs is compared with what the
kernel can have, the CTA's 227 KB less the kernel's static shared memory (480
bytes in the 3D basis kernel), so that no box is accepted whose launch fails.
Boxes of the sizes in between take fewer right-hand sides a round."""
import ctypes

import numpy as np
import pytest

from paper_2404_13811_gb300 import inputs as I

CTA = 227 * 1024
STATIC_LOCAL3D = 480


def test_basis_rounds_leave_room_for_the_static_part():
    from paper_2404_13811_gb300 import build
    size = ctypes.CDLL(build.build())._Z12local3d_smemiiiib   # (precision, nx, ny, nz, particular)
    size.restype = ctypes.c_size_t
    seen = set()
    for shape in ((7, 15, 22), (15, 7, 22), (22, 15, 7), (3, 22, 34), (10, 10, 14), (13, 14, 12)):
        b = size(1, *shape, False)
        seen.add(b)
        # larger than the CTA has in all: refused at creation; never in between
        assert b <= CTA - STATIC_LOCAL3D or b > CTA, (shape, b)
    assert len(seen) > 1


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-8)])
def test_box_between_the_limits_matches_oracle(precision, tol):
    """7 x 15 x 22 cells, three basis functions: three right-hand sides a round take
    232,256 bytes in the mixed form.  (The FP64 form fits with three.)"""
    from oracle import mrcm_oracle as O
    from paper_2404_13811_gb300.solver import MRCM
    prob = I.lognormal_problem((14, 15, 22), sigma2=2.0, corr_len=0.2, seed=50)
    prob.f = np.random.default_rng(17).standard_normal(prob.f.shape)
    ref = O.mrcm_os(prob, (7, 15, 22), 0, 1, 1.0, 1.0, 0)
    s = MRCM(prob, I.Partition((7, 15, 22), 0), space=1, alpha_basis=1.0, alpha_smooth=1.0, precision=precision)
    s.run(0)
    p, u = s.fluxes()
    s.close()
    ep, eu = O.rel_errors(prob, p, u, ref.p, ref.u)
    assert ep <= tol and eu <= tol, (ep, eu)


def test_no_box_of_the_shapes_test_is_refused():
    """The 3D shapes test skips a box that is refused; none of its boxes may be."""
    from paper_2404_13811_gb300 import build
    from tests.test_gpu_local3d import CASES
    lib = ctypes.CDLL(build.build())
    basis, smooth = lib._Z12local3d_smemiiiib, lib._Z13smooth3d_smemiiii
    basis.restype = smooth.restype = ctypes.c_size_t
    for n, sub, ov, _ in CASES:
        # the largest box: inner subdomains grow on both sides, of two on one
        box = [min(n[a], sub[a] + ov * min(2, n[a] // sub[a] - 1)) for a in range(3)]
        for prec in (0, 1):
            assert max(basis(prec, *box, False), basis(prec, *sub, True)) <= CTA - STATIC_LOCAL3D, (box, prec)
            assert smooth(prec, *box) <= CTA - 448, (box, prec)
