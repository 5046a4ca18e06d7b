"""FP32 CG and BiCGSTAB with their vectors in Fourier space against the FP64 mode's CG on real fields, at every axis
length of the z, y and row transforms, through whole planes and through rows and columns.

Tolerance.  The phases' moduli lie between 0.106 and 2 times the reference medium's (3 lambda + 2 mu =
5, 34, 1.8 against 17; 2 mu = 2, 10, 0.6 against 5), so A's spectrum in the C0 product does.  A residual
of 1e-6 ||b|| leaves ||x - x*||_C0 <= 1e-6 / 0.106 ||b||_C0 and ||b||_C0 <= 2 ||x*||_C0; the C0 and the L2
norm differ by sqrt(17 / 5) at most on either side: ||x - x*|| <= 6.4e-5 ||x*||.
"""
import numpy as np
import pytest

from helpers import random_phase
from paper_1712_05145_gb300 import synthetic

pytestmark = pytest.mark.gpu
LAME = np.array([[1.0, 1.0], [8.0, 5.0], [0.4, 0.3]])
BOUND = 6.4e-5
LENGTHS = [2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512]
GRIDS = ([(8, 6, n) for n in [1] + LENGTHS] + [(8, n, 3) for n in LENGTHS] + [(2 * n, 4, 3) for n in LENGTHS]
         + [(64, 48, 32), (96, 32, 12), (256, 64, 8)]
         # whole planes on either side of the lines between their launch shapes
         + [(64, 64, 4), (96, 48, 4), (128, 64, 4), (96, 96, 4), (256, 48, 4), (128, 128, 4), (64, 256, 4)])


def _ms(grid, seed):
    return synthetic.Microstructure(random_phase(grid, 3, seed, p=[0.5, 0.3, 0.2]), LAME, 4.0, 2.5)


def _compare(grid, pass_mode, scheme32):
    from paper_1712_05145_gb300 import hom
    ms = _ms(grid, sum(grid))
    loads = np.eye(6)[[0, 5]] + 0.25 * np.eye(6)[[1, 3]]
    got = []
    for precision, scheme, tol in ((hom.HOM_FP32_REFINE, scheme32, 1e-6), (hom.HOM_FP64, hom.HOM_CG, 1e-10)):
        H = hom.Homogenization(ms, precision=precision, scheme=scheme, pass_mode=pass_mode)
        info = H.solve(0, tol, loads=loads)
        assert all(i["status"] == 0 for i in info), info
        got.append((H.effective(0), [H.field(0, k) for k in range(2)]))
        H.close()
    (c32, e32), (c64, e64) = got
    assert np.linalg.norm(c32 - c64) <= BOUND * np.linalg.norm(c64)
    for a, b in zip(e32, e64):
        assert np.linalg.norm(a - b) <= BOUND * np.linalg.norm(b)


@pytest.mark.parametrize("pass_mode", [0, 2])
@pytest.mark.parametrize("grid", GRIDS, ids=["x".join(map(str, g)) for g in GRIDS])
def test_fp32_cg_matches_fp64_cg(grid, pass_mode):
    from paper_1712_05145_gb300 import hom
    _compare(grid, pass_mode, hom.HOM_CG)


@pytest.mark.parametrize("n3", [1] + LENGTHS)
def test_fp32_bicgstab_matches_fp64_cg(n3):
    from paper_1712_05145_gb300 import hom
    _compare((8, 6, n3), 0, hom.HOM_BICGSTAB)


@pytest.mark.parametrize("grid", [(32, 24, 16), (128, 96, 128)])
def test_loads_per_launch_do_not_change_the_result(grid):
    from paper_1712_05145_gb300 import hom
    ms = _ms(grid, 5)
    out = []
    for chunk in (1, 6):
        H = hom.Homogenization(ms, rhs_chunk=chunk)
        info = H.solve(0, 1e-5)
        out.append((H.effective(0), H.field(0, 4), [i["iterations"] for i in info]))
        H.close()
    assert out[0][2] == out[1][2]
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
