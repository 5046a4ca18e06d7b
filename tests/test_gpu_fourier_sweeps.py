"""FP32 CG and BiCGSTAB in Fourier space: what earlier calls left in the vectors' buffers does not matter, and
BiCGSTAB's passes in the launch shapes of larger grids."""
import numpy as np
import pytest

from helpers import random_phase
from paper_1712_05145_gb300 import synthetic
from test_gpu_spectral_cg import _compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LAME = np.array([[1.0, 1.0], [8.0, 5.0], [0.4, 0.3]])


def _ms(grid, seed):
    return synthetic.Microstructure(random_phase(grid, 3, seed, p=[0.5, 0.3, 0.2]), LAME, 4.0, 2.5)


@pytest.mark.parametrize("scheme", ["cg", "bicgstab"])
@pytest.mark.parametrize("grid", [(24, 24, 24), (12, 12, 16), (128, 24, 32)], ids=lambda g: "x".join(map(str, g)))
def test_order_1_does_not_read_what_earlier_calls_left_in_the_buffers(grid, scheme):
    """Half spectra of 312, 84 and 1560 columns: the last tile of a vector holds columns past the plane.  A step on
    64 fields of NaN leaves NaN in every work buffer that the order-1 loads take over; the same bits come out."""
    from paper_1712_05145_gb300 import hom
    out = []
    for poison in (False, True):
        H = hom.Homogenization(_ms(grid, 3), scheme={"cg": hom.HOM_CG, "bicgstab": hom.HOM_BICGSTAB}[scheme])
        assert all(i["status"] == 0 for i in H.solve(0, 1e-6))
        if poison:
            eps = torch.full((64, 6) + tuple(reversed(grid)), float("nan"), dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()   # the handle has a stream of its own
            hom.hom_ls_apply(H.h, 64, eps, None, eps)
            assert torch.isnan(eps).all()
        info = H.solve(1, 1e-6)
        assert all(i["status"] == 0 for i in info), info
        out.append((H.effective(1), [i["iterations"] for i in info]))
        H.close()
    assert out[0][1] == out[1][1] and np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("grid,pass_mode", [((128, 128, 96), 0),    # whole planes, wide z tiles, two of them per CTA
                                            ((128, 128, 96), 2),    # the same by rows and columns
                                            ((256, 192, 16), 0),    # rows and columns, wide tiles, one per CTA
                                            ((384, 256, 24), 0),    # ... and three per CTA, odd row blocks
                                            ((48, 24, 32), 2)],     # narrow tiles, the last one partly past the plane
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_bicgstab_in_the_launch_shapes_of_larger_grids(grid, pass_mode):
    from paper_1712_05145_gb300 import hom
    _compare(grid, pass_mode, hom.HOM_BICGSTAB)


@pytest.mark.parametrize("grid", [(32, 24, 16), (128, 96, 128)], ids=lambda g: "x".join(map(str, g)))
def test_bicgstab_loads_per_launch_do_not_change_the_result(grid):
    from paper_1712_05145_gb300 import hom
    out = []
    for chunk in (1, 6):
        H = hom.Homogenization(_ms(grid, 5), scheme=hom.HOM_BICGSTAB, rhs_chunk=chunk)
        info = H.solve(0, 1e-5)
        assert all(i["status"] == 0 for i in info), info
        out.append((H.effective(0), H.field(0, 4), [i["iterations"] for i in info]))
        H.close()
    assert out[0][2] == out[1][2]
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
