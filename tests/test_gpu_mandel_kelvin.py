"""Mandel fields on their way into the FP32 step: the sums of a voxel's components are formed in 64 bits before they are
rounded to FP32, from 16-byte aligned arrays (two voxels per thread on fields of this size) and from ones that are
not (one)."""
import numpy as np
import pytest

from oracle.lippmann_schwinger import Problem
from paper_1712_05145_gb300 import synthetic
from tests.helpers import TOL, oracle_ls_step_mandel, random_phase, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
GRID = (64, 48, 32)   # 98304 voxels: two fields lie above the line for two voxels per thread
SHAPE = (2, 6) + tuple(reversed(GRID))


def _at(values, offset):
    """values on the device, `offset` doubles past a 16-byte boundary"""
    buf = torch.zeros(values.numel() + 2, dtype=torch.float64, device="cuda")
    out = buf[offset:offset + values.numel()].view(values.shape)
    out.copy_(values)
    assert out.data_ptr() % 16 == 8 * offset
    return out


@pytest.mark.parametrize("offsets", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("precision", [0, 1])
def test_differences_of_close_components_keep_their_digits(precision, offsets):
    """eps = (c + d, c - d, c, 0, 0, 0) with c in [1, 2) and |d| <= 2^-40 in steps of 2^-52 and 2^-50: all exact in
    FP64, and so are the sums and differences, while c takes more bits than two floats hold.  Phases without a
    bulk contrast do not see c: the step is that of the field (d, -d, 0, ...), at the tolerance of any other field."""
    from paper_1712_05145_gb300 import hom
    lame = np.array([[3.0, 2.5], [4.5, 0.25]])
    assert np.all(3 * lame[:, 0] + 2 * lame[:, 1] == 14.0)
    ms = synthetic.Microstructure(random_phase(GRID, 2, 8), lame, 4.0, 1.0)
    assert 3 * ms.lam0 + 2 * ms.mu0 == 14.0
    rng = np.random.default_rng(4)
    d = rng.integers(-1024, 1025, size=(2,) + SHAPE[2:]) * 2.0 ** -50
    eps = np.zeros(SHAPE)
    c = 1.0 + (rng.integers(0, 2 ** 51, size=d.shape) + 2 ** 50) * 2.0 ** -52
    eps[:, 0], eps[:, 1], eps[:, 2] = c + d, c - d, c
    pure = np.zeros(SHAPE)
    pure[:, 0], pure[:, 1] = d, -d
    pb = Problem(ms.phase, ms.lame, ms.lam0, ms.mu0)
    ref = np.stack([oracle_ls_step_mandel(pb, pure[i], np.zeros(6)) for i in range(2)])
    H = hom.Homogenization(ms, precision=precision)
    src, dst = _at(torch.from_numpy(eps).cuda(), offsets[0]), _at(torch.zeros(SHAPE, dtype=torch.float64), offsets[1])
    torch.cuda.synchronize()   # the handle has a stream of its own
    hom.hom_ls_apply(H.h, 2, src, None, dst)
    H.close()
    assert rel_err(dst.cpu().numpy(), ref) < TOL[precision]


@pytest.mark.parametrize("offset", [0, 1])
def test_sums_whose_terms_exceed_fp32_are_finite_where_the_result_is(offset):
    """(2.5e38, 1e38, -1.5e38): eps_11 + eps_22 is above the largest FP32 number, the Kelvin components are not.  A
    homogeneous cell equal to the reference medium has no polarization: the step is 0."""
    from paper_1712_05145_gb300 import hom
    ms = synthetic.Microstructure(np.zeros(tuple(reversed(GRID)), np.uint8), np.array([[4.0, 2.5]]), 4.0, 2.5)
    eps = torch.zeros(SHAPE, dtype=torch.float64)
    eps[:, 0], eps[:, 1], eps[:, 2] = 2.5e38, 1e38, -1.5e38
    H = hom.Homogenization(ms, precision=1)
    src, dst = _at(eps.cuda(), offset), torch.full(SHAPE, 7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()   # the handle has a stream of its own
    hom.hom_ls_apply(H.h, 2, src, None, dst)
    H.close()
    assert not dst.any()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("scale", [1.0, 1e-25, 3e24])
def test_two_voxels_per_thread_match_the_oracle(scale, offset):
    from paper_1712_05145_gb300 import hom
    ms = synthetic.Microstructure(random_phase(GRID, 2, 9), np.array([[1.0, 1.0], [8.0, 5.0]]), 4.0, 2.5)
    pb = Problem(ms.phase, ms.lame, ms.lam0, ms.mu0)
    eps = np.random.default_rng(5).uniform(-1, 1, size=SHAPE)
    ref = np.stack([oracle_ls_step_mandel(pb, eps[i], np.zeros(6)) for i in range(2)])
    H = hom.Homogenization(ms, precision=1)
    src, dst = _at(torch.from_numpy(scale * eps).cuda(), offset), _at(torch.zeros(SHAPE, dtype=torch.float64), offset)
    torch.cuda.synchronize()   # the handle has a stream of its own
    hom.hom_ls_apply(H.h, 2, src, None, dst)
    H.close()
    assert rel_err(dst.cpu().numpy() / scale, ref) < TOL[1]
