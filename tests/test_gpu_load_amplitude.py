"""Loads of any amplitude: A x = b is linear, so a load scaled by a power of two gives the solution scaled by it, in as
many iterations, and its certified residual is the true one.

Measured from outside: the residual ||T(x) - x|| / ||T(0)|| of the Lippmann-Schwinger step T in FP64 on the returned
strain.  The solve certifies it below its tolerance relative to a norm of b that it computes in FP32, so the FP64 value
may exceed the tolerance by a relative 1e-5 (some ten FP32 roundings) at most.  Solutions of two residuals of 1e-6 ||b|| differ by 1.3e-4 of
their norm at most (twice the bound derived in test_gpu_spectral_cg.py for these moduli)."""
import numpy as np
import pytest

from helpers import random_phase
from paper_1712_05145_gb300 import synthetic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LAME = np.array([[1.0, 1.0], [8.0, 5.0], [0.4, 0.3]])
UNIT = np.eye(6)[[0, 5]] + 0.25 * np.eye(6)[[1, 3]]
TOL = 1e-6
AMPLITUDES = [-30, -40, -60, -100, 20, 80]


def _ms(grid, seed):
    return synthetic.Microstructure(random_phase(grid, 3, seed, p=[0.5, 0.3, 0.2]), LAME, 4.0, 2.5)


def _fields(H, order, amp):
    """the strains of two loads over their amplitudes.  The handle has a stream of its own: torch is done with a
    field before its memory can be the next one's."""
    out = []
    for k in range(2):
        out.append(H.field(order, k, device=True) / float(amp[k]))
        torch.cuda.synchronize()
    return out


def _residuals(ms, fields, loads):
    """||T(x) - x|| / ||T(0)|| per load, computed in FP64 for the loads scaled to amplitude 1"""
    from paper_1712_05145_gb300 import hom
    H = hom.Homogenization(ms, precision=hom.HOM_FP64)
    x = torch.stack(fields)
    t, b = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    hom.hom_ls_apply(H.h, len(fields), x, loads, t)
    hom.hom_ls_apply(H.h, len(fields), None, loads, b)
    H.close()
    # Mandel components: the Euclidean norm is the tensor's
    return [float((t[i] - x[i]).norm() / b[i].norm()) for i in range(len(fields))]


@pytest.mark.parametrize("scheme", ["cg", "bicgstab"])
@pytest.mark.parametrize("grid", [(64, 48, 32), (8, 6, 3), (48, 32, 1)], ids=lambda g: "x".join(map(str, g)))
def test_order_0_loads_of_any_amplitude(grid, scheme):
    from paper_1712_05145_gb300 import hom
    ms = _ms(grid, 11)
    H = hom.Homogenization(ms, scheme={"cg": hom.HOM_CG, "bicgstab": hom.HOM_BICGSTAB}[scheme])
    base = H.solve(0, TOL, loads=UNIT)
    x0 = _fields(H, 0, np.ones(2))
    c0 = H.effective(0)
    for e in AMPLITUDES + [None]:
        amp = np.array([2.0 ** -45, 1.0]) if e is None else np.full(2, 2.0 ** e)   # None: loads of both kinds in one call
        info = H.solve(0, TOL, loads=UNIT * amp[:, None])
        x = _fields(H, 0, amp)
        assert [i["status"] for i in info] == [0, 0], (e, info)
        assert [i["iterations"] for i in info] == [i["iterations"] for i in base], e
        assert all(r < TOL * (1 + 1e-5) for r in _residuals(ms, x, UNIT)), e
        for k in range(2):
            assert float((x[k] - x0[k]).norm()) <= 1.3e-4 * float(x0[k].norm()), e
        assert np.linalg.norm(H.effective(0) / amp - c0) <= 1.3e-4 * np.linalg.norm(c0), e
    H.close()


@pytest.mark.parametrize("scheme", ["cg", "bicgstab"])
@pytest.mark.parametrize("grid", [(32, 24, 16), (24, 16, 8)], ids=lambda g: "x".join(map(str, g)))
def test_order_1_loads_of_any_amplitude(grid, scheme):
    from paper_1712_05145_gb300 import hom
    ms = _ms(grid, 12)
    H = hom.Homogenization(ms, scheme={"cg": hom.HOM_CG, "bicgstab": hom.HOM_BICGSTAB}[scheme])
    assert all(i["status"] == 0 for i in H.solve(0, TOL))
    W = np.zeros((2, 18))
    W[0, 4] = W[1, 9] = 1.0
    W[1, 2] = -0.5
    base = H.solve(1, TOL, loads=W)
    x0 = _fields(H, 1, np.ones(2))
    c0 = H.effective(1)
    for e in AMPLITUDES:
        info = H.solve(1, TOL, loads=W * 2.0 ** e)
        assert [i["status"] for i in info] == [0, 0], (e, info)
        assert [i["iterations"] for i in info] == [i["iterations"] for i in base], e
        for a, b in zip(_fields(H, 1, np.full(2, 2.0 ** e)), x0):
            assert float((a - b).norm()) <= 1.3e-4 * float(b.norm()), e
        assert np.linalg.norm(H.effective(1) / 2.0 ** e - c0) <= 1.3e-4 * np.linalg.norm(c0), e
    H.close()


def test_a_load_of_zero_and_a_load_of_nan_end_as_before():
    from paper_1712_05145_gb300 import hom
    H = hom.Homogenization(_ms((16, 12, 16), 13))
    info = H.solve(0, TOL, loads=np.stack([UNIT[0], np.zeros(6)]))
    assert [i["status"] for i in info] == [0, 0] and info[1]["iterations"] == 0
    assert not H.field(0, 1).any()
    with pytest.raises(hom.HomError):
        H.solve(0, TOL, loads=np.stack([UNIT[0], np.full(6, np.nan)]))
    H.close()
