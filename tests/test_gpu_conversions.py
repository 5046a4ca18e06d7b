"""Mandel fields in and out of the step, whose types change by integer arithmetic on the bits: the step is
linear, so scaled inputs give scaled results, from aligned arrays (two voxels per thread) and from ones that
are not (one)."""
import numpy as np
import pytest

from oracle.lippmann_schwinger import Problem
from paper_1712_05145_gb300 import synthetic
from tests.helpers import TOL, oracle_ls_step_mandel, random_mandel_fields, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("scale", [1.0, 1e-25, 3e24, -1e-30])
@pytest.mark.parametrize("precision", [0, 1])
def test_ls_step_is_linear_over_magnitudes_and_alignments(precision, scale, offset):
    """The tolerance is the one of the unscaled step: rounding is relative, and 1e-30 keeps the smallest
    products within the normal FP32 range."""
    from paper_1712_05145_gb300 import hom
    ms = synthetic.centred_sphere(8)
    pb = Problem(ms.phase, ms.lame, ms.lam0, ms.mu0)
    eps = random_mandel_fields(2, ms.grid, 31)
    E = np.random.default_rng(6).uniform(-1, 1, size=(2, 6))
    ref = np.stack([oracle_ls_step_mandel(pb, eps[i], E[i]) for i in range(2)])
    H = hom.Homogenization(ms, precision=precision)
    src = torch.zeros(eps.size + 2, dtype=torch.float64, device="cuda")
    dst = torch.zeros_like(src)
    ed, out = (t[offset:offset + eps.size].view(eps.shape) for t in (src, dst))
    ed.copy_(torch.from_numpy(scale * eps))
    hom.hom_ls_apply(H.h, 2, ed, scale * E, out)
    assert rel_err(out.cpu().numpy() / scale, ref) < TOL[precision]
    assert dst[eps.size + offset:].abs().sum() == 0 and dst[:offset].abs().sum() == 0
    H.close()
