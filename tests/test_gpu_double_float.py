"""Double-float operations of the FP32 mode's FP64-accurate passes against exact rational arithmetic, and the wave
vectors of its solvers.

Two floats hold a number to 2^-49 of its size: the low one lies below half an ulp of the high one, 2^-24, and is
rounded to 24 bits.  An FP64 operation rounded to two floats adds its own 2^-53, and the operations here are to be as
good."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1712_05145_gb300 import build

pytestmark = pytest.mark.gpu
BOUND = Fraction(1, 2 ** 49) + Fraction(1, 2 ** 53)
N = 20000


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = tmp_path_factory.mktemp("df") / "double_float_ops.so"
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "double_float_ops.cu")
    r = subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-shared", src, "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


def _df(x):
    """float64 array -> [n][2] float32, high and low part"""
    hi = x.astype(np.float32)
    return np.ascontiguousarray(np.stack([hi, (x - hi).astype(np.float32)], axis=1))


def _exact(df):
    return [Fraction(float(h)) + Fraction(float(l)) for h, l in df]


def _ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


@pytest.mark.parametrize("exponents", [(0, 0), (-20, 30), (30, -20)])
def test_division(lib, exponents):
    """Operands over eight binades each, of both signs, the kernels' 1 / |xi|^2 among them."""
    rng = np.random.default_rng(3)
    a, b = (_df(rng.choice([-1.0, 1.0], N) * 2.0 ** rng.uniform(e, e + 8, N)) for e in exponents)
    a[:N // 2] = [1.0, 0.0]
    out = np.zeros_like(a)
    assert lib.df_divide(_ptr(a), _ptr(b), _ptr(out), N) == 0
    worst = max(abs(q / (x / y) - 1) for q, x, y in zip(_exact(out), _exact(a), _exact(b)))
    assert worst <= BOUND, float(worst * 2 ** 49)


@pytest.mark.parametrize("grid", [(512, 384, 96), (48, 512, 192), (12, 24, 512)])
def test_wave_numbers(lib, grid):
    g = (ctypes.c_int * 3)(*grid)
    for axis in range(3):
        n = 513
        out, scale = np.zeros((n, 2), np.float32), ctypes.c_double()
        assert lib.df_waves(g, axis, -256, n, _ptr(out), ctypes.byref(scale)) == 0
        for k, x in zip(range(-256, 257), _exact(out)):
            assert abs(x - k * Fraction(scale.value)) <= BOUND * abs(k) * Fraction(scale.value), (axis, k)


@pytest.mark.parametrize("grid", [(64, 48, 32), (24, 3, 16), (8, 6, 1), (256, 4, 2)])
def test_rotated_wave_vectors(lib, grid):
    """The rotated symbol p = (s1 c2 c3, c1 s2 c3, c1 c2 s3), s and c at pi j / N, up to a factor: tangents, each
    rounded once to FP32 (2^-24, and some 2^-52 of the FP64 table and of p here); where a cosine is 0, the axis of p."""
    axes = [np.arange(n) for n in (grid[0] // 2 + 1, grid[1], grid[2])]
    sin = [np.sin(np.pi * j / n) for j, n in zip(axes, grid)]
    cos = [np.where(2 * j == n, 0.0, np.cos(np.pi * j / n)) for j, n in zip(axes, grid)]
    tan = [np.where(2 * j == n, 0.0, np.tan(np.pi * j / n)) for j, n in zip(axes, grid)]
    tab = np.concatenate([v for s, c in zip(sin, cos) for v in (s, c)] + tan)
    shape = tuple(len(a) for a in reversed(axes))
    q = np.zeros(shape + (3,), np.float32)
    assert lib.rotated_vectors((ctypes.c_int * 3)(*grid), _ptr(tab), len(tab), _ptr(q)) == 0
    s3, s2, s1 = np.meshgrid(*reversed(sin), indexing="ij")
    c3, c2, c1 = np.meshgrid(*reversed(cos), indexing="ij")
    p = np.stack([s1 * c2 * c3, c1 * s2 * c3, c1 * c2 * s3], axis=-1)
    c = (c1 * c2 * c3)[..., None]
    inner = c[..., 0] != 0
    assert np.all(np.abs(q * c - p)[inner] <= (2.0 ** -24 + 2.0 ** -48) * np.abs(p)[inner])
    assert np.array_equal(q[~inner], (p != 0)[~inner].astype(np.float32))
