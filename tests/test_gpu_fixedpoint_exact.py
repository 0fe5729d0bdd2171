"""The FP64 fixed-point sweeps against exact integer arithmetic, bit for bit.

Python integers evaluate the definition of the resident fixed-point form: the
input truncated onto the 2^-F grid, each intermediate sweep rounded to nearest
(ties up) on it, the last sweep's exact value rounded once to FP64.  Sizes sit
at the edges of the kernels' tiles (32 columns; 2 or 4 rows per thread) and of
their plane chunks; every residual must agree exactly too.
"""
from fractions import Fraction
import math

import numpy as np
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu


def frac_bits(u):
    return 57 - math.frexp(float(np.max(np.abs(u))))[1]


def to_fixed(u, F):
    return np.vectorize(lambda x: int(Fraction(float(x)) * 2 ** F), otypes=[object])(u)


def as_f64(q, E):
    """q 2^-E, correctly rounded."""
    return np.vectorize(lambda v: float(Fraction(int(v), 1) / 2 ** E), otypes=[np.float64])(q)


def weights(coeffs):
    """Integers w_j and K with coeffs[j] = w_j 2^-K exactly."""
    fr = [Fraction(float(c)) for c in coeffs]
    K = max(f.denominator.bit_length() - 1 for f in fr)
    return [int(f * 2 ** K) for f in fr], K


def round_up(x, k):
    return (x + (1 << (k - 1))) >> k if k else x


def box_sum(q, w):
    out = 0
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                out = out + np.roll(q, (dz, dy, dx), (0, 1, 2)) * w[abs(dz) + abs(dy) + abs(dx)]
    return out


def run(k, u, n):
    a = torch.from_numpy(u).cuda()
    b = torch.zeros_like(a)
    res = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    fb = jacc.sweep(k, a, b, n, res)
    return (b if fb else a).cpu().numpy(), res.cpu().numpy()


BOX_FP32 = tuple(float(w) for w in inputs.box27_weights())      # factors below 2^31
BOX_FP64 = (6 / 11, 1 / 22, 1 / 88, 1 / 176)                    # 53-bit factors
BOX_ONE = (1.0, 0.0, 0.0, 0.0)                                  # K = 0
BOX_EIGHTHS = (0.5, 1 / 16, 1 / 128, 1 / 256)                   # sums to 1 exactly


@pytest.mark.parametrize("coeffs", [BOX_FP32, BOX_FP64, BOX_ONE, BOX_EIGHTHS])
@pytest.mark.parametrize("shape", [(3, 3, 3), (5, 17, 33), (4, 15, 64), (18, 16, 32), (3, 33, 31)])
@pytest.mark.parametrize("tile,jit", [(-1, False), (0, False), (22, False), (-1, True)])
def test_box27_f64_equals_integer_arithmetic(coeffs, shape, tile, jit):
    nz, ny, nx = shape
    u = 2.0 * inputs.uniform64(31, nx * ny * nz).reshape(shape) - 1.0
    F = frac_bits(u)
    w, K = weights(coeffs)
    k = jacc.Kernel(jacc.STENCIL_27PT, jacc.F64, nx, ny, nz, coeffs=coeffs, tile_id=tile, jit=jit)
    assert k.info()["fixed_point"]
    q = to_fixed(u, F)
    sums = []
    for i in range(3):
        exact = box_sum(q, w)
        q = np.vectorize(lambda x: round_up(x, K), otypes=[object])(exact)
        sums.append(float(Fraction(int(q.sum()), 2 ** F)))
    g, gs = run(k, u, 3)
    assert np.array_equal(g, as_f64(exact, F + K))
    # the field sum: exact per thread, then FP64 additions of the threads' parts
    assert np.max(np.abs(gs - np.array(sums))) <= 1e-12 * float(np.sum(np.abs(u)))


def heat_sum(q):
    c = q[1:-1, 1:-1, 1:-1]
    return (q[1:-1, 1:-1, :-2] + q[1:-1, 1:-1, 2:] + q[1:-1, :-2, 1:-1] + q[1:-1, 2:, 1:-1] + q[:-2, 1:-1, 1:-1]
            + q[2:, 1:-1, 1:-1] - 6 * c)


@pytest.mark.parametrize("r", [0.125, 0.0625, 3 / 64, 0.1, 1 / 6, 0.003, 0.0])
@pytest.mark.parametrize("shape", [(3, 3, 3), (5, 17, 33), (9, 18, 64), (17, 16, 31), (4, 35, 97)])
@pytest.mark.parametrize("tile,jit", [(-1, False), (0, False), (3, False), (22, False), (-1, True)])
def test_heat3d_f64_equals_integer_arithmetic(r, shape, tile, jit):
    nz, ny, nx = shape
    if tile == 3 and nx % 2:
        tile = 2
    u = 2.0 * inputs.uniform64(32, nx * ny * nz).reshape(shape) - 1.0
    F = frac_bits(u)
    w, k2 = weights([r])
    k = jacc.Kernel(jacc.STENCIL_7PT, jacc.F64, nx, ny, nz, coeffs=(r,), tile_id=tile, jit=jit)
    assert k.info()["fixed_point"]
    inner = (slice(1, -1),) * 3
    q = to_fixed(u, F)
    resids = []
    for n in range(1, 5):
        exact = q * (1 << k2)
        exact[inner] = exact[inner] + w[0] * heat_sum(q)
        new = np.vectorize(lambda x: round_up(x, k2), otypes=[object])(exact)
        d = new - q
        resids.append(max(int(x) if x >= 0 else -int(x) - 1 for x in d[inner].ravel()))
        if n in (1, 2, 4):
            g, gr = run(k, u, n)
            want = as_f64(exact, F + k2)
            if n == 1:  # a single sweep copies the boundary
                edge = np.ones(shape, bool)
                edge[inner] = False
                want[edge] = u[edge]
            assert np.array_equal(g, want)
            assert np.array_equal(gr, as_f64(np.array(resids, dtype=object), F))
        q = new
    assert k.status() == 0
