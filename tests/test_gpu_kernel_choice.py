"""The kernels that the library chooses by itself (no tile asked for), at the
edges of their tiles, against exact integer arithmetic, FP32 arithmetic in the
defined order, or the kernel of an explicit tile: bit for bit throughout.
"""
import math

import numpy as np
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu


def run(k, u, n):
    a = torch.from_numpy(u).cuda()
    b = torch.zeros_like(a)
    res = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    fb = jacc.sweep(k, a, b, n, res)
    out = (b if fb else a).cpu().numpy(), (a if fb else b).cpu().numpy(), res.cpu().numpy()
    assert k.status() == 0
    return out


def faces2d(q):
    return (q[:-2, 1:-1] + q[2:, 1:-1]) + (q[1:-1, :-2] + q[1:-1, 2:])


# a warp's strip is 30 columns (odd widths) or 60 (even), a CTA's 30 to 240
@pytest.mark.parametrize("nx", [3, 4, 29, 31, 32, 33, 59, 60, 62, 121, 122, 241, 242])
@pytest.mark.parametrize("ny", [3, 4, 11, 34])
def test_jacobi2d_f64_strips_equal_integer_arithmetic(nx, ny):
    check_jacobi2d_f64(nx, ny, -1, False)


@pytest.mark.parametrize("nx", [4, 31, 62, 122])
@pytest.mark.parametrize("tile", [-1, 0, 1, 9])
def test_jacobi2d_f64_folded_strips_equal_integer_arithmetic(nx, tile):
    if tile in (1, 9) and nx % 2:
        tile = 2
    check_jacobi2d_f64(nx, 11, tile, True)


# the pre-pass reads 2048 values at a time: the largest on both sides of a block's end
@pytest.mark.parametrize("nx,ny", [(23, 89), (512, 4), (683, 3), (64, 64), (241, 17)])
@pytest.mark.parametrize("at", [0, 2047, -1])
def test_fixed_point_scale_follows_the_largest_value_wherever_it_is(nx, ny, at):
    check_jacobi2d_f64(nx, ny, -1, False, spike=min(at, nx * ny - 1))


def test_a_field_of_subnormals_takes_native_arithmetic():
    u = np.zeros((9, 62))
    u[4, 30] = 5e-324
    u[5, 31] = 4e-310
    g, _, gr = run(jacc.Kernel(jacc.STENCIL_5PT, jacc.F64, 62, 9, 1), u, 2)
    t, _, tr = run(jacc.Kernel(jacc.STENCIL_5PT, jacc.F64, 62, 9, 1, arith=jacc.ARITH_NATIVE), u, 2)
    assert np.array_equal(g, t) and np.array_equal(gr, tr)


def check_jacobi2d_f64(nx, ny, tile, jit, spike=None):
    u = 2.0 * inputs.uniform64(41, nx * ny).reshape(ny, nx) - 1.0
    if spike is not None:
        u.ravel()[spike] = -1000.0
    F = 57 - math.frexp(float(np.max(np.abs(u))))[1]
    k = jacc.Kernel(jacc.STENCIL_5PT, jacc.F64, nx, ny, 1, tile_id=tile, jit=jit)
    assert k.info()["fixed_point"]
    # |u| < 2^(57 - F): u 2^F is below 2^57, and its product and sums are exact
    q = np.trunc(np.ldexp(u, F)).astype(np.int64)
    resid = []
    for n in range(1, 5):
        s = faces2d(q)
        d = s - 4 * q[1:-1, 1:-1]
        resid.append(int(np.max(np.where(d < 0, -d - 1, d))))
        if n in (1, 2, 4):
            g, _, gr = run(k, u, n)
            want = u.copy() if n == 1 else np.ldexp(q.astype(np.float64), -F)  # a single sweep copies the boundary
            want[1:-1, 1:-1] = np.ldexp(s.astype(np.float64), -F - 2)          # int64 to FP64 rounds to nearest even
            assert np.array_equal(g, want)
            assert np.array_equal(gr, [math.ldexp(float(r), -F - 2) for r in resid])
        q = q.copy()
        q[1:-1, 1:-1] = (s + 2) >> 2


@pytest.mark.parametrize("nx", [3, 5, 29, 31, 33, 64, 119, 120, 124, 241, 244])
@pytest.mark.parametrize("ny", [3, 11, 34])
def test_jacobi2d_f32_strips_equal_ordered_fp32(nx, ny):
    u = (2.0 * inputs.uniform64(42, nx * ny).reshape(ny, nx) - 1.0).astype(np.float32)
    k = jacc.Kernel(jacc.STENCIL_5PT, jacc.F32, nx, ny, 1)
    g, _, gr = run(k, u, 3)
    resid = []
    for _ in range(3):
        v = u.copy()
        v[1:-1, 1:-1] = np.float32(0.25) * faces2d(u)
        resid.append(float(np.max(np.abs(v - u))))
        u = v
    assert np.array_equal(g, u)
    assert np.array_equal(gr, resid)


# sizes on both sides of the no-staging, ring and bulk-copy ranges; tile 0 has
# scalar columns, tile 1 16-byte ones
@pytest.mark.parametrize("nx,ny,nz", [(3, 3, 3), (31, 9, 5), (33, 17, 6), (64, 8, 9), (68, 10, 33), (129, 33, 40),
                                      (300, 200, 140), (301, 200, 140)])
@pytest.mark.parametrize("stencil", [jacc.STENCIL_7PT, jacc.STENCIL_27PT])
def test_f32_3d_choice_equals_table_tile(stencil, nx, ny, nz):
    u = (2.0 * inputs.uniform64(43, nx * ny * nz).reshape(nz, ny, nx) - 1.0).astype(np.float32)
    coeffs = (0.1,) if stencil == jacc.STENCIL_7PT else tuple(float(w) for w in inputs.box27_weights())
    tile = 1 if nx % 4 == 0 else 0
    g, o, gr = run(jacc.Kernel(stencil, jacc.F32, nx, ny, nz, coeffs=coeffs), u, 3)
    t, to, tr = run(jacc.Kernel(stencil, jacc.F32, nx, ny, nz, coeffs=coeffs, tile_id=tile), u, 3)
    assert np.array_equal(g, t) and np.array_equal(o, to)
    if stencil == jacc.STENCIL_7PT:
        assert np.array_equal(gr, tr)
    else:  # error-free per thread, then FP64 additions of the threads' parts in any order
        assert np.max(np.abs(gr - tr)) <= 1e-12 * float(np.sum(np.abs(u)))


@pytest.mark.parametrize("stencil,shape", [(5, (1, 9, 61)), (5, (1, 9, 62)), (7, (9, 17, 33)), (7, (9, 17, 64)),
                                           (7, (70, 130, 129)), (7, (70, 130, 130)), (27, (9, 17, 33))])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_f64_choice_takes_native_arithmetic_for_non_finite_fields(stencil, shape, bad):
    nz, ny, nx = shape
    u = 2.0 * inputs.uniform64(44, nx * ny * nz).reshape(shape) - 1.0
    u[nz // 2, ny // 2, nx // 2] = bad
    u = u[0] if stencil == 5 else u
    coeffs = {5: (0.0,), 7: (0.1,), 27: (0.5, 1 / 16, 1 / 128, 1 / 256)}[stencil]
    g, _, gr = run(jacc.Kernel(stencil, jacc.F64, nx, ny, nz, coeffs=coeffs), u, 2)
    t, _, tr = run(jacc.Kernel(stencil, jacc.F64, nx, ny, nz, coeffs=coeffs, arith=jacc.ARITH_NATIVE), u, 2)
    assert np.array_equal(g, t, equal_nan=True)
    assert np.array_equal(gr, tr, equal_nan=True)


# a folded grid that streams from HBM has more rows in flight and per warp
def test_jacobi2d_f64_large_folded_strips_equal_the_precompiled_kernel():
    nx, ny = 4098, 2051
    assert nx * ny > 1 << 23
    u = 2.0 * inputs.uniform64(46, nx * ny).reshape(ny, nx) - 1.0
    got = run(jacc.Kernel(jacc.STENCIL_5PT, jacc.F64, nx, ny, 1, jit=True), u, 3)
    want = run(jacc.Kernel(jacc.STENCIL_5PT, jacc.F64, nx, ny, 1, tile_id=1), u, 3)
    for g, w in zip(got, want):
        assert np.array_equal(g.view(np.int64), w.view(np.int64))


# the converting kernel has a plane count of its own where the library chooses
@pytest.mark.parametrize("nx,ny,nz", [(130, 66, 70), (131, 67, 71), (256, 200, 131)])
@pytest.mark.parametrize("stencil,coeffs", [(7, (0.125,)), (7, (0.1,)), (27, (0.5, 1 / 16, 1 / 128, 1 / 256))])
def test_f64_single_launch_equals_table_tile(stencil, coeffs, nx, ny, nz):
    u = 2.0 * inputs.uniform64(47, nx * ny * nz).reshape(nz, ny, nx) - 1.0
    g, _, gr = run(jacc.Kernel(stencil, jacc.F64, nx, ny, nz, coeffs=coeffs), u, 1)
    t, _, tr = run(jacc.Kernel(stencil, jacc.F64, nx, ny, nz, coeffs=coeffs, tile_id=0), u, 1)
    assert np.array_equal(g, t)
    if stencil == 7:
        assert np.array_equal(gr, tr)
    else:
        assert np.max(np.abs(gr - tr)) <= 1e-12 * float(np.sum(np.abs(u)))


def check_until(k, u, stops, most):
    _, _, r = run(k, u, most)
    assert np.all(np.diff(r) < 0)
    for stop in stops:
        a = torch.from_numpy(u).cuda()
        b = torch.zeros_like(a)
        res = torch.full((most,), -1.0, dtype=torch.float64, device="cuda")
        st = torch.full((2,), -7, dtype=torch.int32, device="cuda")
        tol = float(r[stop - 1]) if stop < most else 0.0
        jacc.sweep_until(k, a, b, most, tol, res, st)
        assert st.cpu().tolist() == [stop, stop % 2]
        want, other, wr = run(k, u, stop)
        g, o = (b, a) if stop % 2 else (a, b)
        assert np.array_equal(g.cpu().numpy(), want)
        if stop > 1:
            assert np.array_equal(o.cpu().numpy().view(np.uint8), other.view(np.uint8))
        assert np.array_equal(res.cpu().numpy(), np.concatenate([wr, np.full(most - stop, -1.0)]))


# chunks of 4 sweeps up to the 20th, then 5, 6, 7, ...: stops on, before and
# after their ends; 330 x 390 has more column pairs than a thread keeps items for
@pytest.mark.parametrize("nx,ny", [(3, 3), (70, 48), (71, 49), (129, 200), (330, 390)])
@pytest.mark.parametrize("arith", [jacc.ARITH_AUTO, jacc.ARITH_NATIVE])
def test_until_in_one_cluster_stops_anywhere_in_a_chunk(nx, ny, arith):
    y, x = np.meshgrid(np.sin(np.pi * np.arange(ny) / (ny - 1)), np.sin(np.pi * np.arange(nx) / (nx - 1)), indexing="ij")
    u = y * x + 1e-3 * y  # decays: strictly decreasing residuals
    k = jacc.Kernel(jacc.STENCIL_5PT, jacc.F64, nx, ny, 1, arith=arith)
    few = (nx, ny) == (3, 3)  # one interior point: at its fixed point after one sweep
    check_until(k, u, [1] if few else [1, 3, 4, 5, 8, 20, 21, 25, 26, 31, 60], 2 if few else 60)


@pytest.mark.parametrize("dtype", [jacc.F32, jacc.F64])
def test_until_in_guarded_sweeps_stops_anywhere_in_a_turn(dtype):
    nx, ny, nz = 33, 17, 9
    u = inputs.heat3d_field(nx, ny=ny, nz=nz, seed=45)
    u = u.astype(np.float32) if dtype == jacc.F32 else u
    k = jacc.Kernel(jacc.STENCIL_7PT, dtype, nx, ny, nz, coeffs=(0.125,))
    check_until(k, u, [1, 2, 15, 16, 17, 18, 33, 34, 50], 50)
