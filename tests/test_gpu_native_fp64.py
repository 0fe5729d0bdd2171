"""FP64 handles that always run native arithmetic (JACC_ARITH_NATIVE, and
coefficients outside the fixed-point range), at the edges of their tiles,
against the definition in plain FP64.
"""
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def step(stencil, u, c):
    if stencil == 27:
        def near(t, d):
            return torch.roll(t, 1, d) + torch.roll(t, -1, d)
        x, y, z = near(u, 2), near(u, 1), near(u, 0)
        xy, xz, yz = near(x, 1), near(x, 0), near(y, 0)
        v = c[0] * u + c[1] * (x + y + z) + c[2] * (xy + xz + yz) + c[3] * near(xy, 0)
        return v, v.sum()
    v = u.clone()
    i = (slice(1, -1),) * u.dim()
    s = 0
    for d in range(u.dim()):
        for sl in (slice(None, -2), slice(2, None)):
            at = list(i)
            at[d] = sl
            s = s + u[tuple(at)]
    v[i] = 0.25 * s if stencil == 5 else u[i] + c[0] * (s - 6 * u[i])
    return v, (v - u).abs().max()


# widths on both sides of a tile's 32 to 256 columns, heights and depths of one
# row or plane over a tile's; a folded 5-point grid this small marches strips
@pytest.mark.parametrize("nx,ny,nz", [(3, 3, 3), (33, 9, 17), (62, 5, 65), (64, 17, 16), (65, 8, 18), (258, 11, 7)])
@pytest.mark.parametrize("tile,jit", [(-1, False), (-1, True), (0, False), (3, False), (3, True), (6, False), (14, False),
                                      (16, False), (21, False)])
@pytest.mark.parametrize("stencil,coeffs", [(5, ()), (7, (0.125,)), (7, (0.2,)), (27, (0.5, 1 / 16, 1 / 128, 1 / 256)),
                                            (27, (1.5, -0.1, 0.01, 0.0))])
def test_native_fp64_follows_the_definition(stencil, coeffs, tile, jit, nx, ny, nz):
    if nx % 2 and tile in (3, 21):
        tile -= 1
    nz = 1 if stencil == 5 else nz
    arith = jacc.ARITH_AUTO if coeffs in ((0.2,), (1.5, -0.1, 0.01, 0.0)) else jacc.ARITH_NATIVE
    k = jacc.Kernel(stencil, jacc.F64, nx, ny, nz, coeffs=coeffs, tile_id=tile, jit=jit, arith=arith)
    assert not k.info()["fixed_point"]
    u = torch.from_numpy(2.0 * inputs.uniform64(54, nx * ny * nz).reshape(k.shape) - 1.0).cuda()
    # sum of the coefficients' magnitudes: the growth of a value per sweep
    if stencil == 27:
        g = abs(coeffs[0]) + 6 * abs(coeffs[1]) + 12 * abs(coeffs[2]) + 8 * abs(coeffs[3])
    else:
        g = 1.0 if stencil == 5 else 1.0 + 12 * coeffs[0]
    # at most 30 roundings a value on either side, of terms below g per unit of input
    tol = [2 * 30 * EPS * g, 2 * 30 * EPS * (g * g + g * g)]
    a, b = u.clone(), torch.zeros_like(u)
    res = torch.full((2,), -1.0, dtype=torch.float64, device="cuda")
    assert jacc.sweep(k, a, b, 2, res) == 0
    v1, r1 = step(stencil, u, coeffs)
    v2, r2 = step(stencil, v1, coeffs)
    assert float((b - v1).abs().max()) <= tol[0]
    assert float((a - v2).abs().max()) <= tol[1]
    n = u.numel() if stencil == 27 else 2  # a sum over the field, or the difference of two values
    assert abs(float(res[0] - r1)) <= n * tol[0] and abs(float(res[1] - r2)) <= n * tol[1]
    out = torch.zeros_like(u)
    jacc.launch(k, u, out, res)
    assert torch.equal(out, b)


# the scalar 32 x 8 tiles stage nothing up to 2^24 points, the library's choice neither
@pytest.mark.parametrize("nx,ny,nz", [(161, 131, 101), (256, 256, 256), (257, 256, 256)])
@pytest.mark.parametrize("tile", [-1, 4, 6])
def test_native_heat3d_of_large_grids_equals_tile_0(tile, nx, ny, nz):
    g = torch.Generator(device="cuda")
    g.manual_seed(57)
    u = torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    out = []
    for t in (tile, 0):
        k = jacc.Kernel(7, jacc.F64, nx, ny, nz, coeffs=(0.1,), tile_id=t, arith=jacc.ARITH_NATIVE)
        a, b = u.clone(), torch.zeros_like(u)
        res = torch.full((3,), -1.0, dtype=torch.float64, device="cuda")
        assert jacc.sweep(k, a, b, 3, res) == 1
        out.append((a, b, res))
    for x, y in zip(*out):
        assert torch.equal(x, y)
