"""7-point grids of very many planes: every kernel marches enough planes per
CTA to stay within a grid dimension's 65535 CTAs.  Compared bit for bit with
tile 2, whose 64 planes per CTA suffice throughout.
"""
import pytest
import torch

from paper_2110_14340_gb300 import jacc

pytestmark = pytest.mark.gpu


def field(dtype, nx, ny, nz):
    g = torch.Generator(device="cuda")
    g.manual_seed(51)
    return torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64 if dtype == 64 else torch.float32)


def run(k, u, n):
    a, b = u.clone(), torch.zeros_like(u)
    res = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    if n == 1:
        jacc.launch(k, a, b, res)
        fb = 1
    else:
        fb = jacc.sweep(k, a, b, n, res)
    assert k.status() == 0
    return (b if fb else a), res


# the first plane count of each kernel whose own planes per CTA give more than
# 65535 CTAs: no staging (2 planes), rings of 16 (FP32) and 24 planes (FP64), bulk
# copies of 16; scalar and 16-byte columns
@pytest.mark.parametrize("dtype,nx,ny,nz,tile,jit", [
    (32, 4, 3, 131071, -1, False), (64, 4, 3, 131071, -1, False),
    (32, 4, 3, 131074, -1, True), (64, 4, 3, 131074, -1, True),
    (32, 3, 3, 1048577, -1, False), (32, 8, 8, 1048592, -1, False),
    (64, 3, 3, 1572865, -1, False), (64, 4, 3, 1572865, -1, False),
    (32, 5, 3, 131073, 4, False), (32, 5, 3, 131073, 6, False),
    (64, 5, 3, 131073, 4, False), (64, 5, 3, 131073, 6, False),
])
def test_heat3d_of_many_planes_equals_the_64_plane_tile(dtype, nx, ny, nz, tile, jit):
    u = field(dtype, nx, ny, nz)
    k = jacc.Kernel(jacc.STENCIL_7PT, dtype, nx, ny, nz, coeffs=(0.1,), tile_id=tile, jit=jit)
    assert max(k.info()["grid"][1:]) <= 65535
    w = jacc.Kernel(jacc.STENCIL_7PT, dtype, nx, ny, nz, coeffs=(0.1,), tile_id=2)
    for n in (1, 3):
        got, gr = run(k, u, n)
        want, wr = run(w, u, n)
        assert torch.equal(got, want) and torch.equal(gr, wr)


@pytest.mark.parametrize("dtype", [32, 64])
def test_autotuner_times_every_tile_of_a_grid_of_many_planes(dtype):
    nx, ny, nz = 5, 3, 131073
    u = field(dtype, nx, ny, nz)
    jacc.autotune_forget()
    r = jacc.autotune(dict(stencil=7, dtype=dtype, nx=nx, ny=ny, nz=nz, coeffs=(0.1,)), u, torch.empty_like(u), 1, 1)
    assert r["valid"] == [not jacc.tile_info(t)["vec16"] for t in range(24)]
    jacc.autotune_forget()
