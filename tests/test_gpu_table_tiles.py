"""FP64 7-point table tiles with scalar columns, whose kernel and planes per CTA
follow the grid's size, against the bulk-copy kernel of tile 3: bit for bit.
"""
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu


# tiles 4 and 6 stage nothing up to 2^20 points; the others take fewer planes
# than their own (16 or 64) where the grid is small
@pytest.mark.parametrize("nx,ny,nz", [(34, 9, 5), (66, 33, 70), (128, 128, 64), (128, 128, 65), (130, 101, 131)])
@pytest.mark.parametrize("tile", [0, 4, 6, 10, 14, 22])
@pytest.mark.parametrize("r", [0.125, 0.1])
def test_heat3d_f64_scalar_tiles_equal_the_bulk_copy_tile(tile, nx, ny, nz, r):
    u = torch.from_numpy(2.0 * inputs.uniform64(53, nx * ny * nz).reshape(nz, ny, nx) - 1.0).cuda()
    for n in (1, 3):
        out = []
        for t in (tile, 3):
            k = jacc.Kernel(jacc.STENCIL_7PT, jacc.F64, nx, ny, nz, coeffs=(r,), tile_id=t)
            a, b = u.clone(), torch.zeros_like(u)
            res = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
            assert jacc.sweep(k, a, b, n, res) == 1
            assert k.status() == 0
            out.append((a, b, res))
        for x, y in zip(*out):
            assert torch.equal(x.view(torch.int64), y.view(torch.int64))
