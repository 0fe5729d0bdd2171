"""The folded FP32 27-point kernels staged by bulk copies, whose staged rows and
planes wrap once at most from as many rows on as a stage holds, against the
precompiled kernel of the same tile: bit for bit.
"""
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu
W = tuple(float(w) for w in inputs.box27_weights())


# a stage of tiles 1 and 3 holds 10 rows, of tile 13 18
@pytest.mark.parametrize("nx,ny,nz", [(4, 3, 3), (128, 9, 4), (132, 10, 3), (124, 11, 33), (4, 15, 34), (256, 17, 3),
                                      (136, 18, 5), (128, 19, 40)])
@pytest.mark.parametrize("tile", [1, 3, 13])
def test_folded_equals_precompiled(tile, nx, ny, nz):
    u = torch.from_numpy(2.0 * inputs.uniform64(52, nx * ny * nz).reshape(nz, ny, nx) - 1.0).float().cuda()
    out = []
    for jit in (False, True):
        k = jacc.Kernel(jacc.STENCIL_27PT, jacc.F32, nx, ny, nz, coeffs=W, tile_id=tile, jit=jit)
        a, b = u.clone(), torch.zeros_like(u)
        res = torch.full((3,), -1.0, dtype=torch.float64, device="cuda")
        assert jacc.sweep(k, a, b, 3, res) == 1
        assert k.status() == 0
        out.append((a, b, res))
    (a0, b0, r0), (a1, b1, r1) = out
    assert torch.equal(a0, a1) and torch.equal(b0, b1)
    # error-free per thread, then FP64 additions of the threads' parts in any order
    assert float((r0 - r1).abs().max()) <= 1e-12 * float(u.abs().sum(dtype=torch.float64))
