"""The library's own choice for fields that stream from HBM, planes staged by
bulk copies, at the sizes that select it and with a last chunk of one plane,
against the kernel of tile 3: bit for bit.
"""
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu
W = tuple(float(w) for w in inputs.box27_weights())


# from 2^28 bytes a field on (7-point; FP64 folded only), or 2^30 (27-point FP32,
# folded); chunks of 16 planes (FP32 7-point), 40 and 32
@pytest.mark.parametrize("stencil,dtype,nx,ny,nz,planes,jit", [
    (7, 32, 512, 256, 513, 16, False), (7, 32, 512, 256, 513, 16, True), (7, 64, 512, 256, 361, 40, True),
    (27, 32, 1024, 512, 513, 32, True),
])
def test_bulk_copy_choice_equals_tile_3(stencil, dtype, nx, ny, nz, planes, jit):
    g = torch.Generator(device="cuda")
    g.manual_seed(56)
    t = torch.float64 if dtype == 64 else torch.float32
    u = torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=t)
    coeffs = W if stencil == 27 else (0.1,)
    own = jacc.Kernel(stencil, dtype, nx, ny, nz, coeffs=coeffs, jit=jit)
    tile = jacc.Kernel(stencil, dtype, nx, ny, nz, coeffs=coeffs, tile_id=3)
    assert own.info()["grid"][2] == (nz + planes - 1) // planes and nz % planes == 1
    for n in (1, 3):
        out = []
        for k in (own, tile):
            a, b = u.clone(), torch.zeros_like(u)
            res = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
            assert jacc.sweep(k, a, b, n, res) == 1
            assert k.status() == 0
            out.append((b, res))
        (x, rx), (y, ry) = out
        assert torch.equal(x, y)
        if stencil == 7:
            assert torch.equal(rx, ry)
        else:  # error-free per thread, then FP64 additions of the threads' parts in any order
            assert float((rx - ry).abs().max()) <= 1e-12 * float(u.sum(dtype=torch.float64))
