"""jacc_sweep_until's graph: loops of shorter and longer turns one after the
other, stopped on, before and after the ends of their turns.
"""
import numpy as np
import pytest
from test_gpu_kernel_choice import check_until

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu


# turns of 4 sweeps up to the 17th, then of 16; 4 throughout from 2^22 points on
@pytest.mark.parametrize("shape,stops,most", [((33, 17, 9), list(range(1, 22)) + [32, 33, 34, 49, 50, 60], 60),
                                              ((164, 160, 160), [1, 2, 5, 6, 9], 10)])
@pytest.mark.parametrize("dtype", [jacc.F32, jacc.F64])
def test_until_stops_anywhere_in_a_turn_3d(dtype, shape, stops, most):
    nx, ny, nz = shape
    u = inputs.heat3d_field(nx, ny=ny, nz=nz, seed=45)
    u = u.astype(np.float32) if dtype == jacc.F32 else u
    check_until(jacc.Kernel(jacc.STENCIL_7PT, dtype, nx, ny, nz, coeffs=(0.125,)), u, stops, most)


# a graph is replayed with other fields' contents: what one run leaves set must not steer the next
def test_until_repeats_with_other_counts():
    import torch
    nx, ny = 70, 48
    y, x = np.meshgrid(np.sin(np.pi * np.arange(ny) / (ny - 1)), np.sin(np.pi * np.arange(nx) / (nx - 1)), indexing="ij")
    u = torch.from_numpy((y * x).astype(np.float32)).cuda()
    k = jacc.Kernel(jacc.STENCIL_5PT, jacc.F32, nx, ny, 1)
    a, b, w = u.clone(), torch.zeros_like(u), u.clone()
    r = torch.zeros(40, dtype=torch.float64, device="cuda")
    res, st = torch.zeros_like(r), torch.zeros(2, dtype=torch.int32, device="cuda")
    jacc.sweep(k, w, b, 40, r)
    tol = float(r[29])
    for scale in (1.0, 0.5, 4.0, 0.9, 2.0 ** -10, 1.0):
        w.copy_(u * scale)
        jacc.sweep(k, w, b, 40, r)
        hit = (r <= tol).nonzero()
        n = int(hit[0]) + 1 if len(hit) else 40
        a.copy_(u * scale)
        jacc.sweep_until(k, a, b, 40, tol, res, st)
        assert st.cpu().tolist() == [n, n % 2]
        assert torch.equal(res[:n], r[:n])
