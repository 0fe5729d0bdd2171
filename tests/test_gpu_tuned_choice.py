"""What a handle runs after tuning, with no tile asked for: the fastest tile
where it is ahead of the library's own kernel, that kernel otherwise.
"""
import pytest
import torch

from paper_2110_14340_gb300 import inputs, jacc

pytestmark = pytest.mark.gpu
W = tuple(float(w) for w in inputs.box27_weights())


@pytest.fixture(autouse=True)
def forget():
    jacc.autotune_forget()
    yield
    jacc.autotune_forget()


def geometry(**args):
    i = jacc.Kernel(**args).info()
    return i["block"], i["grid"]


def fields(args):
    shape = jacc.Desc(**args).shape
    t = torch.float64 if args["dtype"] == 64 else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(55)
    return torch.rand(shape, generator=g, device="cuda", dtype=t), torch.zeros(shape, device="cuda", dtype=t)


def result(args):
    k = jacc.Kernel(**args)
    a, b = fields(args)
    assert jacc.sweep(k, a, b, 3) == 1
    return b


# grids on which the library's own kernel takes half of the fastest tile's time
CLEAR = [dict(stencil=27, dtype=32, nx=64, ny=64, nz=64, coeffs=W),
         dict(stencil=7, dtype=32, nx=301, ny=99, nz=97, coeffs=(0.1,)),
         dict(stencil=27, dtype=64, nx=48, ny=48, nz=48, coeffs=W)]


@pytest.mark.parametrize("args", CLEAR)
@pytest.mark.parametrize("jit", [False, True])
def test_tuning_does_not_displace_a_faster_kernel(args, jit):
    own, want = geometry(jit=jit, **args), result(args)
    a, b = fields(args)
    r = jacc.autotune(args, a, b, sweeps_per_rep=4, reps=3)
    assert geometry(jit=jit, **args) == own
    assert jacc.Kernel(**args).info()["tile_id"] == r["best_tile"]
    assert torch.equal(result(args), want)


@pytest.mark.parametrize("args", [dict(stencil=5, dtype=64, nx=511, ny=513), dict(stencil=7, dtype=64, nx=101, ny=99, nz=97,
                                                                                  coeffs=(0.125,))])
def test_a_tuned_handle_runs_the_pick_or_the_own_kernel(args):
    own, want = geometry(**args), result(args)
    a, b = fields(args)
    r = jacc.autotune(args, a, b, sweeps_per_rep=20, reps=5)
    assert geometry(**args) in (own, geometry(tile_id=r["best_tile"], **args))
    assert jacc.Kernel(**args).info()["tile_id"] == r["best_tile"]
    assert torch.equal(result(args), want)


def test_a_model_pick_is_named_and_displaces_nothing():
    args = CLEAR[0]
    own = geometry(**args)
    m = jacc.CostModel(seed=5)
    m.set_range(1.0, 4096.0, 0.0)
    t, fallback = m.choose(args)
    assert not fallback
    assert jacc.Kernel(**args).info()["tile_id"] == t
    assert geometry(**args) == own


# more rows than the own kernel's tile covers in a grid: only the tiles of eight
# thread rows and the long march do
def test_a_grid_that_only_large_tiles_cover_is_tuned():
    args = dict(stencil=5, dtype=32, nx=3, ny=4194305)
    with pytest.raises(jacc.JaccError):
        jacc.Kernel(**args)
    a, b = fields(args)
    r = jacc.autotune(args, a, b, sweeps_per_rep=1, reps=1)
    assert r["valid"][6] and not r["valid"][2]
    assert torch.equal(result(args), result(dict(args, tile_id=6)))
    jacc.autotune_forget()
    m = jacc.CostModel(seed=5)
    m.set_range(1.0, 1e9, 0.0)
    t, fallback = m.choose(args)
    assert not fallback and jacc.Kernel(**args).info()["tile_id"] == t
