"""FP32 lattices at tau = 1 with the velocity shift are held by their moments
from the first step on (the default tile height); with a tile height asked
for they are held by their populations.  Both evaluate the same operations on
the same values, so populations, fields and wall stress are bitwise the same:
at the edges of the tiles, the smallest sizes, with walls and body forces, over
a change of form in a pool, and through checkpoint and restart."""
import numpy as np
import pytest

from _pair import gpu_params, model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("a CUDA GPU is required for -m gpu tests")
    import paper_0807_4471_gb300 as lb
    from paper_0807_4471_gb300 import build
    build.build()
    lb.load()
    return lb


def run(lb, m, rows, steps, seed=5):
    p = gpu_params(lb, m, "fp32")
    p.tile_rows = rows
    g = lb.Lattice(p).init_seeded(seed)
    for n in steps:
        g.step(n)
    out = g.populations(), g.fields(), g.checkpoint()[0], g.stress()
    g.close()
    return out


def same(a, b):
    return (np.array_equal(a[0], b[0]) and all(np.array_equal(x, y) for x, y in zip(a[1], b[1]))
            and np.array_equal(a[2], b[2]) and a[3] == b[3])


# around one and two tiles (60 x 8) and the wrap of the ring, the smallest
# lattices (loads wrap more than once), one and two CTAs per SM (1020 x 256)
@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 9), (8, 17), (59, 15), (60, 16), (61, 8), (121, 33), (63, 130),
                                   (1020, 256)])
def test_moments_equal_populations(lb, nx, ny, boundary):
    m = model(nx, ny, boundary=boundary, u_wall=0.02 if boundary else 0.0, init_shear=boundary)
    assert same(run(lb, m, 0, [1, 2, 40]), run(lb, m, 8, [43]))


@pytest.mark.parametrize("boundary", [0, 1])
def test_moments_with_body_forces(lb, boundary):
    m = model(130, 41, boundary=boundary, u_wall=0.01 if boundary else 0.0, g_x=1e-4, kolmo_amp=2e-4, kolmo_k=1.0)
    assert same(run(lb, m, 0, [30]), run(lb, m, 16, [30]))


def test_pool_changes_form(lb):
    """Default tiles, then a height asked for, then default again, with a
    member admitted in between; and a lattice restarted from a checkpoint of
    the moment form."""
    kw = [dict(nx=130, ny=40), dict(nx=64, ny=33, boundary=1, u_wall=0.02, init_shear=1)]
    with lb.Pool(gpu_params(lb, model(64, 64), "fp32"), budget=1 << 28, max_jobs=4) as pool:
        jobs = [pool.admit(gpu_params(lb, model(**k), "fp32"), 7 + i, 90) for i, k in enumerate(kw)]
        pool.run(30)
        pool.set_tile_rows(16)
        pool.run(21)
        late = pool.admit(gpu_params(lb, model(200, 24), "fp32"), 9, 39)
        pool.set_tile_rows(0)
        assert pool.run(39) == 0
        for j, k, seed, n in [(jobs[0], kw[0], 7, 90), (jobs[1], kw[1], 8, 90), (late, dict(nx=200, ny=24), 9, 39)]:
            want = run(lb, model(**k), 8, [n], seed)
            assert all(np.array_equal(x, y) for x, y in zip(pool.fields(j), want[1]))
            st = pool.stress(j)
            assert st["sigma_bot"] == want[3]["sigma_bot"] and st["samples"] == want[3]["samples"]
    p = gpu_params(lb, model(100, 30), "fp32")
    g = lb.Lattice(p).init_seeded(3).step(17)
    h = lb.Lattice(p).resume(*g.checkpoint())
    assert all(np.array_equal(x, y) for x, y in zip(g.step(20).fields(), h.step(20).fields()))


def test_nonfinite_density_is_latched(lb):
    ra = np.full((16, 64), 0.7)
    ra[3, 5] = np.nan
    g = lb.Lattice(gpu_params(lb, model(64, 16), "fp32")).init_fields(ra, np.full((16, 64), 0.7)).step(3)
    with pytest.raises(lb.LbError) as e:
        g.sync()
    assert e.value.status == lb.LB_ERR_NONFINITE
    g.close()
