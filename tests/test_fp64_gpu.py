"""The FP64 step's table-driven exp(x) - 1 at and beyond the ends of its table
(-(rho - rho_ref)/rho0 in [-3.47, 2.08], the library function outside): populations against the FP64 oracle after three steps.  Tolerance 1e-13 relative to the largest
population: a step rounds each population through some 60 operations of at
most an ulp each, so three steps stay below 200 2^-53 = 2.2e-14 times the
force terms' cancellation, here below 4."""
import numpy as np
import pytest

from _pair import gpu_params, gpu_pops_as_oracle, model, oracle_params, rel_err

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


# (rho0, rho_ref or 0, lowest and highest density)
RANGES = [(0.7, 0.0, 0.01, 3.0), (0.1, 0.0, 0.42, 0.47), (0.1, 0.0, 0.3, 2.0), (0.5, 1.6, 0.4, 0.7)]


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("rho0,rho_ref,lo,hi", RANGES)
def test_fp64_density_range(lb, O, rho0, rho_ref, lo, hi, boundary):
    nx, ny = 61, 19
    m = model(nx, ny, rho0=rho0, Ga=(-0.05, -0.04), Gr=(0.04, 0.05), GX=0.02, boundary=boundary,
              u_wall=0.01 if boundary else 0.0)
    rng = np.random.default_rng(9)
    f0 = [lo + (hi - lo) * rng.random((ny, nx)) for _ in range(2)] + [0.01 * rng.standard_normal((ny, nx))
                                                                     for _ in range(2)]
    P = oracle_params(O, m)
    f = O.init_fields(P, *f0)
    O.run(P, f, 3)
    p = gpu_params(lb, m, "fp64")
    p.rho_ref = rho_ref
    g = lb.Lattice(p).init_fields(*f0)
    g.step(3)
    assert rel_err(gpu_pops_as_oracle(g.populations()), f) < 1e-13
    g.close()


@pytest.mark.parametrize("nx,ny", [(84, 152), (28, 304), (112, 152), (85, 151)])
def test_fp64_pool_with_more_items_than_tiles(lb, nx, ny):
    """A pool's FP64 work items are runs of rows: a small set has more of them
    than 8-row tiles (84 x 152: 152 items, 57 tiles).  Bitwise the lattice
    handle's populations."""
    p = lb.make_params(nx, ny, "fp64", psi_form=lb.LB_PSI_RHO0)
    g = lb.Lattice(p).init_seeded(4)
    g.step(5)
    pool = lb.Pool(p, 64 << 20, max_jobs=2)
    j = pool.admit(p, seed=4, steps=5)
    pool.run(5)
    ra, rb = pool.fields(j)[:2]
    ga, gb = g.fields()[:2]
    assert np.array_equal(ra, ga) and np.array_equal(rb, gb)
    pool.close()
    g.close()
