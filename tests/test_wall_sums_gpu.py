"""Wall stress sums over windows of steps: a launch adds up the previous step's
wall momentum, a window's last launch its own too, so the sums may not depend
on how a run is cut into windows.  Bitwise: the order of additions is the same."""
import pytest

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


def params(lb, precision, nx, ny, tau, every, t0=2):
    return lb.make_params(nx, ny, precision, psi_form=lb.LB_PSI_RHO0, boundary=lb.LB_COUETTE, u_wall=0.02,
                          init_shear=1, tau_A=tau, stress_every=every, stress_t0=t0)


# direct, moment, tile and two-CTA kernels; one row of tiles, ragged strips
CASES = [("fp16", 61, 8, 1.0), ("fp32", 61, 9, 0.8), ("fp32", 130, 50, 1.0), ("fp32", 700, 500, 1.0),
         ("fp32", 700, 300, 0.8), ("fp16", 700, 300, 1.0), ("bf16", 700, 500, 0.8), ("fp64", 61, 19, 1.0),
         ("fp64", 500, 130, 0.8)]


@pytest.mark.parametrize("every", [1, 3])
@pytest.mark.parametrize("precision,nx,ny,tau", CASES)
def test_sums_do_not_depend_on_windows(lb, precision, nx, ny, tau, every):
    p = params(lb, precision, nx, ny, tau, every)
    out = []
    for windows in ([1] * 11, [11], [3, 2, 6], [2, 9]):
        g = lb.Lattice(p).init_seeded(7)
        for n in windows:
            g.step(n)
        out.append(g.stress())
        g.close()
    assert out[0]["samples"] > 0
    assert out[1:] == out[:1] * 3


@pytest.mark.parametrize("precision,tau", [("fp32", 1.0), ("fp32", 0.8), ("fp16", 1.0), ("fp64", 1.0)])
def test_pool_sums_are_the_lattices(lb, precision, tau):
    ps = [params(lb, precision, 130, 50, tau, 1), params(lb, precision, 61, 97, tau, 2, 3),
          params(lb, precision, 300, 40, tau, 3, 0)]
    pool = lb.Pool(ps[0], 256 << 20, max_jobs=4)
    jobs = [pool.admit(p, seed=5, steps=600) for p in ps]
    for n in (1, 7, 592):   # (the last through a captured graph)
        pool.run(n)
    for p, j in zip(ps, jobs):
        g = lb.Lattice(p).init_seeded(5)
        g.step(600)
        assert pool.stress(j) == g.stress()
        g.close()
    pool.close()
