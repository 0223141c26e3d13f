"""FP64 work items are runs of rows, cut anywhere: next to a wall, inside the two
mirrored rows, single rows.  A pool with every partition gives bitwise the same
fields, populations' totals and wall stress as every other."""
import numpy as np
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


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("dims", [[(28, 8)], [(29, 9), (30, 10), (28, 11)], [(57, 17)], [(140, 31), (20, 33)],
                                  [(300, 121)], [(700, 333)]])
def test_fp64_partitions_agree(lb, dims, boundary):
    ps = [lb.make_params(nx, ny, "fp64", psi_form=1, boundary=boundary, u_wall=0.02 if boundary else 0.0,
                         tau_A=0.9, tau_B=1.1, stress_every=2) for nx, ny in dims]
    want = None
    for seg in (-1, 1, 2, 3, 64):
        pool = lb.Pool(ps[0], sum(map(lb.Pool.footprint, ps)), max_jobs=len(ps))
        pool.set_partition(seg)
        jobs = [pool.admit(p, seed=5, steps=9) for p in ps]
        while pool.run(4):
            pass
        got = [(pool.fields(j), pool.stress(j)) for j in jobs]
        assert pool.segment == seg
        pool.close()
        if want is None:
            want = got
        for (fa, sa), (fb, sb) in zip(got, want):
            assert all(np.array_equal(x, y) for x, y in zip(fa, fb)), seg
            assert sa == sb, seg


def test_larger_tables_while_steps_are_on_their_way(lb):
    """Partitions with more items than the pool's buffers were taken for, set while
    earlier steps are still enqueued."""
    p = lb.make_params(2048, 2048, "fp16", psi_form=1)
    g = lb.Lattice(p).init_seeded(3)
    g.step(120)
    pool = lb.Pool(p, lb.Pool.footprint(p), max_jobs=1)
    j = pool.admit(p, seed=3, steps=120)
    for seg in (-1, 1, 5, 2, 1, -1):
        pool.set_partition(seg)
        pool.run(20)
    assert all(np.array_equal(a, b) for a, b in zip(pool.fields(j), g.fields()))
    pool.close()
    g.close()
