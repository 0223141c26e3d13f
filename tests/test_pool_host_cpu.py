"""Host side of the lattice pool, without a GPU (see _fake_host)."""
import pytest

from _fake_host import run

GROW = """
small = lb.make_params(40, 40, "fp64", psi_form=1)
big = lb.make_params(600, 900, "fp64", psi_form=1)
pool = lb.lb_pool_create(small, 1 << 30, 4)
j = lb.lb_pool_admit(pool, small, 1, 1000)
lb.lb_pool_run(pool, 3)
assert lb.lb_pool_segment(pool) == -1
lb.lb_pool_admit(pool, big, 2, 1000)      # more items than the tables hold
"""


@pytest.mark.parametrize("api", ["cudaMalloc", "cudaMemcpyAsync"])
def test_failed_prepare_leaves_the_pool_unbuilt(api):
    """A member set whose launch could not be built has none: the next run builds
    it, and does not step the previous set's launch."""
    run(GROW + f"""
fk.fk_fail(b"{api}", 1, 2)
assert status(lb.lb_pool_prepare, pool) == lb.LB_ERR_NOMEM
assert lb.lb_pool_segment(pool) == 0 and lb.lb_pool_tile_rows(pool) == 0
fk.fk_reset()
lb.lb_pool_run(pool, 5)
steps = launches("k_step")
assert len(steps) == 5
assert {{i[1] for i in step_items(steps[0])}} == {{0, 1}}     # both members
lb.lb_pool_destroy(pool)
""")


def test_pool_runs_on_after_a_failed_growth():
    """No room for larger item tables: the smaller set runs once the large member
    is gone."""
    run(GROW + """
fk.fk_reset()
fk.fk_fail(b"cudaMalloc", 1, 2)
assert status(lb.lb_pool_run, pool, 5) == lb.LB_ERR_NOMEM
assert not launches("k_step")
lb.lb_pool_release(pool, 1)
lb.lb_pool_run(pool, 5)
assert len(launches("k_step")) == 5
lb.lb_pool_destroy(pool)
""")


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("sizes", [[(128, 128)], [(64 + 8 * k, 200 - 5 * k) for k in range(24)],
                                   [(512, 512)] * 40, [(4096, 4096)], [(2048, 2048), (30, 3000)]])
def test_runs_allocate_nothing(prec, sizes):
    """The buffers a launch's tables go through are there before the first run of a
    member set; a run neither allocates nor frees (either may wait for the steps
    that are enqueued)."""
    run(f"""
ps = [lb.make_params(nx, ny, "{prec}", psi_form=1) for nx, ny in {sizes}]
pool = lb.lb_pool_create(ps[0], sum(map(lb.lb_pool_footprint, ps)), len(ps))
for p in ps:
    lb.lb_pool_admit(pool, p, 1, 100)
    fk.fk_reset()
    lb.lb_pool_run(pool, 2)
    assert len(launches("k_step")) == 2
    for api in ("cudaHostAlloc", "cudaFreeHost", "cudaEventCreate"):
        assert count(api) == 0, api
fk.fk_reset()
lb.lb_pool_destroy(pool)
""")


def test_larger_tables_keep_the_old_buffers():
    """Partitions with more items than the buffers hold (one tile each): new buffers,
    and the old ones, out of which copies may be on their way, stay to the end."""
    run("""
p = lb.make_params(4096, 2048, "fp16", psi_form=1)
pool = lb.lb_pool_create(p, lb.lb_pool_footprint(p), 1)
lb.lb_pool_admit(pool, p, 1, 100)
lb.lb_pool_run(pool, 2)
lb.lb_pool_set_partition(pool, 1)
fk.fk_reset()
lb.lb_pool_run(pool, 2)
assert count("cudaHostAlloc") == 1 and count("cudaFreeHost") == 0
assert len(step_items(launches("k_step")[0])) == 69 * 256
lb.lb_pool_destroy(pool)
assert count("cudaFreeHost") == 2
""")


def test_pool_runs_without_pinned_memory():
    """No pinned memory to be had: tables go through pageable memory, as they do for
    a lattice handle."""
    run("""
p = lb.make_params(64, 48, "fp32", psi_form=1)
fk.fk_fail(b"cudaHostAlloc", 1, 2)
pool = lb.lb_pool_create(p, 64 << 20, 2)
for seed in (1, 2):
    fk.fk_fail(b"cudaHostAlloc", 1, 2)
    lb.lb_pool_admit(pool, p, seed, 100)
    fk.fk_reset()
    fk.fk_fail(b"cudaHostAlloc", 1, 2)
    lb.lb_pool_run(pool, 3)
    assert len(launches("k_step")) == 3 and count("cudaStreamSynchronize") >= 1
fk.fk_fail(b"cudaHostAlloc", 1 << 30, 2)
lb.lb_pool_set_partition(pool, 1)
fk.fk_reset()
lb.lb_pool_run(pool, 3)
assert count("cudaStreamSynchronize") == 0       # pinned again
lb.lb_pool_destroy(pool)
""")
