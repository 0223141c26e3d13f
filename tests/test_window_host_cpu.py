"""A step launch that fails part way through a call (host side, no GPU: see
_fake_host).  The launches of a call leave the step counters to the last one, so
a lattice whose call broke off has overwritten buffers under old counters: it
refuses work until it is initialised again."""
from _fake_host import run


def test_lattice_refuses_after_a_broken_call():
    run("""
p = lb.make_params(64, 48, "fp16", psi_form=1)
h = lb.lb_create(p)
lb.lb_init_seeded(h, 1)
lb.lb_step(h, 4)
fk.fk_fail(b"launch", 3, 700)
assert status(lb.lb_step, h, 5) == lb.LB_ERR_CUDA
a, f = np.zeros((48, 64)), np.zeros((2, 9, 48, 64))
fk.fk_reset()
for call in (lambda: lb.lb_step(h, 1), lambda: lb.lb_fields(h, a), lambda: lb.lb_stress(h),
             lambda: lb.lb_populations(h, f), lambda: lb.lb_checkpoint(h, f)):
    assert status(call) == lb.LB_ERR_STATE
assert not launches()
lb.lb_restore(h, f, 3, 1)
lb.lb_step(h, 2)
assert lb.lb_time(h) == 5
lb.lb_destroy(h)
""")


def test_lattice_goes_on_when_no_step_was_enqueued():
    run("""
h = lb.lb_create(lb.make_params(64, 48, "fp32", psi_form=1))
lb.lb_init_seeded(h, 1)
lb.lb_step(h, 4)
fk.fk_fail(b"launch", 1, 700)
assert status(lb.lb_step, h, 5) == lb.LB_ERR_CUDA
lb.lb_step(h, 2)
assert lb.lb_time(h) == 6
lb.lb_destroy(h)
""")


def test_pool_refuses_broken_members():
    run("""
p = lb.make_params(64, 48, "fp32", psi_form=1)
pool = lb.lb_pool_create(p, 64 << 20, 2)
j = [lb.lb_pool_admit(pool, p, s, 100) for s in (1, 2)]
lb.lb_pool_run(pool, 4)
fk.fk_fail(b"launch", 2, 700)
assert status(lb.lb_pool_run, pool, 5) == lb.LB_ERR_CUDA
assert lb.lb_pool_poll(pool, j[0]) == (4, False)
a = np.zeros((48, 64))
fk.fk_reset()
for call in (lambda: lb.lb_pool_run(pool, 1), lambda: lb.lb_pool_prepare(pool),
             lambda: lb.lb_pool_fields(pool, j[0], a), lambda: lb.lb_pool_stress(pool, j[1])):
    assert status(call) == lb.LB_ERR_STATE
assert not launches()
lb.lb_pool_init_fields(pool, j[0], a, a)
lb.lb_pool_release(pool, j[1])
lb.lb_pool_run(pool, 3)
assert len(launches("k_step")) == 3
lb.lb_pool_fields(pool, j[0], a)
lb.lb_pool_destroy(pool)
""")


def test_pool_books_the_steps_that_were_taken():
    """Whole graph chunks before the one that failed are steps taken."""
    run("""
p = lb.make_params(64, 48, "fp32", psi_form=1)
pool = lb.lb_pool_create(p, 64 << 20, 2)
j = lb.lb_pool_admit(pool, p, 1, 10000)
lb.lb_pool_prepare(pool)
fk.fk_fail(b"cudaGraphLaunch", 3, 700)
assert status(lb.lb_pool_run, pool, 100) == lb.LB_ERR_CUDA
assert lb.lb_pool_poll(pool, j) == (32, False)
lb.lb_pool_run(pool, 16)
assert lb.lb_pool_poll(pool, j) == (48, False)
lb.lb_pool_destroy(pool)
""")
