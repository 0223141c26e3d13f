"""What a process's first calls make the driver load and set up (host side, no
GPU: see _fake_host): the kernels that run, not all of a precision's."""
import pytest

from _fake_host import run

CASES = [("fp64", 128, 1.0, 0), ("fp32", 128, 1.0, 0), ("fp32", 512, 1.0, 0), ("fp32", 128, 0.8, 0),
         ("fp32", 512, 0.8, 0), ("fp16", 128, 1.0, 0), ("fp16", 256, 1.0, 0), ("fp16", 512, 1.0, 0),
         ("bf16", 512, 1.0, 16)]


@pytest.mark.parametrize("prec,n,tau,rows", CASES)
def test_first_calls_touch_what_they_run(prec, n, tau, rows):
    run(f"""
p = lb.make_params({n}, {n}, "{prec}", psi_form=1, tau_A={tau}, tau_B={tau}, tile_rows={rows})
h = lb.lb_create(p)
lb.lb_init_seeded(h, 1)
assert count("cudaFuncSetAttribute") == 0
(k,) = launches("k_init")
base = fk.fk_module(fk.fk_launch_name(k))
fk.fk_reset()
lb.lb_step(h, 3)
assert count("cudaFuncSetAttribute") == 2            # shared memory and carveout of one kernel
step = fk.fk_launch_name(launches("k_step")[0])
assert count("attribute " + step.decode()) == 2
m = fk.fk_module(step)
assert m != base and 0 < fk.fk_module_kernels(m, b"k_") <= 8     # one tile shape's variants
assert fk.fk_module_kernels(base, b"k_step") == 0    # initialise, observe, probes
fk.fk_reset()
lb.lb_step(h, 2)
lb.lb_stress(h)
lb.lb_stress(h)
assert count("cudaFuncSetAttribute") == 2             # the observe kernel, once
lb.lb_destroy(h)
""")


def test_pool_makes_its_kernel_ready_before_the_capture():
    run("""
p = lb.make_params(300, 200, "fp16", psi_form=1)
pool = lb.lb_pool_create(p, 64 << 20, 1)
lb.lb_pool_admit(pool, p, 1, 100)
fk.fk_fail(b"cudaStreamBeginCapture", 1, 900)
assert status(lb.lb_pool_prepare, pool) == lb.LB_ERR_CUDA
assert count("cudaFuncSetAttribute") == 2 and not launches("k_step")
lb.lb_pool_prepare(pool)
assert count("cudaFuncSetAttribute") == 2
lb.lb_pool_destroy(pool)
""")
