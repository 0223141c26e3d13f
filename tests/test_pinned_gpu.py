"""Fields, populations and initial states go between the device and pinned host
arrays directly (the kernels read and write them), and through copies for
pageable, unaligned or shared arrays: the same values either way, for every
output alone and together."""
import ctypes

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


def pinned(*shape):
    import torch
    return torch.zeros(shape, dtype=torch.float64, pin_memory=True).numpy()


def pinned_unaligned(n):
    """n doubles of pinned memory that start 4 bytes off a double's boundary."""
    import torch
    raw = torch.zeros(8 * n + 8, dtype=torch.uint8, pin_memory=True).numpy()
    return raw, raw.ctypes.data + 4


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("nx,ny,boundary", [(33, 17, 1), (100, 27, 0), (260, 136, 0)])
def test_pinned_equals_pageable(lb, prec, nx, ny, boundary):
    m = model(nx, ny, boundary=boundary, u_wall=0.02 if boundary else 0.0)
    rng = np.random.default_rng(2)
    src = [0.7 * (1 + 0.03 * (2 * rng.random((ny, nx)) - 1)) for _ in range(2)]
    src += [0.01 * rng.standard_normal((ny, nx)) for _ in range(2)]
    pin = [pinned(ny, nx) for _ in range(4)]
    for a, b in zip(pin, src):
        a[:] = b
    g, h = (lb.Lattice(gpu_params(lb, m, prec)) for _ in range(2))
    for nv in (0, 1, 2):   # without velocities, with u_x, with both
        g.init_fields(*src[:2 + nv]).step(7)
        lb.lb_init_fields(h.h, *pin[:2 + nv])
        h.step(7)
        want = g.fields()
        out = [pinned(ny, nx) for _ in range(4)]
        lb.lb_fields(h.h, *out)
        assert all(np.array_equal(a, b) for a, b in zip(out, want))
    for k in range(4):   # one at a time
        one = [pinned(ny, nx) if j == k else None for j in range(4)]
        lb.lb_fields(h.h, *one)
        assert np.array_equal(one[k], want[k])
    both = pinned(ny, nx)   # one array for two outputs: the later copy's values
    lb.lb_fields(h.h, both, None, None, both)
    assert np.array_equal(both, want[3])
    raw, addr = pinned_unaligned(nx * ny)
    st = lb.load().lb_fields(ctypes.c_void_p(h.h), ctypes.cast(addr, ctypes.POINTER(ctypes.c_double)), None, None,
                             None)
    assert st == lb.LB_OK
    assert np.array_equal(np.frombuffer(raw[4:4 + 8 * nx * ny].tobytes()).reshape(ny, nx), want[0])
    pops, state = pinned(2, 9, ny, nx), pinned(2, 9, ny, nx)
    lb.lb_populations(h.h, pops)
    assert np.array_equal(pops, g.populations())
    ref, t, pulled = g.checkpoint()
    assert lb.lb_checkpoint(h.h, state) == (t, pulled) and np.array_equal(state, ref)
    lb.lb_restore(h.h, state, t, pulled)
    g.resume(ref, t, pulled)
    assert all(np.array_equal(a, b) for a, b in zip(h.step(5).fields(), g.step(5).fields()))
    assert h.t == g.t == t + 5
    sg, sh = g.stress(), h.stress()
    assert sg == sh
    g.close()
    h.close()
