"""Lattices whose 8-row tiles do not fill the SMs run the direct kernel (one
tile per SM at most, on 152 SMs), then the one-site tile kernel (up to 1.5), then
two CTAs per SM: each against the 16-row kernel, bitwise, at the smallest and
ragged sizes and on both sides of the lines (480 x 152: 152 tiles; 540 x 136:
153; 600 x 184: 230), over a first step from the initial state and later ones."""
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


def run(lb, m, prec, rows, steps):
    p = gpu_params(lb, m, prec)
    p.tile_rows = rows
    g = lb.Lattice(p).init_seeded(4)
    for n in steps:
        g.step(n)
    out = g.populations(), g.stress()
    g.close()
    return out


@pytest.mark.parametrize("prec,tau", [("fp32", (0.8, 1.0)), ("fp16", (1.0, 1.0)), ("fp16", (0.9, 0.8)),
                                      ("bf16", (1.0, 1.0))])
@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("nx,ny", [(8, 8), (9, 9), (59, 15), (61, 17), (120, 16), (480, 152), (540, 136), (600, 184)])
def test_few_tiles_bitwise(lb, nx, ny, boundary, prec, tau):
    m = model(nx, ny, boundary=boundary, u_wall=0.02 if boundary else 0.0, init_shear=boundary, tau=tau)
    a, b = run(lb, m, prec, 8, [1, 2, 18]), run(lb, m, prec, 16, [21])
    assert np.array_equal(a[0], b[0]) and a[1] == b[1]


@pytest.mark.parametrize("boundary", [0, 1])
def test_few_tiles_source_and_forces(lb, boundary):
    c = model(70, 41)
    m = model(70, 41, boundary=boundary, force_scheme=1, Ga=tuple(0.5 * v for v in c["Ga"]),
              Gr=tuple(0.5 * v for v in c["Gr"]), g_x=1e-4, kolmo_amp=2e-4, kolmo_k=1.0)
    a, b = run(lb, m, "fp32", 8, [25]), run(lb, m, "fp32", 16, [25])
    assert np.array_equal(a[0], b[0]) and a[1] == b[1]
