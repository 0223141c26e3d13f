"""FP64 where Psi's scale exp(-rho_ref/rho0) is small: its square, by which the
step's forces may be folded, leaves the range of FP64 numbers from
rho_ref/rho0 = 354 on; the scale itself stays within it to 708.  Fields and
populations against the FP64 oracle after three steps.  Tolerance: the window values
exp(-(rho - rho_ref)/rho0) - 1 carry the rounding of their argument, at most
700 x 3 x 2^-53 = 2.4e-13 relative, so forces are good to twice that times the
cancellation of a stencil sum (below 8 here), 4e-12; a population changes by
at most the force's share of it, below 1."""
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


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("psi_form", [0, 1])
@pytest.mark.parametrize("ratio", [40.0, 300.0, 345.0, 352.0, 400.0, 650.0])
def test_fp64_small_psi_scale(lb, O, ratio, psi_form, boundary):
    nx, ny, rho0 = 45, 21, 0.5
    # like-species forces of about a tenth of the density
    g = 0.1 if psi_form else 0.1 * rho0
    m = model(nx, ny, rho0=rho0, Ga=(-g, -0.8 * g), Gr=(0.8 * g, g), GX=0.05, boundary=boundary, psi_form=psi_form,
              u_wall=0.01 if boundary else 0.0)
    rng = np.random.default_rng(3)
    f0 = [rho0 * (0.5 + rng.random((ny, nx))) for _ in range(2)] + [0.01 * rng.standard_normal((ny, nx))
                                                                   for _ in range(2)]
    P = oracle_params(O, m)
    f = O.init_fields(P, *f0)
    O.run(P, f, 3)
    p = gpu_params(lb, m, "fp64")
    p.rho_ref = ratio * rho0
    h = lb.Lattice(p).init_fields(*f0)
    h.step(3)
    # populations are stored as offsets from w_i rho_ref: their ulp is that of rho_ref
    assert rel_err(gpu_pops_as_oracle(h.populations()), f) < 4e-12 + 60 * 2.0 ** -53 * ratio
    for a, b in zip(h.fields(), O.fields(P, f)):
        assert np.abs(a - b).max() < (4e-12 + 60 * 2.0 ** -53 * ratio) * max(1.0, np.abs(b).max())
    h.close()
