"""The FP64 force's x and y components are equally exact.  On a field that is
symmetric under transposition the two differ only in how their stencil sums are
taken; smooth fields, where a sum is a small difference of large values, show
the order of subtraction and weighting.  At rest u = F / (2 rho).  The errors
against a longdouble evaluation of Eq. (2) come mostly from the inputs'
rounding, the same for both, and 6.5 x 10^4 sites settle the ratio of their root
mean squares to a per cent; 8 % is allowed (subtracting weighted columns instead
of weighting differences makes it 1.6 or more)."""
import numpy as np
import pytest

import lbinputs

pytestmark = pytest.mark.gpu
LD = np.longdouble


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


def exact_velocity(ra, rb, rho0):
    """u = (F_A + F_B) / (2 (rho_A + rho_B)) of Eq. (2), in longdouble."""
    c = lbinputs.CAPTION
    w = {1: LD(1) / 9, 2: LD(1) / 36}
    p = {1: LD(4) / 63, 2: LD(4) / 135, 4: LD(1) / 180, 5: LD(2) / 945, 8: LD(1) / 15120}
    r = [ra.astype(LD), rb.astype(LD)]
    psi = [LD(rho0) * -np.expm1(-q / LD(rho0)) for q in r]
    f = [np.zeros_like(r[0]), np.zeros_like(r[0])]

    def at(q, dx, dy):
        return np.roll(q, (-dy, -dx), (0, 1))

    for dx in range(-2, 3):
        for dy in range(-2, 3):
            d2 = dx * dx + dy * dy
            if d2 == 0:
                continue
            for s in range(2):
                k = LD(c["Gr"][s]) * p[d2] + (LD(c["Ga"][s]) * w[d2] if d2 <= 2 else 0)
                t = -k * psi[s] * at(psi[s], dx, dy)
                if d2 <= 2:
                    t = t - LD(c["GX"]) / LD(rho0) * w[d2] * r[s] * at(r[1 - s], dx, dy)
                f[0] = f[0] + dx * t
                f[1] = f[1] + dy * t
    return [q / (2 * (r[0] + r[1])) for q in f]


@pytest.mark.parametrize("amp,k", [(0.02, 1), (0.02, 3), (0.3, 1), (0.3, 4)])
def test_x_and_y_force_equally_exact(lb, amp, k):
    n, rho0 = 256, 0.7
    y, x = np.mgrid[0:n, 0:n]

    def field(shift):
        cx, cy = (np.cos(2 * np.pi * k * (v + shift) / n) for v in (x, y))
        return rho0 * (1 + amp / 1.3 * (cx + cy + 0.3 * np.cos(2 * np.pi * k * (x + y) / n)))

    ra, rb = field(0.0), field(31.0)
    assert np.allclose(ra, ra.T, rtol=1e-14) and np.allclose(rb, rb.T, rtol=1e-14)
    p = lb.make_params(n, n, "fp64", psi_form=lb.LB_PSI_RHO0, rho0=rho0)
    g = lb.Lattice(p).init_fields(ra, rb)
    _, _, ux, uy = g.fields()
    g.close()
    ex, ey = exact_velocity(ra, rb, rho0)
    rms = [float(np.sqrt(((a - b) ** 2).mean())) for a, b in ((ux, ex), (uy, ey))]
    print(f"amp {amp} k {k}: rms error of u_x {rms[0]:.3e}, of u_y {rms[1]:.3e}")
    assert rms[0] <= 1.08 * rms[1]
