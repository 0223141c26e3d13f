"""lb_totals_noalloc against exact sums at the sizes where its paths change:
one CTA and several, whole and partial chunks (2048 sites of a CTA at a time),
16-byte aligned arrays and not, densities on the integer path (positive, within
a factor 2^31) and off it (zero, negative, spread out, non-finite).

Tolerance: every partial sum is a chain of at most 8 fused operations per
chunk turn (at most 28 turns at the largest size), 5 shuffles, 8 warps and the
slots' chain, below 300 roundings in all, so |error| <= 300 2^-53 sum |terms|."""
import math

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


def totals(lb, nx, ny, arrays, shift=0):
    import torch
    n = nx * ny
    dev = []
    for a in arrays:
        t = torch.zeros(n + 2, dtype=torch.float64, device="cuda")
        t[shift:shift + n] = torch.from_numpy(a).cuda()
        dev.append(t)
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    lb.lb_totals_noalloc(nx, ny, *[t.data_ptr() + 8 * shift for t in dev], out.data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy()


@pytest.mark.parametrize("kind", ["densities", "mixed"])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2047, 1), (2048, 1), (2049, 1), (8192, 1), (8193, 1), (100, 333),
                                   (1024, 700)])
def test_totals_sizes(lb, nx, ny, shift, kind):
    n = nx * ny
    rng = np.random.default_rng(n + shift)
    a, b = 0.7 * (1 + 0.9 * (2 * rng.random((2, n)) - 1))
    ux, uy = 0.02 * rng.standard_normal((2, n))
    if kind == "mixed":   # some groups leave the integer path
        a[rng.random(n) < 0.1] = 0.0
        b[rng.random(n) < 0.1] *= -1.0
        a[rng.random(n) < 0.1] *= 2.0 ** -40
        b[rng.random(n) < 0.05] *= 2.0 ** -31
    got = totals(lb, nx, ny, (a, b, ux, uy), shift)
    t = a + b
    terms = (a, b, t * ux, t * uy)
    for g, x in zip(got, terms):
        assert abs(g - math.fsum(x)) <= 300 * 2.0 ** -53 * np.abs(x).sum() + n * 2.0 ** -1074


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_totals_nonfinite(lb, value):
    n = 5000
    a = np.full(n, 0.7)
    a[1234] = value
    got = totals(lb, n, 1, (a, np.full(n, 0.5), np.ones(n), np.zeros(n)))
    assert np.isnan(got[0]) if np.isnan(value) else np.isinf(got[0])
    assert abs(got[1] - 0.5 * n) <= 1e-12 * n
