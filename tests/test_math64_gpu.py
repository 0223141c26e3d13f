"""The FP64 functions of the step and of the fields next to CUDA's (through
lb_selftest_math64)."""
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


def probe(lb, x, y=None, rho0=0.7):
    """(expm1, library expm1, reciprocal, 1/x, quotient, y/x) of each argument"""
    import torch
    x = torch.from_numpy(np.array(x, dtype=np.float64)).cuda()
    y = torch.zeros_like(x) if y is None else torch.from_numpy(np.array(y, dtype=np.float64)).cuda()
    out = torch.empty(6 * x.numel(), dtype=torch.float64, device="cuda")
    lb.lb_selftest_math64(rho0, x.data_ptr(), y.data_ptr(), out.data_ptr(), x.numel(),
                          torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy().reshape(-1, 6).T


@pytest.mark.parametrize("lo,hi", [(0.5, 2.5), (1e-6, 1e6), (2.0 ** -1022, 2.0 ** -900), (2.0 ** 900, 2.0 ** 1021)])
def test_reciprocal_is_the_division(lb, lo, hi):
    """Rounded as the division, but for arguments whose reciprocal lies within
    2^-26 ulp of the middle between two numbers (the series' rest, 2^-79
    relative): none to be expected of 2 x 10^6, two at most."""
    rng = np.random.default_rng(5)
    x = np.exp(np.log(lo) + (np.log(hi) - np.log(lo)) * rng.random(2_000_000)) if hi > 10 * lo else \
        lo + (hi - lo) * rng.random(2_000_000)
    x[::2] *= -1.0
    _, _, r, want, _, _ = probe(lb, x)
    assert np.count_nonzero(r != want) <= 2


def test_reciprocal_special_values(lb):
    """Subnormal arguments and results, zeros, infinities: the division's."""
    tiny = np.finfo(np.float64).tiny
    x = np.array([tiny, tiny / 2, 2e-310, 5.6e-309, 4e-320, 5e-324, 0.0, -0.0, 2.0 ** 1020, 2.0 ** 1021, 8.9e307, 1e308,
                  np.finfo(np.float64).max, np.inf, -np.inf, -1e308, -2e-310, np.nan])
    _, _, r, want, _, _ = probe(lb, x)
    assert np.array_equal(r, want, equal_nan=True)
