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


def expm1_error(got, x, rho0):
    """Error relative to exp(-x/rho0) - 1, in 2^-52."""
    exact = np.expm1(-x.astype(np.longdouble) / np.longdouble(rho0))
    return ((got - exact) / exact * 2.0 ** 52).astype(np.float64)


@pytest.mark.parametrize("rho0", [0.51, 0.55, 0.6, 0.7, 0.83, 0.97, 0.1])
@pytest.mark.parametrize("amp", [1e-6, 1e-3, 0.03, 0.3, 0.9])
def test_expm1_is_as_good_as_the_library(lb, rho0, amp):
    """Half a unit each from 1/rho0, from the argument, and from the last of the
    operations that follow; the table and the series add less than a tenth.  The
    root mean square is no larger than that of the library's expm1 of the same
    argument (2 % for the sampling)."""
    assert np.finfo(np.longdouble).nmant >= 63
    rng = np.random.default_rng(11)
    x = amp * rho0 * (2.0 * rng.random(400_000) - 1.0)
    x = x[x != 0.0]
    ours, lib = probe(lb, x, x, rho0)[:2]
    e, el = expm1_error(ours, x, rho0), expm1_error(lib, x, rho0)
    print(f"rho0 {rho0} |x| <= {amp} rho0: max {np.abs(e).max():.3f} (library {np.abs(el).max():.3f}), "
          f"rms {np.sqrt((e * e).mean()):.4f} ({np.sqrt((el * el).mean()):.4f})")
    assert np.abs(e).max() <= 1.6
    assert np.sqrt((e * e).mean()) <= 1.02 * np.sqrt((el * el).mean())


def test_expm1_at_and_beyond_the_table(lb):
    """The table's ends (-x/rho0 = -3.47 and 2.07), its inner steps (the multiples
    of ln2/128), and the library outside, for huge and non-finite arguments too."""
    rho0 = 0.7
    steps = -rho0 * np.log(2.0) / 128.0 * np.arange(-641, 385)
    x = np.concatenate([steps, np.nextafter(steps, 1.0), np.nextafter(steps, -1.0), steps * (1 + 1e-9)])
    x = x[x != 0.0]
    ours, lib = probe(lb, x, x, rho0)[:2]
    tiny = np.abs(x) < np.finfo(np.float64).tiny   # (no relative error there)
    assert np.array_equal(ours[tiny], lib[tiny])
    assert np.abs(expm1_error(ours[~tiny], x[~tiny], rho0)).max() <= 1.6
    far = np.array([0.0, 2.6, 30.0, 500.0, 1e10, 1e300, np.inf, -1.5, -2.0, -400.0, -1e10, -1e300, -np.inf, np.nan])
    # (the pair's other value is inside the table: one outside takes both to the library)
    ours, lib = probe(lb, far, np.full(far.size, 0.01), rho0)[:2]
    assert np.array_equal(ours, lib, equal_nan=True)


@pytest.mark.parametrize("lo,hi", [(0.5, 2.5), (1e-6, 1e6), (1e-80, 1e80)])
@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e-150, 1e-290, 1e-310, 1e200])
def test_quotient_is_the_division(lb, lo, hi, scale):
    """Velocities, momentum / density: rounded as the division (but for the few
    reciprocals that are not, see above: four at most of 10^6)."""
    rng = np.random.default_rng(7)
    t = np.exp(np.log(lo) + (np.log(hi) - np.log(lo)) * rng.random(1_000_000))
    m = scale * (2.0 * rng.random(t.size) - 1.0)
    m[:100] = 0.0
    m[100:200] = -0.0
    got, want = probe(lb, t, m)[4:]
    assert np.count_nonzero(got != want) <= 4
    assert np.array_equal(np.signbit(got), np.signbit(want))


def test_quotient_special_values(lb):
    t = np.array([1.3, 1e-300, 1e300, -1.3, np.inf, 2e-310, np.nan])
    m = np.array([0.0, -0.0, 1.0, -2e-310, 1e308, -np.inf, np.nan])
    t, m = (a.ravel() for a in np.meshgrid(t, m))
    got, want = probe(lb, t, m)[4:]
    assert np.array_equal(got, want, equal_nan=True)
