"""lb_totals_noalloc where a thread sums many groups: a CTA takes chunks of 1024
sites, 608 CTAs at most, so a thread has up to 27 groups of four at 4096^2.  Its
64-bit sum of mantissas is rounded to FP64 after 32 terms of up to 2^58; the
densities here are such that 27 groups without that would overflow it: the
first groups, which set the reference, a quarter of the others.  And the edges
of a chunk.

Tolerance: a thread rounds its mass sums at most 5 times (27 groups, 8 at a time)
and its momenta 108 times, then follow 5 + 3 additions in the block, 3 slots a
thread and 8 more: below 300 roundings, |error| <= 300 2^-53 sum |terms|, as for
the smaller sizes."""
import numpy as np
import pytest

from test_totals_gpu import lb, totals  # noqa: F401

pytestmark = pytest.mark.gpu


def check(lb, nx, ny, a, b, ux, uy, shift=0):
    got = totals(lb, nx, ny, (a, b, ux, uy), shift)
    t = a + b
    for g, x in zip(got, (a, b, t * ux, t * uy)):
        exact = np.sum(x, dtype=np.longdouble)
        assert abs(g - exact) <= 300 * 2.0 ** -53 * np.abs(x).sum()


@pytest.mark.parametrize("nx,ny", [(4096, 4096), (2503, 2531), (4095, 1537)])
def test_many_groups_near_the_top_of_a_binade(lb, nx, ny):  # noqa: F811
    n = nx * ny
    rng = np.random.default_rng(n)
    first = 608 * 1024
    a, b = 4.0 * (1.0 - 2.0 ** -20 * rng.random((2, n)))
    a[:first] /= 4.0
    b[:first] /= 4.0
    ux, uy = 0.02 * rng.standard_normal((2, n))
    check(lb, nx, ny, a, b, ux, uy)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 8 * 1024 - 1, 8 * 1024 + 1, 608 * 1024 - 1, 608 * 1024,
                               608 * 1024 + 1, 609 * 1024])
def test_chunk_edges(lb, n, shift):  # noqa: F811
    rng = np.random.default_rng(n)
    a, b = 0.7 * (1 + 0.9 * (2 * rng.random((2, n)) - 1))
    ux, uy = 0.02 * rng.standard_normal((2, n))
    check(lb, n, 1, a, b, ux, uy, shift)
