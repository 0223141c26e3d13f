"""Which host arrays the kernels read and write themselves (host side, no GPU: see
_fake_host): those that lie in one pinned allocation or registration as a
whole.  All others go through copies."""
import pytest

from _fake_host import run

# pinned: (offset, bytes) of the ranges that are pinned in a buffer that holds
# the array from byte 4096 on, `n` bytes long
CASES = {
    "whole": ("[(0, 4096 + n + 4096)]", True),
    "exact": ("[(4096, n)]", True),
    "pageable": ("[]", False),
    "first half": ("[(0, 4096 + n // 2)]", False),
    "last half": ("[(4096 + n // 2, n)]", False),
    "gap": ("[(0, 8192), (4096 + n - 4096, 8192)]", False),
    "two that meet": ("[(0, 4096 + n // 2), (4096 + n // 2, n)]", False),
    "one byte short": ("[(4096, n - 1)]", False),
}


@pytest.mark.parametrize("pinned", CASES)
def test_direct_only_inside_one_pinned_range(pinned):
    ranges, direct = CASES[pinned]
    run(f"""
nx, ny = 96, 80
p = lb.make_params(nx, ny, "fp32", psi_form=1)
h = lb.lb_create(p)
for planes, what in ((1, "fields"), (18, "pops")):
    n = 8 * planes * nx * ny
    raw = np.zeros(n + 16384, dtype=np.uint8)
    raw = raw[-raw.ctypes.data % 8:]
    base = raw.ctypes.data
    for at, size in {ranges}:
        fk.fk_pin(base + at, size)
    a = raw[4096:4096 + n].view(np.float64)
    lb.lb_init_seeded(h, 1)
    fk.fk_reset()
    if what == "fields":
        lb.lb_fields(h, a.reshape(ny, nx))
    else:
        lb.lb_populations(h, a)
    out = [fk.fk_launch_dst(k, 0) for k in launches("k_observe")]
    assert all((d == base + 4096) == {direct} for d in out) and out
    assert (count("cudaMemcpyAsync") == 1) == {direct}     # the counters alone
    fk.fk_reset()
    if what == "fields":
        lb.lb_init_fields(h, a.reshape(ny, nx), a.reshape(ny, nx))
    else:
        lb.lb_restore(h, a, 0, 0)
    assert (count("cudaMemcpyAsync") == 0) == {direct}
lb.lb_destroy(h)
""")
