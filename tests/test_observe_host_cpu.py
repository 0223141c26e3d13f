"""Launch shape of the observables (host side, no GPU: see _fake_host)."""
import pytest

from _fake_host import run


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_totals_do_not_depend_on_the_gpu(prec):
    """lb_stress adds per-CTA sums: the CTAs, and with them the order of the
    additions, are the same on every GPU."""
    run(f"""
grids = set()
for sms in (7, 108, 152, 300):
    fk.fk_sms(sms)
    h = lb.lb_create(lb.make_params(2000, 700, "{prec}", psi_form=1))
    lb.lb_init_seeded(h, 1)
    fk.fk_reset()
    lb.lb_stress(h)
    (k,) = launches("k_observe")
    grids.add(fk.fk_launch_grid(k))
    lb.lb_destroy(h)
assert len(grids) == 1, grids
""")
