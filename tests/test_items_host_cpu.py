"""The work items of real step launches (host side, no GPU: see _fake_host, which
checks that every table lies inside its allocation and every item inside its
lattice): each row (FP64) or tile is updated once, and the tables hold the most
items a launch can have."""
import pytest

from _fake_host import run

COVER = """
def units(p, nlat_items, rows):
    n = {}
    for _, l, s, a, b in nlat_items:
        for u in range(a, b):
            n[l, s, u] = n.get((l, s, u), 0) + 1
    return n

def want(ps, tx, rows):
    return {(l, s, u): 1 for l, p in enumerate(ps) for s in range(-(-p.nx // tx)) for u in range(-(-p.ny // rows))}
"""

SIZES = [(8, 8), (28, 9), (29, 8), (84, 152), (28, 304), (112, 152), (85, 151), (128, 128), (61, 19),
         (300, 211), (512, 512), (1000, 37), (33, 2000)]


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("sms", [1, 7, 132, 152, 256, 1000])
def test_every_unit_once_and_tables_hold(prec, sms):
    """Lattice handles, on GPUs with few and many SMs; tables fit the workspace
    that lb_workspace_size asks for."""
    run(COVER + f"""
fk.fk_sms({sms})
tx, rows = (28, 1) if "{prec}" == "fp64" else (60, 8)
for nx, ny in {SIZES}:
    for tau in (1.0, 0.8):
        p = lb.make_params(nx, ny, "{prec}", psi_form=1, tau_A=tau, tau_B=tau, tile_rows=8)
        n = lb.lb_workspace_size(p)
        h = lb.lb_create_in(p, 0, fk.fk_device(n), n)
        lb.lb_init_seeded(h, 1)
        fk.fk_reset()
        lb.lb_step(h, 1)
        assert not fk.fk_errors(), (nx, ny, tau, fk.fk_errors())
        (k,) = launches("k_step")
        assert units(p, step_items(k), rows) == want([p], tx, rows), (nx, ny)
        lb.lb_destroy(h)
""")


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("seg", [0, -1, 1, 3])
def test_pool_covers_its_members(prec, seg):
    run(COVER + f"""
tx, rows = (28, 1) if "{prec}" == "fp64" else (60, 8)
ps = [lb.make_params(nx, ny, "{prec}", psi_form=1) for nx, ny in ((84, 152), (8, 8), (61, 37), (200, 24))]
pool = lb.lb_pool_create(ps[0], 64 << 20, 4)
lb.lb_pool_set_partition(pool, {seg})
lb.lb_pool_set_tile_rows(pool, 8)
for p in ps:
    lb.lb_pool_admit(pool, p, 1, 10)
    fk.fk_reset()
    lb.lb_pool_run(pool, 1)
(k,) = launches("k_step")
assert units(ps[0], step_items(k), rows) == want(ps, tx, rows)
lb.lb_pool_destroy(pool)
""")


def test_workspace_sizes_do_not_shrink_or_grow():
    """What callers were told to reserve stays enough, and a lattice handle's memory
    keeps its extent."""
    run("""
for (nx, ny, prec), n in {(64, 64, "fp64"): 1467392, (37, 155, "fp32"): 1589760, (128, 128, "fp16"): 1407744,
                          (512, 512, "fp32"): 38850048}.items():
    assert lb.lb_workspace_size(lb.make_params(nx, ny, prec)) == n, (nx, ny, prec)
""")
