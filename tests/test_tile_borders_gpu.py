"""Step-kernel tiles that begin on a wall (GPU).  In FP32 arithmetic a node sees
the wall's own velocity across a border of the step kernel's tiles and the
extrapolated wall node's inside a tile; the two differ by rounding.  A resident
launch follows the borders of the step kernel that the handle would otherwise
run, so steps agree bit for bit however they are divided over calls; shapes of
equal borders agree bit for bit, and others to rounding."""

import numpy as np
import pytest

import paper_1908_08386_gb300 as L
from paper_1908_08386_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


def start(c, seed=3):
    u, v = WL.random_velocity(c.ny, c.nx, seed, 0.01)
    c.set_state(*[a.astype(np.float32) for a in (u, v, WL.random_temperature(c.ny, c.nx, seed + 1))])
    return c


# the last row (column) alone in a tile of 8 or 16 rows (64 columns), inside resident tiles of 16, 32 and 40 rows and at
# their borders
@pytest.mark.parametrize("nx,ny", [(100, 9), (65, 65), (256, 265), (257, 265), (321, 201), (300, 273), (503, 497), (610, 489), (640, 465),
                                   (600, 600)])
@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("scheme,m,lid", [("central", 1, 0.0), ("central", 1, 0.05), ("quick", 1, 0.0), ("central", 2, 0.0)])
def test_resident_steps_at_tile_borders_beside_walls(nx, ny, store, scheme, m, lid):
    kw = dict(nu=0.03, alpha=0.05 * m, gbeta=1e-4, force=(1e-6, -2e-6), store=store, fv_scheme=scheme, fv_substeps=m)
    if lid:
        A, M = L.LBMFVM_BC_ADIABATIC, L.LBMFVM_BC_MOVING
        kw.update(bc=(M, A, A, M), u_lid=lid)
    whole, parts, one = (start(L.Cavity(nx, ny, kernel=k, **kw)) for k in ("auto", "auto", "tma"))
    whole.step(60)
    one.step(60)
    for n in (9, 3, 40, 8):
        parts.step(n)
    want = np.stack(one.fields())
    assert np.array_equal(np.stack(whole.fields()), want)
    assert np.array_equal(np.stack(parts.fields()), want)
    for c in (whole, parts, one):
        c.close()


# a height that begins a tile of 16 rows, one that begins a tile of 8 only, one that begins neither
@pytest.mark.parametrize("nx,ny", [(150, 97), (129, 89), (334, 203)])
@pytest.mark.parametrize("store", ["f32", "f16"])
def test_shapes_with_a_body_force_at_tile_borders(nx, ny, store):
    """Both components of the force in every product and sum of the collision."""
    kw = dict(nu=0.03, alpha=0.05, gbeta=1e-4, force=(3e-6, -2e-6), store=store, t_ref=0.3, kernel="tma",
              mask=WL.rasterize([("circle", 0.4 * nx, 0.45 * ny, 0.31 * ny)], nx, ny))
    got = {}
    for cfg in range(6):
        c = start(L.Cavity(nx, ny, tma_config=cfg, **kw))
        c.step(37)
        got[cfg] = np.stack(c.fields())
        c.close()
    for cfg in (1, 4, 5):
        assert np.array_equal(got[cfg], got[0]), cfg
    for cfg in (2, 3):
        if (ny - 1) % 8 or (ny - 1) % 16 == 0:
            if cfg == 2 or (nx - 1) % 64:
                assert np.array_equal(got[cfg], got[0]), cfg
        # a wall velocity differs by at most a few ulp of the populations (2^-23 of 1/9 after division by rho about 1) and
        # moves T by its product with a temperature difference: below 2^-22 a step, 37 steps
        d = np.abs(got[cfg] - got[0])
        assert d.max() <= (37 * 2.0 ** -22 if store == "f32" else 2e-3), (cfg, d.max())
