"""Tile shapes whose threads take pairs of neighbouring nodes (GPU) against the
one that takes single nodes: the same roundings, so the same bits, with
obstacles that cut through pairs and tiles, rows and columns that end inside a
pair, and moving and adiabatic walls."""

import numpy as np
import pytest

import paper_1908_08386_gb300 as L
from paper_1908_08386_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny,moving", [(3, 3, False), (31, 18, False), (63, 50, True), (150, 90, False), (334, 203, True)])
def test_paired_shapes_equal_the_single_one(nx, ny, moving, store):
    mask = None
    if ny > 12:
        mask = WL.rasterize([("circle", 0.4 * nx, 0.45 * ny, 0.31 * ny), ("rect", 0.75 * nx, 0.6 * ny, 0.2 * nx, 0.15 * ny)],
                            nx, ny)
    kw = dict(nu=0.03, alpha=0.05, gbeta=1e-4, mask=mask, store=store, t_ref=0.3, kernel="tma")
    if moving:
        kw.update(bc=(L.LBMFVM_BC_DIRICHLET, L.LBMFVM_BC_DIRICHLET, L.LBMFVM_BC_ADIABATIC, L.LBMFVM_BC_MOVING), u_lid=0.04)
    u, v = WL.random_velocity(ny, nx, 3, 0.01)
    T = WL.random_temperature(ny, nx, 4)
    got = {}
    for cfg in (2, 1, 4, 5):
        c = L.Cavity(nx, ny, tma_config=cfg, **kw)
        c.set_state(u.astype(np.float32), v.astype(np.float32), T.astype(np.float32))
        c.step(37)
        got[cfg] = np.stack(c.fields())
        c.close()
    for cfg in (1, 4, 5):
        assert np.array_equal(got[cfg], got[2]), (cfg, np.abs(got[cfg] - got[2]).max())
