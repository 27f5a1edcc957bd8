"""Many steps per launch with the state on the chip (GPU) against one launch
per step.

A handle whose kernel is left to the library keeps small cavities in shared
memory over a whole `step` call; naming the kernel gives one launch per step.
Both take the same arithmetic per node, so every field, the residual and the
Nusselt numbers agree bit for bit (sizes are kept off the one alignment where
the kernels' own tile shapes round differently: a tile border beside a wall).
"""

import numpy as np
import pytest

import paper_1908_08386_gb300 as L
from paper_1908_08386_gb300 import workloads as WL

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def state(nx, ny, seed):
    u, v = WL.random_velocity(ny, nx, seed, 0.01)
    T = WL.random_temperature(ny, nx, seed + 1)
    return [a.astype(np.float32) for a in (u, v, T)]


def obstacles(nx, ny):
    return WL.rasterize([("circle", 0.4 * nx, 0.45 * ny, 0.31 * ny), ("rect", 0.75 * nx, 0.6 * ny, 0.2 * nx, 0.15 * ny)],
                        nx, ny)


def outcome(c):
    r = c.residual()
    hot, loc, cold = c.nusselt()
    return np.stack(c.fields()), r, hot, cold, loc


def same(a, b):
    for x, y in zip(outcome(a), outcome(b)):
        assert np.array_equal(x, y), np.abs(np.asarray(x) - np.asarray(y)).max()


# one node inside the walls; a single tile, exactly and by a node more; ragged tiles of every shape up to the largest
# that fits (64 x 40 nodes on each of 152 SMs for 2-byte types, 64 x 32 for 4-byte, 32 x 16 for 8-byte), and beyond
SIZES = [(3, 3), (16, 8), (18, 11), (64, 64), (63, 130), (203, 127), (302, 200), (404, 344), (503, 500), (616, 480), (800, 454)]


@pytest.mark.parametrize("store", ["f32", "f16", "bf16", "f32x2", "f64"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_resident_steps_equal_one_launch_per_step(nx, ny, store):
    mask = obstacles(nx, ny) if min(nx, ny) > 12 else None
    kw = dict(nu=0.03, alpha=0.05, gbeta=1e-4, mask=mask, store=store, t_ref=0.3)
    a, b = L.Cavity(nx, ny, **kw), L.Cavity(nx, ny, kernel="tma", **kw)
    for c in (a, b):
        c.set_state(*state(nx, ny, 5))
    # below the limit, just above it, odd and even, and after ordinary steps of either parity
    for n in (3, 8, 9, 31, 1, 64):
        a.step(n)
        b.step(n)
        assert a.steps == b.steps
    same(a, b)
    a.close()
    b.close()


@pytest.mark.parametrize("store", ["f32", "f32x2", "f16", "f64"])
@pytest.mark.parametrize("scheme,m", [("quick", 1), ("central", 2), ("quick", 3)])
@pytest.mark.parametrize("nx,ny", [(18, 11), (63, 130), (302, 200)])
def test_resident_energy_options_equal_one_launch_per_step(nx, ny, scheme, m, store):
    kw = dict(nu=0.03, alpha=0.05 * m, gbeta=1e-4, mask=obstacles(nx, ny) if ny > 12 else None, store=store,
              fv_scheme=scheme, fv_substeps=m)
    a, b = L.Cavity(nx, ny, **kw), L.Cavity(nx, ny, kernel="tma", **kw)
    for c in (a, b):
        c.set_state(*state(nx, ny, 7))
    for n in (9, 22, 1):
        a.step(n)
        b.step(n)
    same(a, b)
    a.close()
    b.close()


def test_resident_walls_that_move_and_all_adiabatic():
    bc = (L.LBMFVM_BC_MOVING, L.LBMFVM_BC_ADIABATIC, L.LBMFVM_BC_ADIABATIC, L.LBMFVM_BC_MOVING)
    kw = dict(nu=0.02, alpha=0.03, gbeta=2e-4, force=(1e-6, -2e-6), bc=bc, u_lid=0.05)
    a, b = L.Cavity(100, 75, **kw), L.Cavity(100, 75, kernel="tma", **kw)
    for c in (a, b):
        c.set_state(*state(100, 75, 3))
        c.step(40)
    same(a, b)


def test_resident_batch_with_uneven_substeps_and_leaving_cavities():
    """Cavities of different sizes and numbers of sub-steps in one resident
    launch, and again after some have left it (a new, larger-area choice of
    tiles): equal to the batch pinned to one tile shape."""
    cases = [WL.CavityCase(n, k, Ra, 0.71, 0.1 * 3 ** 0.5) for n, k, Ra in
             ((40, 44, 1e3), (96, 63, 3e4), (70, 30, 1e5), (30, 90, 1e3))]
    runs = []
    for cfg in ("default", 1):
        b = L.Batch(cases, store="f32", tma_config=cfg, fv_substeps=0)
        assert len({b.substeps(i) for i in range(4)}) > 1
        b.step(77)
        r = [b.residuals()]
        b.run(tol=3e-3, check_every=200, max_steps=4000)
        b.step(33)
        r += [b.residuals()] + [np.stack(b.fields(i)) for i in range(4)] + [[b.info(i)[:2] for i in range(4)]]
        runs.append(r)
        b.close()
    for x, y in zip(*runs):
        assert np.array_equal(x, y)


def test_resident_launches_of_many_streams_and_threads():
    """Handles on streams of their own, stepped from threads at once: their
    launches go one after another, and each result is its own."""
    import threading

    kw = dict(nu=0.03, alpha=0.05, gbeta=1e-4)
    want, cav, done = [], [], []
    for i in range(4):
        ref = L.Cavity(150, 140 + i, kernel="tma", **kw)
        ref.set_state(*state(150, 140 + i, i))
        ref.step(300)
        want.append(np.stack(ref.fields()))
        ref.close()
        with torch.cuda.stream(torch.cuda.Stream()):
            c = L.Cavity(150, 140 + i, **kw)
            c.set_state(*state(150, 140 + i, i))
            cav.append(c)

    def go(i):
        for _ in range(30):
            cav[i].step(10)
        done.append((i, np.stack(cav[i].fields())))

    ts = [threading.Thread(target=go, args=(i,)) for i in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert len(done) == 4
    for i, got in done:
        assert np.array_equal(got, want[i]), i


def test_resident_run_resumes_from_a_checkpoint(tmp_path):
    kw = dict(nu=0.03, alpha=0.05, gbeta=1e-4)
    a, b = L.Cavity(90, 77, **kw), L.Cavity(90, 77, **kw)
    a.set_state(*state(90, 77, 1))
    a.step(45)
    a.save(str(tmp_path / "c"))
    b.load(str(tmp_path / "c"))
    for c in (a, b):
        c.step(50)
    same(a, b)


def test_resident_launch_beside_other_work_on_the_gpu():
    """Another stream keeps every SM busy while a resident launch comes up: its
    blocks start as SMs free up, and the result is the same."""
    kw = dict(nu=0.03, alpha=0.05, gbeta=1e-4)
    a, b = L.Cavity(300, 280, **kw), L.Cavity(300, 280, kernel="tma", **kw)
    m = torch.randn(8192, 8192, device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        for _ in range(300):
            out = m @ m
    for n in (9, 50, 200):
        a.step(n)
    for n in (9, 50, 200):
        b.step(n)
    same(a, b)
    del out
