"""Device-side waits that run out (GPU): the kernel gives up, the next
synchronising call reports it, and the handle and the context stay usable.
Nothing here faults or hangs: the hooks make a thread take a wait for one that
ran out, or leave out what it waits for."""

import numpy as np
import pytest

import paper_1908_08386_gb300 as L
from paper_1908_08386_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

KW = dict(nu=0.03, alpha=0.05, gbeta=1e-4)


def state(nx, ny, seed):
    u, v = WL.random_velocity(ny, nx, seed, 0.01)
    T = WL.random_temperature(ny, nx, seed + 1)
    return [a.astype(np.float32) for a in (u, v, T)]


def reports_and_recovers(c, ref, steps):
    """The armed call's failure is reported once; from a new state the handle
    computes what an undisturbed one does."""
    with pytest.raises(L.LbmfvmError) as e:
        c.residual()
    assert e.value.code == L.LBMFVM_ERR_TIMEOUT
    for h in (c, ref):
        h.set_state(*state(c.nx, c.ny, 5))
        h.step(steps)
    assert np.array_equal(np.stack(c.fields()), np.stack(ref.fields()))
    c.close()
    ref.close()


@pytest.mark.parametrize("store", ["f32", "f16"])
# fewer tiles than blocks' stages, several rounds of tiles, tiles drawn from the counter
@pytest.mark.parametrize("nx,ny", [(100, 60), (900, 700), (2000, 1500)])
def test_a_timeout_beside_the_end_mark_leaves_the_block(nx, ny, store):
    """Copying-warp shape: some threads of a block see the end of its tiles,
    others a wait that ran out; all of them leave."""
    kw = dict(KW, store=store, kernel="tma", tma_config=5)
    c = L.Cavity(nx, ny, **kw)
    L.lbmfvm_inject_fault(c.h, L.LBMFVM_FAULT_END)
    c.step(1)
    reports_and_recovers(c, L.Cavity(nx, ny, **kw), 9)


@pytest.mark.parametrize("nx,ny", [(100, 60), (900, 700)])
def test_a_lost_load_of_the_copying_warp_shape(nx, ny):
    kw = dict(KW, kernel="tma", tma_config=5)
    c = L.Cavity(nx, ny, **kw)
    L.lbmfvm_inject_stall(c.h)
    c.step(1)
    reports_and_recovers(c, L.Cavity(nx, ny, **kw), 9)


@pytest.mark.parametrize("store", ["f32", "f16", "f32x2", "f64"])
@pytest.mark.parametrize("fault,m", [("POST", 1), ("POST", 3), ("SUBPOST", 2), ("SUBPOST", 3)])
def test_a_border_that_is_never_posted_is_reported(store, fault, m):
    """Resident launches: the exchange of a step, of a step with energy
    sub-steps, and between the sub-steps of the last step, which no later
    exchange follows."""
    kw = dict(KW, alpha=0.05 * m, store=store, fv_substeps=m)
    c = L.Cavity(70, 90, **kw)
    L.lbmfvm_inject_fault(c.h, getattr(L, "LBMFVM_FAULT_" + fault))
    c.step(60)
    reports_and_recovers(c, L.Cavity(70, 90, **dict(kw, kernel="tma")), 33)


# two tiles; four and more across in x, in y and in both; shapes of one and of several nodes per thread
@pytest.mark.parametrize("nx,ny,store,m", [(20, 8, "f32", 1), (120, 20, "f32", 1), (20, 120, "f32", 3), (300, 280, "f32", 1),
                                           (300, 280, "f16", 2), (90, 60, "f32x2", 2), (60, 60, "f64", 1)])
def test_a_block_that_starts_late_is_waited_for(nx, ny, store, m):
    """A resident launch whose first block is kept off its SM for longer than
    the limit of a running exchange: every block waits for it, however far away."""
    kw = dict(KW, alpha=0.05 * m, store=store, fv_substeps=m)
    c, ref = L.Cavity(nx, ny, **kw), L.Cavity(nx, ny, kernel="tma", **kw)
    for h in (c, ref):
        h.set_state(*state(nx, ny, 9))
    L.lbmfvm_inject_fault(c.h, L.LBMFVM_FAULT_LATE)
    for n in (60, 9):
        c.step(n)
        ref.step(n)
    assert c.residual() == ref.residual()
    assert np.array_equal(np.stack(c.fields()), np.stack(ref.fields()))
    c.close()
    ref.close()


@pytest.mark.parametrize("store,m", [("f32", 1), ("f64", 2)])
def test_a_refused_resident_launch_leaves_ordinary_steps(store, m):
    kw = dict(KW, alpha=0.05 * m, store=store, fv_substeps=m)
    c, ref = L.Cavity(70, 90, **kw), L.Cavity(70, 90, kernel="tma", **kw)
    for h in (c, ref):
        h.set_state(*state(70, 90, 9))
    L.lbmfvm_inject_fault(c.h, L.LBMFVM_FAULT_REFUSED)
    for n in (60, 9):
        c.step(n)
        ref.step(n)
    assert c.steps == ref.steps == 69
    assert np.array_equal(np.stack(c.fields()), np.stack(ref.fields()))
    c.close()
    ref.close()


def test_hooks_of_kernels_that_are_not_in_use_are_refused():
    for kw in (dict(tma_config=4, kernel="tma"), dict(store="f64"), dict(kernel="generic")):
        c = L.Cavity(40, 40, **dict(KW, **kw))
        with pytest.raises(L.LbmfvmError) as e:
            L.lbmfvm_inject_fault(c.h, L.LBMFVM_FAULT_END)
        assert e.value.code == L.LBMFVM_ERR_ARG
        with pytest.raises(L.LbmfvmError) as e:
            L.lbmfvm_inject_fault(c.h, 99)
        assert e.value.code == L.LBMFVM_ERR_ARG
        with pytest.raises(L.LbmfvmError) as e:
            L.lbmfvm_inject_fault(c.h, L.LBMFVM_FAULT_SUBPOST)
        assert e.value.code == L.LBMFVM_ERR_ARG
        c.close()
