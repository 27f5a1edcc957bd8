"""Fields, residual and Nusselt numbers into every kind of memory a caller may
hand over (GPU): device arrays written in place, arrays that are not aligned
for their element, host arrays, a subset of the fields, none of them."""

import ctypes

import numpy as np
import pytest

import paper_1908_08386_gb300 as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("store", ["f32", "f64", "f32x2", "bf16"])
@pytest.mark.parametrize("wide", [False, True])
def test_fields_reach_every_kind_of_memory(store, wide):
    nx, ny = 75, 43
    c = L.Cavity(nx, ny, Ra=1e4, Pr=0.71, Ma=0.17, store=store)
    c.step(21)
    dt, call = (torch.float64, L.lbmfvm_fields) if wide else (torch.float32, L.lbmfvm_fields_f32)
    size = 8 if wide else 4
    host = [np.full((ny, nx), -7.0, np.float64 if wide else np.float32) for _ in range(4)]
    call(c.h, *host)
    dev = torch.full((4, ny, nx), -7.0, dtype=dt, device="cuda")
    call(c.h, *dev)
    assert np.array_equal(dev.cpu().numpy(), np.stack(host))
    # one byte off its alignment, in device memory
    raw = torch.zeros(4, nx * ny * size + 8, dtype=torch.uint8, device="cuda")
    fn = getattr(L.lib(), "lbmfvm_fields" if wide else "lbmfvm_fields_f32")
    assert fn(c.h, *[ctypes.c_void_p(raw[i].data_ptr() + 1) for i in range(4)]) == 0
    got = raw[:, 1:1 + nx * ny * size].cpu().numpy().copy().view(host[0].dtype).reshape(4, ny, nx)
    assert np.array_equal(got, np.stack(host))
    # some of them, from both kinds; none
    u = torch.zeros(ny, nx, dtype=dt, device="cuda")
    T = np.zeros((ny, nx), host[0].dtype)
    call(c.h, None, u, None, T)
    assert np.array_equal(u.cpu().numpy(), host[1]) and np.array_equal(T, host[3])
    call(c.h)
    pin = torch.zeros(ny, nx, dtype=dt).pin_memory()
    call(c.h, v=pin)
    assert np.array_equal(pin.numpy(), host[2])


def test_nusselt_and_residual_into_host_and_device_memory():
    c = L.Cavity(60, 50, Ra=1e4, Pr=0.71, Ma=0.17)
    c.step(30)
    loc = np.zeros(50)
    hot, cold = L.lbmfvm_nusselt(c.h, loc)
    d = torch.zeros(50, dtype=torch.float64, device="cuda")
    assert L.lbmfvm_nusselt(c.h, d) == (hot, cold) and L.lbmfvm_nusselt(c.h) == (hot, cold)
    assert np.array_equal(d.cpu().numpy(), loc)
    w = np.ones(50)
    w[0] = w[-1] = 0.5
    assert hot == pytest.approx((w * loc).sum() / 49, rel=1e-12)
    r = c.residual()
    assert r > 0 and c.residual() == 0.0  # against its own snapshot


def test_batch_fields_into_device_memory():
    from paper_1908_08386_gb300 import workloads as WL

    cases = [WL.CavityCase(40, 37, 1e4, 0.71, 0.17), WL.CavityCase(70, 33, 1e5, 0.71, 0.17)]
    b = L.Batch(cases, store="f16")
    b.step(25)
    for i, (ny, nx) in enumerate(b.shapes):
        want = np.stack(b.fields(i))
        out = torch.zeros(4, ny, nx, dtype=torch.float64, device="cuda")
        L._bcheck(L.lib().lbmfvm_batch_fields(b.b, i, *[L._addr(out[j]) for j in range(4)]), b.b)
        assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("store", ["f32", "f16", "f32x2", "f64"])
def test_batch_residuals_equal_the_single_handles(store):
    """One launch over all active cavities (one of more rows than a cavity has
    blocks, one at step 0, one that has left) against a handle each: the same
    sums in the same order, so they agree to a few roundings of the FP64 sums."""
    from paper_1908_08386_gb300 import workloads as WL

    mask = np.zeros((33, 70), np.uint8)
    mask[10:20, 20:40] = 1
    cases = [WL.CavityCase(40, 37, 1e4, 0.71, 0.17), WL.CavityCase(70, 33, 1e5, 0.71, 0.17, mask=mask),
             WL.CavityCase(20, 700, 1e6, 0.71, 0.05), WL.CavityCase(50, 50, 1e5, 7.0, 0.17)]
    b = L.Batch(cases, store=store, tma_config="default")
    singles = [L.Cavity(c.nx, c.ny, Ra=c.Ra, Pr=c.Pr, Ma=c.Ma, mask=c.mask, store=store) for c in cases]
    for n in (7, 12):
        b.step(n)
        got = b.residuals()
        for i, c in enumerate(singles):
            c.step(n)
            assert got[i] == pytest.approx(c.residual(), rel=1e-12), i
    b.set_state(3)  # back to step 0: its snapshot is its state
    got = b.residuals()
    assert got[3] == 0.0 and list(got[:3]) == [0.0] * 3
    b.close()
