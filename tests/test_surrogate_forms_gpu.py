"""The surrogate's elementwise and output-layer kernels in the two forms that
their entry points choose between (GPU): 16-byte words for aligned slices whose
channels come in eights, single elements for every other slice.  Both compute
the same rounded values, so the elementwise results are equal bit for bit and
the output layer's FP32 sums agree to their own rounding."""

import numpy as np
import pytest

from oracle import surrogate_ref as R
from paper_1908_08386_gb300 import surrogate as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def slice_of(a, pad):
    """`a` (BF16, NHWC) as a channel slice: pad = 0 dense, 8 an aligned slice of
    a wider tensor, 1 a slice that no 16-byte word fits."""
    B, H, W, C = a.shape
    t = torch.zeros(B, H, W, C + 2 * pad, dtype=torch.bfloat16, device="cuda")
    v = t[..., pad:pad + C]
    v.copy_(a)
    return t, v, t.data_ptr() + 2 * pad, C + 2 * pad


def rand(rng, *s):
    return torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda().to(torch.bfloat16)


# one pixel pair; odd pixel counts in every dimension; the last block partly filled; 8 and 160 channels
@pytest.mark.parametrize("B,H,W,C", [(1, 2, 2, 8), (3, 6, 10, 24), (2, 16, 32, 32), (1, 8, 18, 160)])
def test_word_and_element_forms_agree(B, H, W, C):
    rng = np.random.default_rng(B + H + W + C)
    x, dy, up = rand(rng, B, H, W, C), rand(rng, B, H // 2, W // 2, C), rand(rng, B, 2 * H, 2 * W, C)
    add, m = rand(rng, B, H, W, C), rand(rng, B, H, W, C)
    got = {}
    for pad in (0, 8, 1):
        z = lambda *s: slice_of(torch.zeros(*s, dtype=torch.bfloat16, device="cuda"), pad)
        held = [slice_of(t, pad) for t in (x, dy, up, add, m)]  # the slices stay alive until the kernels have run
        (xp, ldx), (dp, ldd), (upp, ldu), (ap, lda), (mp, ldm) = (h[2:] for h in held)
        t1, y1, p1, l1 = z(B, H // 2, W // 2, C)
        S.call("lbmfvm_sg_pool2", xp, ldx, p1, l1, B, H, W, C, S._stream())
        outs = [y1]
        for a, mm in ((ap, mp), (None, None), (ap, None), (None, mp)):
            t2, y2, p2, l2 = z(B, H, W, C)
            S.call("lbmfvm_sg_pool2_backward", dp, ldd, a, lda, mm, ldm, p2, l2, B, H, W, C, S._stream())
            outs.append(y2)
        t3, y3, p3, l3 = z(B, 2 * H, 2 * W, C)
        S.call("lbmfvm_sg_upsample2", xp, ldx, p3, l3, B, H, W, C, S._stream())
        outs.append(y3)
        for mm in (mp, None):
            t4, y4, p4, l4 = z(B, H, W, C)
            S.call("lbmfvm_sg_upsample2_backward", upp, ldu, mm, ldm, p4, l4, B, H, W, C, S._stream())
            outs.append(y4)
        torch.cuda.synchronize()
        for t in (t1, t3):  # nothing outside the slices
            if pad:
                assert not t[..., :pad].any() and not t[..., pad + C:].any()
        got[pad] = [o.clone() for o in outs]
    for k in range(len(got[1])):
        assert torch.equal(got[0][k], got[1][k]) and torch.equal(got[8][k], got[1][k]), k


@pytest.mark.parametrize("P,C,CO,pad", [(1, 32, 3, 0), (63, 32, 3, 8), (65, 64, 3, 0), (100003, 32, 3, 0), (257, 64, 3, 8),
                                        (300, 32, 3, 1), (77, 24, 3, 0), (77, 16, 2, 0), (130, 64, 8, 0)])
def test_output_layer_over_its_forms(P, C, CO, pad):
    rng = np.random.default_rng(P + C + CO)
    xt, xv, xp, ldx = slice_of(rand(rng, 1, 1, P, C), pad)
    f = lambda *s: torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
    w, b, dy = f(CO, C), f(CO), f(P, CO)
    y = torch.zeros(P, CO, device="cuda")
    S.call("lbmfvm_sg_conv1x1", xp, ldx, w.data_ptr(), b.data_ptr(), y.data_ptr(), P, C, CO, S._stream())
    dxt, dxv, dxp, lddx = slice_of(torch.zeros(1, 1, P, C, dtype=torch.bfloat16, device="cuda"), pad)
    dw, db = torch.ones(CO, C, device="cuda"), torch.ones(CO, device="cuda")  # added to
    S.call("lbmfvm_sg_conv1x1_backward", xp, ldx, w.data_ptr(), dy.data_ptr(), dxp, lddx, dw.data_ptr(), db.data_ptr(),
           P, C, CO, S._stream())
    dw2 = torch.ones(CO, C, device="cuda")  # neither dx nor db
    S.call("lbmfvm_sg_conv1x1_backward", xp, ldx, w.data_ptr(), dy.data_ptr(), None, 0, dw2.data_ptr(), None, P, C, CO,
           S._stream())
    torch.cuda.synchronize()
    h = lambda t: t.double().cpu().numpy()
    xr, wr, dyr = h(xv).reshape(P, C), h(w), h(dy)
    ulp = 2.0 ** -23
    # a sum of n FP32 products: at most about n / 2 ulp of the sum of their sizes
    assert np.all(np.abs(h(y) - (xr @ wr.T + h(b))) <= (C + 1) * ulp * (np.abs(xr) @ np.abs(wr).T + np.abs(h(b))))
    for got in (dw, dw2):
        assert np.all(np.abs(h(got) - 1 - dyr.T @ xr) <= (P + 1) * ulp * (np.abs(dyr).T @ np.abs(xr) + 1))
    assert np.all(np.abs(h(db) - 1 - dyr.sum(0)) <= (P + 1) * ulp * (np.abs(dyr).sum(0) + 1))
    ref = R.leaky_backward(xr, dyr @ wr)
    assert np.abs(h(dxv).reshape(P, C) - ref).max() <= 2.0 ** -8 * np.abs(ref).max()
    if pad:
        assert not dxt[..., :pad].any() and not dxt[..., pad + C:].any()


# one piece of 8 x 16 pixels; fewer pieces than a block has warps; pieces that do not fill the last round; sliced
# channels; the widest layer's 160 x 160; with and without the bias gradient
@pytest.mark.parametrize("B,H,W,cin,cout,pad,bias", [(1, 8, 16, 16, 32, 0, True), (1, 24, 16, 48, 64, 8, True),
                                                     (3, 16, 48, 32, 32, 8, False), (5, 16, 16, 160, 160, 0, True),
                                                     (2, 128, 128, 96, 32, 0, True), (1, 64, 240, 16, 96, 16, True)])
def test_weight_and_bias_gradient_over_their_shapes(B, H, W, cin, cout, pad, bias):
    rng = np.random.default_rng(B + H + W + cin + cout)
    xt, xv, xp, ldx = slice_of(rand(rng, B, H, W, cin), pad)
    dt, dv, dp, ldd = slice_of(rand(rng, B, H, W, cout), pad)
    if pad:  # what lies beside the slices is not read
        for t, c in ((xt, cin), (dt, cout)):
            t[..., :pad] = t[..., pad + c:] = float("nan")
    dw, db = torch.ones(cout, 9, cin, device="cuda"), torch.ones(cout, device="cuda")
    S.call("lbmfvm_sg_conv3x3_wgrad", xp, ldx, dp, ldd, dw.data_ptr(), db.data_ptr() if bias else None, B, H, W, cin,
           cout, S._stream())
    torch.cuda.synchronize()
    x, dy = xv.double(), dv.double().reshape(-1, cout)
    xpad = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    taps = [xpad[:, k // 3:k // 3 + H, k % 3:k % 3 + W].reshape(-1, cin) for k in range(9)]
    want = torch.stack([dy.t() @ t for t in taps], 1)
    size = torch.stack([dy.abs().t() @ t.abs() for t in taps], 1)
    # FP32 sums of exact BF16 products: a warp's chain is some hundred terms, so 64 ulp of the sum of sizes is ample
    assert bool(((dw.double() - 1 - want).abs() <= 64 * 2.0 ** -23 * (size + 1)).all())
    if bias:
        assert bool(((db.double() - 1 - dy.sum(0)).abs() <= 64 * 2.0 ** -23 * (dy.abs().sum(0) + 1)).all())
    else:
        assert bool((db == 1).all())
