"""Infinite and NaN image values (overflowed 16-bit highlights) in the render from a re-laid bank: a pixel
takes them through its non-zero taps only.  The expected pixels follow from counting, per pixel, the
non-zero taps that lie over a +inf, a -inf and a NaN; all others must equal the render of the image with
those values set to 0."""
import ctypes

import numpy as np
import pytest
import torch
import torch.nn.functional as F

pytestmark = pytest.mark.gpu

F32, BF, HF = torch.float32, torch.bfloat16, torch.float16


def render_ws(sd, aif, depth, bank, lay):
    from paper_2503_11213_gb300 import api, _lib as L
    N, C, H, W = aif.shape
    c, n = lay.c(), ctypes.c_size_t(0)
    L.check(L.lib().sd_dp_render_workspace(ctypes.byref(c), N, C, H, W, ctypes.byref(n)), "ws")
    ws = torch.full((n.value,), 255, dtype=torch.uint8, device="cuda")
    out = torch.empty((N, 2 * C, H, W), dtype=aif.dtype, device="cuda")
    L.check(L.lib().sd_dp_render_ws(api._ptr(aif), api._ptr(depth), api._ptr(bank),
                                    ctypes.byref(c), N, C, H, W, api._DT[aif.dtype],
                                    api._ptr(out), api._ptr(ws), n.value, api._stream()), "render")
    return out


@pytest.mark.parametrize("H,W,C,ks,quadrant,image,bank", [
    (33, 47, 1, 1, False, F32, F32),
    (40, 61, 1, 65, False, F32, F32),       # eight warps a group
    (70, 66, 2, 31, True, HF, HF),          # four
    (130, 121, 3, 17, False, F32, HF),      # one
    (411, 509, 2, 5, True, BF, BF),         # two groups a warp
    (1025, 1031, 2, 7, False, F32, F32),    # four
])
def test_only_non_zero_taps_take_non_finite_values(sdlib, H, W, C, ks, quadrant, image, bank):
    sd = sdlib
    rng = np.random.default_rng(ks)
    lay = sd.BankLayout([0.0], [1.0], 1, ks, 0.002, bank,
                        sd.SD_FIELD_QUADRANT if quadrant else sd.SD_FIELD_RADIAL)
    # a disc off centre with holes, the left half in L and the right half in R
    a = np.arange(ks) - (ks - 1) / 2
    k = rng.random((2, ks, ks)) + 0.1
    k *= ((a[:, None] - 0.1 * ks) ** 2 + a ** 2 <= (0.35 * ks + 0.5) ** 2) & (rng.random((2, ks, ks)) < 0.8)
    k[:, 0, ks - 1] = 0.25  # and a corner, so that the footprint's edges are in use
    k[0] *= a < 0.2 * ks
    K = torch.tensor(k / k.sum(), dtype=bank)
    img = torch.tensor(rng.random((1, C, H, W)), dtype=image)
    bad = torch.zeros((3, 1, C, H, W), dtype=torch.bool)
    for i, v in enumerate((float("inf"), float("-inf"), float("nan"))):
        for _ in range(2):
            c, y, x = rng.integers(C), rng.integers(H), rng.integers(W)
            img[0, c, y, x] = v
    img[0, 0, 0, W - 1] = float("inf")  # replicated into the border
    bad[0], bad[1], bad[2] = img == float("inf"), img == float("-inf"), img.isnan()
    depth = torch.ones((1, H, W), device="cuda")
    if quadrant:  # the flip classes exchange sides and mirror: render the indicators to count
        clean = torch.where(bad.any(0), torch.zeros_like(img), img)
        ones = (K != 0).to(bank)
        cnt = [render_ws(sd, m.to(image).cuda(), depth, ones.cuda(), lay).cpu() > 0.5 for m in bad]
        want = render_ws(sd, clean.cuda(), depth, K.cuda(), lay).cpu()
    else:
        clean = torch.where(bad.any(0), torch.zeros_like(img), img)
        p = (ks - 1) // 2
        flip = K.double().flip(-1, -2)[:, None]

        def conv(x, w):
            y = F.conv2d(F.pad(x.double().transpose(0, 1), (p,) * 4, mode="replicate"), w)
            return y.permute(1, 0, 2, 3).reshape(1, 2 * C, H, W)
        cnt = [conv(m, (flip != 0).double()) > 0.5 for m in bad]
        want = render_ws(sd, clean.cuda(), depth, K.cuda(), lay).cpu()
        assert torch.allclose(want.double(), conv(clean, flip), rtol=2.0 ** -8 if image != F32 else 0,
                              atol=1e-6)
    got = render_ws(sd, img.cuda(), depth, K.cuda(), lay).cpu()
    pos, neg, nan = cnt
    nan = nan | (pos & neg)
    fine = ~(pos | neg | nan)
    assert bool(fine.any()) and bool(pos.any()) and bool(nan.any())
    assert torch.equal(got[fine], want[fine])
    assert bool(got[nan].isnan().all())
    assert bool((got[pos & ~nan] == float("inf")).all())
    assert bool((got[neg & ~nan] == float("-inf")).all())
