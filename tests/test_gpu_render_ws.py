"""sd_dp_render_ws (the re-laid bank) against sd_dp_render (the bank itself): both sum up to 2 ks^2
FP32 products per pixel and plane, |I K| summing to at most 1 per slice (images in [0, 1],
sum-normalised PSF pairs), so each is within n 2^-24 of the exact sum."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

EPS = {torch.float32: 0.0, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -11}


def scene(sd, shape, F, Z, NL, ks, quadrant, image, bank, seed=0):
    N, C, H, W = shape
    rng = np.random.default_rng(seed)
    lay = sd.BankLayout(np.linspace(0.0, 0.06, F), np.linspace(0.4, 3.0, Z), NL, ks, 0.002, bank,
                        sd.SD_FIELD_QUADRANT if quadrant else sd.SD_FIELD_RADIAL)
    k = rng.random(lay.shape())
    # discs of every size down to one tap, off centre: empty rows, columns and corners
    a = np.arange(ks) - (ks - 1) / 2
    r = rng.uniform(0.3, 0.8 * ks, lay.shape()[:3])[..., None, None, None]
    cy, cx = rng.uniform(-0.2 * ks, 0.2 * ks, (2,) + r.shape)
    k *= (a[:, None] - cy) ** 2 + (a - cx) ** 2 <= r * r
    k /= np.maximum(k.sum((-1, -2, -3), keepdims=True), 1e-30)
    aif = torch.tensor(rng.random(shape), dtype=image, device="cuda")
    depth = torch.tensor(rng.uniform(0.3, 3.5, (N, H, W)), dtype=torch.float32, device="cuda")
    depth[..., : W // 2] = 0.4  # exactly on the first slice (weight 0)
    return lay, aif, depth, torch.tensor(k, dtype=bank, device="cuda")


F32, BF, HF = torch.float32, torch.bfloat16, torch.float16


@pytest.mark.parametrize("shape,F,Z,NL,ks,quadrant,image,bank", [
    ((1, 1, 1, 1), 1, 1, 1, 1, False, F32, F32),
    ((1, 1, 3, 17), 3, 2, 1, 3, False, F32, F32),
    ((1, 1, 40, 39), 4, 5, 1, 65, False, F32, F32),       # eight warps a group
    ((1, 2, 31, 63), 4, 5, 2, 127, True, F32, F32),
    ((1, 3, 70, 66), 4, 5, 3, 31, False, BF, BF),         # four
    ((2, 3, 130, 121), 3, 4, 1, 15, True, F32, HF),       # one, one wavelength for all channels
    ((1, 1, 200, 33), 4, 1, 1, 33, True, HF, HF),
    ((1, 3, 411, 509), 3, 4, 3, 5, True, F32, BF),        # two groups a warp
    ((2, 1, 1025, 1031), 3, 4, 1, 7, True, F32, F32),     # four
])
def test_ws_equals_direct(sdlib, shape, F, Z, NL, ks, quadrant, image, bank):
    sd = sdlib
    from paper_2503_11213_gb300 import api, _lib as L
    N, C, H, W = shape
    lay, aif, depth, k = scene(sd, shape, F, Z, NL, ks, quadrant, image, bank)
    c, out, n = lay.c(), [], ctypes.c_size_t(0)
    L.check(L.lib().sd_dp_render_workspace(ctypes.byref(c), N, C, H, W, ctypes.byref(n)), "ws")
    for ws_bytes in (0, n.value, n.value):
        o = torch.full((N, 2 * C, H, W), float("nan"), dtype=image, device="cuda")
        ws = torch.full((ws_bytes,), 255, dtype=torch.uint8, device="cuda") if ws_bytes else None
        L.check(L.lib().sd_dp_render_ws(api._ptr(aif), api._ptr(depth), api._ptr(k),
                                        ctypes.byref(c), N, C, H, W, api._DT[image], api._ptr(o),
                                        api._ptr(ws), ws_bytes, api._stream()), "render")
        out.append(o)
    direct, a, b = out
    assert torch.equal(a, b)
    tol = 4 * (ks * ks + 32) * 2.0 ** -24 + EPS[image]
    assert float((a.double() - direct.double()).abs().max()) <= tol
    # a short or misaligned workspace is refused
    ws = torch.empty(n.value + 256, dtype=torch.uint8, device="cuda")
    for ptr, size in ((ws.data_ptr(), n.value - 1), (ws.data_ptr() + 16, n.value)):
        st = L.lib().sd_dp_render_ws(api._ptr(aif), api._ptr(depth), api._ptr(k), ctypes.byref(c),
                                     N, C, H, W, api._DT[image], api._ptr(o),
                                     ctypes.c_void_p(ptr), size, api._stream())
        assert st == 1  # SD_ERR_ARG
