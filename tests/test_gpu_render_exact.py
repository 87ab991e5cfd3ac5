"""Both forms of the bank render (sd_dp_render and, through a workspace, the re-laid bank) on inputs whose
sums are exact: small whole image values and taps and depth weights of 0, 1/2 and 1, so that every partial
sum is a multiple of 1/2 below 2^24 and FP32 rounds nothing.  One tap dropped, doubled or misplaced
changes a result, whatever the kernel's size, so the outputs must equal the FP64 oracle's (rounded to the
image's type).  Shapes reach every launch of both forms."""
import ctypes

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

F32, BF, HF = torch.float32, torch.bfloat16, torch.float16
DEPTHS = {1: [1.0], 2: [0.5, 1.0], 3: [0.25, 0.5, 1.0]}


@pytest.mark.parametrize("shape,F,Z,NL,ks,quadrant,image,bank", [
    ((1, 1, 1, 1), 1, 1, 1, 1, False, F32, F32),
    ((1, 1, 3, 17), 3, 2, 1, 3, False, F32, F32),
    ((1, 1, 40, 39), 4, 3, 1, 65, False, F32, F32),      # re-laid: eight warps a group
    ((1, 2, 31, 63), 3, 3, 2, 127, True, F32, F32),
    ((1, 1, 37, 130), 2, 2, 1, 101, False, F32, BF),     # direct: four columns at a time
    ((1, 3, 70, 66), 4, 3, 3, 31, False, BF, BF),        # four warps a group
    ((2, 3, 130, 121), 3, 2, 1, 15, True, F32, HF),      # one
    ((1, 1, 200, 33), 4, 1, 1, 33, True, HF, HF),
    ((1, 3, 411, 509), 3, 3, 3, 5, True, F32, BF),       # two groups a warp
    ((2, 1, 1025, 1031), 3, 3, 1, 7, True, F32, F32),    # four
    ((1, 1, 1, 300), 5, 2, 1, 9, False, F32, F32),       # one row, one column
    ((1, 1, 301, 1), 5, 2, 1, 9, True, F32, F32),
])
def test_exact_sums(sdlib, shape, F, Z, NL, ks, quadrant, image, bank):
    sd = sdlib
    from paper_2503_11213_gb300 import api, _lib as L
    N, C, H, W = shape
    rng = np.random.default_rng(ks * H)
    fh = np.linspace(0.0, 0.45 * 0.002 * max(H, W, 2), F).astype(np.float32)
    lay = sd.BankLayout(fh, DEPTHS[Z], NL, ks, 0.002, bank,
                        sd.SD_FIELD_QUADRANT if quadrant else sd.SD_FIELD_RADIAL)
    # discs of every size, off centre, with zeros inside
    k = rng.integers(0, 4, lay.shape()).astype(np.float64)
    a = np.arange(ks) - (ks - 1) / 2
    r = rng.uniform(0.6, 0.75 * ks, lay.shape()[:3])[..., None, None, None]
    cy, cx = rng.uniform(-0.2 * ks, 0.2 * ks, (2,) + r.shape)
    k *= (a[:, None] - cy) ** 2 + (a - cx) ** 2 <= r * r
    aif = rng.integers(0, 8, shape).astype(np.float64) / (16 if image == HF else 1)
    depth = rng.choice(np.array([0.2, 0.25, 1 / 3, 0.5, 2 / 3, 1.0, 4.0], dtype=np.float32), (N, H, W))
    ref = O.render_bank(aif, depth, k, fh, np.array(DEPTHS[Z], np.float32), 0.002, n_threads=8,
                        field_mode=O.FIELD_QUADRANT if quadrant else O.FIELD_RADIAL)
    want = torch.tensor(ref, dtype=F32)
    assert np.array_equal(want.double().numpy(), ref) and ref.max() < 2 ** 23
    assert ks == 1 or ref.max() > 0
    want = want.to(image)
    ta = torch.tensor(aif, dtype=image, device="cuda")
    tk = torch.tensor(k, dtype=bank, device="cuda")
    td = torch.tensor(depth, device="cuda")
    c, n = lay.c(), ctypes.c_size_t(0)
    L.check(L.lib().sd_dp_render_workspace(ctypes.byref(c), N, C, H, W, ctypes.byref(n)), "ws")
    for size in (0, n.value):
        out = torch.full((N, 2 * C, H, W), float("nan"), dtype=image, device="cuda")
        ws = torch.full((size,), 255, dtype=torch.uint8, device="cuda") if size else None
        L.check(L.lib().sd_dp_render_ws(api._ptr(ta), api._ptr(td), api._ptr(tk), ctypes.byref(c),
                                        N, C, H, W, api._DT[image], api._ptr(out), api._ptr(ws),
                                        size, api._stream()), "render")
        assert torch.equal(out.cpu(), want), "re-laid" if size else "direct"
