"""Which form dp_render takes: the bank as it is for small kernels on large images, the re-laid bank for
the rest (sd_dp_render_advised_workspace).  The rule needs no GPU; that dp_render follows it, does."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2503_11213_gb300 import _lib as L
from paper_2503_11213_gb300 import build as B


def layout(ks, F=16, Z=16, nl=1, quadrant=False):
    fh = np.linspace(0.0, 1.0, F).astype(np.float32)
    dm = np.linspace(0.5, 3.0, Z).astype(np.float32)
    lay = L.SdBankLayout(F, Z, nl, ks, L.SD_F32, int(quadrant),
                         fh.ctypes.data_as(ctypes.POINTER(ctypes.c_float)),
                         dm.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), 0.002, 0.0)
    return lay, (fh, dm)


def query(name, lay, N, C, H, W):
    n = ctypes.c_size_t(7)
    st = getattr(L.lib(), name)(ctypes.byref(lay), N, C, H, W, ctypes.byref(n))
    return st, n.value


@pytest.mark.parametrize("ks,N,C,H,W,quadrant,direct", [
    (1, 1, 1, 64, 64, False, False),
    (65, 1, 3, 1024, 1024, False, False),
    (3, 1, 3, 1024, 1024, False, True),
    (21, 1, 3, 2048, 2048, False, True),
    (25, 1, 3, 2048, 2048, False, False),
    (15, 1, 3, 512, 512, False, False),
    (21, 1, 3, 512, 512, True, True),
    (31, 2, 3, 1000, 1000, True, True),
    (65, 1, 3, 2048, 2048, True, False),
    (31, 1, 1, 64, 64, True, False),
])
def test_advice_by_size(ks, N, C, H, W, quadrant, direct):
    B.build()
    lay, keep = layout(ks, F=8 if quadrant else 16, Z=8 if quadrant else 16, quadrant=quadrant)
    st, full = query("sd_dp_render_workspace", lay, N, C, H, W)
    assert st == L.SD_OK and full > 0
    st, advised = query("sd_dp_render_advised_workspace", lay, N, C, H, W)
    assert st == L.SD_OK and advised == (0 if direct else full)


def test_advice_arguments():
    B.build()
    lay, keep = layout(3)
    f = L.lib().sd_dp_render_advised_workspace
    assert f(ctypes.byref(lay), 1, 1, 8, 8, None) == L.SD_ERR_ARG
    for args, st in (((1, 0, 8, 8), L.SD_ERR_ARG), ((-1, 1, 8, 8), L.SD_ERR_ARG),
                     ((70000, 1, 8, 8), L.SD_ERR_UNSUPPORTED), ((0, 1, 8, 8), L.SD_OK)):
        for name in ("sd_dp_render_workspace", "sd_dp_render_advised_workspace"):
            assert query(name, lay, *args) == (st, 0 if st == L.SD_OK else 7), (name, args)
    lay, keep = layout(4)
    assert query("sd_dp_render_advised_workspace", lay, 1, 1, 8, 8)[0] == L.SD_ERR_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("ks,C,H,W,quadrant,direct", [
    (3, 1, 64, 64, False, False), (7, 3, 512, 511, False, True), (17, 3, 512, 512, False, False),
    (19, 3, 509, 512, True, True), (33, 1, 512, 512, True, False)])
def test_dp_render_takes_the_advised_form(sdlib, ks, C, H, W, quadrant, direct):
    """Bit for bit the output of that form (dense random kernels: the other form's sums, taken in
    another order, differ in some of so many pixels)."""
    sd = sdlib
    from paper_2503_11213_gb300 import api
    F = 8 if quadrant else 16
    lay = sd.BankLayout(np.linspace(0.0, 0.5, F), np.linspace(0.4, 3.0, F), C, ks, 0.002,
                        field_mode=sd.SD_FIELD_QUADRANT if quadrant else sd.SD_FIELD_RADIAL)
    g = torch.Generator("cuda").manual_seed(ks)
    bank = torch.rand(lay.shape(), device="cuda", generator=g)
    aif = torch.rand((1, C, H, W), device="cuda", generator=g)
    depth = 0.3 + 3 * torch.rand((1, H, W), device="cuda", generator=g)
    got = sd.dp_render(aif, depth, bank, lay)
    c, n = lay.c(), ctypes.c_size_t(0)
    L.check(L.lib().sd_dp_render_workspace(ctypes.byref(c), 1, C, H, W, ctypes.byref(n)), "ws")
    ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    form = []
    for w, size in ((None, 0), (ws, n.value)):
        o = torch.empty_like(got)
        L.check(L.lib().sd_dp_render_ws(api._ptr(aif), api._ptr(depth), api._ptr(bank),
                                        ctypes.byref(c), 1, C, H, W, L.SD_F32, api._ptr(o),
                                        api._ptr(w), size, api._stream()), "render")
        form.append(o)
    assert not torch.equal(*form)
    assert torch.equal(got, form[0 if direct else 1])
