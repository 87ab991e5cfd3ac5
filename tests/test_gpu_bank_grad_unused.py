"""Bank gradients of banks most of whose slices no tile uses (a nearly flat depth map; a quadrant bank's
far cells), from workspaces full of NaN: the blocks of unused keys write a radial bank's zeros and write
nothing of a quadrant bank, whose fold must not read them.  Against the oracle (max|err| <= 1e-4 max|ref|
in FP32, 8 * 2^-9 on the tensor cores), with exact zeros where no pixel uses a slice."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from test_gpu_render import rand_bank

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("quadrant", [False, True])
@pytest.mark.parametrize("N,C,H,Wd,F,Z,NL,ks", [
    (1, 2, 24, 37, 5, 9, 2, 15),
    (2, 1, 40, 70, 6, 8, 1, 65),
    (1, 1, 33, 20, 4, 12, 1, 91),
])
def test_unused_slices(sdlib, quadrant, N, C, H, Wd, F, Z, NL, ks):
    sd = sdlib
    rng = np.random.default_rng(ks)
    mode = sd.SD_FIELD_QUADRANT if quadrant else sd.SD_FIELD_RADIAL
    aif = rng.uniform(0, 1, (N, C, H, Wd)).astype(np.float32)
    depth = rng.uniform(0.8, 1.0, (N, H, Wd)).astype(np.float32)
    fh = np.linspace(0.0, 1.5 * max(H, Wd) * 0.002, F).astype(np.float32)  # past the corners
    dm = (W.inverse_uniform_depths(300.0, 3000.0, Z) / 1000.0).astype(np.float32)
    bank = rand_bank(rng, F * F if quadrant else F, Z, NL, ks)
    g = rng.normal(size=(N, 2 * C, H, Wd)).astype(np.float32)
    a, d, gt = (torch.tensor(x, device="cuda") for x in (aif, depth, g))
    b = torch.tensor(bank, dtype=torch.float32, device="cuda").reshape(-1)

    def check(gb, ref, tol):
        gb = gb.cpu().numpy().reshape(bank.shape)
        assert np.isfinite(gb).all()
        unused = ~np.any(ref != 0, axis=(-1, -2, -3))
        assert unused.any() and (gb[unused] == 0).all()
        assert np.abs(gb - ref).max() <= tol * np.abs(ref).max()

    field = O.FIELD_QUADRANT if quadrant else 0
    lay = sd.BankLayout(fh, dm, NL, ks, 0.002, field_mode=mode)
    ws = torch.full((sd.api.render_backward_workspace(lay, N, C, H, Wd),), 255, dtype=torch.uint8,
                    device="cuda")
    _, gb = sd.dp_render_backward(gt, a, d, b, lay, need_aif=False, workspace=ws)
    check(gb, O.render_bank_bwd(g, aif, depth, bank, fh, dm, 0.002, field_mode=field)[1], 1e-4)
    if ks > 65:
        return
    a16 = a.to(torch.bfloat16)
    lay16 = sd.BankLayout(fh, dm, NL, ks, 0.002, dtype=torch.bfloat16, field_mode=mode)
    wst = torch.full((sd.api.bank_grad_tc_workspace(lay16, N, C, H, Wd),), 255, dtype=torch.uint8,
                     device="cuda")
    out = torch.full(lay16.shape(), float("nan"), device="cuda")
    sd.dp_render_bank_grad_tc(gt, a16, d, lay16, out=out, workspace=wst)
    sd.sync_status(wst[:4].view(torch.int32))
    ref = O.render_bank_bwd(g, a16.float().cpu().numpy(), depth, bank, fh, dm, 0.002,
                            field_mode=field)[1]
    check(out, ref, 8 * 2.0 ** -9)
