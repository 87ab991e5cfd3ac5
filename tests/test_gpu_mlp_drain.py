"""PSF network with wait limits that give up in mid-pipeline, while weight copies and products are in
flight: whichever wait gives up first, the call ends soon (the drain waits for each buffer's last copy,
not for a phase that never comes), says so in its status word, and leaves the next call right.  A call
that gives up nowhere must be right itself."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ks", [1, 21])
def test_give_up_anywhere_drains(sdlib, ks):
    sd = sdlib
    rng = np.random.default_rng(ks)
    shapes = sd.MLP_SHAPES(ks)
    net = sd.PsfMLP([rng.normal(0, np.sqrt(2.0 / s[1]), size=s).astype(np.float32)
                     for s in shapes],
                    [rng.normal(0, 0.05, size=s[0]).astype(np.float32) for s in shapes], ks)
    # more than one CTA an SM, the last one ragged
    depth = torch.tensor(rng.uniform(0.5, 20.0, size=(151, 143)).astype(np.float32), device="cuda")
    st = torch.empty(1, dtype=torch.int32, device="cuda")
    good = sd.mlp_psf_map(net, depth, 0.5, 20.0, status=st)[0].clone()
    sd.sync_status(st)
    gave_up = 0
    for limit in (0, 1, 2, 3, 5, 8, 13, 21, 34, 55, 89, 144, 377, 987, 10000):
        out = torch.full_like(good, float("nan"))
        try:
            sd.set_wait_limit(limit)
            t0 = time.perf_counter()
            sd.mlp_psf_map(net, depth, 0.5, 20.0, out=out, status=st)
            torch.cuda.synchronize()
            assert time.perf_counter() - t0 < 1.0, limit
        finally:
            sd.set_wait_limit(None)
        if int(st.item()):
            gave_up += 1
        else:
            assert torch.equal(out, good), limit
    assert gave_up >= 1
    again = sd.mlp_psf_map(net, depth, 0.5, 20.0, status=st)[0]
    sd.sync_status(st)
    assert torch.equal(again, good)
