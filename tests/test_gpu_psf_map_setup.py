"""A map's set-up in its own kernel (more than 1024 pixels whose PSFs hold it) and in the pixels' blocks
(the rest): every valid pixel's PSF and statistics are those of the request-array trace bit for bit, and a
pixel of invalid depth keeps its output and has no rays."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

F32, BF, HF = torch.float32, torch.bfloat16, torch.float16


@pytest.mark.parametrize("H,Wd", [(32, 32), (25, 41)])  # 1024 and 1025 pixels
@pytest.mark.parametrize("lens_of,ks,dtype", [
    (W.canon_rf50, 3, F32), (W.canon_rf50, 5, F32), (W.canon_rf50, 5, BF), (W.canon_rf50, 21, HF),
    (W.singlet_f2, 1, F32), (W.singlet_f2, 3, F32), (W.singlet_f2, 15, BF),
])
def test_map_equals_request_trace(sdlib, H, Wd, lens_of, ks, dtype):
    sd = sdlib
    rng = np.random.default_rng(ks)
    pitch, lam, n = 0.01, 550.0, 33
    depth = rng.uniform(0.4, 4.0, (H, Wd)).astype(np.float32)
    bad = rng.random((H, Wd)) < 0.02
    bad[0, 0] = bad[H - 1, Wd - 1] = True
    depth[bad] = rng.choice(np.array([0.0, -1.0, np.nan], dtype=np.float32), int(bad.sum()))
    lens, sen = sd.Lens(lens_of(), 1000.0), sd.DPSensor(pitch)
    out = torch.full((H, Wd, 2, ks, ks), 7.0, dtype=dtype, device="cuda")
    stats = torch.full((H * Wd, 8), -1, dtype=torch.int64, device="cuda")
    sd.dp_psf_map(lens, sen, torch.tensor(depth, device="cuda"), lam, n, ks, out=out, stats=stats)
    rows, cols = np.nonzero(~bad)
    reqs = W.map_requests(depth, rows, cols, pitch, lam, n, ks)
    dev, total, _ = sd.make_requests(reqs)
    bank, st = sd.dp_psf_trace(lens, sen, dev, len(reqs), total, max_ks=ks, max_n=n, dtype=dtype)
    torch.cuda.synchronize()
    good = torch.tensor(~bad, device="cuda")
    stats = stats.view(H, Wd, 8)
    assert torch.equal(out[good], bank.view(-1, 2, ks, ks))
    assert torch.equal(stats[good], st) and int(st[:, 1].sum()) > 0
    assert bool((out[~good] == 7.0).all()) and bool((stats[~good] == 0).all())
    lens.free()
