"""The per-lens sum of the adjoint's per-request gradients: four contiguous request ranges per lens,
each added in request order, then the four in range order, in FP32 (bit for bit the sum below)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 31, 128, 129, 257, 513])
def test_lens_sums(sdlib, n):
    sd = sdlib
    rng = np.random.default_rng(n)
    reqs = np.zeros(n, dtype=W.REQ_DTYPE)
    reqs["h_mm"], reqs["depth_mm"] = rng.uniform(0, 1.4, n), rng.uniform(300, 3000, n)
    reqs["lambda_nm"], reqs["n_grid"], reqs["ks"] = W.LAMBDA_D, 16, 15
    reqs["lens"] = rng.integers(0, 2, n)
    lenses = [sd.Lens(W.doublet_pair_f18(), 1000.0), sd.Lens(W.spherical4(), 1000.0)]
    dev, total, _ = sd.make_requests(reqs)
    g = torch.tensor(rng.standard_normal(total), dtype=torch.float32, device="cuda")
    greq, glens = sd.dp_psf_trace_backward(lenses, sd.DPSensor(0.004), dev, n, g, max_ks=15, max_n=16)
    greq, glens = greq.cpu().numpy(), glens.cpu().numpy()
    for l in range(2):
        part = []
        for c in range(4):
            a = np.zeros((32, 8), dtype=np.float32)
            for r in range(n * c // 4, n * (c + 1) // 4):
                if reqs["lens"][r] == l:
                    a += greq[r]
            part.append(a)
        assert np.array_equal(glens[l], ((part[0] + part[1]) + part[2]) + part[3])
    for l in lenses:
        l.free()
