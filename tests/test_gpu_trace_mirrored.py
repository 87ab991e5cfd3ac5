"""Requests on the sensor's x axis (v = 0): only the pupil rows up to the middle one are traced and
every ray above it stands for its mirrored ray too.  The same request with v = 1e-30 mm takes the
general path (every ray traced) and must give the same bank, statistics and landing mask: v is far
below the rounding of every position it enters."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def requests(v):
    """Edge grids (2 and 3 samples a side; even and odd; rows ending inside and at a warp), patches
    from one pixel up, fields on both sides of the axis, three lenses."""
    reqs = []
    for lens in range(3):
        for n, ks in ((2, 1), (3, 3), (32, 127), (33, 31), (64, 65), (97, 15), (160, 31)):
            for h, d in ((0.0, 1000.0), (0.9, 400.0), (-1.2, 2500.0)):
                reqs.append((h, d, W.LAMBDA_F, n, ks, lens, v))
    return np.array(reqs, dtype=W.REQ_DTYPE)


def words(mask, reqs, launched, max_n):
    m = mask.cpu().numpy().view(np.uint32).reshape(len(reqs), -1)
    assert m.shape[1] == (max_n * max_n + 31) // 32
    return [m[r, :(launched[r] + 31) // 32] for r in range(len(reqs))]


@pytest.mark.parametrize("mode,norm", [("hard", "none"), ("hard", "joint"), ("bilinear", "none")])
@pytest.mark.parametrize("batched", [None, (96, 1, 1), (256, 700, 2)])
def test_mirrored_rays_equal_the_general_path(sdlib, mode, norm, batched):
    sd = sdlib
    if batched and mode == "bilinear":
        pytest.skip("the batched trace bins hard")
    lenses = [sd.Lens(t, 1000.0) for t in (W.doublet_pair_f18(), W.spherical4(), W.canon_rf50())]
    sensor = sd.DPSensor(0.004)
    mode_id = {"hard": sd.SD_BIN_HARD, "bilinear": sd.SD_BIN_BILINEAR}[mode]
    norm_id = {"none": sd.SD_NORM_NONE, "joint": sd.SD_NORM_JOINT}[norm]
    got = []
    for v in (0.0, 1e-30):
        reqs = requests(v)
        dev, total, _ = sd.make_requests(reqs)
        mask = sd.land_mask(len(reqs), 160)
        mask.fill_(-1)
        if batched and v == 0.0:
            bt = sd.BatchedTrace(lenses, sensor, dev, len(reqs), total, max_ks=127, max_n=160,
                                 norm=norm_id, config=batched, mask=mask)
            out, stats = bt.run()
        else:
            out, stats = sd.dp_psf_trace(lenses, sensor, dev, len(reqs), total, max_ks=127,
                                         max_n=160, mode=mode_id, norm=norm_id, mask=mask)
        torch.cuda.synchronize()
        launched = stats[:, 0].cpu().numpy()
        got.append((out, stats, words(mask, reqs, launched, 160)))
    (a, sa, ma), (b, sb, mb) = got
    assert torch.equal(sa, sb)
    assert int(sa[:, 1].sum()) > 0.5 * int(sa[:, 0].sum())
    if mode == "hard":  # bilinear sums depend on the order of their additions
        assert torch.equal(a, b)
    for x, y in zip(ma, mb):
        assert np.array_equal(x, y)
    for l in lenses:
        l.free()


@pytest.mark.parametrize("n_req", [1, 152, 153, 304, 305])
@pytest.mark.parametrize("v", [0.0, 0.3])
def test_block_sizes_equal_the_batched_trace(sdlib, n_req, v):
    """The per-request kernel's 1024, 512 and 256 threads a block (chosen by the number of requests)
    give the batched trace's counts and masks."""
    sd = sdlib
    rng = np.random.default_rng(n_req)
    reqs = np.zeros(n_req, dtype=W.REQ_DTYPE)
    reqs["h_mm"], reqs["v_mm"] = rng.uniform(0, 1.4, n_req), v
    reqs["depth_mm"], reqs["lambda_nm"] = rng.uniform(300, 3000, n_req), W.LAMBDA_C
    reqs["n_grid"], reqs["ks"] = rng.integers(16, 81, n_req), rng.choice([1, 15, 65], n_req)
    lens = sd.Lens(W.doublet_pair_f18(), 1000.0)
    dev, total, _ = sd.make_requests(reqs)
    masks = [sd.land_mask(n_req, 80).fill_(-1) for _ in range(2)]
    a, sa = sd.dp_psf_trace(lens, sd.DPSensor(0.002), dev, n_req, total, max_ks=65, max_n=80,
                            mask=masks[0])
    bt = sd.BatchedTrace(lens, sd.DPSensor(0.002), dev, n_req, total, max_ks=65, max_n=80,
                         mask=masks[1])
    b, sb = bt.run()
    torch.cuda.synchronize()
    assert torch.equal(a, b) and torch.equal(sa, sb)
    launched = sa[:, 0].cpu().numpy()
    for x, y in zip(words(masks[0], reqs, launched, 80), words(masks[1], reqs, launched, 80)):
        assert np.array_equal(x, y)
    lens.free()
