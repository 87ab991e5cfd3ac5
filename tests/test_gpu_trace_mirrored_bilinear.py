"""Values of the bilinear bank whose mirrored rays are splatted, not traced, against the general path's
(the same request with v = 1e-30 mm, every ray traced).  Both add the same weights in some order: a sum of
n non-negative terms is within (n - 1) 2^-24 of the exact one, relative, to first order, so two of them are
within 2 n 2^-24.  n is at most the number of rays whose nearest pixel is the pixel or one of its eight
neighbours: the hard count of a patch one pixel wider, summed over 3 x 3."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ks", [(2, 1), (3, 3), (32, 125), (33, 31), (64, 65), (97, 15), (160, 31)])
def test_bilinear_values(sdlib, n, ks):
    sd = sdlib
    tables = (W.doublet_pair_f18(), W.spherical4(), W.canon_rf50())
    lenses, sensor = [sd.Lens(t, 1000.0) for t in tables], sd.DPSensor(0.004)

    def trace(v, size, mode):
        reqs = np.array([(h, d, W.LAMBDA_F, n, size, lens, v) for lens in range(3)
                         for h, d in ((0.0, 1000.0), (0.9, 400.0), (-1.2, 2500.0))], dtype=W.REQ_DTYPE)
        dev, total, _ = sd.make_requests(reqs)
        out, _ = sd.dp_psf_trace(lenses, sensor, dev, len(reqs), total, max_ks=size, max_n=n,
                                 mode=mode, norm=sd.SD_NORM_NONE)
        return out.view(len(reqs), 2, size, size).double()

    count = trace(1e-30, ks + 2, sd.SD_BIN_HARD)
    terms = 9 * torch.nn.functional.avg_pool2d(count, 3, stride=1)
    a, b = (trace(v, ks, sd.SD_BIN_BILINEAR) for v in (0.0, 1e-30))
    assert float(b.sum()) > 0 or n < 4
    assert bool(((a - b).abs() <= 2.01 * terms * 2.0 ** -24 * torch.maximum(a, b)).all())
    for l in lenses:
        l.free()
