"""Renders through both forms of the bank render at the shapes that reach each of their launches, reduced
to a SHA-256 per output.  Run by test_gpu_checked_render.py in the normal build and, as a child process
with SDIRT_CHECKED=1, in the build whose kernels check their indices."""
import ctypes
import json
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
for d in (ROOT, os.path.join(ROOT, "tests")):
    if d not in sys.path:
        sys.path.insert(0, d)

from checked_workload import _h  # noqa: E402

SHAPES = {  # N, C, H, W, F, Z, NL, ks, quadrant
    "tiny": (1, 1, 1, 1, 1, 1, 1, 1, False),
    "split8": (1, 1, 29, 41, 3, 4, 1, 65, False),
    "split4": (1, 3, 70, 66, 3, 4, 3, 31, True),
    "one": (2, 1, 130, 121, 3, 4, 1, 17, False),
    "two": (1, 3, 411, 509, 2, 3, 1, 5, True),
    "four": (2, 1, 1025, 1031, 2, 3, 1, 3, False),
    "wide": (1, 1, 40, 130, 2, 3, 1, 127, False),
    "wide4": (1, 1, 37, 70, 2, 3, 1, 101, True),
}


def run(sd):
    from paper_2503_11213_gb300 import api, _lib as L
    out = {}
    for name, (N, C, H, W, F, Z, NL, ks, quadrant) in SHAPES.items():
        rng = np.random.default_rng(ks)
        lay = sd.BankLayout(np.linspace(0.0, 0.001 * max(H, W, 2), F), np.linspace(0.4, 3.0, Z), NL,
                            ks, 0.002, field_mode=int(quadrant))
        aif = rng.random((N, C, H, W)).astype(np.float32)
        for what in ("finite", "infinite"):  # the second takes the blocks that skip zero taps
            if what == "infinite":
                aif[:, :, H // 2, W // 2] = np.inf
            a, d, b = (torch.tensor(x, dtype=torch.float32, device="cuda") for x in
                       (aif, rng.uniform(0.3, 3.5, (N, H, W)), rng.random(lay.shape())))
            c, n = lay.c(), ctypes.c_size_t(0)
            L.check(L.lib().sd_dp_render_workspace(ctypes.byref(c), N, C, H, W, ctypes.byref(n)), "ws")
            for size in (0, n.value):
                o = torch.empty((N, 2 * C, H, W), device="cuda")
                ws = torch.empty(size, dtype=torch.uint8, device="cuda") if size else None
                L.check(L.lib().sd_dp_render_ws(api._ptr(a), api._ptr(d), api._ptr(b),
                                                ctypes.byref(c), N, C, H, W, L.SD_F32, api._ptr(o),
                                                api._ptr(ws), size, api._stream()), "render")
                out[f"{name}_{what}_{'relaid' if size else 'direct'}"] = _h(o)
    torch.cuda.synchronize()
    return out


if __name__ == "__main__":
    import paper_2503_11213_gb300 as sd
    res = run(sd)
    site, index, bound, count = sd.api.check_status()
    print(json.dumps({"hashes": res, "site": site, "index": index, "bound": bound, "count": count}))
