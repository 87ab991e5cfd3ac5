"""Performance cases: the calls a user of the dual-pixel simulator makes, over the sizes, storage types
and options they are made with.

Every family below is one public entry point (or the two of a training step):

  trace         dp_psf_trace: a PSF bank over fields x depths x wavelengths
  batch         BatchedTrace.run: uneven requests in one persistent launch
  psf_map       dp_psf_map: a traced PSF for every pixel of a depth map
  lens_grad     dp_psf_trace_autograd and its backward: gradients of the lens parameters
  render        dp_render: an image rendered through a bank
  render_tc     dp_render_tc: the same for 16-bit images on the tensor cores
  render_grad   dp_render_autograd and its backward: gradients of image and bank
  bank_grad_tc  dp_render_bank_grad_tc: the bank's gradient for 16-bit images
  mlp_map       mlp_psf_map: the PSF network's map of a depth map
  render_map    dp_render_map: an image rendered through a per-pixel map

Inputs are synthetic and made on the GPU from a seed: 1/f images, gradient-noise depth maps, and banks of
defocus discs sampled with as many rays as a trace would launch (so with a traced bank's zeros).  exact() is
the same mathematics in 64 bits, written here in plain torch.
"""
import math

import numpy as np
import torch

import paper_2503_11213_gb300 as sd

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f32": 4, "bf16": 2, "f16": 2}
LAMBDAS = (656.2725, 587.5618, 486.1327)
MAX_RAY_SURFACES = 512 * 768 * 3228 * 12  # the largest listed case's

# ---------------------------------------------------------------------------------------------------
# Lenses: (radius, thickness, nd, Vd, semi-diameter, conic, a4..a12) per surface, radius None = the stop
# ---------------------------------------------------------------------------------------------------
CROWN, FLINT, AIR = (1.5168, 64.17), (1.62004, 36.37), (1.0, 0.0)
LENSES = {
    # f/2 singlet
    "singlet": dict(focus=1000.0, pitch=0.004, half_field=0.12, depth_m=(0.5, 3.0), surfaces=[
        (None, 0.0, AIR, 12.5), (51.68, 5.0, (1.5168, 0.0), 14.0), (-51.68, 50.0, AIR, 14.0)]),
    # f/1.8 doublet pair with two aspheres
    "doublet": dict(focus=1000.0, pitch=0.002, half_field=1.448, depth_m=(0.3, 3.0), surfaces=[
        (None, 0.0, AIR, 24.0 / 3.6),
        (19.30630884225998, 4.0, CROWN, 8.0, -0.8276327856667939, (1e-5, -1e-7, 1e-9, 1e-12, 0.0)),
        (-16.08859070188332, 1.5, FLINT, 8.0), (-51.48349024602662, 1.5, AIR, 8.0), (25.74174512301331, 3.5, CROWN, 8.0),
        (-19.30630884225998, 1.5, FLINT, 8.0),
        (128.70872561506656, 17.0, AIR, 8.0, -0.7345202837075637, (-1e-5, -1e-7, 1e-9, 1e-12, 0.0))]),
    # four-surface spherical lens
    "spherical": dict(focus=1000.0, pitch=0.004, half_field=1.448, depth_m=(0.3, 3.0), surfaces=[
        (None, 0.0, AIR, 6.0), (37.03, 4.0, CROWN, 9.0), (-59.99, 2.0, AIR, 9.0), (30.61, 3.5, FLINT, 9.0),
        (-90.57, 30.0, AIR, 9.0)]),
    # Canon RF50 (the paper's Table S1) with its stop scaled to F/4
    "rf50": dict(focus=1000.0, pitch=36.0 / 768, half_field=18.0, depth_m=(0.5, 20.0), surfaces=[
        (28.621, 4.20, (1.83481, 42.7), 14.995), (68.136, 0.18, AIR, 14.24), (17.772, 6.70, (1.79952, 42.2), 11.95),
        (59.525, 1.10, (1.80518, 25.4), 10.39), (11.427, 5.27, AIR, 8.39), (None, 6.20, AIR, 8.12 * 1.85 / 4.0),
        (-16.726, 0.90, (1.67270, 32.1), 7.475), (-29.829, 0.83, AIR, 7.73),
        (-25.000, 2.95, (1.53110, 55.9), 7.76, 0.0, (-4.12032e-05, -2.90015e-07, -4.67119e-09, 7.90646e-11, -9.28470e-13)),
        (-18.373, 0.98, AIR, 9.07, 0.0, (-2.41619e-05, -3.29146e-07, 1.91098e-10, -9.28593e-13, -2.29193e-13)),
        (280.004, 4.60, (1.73400, 51.5), 12.215), (-34.002, 25.67, AIR, 12.855)]),
}


def _table(name):
    rows = []
    for s in LENSES[name]["surfaces"]:
        r, t, (nd, vd), semi = s[:4]
        conic, asph = (s[4], s[5]) if len(s) > 4 else (0.0, (0.0,) * 5)
        rows.append([1.0 if r is None else 0.0, 0.0 if r is None else r, t, nd, vd, semi, conic, *asph])
    return np.array(rows)


def _n_surf(name):
    return len(LENSES[name]["surfaces"])


# parameters of a lens a user fits: curvatures and thicknesses, and the conics and a4..a10 of the aspheres
def _param_ids(name):
    ids = []
    for i, s in enumerate(LENSES[name]["surfaces"]):
        if s[0] is not None:
            ids += [8 * i, 8 * i + 7]
            if len(s) > 4:
                ids += [8 * i + j for j in range(1, 6)]
    return ids


def _param_value(lens, pid):
    """The value of a parameter in the lens as focused (lens: the FP64 form of _lens64)."""
    s, j = divmod(pid, 8)
    return {0: lens["c"][s], 1: lens["k"][s], 7: lens["t"][s]}[j] if j in (0, 1, 7) else lens["a"][s][j - 2]


# ---------------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------------
def listed():
    return [
        # a first look at a lens: 32 small PSFs of a singlet (launch-bound)
        dict(name="trace_singlet", family="trace", lens="singlet", F=8, Z=4, NL=1, n=64, ks=31, quadrant=False, dtype="f32"),
        # the bank a renderer needs: 3072 PSFs of 65 x 65 at 256 x 256 pupil samples
        dict(name="trace_bank", family="trace", lens="doublet", F=32, Z=32, NL=3, n=256, ks=65, quadrant=False, dtype="f32"),
        # a service answering requests of any size for two lenses
        dict(name="batch_uneven", family="batch", n_req=4096, n_max=512, dtype="f32"),
        # the paper's own timed workload: a traced PSF for every pixel
        dict(name="psf_map_rf50", family="psf_map", lens="rf50", H=512, W=768, n=64, ks=21, dtype="f32"),
        # a step of a lens fit: the bank traced bilinearly and the gradient of 22 lens parameters
        dict(name="lens_gradient", family="lens_grad", lens="doublet", F=32, Z=32, NL=3, n=128, ks=65),
        # the smallest render: one gray thumbnail
        dict(name="render_thumbnail", family="render", N=1, C=1, H=64, W=64, F=8, Z=4, ks=31, quadrant=False, image="f32", bank="f32"),
        # one RGB image through the full bank in FP32
        dict(name="render_1024", family="render", N=1, C=3, H=1024, W=1024, F=32, Z=32, ks=65, quadrant=False, image="f32", bank="f32"),
        # full-resolution BF16 images for a data set
        dict(name="render_tc_2048", family="render_tc", N=2, C=3, H=2048, W=1536, F=64, Z=64, ks=65, quadrant=False, image="bf16", bank="bf16"),
        # a training step through the render: 8 RGB images, both gradients
        dict(name="render_grad_512", family="render_grad", N=8, C=3, H=512, W=512, F=32, Z=32, ks=65, quadrant=False, image="f32", bank="f32"),
        # the bank's gradient with FP16 images, ragged sizes and a quadrant bank
        dict(name="bank_grad_tc_ragged", family="bank_grad_tc", N=3, C=3, H=397, W=611, F=12, Z=16, ks=51, quadrant=True, image="f16"),
        # the PSF network's map at the paper's size
        dict(name="mlp_map_512", family="mlp_map", H=512, W=768, ks=21, dtype="f32"),
        # an RGB image through a BF16 per-pixel map
        dict(name="render_map_bf16", family="render_map", N=1, C=3, H=512, W=768, ks=21, image="bf16", map="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, lo, hi):
    return min(hi, _log(rng, lo, hi) | 1)


def draw(rng):
    while True:
        c = _draw(rng)
        if _cost(c) <= 1.0:
            return c


def _draw(rng):
    fam = rng.choice(["trace", "trace", "batch", "psf_map", "lens_grad", "render", "render", "render_tc", "render_grad",
                      "bank_grad_tc", "mlp_map", "render_map"])
    if fam in ("trace", "lens_grad"):
        lens = rng.choice(["singlet", "doublet", "spherical"] + (["rf50"] if fam == "trace" else []))
        c = dict(family=fam, lens=lens, F=_log(rng, 2, 32), Z=_log(rng, 2, 32), NL=rng.choice([1, 3]),
                 n=_log(rng, 32, 256 if fam == "trace" else 128), ks=_odd(rng, 15, 127))
        if fam == "trace":
            c.update(quadrant=rng.random() < 0.25, dtype=rng.choice(list(DTYPES)))
            if c["quadrant"]:
                c["F"] = min(c["F"], 12)
        return c
    if fam == "batch":
        return dict(family=fam, n_req=_log(rng, 16, 4096), n_max=_log(rng, 64, 512), dtype=rng.choice(list(DTYPES)))
    if fam == "psf_map":
        return dict(family=fam, lens=rng.choice(list(LENSES)), H=_log(rng, 48, 512), W=_log(rng, 48, 768), n=_log(rng, 16, 64),
                    ks=_odd(rng, 7, 31), dtype=rng.choice(["f32", "bf16"]))
    if fam == "mlp_map":
        return dict(family=fam, H=_log(rng, 48, 512), W=_log(rng, 48, 768), ks=_odd(rng, 11, 31), dtype=rng.choice(["f32", "bf16"]))
    if fam == "render_map":
        image, mp = rng.choice([("f32", "f32"), ("f32", "bf16"), ("bf16", "bf16"), ("f16", "f16")])
        return dict(family=fam, N=rng.choice([1, 1, 2]), C=rng.choice([1, 3]), H=_log(rng, 48, 512), W=_log(rng, 48, 768),
                    ks=_odd(rng, 7, 31), image=image, map=mp)
    big = fam in ("render", "render_tc")
    quadrant = rng.random() < 0.25
    c = dict(family=fam, N=rng.choice([1, 2, 4]), C=rng.choice([1, 3]), H=_log(rng, 64, 1024 if big else 512),
             W=_log(rng, 64, 1024 if big else 512), F=_log(rng, 4, 12 if quadrant else 48), Z=_log(rng, 4, 48),
             ks=_odd(rng, 15, 65), quadrant=quadrant)
    if fam in ("render", "render_grad"):
        c["ks"] = _odd(rng, 15, 127)
        c["image"], c["bank"] = rng.choice([("f32", "f32"), ("f32", "f32"), ("bf16", "bf16"), ("f16", "f16")])
        if fam == "render_grad":
            c["image"] = c["bank"] = "f32"
    else:
        c["image"] = rng.choice(["bf16", "f16"])
        if fam == "render_tc":
            c["bank"] = rng.choice([c["image"], "f32"])
    return c


def _rays(n):
    """In-pupil samples of an n x n pupil grid."""
    a = np.arange(n) * 2 + 1 - n
    return int((a[:, None] ** 2 + a[None, :] ** 2 <= n * n).sum())


def _cells(c):
    return c["F"] ** 2 if c.get("quadrant") else c["F"]


def _ray_surfaces(c):
    if c["family"] in ("trace", "lens_grad"):
        return _cells(c) * c["Z"] * c["NL"] * _rays(c["n"]) * _n_surf(c["lens"])
    if c["family"] == "batch":
        n = c["n_max"]
        mean = (n * n - 32 * 32) / (2 * math.log(max(n, 33) / 32)) * math.pi / 4
        return c["n_req"] * mean * 6
    return c["H"] * c["W"] * _rays(c["n"]) * _n_surf(c["lens"])


def _cost(c):
    """Rough share of the largest listed case's work."""
    if c["family"] in ("trace", "batch", "psf_map", "lens_grad"):
        return _ray_surfaces(c) * (4 if c["family"] == "lens_grad" else 1) / MAX_RAY_SURFACES
    if c["family"] in ("mlp_map", "render_map"):
        return 0.1
    return c["N"] * c["C"] * c["H"] * c["W"] * c["ks"] ** 2 / (8 * 3 * 1024 * 1024 * 65 ** 2)


def work(case):
    c = case
    f = c["family"]
    if f in ("trace", "lens_grad", "batch", "psf_map"):
        flops = 120.0 * _ray_surfaces(c)  # conic root, Newton steps of the aspheres, Snell's law
        if f == "batch":
            out = c["n_req"] * 2 * (15 ** 2 + 31 ** 2 + 65 ** 2 + 127 ** 2) / 4
        else:
            n = c["H"] * c["W"] if f == "psf_map" else _cells(c) * c["Z"] * c["NL"]
            out = n * 2 * c["ks"] ** 2
        nbytes = out * BYTES[c.get("dtype", "f32")]
        if f == "lens_grad":  # the forward, and the rays again with their reverse sweep; the bank's gradient read
            flops, nbytes = flops * 3.5, 2 * nbytes
        return {"bytes": nbytes, "flops": flops}
    px = c["H"] * c["W"]
    if f == "mlp_map":
        nout = 2 * c["ks"] ** 2
        return {"bytes": px * (4 + nout * BYTES[c["dtype"]]) + 2 * 512 * (4 * 512 + nout),
                "flops": 2.0 * px * (3 * 512 + 4 * 512 * 512 + 512 * nout)}
    if f == "render_map":
        return {"bytes": px * 2 * c["ks"] ** 2 * BYTES[c["map"]] + 3 * c["N"] * c["C"] * px * BYTES[c["image"]],
                "flops": 4.0 * c["N"] * c["C"] * px * c["ks"] ** 2}
    img = c["N"] * c["C"] * px
    bank = _cells(c) * c["Z"] * c["C"] * 2 * c["ks"] ** 2
    render = 8.0 * img * c["ks"] ** 2  # two sides, two depth slices, multiply and add
    if f in ("render", "render_tc"):
        return {"bytes": 3 * img * BYTES[c["image"]] + 4 * c["N"] * px + bank * BYTES[c["bank"]], "flops": render}
    if f == "render_grad":  # the forward, then image and bank gradients
        return {"bytes": 4 * (img + 2 * img + c["N"] * px + bank) + 4 * (2 * img + img + c["N"] * px + bank + img + bank),
                "flops": 3 * render}
    return {"bytes": 4 * 2 * img + img * BYTES[c["image"]] + 4 * c["N"] * px + 4 * bank, "flops": render}


# ---------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _pink(seed, n, c, h, w):
    """Images with a 1/f amplitude spectrum, each plane scaled to [0, 1]."""
    fy, fx = torch.fft.fftfreq(h, device="cuda")[:, None], torch.fft.rfftfreq(w, device="cuda")[None]
    f = torch.sqrt(fx * fx + fy * fy)
    f[0, 0] = math.inf
    out = torch.empty((n, c, h, w), device="cuda")
    for i in range(n):
        white = torch.randn((c, h, w), device="cuda", generator=_gen(seed, 100 + i))
        x = torch.fft.irfft2(torch.fft.rfft2(white) / f, s=(h, w))
        lo, hi = x.amin((1, 2), keepdim=True), x.amax((1, 2), keepdim=True)
        out[i] = (x - lo) / (hi - lo)
    return out


def _depth(seed, n, h, w, lo, hi):
    """Smooth depth maps in metres: four octaves of gradient noise, scaled to [lo, hi]."""
    out = torch.empty((n, h, w), device="cuda")
    for i in range(n):
        g = _gen(seed, 200 + i)
        acc = torch.zeros((h, w), device="cuda")
        for o in range(4):
            cells = 4 << o
            ang = torch.rand((cells + 1, cells + 1), device="cuda", generator=g) * (2 * math.pi)
            ys = ((torch.arange(h, device="cuda") + 0.5) / h * cells)[:, None]
            xs = ((torch.arange(w, device="cuda") + 0.5) / w * cells)[None]
            y0, x0 = ys.floor().long(), xs.floor().long()
            fy, fx = ys - y0, xs - x0
            def dot(j, k):
                a = ang[y0 + j, x0 + k]
                return a.cos() * (fx - k) + a.sin() * (fy - j)
            sy, sx = fy ** 3 * (fy * (fy * 6 - 15) + 10), fx ** 3 * (fx * (fx * 6 - 15) + 10)
            top, bottom = torch.lerp(dot(0, 0), dot(0, 1), sx), torch.lerp(dot(1, 0), dot(1, 1), sx)
            acc += 0.5 ** o * (top + (bottom - top) * sy)
        acc = (acc - acc.min()) / (acc.max() - acc.min())
        out[i] = lo + acc * (hi - lo)
    return out


def _psfs(seed, ks, defocus, field, rays):
    """PSF pairs (n, 2, ks, ks): defocus discs, vignetted off axis and split by the dual pixel along x,
    as counts of `rays` rays over the whole disc, sum-normalised.  defocus and field (0..1): (n,) tensors."""
    p = (ks - 1) // 2
    a = torch.arange(-p, p + 1, device="cuda", dtype=torch.float32)
    x, y = a[None, None, :], a[None, :, None]
    r = (defocus.abs() * ks * 1.2 + 1.5)[:, None, None]
    sx = torch.where(defocus < 0, -1.0, 1.0)[:, None, None]
    disc = torch.sigmoid(2.0 * (r - torch.sqrt(x * x + y * y)))
    xs = x - field[:, None, None] * 0.6 * r
    disc = disc * torch.sigmoid(2.0 * (r - torch.sqrt(xs * xs + y * y)))
    left = (0.5 + 0.9 * sx * x / r).clamp(0.02, 0.98)
    mean = torch.stack([disc * left, disc * (1 - left)], 1) * (0.8 * rays / (math.pi * r * r))[:, None]
    counts = torch.poisson(mean, generator=_gen(seed, 300))
    return counts / counts.sum((1, 2, 3), keepdim=True).clamp_min(1.0)


def _axes(c, lens):
    o = LENSES[lens]
    inv = np.linspace(1 / o["depth_m"][0], 1 / o["depth_m"][1], c["Z"])
    return o, 1 / inv


def _bank(c, seed):
    """A bank over fields (or the first quadrant's) x depths x wavelengths, its heights and depths."""
    o, depths = _axes(c, "doublet")
    half = 0.5 * math.hypot(c["H"], c["W"]) * o["pitch"]
    heights = np.linspace(0.0, half, c["F"])
    h = np.hypot(heights[:, None], heights[None]).reshape(-1) / math.hypot(half, half) if c["quadrant"] else heights / half
    f = torch.tensor(h, device="cuda", dtype=torch.float32)
    z = torch.tensor(1 / depths - 1.0, device="cuda", dtype=torch.float32)
    field = f[:, None, None].expand(len(h), c["Z"], c["C"])
    lam = torch.tensor([0.03 * (i - (c["C"] - 1) / 2) for i in range(c["C"])], device="cuda")
    defocus = (z[None, :, None] + lam).expand_as(field)
    bank = _psfs(seed, c["ks"], defocus.reshape(-1), field.reshape(-1), 12868)
    return bank.view(len(h), c["Z"], c["C"], 2, c["ks"], c["ks"]), heights, depths, o["pitch"]


def _requests(c, seed):
    """Requests as a structured array (fields of the entry points' request record)."""
    rng = np.random.default_rng(seed)
    names = [("h_mm", "f8"), ("depth_mm", "f8"), ("lambda_nm", "f8"), ("n_grid", "i4"), ("ks", "i4"), ("lens", "i4"), ("v_mm", "f8")]
    if c["family"] == "batch":
        q = np.zeros(c["n_req"], dtype=names)
        n = len(q)
        q["n_grid"] = np.exp(rng.uniform(math.log(32), math.log(c["n_max"]), n)).astype(np.int32)
        q["ks"] = rng.permutation(np.resize([15, 31, 65, 127], n))
        q["h_mm"], q["depth_mm"] = rng.uniform(0, 1.448, n), 1 / rng.uniform(1 / 3000.0, 1 / 300.0, n)
        q["lambda_nm"], q["lens"] = rng.choice(LAMBDAS, n), rng.integers(0, 2, n)
        return q
    o, depths = _axes(c, c["lens"])
    # the field of a bank ends where its image does, the depths where the scene does: both vary
    h = np.linspace(0.0, o["half_field"] * rng.uniform(0.85, 1.0), c["F"])
    depths = depths * rng.uniform(0.95, 1.05)
    lam = LAMBDAS if c["NL"] == 3 else LAMBDAS[1:2]
    if c["quadrant"]:
        g = np.array([(x, y, d, w) for x in h for y in h for d in depths for w in lam])
    else:
        g = np.array([(x, 0.0, d, w) for x in h for d in depths for w in lam])
    q = np.zeros(len(g), dtype=names)
    q["h_mm"], q["v_mm"], q["depth_mm"], q["lambda_nm"] = g[:, 0], g[:, 1], g[:, 2] * 1000, g[:, 3]
    q["n_grid"], q["ks"] = c["n"], c["ks"]
    return q


def _lens(name):
    return sd.Lens(_table(name), LENSES[name]["focus"])


BATCH_LENSES = ("doublet", "spherical")


def _network(seed, ks):
    """A network of trained scale: He-initialised, the last layer biased like a blur disc."""
    g = torch.Generator().manual_seed(1000003 * int(seed) + 7)
    w, b = [], []
    for out, inp in sd.MLP_SHAPES(ks):
        w.append((torch.randn((out, inp), generator=g) * math.sqrt(2.0 / inp)).numpy())
        b.append((torch.randn(out, generator=g) * 0.1).numpy())
    return w, b


def _map(c, seed):
    depth = _depth(seed, 1, c["H"], c["W"], 0.5, 20.0)[0].reshape(-1)
    out = torch.empty((c["H"] * c["W"], 2, c["ks"], c["ks"]), device="cuda", dtype=DTYPES[c["map"]])
    for i in range(0, len(out), 65536):
        d = depth[i:i + 65536]
        out[i:i + 65536] = _psfs(seed + i, c["ks"], 0.25 * (1 / d - 1), torch.linspace(0, 1, len(d), device="cuda"), 3228)
    return out.view(c["H"], c["W"], 2, c["ks"], c["ks"])


def _images(c, seed):
    o = LENSES["doublet"]["depth_m"]
    return _pink(seed, c["N"], c["C"], c["H"], c["W"]).to(DTYPES[c["image"]]), _depth(seed, c["N"], c["H"], c["W"], *o)


def _layout(c, heights, depths, pitch, dtype):
    return sd.BankLayout(heights, depths, c["C"], c["ks"], pitch, DTYPES[dtype],
                         sd.SD_FIELD_QUADRANT if c["quadrant"] else sd.SD_FIELD_RADIAL)


def _upstream(c, seed, n_req):
    """A loss's gradient of the bank: smooth patches, zero for the PSFs that no pixel uses."""
    g = torch.randn((n_req, 2, c["ks"], c["ks"]), device="cuda", generator=_gen(seed, 400))
    g = torch.nn.functional.avg_pool2d(g, 5, 1, 2)
    return (g * (torch.rand((n_req, 1, 1, 1), device="cuda", generator=_gen(seed, 401)) < 0.6)).reshape(-1)


def prepare(case, seed):
    c, f = case, case["family"]
    s = {"case": c}
    if f in ("trace", "lens_grad", "batch"):
        q = _requests(dict(quadrant=False, **c) if f != "trace" else c, seed)
        s["req"], s["total"], _ = sd.make_requests(q)
        s["n_req"] = len(q)
        s["sensor"] = sd.DPSensor(LENSES[c["lens"]]["pitch"] if f != "batch" else 0.002)
    if f == "batch":
        s["trace"] = sd.BatchedTrace([_lens(n) for n in BATCH_LENSES], s["sensor"], s["req"], s["n_req"], s["total"], max_ks=127,
                                     max_n=c["n_max"], dtype=DTYPES[c["dtype"]])
    elif f == "trace":
        s["lens"] = _lens(c["lens"])
    elif f == "psf_map":
        s["lens"], s["sensor"] = _lens(c["lens"]), sd.DPSensor(2 * LENSES[c["lens"]]["half_field"] / 768)
        s["depth"] = _depth(seed, 1, c["H"], c["W"], *LENSES[c["lens"]]["depth_m"])[0]
    elif f == "lens_grad":
        s["lens"], s["pids"], s["g"] = _lens(c["lens"]), _param_ids(c["lens"]), _upstream(c, seed, s["n_req"])
        l64 = _lens64(c["lens"])
        s["theta"] = torch.tensor([_param_value(l64, i) for i in s["pids"]], dtype=torch.float64, requires_grad=True)
    elif f == "mlp_map":
        s["net"] = sd.PsfMLP(*_network(seed, c["ks"]), c["ks"])
        s["depth"] = _depth(seed, 1, c["H"], c["W"], 0.5, 20.0)[0]
    elif f == "render_map":
        s["aif"], s["map"] = _pink(seed, c["N"], c["C"], c["H"], c["W"]).to(DTYPES[c["image"]]), _map(c, seed)
    else:
        s["aif"], s["depth"] = _images(c, seed)
        bank, *axes = _bank(c, seed)
        s["layout"] = _layout(c, *axes, c.get("bank", "f32"))
        s["bank"] = bank.to(DTYPES[c.get("bank", "f32")])
        if f in ("render_grad", "bank_grad_tc"):
            s["g"] = torch.randn((c["N"], 2 * c["C"], c["H"], c["W"]), device="cuda", generator=_gen(seed, 500)) * 1e-3
        if f == "render_grad":
            s["aif"].requires_grad_(True)
            s["bank"].requires_grad_(True)
    return s


def run(s):
    c, f = s["case"], s["case"]["family"]
    if f == "trace":
        return sd.dp_psf_trace(s["lens"], s["sensor"], s["req"], s["n_req"], s["total"], max_ks=c["ks"], max_n=c["n"],
                               dtype=DTYPES[c["dtype"]])
    if f == "batch":
        return s["trace"].run()
    if f == "psf_map":
        return sd.dp_psf_map(s["lens"], s["sensor"], s["depth"], 550.0, c["n"], c["ks"], dtype=DTYPES[c["dtype"]])
    if f == "lens_grad":
        psf = sd.dp_psf_trace_autograd(s["theta"], s["lens"], s["pids"], s["sensor"], s["req"], s["n_req"], s["total"],
                                       max_ks=c["ks"], max_n=c["n"])
        return psf.detach(), torch.autograd.grad(psf, s["theta"], s["g"])[0]
    if f == "render":
        return sd.dp_render(s["aif"], s["depth"], s["bank"], s["layout"])
    if f == "render_tc":
        return sd.dp_render_tc(s["aif"], s["depth"], s["bank"], s["layout"])
    if f == "render_grad":
        out = sd.dp_render_autograd(s["aif"], s["bank"], s["depth"], s["layout"])
        return (out.detach(), *torch.autograd.grad(out, (s["aif"], s["bank"]), s["g"]))
    if f == "bank_grad_tc":
        return sd.dp_render_bank_grad_tc(s["g"], s["aif"], s["depth"], s["layout"])
    if f == "mlp_map":
        return sd.mlp_psf_map(s["net"], s["depth"], 0.5, 20.0, dtype=DTYPES[c["dtype"]])
    return sd.dp_render_map(s["aif"], s["map"])


# ---------------------------------------------------------------------------------------------------
# The same in 64 bits: the trace
# ---------------------------------------------------------------------------------------------------
def _lens64(name):
    """FP64 lens: curvatures, thicknesses (focused), conics, aspheres, apertures, Cauchy coefficients."""
    L = dict(c=[], t=[], k=[], a=[], sd=[], A=[], B=[], stop=[])
    for s in LENSES[name]["surfaces"]:
        r, t, (nd, vd), semi = s[:4]
        L["c"].append(0.0 if r is None else 1.0 / r)
        L["t"].append(t)
        L["k"].append(s[4] if len(s) > 4 else 0.0)
        L["a"].append(tuple(s[5]) if len(s) > 4 else (0.0,) * 5)
        L["sd"].append(semi)
        L["stop"].append(r is None)
        b = 0.0 if vd <= 0 or nd == 1 else (nd - 1) / vd / (0.4861327 ** -2 - 0.6562725 ** -2)
        L["B"].append(b)
        L["A"].append(nd - b / 0.5875618 ** 2)
    n = len(L["c"])
    y, u, n1 = 1.0, 1.0 / LENSES[name]["focus"], 1.0
    for s in range(n):  # the sensor in focus for the focus distance
        n2 = L["A"][s] + L["B"][s] / 0.5875618 ** 2
        u, n1 = (n1 * u - y * (n2 - n1) * L["c"][s]) / n2, n2
        y = y + (L["t"][s] if s < n - 1 else 0.0) * u
    L["t"][-1] = -y / u
    return L


def _parax(L, nl, y, u, to):
    n1 = torch.ones_like(nl[0])
    for s in range(to):
        if not L["stop"][s]:
            u = (n1 * u - y * (nl[s] - n1) * L["c"][s]) / nl[s]
        n1 = nl[s]
        y = y + L["t"][s] * u
    return y


def _trace64(L, q, theta=None):
    """All in-pupil rays of the requests q (dict of per-request FP64 tensors) through the lens.  Returns the
    request of each ray, the landing points, tan(theta) and whether it arrives.  theta: {(surface, j): tensor}
    replaces parameters in the surfaces (not in the ray generation)."""
    n = len(L["c"])
    stop = L["stop"].index(True)
    nl = [L["A"][s] + L["B"][s] / (q["lam"] * 1e-3) ** 2 for s in range(n)]
    one, zero = torch.ones_like(q["h"]), torch.zeros_like(q["h"])
    ay, by = _parax(L, nl, one, zero, stop), _parax(L, nl, zero, one, stop)
    z_ep, r_ep = by / ay, (L["sd"][stop] / ay).abs()
    u0 = -1 / (z_ep + q["depth"])
    m = _parax(L, nl, 1 + u0 * q["depth"], u0, n)
    z_front = 0.0
    if not L["stop"][0]:
        c, u = L["c"][0], L["sd"][0] ** 2
        z_front = min(0.0, c * u / (1 + math.sqrt(max(0.0, 1 - c * c * u))))
    z0 = torch.where(z_ep <= z_front, z_ep, torch.full_like(z_ep, z_front - 1.0))
    # the pupil grid of every request, cut to the disc
    cells = q["n"] ** 2
    req = torch.repeat_interleave(torch.arange(len(cells), device="cuda"), cells)
    first = torch.cumsum(cells, 0) - cells
    k = torch.arange(len(req), device="cuda") - first[req]
    iy = torch.div(k, q["n"][req], rounding_mode="floor")
    ax, ayy = 2 * (k - iy * q["n"][req]) + 1 - q["n"][req], 2 * iy + 1 - q["n"][req]
    keep = ax * ax + ayy * ayy <= q["n"][req] ** 2
    req, ax, ayy = req[keep], ax[keep], ayy[keep]
    sc = (r_ep / q["n"])[req]
    xo, yo = (q["h"] / m)[req], (q["v"] / m)[req]
    vx, vy, vz = ax * sc - xo, ayy * sc - yo, (z_ep + q["depth"])[req]
    inv = 1 / torch.sqrt(vx * vx + vy * vy + vz * vz)
    dx, dy, dz = vx * inv, vy * inv, vz * inv
    f = ((z0 + q["depth"]) / (z_ep + q["depth"]))[req]
    x, y, z = xo + f * vx, yo + f * vy, z0[req]
    ok = torch.ones_like(x, dtype=torch.bool)
    get = (lambda s, j, v: theta.get((s, j), v)) if theta else (lambda s, j, v: v)
    n1 = torch.ones_like(nl[0])
    for s in range(n):
        c, kk, asph = get(s, 0, L["c"][s]), 1 + get(s, 1, L["k"][s]), [get(s, 2 + j, L["a"][s][j]) for j in range(5)]
        newton = any(v != 0 for v in L["a"][s])
        if L["c"][s] == 0:
            t = -z / dz
        else:
            A = c * (1 + (kk - 1) * dz * dz)
            B = dz - c * (x * dx + y * dy + kk * z * dz)
            C = c * (x * x + y * y + kk * z * z) - 2 * z
            disc = B * B - A * C
            ok = ok & (disc >= 0)
            t = C / (B + torch.sqrt(disc.clamp_min(1e-30)))

        def sag(u):
            root = torch.sqrt((1 - kk * c * c * u).clamp_min(1e-30))
            poly = u * u * (asph[0] + u * (asph[1] + u * (asph[2] + u * (asph[3] + u * asph[4]))))
            d = 0.5 * c / root + u * (2 * asph[0] + u * (3 * asph[1] + u * (4 * asph[2] + u * (5 * asph[3] + u * 6 * asph[4]))))
            return c * u / (1 + root) + poly, d

        if newton:
            with torch.no_grad():
                for _ in range(7):
                    px, py = x + t * dx, y + t * dy
                    zs, d = sag(px * px + py * py)
                    t = t - (z + t * dz - zs) / (dz - 2 * d * (px * dx + py * dy))
                px, py = x + t * dx, y + t * dy
                dF = dz - 2 * sag(px * px + py * py)[1] * (px * dx + py * dy)
            px, py = x + t * dx, y + t * dy  # one differentiable step at the root
            t = t - (z + t * dz - sag(px * px + py * py)[0]) / dF
        x, y, z = x + t * dx, y + t * dy, z + t * dz
        u = x * x + y * y
        ok = ok & (u <= L["sd"][s] ** 2)
        if not L["stop"][s]:
            d = sag(u)[1]
            nx, ny = -2 * x * d, -2 * y * d
            inv = 1 / torch.sqrt(nx * nx + ny * ny + 1)
            nx, ny, nz = nx * inv, ny * inv, inv
            e = (n1 / nl[s])[req]
            cosi = nx * dx + ny * dy + nz * dz
            k2 = 1 - e * e * (1 - cosi * cosi)
            ok = ok & (k2 >= 0)
            g = torch.sqrt(k2.clamp_min(1e-30)) - e * cosi
            dx, dy, dz = e * dx + g * nx, e * dy + g * ny, e * dz + g * nz
        n1 = nl[s]
        z = z - get(s, 7, L["t"][s])
    ok = ok & (dz > 0)
    t = -z / dz
    return req, x + t * dx, y + t * dy, dx / dz, ok


def _binned64(L, pitch, q, ks, bilinear, theta=None):
    """Summed PSF pairs of the requests, flat at each one's offset `at` (bilinear: and by the launched rays)."""
    req, x, y, tan, ok = _trace64(L, q, theta)
    p = (q["ks"][req] - 1) // 2
    fx, fy = (x - q["h"][req]) / pitch + p, (y - q["v"][req]) / pitch + p
    with torch.no_grad():
        af, bf = torch.floor(fx + 0.5), torch.floor(fy + 0.5)
        ex, ey = (fx - af) * pitch, (fy - bf) * pitch
        h, fl, w, r = 0.78 * pitch, 1.44 * pitch, 0.30 * pitch, 0.50 * pitch
        sp = torch.where(ex * ex + ey * ey <= r * r, ex * (fl - h) / fl, ex) + h * tan
        side = torch.where(sp >= 0, 0, 1)
        ok = ok & (sp >= -w) & (sp < w)
    k = q["ks"][req]
    out = torch.zeros(int(2 * (q["ks"] ** 2).sum()), device="cuda", dtype=torch.float64)

    def put(out, a, b, wgt):
        hit = ok & (a >= 0) & (a < k) & (b >= 0) & (b < k)
        i = q["at"][req] + side * k * k + b * k + a
        return out.index_add(0, i[hit], wgt[hit])

    if not bilinear:
        out = put(out, af.long(), bf.long(), torch.ones_like(fx))
    else:
        a0, b0 = torch.floor(fx.detach()), torch.floor(fy.detach())
        wx, wy = fx - a0, fy - b0
        for j in (0, 1):
            for i in (0, 1):
                out = put(out, (a0 + i).long(), (b0 + j).long(), (wx if i else 1 - wx) * (wy if j else 1 - wy))
        n = torch.bincount(req, minlength=len(q["n"])).double()
        out = out / torch.repeat_interleave(n, 2 * q["ks"] ** 2)
    return out


def _chunks(q, most):
    """Slices of the requests with at most `most` pupil samples each."""
    cells = np.asarray(q["n_grid"], dtype=np.int64) ** 2
    i = 0
    while i < len(q):
        j, n = i, 0
        while j < len(q) and (j == i or n + cells[j] <= most):
            n, j = n + cells[j], j + 1
        yield i, j
        i = j


def _q64(q):
    ks = torch.tensor(q["ks"].astype(np.int64), device="cuda")
    d = {n: torch.tensor(np.ascontiguousarray(q[f]), device="cuda", dtype=torch.float64)
         for n, f in (("h", "h_mm"), ("v", "v_mm"), ("depth", "depth_mm"), ("lam", "lambda_nm"))}
    return {**d, "n": torch.tensor(q["n_grid"].astype(np.int64), device="cuda"), "ks": ks,
            "at": torch.cumsum(2 * ks * ks, 0) - 2 * ks * ks}


def _normalised(psf, ks):
    """Flat PSF pairs divided by their sums."""
    size = torch.as_tensor(2 * np.asarray(ks, dtype=np.int64) ** 2, device="cuda")
    pair = torch.repeat_interleave(torch.arange(len(size), device="cuda"), size)
    total = torch.zeros(len(size), device="cuda", dtype=torch.float64).index_add(0, pair, psf)
    return psf / total.clamp_min(1.0)[pair]


def _exact_trace(c, seed):
    q = _requests(c, seed)
    L = _lens64(c["lens"])
    parts = [_binned64(L, LENSES[c["lens"]]["pitch"], _q64(q[i:j]), c["ks"], False) for i, j in _chunks(q, 4 << 20)]
    return _normalised(torch.cat(parts), q["ks"]), None


def _exact_batch(c, seed):
    q = _requests(c, seed)
    size = 2 * q["ks"].astype(np.int64) ** 2
    at = np.cumsum(size) - size
    out = torch.zeros(int(size.sum()), device="cuda", dtype=torch.float64)
    for li, name in enumerate(BATCH_LENSES):
        mine = np.flatnonzero(q["lens"] == li)
        L = _lens64(name)
        for i, j in _chunks(q[mine], 4 << 20):
            idx = mine[i:j]
            part = _binned64(L, 0.002, _q64(q[idx]), None, False)
            n = 0
            for r in idx:
                out[at[r]:at[r] + size[r]] = part[n:n + size[r]]
                n += size[r]
    return _normalised(out, q["ks"]), None


def _exact_psf_map(c, seed):
    L, o = _lens64(c["lens"]), LENSES[c["lens"]]
    pitch = 2 * o["half_field"] / 768
    depth = _depth(seed, 1, c["H"], c["W"], *o["depth_m"])[0].double()
    row, col = torch.meshgrid(torch.arange(c["H"], device="cuda"), torch.arange(c["W"], device="cuda"), indexing="ij")
    h, v = (col - 0.5 * (c["W"] - 1)).double().mul(pitch).reshape(-1), (row - 0.5 * (c["H"] - 1)).double().mul(pitch).reshape(-1)
    out = torch.empty((c["H"] * c["W"], 2 * c["ks"] ** 2), device="cuda")
    step = max(1, (8 << 20) // c["n"] ** 2)
    for i in range(0, len(out), step):
        n = len(h[i:i + step])
        ks = torch.full((n,), c["ks"], device="cuda")
        q = dict(h=h[i:i + step], v=v[i:i + step], depth=depth.reshape(-1)[i:i + step] * 1000, lam=torch.full((n,), 550.0, device="cuda").double(),
                 n=torch.full((n,), c["n"], device="cuda"), ks=ks, at=torch.arange(n, device="cuda") * 2 * c["ks"] ** 2)
        psf = _binned64(L, pitch, q, c["ks"], False).view(n, -1)
        out[i:i + step] = psf / psf.sum(1, keepdim=True).clamp_min(1.0)
    return out.view(c["H"], c["W"], 2, c["ks"], c["ks"]), None


def _exact_lens_grad(c, seed):
    c = dict(quadrant=False, **c)
    q, L, pids = _requests(c, seed), _lens64(c["lens"]), _param_ids(c["lens"])
    theta = torch.tensor([_param_value(L, i) for i in pids], device="cuda", dtype=torch.float64, requires_grad=True)
    g = _upstream(c, seed, len(q)).double()
    psf, grad, size = [], torch.zeros_like(theta), 2 * c["ks"] ** 2
    for i, j in _chunks(q, 1 << 20):
        part = _binned64(L, LENSES[c["lens"]]["pitch"], _q64(q[i:j]), c["ks"], True,
                         {divmod(p, 8): theta[k] for k, p in enumerate(pids)})
        grad += torch.autograd.grad(part, theta, g[i * size:j * size])[0]
        psf.append(part.detach())
    return torch.cat(psf), grad.cpu()


# ---------------------------------------------------------------------------------------------------
# The same in 64 bits: the renders and the network
# ---------------------------------------------------------------------------------------------------
def _select(c, heights, depths, pitch, depth):
    """Each pixel's bank key and depth weight, in the entry points' FP32 operations: the nearest field height
    and the depth's bracket in inverse depth."""
    H, W = depth.shape[-2:]
    fh = torch.tensor(heights, device="cuda", dtype=torch.float32)
    iq = 1.0 / torch.tensor(depths, device="cuda", dtype=torch.float32)
    ps = torch.tensor(pitch, device="cuda", dtype=torch.float32)
    X = ((torch.arange(W, device="cuda").float() - 0.5 * (W - 1)) * ps)[None, :].expand(H, W)
    Y = ((torch.arange(H, device="cuda").float() - 0.5 * (H - 1)) * ps)[:, None].expand(H, W)

    def nearest(r):
        lo = (torch.searchsorted(fh, r.contiguous(), right=True) - 1).clamp(0, len(fh) - 1)
        hi = (lo + 1).clamp_max(len(fh) - 1)
        return torch.where(fh[hi] - r < r - fh[lo], hi, lo)

    if c["quadrant"]:
        f = ((X < 0).long() + 2 * (Y < 0).long()) * c["F"] ** 2 + nearest(X.abs()) * c["F"] + nearest(Y.abs())
    else:
        f = nearest(torch.sqrt(X * X + Y * Y))
    q = 1.0 / depth
    z = (torch.searchsorted(-iq, -q, right=True) - 1).clamp(0, len(iq) - 2)
    t = ((iq[z] - q) / (iq[z] - iq[z + 1])).clamp(0, 1)
    return f[None] * c["Z"] + z, t.double()


def _flip_classes(c, bank):
    """The quadrant bank's four flip classes stacked (a radial bank as it is)."""
    if not c["quadrant"]:
        return bank
    fx = bank.flip(-1).flip(-3)
    return torch.cat([bank, fx, bank.flip(-2), fx.flip(-2)])


def _exact_render(c, seed, backward=False):
    aif, depth = _images(c, seed)
    bank, heights, depths, pitch = _bank(c, seed)
    dt = DTYPES[c.get("bank", "f32")]
    if c["family"] == "render_tc":
        dt = DTYPES[c["image"]]  # the tensor cores' operands share the image's type
    if c["family"] in ("render_tc", "render") and 8.0 * aif.numel() * c["ks"] ** 2 > 2e12:
        return None
    ks, p = c["ks"], (c["ks"] - 1) // 2
    K = _flip_classes(c, bank.to(dt)).double().flip(-1, -2).reshape(-1, c["C"], 2, ks * ks)
    key, t = _select(c, heights, depths, pitch, depth)
    N, C, H, W = aif.shape
    pad = torch.nn.functional.pad(aif.double(), (p, p, p, p), mode="replicate")
    Hp, Wp = pad.shape[-2:]
    offs = (torch.arange(ks, device="cuda")[:, None] * Wp + torch.arange(ks, device="cuda")).reshape(-1)
    key, t = key.reshape(-1), t.reshape(-1)
    order = torch.argsort(key)
    keys, counts = torch.unique_consecutive(key[order], return_counts=True)
    out = torch.empty((N * H * W, C, 2), device="cuda", dtype=torch.float64)
    flat = pad.permute(1, 0, 2, 3).reshape(C, -1)
    if backward:
        g = (torch.randn((N, 2 * C, H, W), device="cuda", generator=_gen(seed, 500)) * 1e-3).double()
        g = g.view(N, 2, C, H * W).permute(0, 3, 2, 1).reshape(-1, C, 2)
        gK, gI = torch.zeros_like(K), torch.zeros_like(flat)
    at = 0
    most = max(1, (1 << 27) // (ks * ks))
    for k, n in zip(keys.tolist(), counts.tolist()):
        for i in range(at, at + n, most):
            px = order[i:min(i + most, at + n)]
            img, rc = px // (H * W), px % (H * W)
            base = img * (Hp * Wp) + (rc // W) * Wp + rc % W
            idx = base[:, None] + offs
            w = t[px][:, None]
            for ch in range(C):
                patch = flat[ch][idx]
                pair = K[k:k + 2, ch].reshape(-1, ks * ks)  # (slice, side)
                r = (patch @ pair.T).view(-1, 2, 2)
                out[px, ch] = (1 - w) * r[:, 0] + w * r[:, 1]
                if backward:
                    wg = torch.cat([(1 - w) * g[px, ch], w * g[px, ch]], 1)
                    gK[k:k + 2, ch] += (wg.T @ patch).view(2, 2, -1)
                    gI[ch].index_add_(0, idx.reshape(-1), (wg @ pair).reshape(-1))
        at += n
    out = out.view(N, H * W, C, 2).permute(0, 3, 2, 1).reshape(N, 2 * C, H, W)
    if not backward:
        return out
    # the padding folds onto the edges; the flip classes onto the stored quadrant
    gI = gI.view(C, N, Hp, Wp).permute(1, 0, 2, 3)
    for dim, n in ((2, H), (3, W)):
        i = (torch.arange(n + 2 * p, device="cuda") - p).clamp(0, n - 1)
        shape = list(gI.shape)
        shape[dim] = n
        gI = torch.zeros(shape, device="cuda", dtype=torch.float64).index_add_(dim, i, gI)
    gK = gK.view(-1, c["Z"], C, 2, ks, ks).flip(-1, -2)
    if c["quadrant"]:
        a, b, d, e = gK.chunk(4)
        gK = a + b.flip(-3).flip(-1) + d.flip(-2) + e.flip(-2).flip(-3).flip(-1)
    return out, gI, gK


def _exact_mlp(c, seed):
    w, b = _network(seed, c["ks"])
    w, b = ([torch.tensor(v, device="cuda").double() for v in x] for x in (w, b))
    depth = _depth(seed, 1, c["H"], c["W"], 0.5, 20.0)[0].double()
    H, W = depth.shape
    y, x = torch.meshgrid(torch.arange(H, device="cuda").double(), torch.arange(W, device="cuda").double(), indexing="ij")
    pts = torch.stack([(x - 0.5 * (W - 1)) / (0.5 * W), (y - 0.5 * (H - 1)) / (0.5 * H), 2 * (depth - 0.5) / 19.5 - 1], -1).view(-1, 3)
    out = torch.empty((H * W, 2 * c["ks"] ** 2), device="cuda")
    for i in range(0, H * W, 32768):
        h = pts[i:i + 32768]
        for l in range(6):
            h = torch.relu(h @ w[l].T + b[l])
        s = h.sum(1, keepdim=True)
        out[i:i + 32768] = torch.where(s > 0, h / s.clamp_min(1e-300), torch.zeros_like(h))
    return out.view(H, W, 2, c["ks"], c["ks"]), None


def _exact_render_map(c, seed):
    aif = _pink(seed, c["N"], c["C"], c["H"], c["W"]).to(DTYPES[c["image"]]).double()
    mp, ks, p = _map(c, seed), c["ks"], (c["ks"] - 1) // 2
    pad = torch.nn.functional.pad(aif, (p, p, p, p), mode="replicate")
    out = torch.zeros((c["N"], 2, c["C"], c["H"], c["W"]), device="cuda", dtype=torch.float64)
    for u in range(ks):
        for v in range(ks):
            k = mp[:, :, :, ks - 1 - u, ks - 1 - v].double().permute(2, 0, 1)
            out += pad[:, None, :, u:u + c["H"], v:v + c["W"]] * k[None, :, None]
    return out.view(c["N"], 2 * c["C"], c["H"], c["W"])


def exact(case, seed):
    f = case["family"]
    if f == "render_grad":
        return _exact_render(case, seed, backward=True)
    if f == "bank_grad_tc":
        return _exact_render(case, seed, backward=True)[2]
    return {"trace": _exact_trace, "batch": _exact_batch, "psf_map": _exact_psf_map, "lens_grad": _exact_lens_grad,
            "render": _exact_render, "render_tc": _exact_render, "mlp_map": _exact_mlp,
            "render_map": _exact_render_map}[f](case, seed)
