"""The work this framework is used for, as cases that can be timed and compared.

A case is one call (or one pass of a request loop) through the public Python
entry points on seeded synthetic frames: whole-frame extraction from 1 to
151 megapixels in both pixel types, with and without a bad-pixel mask, at
aligned and ragged sizes; several small frames in one batched call; the request
server with frames in host memory; the learned background's extraction and its
training step; photometry at a list of known stars; the cosmetic filters; the
second detection pass with a varying PSF; and deblending.  The frames follow
the recipes of synth/ (FP32 with a sky gradient, a uint16 CCD with hot pixels
and cosmic rays, a dense uint16 field with nebulosity), drawn on the GPU.

listed() holds one case per use; draw() gives others from the same ranges.
exact() evaluates the same quantities in 64 bits with plain torch and numpy.
"""
import math

import numpy as np
import torch

import paper_2609_32375_gb300 as gp
from paper_2609_32375_gb300 import learned

DEV = "cuda"
MINAREA = 5
SAT = 65535.0

# Frame recipes: dtype, sky level (ADU), gain (e-/ADU), read noise (e-), stars
# per megapixel, their flux range (F^-1.5), FWHM range (px).
RECIPES = {
    "sky_f32": dict(u16=False, sky=1000.0, gain=1.0, rn=5.0, stars=286.0, flux=(1e2, 1e5), fwhm=(3.0, 3.0)),
    "ccd_u16": dict(u16=True, sky=800.0, gain=1.5, rn=8.0, stars=477.0, flux=(2e2, 2e5), fwhm=(2.0, 5.0)),
    "dense_u16": dict(u16=True, sky=2000.0, gain=1.0, rn=3.0, stars=886.0, flux=(1e2, 1e5), fwhm=(3.0, 3.0)),
}


def listed():
    return [
        # the smallest whole frame of the configurations: launches and single-CTA stages count
        dict(name="extract 1MP f32", kind="extract", recipe="sky_f32", w=1024, h=1024, mesh=64, taps=5, thresh=1.5,
             radii="3,5,8", masked=False),
        # an ordinary CCD frame (the paper's smallest camera): hot pixels, cosmic rays, saturation
        dict(name="extract 4MP ccd u16", kind="extract", recipe="ccd_u16", w=2048, h=2048, mesh=128, taps=5,
             thresh=3.0, radii="4,8", masked=False),
        # a calibrated FP32 frame of a ragged size with its bad-pixel mask, unaligned rows
        dict(name="extract 9MP f32 masked", kind="extract", recipe="sky_f32", w=3001, h=2999, mesh=64, taps=5,
             thresh=1.5, radii="3,6,10", masked=True),
        # the headline: the dense 151 MP uint16 frame
        dict(name="extract 151MP dense u16", kind="extract", recipe="dense_u16", w=12288, h=12304, mesh=256, taps=5,
             thresh=1.5, radii="3,6,10", masked=False),
        # a burst of small frames extracted in one call
        dict(name="batch 8x4MP dense u16", kind="batch", recipe="dense_u16", w=2048, h=2048, frames=8, mesh=256,
             taps=5, thresh=1.5, radii="3,6,10"),
        # the serving loop: frames of two sizes arrive in pinned host memory, catalogs go back to the host
        dict(name="serve 6x4MP 2x17MP", kind="serve", recipe="dense_u16", w=2048, h=2048, frames=6, big=2, mesh=256,
             taps=5, thresh=1.5, radii="3,6,10"),
        # extraction with the network's background, on the frames it was trained for
        dict(name="learned 17MP f32", kind="learned", recipe="sky_f32", w=4096, h=4096, mesh=64, taps=5, thresh=1.5,
             radii="3,5,8"),
        # one training step of that network (forward, backward, AdamW) at its training batch
        dict(name="train 32x64x64", kind="train", n=32, h=64, w=64),
        # photometry at a list of known stars: exact apertures, growth curves, the optimal radius
        dict(name="photometry 17MP 15k", kind="photometry", recipe="dense_u16", w=4096, h=4096, mesh=256, taps=5,
             radii="3,6,10", rows=15000),
        # cosmic rays and salt-and-pepper noise taken out of a raw CCD frame
        dict(name="cosmetic 17MP ccd u16", kind="cosmetic", recipe="ccd_u16", w=4096, h=4096, rtn=True, cr=True),
        # the second detection pass, a 13 x 13 reference PSF and 5 modes
        dict(name="psf 17MP 5 modes", kind="psf", recipe="dense_u16", w=4096, h=4096, mesh=256, size=13, modes=5,
             tile=2048, thresh=1.5),
        # deblending of a crowded field's segments
        dict(name="deblend 17MP dense u16", kind="deblend", recipe="dense_u16", w=4096, h=4096, mesh=256, taps=5,
             thresh=1.5),
    ]


def _size(rng, lo_mp, hi_mp):
    """Width and height of log-uniform area and an aspect ratio up to 2; a third multiples of 64, a third odd."""
    while True:
        area = math.exp(rng.uniform(math.log(lo_mp), math.log(hi_mp))) * 1e6
        w = math.sqrt(area * 2.0 ** rng.uniform(-1, 1))
        h = area / w
        form = rng.randrange(3)
        w, h = [(max(1, round(v / 64)) * 64, round(v) | 1, round(v))[form] for v in (w, h)]
        if w * h <= hi_mp * 1.02e6:
            return w, h


def draw(rng):
    kind = rng.choice(["extract", "extract", "extract", "batch", "serve", "learned", "train", "photometry",
                       "cosmetic", "psf", "deblend"])
    recipe = rng.choice(sorted(RECIPES))
    u16 = RECIPES[recipe]["u16"]
    det = dict(mesh=rng.choice((32, 64, 128, 256) if u16 else (32, 64, 128)), taps=rng.choice((3, 5, 5, 7)),
               thresh=rng.choice((1.5, 2.0, 3.0)))
    radii = rng.choice(("3,6,10", "4,8", "3,5,8", "2.5", "2,3,4.5,7,12"))
    if kind == "extract":
        w, h = _size(rng, 0.25, 151.0)
        return dict(kind=kind, recipe=recipe, w=w, h=h, radii=radii, masked=rng.random() < 0.25, **det)
    if kind == "batch":
        frames = rng.randint(2, 8)
        w, h = _size(rng, 0.25, 34.0 / frames)
        return dict(kind=kind, recipe=recipe, w=w, h=h, frames=frames, radii=radii, **det)
    if kind == "serve":
        frames = rng.randint(2, 8)
        w, h = _size(rng, 0.25, 4.2)
        return dict(kind=kind, recipe=recipe, w=w, h=h, frames=frames, big=rng.randint(0, 2), radii=radii, **det)
    if kind == "learned":
        w, h = _size(rng, 1.0, 17.0)
        if u16:
            det["mesh"] = rng.choice((64, 256))
        else:
            det["mesh"] = 64
        return dict(kind=kind, recipe=recipe, w=w, h=h, radii=radii, **det)
    if kind == "train":
        return dict(kind=kind, n=rng.randint(2, 32), h=rng.randint(16, 64), w=rng.randint(16, 64))
    if kind == "photometry":
        w, h = _size(rng, 0.25, 17.0)
        return dict(kind=kind, recipe=recipe, w=w, h=h, mesh=det["mesh"], taps=det["taps"], radii=radii,
                    rows=int(math.exp(rng.uniform(math.log(100), math.log(15000)))))
    if kind == "cosmetic":
        w, h = _size(rng, 0.25, 17.0)
        cr = rng.random() < 0.7
        return dict(kind=kind, recipe=recipe, w=w, h=h, rtn=not cr or rng.random() < 0.5, cr=cr)
    if kind == "psf":
        w, h = _size(rng, 0.25, 17.0)
        return dict(kind=kind, recipe=recipe, w=w, h=h, mesh=det["mesh"], size=rng.choice((5, 7, 9, 13)),
                    modes=rng.randint(0, 5), tile=rng.choice((512, 1024, 2048)), thresh=det["thresh"])
    w, h = _size(rng, 0.25, 17.0)
    return dict(kind=kind, recipe=recipe, w=w, h=h, **det)


# ---------------------------------------------------------------- frames ---
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _stars(g, rec, w, h, n):
    """Positions, fluxes and FWHM of n stars; one in twenty sits beside the star before it."""
    u = torch.rand((5, n), generator=g, device=DEV, dtype=torch.float64)
    x, y = u[0] * w - 0.5, u[1] * h - 0.5
    lo, hi = (f ** -0.5 for f in rec["flux"])
    fwhm = rec["fwhm"][0] + u[3] * (rec["fwhm"][1] - rec["fwhm"][0])
    k = torch.arange(n // 20, device=DEV) * 20 + 1
    sep = (1.0 + torch.frac(u[4][k] * 7.0)) * fwhm[k]
    x[k] = x[k - 1] + sep * torch.cos(2 * math.pi * u[4][k])
    y[k] = y[k - 1] + sep * torch.sin(2 * math.pi * u[4][k])
    return x, y, (lo + u[2] * (hi - lo)) ** -2.0, fwhm


def _star_light(x, y, flux, fwhm, w, h, beta=2.5, reach=10):
    """Moffat profiles sampled at pixel centres, summed in fixed point so that the order does not matter."""
    out = torch.zeros(h * w, dtype=torch.int32, device=DEV)
    off = torch.arange(-reach, reach + 1, device=DEV)
    for c in range(0, len(x), 16384):
        xc, yc = x[c:c + 16384, None, None], y[c:c + 16384, None, None]
        a2 = (fwhm[c:c + 16384, None, None] / (2 * math.sqrt(2 ** (1 / beta) - 1))) ** 2
        px, py = xc.round().long() + off[None, None, :], yc.round().long() + off[None, :, None]
        r2 = ((px - xc) ** 2 + (py - yc) ** 2) / a2
        v = flux[c:c + 16384, None, None] * (beta - 1) / (math.pi * a2) * (1 + r2) ** -beta
        ok = (px >= 0) & (px < w) & (py >= 0) & (py < h)
        out.index_add_(0, (py * w + px)[ok], (v[ok] * 1024).round().to(torch.int32))
    return out.view(h, w).float() / 1024


def _sky(g, recipe, w, h):
    rec = RECIPES[recipe]
    xx = torch.linspace(0, 1, w, device=DEV)[None, :]
    yy = torch.linspace(0, 1, h, device=DEV)[:, None]
    if recipe == "sky_f32":
        return rec["sky"] + 50.0 * xx + 0.0 * yy
    if recipe == "ccd_u16":
        return rec["sky"] * (1 - 0.02 * ((2 * xx - 1) ** 2 + (2 * yy - 1) ** 2) / 2)
    gh, gw = h // 15 + 2, w // 15 + 2         # 100 ADU of nebulosity, correlated over 300 px
    noise = torch.randn((gh, gw), generator=g, device=DEV)
    ky, kx = torch.fft.fftfreq(gh, device=DEV)[:, None], torch.fft.fftfreq(gw, device=DEV)[None, :]
    field = torch.fft.ifft2(torch.fft.fft2(noise) * torch.exp(-2 * math.pi ** 2 * (kx ** 2 + ky ** 2) * 400.0)).real
    field = field * (100.0 / (field.std() + 1e-6))
    up = torch.nn.functional.interpolate(field[None, None], size=(h, w), mode="bilinear", align_corners=False)
    return rec["sky"] + up[0, 0].clamp(-400.0, 400.0)


def _as_u16(v):
    v = v.round_().clamp_(0, 65535).to(torch.int32)
    return torch.where(v > 32767, v - 65536, v).to(torch.int16).view(torch.uint16)


def _frame(recipe, w, h, seed, stars=None):
    """The frame as the camera or the calibration step leaves it, its sky and its stars."""
    rec, g = RECIPES[recipe], _gen(seed)
    sky = _sky(g, recipe, w, h)
    n = stars if stars is not None else max(4, round(rec["stars"] * w * h / 1e6))
    x, y, flux, fwhm = _stars(g, rec, w, h, n)
    img = torch.poisson((sky + _star_light(x, y, flux, fwhm, w, h)) * rec["gain"], generator=g)
    img += rec["rn"] * torch.randn((h, w), generator=g, device=DEV)
    img /= rec["gain"]
    if recipe == "ccd_u16":
        hot = torch.rand((h, w), generator=g, device=DEV)
        img = torch.where(hot < 5e-4, 5e3 + hot * ((SAT - 5e3) / 5e-4), img)
        t = torch.arange(0.0, 60.0, 0.5, device=DEV)
        for _ in range(max(1, round(20 * w * h / 4.2e6))):
            u = torch.rand(5, generator=g, device=DEV)
            tt = t[None, :] * (0.1 + 0.9 * u[2])
            tx = (u[0] * w + tt * torch.cos(math.pi * u[3])).round().long().clamp(0, w - 1)
            ty = (u[1] * h + tt * torch.sin(math.pi * u[3])).round().long().clamp(0, h - 1)
            img[ty, tx] = 500 + 19500 * u[4]
    return (_as_u16(img) if rec["u16"] else img), sky, (x, y)


def _bad_pixels(w, h, seed):
    """A detector's defect map: one pixel in a thousand, and some columns."""
    g = _gen(seed + 7919)
    bad = (torch.rand((h, w), generator=g, device=DEV) < 1e-3).to(torch.uint8)
    bad[:, torch.randint(0, w, (max(1, w // 1000),), generator=g, device=DEV)] = 1
    return bad


def _taps(size, fwhm=3.0):
    u = np.arange(size) - size // 2
    return np.exp(-(u[None, :] ** 2 + u[:, None] ** 2) * (4 * math.log(2) / fwhm ** 2)).astype(np.float32)


def _radii(case):
    return [float(r) for r in case["radii"].split(",")]


def _capacity(w, h):
    return max(8192, w * h // 378)      # 400,000 rows for the 151 MP frame


def _meshes(sky, rec, mesh):
    """Background and noise meshes of the known sky."""
    m = torch.nn.functional.avg_pool2d(sky[None, None].float(), mesh, ceil_mode=True)[0, 0].contiguous()
    return m, torch.sqrt(m / rec["gain"] + (rec["rn"] / rec["gain"]) ** 2).contiguous()


def _psf_model(case, seed):
    size, h = case["size"], case["size"] // 2
    yy, xx = np.mgrid[-h:h + 1, -h:h + 1].astype(np.float64)
    s2 = (3.0 / 2.3548) ** 2
    p0 = np.exp(-(xx * xx + yy * yy) / (2 * s2))
    p0 /= p0.sum()
    shapes = [xx * p0, yy * p0, (xx * xx + yy * yy - 2 * s2) * p0, (xx * xx - yy * yy) * p0, xx * yy * p0]
    k = case["modes"]
    modes = np.array(shapes[:k], np.float32).reshape(k, size, size)
    grid = (k, -(-case["h"] // case["tile"]), -(-case["w"] // case["tile"]))
    coef = torch.rand(grid, generator=_gen(seed + 104729), device=DEV) * 0.6 - 0.3 if k else None
    return p0.astype(np.float32), modes, coef


def _train_inputs(case, seed):
    g = _gen(seed)
    n, h, w = case["n"], case["h"], case["w"]
    centre = torch.randn((n, h, w, 1), generator=g, device=DEV)
    spread = 1 + 0.2 * torch.rand((n, h, w, 1), generator=g, device=DEV)
    q = centre + spread * torch.tensor([-1.28, -0.67, 0.0, 0.67, 1.28], device=DEV)
    feat = torch.zeros((n, h, w, 16), dtype=torch.bfloat16, device=DEV)
    feat[..., :5] = q.to(torch.bfloat16)
    ch = (5, 32, 48, 48, 32, 32, 2)
    weights = [torch.randn((b, a, 3, 3), generator=g, device=DEV) * math.sqrt(2 / (9 * a)) for a, b in zip(ch, ch[1:])]
    return feat, torch.cat([centre - 0.05 * spread, 0.95 * spread], dim=3).contiguous(), weights


# --------------------------------------------------------------- prepare ---
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "train":
        s["feat"], s["target"], weights = _train_inputs(case, seed)
        s["net"] = learned.Network(DEV)
        s["net"].load_state_dict({"W": weights})
        return s
    rec, w, h = RECIPES[case["recipe"]], case["w"], case["h"]
    sat = SAT if rec["u16"] else 0.0
    if kind == "serve":
        sizes = [(w, h)] * case["frames"] + [(2 * w, 2 * h)] * case["big"]
        s["frames"] = [_frame(case["recipe"], a, b, seed + 1000 * k)[0].cpu().pin_memory()
                       for k, (a, b) in enumerate(sizes)]
        s["caps"] = [_capacity(a, b) for a, b in sizes]
        s["tables"] = [{k: np.zeros((c, len(_radii(case))) if k.startswith("flux") else c, dt)
                        for k, dt in (("label", np.uint32), ("x", float), ("y", float), ("flux", float),
                                      ("fluxerr", float))} for c in s["caps"]]
        s["sat"] = sat
        s["server"] = gp.Server(0, hbm_budget=3 << 30, host_budget=128 << 20, slots=4, batch_pixels=8 << 20,
                                max_batch=8, mesh=case["mesh"], kernel=_taps(case["taps"]), thresh=case["thresh"],
                                minarea=MINAREA, radii=_radii(case), gain=rec["gain"])
        return s
    s["ctx"] = ctx = gp.Context(0)
    if kind == "batch":
        s["images"] = [_frame(case["recipe"], w, h, seed + 1000 * k)[0] for k in range(case["frames"])]
        s["ex"] = gp.BatchExtractor(ctx, [(h, w)] * case["frames"], s["images"][0].dtype, case["mesh"],
                                    _taps(case["taps"]), case["thresh"], MINAREA, _radii(case), rec["gain"],
                                    _capacity(w, h), saturation=sat)
        return s
    if kind == "photometry":
        n = max(case["rows"], 100)
        s["img"], sky, (x, y) = _frame(case["recipe"], w, h, seed, stars=n)
        bm, rm = _meshes(sky, rec, case["mesh"])
        s["bkg"] = {"bkg_mesh": bm, "rms_mesh": rm, "mesh": case["mesh"]}
        s["cat"], _ = gp.allocate_catalog(n, DEV)
        s["cat"]["n"].fill_(n)
        s["cat"]["x"].copy_(x)
        s["cat"]["y"].copy_(y)
        s["cat"]["xpeak"].copy_(x.round().clamp(0, w - 1))
        s["cat"]["ypeak"].copy_(y.round().clamp(0, h - 1))
        s["sat"], s["gain"] = sat, rec["gain"]
        return s
    s["img"], sky, _ = _frame(case["recipe"], w, h, seed)
    s["sat"], s["gain"] = sat, rec["gain"]
    if kind == "cosmetic":
        s["args"] = dict(rtn_t=150.5 if case["rtn"] else 0.0, cr_gain=rec["gain"] if case["cr"] else 0.0,
                         cr_read_noise=rec["rn"] if case["cr"] else 0.0)
        return s
    if kind == "psf":
        bm, rm = _meshes(sky, rec, case["mesh"])
        s["bkg"] = {"bkg_mesh": bm, "rms_mesh": rm, "mesh": case["mesh"]}
        s["p0"], s["modes"], s["coef"] = _psf_model(case, seed)
        return s
    net = learned.load(learned.weights_for_mesh(case["mesh"]), DEV) if kind == "learned" else None
    s["mask"] = _bad_pixels(w, h, seed) if case.get("masked") else None
    s["ex"] = gp.Extractor(ctx, (h, w), s["img"].dtype, case["mesh"], _taps(case["taps"]), case["thresh"], MINAREA,
                           _radii(case) if "radii" in case else [3.0], rec["gain"], _capacity(w, h), saturation=sat,
                           net=net)
    if kind == "deblend":
        o = s["ex"].run(s["img"])
        n = int(o["catalog"]["n"].item())
        s["cat"] = {k: v if k == "n" else v[:max(n, 1)].clone() for k, v in o["catalog"].items()}
        s["bkg"] = {k: o[k] for k in ("bkg_mesh", "rms_mesh", "mesh")}
        s["segmap"] = o["segmap"]
    return s


# ------------------------------------------------------------------- run ---
def _extraction(o):
    return {k: o[k] for k in ("bkg_mesh", "rms_mesh", "segmap", "catalog", "flux", "fluxerr", "apflags")}


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind in ("extract", "learned"):
        return _extraction(s["ex"].run(s["img"], mask=s["mask"]))
    if kind == "batch":
        return [dict({k: o["catalog"][k] for k in ("n", "label", "x", "y")}, segmap=o["segmap"], flux=o["flux"],
                     fluxerr=o["fluxerr"], bkg_mesh=o["bkg_mesh"]) for o in s["ex"].run(s["images"])]
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit(f, c, saturation=s["sat"]) for f, c in zip(s["frames"], s["caps"])]
        out = []
        for t, table in zip(tickets, s["tables"]):      # the rows go into the caller's tables, frame by frame
            r = srv.result(t)
            for k, v in table.items():
                rows = r["catalog"][k]
                v[:len(rows)] = rows
                v[len(rows):] = 0
            out.append(dict(table, bkg_mesh=r["bkg_mesh"]))
        return out
    if kind == "train":
        net = s["net"]
        acts, logits = net.forward(s["feat"])
        loss, grads = net.backward(acts, logits, s["target"])
        net.adamw(grads, lr=1e-3)
        return {"logits": logits, "loss": loss, "grads": grads, "W": net.W, "b": net.b}
    ctx, img = s["ctx"], s["img"]
    if kind == "photometry":
        cat = s["cat"]
        flux, err, flags = ctx.gp_aperture(img, s["bkg"], cat["x"], cat["y"], _radii(case), gain=s["gain"],
                                           saturation=s["sat"])
        ro = ctx.gp_optimal_radius(img, s["bkg"], _taps(case["taps"]), cat, range(3, 16), gain=s["gain"],
                                   snr_min=20.0, d_iso=30.0, saturation=s["sat"])
        return {"flux": flux, "fluxerr": err, "flags": flags, "radius": ro}
    if kind == "cosmetic":
        return ctx.gp_cosmetic(img, **s["args"])
    if kind == "psf":
        return ctx.gp_detect_psf(img, s["bkg"], s["p0"], s["modes"], s["coef"], case["tile"], case["thresh"],
                                 MINAREA, _capacity(case["w"], case["h"]), saturation=s["sat"])
    seg = s["segmap"].clone()      # the undivided map is kept
    r = ctx.gp_deblend(img, s["bkg"], _taps(case["taps"]), case["thresh"], MINAREA, seg, s["cat"],
                       saturation=s["sat"])
    return {"segmap": seg, "objects": r["objects"], "counts": r["counts"]}


# ------------------------------------------------------------------ work ---
def work(case):
    kind = case["kind"]
    if kind == "train":
        pos, ch = case["n"] * case["h"] * case["w"], (5, 32, 48, 48, 32, 32, 2)
        macs = [9 * a * b for a, b in zip(ch, ch[1:])]
        # activations written and read once each way, in bf16
        return {"bytes": pos * 2.0 * (4 * sum(ch[1:6]) + ch[0]), "flops": 2.0 * pos * (3 * sum(macs) - macs[0])}
    px, b = case["w"] * case["h"], 2 if RECIPES[case["recipe"]]["u16"] else 4
    if kind in ("extract", "learned"):
        # the frame in, the segmentation map out, about ten operations a pixel (the separable filter)
        return {"bytes": px * (b + 4.0 + (1.0 if case.get("masked") else 0.0)), "flops": 4.0 * case["taps"] * px}
    if kind == "batch":
        return {"bytes": px * (b + 4.0) * case["frames"], "flops": 4.0 * case["taps"] * px * case["frames"]}
    if kind == "serve":
        px *= case["frames"] + 4 * case["big"]
        return {"bytes": px * float(b), "flops": 4.0 * case["taps"] * px}
    if kind == "photometry":
        n, r = max(case["rows"], 100), max(15.0, max(_radii(case)))
        nr = len(_radii(case)) + 13
        return {"bytes": n * (math.pi * r * r * b + 20.0 * nr), "flops": n * 4.0 * math.pi * r * r}
    if kind == "cosmetic":
        # selecting networks of 9, 25, 25 and 49 values take some 600 minima and maxima a pixel
        return {"bytes": px * (b + 5.0), "flops": px * ((20.0 if case["rtn"] else 0.0) + (300.0 if case["cr"] else 0.0))}
    if kind == "psf":
        return {"bytes": px * (b + 4.0), "flops": 2.0 * px * (case["modes"] + 1) * case["size"] ** 2}
    return {"bytes": px * (b + 8.0), "flops": 4.0 * case["taps"] * px}


# ----------------------------------------------------------------- exact ---
# The method in 64 bits: definitions as the C header states them.
F64 = torch.float64


def _box_stats(img, bad, mesh, k=3.0, maxiter=10):
    """Sigma-clipped background and noise of each box from its sorted good values."""
    h, w = img.shape
    my, mx = -(-h // mesh), -(-w // mesh)
    bkg = torch.zeros((my, mx), dtype=F64, device=DEV)
    rms = torch.zeros((my, mx), dtype=F64, device=DEV)
    for j in range(my):
        row = torch.full((mesh, mx * mesh), math.inf, dtype=F64, device=DEV)
        part = img[j * mesh:(j + 1) * mesh]
        row[:part.shape[0], :w] = part if bad is None else part.masked_fill(bad[j * mesh:(j + 1) * mesh], math.inf)
        v = row.view(mesh, mx, mesh).permute(1, 0, 2).reshape(mx, -1).sort(dim=1).values
        cnt = torch.isfinite(v).sum(dim=1)
        ref = v[:, :1]
        d = torch.where(torch.isfinite(v), v - ref, torch.zeros_like(v))
        z = torch.zeros((mx, 1), dtype=F64, device=DEV)
        c1, c2 = torch.cat([z, d.cumsum(1)], 1), torch.cat([z, (d * d).cumsum(1)], 1)
        at = lambda t, i: t.gather(1, i[:, None])[:, 0]                                    # noqa: E731
        lo, hi = torch.zeros_like(cnt), cnt.clone()
        for it in range(maxiter + 1):
            n = (hi - lo).clamp(min=1)
            med = 0.5 * (at(v, lo + (n - 1) // 2) + at(v, lo + n // 2))
            mean = (at(c1, hi) - at(c1, lo)) / n
            std = ((at(c2, hi) - at(c2, lo)) / n - mean * mean).clamp(min=0).sqrt()
            if it == maxiter:
                break
            lo2 = torch.searchsorted(v, (med - k * std)[:, None])[:, 0].maximum(lo)
            hi2 = torch.searchsorted(v, (med + k * std)[:, None], right=True)[:, 0].minimum(hi)
            if torch.equal(lo2, lo) and torch.equal(hi2, hi):
                break
            lo, hi = lo2, hi2
        mean = mean + ref[:, 0]
        skew = (mean - med).abs() > 0.3 * std
        bkg[j] = torch.where((std == 0) | skew, med, 2.5 * med - 1.5 * mean)
        rms[j] = std
    return bkg, rms


def _mesh_median(m):
    p = torch.nn.functional.pad(m[None, None], (1, 1, 1, 1), value=math.nan)[0, 0]
    win = p.unfold(0, 3, 1).unfold(1, 3, 1).reshape(*m.shape, 9)
    n = (~win.isnan()).sum(-1, keepdim=True)
    v = win.nan_to_num(nan=math.inf).sort(dim=-1).values
    return 0.5 * (v.gather(-1, (n - 1) // 2) + v.gather(-1, n // 2))[..., 0]


def _spline_matrix(size, mesh):
    """Pixels from nodes: the natural cubic spline through the box centres, continued by its end slopes."""
    n = -(-size // mesh)
    start = np.arange(n) * float(mesh)
    t = start + (np.minimum(start + mesh, size) - start - 1) / 2
    if n == 1:
        return torch.ones((size, 1), dtype=F64, device=DEV)
    step = np.diff(t)
    a, r = np.eye(n), np.zeros((n, n))
    for i in range(1, n - 1):
        a[i, i - 1:i + 2] = step[i - 1] / 6, (step[i - 1] + step[i]) / 3, step[i] / 6
        r[i, i - 1:i + 2] = 1 / step[i - 1], -1 / step[i - 1] - 1 / step[i], 1 / step[i]
    m = np.linalg.solve(a, r)
    x = np.arange(size, dtype=np.float64)
    i = np.clip(np.searchsorted(t, x, side="right") - 1, 0, n - 2)
    s, b = step[i], (x - t[i]) / step[i]
    bi = np.clip(b, 0, 1)
    eye = np.eye(n)
    out = (1 - b)[:, None] * eye[i] + b[:, None] * eye[i + 1]
    # the cubic part inside the nodes; outside, its end slope times the distance
    c0 = np.where(b < 0, -b * s * s / 3, np.where(b > 1, (b - 1) * s * s / 6, s * s / 6 * ((1 - bi) ** 3 - (1 - bi))))
    c1 = np.where(b < 0, -b * s * s / 6, np.where(b > 1, (b - 1) * s * s / 3, s * s / 6 * (bi ** 3 - bi)))
    out += c0[:, None] * m[i] + c1[:, None] * m[i + 1]
    return torch.from_numpy(out).to(DEV)


def _map(nodes, h, w, mesh):
    return _spline_matrix(h, mesh) @ nodes.to(F64) @ _spline_matrix(w, mesh).T


def _correlate(m, kernel):
    kh, kw = kernel.shape
    k = torch.from_numpy(np.asarray(kernel, np.float64)).to(DEV)
    p = torch.nn.functional.pad(m[None, None], (kw // 2, kw // 2, kh // 2, kh // 2), mode="reflect")[0, 0]
    out = torch.zeros_like(m)
    for v in range(kh):
        for u in range(kw):
            out += k[v, u] * p[v:v + m.shape[0], u:u + m.shape[1]]
    return out


def _labels(fg):
    """1 + the smallest linear index of each 8-connected component, 0 elsewhere."""
    h, w = fg.shape
    n = h * w
    val = torch.where(fg, n - torch.arange(n, device=DEV, dtype=F64).view(h, w), torch.zeros((), dtype=F64, device=DEV))
    while True:
        new = torch.nn.functional.max_pool2d(val[None, None], 3, 1, 1)[0, 0] * fg
        root = (n - new).clamp(max=n - 1).long()
        new = torch.where(fg, new.view(-1)[root].maximum(new), new)
        if torch.equal(new, val):
            break
        val = new
    return torch.where(fg, n - val + 1, torch.zeros_like(val)).long()


def _catalog(m, fg, cap):
    """Per kept segment in label order, in arrays of `cap` rows: flux, centroid, second moments, peak; their count."""
    h, w = m.shape
    lab = _labels(fg)
    py, px = torch.nonzero(lab, as_tuple=True)
    ids, inv, cnt = torch.unique(lab[py, px], return_inverse=True, return_counts=True)
    keep = cnt >= MINAREA
    sel = keep[inv]
    inv, py, px = (keep.cumsum(0) - 1)[inv][sel], py[sel].double(), px[sel].double()
    v, n = m[py.long(), px.long()], int(keep.sum())
    add = lambda t: torch.zeros(n, dtype=F64, device=DEV).index_add_(0, inv, t)           # noqa: E731
    s = add(v)
    wt = torch.where((s > 0)[inv], v, torch.ones_like(v))
    sw = add(wt)
    x, y = add(px * wt) / sw, add(py * wt) / sw
    dx, dy = px - x[inv], py - y[inv]
    peak = torch.full((n,), -math.inf, dtype=F64, device=DEV).scatter_reduce_(0, inv, v, "amax")
    full = lambda t: torch.nn.functional.pad(t[:cap], (0, max(0, cap - n)))                # noqa: E731
    return n, {k: full(t) for k, t in dict(flux_iso=s, x=x, y=y, x2=add(dx * dx * wt) / sw, y2=add(dy * dy * wt) / sw,
                                           xy=add(dx * dy * wt) / sw, peak=peak).items()}


def _disc_below(a, b, r):
    """Area of the disc of radius r about the origin with X <= a and Y <= b."""
    a, b = a.clamp(-r, r), b.clamp(-r, r)
    c = (r * r - b * b).clamp(min=0).sqrt()
    g = lambda t: 0.5 * (t * (r * r - t * t).clamp(min=0).sqrt() + r * r * (t / r).clamp(-1, 1).asin())  # noqa: E731
    a1, a2, a3 = torch.minimum(a, -c), torch.minimum(torch.maximum(a, -c), c), torch.maximum(a, c)
    ends = 2 * (g(a1) - g(torch.full_like(a, -r)) + g(a3) - g(c))
    return torch.where(b >= 0, ends, torch.zeros_like(ends)) + b * (a2 + c) + g(a2) - g(-c)


def _windows(m, var, x, y, reach, weigh, gain):
    """Sums of weigh(dx, dy) m and of weigh var over each source's window, as flux and its error."""
    h, w = m.shape
    off = torch.arange(-reach, reach + 1, device=DEV)
    flux, err = [], []
    for c in range(0, len(x), 4096):
        xc, yc = x[c:c + 4096, None, None], y[c:c + 4096, None, None]
        px, py = torch.floor(xc + 0.5).long() + off[None, None, :], torch.floor(yc + 0.5).long() + off[None, :, None]
        ok = (px >= 0) & (px < w) & (py >= 0) & (py < h)
        at = py.clamp(0, h - 1) * w + px.clamp(0, w - 1)
        a = torch.where(ok, weigh(px - xc, py - yc), torch.zeros((), dtype=F64, device=DEV))
        f = (a * m.reshape(-1)[at]).sum((1, 2))
        flux.append(f)
        err.append(((a * var.reshape(-1)[at]).sum((1, 2)) + (f.clamp(min=0) / gain if gain > 0 else 0.0)).sqrt())
    return torch.cat(flux), torch.cat(err)


def _apertures(m, var, x, y, radii, gain):
    flux, err = [], []
    for r in radii:
        r = float(np.float32(r))

        def weigh(dx, dy):
            below = lambda u, v: _disc_below(dx + u, dy + v, r)                            # noqa: E731
            return below(0.5, 0.5) - below(-0.5, 0.5) - below(0.5, -0.5) + below(-0.5, -0.5)
        f, e = _windows(m, var, x, y, math.ceil(r) + 2, weigh, gain)
        flux.append(f)
        err.append(e)
    return torch.stack(flux, 1), torch.stack(err, 1)


def _pixels(img):
    return (img.to(torch.int32) if img.dtype == torch.uint16 else img).to(F64)


def _exact_extract(case, seed):
    rec, w, h = RECIPES[case["recipe"]], case["w"], case["h"]
    img = _pixels(_frame(case["recipe"], w, h, seed)[0])
    bad = _bad_pixels(w, h, seed) != 0 if case.get("masked") else None
    bkg, rms = (_mesh_median(t) for t in _box_stats(img, bad, case["mesh"]))
    none = dict.fromkeys(("segmap", "apflags"))
    if w * h > 20e6:
        return dict(none, bkg_mesh=bkg, rms_mesh=rms)
    m, sig = img - _map(bkg, h, w, case["mesh"]), _map(rms, h, w, case["mesh"])
    var = sig * sig
    if bad is not None:
        m, var = m.masked_fill(bad, 0.0), var.masked_fill(bad, 0.0)
    k = _taps(case["taps"]).astype(np.float64)
    fg = _correlate(m, k / k.sum()) > case["thresh"] * sig
    fg = fg if bad is None else fg & ~bad
    cap = _capacity(w, h)
    n, cat = _catalog(m, fg, cap)
    f, e = _apertures(m, var, cat["x"][:n], cat["y"][:n], _radii(case), rec["gain"])
    full = lambda t: torch.nn.functional.pad(t[:cap], (0, 0, 0, max(0, cap - n)))          # noqa: E731
    return dict(none, bkg_mesh=bkg, rms_mesh=rms, catalog=cat, flux=full(f), fluxerr=full(e))


def _exact_photometry(case, seed):
    rec, w, h, n = RECIPES[case["recipe"]], case["w"], case["h"], max(case["rows"], 100)
    img, sky, (x, y) = _frame(case["recipe"], w, h, seed, stars=n)
    bm, rm = _meshes(sky, rec, case["mesh"])
    m, sig = _pixels(img) - _map(bm, h, w, case["mesh"]), _map(rm, h, w, case["mesh"])
    flux, err = _apertures(m, sig * sig, x, y, _radii(case), rec["gain"])
    gx, gy = torch.floor(x + 0.5), torch.floor(y + 0.5)
    rings = [_windows(m, sig * sig, gx, gy, r, lambda dx, dy, r=r: (dx * dx + dy * dy <= r * r).to(F64), rec["gain"])
             for r in range(3, 16)]
    k = _taps(case["taps"]).astype(np.float64)
    nu = _correlate(m, k / k.sum()) / sig
    at = y.round().clamp(0, h - 1).long(), x.round().clamp(0, w - 1).long()
    return {"flux": flux, "fluxerr": err,
            "radius": {"flux": torch.stack([f for f, _ in rings], 1), "fluxerr": torch.stack([e for _, e in rings], 1),
                       "nu": nu[at]}}


def _window(v, size):
    """The size x size values around each pixel of rows with a mirror border."""
    p = size // 2
    p = torch.nn.functional.pad(v[None, None], (p, p, p, p), mode="reflect")[0, 0]
    return p.unfold(0, size, 1).unfold(1, size, 1).reshape(*v.shape, size * size)


def _median(v, size, rows=256):
    out = torch.empty_like(v)
    p = size // 2
    q = torch.nn.functional.pad(v[None, None], (p, p, p, p), mode="reflect")[0, 0]
    for r in range(0, v.shape[0], rows):
        part = q[r:r + rows + 2 * p]
        win = part.unfold(0, size, 1).unfold(1, size, 1).reshape(part.shape[0] - 2 * p, v.shape[1], size * size)
        out[r:r + rows] = win.sort(dim=-1).values[..., size * size // 2]
    return out


def _exact_cosmetic(case, seed):
    rec, w, h = RECIPES[case["recipe"]], case["w"], case["h"]
    img = _pixels(_frame(case["recipe"], w, h, seed)[0])
    if case["cr"]:
        gain, rn = rec["gain"], rec["rn"]
        lap = _correlate(img, np.array([[0, -1, 0], [-1, 4, -1], [0, -1, 0]])).clamp(min=0)
        noise = (_median(img, 5).clamp(min=0) * gain + rn * rn).sqrt() / gain
        s = lap / (math.sqrt(20) * noise)
        s = s - _median(s, 5)
        med3 = _median(img, 3)
        fine = (med3 - _median(med3, 7)).clamp(min=0.01)
        hit = (s > 4.5) & (lap / fine > 5.0)
        clean = _window(img.masked_fill(hit, math.inf).float(), 5)[hit].double().sort(dim=-1).values
        n = torch.isfinite(clean).sum(-1, keepdim=True)
        fill = 0.5 * (clean.gather(-1, ((n - 1) // 2).clamp(min=0)) + clean.gather(-1, (n // 2).clamp(max=24)))[:, 0]
        img = img.clone()
        img[hit] = torch.where(n[:, 0] > 0, fill, img[hit])
    if case["rtn"]:
        med = _median(img, 3)
        out = (img - med).abs() > 150.5
        near = torch.nn.functional.conv2d(torch.nn.functional.pad(out[None, None].double(), (1, 1, 1, 1)),
                                          torch.ones((1, 1, 3, 3), dtype=F64, device=DEV))[0, 0]
        img = torch.where(out & (near < 1.5), med, img)
    return {"image": img}


def _exact_psf(case, seed):
    rec, w, h = RECIPES[case["recipe"]], case["w"], case["h"]
    img, sky, _ = _frame(case["recipe"], w, h, seed)
    bm, rm = _meshes(sky, rec, case["mesh"])
    m = _pixels(img) - _map(bm, h, w, case["mesh"])
    p0, modes, coef = _psf_model(case, seed)
    s = _correlate(m, p0)
    for k in range(case["modes"]):
        s += _map(coef[k], h, w, case["tile"]) * _correlate(m, modes[k])
    return {"catalog": _catalog(m, s > case["thresh"] * _map(rm, h, w, case["mesh"]), _capacity(w, h))[1]}


def _exact_train(case, seed):
    feat, target, weights = _train_inputs(case, seed)
    ws = [t.to(F64).requires_grad_() for t in weights]
    bs = [torch.zeros(len(t), dtype=F64, device=DEV, requires_grad=True) for t in weights]
    x = feat[..., :5].to(F64).permute(0, 3, 1, 2)
    for k, (wt, b) in enumerate(zip(ws, bs)):
        cols = torch.nn.functional.unfold(x, 3, padding=1)
        x = (wt.reshape(wt.shape[0], -1) @ cols + b[:, None]).view(x.shape[0], -1, case["h"], case["w"])
        x = x if k == 5 else x.relu()
    out = x.permute(0, 2, 3, 1)
    loss = (out - target.to(F64)).square().mean()
    grads = torch.autograd.grad(loss, ws + bs)
    return {"logits": out.detach(), "loss": loss.detach()[None], "grads": [(grads[k], grads[6 + k]) for k in range(6)],
            "W": None, "b": None}


def exact(case, seed):
    """What run() returns, from the definitions in 64 bits; None for the outputs that are decisions (labels, flags,
    radii), for the network's meshes and for deblending, whose objects are decisions throughout.  A whole frame above
    20 megapixels gives its meshes only, and the batch and the server, whose frames are those of the other cases,
    give their meshes."""
    kind = case["kind"]
    if kind == "extract":
        return _exact_extract(case, seed)
    if kind in ("batch", "serve"):
        sizes = [(case["w"], case["h"])] * case["frames"] + [(2 * case["w"], 2 * case["h"])] * case.get("big", 0)
        return [{"bkg_mesh": _mesh_median(_box_stats(_pixels(_frame(case["recipe"], a, b, seed + 1000 * k)[0]), None,
                                                     case["mesh"])[0])} for k, (a, b) in enumerate(sizes)]
    if kind == "photometry":
        return _exact_photometry(case, seed)
    if kind == "cosmetic":
        return _exact_cosmetic(case, seed)
    if kind == "psf":
        return _exact_psf(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return None
