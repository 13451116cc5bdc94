"""Apertures for every number of radii (seven run in the kernel of eight):
listed positions against the oracle, and an extraction's rows, single and
batched, against the listed call at their centroids."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

RADII = (2.0, 3.3, 4.0, 5.5, 6.0, 7.25, 9.0, 12.0)
U8 = 8 * 2.0 ** -24


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("nr", range(1, 9))
def test_listed_positions(nr, f32):
    rng = np.random.default_rng(nr)
    H, W, mesh = 220, 260, 32
    img = np.round(rng.normal(1000.0, 20.0, (H, W)))
    img[rng.random((H, W)) < 0.002] = 60000.0
    img = img.astype(np.float32 if f32 else np.uint16)
    mask = (rng.random((H, W)) < 0.001).astype(np.uint8)
    my, mx = -(-H // mesh), -(-W // mesh)
    bm = rng.normal(1000.0, 5.0, (my, mx)).astype(np.float32)
    rm = rng.uniform(15.0, 25.0, (my, mx)).astype(np.float32)
    xs, ys = rng.uniform(-8, W + 8, 400), rng.uniform(-8, H + 8, 400)
    radii = RADII[8 - nr:]
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    bkg = {"bkg_mesh": torch.from_numpy(bm).cuda(), "rms_mesh": torch.from_numpy(rm).cuda(), "mesh": mesh}
    f, e, fl = ctx.gp_aperture(torch.from_numpy(img).cuda(), bkg, torch.from_numpy(xs), torch.from_numpy(ys), radii,
                               gain=1.5, mask=torch.from_numpy(mask).cuda(), saturation=50000.0)
    ctx.sync()
    vals, bad = oracle.pixel_values(img, mask)
    bmap, rmap = oracle.spline_map(bm.astype(np.float64), W, H, mesh), oracle.spline_map(rm.astype(np.float64), W, H, mesh)
    m, var, sat = np.where(bad, 0.0, vals - bmap), np.where(bad, 0.0, rmap ** 2), oracle.saturated(img, 50000.0)
    rf, re, rfl = oracle.apertures(m, var, bad, sat, xs, ys, radii, 1.5)
    scale, _, _ = oracle.apertures(np.abs(m) + U8 / 1e-5 * np.abs(bmap), var, bad, sat, xs, ys, radii, 0.0)
    assert np.all(np.abs(f.cpu().numpy() - rf) <= 1e-5 * scale + 1e-6)
    # the root of the sum of A sigma^2: areas are good to 1e-6 pixels, so 1e-5 of it needs a pixel in the frame
    area, _, _ = oracle.apertures(np.ones_like(m), var, np.zeros_like(bad), sat, xs, ys, radii, 0.0)
    whole = area >= 1.0
    assert whole.sum() > 300 * nr and np.all((np.abs(e.cpu().numpy() - re) <= 1e-5 * np.maximum(re, 1.0))[whole])
    assert np.array_equal(fl.cpu().numpy().view(np.uint32), rfl.astype(np.uint32))


@pytest.mark.parametrize("nr", (5, 6, 7, 8))
def test_extraction_and_batch(nr):
    cfg = synth.scaled_config(synth.CONFIGS["plain_2048x2048_u16"], 420, 390, name="aperture_radii_420x390_u16")
    t = torch.from_numpy(synth.make_frame(cfg, 11, cache=False)[0]).cuda()
    radii, args = RADII[:nr], (64, cfg.kernel, cfg.thresh, cfg.minarea)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    one = ctx.gp_extract(t, *args, radii, cfg.gain, capacity=4096, saturation=cfg.saturation)
    ctx.sync()
    n = int(one["catalog"]["n"].item())
    assert n > 50
    f, e, fl = ctx.gp_aperture(t, one, one["catalog"]["x"][:n], one["catalog"]["y"][:n], radii, gain=cfg.gain,
                               saturation=cfg.saturation)
    ctx.sync()
    for k, v in (("flux", f), ("fluxerr", e), ("apflags", fl)):
        assert torch.equal(one[k].reshape(-1)[:n * nr].view(n, nr), v), k
    bx = gp.BatchExtractor(ctx, [t.shape] * 2, t.dtype, *args, radii, cfg.gain, 4096, saturation=cfg.saturation)
    bx.run([t, t.clone()])
    ctx.sync()
    for o in bx.outs:
        for k in ("flux", "fluxerr", "apflags"):
            assert torch.equal(o[k][:n], one[k][:n]), k
