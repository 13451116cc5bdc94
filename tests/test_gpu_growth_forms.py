"""Growth curves by ring lists and by columns: radii sets on both sides of
each form's limits (few and many radii, radius 0, lists too long), sources
inside one interval of the mesh rows, across one, and over the frame's edge,
bad and saturated pixels; against the oracle.  The optimal-radius step's
isolation scan around its chunk length, and its fit."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

U8 = 8 * 2.0 ** -24


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("radii", ((0,), (5,), (0, 1, 2), tuple(range(1, 9)), tuple(range(1, 10)), tuple(range(3, 19)),
                                   tuple(range(2, 19)), tuple(range(1, 33)), (3, 20, 35), (2, 40), (1, 41, 60)))
def test_forms_match_the_oracle(radii, f32):
    rng = np.random.default_rng(len(radii) + radii[-1])
    H, W, mesh = 300, 410, 64
    img = np.round(rng.normal(1000.0, 20.0, (H, W)))
    img[rng.random((H, W)) < 0.002] = 60000.0
    img = img.astype(np.float32 if f32 else np.uint16)
    mask = (rng.random((H, W)) < 0.001).astype(np.uint8)
    my, mx = -(-H // mesh), -(-W // mesh)
    bm = rng.normal(1000.0, 5.0, (my, mx)).astype(np.float32)
    rm = rng.uniform(15.0, 25.0, (my, mx)).astype(np.float32)
    xs = np.concatenate([rng.uniform(-5, W + 5, 120), [200.5, 200.49999, W - 1.0, -1e9, np.nan]])
    ys = np.concatenate([rng.uniform(-5, H + 5, 120), [96.0, 128.5, 5.0, 10.0, 20.0]])
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    bkg = {"bkg_mesh": torch.from_numpy(bm).cuda(), "rms_mesh": torch.from_numpy(rm).cuda(), "mesh": mesh}
    f, e, fl = ctx.gp_growth(torch.from_numpy(img).cuda(), bkg, torch.from_numpy(xs).cuda(), torch.from_numpy(ys).cuda(),
                             radii, gain=1.5, mask=torch.from_numpy(mask).cuda(), saturation=50000.0)
    ctx.sync()
    vals, bad = oracle.pixel_values(img, mask)
    bmap, rmap = oracle.spline_map(bm.astype(np.float64), W, H, mesh), oracle.spline_map(rm.astype(np.float64), W, H, mesh)
    m, var, sat = np.where(bad, 0.0, vals - bmap), rmap ** 2, oracle.saturated(img, 50000.0)
    ok = np.abs(xs) < 1e6                            # the far and the undefined position: empty sums
    rf, re, rfl = oracle.growth(m, var, bad, sat, xs[ok], ys[ok], radii, 1.5)
    scale, _, _ = oracle.growth(np.abs(m) + U8 / 1e-5 * np.abs(bmap), var, bad, sat, xs[ok], ys[ok], radii, 0.0)
    got = f.cpu().numpy()
    assert np.all(np.abs(got[ok] - rf) <= 1e-5 * scale + 1e-6)
    assert np.all(np.abs(e.cpu().numpy()[ok] - re) <= 1e-5 * np.maximum(re, 1.0))
    assert np.array_equal(fl.cpu().numpy()[ok].view(np.uint32), rfl.astype(np.uint32))
    assert not got[~ok].any() and np.all(fl.cpu().numpy()[~ok] == gp.GP_FLAG_TRUNCATED)


@pytest.mark.parametrize("w,h,n,d_iso", ((200, 150, 1, 5.0), (500, 400, 63, 3.0), (500, 400, 65, 9.0), (910, 905, 900, 10.0),
                                         (900, 700, 4000, 1.0), (2000, 1500, 3000, 12.0)))
def test_optimal_radius_steps(w, h, n, d_iso):
    rng = np.random.default_rng(n)
    xs, ys = rng.uniform(0, w - 1, n), rng.uniform(0, h - 1, n)
    img = rng.normal(1000.0, 10.0, (h, w))
    for x, y, f in zip(xs, ys, rng.uniform(200, 60000, n)):
        x0, y0 = int(round(x)), int(round(y))
        sl = np.s_[max(0, y0 - 8):min(h, y0 + 9), max(0, x0 - 8):min(w, x0 + 9)]
        yy, xx = np.mgrid[sl]
        img[sl] += f / 12.0 * np.exp(-((yy - y) ** 2 + (xx - x) ** 2) / 4.0)
    img = img.astype(np.float32)
    mesh = 64
    my, mx = -(-h // mesh), -(-w // mesh)
    bm, rm = np.full((my, mx), 1000.0, np.float32), np.full((my, mx), 10.0, np.float32)
    kern = np.ones((3, 3), np.float32)
    ctx = gp.Context(0, workspace_bytes=128 << 20)
    cat, _ = gp.allocate_catalog(n, "cuda")
    cat["n"].fill_(n)
    xp, yp = np.clip(np.round(xs), 0, w - 1), np.clip(np.round(ys), 0, h - 1)
    for k, v in (("x", xs), ("y", ys), ("xpeak", xp), ("ypeak", yp)):
        cat[k].copy_(torch.from_numpy(v))
    radii = tuple(range(2, 12))
    ro = ctx.gp_optimal_radius(torch.from_numpy(img).cuda(), {"bkg_mesh": torch.from_numpy(bm).cuda(),
                               "rms_mesh": torch.from_numpy(rm).cuda(), "mesh": mesh}, kern, cat, radii, gain=1.0,
                               snr_min=20.0, d_iso=d_iso)
    ctx.sync()
    o = {k: v.cpu().numpy() for k, v in ro.items()}
    # each step from the outputs of the one before, in float64
    snr = np.where(o["fluxerr"] > 0, o["flux"] / np.where(o["fluxerr"] > 0, o["fluxerr"], 1.0), 0.0)
    assert np.array_equal(o["kopt"], snr.argmax(axis=1))
    iso = oracle.isolated(xs, ys, d_iso)
    best = snr[np.arange(n), o["kopt"]]
    cal = iso & (o["flags"].max(axis=1) == 0) & (o["nu"] > 0) & (best >= 20.0)
    assert np.array_equal(o["calib"] != 0, cal)
    a, b, cnt, status = o["fit"]
    assert int(cnt) == int(cal.sum())
    if cal.sum() >= 3 and len(np.unique(o["nu"][cal])) > 1:
        x, y = np.log10(o["nu"][cal].astype(np.float64)), np.log10(np.asarray(radii, float)[o["kopt"][cal]])
        sxx = ((x - x.mean()) ** 2).sum()
        ra = ((x - x.mean()) * (y - y.mean())).sum() / sxx
        # float64 sums of cal.sum() terms, conditioned by the spread of x
        tol = 1e-13 * cal.sum() * max(1.0, np.abs(x).max() ** 2 / (sxx / cal.sum()))
        assert status == 0 and abs(a - ra) <= tol and abs(b - (y.mean() - ra * x.mean())) <= tol * max(1.0, np.abs(x.mean()))
    else:
        assert status == 1
