"""Circular apertures over windows of one and several chunks of 32 rows and
columns: small and large radii, one to eight of them, positions at pixel
centres, at the frame's edge and outside, undefined ones, bad and saturated
pixels, a mesh whose rows change inside the window; against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

U8 = 8 * 2.0 ** -24


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("radii", ((0.4,), (2.5, 3.0), (3.0, 6.0, 10.0), (13.9, 14.1, 14.9), (1.0, 2.0, 3.0, 40.0),
                                   (0.5, 1.5, 2.5, 3.5, 4.5, 5.5, 6.5, 7.5)))
def test_apertures_match_the_oracle(radii, f32):
    rng = np.random.default_rng(len(radii))
    H, W, mesh = 150, 210, 24
    img = np.round(rng.normal(1000.0, 20.0, (H, W)))
    img[rng.random((H, W)) < 0.002] = 60000.0
    img = img.astype(np.float32 if f32 else np.uint16)
    mask = (rng.random((H, W)) < 0.001).astype(np.uint8)
    my, mx = -(-H // mesh), -(-W // mesh)
    bm = rng.normal(1000.0, 5.0, (my, mx)).astype(np.float32)
    rm = rng.uniform(15.0, 25.0, (my, mx)).astype(np.float32)
    xs = np.concatenate([rng.uniform(-8, W + 8, 150), [100.0, 100.5, 0.0, W - 1.0, -1e9, np.nan]])
    ys = np.concatenate([rng.uniform(-8, H + 8, 150), [50.0, 50.5, 0.0, H - 1.0, 10.0, 20.0]])
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    bkg = {"bkg_mesh": torch.from_numpy(bm).cuda(), "rms_mesh": torch.from_numpy(rm).cuda(), "mesh": mesh}
    f, e, fl = ctx.gp_aperture(torch.from_numpy(img).cuda(), bkg, torch.from_numpy(xs), torch.from_numpy(ys), radii,
                               gain=1.5, mask=torch.from_numpy(mask).cuda(), saturation=50000.0)
    ctx.sync()
    vals, bad = oracle.pixel_values(img, mask)
    bmap, rmap = oracle.spline_map(bm.astype(np.float64), W, H, mesh), oracle.spline_map(rm.astype(np.float64), W, H, mesh)
    m, var, sat = np.where(bad, 0.0, vals - bmap), np.where(bad, 0.0, rmap ** 2), oracle.saturated(img, 50000.0)
    ok = np.abs(xs) < 1e6                            # the far and the undefined position: empty sums
    rf, re, rfl = oracle.apertures(m, var, bad, sat, xs[ok], ys[ok], radii, 1.5)
    scale, _, _ = oracle.apertures(np.abs(m) + U8 / 1e-5 * np.abs(bmap), var, bad, sat, xs[ok], ys[ok], radii, 0.0)
    got = f.cpu().numpy()
    assert np.all(np.abs(got[ok] - rf) <= 1e-5 * scale + 1e-6)
    assert np.all(np.abs(e.cpu().numpy()[ok] - re) <= 1e-5 * np.maximum(re, 1.0))
    assert np.array_equal(fl.cpu().numpy()[ok].view(np.uint32), rfl.astype(np.uint32))
    assert not got[~ok].any()
