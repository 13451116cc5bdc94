"""Clip bounds that fall on pixel values: boxes of two values, half each, at
clip_k = 1, where med -/+ sigma are the values themselves.  The exact bounds
keep every pixel, so the box's background is the values' mean and its noise
half their difference; a bound rounded inward would drop them all.  Ragged
boxes (pixel counts that are no powers of two), values inside the uint16
histogram window and outside it, adjacent values, every pixel type."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

BOXES = ((255, 254), (256, 256), (251, 250), (199, 248), (128, 127), (100, 99), (62, 37), (50, 50), (17, 18))


def half_and_half(h, w, lo, hi, dtype):
    img = np.full(h * w, lo, dtype)
    img[::2] = hi
    return np.random.default_rng(h + w).permutation(img).reshape(h, w)


def pairs(seed):
    """Values in one window, around its width, far apart, and adjacent."""
    rng = np.random.default_rng(seed)
    out = [(100, 2993), (100, 101), (0, 65535), (7, 4102), (7, 4104), (100, 52993)]
    for span in (8, 500, 3000, 60000):
        for _ in range(12):
            lo = int(rng.integers(0, 65535 - span))
            out.append((lo, lo + int(rng.integers(1, span + 1))))
    return out


@pytest.mark.parametrize("h,w", BOXES)
def test_two_valued_uint16_boxes_stay_whole(h, w):
    mesh = max(h, w, 16)
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    for lo, hi in pairs(h * w):
        t = torch.from_numpy(half_and_half(h, w, lo, hi, np.uint16)).cuda()
        o = ctx.gp_background(t, mesh, filter_size=1, clip_k=1.0)
        ctx.sync()
        b, r = o["bkg_mesh"].item(), o["rms_mesh"].item()
        # float32 results of float64 statistics
        assert abs(b - (lo + hi) / 2) <= 1e-6 * hi and abs(r - (hi - lo) / 2) <= 1e-6 * hi, (lo, hi, b, r)


@pytest.mark.parametrize("k", (1.0, 1.5, 2.5))
def test_ties_beside_the_median_clip_alike(k):
    """A fifth of the pixels at distance D from the rest puts k sigma = D at k = 2.5: float64 decides such ties, the
    same in every box layout."""
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    for side in (20, 50, 100, 200, 250):
        for d in (5, 10, 400, 1111):
            img = np.full(side * side, 1000, np.uint16)
            img[::5] = 1000 + d
            t = torch.from_numpy(img.reshape(side, side)).cuda()
            o = ctx.gp_background(t, side, filter_size=1, clip_k=k, clip_maxiter=1)
            ctx.sync()
            sd = 0.4 * d
            kept = d <= k * sd * (1 + 1e-12)
            want = (sd if kept else 0.0,)
            got = o["rms_mesh"].item()
            if abs(d - k * sd) > 1e-9 * d:
                assert abs(got - want[0]) <= 1e-6 * max(sd, 1.0), (side, d, got)
            else:                                    # on the bound: one of the two whole sets
                assert min(abs(got - sd), abs(got)) <= 1e-6 * sd, (side, d, got)
