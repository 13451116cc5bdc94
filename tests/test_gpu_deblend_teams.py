"""Deblending by every team: segments whose boxes suit a warp, a CTA and a
cluster of CTAs, in one frame, against the oracle; more large segments than
the cluster list holds; and objects whose catalog rows a whole team sums."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


def blob(img, y, x, s, peak):
    yy, xx = np.mgrid[:img.shape[0], :img.shape[1]]
    img += peak * np.exp(-((yy - y) ** 2 + (xx - x) ** 2) / (2 * s * s))


def run(img, f32, minarea=5):
    kern = synth.gaussian_kernel(5, 3.0)
    a = img.astype(np.float32) if f32 else np.clip(np.round(img), 0, 65535).astype(np.uint16)
    H, W = a.shape
    ctx = gp.Context(0, workspace_bytes=512 << 20)
    t = torch.from_numpy(a).cuda()
    mesh = 128
    my, mx = -(-H // mesh), -(-W // mesh)
    bkg = {"bkg_mesh": torch.full((my, mx), 1000.0, device="cuda"),
           "rms_mesh": torch.full((my, mx), 30.0, device="cuda"), "mesh": mesh}
    det = ctx.gp_detect(t, bkg, kern, 1.5, minarea, 20000, saturation=20000.0)
    seg = det["segmap"].clone()
    db = ctx.gp_deblend(t, bkg, kern, 1.5, minarea, seg, det["catalog"], saturation=20000.0)
    ctx.sync()
    m = a.astype(np.float64) - 1000.0
    F = oracle.matched_filter(m, kern)
    margins = {}
    seg0 = det["segmap"].cpu().numpy().view(np.uint32)
    ref, nsplit = oracle.deblend(seg0, F / 30.0, m, 1.5, minarea, margins=margins)
    return seg0, seg.cpu().numpy().view(np.uint32), ref, nsplit, margins, db, m, a


def check(seg0, got, ref, nsplit, margins, db, m, a):
    labels = np.unique(seg0[seg0 > 0])
    clear = np.array([L for L in labels if margins[int(L)]["nu"] > 1e-5 and margins[int(L)]["flux"] > 1e-5], np.uint32)
    inclear = np.isin(seg0, clear)
    assert np.array_equal(got[inclear], ref[inclear])
    # a segment near a bound: the same or another partition into valid objects
    differ = [L for L in labels if not np.array_equal(got[seg0 == L], ref[seg0 == L])]
    assert len(differ) <= 2
    n = int(db["objects"]["n"].item())
    assert n == int(db["counts"][1].item())
    cat = {k: v[:n].cpu().numpy() for k, v in db["objects"].items() if k != "n"}
    rc = oracle.moments(got, m, oracle.saturated(a, 20000.0))
    pos = np.searchsorted(rc["label"], cat["label"])
    for k in ("label", "npix", "xmin", "xmax", "ymin", "ymax", "xpeak", "ypeak", "flags"):
        assert np.array_equal(cat[k], rc[k][pos]), k
    # float32 m and float64 sums: m is exact to 8 u |B|, so the flux to 8 u 1000 npix
    tol = 8 * 2.0 ** -24 * 1000.0 * cat["npix"] + 1e-6
    assert np.all(np.abs(cat["flux_iso"] - rc["flux"][pos]) <= tol)
    return len(labels)


@pytest.mark.parametrize("f32", (False, True))
def test_warp_cta_and_cluster_boxes(f32):
    rng = np.random.default_rng(5)
    img = 1000.0 + rng.normal(0, 4.0, (420, 560))
    blob(img, 150, 170, 45, 900)                      # over 8192 box pixels: a cluster, rows by the whole team
    for y, x in rng.uniform(70, 240, (14, 2)):
        blob(img, y, x, 1.6, rng.uniform(400, 25000))
    blob(img, 340, 120, 18, 500)                      # over 1024: a CTA
    for y, x in ((332, 110), (345, 131), (350, 118)):
        blob(img, y, x, 1.5, 3000)
    for y, x in ((40, 420), (90, 460), (200, 430), (300, 470)):
        blob(img, y, x, 1.6, 2500)                    # pairs: a warp
        blob(img, y + 3, x + 5, 1.6, 2000)
    res = run(img, f32)
    seg0 = res[0]
    area = []
    for L in np.unique(seg0[seg0 > 0]):
        y, x = np.nonzero(seg0 == L)
        area.append((np.ptp(y) + 1) * (np.ptp(x) + 1))
    assert max(area) > 8192 and any(1024 < v <= 8192 for v in area) and any(v <= 1024 for v in area)
    assert res[3] >= 3
    check(*res)


def test_more_large_segments_than_the_list_holds():
    rng = np.random.default_rng(6)
    img = 1000.0 + rng.normal(0, 4.0, (1300, 1300))
    for j in range(8):
        for i in range(8):                            # 64 boxes of some 120 x 120
            y, x = 80 + 160 * j, 80 + 160 * i
            img[y - 55:y + 55, x - 55:x + 55] += 200 + 2 * (i + j)
            blob(img[y - 60:y + 60, x - 60:x + 60], 40 + i, 40, 1.6, 4000)
            blob(img[y - 60:y + 60, x - 60:x + 60], 75, 70 - j, 1.6, 5000)
    res = run(img, False)
    assert check(*res) >= 64 and int(res[5]["counts"][0].item()) >= 60


def test_repeated_calls_give_the_same_bits():
    rng = np.random.default_rng(7)
    img = 1000.0 + rng.normal(0, 20.0, (300, 400))
    blob(img, 150, 180, 40, 400)
    for y, x in rng.uniform(30, 270, (60, 2)):
        blob(img, y, x, 1.6, rng.uniform(300, 9000))
    first = run(img, False, minarea=1)
    for _ in range(4):
        again = run(img, False, minarea=1)
        assert np.array_equal(again[1], first[1])
        for k in first[5]["objects"]:
            assert torch.equal(again[5]["objects"][k], first[5]["objects"][k]), k
