"""Meshes beyond the fused kernel's shared memory: box filling, the median
filter at every size, and the chunked spline solves, at node counts around
the chunk length, against the oracle's whole-line solves; the coefficient
maps of the varying filter go through the same solves at any size."""
import numpy as np
import pytest

import oracle
from parity import assert_close

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fsize", (1, 3, 5, 7))
@pytest.mark.parametrize("mx,my,masked", ((65, 64, False), (64, 130, True), (129, 33, False), (1300, 4, False),
                                          (3, 1400, True), (161, 97, True)))
def test_meshes_and_maps(mx, my, masked, fsize):
    """mesh 16; the last boxes 9 columns wide and 7 rows high."""
    rng = np.random.default_rng(mx + fsize)
    W, H = 16 * (mx - 1) + 9, 16 * (my - 1) + 7
    base = 1000.0 + 300.0 * rng.normal(0, 1, (my, mx)).repeat(16, 0).repeat(16, 1)[:H, :W]
    img = np.clip(np.round(base + rng.normal(0, 20, (H, W))), 0, 65535).astype(np.uint16)
    mask = None
    if masked:                                       # whole boxes without a good pixel, one region three boxes wide
        mask = np.zeros((H, W), np.uint8)
        for _ in range(40):
            i, j = rng.integers(0, mx), rng.integers(0, my)
            mask[16 * j:16 * j + 16, 16 * i:16 * i + 16] = 1
        mask[:48, :48] = 1
    vals, bad = oracle.pixel_values(img, mask)
    bm, rm, _ = oracle.background_meshes(vals, bad, 16, fsize=fsize)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    out = ctx.gp_background(torch.from_numpy(img).cuda(), 16, filter_size=fsize, maps=True,
                            mask=None if mask is None else torch.from_numpy(mask).cuda())
    ctx.sync()
    assert mx * my > 4096 or mx * my == 4160
    assert_close("bkg_mesh", out["bkg_mesh"].cpu().numpy(), bm, np.abs(bm) + 1e-6)
    assert_close("rms_mesh", out["rms_mesh"].cpu().numpy(), rm, np.abs(rm) + 1e-6)
    # the maps from the GPU's own meshes: the spline alone (scale: the nodes' size, as the cubic terms swing as far)
    for name in ("bkg", "rms"):
        nodes = out[name + "_mesh"].cpu().numpy().astype(np.float64)
        ref = oracle.spline_map(nodes, W, H, 16)
        assert_close(name + "_map", out[name + "_map"].cpu().numpy(), ref, np.full(ref.shape, np.abs(nodes).max()))


@pytest.mark.parametrize("tile", (9, 64, 300, 5000))
def test_coefficient_maps(tile):
    """S = c (delta (x) m) over a constant frame reads the coefficient spline back through the threshold."""
    H, W = 520, 700
    rng = np.random.default_rng(tile)
    cy, cx = -(-H // tile), -(-W // tile)
    coef = rng.uniform(0.5, 1.5, (3, cy, cx)).astype(np.float32)
    img = torch.full((H, W), 1100.0, device="cuda")
    bkg = {"bkg_mesh": torch.full((5, 6), 1000.0, device="cuda"), "rms_mesh": torch.full((5, 6), 50.0, device="cuda"),
           "mesh": 128}
    p0 = np.zeros((3, 3), np.float32)
    modes = np.zeros((3, 3, 3), np.float32)
    modes[:, 1, 1] = (1.0, -0.5, 0.25)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    det = ctx.gp_detect_psf(img, bkg, p0, modes, torch.from_numpy(coef).cuda(), tile, 1.5, 1, 200000)
    ctx.sync()
    s = sum(w * oracle.spline_map(c.astype(np.float64), W, H, tile) for w, c in zip((1.0, -0.5, 0.25), coef)) * 100.0
    fg = det["segmap"].cpu().numpy() != 0
    clear = np.abs(s - 75.0) > 1e-3
    assert np.array_equal(fg[clear], (s > 75.0)[clear]) and clear.mean() > 0.99
