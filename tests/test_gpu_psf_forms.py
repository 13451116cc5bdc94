"""The varying-PSF threshold pass at the edges of its tiles: widths around a
128-column strip, heights around a 32-row band and its 16-row halves, every
padded kernel size, none to the most modes, meshes whose rows fall inside a
group of rows filled together; the threshold mask against the oracle's
outside the near-threshold set (|S - k sigma| <= 1e-5 |k sigma|)."""
import numpy as np
import pytest

import oracle
from test_gpu_psf import dev, psf_model

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w,mesh,size,K,tile,f32", (
    (64, 64, 32, 3, 1, 32, False), (31, 127, 16, 5, 2, 40, True), (32, 128, 32, 7, 3, 64, False),
    (33, 129, 32, 9, 8, 33, True), (47, 257, 16, 11, 5, 50, False), (48, 130, 24, 13, 4, 48, True),
    (49, 255, 64, 15, 8, 17, False), (257, 300, 16, 15, 7, 60, True), (17, 40, 16, 13, 6, 16, False)))
def test_mask_at_tile_edges(h, w, mesh, size, K, tile, f32):
    rng = np.random.default_rng(h * w + size)
    img = np.round(rng.normal(1000.0, 20.0, (h, w)))
    img[rng.random((h, w)) < 0.03] += 300.0
    img = img.astype(np.float32 if f32 else np.uint16)
    p0, modes, _ = psf_model(size, 1, w, h, tile, 1)
    modes = rng.normal(0.0, 0.02, (K, size, size)).astype(np.float32)
    coef = rng.uniform(-0.4, 0.4, (K, -(-h // tile), -(-w // tile))).astype(np.float32)
    ref = oracle.detect_psf(img, mesh, p0.astype(np.float64), modes.astype(np.float64), coef.astype(np.float64), tile, 1.0, 1)
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    dimg = dev(img)
    out = ctx.gp_detect_psf(dimg, ctx.gp_background(dimg, mesh), p0, modes, dev(coef), tile, 1.0, 1, capacity=h * w)
    ctx.sync()
    mask = (out["segmap"].cpu().numpy().view(np.uint32) != 0).astype(np.uint8)
    assert ref["fg"].any()
    assert not np.any((mask != ref["fg"]) & ~ref["near"])
