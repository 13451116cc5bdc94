"""uint16 box statistics from the windowed histogram with its list of values
outside the window: none, few, as many as the list holds, one more, far too
many; above, below and on both sides; every thread count (few and many boxes,
small and large)."""
import numpy as np
import pytest

import oracle
from parity import assert_close

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("masked", (False, True))
@pytest.mark.parametrize("side", ("above", "below", "both"))
@pytest.mark.parametrize("mesh,nx,ny", ((32, 40, 40), (128, 5, 4), (128, 40, 20), (256, 3, 2), (100, 7, 3)))
def test_values_outside_the_window(mesh, nx, ny, side, masked):
    rng = np.random.default_rng(mesh + nx)
    H, W = ny * mesh - 3, nx * mesh - 5
    img = rng.normal(20000.0, 40.0, (H, W))
    counts = [0, 3, 40, 300, 1023, 1024, 1025, 3000]
    for b in range(nx * ny):
        y0, x0 = b // nx * mesh, b % nx * mesh
        box = img[y0:y0 + mesh, x0:x0 + mesh]
        n = min(counts[b % len(counts)], box.size // 8)
        at = rng.choice(box.size, n, replace=False)
        hi, lo = rng.uniform(23000, 65535, n), rng.uniform(0, 17000, n)
        v = hi if side == "above" else lo if side == "below" else np.where(rng.random(n) < 0.5, hi, lo)
        flat = box.reshape(-1).copy()
        flat[at] = v
        img[y0:y0 + mesh, x0:x0 + mesh] = flat.reshape(box.shape)
    img = np.round(img).astype(np.uint16)
    mask = (rng.random((H, W)) < 0.05).astype(np.uint8) if masked else None
    vals, bad = oracle.pixel_values(img, mask)
    bm, rm, _ = oracle.background_meshes(vals, bad, mesh, fsize=1)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    t = torch.from_numpy(img).cuda()
    m = None if mask is None else torch.from_numpy(mask).cuda()
    out = ctx.gp_background(t, mesh, filter_size=1, mask=m)
    ctx.sync()
    assert_close("bkg_mesh", out["bkg_mesh"].cpu().numpy(), bm, np.abs(bm))
    assert_close("rms_mesh", out["rms_mesh"].cpu().numpy(), rm, rm)
