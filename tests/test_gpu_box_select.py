"""Float32 box statistics and feature scaling, whose order statistics come
from histograms of a range instead of a sort: every thread layout (box sides
16 to 128), ragged boxes, ties, signed zeros, constants, wide ranges."""
import numpy as np
import pytest

import oracle
from parity import assert_close

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")
from paper_2609_32375_gb300 import learned  # noqa: E402

pytestmark = pytest.mark.gpu


def values(kind, shape, rng):
    sky = rng.normal(0.0, 30.0, shape)
    if kind == "sky":
        v = 1000.0 + sky
        v[rng.random(shape) < 0.01] += 3e4
    elif kind == "integers":                     # many equal values
        v = np.round(200.0 + sky / 6)
    elif kind == "signed":                       # a subtracted sky: both signs, both zeros
        v = np.round(sky / 10)
        v[rng.random(shape) < 0.05] = -0.0
    elif kind == "constant":
        v = np.full(shape, 1234.5)
    else:                                        # "wide": eighteen decades
        v = 10.0 ** rng.uniform(-3, 15, shape) * rng.choice((-1, 1), shape)
    return v.astype(np.float32)


@pytest.mark.parametrize("kind", ("sky", "integers", "signed", "constant", "wide"))
@pytest.mark.parametrize("mesh", (16, 31, 32, 33, 64, 65, 128))
def test_float_box_statistics(mesh, kind):
    rng = np.random.default_rng(mesh)
    H, W = 2 * mesh + 5, 3 * mesh + 1            # last boxes 5 rows high, 1 column wide
    img = values(kind, (H, W), rng)
    mask = (rng.random((H, W)) < 0.2).astype(np.uint8)
    img[rng.random((H, W)) < 0.05] = np.nan
    mask[:mesh, :mesh] = 1                       # a box without a good pixel
    mask[5, 7] = 0
    vals, bad = oracle.pixel_values(img, mask)
    bm, rm, _ = oracle.background_meshes(vals, bad, mesh, fsize=1)
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    out = ctx.gp_background(torch.from_numpy(img).cuda(), mesh, filter_size=1, mask=torch.from_numpy(mask).cuda())
    ctx.sync()
    # the mode estimate is a difference of median and mean: its error scales with sigma too
    assert_close("bkg_mesh", out["bkg_mesh"].cpu().numpy(), bm, np.abs(bm) + rm + 1e-6)
    assert_close("rms_mesh", out["rms_mesh"].cpu().numpy(), rm, rm + 1e-6)
    # quantiles are values of the box, exactly
    q = learned.box_quantiles(ctx, torch.from_numpy(img).cuda(), mesh).cpu().numpy()
    for j in range(q.shape[1]):
        for i in range(q.shape[2]):
            b = img[j * mesh:(j + 1) * mesh, i * mesh:(i + 1) * mesh]
            b = np.sort(b[np.isfinite(b)])
            for k, f in enumerate((0.10, 0.25, 0.50, 0.75, 0.90)):
                want = b[int(np.floor(np.float64(np.float32(f)) * (b.size - 1) + 0.5))] if b.size else 0.0
                assert q[k, j, i] == want


@pytest.mark.parametrize("nbox", (1, 2, 31, 1024, 1025, 5000))
def test_feature_scaling(nbox):
    rng = np.random.default_rng(nbox)
    q = np.sort(1000.0 + rng.normal(0, 20, (2, nbox, 5)), axis=2).transpose(0, 2, 1).astype(np.float32)
    q[1] = np.round(q[1])                        # ties
    if nbox > 4:
        q[0, :, :3] = 0.0                        # empty boxes
    feat, norm = learned.features(torch.from_numpy(q[:, :, None, :].copy()).cuda())
    c = np.median(q[:, 2], axis=1)
    s = np.median(q[:, 3] - q[:, 1], axis=1) / np.float32(1.349)
    s = np.where(s > 0, s, np.float32(1.0))
    n = norm.cpu().numpy()
    assert np.array_equal(n[:, 0], c) and np.array_equal(n[:, 1], s.astype(np.float32))
    want = torch.from_numpy(((q - c[:, None, None]) / s[:, None, None]).astype(np.float32)).to(torch.bfloat16)
    got = feat.cpu().reshape(2, nbox, 16)
    assert torch.equal(got[..., :5], want.permute(0, 2, 1)) and not got[..., 5:].any()
