"""The cosmetic filters' certain "no" and exact rest, at the edges of their
blocks and rows: small and ragged frames, both pixel types, blocks with and
without bad pixels, unaligned rows, and a sharpness limit every pixel
passes.  Decisions as in test_gpu_cosmetic.py: exact except within 1e-4 of a
threshold; the salt-and-pepper filter exact on integer frames."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

SIZES = ((3, 5), (16, 31), (33, 64), (45, 100), (70, 131), (64, 260))


def frame(h, w, seed):
    rng = np.random.default_rng(seed)
    img = rng.poisson(800.0, (h, w)).astype(np.float64)
    yy, xx = np.mgrid[:h, :w]
    for _ in range(max(1, h * w // 400)):                      # stars
        y, x, f = rng.uniform(0, h), rng.uniform(0, w), rng.uniform(300, 20000)
        img += f * np.exp(-((yy - y) ** 2 + (xx - x) ** 2) / 4.0)
    n = max(2, h * w // 150)                                   # hits, pairs, dark pixels
    img[rng.integers(0, h, n), rng.integers(0, w, n)] += rng.uniform(200, 5000, n)
    img[rng.integers(0, h, n), rng.integers(0, w, n)] -= rng.uniform(160, 700, n)
    img[0, :3] += 900
    img[h - 1, w - 1] += 2500
    return np.clip(np.round(img), 0, 65535).astype(np.uint16), rng


def unaligned(t, pad):
    big = torch.zeros((t.shape[0], t.shape[1] + pad), dtype=torch.int16 if t.element_size() == 2 else t.dtype,
                      device="cuda").view(t.dtype)
    v = big[:, 1:1 + t.shape[1]]
    v.copy_(t)
    return v


@pytest.mark.parametrize("kind", ("u16", "u16 mask", "f32", "f32 bad"))
@pytest.mark.parametrize("h,w", SIZES)
def test_filters(h, w, kind):
    img, rng = frame(h, w, h * w)
    mask = None
    if kind == "u16 mask":
        mask = (rng.random((h, w)) < 0.01).astype(np.uint8)
    if kind.startswith("f32"):
        img = img.astype(np.float32)
    if kind == "f32 bad":                                      # bad pixels in a corner: other blocks hold none
        img[:9, :9][rng.random(img[:9, :9].shape) < 0.2] = np.nan
        img[h // 2, 0] = np.inf
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    t = torch.from_numpy(img).cuda()
    m = None if mask is None else torch.from_numpy(mask).cuda()
    ref, rep = oracle.rtn_filter(img, 150.5, mask=mask)
    for x in (t, unaligned(t, 3), unaligned(t, 8)):
        out = ctx.gp_cosmetic(x, rtn_t=150.5, mask=m)
        ctx.sync()
        assert np.array_equal(out["flags"].cpu().numpy() == 1, rep)
        assert np.array_equal(out["image"].cpu().numpy().astype(np.float64), ref, equal_nan=True)
        assert out["counts"].cpu().numpy().tolist() == [int(rep.sum()), 0]
    for clip, lim in ((4.5, 5.0), (0.0, 2.0), (-1.0, 0.5)):
        c, flag, d = oracle.cr_filter(img, 1.5, 8.0, clip, lim, mask=mask, details=True)
        amb = (np.abs(d["sp"] - clip) <= 1e-4 * max(abs(clip), 1)) | (np.abs(d["ratio"] - lim) <= 1e-4 * lim)
        near = np.zeros_like(amb)
        for y, x in np.argwhere(amb):
            near[max(0, y - 2):y + 3, max(0, x - 2):x + 3] = True
        first = None
        for x in (t, unaligned(t, 3), unaligned(t, 8)):
            out = ctx.gp_cosmetic(x, cr_gain=1.5, cr_read_noise=8.0, cr_sigclip=clip, cr_objlim=lim, mask=m)
            ctx.sync()
            f, g = out["flags"].cpu().numpy(), out["image"].cpu().numpy()
            assert np.array_equal((f == 2)[~amb], flag[~amb])
            assert np.array_equal(g.astype(np.float64)[~near], c[~near], equal_nan=True)
            assert int(out["counts"][1].item()) == int((f == 2).sum())
            first = first or (f, g)
            assert np.array_equal(f, first[0]) and np.array_equal(g, first[1], equal_nan=True)
