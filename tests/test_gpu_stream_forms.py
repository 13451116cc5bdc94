"""The streaming pass's forms on one frame: tensor-map staging against the
direct one (vector loads and element loads), with and without a mask, fast
and general, single and batched, at heights around its row chunks and widths
around its strips.  All read the same pixels, so every output is the same;
the general one is checked against the oracle."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

SIZES = ((17, 16), (31, 40), (33, 600), (64, 512), (65, 513), (129, 1030), (160, 2056))


def frame(h, w, f32, seed):
    cfg = synth.scaled_config(synth.CONFIGS["plain_1024x1024_f32" if f32 else "plain_2048x2048_u16"], w, h,
                              nsrc=max(3, h * w // 1500), name="stream")
    return cfg, synth.make_frame(cfg, seed, cache=False)[0]


def unaligned(t, pad):
    """The same frame with rows `pad` elements longer, starting one element in."""
    big = torch.zeros((t.shape[0], t.shape[1] + pad), dtype=torch.int16 if t.element_size() == 2 else t.dtype,
                      device="cuda").view(t.dtype)
    v = big[:, 1:1 + t.shape[1]]
    v.copy_(t)
    return v


def same(a, b):
    assert torch.equal(a["segmap"], b["segmap"])
    n = int(a["catalog"]["n"].item())
    assert n == int(b["catalog"]["n"].item())
    for k in a["catalog"]:
        assert torch.equal(a["catalog"][k][:n], b["catalog"][k][:n]), k
    assert torch.equal(a["flux"][:n], b["flux"][:n])


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("ks", (3, 5, 7, 15))
@pytest.mark.parametrize("h,w", SIZES)
def test_stagings_agree(h, w, ks, f32):
    cfg, img = frame(h, w, f32, 3 * h + w)
    if f32:
        img = img.copy()
        img[h // 2, w // 3] = np.nan
        img[0, 0] = np.inf
    kern = synth.gaussian_kernel(ks, 3.0)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    t = torch.from_numpy(img).cuda()

    def run(x, **kw):
        out = ctx.gp_extract(x, 32, kern, 2.0, 3, (3.0,), cfg.gain, capacity=4096, saturation=cfg.saturation, **kw)
        ctx.sync()
        return out

    general = run(t, mask_out=True)
    mask = general["mask"].cpu().numpy()
    ref = oracle.extract(img, 32, kern, 2.0, 3, (3.0,), cfg.gain, saturation=cfg.saturation)
    assert not np.any((mask != ref["fg"]) & ~ref["near"])
    assert np.array_equal(general["segmap"].cpu().numpy().view(np.uint32), oracle.label(mask, 3)[0])
    fast = run(t)
    same(fast, general)
    for pad in (4, 16, 17):
        same(run(unaligned(t, pad)), fast)
    # a mask without a bad pixel, then one that repeats the frame's own bad pixels
    zero = torch.zeros((h, w), dtype=torch.uint8, device="cuda")
    same(run(t, mask=zero), fast)
    if f32:
        same(run(t, mask=(~torch.isfinite(t)).to(torch.uint8)), fast)
    bx = gp.BatchExtractor(ctx, [(h, w), (40, 64)], t.dtype, 32, kern, 2.0, 3, (3.0,), cfg.gain, 4096,
                           saturation=cfg.saturation)
    other = torch.from_numpy(frame(40, 64, f32, 7)[1]).cuda()
    for x in (t, unaligned(t, 17)):
        same(bx.run([x, other])[0], fast)


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("h,w", ((40, 530), (131, 1040), (33, 2048), (64, 63)))
def test_masked_pixels(h, w, f32):
    cfg, img = frame(h, w, f32, h + w)
    rng = np.random.default_rng(h)
    bad = (rng.random((h, w)) < 0.03).astype(np.uint8)
    bad[:, w // 2] = 7
    bad[0], bad[:, -1] = 1, 1
    kern = synth.gaussian_kernel(5, 3.0)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    t, m = torch.from_numpy(img).cuda(), torch.from_numpy(bad).cuda()
    outs = []
    for x in (t, unaligned(t, 17), unaligned(t, 16)):
        outs.append(ctx.gp_extract(x, 32, kern, 2.0, 3, (3.0,), cfg.gain, capacity=4096, mask=m, mask_out=True,
                                   saturation=cfg.saturation))
        ctx.sync()
    got = outs[0]["mask"].cpu().numpy()
    ref = oracle.extract(img, 32, kern, 2.0, 3, (3.0,), cfg.gain, mask=bad, saturation=cfg.saturation)
    assert not np.any((got != ref["fg"]) & ~ref["near"])
    assert not np.any(got[bad != 0])
    assert np.array_equal(outs[0]["segmap"].cpu().numpy().view(np.uint32), oracle.label(got, 3)[0])
    for o in outs[1:]:
        same(o, outs[0])
        assert torch.equal(o["mask"], outs[0]["mask"])
