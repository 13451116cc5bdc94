"""The salt-and-pepper filter's two forms, chosen by the frame's size: blocks
in shared memory for small frames, warps walking 2 or 8 rows for larger ones.
Every form gives the same pixels: a large frame against its parts filtered
alone (a pixel's fate depends on the 5 x 5 pixels around it), at odd sizes,
unaligned rows, with a mask, with bad float pixels; and against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

BLOCK, FEW = 2 << 20, 6 << 20       # most pixels of the block form; of 2 rows a warp
SIZES = ((1024, 2048), (1025, 2048), (1601, 1503), (2900, 2113), (2731, 2401), (70001, 33), (37, 90001))


def frame(h, w, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    img = torch.randn((h, w), generator=g, device="cuda") * 20 + 1000
    img[torch.rand((h, w), generator=g, device="cuda") < 2e-3] += 900       # lone and touching outliers
    img[h // 3, : min(w, 300)] += 2000                                      # a track along a row
    img[: min(h, 90), w // 2] += 2000
    return img


def run(ctx, img, mask=None, cr=False):
    o = ctx.gp_cosmetic(img, rtn_t=150.5, mask=mask, **(dict(cr_gain=1.5, cr_read_noise=8.0) if cr else {}))
    ctx.sync()
    return o["image"], o["flags"], o["counts"].cpu().numpy()


@pytest.mark.parametrize("kind", ("u16", "u16 unaligned", "f32", "f32 bad", "u16 masked", "f32 masked"))
@pytest.mark.parametrize("h,w", SIZES)
def test_forms_agree(h, w, kind):
    img = frame(h, w, h + w)
    mask = (torch.rand((h, w), device="cuda") < 0.01).to(torch.uint8) if "masked" in kind else None
    if kind.startswith("u16"):
        img = img.round().to(torch.int16)
        if "unaligned" in kind:
            big = torch.zeros((h, w + 3), dtype=torch.int16, device="cuda")
            big[:, 1:1 + w] = img
            img = big[:, 1:1 + w]
        img = img.view(torch.uint16)
    elif "bad" in kind:
        img[torch.rand((h, w), device="cuda") < 5e-3] = float("nan")
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    full, flags, counts = run(ctx, img, mask)
    assert (h * w > BLOCK) == ((h, w) != (1024, 2048))
    assert int((flags == 1).sum()) == counts[0] > 0
    # parts of at most a quarter of a megapixel, 4 pixels over one another
    step = 512 if min(h, w) >= 512 else 4096
    for y in range(0, h, step):
        for x in range(0, w, step):
            ya, yb, xa, xb = max(y - 2, 0), min(y + step + 2, h), max(x - 2, 0), min(x + step + 2, w)
            part = img[ya:yb, xa:xb]
            m = None if mask is None else mask[ya:yb, xa:xb].contiguous()
            img2, fl2, _ = run(ctx, part, m)
            inner = np.s_[y - ya:y - ya + min(step, h - y), x - xa:x - xa + min(step, w - x)]
            whole = np.s_[y:min(y + step, h), x:min(x + step, w)]
            assert torch.equal(fl2[inner], flags[whole])
            assert torch.equal(img2[inner].view(torch.int32), full[whole].view(torch.int32))


@pytest.mark.parametrize("h,w", ((300, 257), (1601, 1503)))
def test_against_the_oracle(h, w):
    img = frame(h, w, 5).round().to(torch.int16).view(torch.uint16)
    ctx = gp.Context(0, workspace_bytes=256 << 20)
    full, flags, _ = run(ctx, img)
    ref, rep = oracle.rtn_filter(img.cpu().numpy(), 150.5)
    assert np.array_equal(flags.cpu().numpy() == 1, rep) and np.array_equal(full.cpu().numpy(), ref.astype(np.float32))
