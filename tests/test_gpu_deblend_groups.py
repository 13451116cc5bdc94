"""Deblending by groups of warps: segments whose boxes lie on both sides of
the sizes where a warp, a group and a CTA take over from one another (64 and
1,024 pixels), more of them than the chip has groups, and a handful, against
the oracle.  Rectangles with two bumps each and a 1 x 1 kernel, so that the
boxes are exact."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

BOXES = ((7, 9), (8, 8), (5, 13), (16, 16), (12, 43), (31, 33), (32, 32), (25, 41), (40, 40))


def field(copies):
    """Rectangles at + 150 with two bumps of 3 x 3 at + 900 and + 1100 in opposite corners."""
    cell = 44
    n = copies * len(BOXES)
    nx = int(np.ceil(np.sqrt(n)))
    img = np.full((cell * -(-n // nx) + 3, cell * nx + 3), 1000, np.int64)
    for i in range(n):
        h, w = BOXES[i % len(BOXES)]
        y, x = 1 + cell * (i // nx), 1 + cell * (i % nx)
        img[y:y + h, x:x + w] += 150 + i % 7
        img[y:y + 3, x:x + 3] += 900
        img[y + h - 3:y + h, x + w - 3:x + w] += 1100
    return img


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("copies", (1, 9, 160))
def test_box_sizes_around_the_teams(copies, f32):
    a = field(copies).astype(np.float32 if f32 else np.uint16)
    H, W = a.shape
    kern, mesh = np.ones((1, 1), np.float32), 128
    my, mx = -(-H // mesh), -(-W // mesh)
    ctx = gp.Context(0, workspace_bytes=1 << 30)
    t = torch.from_numpy(a).cuda()
    bkg = {"bkg_mesh": torch.full((my, mx), 1000.0, device="cuda"), "rms_mesh": torch.full((my, mx), 30.0, device="cuda"),
           "mesh": mesh}
    det = ctx.gp_detect(t, bkg, kern, 1.5, 5, 20000)
    seg = det["segmap"].clone()
    db = ctx.gp_deblend(t, bkg, kern, 1.5, 5, seg, det["catalog"])
    ctx.sync()
    n = copies * len(BOXES)
    assert int(det["catalog"]["n"].item()) == n
    m = a.astype(np.float64) - 1000.0
    margins = {}
    seg0 = det["segmap"].cpu().numpy().view(np.uint32)
    ref, nsplit = oracle.deblend(seg0, m / 30.0, m, 1.5, 5, margins=margins)
    assert nsplit == n and min(v["nu"] for v in margins.values()) > 1e-5 and min(v["flux"] for v in margins.values()) > 1e-5
    assert np.array_equal(seg.cpu().numpy().view(np.uint32), ref)
    assert db["counts"].cpu().numpy().tolist() == [n, 2 * n]
    cat = {k: v[:2 * n].cpu().numpy() for k, v in db["objects"].items() if k != "n"}
    rc = oracle.moments(ref, m, np.zeros(a.shape, bool))
    for k in ("label", "npix", "xmin", "xmax", "ymin", "ymax", "xpeak", "ypeak", "flags"):
        assert np.array_equal(cat[k], rc[k]), k
    assert np.array_equal(cat["flux_iso"], rc["flux"])       # sums of whole numbers


def test_more_segments_than_the_chip_has_warps():
    """Where warps take larger boxes: every rectangle splits as its like does in a small frame."""
    def patches(copies):
        a = field(copies).astype(np.uint16)
        H, W = a.shape
        kern, mesh = np.ones((1, 1), np.float32), 128
        my, mx = -(-H // mesh), -(-W // mesh)
        ctx = gp.Context(0, workspace_bytes=1 << 30)
        t = torch.from_numpy(a).cuda()
        bkg = {"bkg_mesh": torch.full((my, mx), 1000.0, device="cuda"),
               "rms_mesh": torch.full((my, mx), 30.0, device="cuda"), "mesh": mesh}
        det = ctx.gp_detect(t, bkg, kern, 1.5, 5, 20000)
        seg = det["segmap"].clone()
        db = ctx.gp_deblend(t, bkg, kern, 1.5, 5, seg, det["catalog"])
        ctx.sync()
        n = copies * len(BOXES)
        assert int(det["catalog"]["n"].item()) == n and db["counts"].cpu().numpy().tolist() == [n, 2 * n]
        s, nx = seg.cpu().numpy(), int(np.ceil(np.sqrt(n)))
        for i in range(n):
            (h, w), y, x = BOXES[i % len(BOXES)], 1 + 44 * (i // nx), 1 + 44 * (i % nx)
            yield i, np.unique(s[y:y + h, x:x + w], return_inverse=True)[1].reshape(-1)

    like = {i % 63: p for i, p in patches(9)}                # 9 boxes by 7 levels
    assert len(like) == 63
    for i, p in patches(600):
        assert np.array_equal(p, like[i % 63]), i
