"""Which meshes take the single-kernel mesh stage, whose splines are float32:
up to 4,096 nodes, but not those with so long an axis that the stage never
held them; they keep the float64 solves.  Seen by the launches of a call."""
import numpy as np
import pytest

import oracle
from parity import assert_close

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


def call(mx, my, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    img = torch.rand((16 * my, 16 * mx), generator=g, device="cuda") * 20 + 1000
    ctx = gp.Context(0, workspace_bytes=512 << 20)
    out = ctx.gp_background(img, 16)
    ctx.sync()
    return img, out, ctx.stats()["launches"]


@pytest.mark.parametrize("mx,my,single", ((64, 64, True), (2000, 2, True), (1, 2700, True), (65, 64, False),
                                          (4096, 1, False), (1, 4096, False), (2, 2048, False), (1365, 3, True)))
def test_long_narrow_meshes_keep_float64(mx, my, single):
    img, out, launches = call(mx, my)
    assert (launches == call(64, 64)[2]) == single
    vals, bad = oracle.pixel_values(img.cpu().numpy(), None)
    bm, rm, _ = oracle.background_meshes(vals, bad, 16)
    assert_close("bkg_mesh", out["bkg_mesh"].cpu().numpy(), bm, np.abs(bm))
    assert_close("rms_mesh", out["rms_mesh"].cpu().numpy(), rm, rm)
