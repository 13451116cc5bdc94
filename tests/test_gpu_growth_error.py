"""The growth curve's error is the correctly rounded root of its variance.
With m = K - 1 and sigma = 1 over the frame and a gain of 1 the variance of a
disc of N pixels is the integer N K, exact in the sums; the chosen pairs are
ones whose root lies so close to the middle of two float64 values that a root
without a correct last step takes the other."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,k", ((2, 226131), (10, 44421), (13, 362367), (24, 281239)))
@pytest.mark.parametrize("nr", (1, 2))
def test_error_is_the_rounded_root(r, k, nr):
    n = sum(u * u + v * v <= r * r for u in range(-r, r + 1) for v in range(-r, r + 1))
    img = torch.full((128, 128), float(k - 1), device="cuda")
    bkg = {"bkg_mesh": torch.zeros((2, 2), device="cuda"), "rms_mesh": torch.ones((2, 2), device="cuda"), "mesh": 64}
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    radii = (r,) if nr == 1 else (1, r)
    xs = torch.tensor([60.0, 64.0], dtype=torch.float64)
    f, e, fl = ctx.gp_growth(img, bkg, xs, xs, radii, gain=1.0)
    ctx.sync()
    assert not fl.any() and np.all(f.cpu().numpy()[:, -1] == n * (k - 1))
    assert np.all(e.cpu().numpy()[:, -1] == np.sqrt(np.float64(n) * k))
