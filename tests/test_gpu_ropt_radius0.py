"""Calibrators whose best radius is 0: log10 r is -inf, so the line through
them is undefined (NaN, with status 0 and their count), wherever they stand in
the catalog, and every other row takes the first radius."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

RADII = (0, 2, 3, 4, 5)


@pytest.mark.parametrize("rows,points", ((3, (0,)), (3, (1,)), (3, (2,)), (3, (0, 2)), (40, (39,)), (40, (1, 17)),
                                         (130, (64,)), (130, (129,))))
def test_radius_zero_calibrators(rows, points):
    """Sources 40 px apart: flat patches of 7 x 7 (best at a larger radius), single pixels at `points`."""
    rng = np.random.default_rng(rows)
    nx = 12
    h, w = 40 * (-(-rows // nx)) + 40, 40 * nx + 40
    img = rng.normal(1000.0, 1.0, (h, w))
    xs, ys = 40.0 + 40 * (np.arange(rows) % nx), 40.0 + 40 * (np.arange(rows) // nx)
    for i, (x, y) in enumerate(zip(xs.astype(int), ys.astype(int))):
        img[y, x] += 3000 + 10 * i
        if i not in points:
            img[y - 3:y + 4, x - 3:x + 4] += 2000 + 7 * i
    cat, _ = gp.allocate_catalog(rows + 1, "cuda")
    cat["n"].fill_(rows + 1)                         # one row more, no calibrator: flagged
    for k, v in (("x", xs), ("y", ys), ("xpeak", xs), ("ypeak", ys)):
        cat[k].copy_(torch.from_numpy(np.append(v, v[0] + 20)))
    cat["flags"].copy_(torch.from_numpy(np.append(np.zeros(rows, np.uint32), np.uint32(gp.GP_FLAG_SAT))))
    my, mx = -(-h // 64), -(-w // 64)
    bkg = {"bkg_mesh": torch.full((my, mx), 1000.0, device="cuda"), "rms_mesh": torch.ones((my, mx), device="cuda"), "mesh": 64}
    ctx = gp.Context(0, workspace_bytes=64 << 20)
    o = ctx.gp_optimal_radius(torch.from_numpy(img.astype(np.float32)).cuda(), bkg, np.ones((3, 3), np.float32), cat, RADII,
                              gain=0.0, snr_min=20.0, d_iso=10.0)
    ctx.sync()
    kopt, calib, fit = o["kopt"].cpu().numpy(), o["calib"].cpu().numpy(), o["fit"].cpu().numpy()
    assert [i for i in range(rows) if kopt[i] == 0] == list(points)
    assert calib[:rows].all() and not calib[rows]
    assert np.isnan(fit[0]) and np.isnan(fit[1]) and fit[2] == rows and fit[3] == 0
    assert np.array_equal(o["kfinal"].cpu().numpy(), np.append(kopt[:rows], 0))
