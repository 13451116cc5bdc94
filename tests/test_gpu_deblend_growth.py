"""Growth rounds beyond the common sizes: a box too large for a CTA's shared
memory, whose rounds run in global memory; and a long plateau whose rounds
list more candidates than the shared list holds, so that the rest go to
global memory.  Against the oracle, and repeated to the same bits (the rounds'
accesses to the shared states are all of one size)."""
import numpy as np
import pytest

from test_gpu_deblend_teams import blob, check, run

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

SHARED_BOX = 103000        # pixels of the largest box held in shared memory
SHARED_LIST = 1024         # candidates of a round held there


def large_box():
    img = np.full((420, 420), 1000.0)
    img[40:380, 40:380] += 400
    for y, x in ((100, 110), (150, 300), (300, 120), (290, 310), (200, 200)):
        blob(img, y, x, 6, 6000 + 10 * x)
    return np.round(img), 5, lambda area: area > SHARED_BOX


def long_plateau():
    """Two ridges of 1330 columns: the first round below them opens some 5000 pixels, each of the next as many."""
    img = np.full((90, 1450), 1000.0)
    img[15:75, 30:1420] += 600
    img[30:33, 60:1390] += 3000
    img[50:53, 60:1390] += 3500
    assert 1390 - 60 > SHARED_LIST
    return img, 2, lambda area: 8192 < area <= SHARED_BOX


@pytest.mark.parametrize("f32", (False, True))
@pytest.mark.parametrize("field", (large_box, long_plateau))
def test_growth_beyond_shared_memory(field, f32):
    img, objects, size_ok = field()
    res = run(img, f32)
    seg0, got = res[0], res[1]
    y, x = np.nonzero(seg0)
    assert len(np.unique(seg0)) == 2 and size_ok((np.ptp(y) + 1) * (np.ptp(x) + 1))
    margin = res[4][int(seg0.max())]
    assert margin["nu"] > 1e-5 and margin["flux"] > 1e-5            # no pixel near a level: one right answer
    assert len(np.unique(got[got > 0])) == objects
    check(*res)
    for _ in range(3):
        again = run(img, f32)
        assert np.array_equal(again[1], got)
        for k, v in res[5]["objects"].items():
            assert torch.equal(again[5]["objects"][k], v), k
