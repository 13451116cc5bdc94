"""The network kernels at the edges of their tiles: the four-row and the
one-row convolution tilings give the same bits, and the weight gradient
agrees with the oracle at ragged widths, few rows and unaligned arrays."""
import numpy as np
import pytest

from oracle import cnn as ocnn

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu

PAIRS = [(16, 32), (32, 48), (48, 48), (48, 32), (32, 32), (32, 16)]


def stream():
    return torch.cuda.current_stream().cuda_stream or None


def conv(x, wt, bias, cop, f32):
    n, h, w, cip = x.shape
    y = torch.full((n, h, w, cop), 7.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    assert gp.load_library().gp_cnn_conv3x3(x.data_ptr(), n, h, w, cip, wt.data_ptr(), bias.data_ptr(), cop, 1,
                                            y.data_ptr(), int(f32), cop, stream()) == gp.GP_OK
    return y


@pytest.mark.parametrize("cip,cop", PAIRS)
@pytest.mark.parametrize("h,w", ((1, 1), (3, 64), (4, 65), (9, 31)))
def test_conv_tilings_agree(cip, cop, h, w):
    g = torch.Generator(device="cuda").manual_seed(h * 100 + w)
    n = 160                                      # a tile for every SM: the four-row form
    x = torch.randn((n, h, w, cip), generator=g, device="cuda").to(torch.bfloat16)
    wt = (torch.randn((cop, 9 * cip), generator=g, device="cuda") * 0.1).to(torch.bfloat16)
    b = torch.randn(cop, generator=g, device="cuda")
    for f32 in (False, True):
        y = conv(x, wt, b, cop, f32)
        for k in (0, 1, n - 1):                  # one frame: the one-row form
            assert torch.equal(y[k], conv(x[k:k + 1].contiguous(), wt, b, cop, f32)[0])


@pytest.mark.parametrize("cip,cop", PAIRS)
@pytest.mark.parametrize("n,h,w,nslot", ((1, 1, 1, 4), (2, 3, 63, 64), (1, 5, 65, 2), (3, 4, 128, 5)))
def test_weight_gradient_edges(cip, cop, n, h, w, nslot):
    rng = np.random.default_rng(cip + cop + w)
    x = ocnn.bf16_round(rng.normal(size=(n, h, w, cip)))
    dp = ocnn.bf16_round(rng.normal(size=(n, h, w, cop)))
    zero = np.zeros((cop, cip, 3, 3))
    _, rW, rb = ocnn.conv3x3_backward(x, zero, dp)
    _, sW, sb = ocnn.conv3x3_backward(np.abs(x), zero, np.abs(dp))
    got = []
    for shift in (0, 1):                         # one element off a 16-byte boundary: element loads
        def put(a):
            t = torch.zeros(a.size + 8, dtype=torch.bfloat16, device="cuda")
            t[shift:shift + a.size] = torch.from_numpy(a.astype(np.float32)).to(torch.bfloat16).cuda().reshape(-1)
            return t
        tx, td = put(x), put(dp)
        part = torch.empty(nslot * 9 * cop * cip, device="cuda")
        bpart = torch.empty(nslot * cop, device="cuda")
        dW, db = torch.empty((cop, cip, 3, 3), device="cuda"), torch.empty(cop, device="cuda")
        assert gp.load_library().gp_cnn_conv3x3_wgrad(
            tx.data_ptr() + 2 * shift, td.data_ptr() + 2 * shift, n, h, w, cip, cop, cip, cop, nslot,
            part.data_ptr(), bpart.data_ptr(), dW.data_ptr(), db.data_ptr(), stream()) == gp.GP_OK
        got.append((dW, db))
        # float32 sums of n*h*w products: the bound of the layer tests
        assert (np.abs(dW.cpu().numpy() - rW) / (sW + 1e-6)).max() < 2e-6
        assert (np.abs(db.cpu().numpy() - rb) / (sb + 1e-6)).max() < 2e-6
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("count", (1, 7, 8, 4096, 4099))
def test_relu_backward_vector_tail(count):
    g = torch.Generator(device="cuda").manual_seed(count)
    y = torch.randn(count + 1, generator=g, device="cuda").to(torch.bfloat16)
    y[::5] = 0.0
    y[1::11] = -0.0
    y[::13] = float("inf")
    dy = torch.randn(count + 1, generator=g, device="cuda").to(torch.bfloat16)
    for o in (0, 1):
        out = torch.full((count + 1,), 9.0, dtype=torch.bfloat16, device="cuda")
        assert gp.load_library().gp_cnn_relu_backward(dy.data_ptr() + 2 * o, y.data_ptr() + 2 * o,
                                                      out.data_ptr() + 2 * o, count, stream()) == gp.GP_OK
        want = torch.where(y[o:o + count].float() > 0, dy[o:o + count], torch.zeros_like(dy[o:o + count]))
        assert torch.equal(out[o:o + count], want)
        if o == 0:
            assert out[count] == 9.0
