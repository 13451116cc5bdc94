"""The training step's fused kernels against the separate ones: the gated
data gradient (convolution and ReLU backward in one launch) bit for bit, and the
update of all layers (AdamW and packing in one launch)."""
import pytest

torch = pytest.importorskip("torch")
gp = pytest.importorskip("paper_2609_32375_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,h,w", ((1, 1, 1), (1, 5, 63), (2, 64, 64), (3, 7, 65), (40, 17, 130)))
@pytest.mark.parametrize("cop,cip", ((16, 32), (32, 32), (32, 48), (48, 48), (48, 32)))
def test_gated_gradient_is_convolution_then_relu_backward(n, h, w, cop, cip):
    lib = gp.load_library()
    g = torch.Generator(device="cuda").manual_seed(n * h + w)
    dp = torch.randn((n, h, w, cop), generator=g, device="cuda").bfloat16()
    wtd = (0.1 * torch.randn((cip, 9 * cop), generator=g, device="cuda")).bfloat16()
    act = torch.randn((n, h, w, cip), generator=g, device="cuda").bfloat16()
    act[..., ::5] = 0.0
    act[..., 1::7] = float("nan")
    act[..., 2::9] = -0.0
    zero = torch.zeros(cip, device="cuda")
    dy, ref, got, plain = (torch.full_like(act, 7.0) for _ in range(4))
    s = torch.cuda.current_stream().cuda_stream or None
    for status in (
            lib.gp_cnn_conv3x3(dp.data_ptr(), n, h, w, cop, wtd.data_ptr(), zero.data_ptr(), cip, 0, dy.data_ptr(), 0, 0, s),
            lib.gp_cnn_relu_backward(dy.data_ptr(), act.data_ptr(), ref.data_ptr(), ref.numel(), s),
            lib.gp_cnn_conv3x3_dgrad(dp.data_ptr(), n, h, w, cop, wtd.data_ptr(), cip, act.data_ptr(), got.data_ptr(), s),
            lib.gp_cnn_conv3x3_dgrad(dp.data_ptr(), n, h, w, cop, wtd.data_ptr(), cip, None, plain.data_ptr(), s)):
        assert status == 0
    torch.cuda.synchronize()
    assert torch.equal(got.view(torch.int16), ref.view(torch.int16))
    assert torch.equal(plain.view(torch.int16), dy.view(torch.int16))


def test_update_is_adamw_then_pack():
    from paper_2609_32375_gb300 import learned
    a, b = learned.Network(seed=3), learned.Network(seed=3)
    g = torch.Generator(device="cuda").manual_seed(1)
    s = torch.cuda.current_stream().cuda_stream or None
    for step in (1, 2, 3):
        grads = [(torch.randn(w.shape, generator=g, device="cuda"), torch.randn(c.shape, generator=g, device="cuda"))
                 for w, c in zip(a.W, a.b)]
        a.adamw(grads, lr=1e-2)
        for l, (dw, db) in enumerate(grads):
            for p, d, m, v, wd in ((b.W[l], dw, b.mW[l], b.vW[l], 1e-4), (b.b[l], db, b.mb[l], b.vb[l], 0.0)):
                assert b._lib.gp_cnn_adamw(p.data_ptr(), d.data_ptr(), m.data_ptr(), v.data_ptr(), p.numel(), 1e-2, 0.9,
                                           0.999, 1e-8, wd, step, s) == 0
        b.pack()
    # a few float32 roundings a step, of terms up to 0.1 (steps of size lr) and 1 (moments of gradients)
    for k, scale in (("W", 0.1), ("b", 0.1), ("mW", 1.0), ("mb", 1.0), ("vW", 1.0), ("vb", 1.0)):
        for p, q in zip(getattr(a, k), getattr(b, k)):
            assert torch.all((p - q).abs() <= 3 * 8 * 2.0 ** -24 * (q.abs() + scale))
    wt, wtd, bias = ([t.clone() for t in getattr(a, k)] for k in ("wt", "wtd", "bias"))
    a.pack()                                       # of the same master weights
    for got, ref in ((wt, a.wt), (wtd, a.wtd), (bias, a.bias)):
        assert all(torch.equal(p, q) for p, q in zip(got, ref))
