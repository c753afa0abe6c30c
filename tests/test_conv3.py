"""3 x 3 convolutions with BF16 products against the im2col path they stand
for (nn_im2col3 + nn_gemm_bf16 + nn_bias_act / nn_col2im3_add): the same
products in the same order, so the results are equal bit for bit, whatever the
tiles, the K slices and the alignment."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [  # ci, co, B, H, W
    (1, 1, 1, 1, 1),        # one pixel: nothing but padding around it
    (3, 5, 2, 3, 2),
    (2, 24, 1, 8, 32),      # one 32-pixel segment; weight rows of 18 values
    (24, 24, 2, 9, 64),     # image rows ending inside a tile
    (17, 33, 3, 5, 20),     # the narrowest rows on the tiled kernels, channels off every tile
    (16, 32, 2, 12, 16),    # narrower: gathered forward, tiled weight gradient
    (96, 49, 1, 7, 36),     # a ragged second segment
    (40, 97, 1, 6, 40),     # two row tiles of output channels
    (24, 48, 2, 11, 50),    # rows whose 16-byte groups straddle: gathered
    (72, 24, 1, 25, 25),
    (192, 200, 1, 4, 24),   # deep: three taps, then one tap of weights at a time
    (48, 64, 2, 64, 96),    # enough pixels for K slices of the weight gradient
]


def _path(L, x, w, bias, dy, dx, relu, wk, add):
    import torch
    ci, B, H, W = x.shape
    co, P, K = w.shape[0], B * H * W, 9 * ci
    p = lambda t: t.data_ptr()
    col = torch.empty(K * P, device="cuda")
    y, gw = torch.empty(co, B, H, W, device="cuda"), torch.empty(co, K, device="cuda")
    dx = dx.clone() if add else torch.zeros_like(dx)
    rc = [L.nn_im2col3(p(x), ci, B, H, W, p(col), None),
          L.nn_gemm_bf16(0, 0, co, P, K, 1.0, p(w), K, p(col), P, 0.0, p(y), P, p(wk), wk.numel(), None),
          L.nn_bias_act(p(y), p(bias), co, P, relu, None),
          L.nn_gemm_bf16(0, 1, co, K, P, 1.0, p(dy), P, p(col), P, 0.0, p(gw), K, p(wk), wk.numel(), None),
          L.nn_gemm_bf16(1, 0, K, P, co, 1.0, p(w), K, p(dy), P, 0.0, p(col), P, None, 0, None),
          L.nn_col2im3_add(p(col), ci, B, H, W, p(dx), None)]
    assert rc == [0] * 6
    return y, gw, dx


@pytest.mark.parametrize("relu,work,add,shift", [(1, 1 << 20, 0, 0), (0, 1, 1, 0), (1, 1 << 20, 1, 1)])
@pytest.mark.parametrize("ci,co,B,H,W", SHAPES)
def test_same_bits_as_im2col(ci, co, B, H, W, relu, work, add, shift):
    """shift: tensors that start 4 bytes past a 16-byte boundary."""
    import torch
    from paper_2203_01462_gb300.surrogate import _nn
    L = _nn()
    g = torch.Generator(device="cuda").manual_seed(ci * 1000 + co * 10 + W)

    def rnd(*shape):
        n = 1
        for v in shape:
            n *= v
        return torch.randn(n + shift, generator=g, device="cuda")[shift:].view(*shape)

    x, w, bias, dy, dx = rnd(ci, B, H, W), rnd(co, 9 * ci), rnd(co), rnd(co, B, H, W), rnd(ci, B, H, W)
    wk = torch.empty(work, device="cuda")
    y0, gw0, dx0 = _path(L, x, w, bias, dy, dx, relu, wk, add)
    y, gw = rnd(co, B, H, W), rnd(co, 9 * ci)
    p = lambda t: t.data_ptr()
    assert L.nn_conv3_fwd(p(x), p(w), p(bias), p(y), ci, co, B, H, W, relu, p(wk), work, None) == 0
    assert L.nn_conv3_wgrad(p(dy), p(x), p(gw), ci, co, B, H, W, p(wk), work, None) == 0
    assert L.nn_conv3_dgrad(p(dy), p(w), p(dx), ci, co, B, H, W, add, None) == 0
    torch.cuda.synchronize()
    assert torch.equal(y, y0)
    assert torch.equal(gw, gw0)
    assert torch.equal(dx, dx0)


def test_infinities_and_nan_stay_where_they_were():
    """A NaN and an infinity in the input reach the same outputs and weight
    gradients as through im2col (nothing outside the image or a slice is
    multiplied by them)."""
    import torch
    from paper_2203_01462_gb300.surrogate import _nn
    L = _nn()
    ci, co, B, H, W = 20, 24, 2, 24, 64
    g = torch.Generator(device="cuda").manual_seed(3)
    x, w, bias, dy, dx = (torch.randn(*s, generator=g, device="cuda")
                          for s in ((ci, B, H, W), (co, 9 * ci), (co,), (co, B, H, W), (ci, B, H, W)))
    x[7, 0, 5, 31], x[19, 1, 23, 63] = float("nan"), float("inf")
    wk = torch.empty(1 << 20, device="cuda")
    y0, gw0, _ = _path(L, x, w, bias, dy, dx, 0, wk, 0)
    y, gw = torch.empty_like(y0), torch.empty_like(gw0)
    p = lambda t: t.data_ptr()
    assert L.nn_conv3_fwd(p(x), p(w), p(bias), p(y), ci, co, B, H, W, 0, p(wk), wk.numel(), None) == 0
    assert L.nn_conv3_wgrad(p(dy), p(x), p(gw), ci, co, B, H, W, p(wk), wk.numel(), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(torch.nan_to_num(y, 7.0, 8.0, 9.0), torch.nan_to_num(y0, 7.0, 8.0, 9.0))
    assert torch.equal(torch.nan_to_num(gw, 7.0, 8.0, 9.0), torch.nan_to_num(gw0, 7.0, 8.0, 9.0))
