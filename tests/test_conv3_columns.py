"""3 x 3 convolutions given scratch for the im2col matrix: the same results as
the im2col path (nn_im2col3 + nn_gemm_bf16 + ...), bit for bit, whichever of the
two forms a layer takes, and the convolutions where the scratch is too small."""
import ctypes as C

import pytest

from test_conv3 import _path

pytestmark = pytest.mark.gpu

SHAPES = [  # ci, co, B, H, W, scratch wanted
    (24, 24, 1, 16, 24, False),
    (40, 96, 2, 9, 13, True),    # narrow rows: input gradient only
    (96, 96, 4, 50, 50, True),   # rows that leave no 16-byte groups, forward too
    (96, 192, 1, 32, 32, True),  # whole groups, a deep input gradient
    (64, 384, 2, 7, 7, True),    # depth in K slices
    (96, 96, 8, 64, 64, False),
]


def _lib():
    from paper_2203_01462_gb300.surrogate import _nn
    return _nn()


@pytest.mark.parametrize("ci,co,B,H,W,wanted", SHAPES)
def test_against_im2col(ci, co, B, H, W, wanted):
    import torch
    L = _lib()
    n = C.c_longlong(-1)
    assert L.nn_conv3_col_elems(ci, co, B, H, W, C.byref(n)) == 0
    assert n.value == (9 * ci * B * H * W if wanted else 0)
    gen = torch.Generator(device="cuda").manual_seed(ci * co + W)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda")
    x, w, bias, dy, dx0 = rnd(ci, B, H, W), rnd(co, 9 * ci), rnd(co), rnd(co, B, H, W), rnd(ci, B, H, W)
    wk = torch.zeros(1 << 20, device="cuda")
    p = lambda t: t.data_ptr()
    y_ref, _, _ = _path(L, x, w, bias, dy, dx0, 1, wk, 0)
    for add in (0, 1):
        # the input gradient's GEMM with the scratch of K slices that the call has
        col = torch.empty(9 * ci * B * H * W, device="cuda")
        ref = dx0.clone() if add else torch.zeros_like(dx0)
        P, K = B * H * W, 9 * ci
        assert L.nn_gemm_bf16(1, 0, K, P, co, 1.0, p(w), K, p(dy), P, 0.0, p(col), P, p(wk) if wanted else None,
                              wk.numel() if wanted else 0, None) == 0
        assert L.nn_col2im3_add(p(col), ci, B, H, W, p(ref), None) == 0
        y, dx = torch.zeros_like(y_ref), dx0.clone()
        assert L.nn_conv3_fwd_col(p(x), p(w), p(bias), p(y), ci, co, B, H, W, 1, p(wk), wk.numel(), p(col), n.value, None) == 0
        assert L.nn_conv3_dgrad_col(p(dy), p(w), p(dx), ci, co, B, H, W, add, p(wk), wk.numel(), p(col), n.value, None) == 0
        torch.cuda.synchronize()
        assert torch.equal(y, y_ref)
        assert torch.equal(dx, ref)


def test_too_little_scratch():
    """One word short, or none: the convolutions, whose scratch stays untouched."""
    import torch
    L = _lib()
    ci, co, B, H, W = 96, 96, 4, 50, 50
    gen = torch.Generator(device="cuda").manual_seed(3)
    x, w, dy = (torch.randn(*s, generator=gen, device="cuda") for s in ((ci, B, H, W), (co, 9 * ci), (co, B, H, W)))
    bias, wk = torch.zeros(co, device="cuda"), torch.zeros(1 << 20, device="cuda")
    p = lambda t: t.data_ptr()
    n = 9 * ci * B * H * W - 1
    col = torch.full((n,), 7.0, device="cuda")
    out = []
    for c, k in ((p(col), n), (None, 0)):
        y, dx = torch.zeros(co, B, H, W, device="cuda"), torch.zeros(ci, B, H, W, device="cuda")
        assert L.nn_conv3_fwd_col(p(x), p(w), p(bias), p(y), ci, co, B, H, W, 0, p(wk), wk.numel(), c, k, None) == 0
        assert L.nn_conv3_dgrad_col(p(dy), p(w), p(dx), ci, co, B, H, W, 0, p(wk), wk.numel(), c, k, None) == 0
        out.append((y, dx))
    y, dx = torch.zeros(co, B, H, W, device="cuda"), torch.zeros(ci, B, H, W, device="cuda")
    assert L.nn_conv3_fwd(p(x), p(w), p(bias), p(y), ci, co, B, H, W, 0, p(wk), wk.numel(), None) == 0
    assert L.nn_conv3_dgrad(p(dy), p(w), p(dx), ci, co, B, H, W, 0, None) == 0
    torch.cuda.synchronize()
    assert bool((col == 7.0).all())
    for a in out:
        assert torch.equal(a[0], y) and torch.equal(a[1], dx)
