"""The surrogate's small passes at sizes where their vector forms begin and
end: resampling, bias gradient with ReLU, Adam on several tensors."""
import pytest

pytestmark = pytest.mark.gpu


def _lib():
    from paper_2203_01462_gb300.surrogate import _nn
    return _nn()


def _p(t):
    return t.data_ptr()


@pytest.mark.parametrize("shift", [0, 1])  # planes that start 4 bytes past an aligned address
@pytest.mark.parametrize("n,h,w", [(1, 1, 1), (3, 5, 3), (2, 3, 2), (5, 7, 6), (24, 64, 128), (1, 1, 1024)])
def test_resampling(n, h, w, shift):
    """Sums of four and one product by 0.25 in the order written: exact."""
    import torch
    L = _lib()
    g = torch.Generator(device="cuda").manual_seed(n + h + w)

    def rnd(*s):
        m = s[0] * s[1] * s[2]
        return torch.randn(m + shift, generator=g, device="cuda")[shift:].view(*s)

    def four(a):
        return a[:, 0::2, 0::2] + a[:, 0::2, 1::2] + a[:, 1::2, 0::2] + a[:, 1::2, 1::2]

    def up(a):
        return a.repeat_interleave(2, 1).repeat_interleave(2, 2)

    fine, coarse = rnd(n, 2 * h, 2 * w), rnd(n, h, w)
    out_c, out_f = rnd(n, h, w), rnd(n, 2 * h, 2 * w)
    ref_cb, ref_fb = out_c + four(fine), out_f + 0.25 * up(coarse)
    acc_c, acc_f = out_c.clone() if not shift else out_c, out_f.clone() if not shift else out_f
    assert L.nn_up2_bwd_add(_p(fine), n, h, w, _p(acc_c), None) == 0
    assert L.nn_pool2_bwd_add(_p(coarse), n, 2 * h, 2 * w, _p(acc_f), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(acc_c, ref_cb) and torch.equal(acc_f, ref_fb)
    assert L.nn_pool2(_p(fine), n, 2 * h, 2 * w, _p(acc_c), None) == 0
    assert L.nn_up2(_p(coarse), n, h, w, _p(acc_f), None) == 0
    torch.cuda.synchronize()
    assert torch.equal(acc_c, 0.25 * four(fine)) and torch.equal(acc_f, up(coarse))


@pytest.mark.parametrize("relu", [0, 1])
@pytest.mark.parametrize("co,P", [(1, 32764), (3, 32768), (2, 32772), (5, 131070), (24, 200 * 136 * 5)])
def test_bias_gradient(co, P, relu):
    """The mask is exact; the sum is within its FP32 accumulation bound
    (each term in a chain of fewer than P / 1024 + 14 additions)."""
    import torch
    L = _lib()
    g = torch.Generator(device="cuda").manual_seed(P)
    y, dy = torch.randn(co, P, generator=g, device="cuda"), torch.randn(co, P, generator=g, device="cuda")
    y[0, :3] = torch.tensor([0.0, float("nan"), -0.0])
    ref = torch.where(y > 0, dy, torch.zeros_like(dy)) if relu else dy.clone()
    db = torch.full((co,), 7.0, device="cuda")
    assert L.nn_act_bwd_bias(_p(y), _p(dy), _p(db), co, P, relu, None) == 0
    torch.cuda.synchronize()
    assert torch.equal(dy, ref)
    bound = (P / 1024 + 14) * 2.0 ** -24 * ref.abs().double().sum(1)
    assert bool(((db.double() - ref.double().sum(1)).abs() <= bound).all())


@pytest.mark.parametrize("count", [1, 2, 64, 65])
def test_adam_on_several_tensors_is_adam_on_each(count):
    import torch
    import ctypes as C
    L = _lib()
    g = torch.Generator(device="cuda").manual_seed(count)
    sizes = [(1, 1023, 1024, 1025, 40000)[i % 5] for i in range(count)]
    one = [[torch.rand(n, generator=g, device="cuda") for n in sizes] for _ in range(4)]  # p, g, m, v
    many = [[t.clone() for t in ts] for ts in one]
    for p, gr, m, v in zip(*one):
        assert L.nn_adam(_p(p), _p(gr), _p(m), _p(v), p.numel(), 1e-3, 0.9, 0.999, 1e-8, 3, None) == 0
    arr = [(C.c_void_p * count)(*[t.data_ptr() for t in ts]) for ts in many]
    assert L.nn_adam_multi(count, *arr, (C.c_longlong * count)(*sizes), 1e-3, 0.9, 0.999, 1e-8, 3, None) == 0
    torch.cuda.synchronize()
    for a, b in zip(one, many):
        assert all(torch.equal(s, t) for s, t in zip(a, b))
    arr[2][count - 1] = None  # a missing moment buffer is refused before anything is launched
    assert L.nn_adam_multi(count, *arr, (C.c_longlong * count)(*sizes), 1e-3, 0.9, 0.999, 1e-8, 3, None) == 1


@pytest.mark.parametrize("ta", [0, 1])
@pytest.mark.parametrize("M,N,beta,shift", [(1, 4, 0.0, 0), (8, 1024, 1.0, 0), (9, 1028, 0.5, 0), (24, 4096, 1.0, 0),
                                            (24, 4095, 1.0, 0), (5, 64, 1.0, 1)])
def test_gemm_bf16_of_depth_one(ta, M, N, beta, shift):
    """One product per entry, exact in FP32; alpha = 1, and beta C + product
    rounded once or twice: one unit in the last place of the larger term.
    shift: operands that start 4 bytes past an aligned address."""
    import torch
    L = _lib()
    g = torch.Generator(device="cuda").manual_seed(M * N)
    A = torch.randn(M, generator=g, device="cuda")
    B = torch.randn(N + shift, generator=g, device="cuda")[shift:]
    Cm = torch.randn(M * N + shift, generator=g, device="cuda")[shift:].view(M, N)
    prod = A.bfloat16().double()[:, None] * B.bfloat16().double()[None]
    ref = prod + beta * Cm.double()
    bound = 2.0 ** -23 * (prod.abs() + (beta * Cm.double()).abs())
    assert L.nn_gemm_bf16(ta, 0, M, N, 1, 1.0, _p(A), M if ta else 1, _p(B), N, beta, _p(Cm), N, None, 0, None) == 0
    torch.cuda.synchronize()
    assert bool(((Cm.double() - ref).abs() <= bound).all())
