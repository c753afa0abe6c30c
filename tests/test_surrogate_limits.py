"""The surrogate's kernels at the ends of their integer ranges."""
import pytest


def _lib():
    from paper_2203_01462_gb300.surrogate import _nn
    return _nn()


@pytest.mark.gpu
def test_gemm_of_depth_one_with_the_most_columns():
    """N = 2^31 - 4: the last block reaches past the int range of columns.
    Products of small integers: exact."""
    import torch
    L = _lib()
    N = 2 ** 31 - 4
    if torch.cuda.mem_get_info()[0] < 5 * N * 4:
        pytest.skip("needs 40 GB of free device memory")
    guard = 1 << 16
    buf = torch.full((N + 2 * guard,), 7.0, device="cuda")  # C with untouched words on either side
    B = torch.arange(1 << 7, device="cuda", dtype=torch.float32).repeat(2 ** 24)[:N]
    A = torch.tensor([3.0], device="cuda")
    C = buf[guard:guard + N]
    assert L.nn_gemm_bf16(0, 0, 1, N, 1, 1.0, A.data_ptr(), 1, B.data_ptr(), N, 0.0, C.data_ptr(), N, None, 0, None) == 0
    torch.cuda.synchronize()
    assert bool((buf[:guard] == 7.0).all()) and bool((buf[guard + N:] == 7.0).all())
    step = 1 << 28
    for o in range(0, N, step):
        assert torch.equal(C[o:o + step], 3.0 * B[o:o + step])
