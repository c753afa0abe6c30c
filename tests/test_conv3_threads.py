"""Input gradients of two networks from two host threads, each on its own
stream: a kernel's shared-memory limit is common to all its callers, and the
sizes that two widths need differ."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_widths_do_not_disturb_one_another():
    import torch
    from paper_2203_01462_gb300.surrogate import _nn
    L = _nn()
    ci, B, H, W, calls = 16, 1, 8, 32, 6000
    gen = torch.Generator(device="cuda").manual_seed(5)
    # integers: every sum is exact
    data = {co: [torch.randint(-4, 5, s, generator=gen, device="cuda").float()
                 for s in ((co, B, H, W), (co, 9 * ci))] for co in (8, 64)}
    out = {co: torch.zeros(ci, B, H, W, device="cuda") for co in data}
    bad = {}
    start = threading.Barrier(len(data))
    torch.cuda.synchronize()

    def work(co):
        dy, w = data[co]
        st = torch.cuda.Stream()
        a = (dy.data_ptr(), w.data_ptr(), out[co].data_ptr(), ci, co, B, H, W, 0, st.cuda_stream)
        start.wait()
        bad[co] = sum(L.nn_conv3_dgrad(*a) != 0 for _ in range(calls))
        st.synchronize()

    ts = [threading.Thread(target=work, args=(co,)) for co in data]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert bad == {8: 0, 64: 0}
    for co, (dy, w) in data.items():
        ref = torch.nn.grad.conv2d_input((B, ci, H, W), w.view(co, ci, 3, 3).double(), dy.transpose(0, 1).double(), padding=1)
        assert torch.equal(out[co].transpose(0, 1).double(), ref)
