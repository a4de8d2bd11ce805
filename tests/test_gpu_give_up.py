"""Tensor-core kernels whose waits run out: the products stop before a K step, as after a
wait that ran out, so every other role's waits run out too (after half a millisecond
here).  The call reports HR_ERR_TIMEOUT, every block has waited for its copies and products
under way and has given its tensor memory back: the next call, with the usual bounds, gives
the results of before, bit for bit."""
import ctypes

import pytest

from tests.gpu_common import require_gpu, torch

pytestmark = pytest.mark.gpu

CLOCKS, USUAL = 1 << 20, 1 << 31
# the first step; in the ring's first lap; in later laps of either parity; in a later tile
STOPS = [0, 2, 4, 7, 11, 19]


@pytest.fixture(scope="module")
def B_():
    require_gpu()
    from paper_2107_05509_gb300 import binding
    L = binding.lib()
    for f in (L.hr_internal_context_waits, L.hr_internal_net_waits):
        f.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int]
    return binding


@pytest.mark.parametrize("M,N,K,splits", [(300, 96, 1344, 1), (300, 96, 2688, 2), (2049, 2303, 1088, 1)])
def test_gemm_gives_up(B_, M, N, K, splits):
    """The 128-row kernel, with and without split sums, and the paired one (81 tiles: some
    pairs have a second)."""
    ctx = B_.Context(8, 8, 8, 1, 8, 8)
    gen = torch.Generator(device="cuda").manual_seed(M)
    a, b = (torch.randn((r, K), generator=gen, device="cuda").to(torch.bfloat16) for r in (M, N))
    buf = torch.empty((splits, M, N), device="cuda") if splits > 1 else None

    def product():
        out = torch.zeros((M, N), device="cuda")
        B_.hr_gemm_bf16(ctx, a, b, out, splits=splits, split_buf=buf)
        return out, B_.hr_get_status(ctx)

    ref, status = product()
    assert status == B_.HR_OK
    for stop in STOPS:
        B_.lib().hr_internal_context_waits(ctx.handle, CLOCKS, stop)
        assert product()[1] == B_.HR_ERR_TIMEOUT, stop
        B_.lib().hr_internal_context_waits(ctx.handle, USUAL, -1)
        out, status = product()
        assert status == B_.HR_OK and torch.equal(out, ref), stop


def test_network_gives_up(B_):
    """Convolutions, their input and weight gradients, and the dense layers' ones: a step
    that a kernel does not reach changes nothing there."""
    n, views = 40, 4
    net = B_.Net(n, views)
    gen = torch.Generator(device="cuda").manual_seed(1)
    net.set_params(0.05 * torch.randn(net.P, generator=gen, device="cuda"))
    net.set_inputs_bf16(torch.randn((n * views, 128, 128, 8), generator=gen, device="cuda").to(torch.bfloat16))
    cams, d_out = torch.rand((n * views, 20), generator=gen, device="cuda"), torch.randn((n, 61), generator=gen, device="cuda")

    def step(backward_only=False):
        out, g = torch.zeros((n, 61), device="cuda"), torch.zeros(net.P, device="cuda")
        if not backward_only:
            net.forward(cams, out)
        status = net.status()
        net.backward(d_out)
        net.get_params(grads=g)
        return out, g, status, net.status()

    out0, g0, *status = step()
    assert status == [B_.HR_OK] * 2
    for stop in STOPS:
        B_.lib().hr_internal_net_waits(net.handle, CLOCKS, stop)
        assert step(backward_only=True)[3] == B_.HR_ERR_TIMEOUT, stop
        assert step()[2:] == (B_.HR_ERR_TIMEOUT, B_.HR_ERR_TIMEOUT), stop
        B_.lib().hr_internal_net_waits(net.handle, USUAL, -1)
        out, g, *status = step()
        assert status == [B_.HR_OK] * 2 and torch.equal(out, out0) and torch.equal(g, g0), stop
