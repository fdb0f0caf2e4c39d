"""A bounded device wait that runs out, made to happen without a fault, in the
kernels that have an abort and drain path of their own: the convolution that walks
down the image, the weight gradient from the NHWC operands and the up-convolution's
weight gradient (both inside a network's backward pass).  With the operand-wait
bound at 0 the tensor-core issuer gives up its first wait; the kernel raises the
flag lbm_nn_error reports, drains its copies, frees its tensor memory and returns.
With the default bound back the same call gives the same bits as before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ETIMEOUT = -5


def _gives_up_and_recovers(torch, lib, call):
    torch.cuda.synchronize()
    assert lib.lbm_nn_error(1) == 0
    try:
        assert lib.lbm_nn_set_operand_wait(0) == 0
        call()
        torch.cuda.synchronize()
        assert lib.lbm_nn_error(1) == ETIMEOUT
    finally:
        assert lib.lbm_nn_set_operand_wait(1000000000) == 0
    call()
    torch.cuda.synchronize()
    assert lib.lbm_nn_error(1) == 0


# one and two channel blocks; four, two and one input rows a stage
@pytest.mark.parametrize("C,N", [(32, 32), (64, 64), (128, 64)])
def test_convolution_down_the_image(C, N):
    import torch

    from paper_2209_01444_gb300 import lbm

    lib = lbm.load()
    B, H, width = 3, 160, 256
    g = torch.Generator(device="cuda").manual_seed(C)
    X = torch.randn(B, H, width, C, generator=g, device="cuda").bfloat16()
    Wm = (torch.randn(N, 9 * C, generator=g, device="cuda") / (3 * C ** 0.5)).bfloat16()
    D = torch.full((B, H, width, N), 3.0, device="cuda")
    seen = []

    def call():
        D.fill_(3.0)
        assert lib.lbm_nn_conv3x3(X.data_ptr(), B, H, width, C, C, Wm.data_ptr(), 9 * C, D.data_ptr(), N, None, N, 1, 0,
                                  torch.cuda.current_stream().cuda_stream) == 0
        seen.append(D.clone())

    call()
    _gives_up_and_recovers(torch, lib, call)
    assert bool((seen[1] == 3.0).all())  # nothing was stored
    assert torch.equal(seen[0], seen[2])


# K blocks of 64 and 32 pixels, one and three vertical taps a CTA
@pytest.mark.parametrize("B,H,width", [(1, 16, 64), (2, 64, 512)])
def test_weight_gradients(B, H, width):
    import torch

    from paper_2209_01444_gb300 import lbm, surrogate as S

    g = torch.Generator(device="cuda").manual_seed(H)
    x = torch.randn(B, H, width, 5, generator=g, device="cuda")
    t = x + 0.1 * torch.randn(x.shape, generator=g, device="cuda")
    net = S.UNet(B, H, width, levels=2)
    r = np.random.Generator(np.random.PCG64(2))
    net.set_params(0.05 * r.normal(size=net.param_count).astype(np.float32))
    net.backward(x, t)
    want = net.grads()
    _gives_up_and_recovers(torch, lbm.load(), lambda: net.backward(x, t))
    got = net.grads()
    for name in want:
        assert np.array_equal(got[name], want[name]), name
