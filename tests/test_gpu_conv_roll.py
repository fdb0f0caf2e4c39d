"""Convolutions that walk down the image with every weight tile on chip, and
convolutions of images whose rows fit no run of 128 pixels, at the edges of their
tiles.  Each output against an FP64 convolution of the same BF16 values: the
products are exact in FP32 and their sum is within 9 C rounding steps (2^-23 each,
truncation allowed for) of sum |x||w|, a BF16 result rounds by 2^-9 more."""
import numpy as np
import pytest

from oracle import unet_oracle as U
from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# runs that cross images and columns of tiles and end anywhere in one; images of one and two rows; 32 to 128 channels in, 32 and 64 out, ragged N
@pytest.mark.parametrize("B,H,width,C,N", [
    (1, 230, 256, 32, 32), (230, 1, 256, 32, 64), (120, 2, 256, 64, 32), (3, 100, 256, 64, 64), (2, 79, 384, 32, 40),
    (1, 300, 384, 64, 24), (1, 61, 1024, 32, 8), (4, 127, 128, 64, 56),
    (3, 100, 256, 128, 64), (2, 79, 384, 128, 40)])
@pytest.mark.parametrize("fp32", [0, 1])
def test_outputs_match_fp64(B, H, width, C, N, fp32):
    import torch

    from paper_2209_01444_gb300 import build_ext, lbm

    build_ext.build()
    lib = lbm.load()
    g = torch.Generator(device="cuda").manual_seed(H + C + N)
    X = torch.randn(B, H, width, C + 8, generator=g, device="cuda").bfloat16()
    Wm = (torch.randn(N, 9 * C, generator=g, device="cuda") / (3 * C ** 0.5)).bfloat16()
    bias = torch.randn(N, generator=g, device="cuda")
    D = torch.full((B, H, width, N + 8), 3.0, dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    for relu in (0, 1):
        assert lib.lbm_nn_conv3x3(X.data_ptr(), B, H, width, C, C + 8, Wm.data_ptr(), 9 * C, D.data_ptr(), N + 8,
                                  bias.data_ptr(), N, fp32, relu, torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert lib.lbm_nn_error(1) == 0
        x = X[..., :C].double().cpu().permute(0, 3, 1, 2)
        w = Wm.double().cpu().reshape(N, 3, 3, C).permute(0, 3, 1, 2)
        b = bias.double().cpu()
        conv = torch.nn.functional.conv2d
        want = conv(x, w, b, padding=1).permute(0, 2, 3, 1)
        size = conv(x.abs(), w.abs(), b.abs(), padding=1).permute(0, 2, 3, 1)
        if relu:
            want = want.clamp(min=0.0)
        got = D[..., :N].double().cpu()
        bound = 9 * C * 2.0 ** -23 * size + (0.0 if fp32 else 2.0 ** -8) * want.abs()
        assert bool(((got - want).abs() <= bound).all())
        assert bool((D[..., N:].float() == 3.0).all())


# tiles of 8 to 128 pixels a side over rows of 40, 136, 200 and 272, and the
# masked, FP32 and pooled-output gradients of wide rows (272, 256);
# gradients as in test_gpu_wgrad.py: 2e-3 at one level, 2e-2 at two
@pytest.mark.parametrize("levels,base,B,H,width,tol", [
    (1, 32, 2, 5, 40, 2e-3), (1, 64, 1, 3, 200, 2e-3), (2, 32, 1, 8, 144, 2e-2), (1, 32, 1, 160, 272, 2e-3),
    (2, 32, 1, 240, 256, 2e-2)])
def test_gradients_match_the_oracle(levels, base, B, H, width, tol):
    import torch

    from paper_2209_01444_gb300 import lbm, surrogate as S

    shapes = U.init_shapes(levels, base, 8, 5)
    params = W.unet_params(shapes, 3, out_scale=1.0)
    r = np.random.Generator(np.random.PCG64(9))
    x = W.bf16_exact(r.normal(size=(B, H, width, 5)))
    t = x + 0.1 * r.normal(size=x.shape)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()  # noqa: E731
    net = S.UNet(B, H, width, levels=levels, base=base)
    net.set_params(params)
    net.backward(dev(x), dev(t))
    g = net.grads()
    assert lbm.load().lbm_nn_error(1) == 0
    x8 = np.zeros(x.shape[:-1] + (8,))
    x8[..., :5] = x
    y, cache = U.forward(params, x8, levels, 5, q=U.bf16_round)
    want = U.backward(params, cache, U.mse(y, t)[1], levels, q=U.bf16_round)
    for name, _ in shapes:
        a, b = g[name].astype(np.float64), want[name]
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), name
