"""Weight gradients of 3 x 3 convolutions taken straight from the NHWC input
and output gradient, through networks of one and two levels, against the FP64
network oracle with the same BF16 rounding points.  Tolerances as for the
gradients of such networks elsewhere: 2e-3 of each tensor at one level, 2e-2 at
two (single rounding decisions differ); a tap, row or channel taken from the
wrong place is off by its whole size."""
import numpy as np
import pytest

from oracle import unet_oracle as U
from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# rows of 32, 64 and 96 or 160 pixels (K blocks of 32 and 64, one or several to
# a row), image edges in every block; 32 and 64 channels per block, one and
# several blocks (96, 256), the zero-padded first layer; few slices (one vertical
# tap per CTA) and many (three)
@pytest.mark.parametrize("levels,base,B,H,width,tol", [
    (1, 32, 1, 8, 32, 2e-3), (1, 32, 2, 4, 96, 2e-3), (1, 32, 1, 32, 512, 2e-3), (1, 64, 1, 8, 160, 2e-3),
    (1, 96, 1, 4, 64, 2e-3), (1, 256, 1, 16, 32, 2e-3), (2, 32, 1, 8, 64, 2e-2), (1, 32, 1, 8, 40, 2e-3)])
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
