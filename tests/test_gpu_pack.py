"""Packing of fields into BF16 pixels: a thread per pixel below 32 channels, by
16-byte chunks from there on; every value is one subtraction, one product and one
rounding, so the results are those of the same operations in PyTorch, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


# one pixel, a block's 256 and one more, several blocks; all widths of both forms
@pytest.mark.parametrize("P", [1, 256, 257, 1000])
@pytest.mark.parametrize("F,pitch", [(1, 8), (5, 8), (8, 8), (5, 16), (8, 24), (5, 32), (8, 40), (3, 64)])
def test_packed_pixels(P, F, pitch):
    import torch

    from paper_2209_01444_gb300 import lbm

    g = torch.Generator(device="cuda").manual_seed(P + F)
    f = torch.randn(P, F, generator=g, device="cuda")
    mean, inv = torch.randn(8, generator=g, device="cuda"), torch.rand(8, generator=g, device="cuda") + 0.5
    X = torch.full((P + 1, pitch), 3.0, dtype=torch.bfloat16, device="cuda")
    assert lbm.load().lbm_nn_pack(f.data_ptr(), P, F, mean.data_ptr(), inv.data_ptr(), X.data_ptr(), pitch, None,
                                  torch.cuda.current_stream().cuda_stream) == 0
    want = torch.zeros(P, pitch, device="cuda")
    want[:, :F] = (f - mean[:F]) * inv[:F]
    assert torch.equal(X[:P], want.bfloat16())
    assert bool((X[P] == 3.0).all())
