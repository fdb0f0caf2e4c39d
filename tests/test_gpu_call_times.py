"""Calls whose time follows from another call's of the same build: a kernel form
or a launch that suits one size can lose on another.  Each compares medians of the
two calls, queued in turn on the same stream, so that clocks and neighbours weigh on
both; the bounds lie between the ratio that the operation counts give and the one
the unsuitable form had."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _ratio(torch, a, b, reps=20, rounds=15):
    """Median over rounds of the time of `reps` queued calls of a over those of b."""
    out = []
    for _ in range(rounds):
        t = []
        for fn in (a, b):
            fn()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(reps):
                fn()
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        out.append(t[0] / t[1])
    return float(np.median(out))


@pytest.fixture(scope="module")
def env():
    import torch

    from paper_2209_01444_gb300 import lbm as L

    return torch, L.load()


# twice the fields, twice the products and sums: 1.9 to 2.1 as the kernel stands, 2.5
# and more where four pixels' loads beside the sums leave few warps resident
@pytest.mark.parametrize("P,C", [(4096, 8), (100003, 8), (1 << 20, 32)])
def test_projection_weight_gradients_of_six_fields(env, P, C):
    torch, lib = env
    X = torch.randn(P, C, device="cuda").bfloat16()
    part = torch.empty(1024 * 6 * (C + 1), device="cuda")

    def call(O):
        dY, W = torch.randn(P, O, device="cuda"), torch.randn(O, C, device="cuda")
        dW, db = torch.empty(O, C, device="cuda"), torch.empty(O, device="cuda")

        def fn():
            assert lib.lbm_nn_proj_bwd(dY.data_ptr(), X.data_ptr(), P, C, C, W.data_ptr(), O, None, C, dW.data_ptr(),
                                       db.data_ptr(), part.data_ptr(), 1024,
                                       torch.cuda.current_stream().cuda_stream) == 0
        return fn

    assert _ratio(torch, call(6), call(3)) < 2.3
