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


# calls queued one behind the other take less than a call alone with its launch
# (0.75 as it stands) and 1.1 to 1.2 where the CTAs of kernels that wait for their turn lie on few SMs
def test_projections_queued_one_behind_the_other(env):
    torch, lib = env
    P, C, O = 100003, 256, 8
    X, Wt = torch.randn(P, C, device="cuda").bfloat16(), torch.randn(O, C, device="cuda")
    bias, Y = torch.randn(O, device="cuda"), torch.empty(P, O, device="cuda")

    def fn():
        assert lib.lbm_nn_proj_fwd(X.data_ptr(), P, C, C, Wt.data_ptr(), bias.data_ptr(), O, None, Y.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream) == 0

    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def time(reps):
        torch.cuda.synchronize()
        e[0].record()
        for _ in range(reps):
            fn()
        e[1].record()
        torch.cuda.synchronize()
        return e[0].elapsed_time(e[1]) / reps

    time(20)
    queued, alone = (float(np.median([time(n) for _ in range(25)])) for n in (30, 1))
    assert queued < 0.95 * alone


# a second flow step in the same launch costs less than the first, which takes the
# wall passes and the frozen fields' pass with it; 3.0 where the wall pass's CTAs were
# resident before the step had finished, on the few SMs that it left free
@pytest.mark.parametrize("walls", [("noslip", "noslip", "periodic", "periodic"),
                                   ("inflow", "outflow", "symmetry", "symmetry")])
@pytest.mark.parametrize("nx", [4, 32])
def test_two_flow_steps_of_a_long_strip(env, nx, walls):
    from paper_2209_01444_gb300 import lbm as L, workloads as W

    torch, _ = env
    p = W.thermosolutal_params(nx, 8000, bc=walls, u_in=(0.5, 0.0))
    sim = L.Simulation(p, stream=torch.cuda.current_stream())
    sim.init_seeds(np.array([[0.5 * nx, 4000.0, 1.0, 0.0]]), 0.0, -0.55)
    assert _ratio(torch, lambda: sim.step_flow(2), lambda: sim.step_flow(1)) < 2.0


# fourteen flow steps of a long strip in one call cost no more than one by one, wall
# pass and frozen fields' pass each time; 2 to 4 where they run in regions of which the
# strip fills a small part
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_flow_steps_of_a_long_strip(env, storage):
    from paper_2209_01444_gb300 import lbm as L, workloads as W

    torch, _ = env
    p = W.thermosolutal_params(262140, 4)
    sim = L.Simulation(p, storage, stream=torch.cuda.current_stream())
    sim.init_seeds(np.array([[1000.0, 2.0, 1.0, 0.0]]), 0.0, -0.55)
    one = lambda: [sim.step_flow(1) for _ in range(14)]  # noqa: E731
    assert _ratio(torch, lambda: sim.step_flow(14), one, reps=5) < 1.15


# a quarter of the channels written, two thirds of the bytes in all left out: 0.45 of
# the time, 0.65 where 8 channels went through shared memory by chunks as 32 do
def test_packing_few_channels(env):
    torch, lib = env
    P, F = 4000000, 5
    f = torch.randn(P, F, device="cuda")
    mean, inv = torch.zeros(8, device="cuda"), torch.ones(8, device="cuda")

    def call(pitch):
        X = torch.empty(P, pitch, dtype=torch.bfloat16, device="cuda")

        def fn():
            assert lib.lbm_nn_pack(f.data_ptr(), P, F, mean.data_ptr(), inv.data_ptr(), X.data_ptr(), pitch, None,
                                   torch.cuda.current_stream().cuda_stream) == 0
        return fn

    assert _ratio(torch, call(8), call(32)) < 0.55


# two images of as many pixels and tiles, whose columns of tiles end at the ends of
# CTAs' runs (two columns) and within them (three): 1.0, and 1.2 where the
# column-walking kernel took the second on three tiles per SM as well
@pytest.mark.parametrize("C,N", [(64, 64), (128, 64)])
def test_convolutions_of_three_columns(env, C, N):
    torch, lib = env
    W = torch.randn(N, 9 * C, device="cuda").bfloat16()

    def call(H, width):
        X = torch.randn(H, width, C, device="cuda").bfloat16()
        D = torch.empty(H, width, N, dtype=torch.bfloat16, device="cuda")

        def fn():
            assert lib.lbm_nn_conv3x3(X.data_ptr(), 1, H, width, C, C, W.data_ptr(), 9 * C, D.data_ptr(), N, None, N, 0,
                                      1, torch.cuda.current_stream().cuda_stream) == 0
        return fn

    assert _ratio(torch, call(160, 384), call(240, 256)) < 1.09


# coupled steps with three flow steps each, replayed from a graph on a small grid: 2.2
# times the step with one, 3.5 where the two more went through a region's load and store
def test_small_grid_with_two_time_scales(env):
    from paper_2209_01444_gb300 import lbm as L, workloads as W

    torch, _ = env
    sims = []
    for n_sub in (3, 1):
        sim = L.Simulation(W.thermosolutal_params(48, 48, n_sub=n_sub), stream=torch.cuda.current_stream())
        sim.init_seeds(np.array([[24.0, 24.0, 6.0, 0.0]]), 0.0, -0.55)
        sims.append(sim)
    assert _ratio(torch, lambda: sims[0].step(32), lambda: sims[1].step(32), reps=5) < 2.9
