"""Host reads share one page-locked staging buffer, and none waits for work
queued on another object's stream: a read of a network's parameters leaves the
buffer to others while its own stream is busy, and does without it while a field
read holds it."""
import threading

import numpy as np
import pytest

from paper_2209_01444_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# 103,205 and 1,927,845 parameters: read through plain memory and through the buffer
@pytest.mark.parametrize("levels", [2, 4])
@pytest.mark.parametrize("busy", ["network", "fields"])
def test_a_busy_stream_holds_up_its_own_read_alone(busy, levels):
    import torch

    from paper_2209_01444_gb300 import lbm as L, surrogate as S

    case = W.single_seed_periodic(n=48, steps=1, R=6.0)
    sim = L.Simulation(case.params)
    sim.init_seeds(case.seeds, case.U0, case.theta0)
    net = S.UNet(2, 32, 32, levels=levels)
    vec = np.random.Generator(np.random.PCG64(1)).normal(size=net.param_count).astype(np.float32)
    net.set_params(vec)
    reads = {"network": lambda: np.concatenate([v.reshape(-1) for v in net.params().values()]),
             "fields": lambda: sim.fields(("phi",))["phi"]}
    other = "fields" if busy == "network" else "network"
    want = {k: f() for k, f in reads.items()}  # the buffer has its size now
    assert np.array_equal(want["network"], vec)
    s = torch.cuda.Stream()
    (net if busy == "network" else sim).set_stream(s)
    with torch.cuda.stream(s):
        torch.cuda._sleep(3_000_000_000)  # about 1.5 s
    got = {}
    t = threading.Thread(target=lambda: got.update({busy: reads[busy]()}))
    t.start()
    t.join(0.2)  # it waits for its stream by now
    got[other] = reads[other]()
    still_busy = not s.query()
    t.join()
    assert still_busy
    assert all(np.array_equal(got[k], want[k]) for k in want)
