"""The failure-detection hook over a rollout of many waves of CTAs."""
import time

import numpy as np
import pytest

import scenarios as S
from parity import gpu_step, make_ctrl

pytestmark = pytest.mark.gpu


def test_expired_wait_costs_one_limit(lib):
    """1920 CTAs, two an SM: a step whose waits run out takes about one limit, not one
    for every wave of CTAs (seven); the next step is as before."""
    import torch
    sc = S.scenario("small", K=4096, T=20, N=300, precision=0)
    _, ctrl = make_ctrl(lib, sc)
    ref = gpu_step(lib, ctrl, sc, sc.x0, sc.U0, it=2)
    limit = 0.1
    lib.mppi_set_wait_limit(ctrl, int(limit * 1e9), expire_first=True)
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    Un = torch.empty_like(U)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    lib.mppi_step(ctrl, sc.x0, U, Un)
    torch.cuda.synchronize()
    took = time.perf_counter() - t0
    with pytest.raises(lib.GpmppiError) as ei:
        lib.mppi_device_status(ctrl)
    assert ei.value.code == lib.GPMPPI_ERR_TIMEOUT
    assert limit <= took < 3 * limit
    lib.mppi_set_wait_limit(ctrl, 2_000_000_000, expire_first=False)
    for a, b in zip(ref, gpu_step(lib, ctrl, sc, sc.x0, sc.U0, it=2)):
        assert np.array_equal(a, b)
