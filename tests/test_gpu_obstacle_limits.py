"""Scenes of more obstacles than the stage costs' default shared memory holds."""
import threading

import numpy as np
import pytest

import oracle as O
import scenarios as S
from parity import TOL_COST, assert_close, check_trace, gpu_trace, make_ctrl, reconcile_costs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("obstacles", [1013, 1014, 4096])
def test_many_obstacles(lib, obstacles, precision):
    """Around 48 KB (1013 obstacles) and at the limit."""
    sc = S.scenario("small", K=70, T=3, N=40, O=obstacles, precision=precision)
    _, ctrl = make_ctrl(lib, sc)
    tr = gpu_trace(lib, ctrl, sc, sc.x0, sc.U0, it=1)
    x0 = sc.x0.astype(np.float32).astype(np.float64)
    ro = O.rollout(sc, O.gp_fit(sc.X, sc.Y, sc.hyper), x0, sc.U0, 1)
    check_trace(sc, ro, tr)
    ref, _ = reconcile_costs(sc, ro, tr["costs"], np.arange(70))
    assert_close(tr["costs"], ref, TOL_COST, what="costs")


def test_threads_with_different_scenes(lib):
    """Two host threads step controllers of 1100 and of 4096 obstacles at the same
    time: neither launch sees the other's shared-memory limit."""
    import torch
    made = []
    for o in (1100, 4096):
        sc = S.scenario("small", K=32, T=2, N=10, O=o, precision=0)
        made.append((sc, make_ctrl(lib, sc)[1]))
    errors = []

    def steps(sc, ctrl):
        try:
            st = torch.cuda.Stream()
            U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
            Un = torch.empty_like(U)
            torch.cuda.current_stream().synchronize()
            for _ in range(3000):
                lib.mppi_step(ctrl, sc.x0, U, Un, stream=st)
            st.synchronize()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    ts = [threading.Thread(target=steps, args=m) for m in made]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
