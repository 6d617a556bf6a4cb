"""Forms of a rollout that the other tests do not reach: samples in several pieces on
the tensor cores, workspaces that shrink on a full device, more FP32 controllers in a
batch than lanes, and a terrain without training points beside full ones."""
import numpy as np
import pytest

import oracle as O
import scenarios as S
from parity import TOL_COST, assert_close, check_trace, gpu_trace, make_ctrl, reconcile_costs, to_np
from test_gpu_batch_layouts import _both, _equal
from test_gpu_scratch import _Full

pytestmark = pytest.mark.gpu


def test_split_in_pieces(lib, monkeypatch):
    """2^23 queries are recorded at a time: 5 x 1.7 M samples take two pieces.  Every
    cost of the three-part format as the batched rollout gives it, which has none."""
    sc = S.scenario("small", K=1_700_001, T=5, N=20, precision=3)
    one, many, _ = _both(lib, sc, 2, monkeypatch)
    _equal(one, many)


def test_two_part_split_in_pieces(lib):
    sc = S.scenario("small", K=1_700_001, T=5, N=20, precision=2)
    _, ctrl = make_ctrl(lib, sc)
    rows = np.array([0, 1, 1_677_695, 1_677_696, 1_677_697, 1_677_721, 1_677_722, 1_700_000])
    x0 = sc.x0.astype(np.float32).astype(np.float64)
    tr = gpu_trace(lib, ctrl, sc, x0, sc.U0, it=3)
    ro = O.rollout(sc, O.gp_fit(sc.X, sc.Y, sc.hyper), x0, sc.U0, 3, samples=rows)
    check_trace(sc, ro, tr, rows)
    ref, _ = reconcile_costs(sc, ro, tr["costs"][rows], rows)
    assert_close(tr["costs"][rows], ref, TOL_COST, what="costs")


@pytest.mark.parametrize("precision,N", [(0, 300), (2, 300), (2, 900), (3, 100)])
def test_workspaces_on_a_full_device(lib, precision, N):
    """Smaller pieces of the samples and of the rows of v: the same bits."""
    import torch
    sc = S.scenario("small", K=20000, T=40, N=N, precision=precision)
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    out = [torch.empty_like(U), torch.empty(20000, device="cuda"), torch.empty(20000, device="cuda")]

    def step(ctrl):
        lib.mppi_set_iteration(ctrl, 1)
        lib.mppi_step(ctrl, sc.x0, U, *out)
        lib.mppi_device_status(ctrl)
        return [x.cpu().numpy() for x in out]

    g, ctrl = make_ctrl(lib, sc)
    want = step(ctrl)
    # 9 MB are the controls and costs; the least workspace is a few hundred KB
    for left in (28, 22, 18, 16):
        with _Full(left << 20):
            _, ctrl = make_ctrl(lib, sc, g)
            got = step(ctrl)
            del ctrl
        for a, b in zip(want, got):
            assert np.array_equal(a, b)


def test_more_fp32_controllers_than_lanes(lib):
    """Seven FP32 controllers and two on the tensor cores: each as on its own."""
    import torch
    specs = [(300, 7, 200, 0), (77, 5, 45, 0), (513, 9, 333, 0), (129, 4, 0, 0), (200, 8, 1030, 0), (64, 20, 90, 0),
             (40, 3, 15, 0), (100, 6, 100, 3), (90, 5, 800, 2)]
    scs = [S.scenario("small", K=K, T=T, N=N, O=3, precision=p, seed=20 + i) for i, (K, T, N, p) in enumerate(specs)]
    ctrls = [make_ctrl(lib, sc)[1] for sc in scs]
    b = lib.mppi_batch_create(ctrls)
    for i, sc in enumerate(scs):
        b.state[i].copy_(torch.tensor(sc.x0, dtype=torch.float32))
        b.U_nom[i].copy_(torch.tensor(sc.U0, dtype=torch.float32))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(2):
        lib.mppi_batch_graph(b, st)
    st.synchronize()
    many = [[to_np(x[i]) for x in (b.U_new, b.weights, b.costs)] for i in range(len(scs))]
    for i, sc in enumerate(scs):
        U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
        out = [torch.empty_like(U), torch.empty(sc.params.K, device="cuda"), torch.empty(sc.params.K, device="cuda")]
        lib.mppi_set_iteration(ctrls[i], 1)
        lib.mppi_step(ctrls[i], sc.x0.astype(np.float32), U, *out)
        for a, x in zip(many[i], out):
            assert np.array_equal(a, to_np(x)), i


@pytest.mark.parametrize("empty", [0, 1, 2])
@pytest.mark.parametrize("precision", [0, 2, 3])
def test_ensemble_with_an_empty_terrain(lib, precision, empty):
    sc = S.terrain_scenario("small", M=3, N=140, K=70, T=5, precision=precision)
    terrains = list(sc.terrains)
    terrains[empty] = (np.zeros((0, 4)), np.zeros((0, 2)), terrains[empty][2])
    sc = sc.replace(terrains=terrains)
    _, ctrl = make_ctrl(lib, sc)
    rows = np.arange(70)
    x0 = sc.x0.astype(np.float32).astype(np.float64)
    tr = gpu_trace(lib, ctrl, sc, x0, sc.U0, it=3)
    fits = O.Ensemble([O.gp_fit(*t) for t in sc.terrains], sc.terrain_w)
    ro = O.rollout(sc, fits, x0, sc.U0, 3, samples=rows)
    check_trace(sc, ro, tr, rows)
    ref, _ = reconcile_costs(sc, ro, tr["costs"][rows], rows)
    assert_close(tr["costs"][rows], ref, TOL_COST, what="costs")
