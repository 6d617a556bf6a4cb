"""The batched rollout's tile layouts (2, 4 and 8 threads a sample, scenes in and
out of shared memory, two- and three-part formats) against the single step and the
oracle.  The single step adds its sums in the batched rollout's order, and every cost,
weight and control is the same bits, but for training sets of up to 512 points in two
parts (and there too where the environment asks for the batched order)."""
import numpy as np
import pytest

import oracle as O
import scenarios as S
from parity import TOL_U, check_step, make_ctrl

pytestmark = pytest.mark.gpu


def _both(lib, sc, rps, monkeypatch, U=None, it=5):
    """(U_new, weights, costs) of mppi_step and of a batch of one, and the batch's layout."""
    import torch
    monkeypatch.setenv("GPMPPI_MMA_THREADS_PER_SAMPLE", str(rps))
    g, ctrl = make_ctrl(lib, sc)
    lib.mppi_set_iteration(ctrl, it)
    b = lib.mppi_batch_create([ctrl])
    x0 = torch.tensor(np.asarray(sc.x0), dtype=torch.float32)
    Ud = torch.tensor(np.asarray(sc.U0 if U is None else U), dtype=torch.float32, device="cuda")
    K = sc.params.K
    one = [torch.empty_like(Ud), torch.empty(K, device="cuda"), torch.empty(K, device="cuda")]
    lib.mppi_step(ctrl, x0.numpy(), Ud, *one)
    one = [x.cpu().numpy() for x in one]
    b.state[0].copy_(x0)
    b.U_nom[0].copy_(Ud)
    lib.mppi_batch_step(b)
    lib.mppi_device_status(ctrl)
    assert lib.mppi_batch_layout(b, 0)[0] == rps
    return one, [x.cpu().numpy() for x in (b.U_new[0], b.weights[0], b.costs[0])], (g, ctrl)


def _equal(one, many):
    for a, b in zip(one, many):
        assert np.all(np.isfinite(a)) and np.array_equal(a, b)


# training sets on both sides of the 64-column steps, of an odd and an even count of
# 128-column blocks and of the 256-column passes; ragged sample tiles
@pytest.mark.parametrize("rps", [2, 4, 8])
@pytest.mark.parametrize("precision,N", [(2, 1), (1, 65), (2, 129), (2, 333), (1, 512), (2, 513), (2, 640), (2, 641),
                                         (1, 768), (2, 769), (2, 897), (1, 1025), (2, 1200), (3, 1), (3, 65), (3, 129),
                                         (3, 333), (3, 1025)])
def test_step_and_batch_are_the_same_bits(lib, precision, N, rps, monkeypatch):
    monkeypatch.setenv("GPMPPI_NO_CLUSTER", "1")
    sc = S.scenario("small", K=301, T=5, N=N, O=5, precision=precision)
    one, many, _ = _both(lib, sc, rps, monkeypatch)
    _equal(one, many)


@pytest.mark.parametrize("precision,N", [(3, 150), (2, 90), (1, 300), (2, 800)])
def test_ensemble_step_and_batch_are_the_same_bits(lib, precision, N, monkeypatch):
    sc = S.terrain_scenario("small", M=2, N=N, K=213, T=4, precision=precision)
    one, many, _ = _both(lib, sc, 4, monkeypatch)
    _equal(one, many)


@pytest.mark.parametrize("precision,N", [(2, 2048), (3, 2048), (2, 700)])
def test_large_step_and_batch_are_the_same_bits(lib, precision, N, monkeypatch):
    """Every weight of a step whose queries fill the chip without a split of the passes."""
    sc = S.scenario("small", K=16384, T=30, N=N, O=20, path="eight", precision=precision)
    one, many, _ = _both(lib, sc, 2, monkeypatch)
    _equal(one, many)


@pytest.mark.parametrize("rps", [2, 4, 8])
@pytest.mark.parametrize("precision,N", [(2, 333), (1, 700)])
def test_batch_layouts_against_the_oracle(lib, precision, N, rps, monkeypatch):
    """The oracle's step, and the single step's within the two kernels' rounding."""
    sc = S.scenario("small", K=299, T=6, N=N, O=5, precision=precision)
    one, many, _ = _both(lib, sc, rps, monkeypatch)
    fits = O.gp_fit(sc.X, sc.Y, sc.hyper)
    x0 = sc.x0.astype(np.float32).astype(np.float64)
    check_step(sc, O.rollout(sc, fits, x0, sc.U0, 5), sc.U0, *(x.astype(np.float64) for x in many))
    np.testing.assert_allclose(one[2], many[2], rtol=1e-5, atol=1e-5)
    assert np.max(np.abs(one[0] - many[0])) <= TOL_U


@pytest.mark.parametrize("precision,N", [(2, 1900), (3, 1300)])
def test_batch_scene_in_global_memory(lib, precision, N, monkeypatch):
    """A scene that does not fit beside the ring: read from global memory, ragged samples."""
    sc = S.scenario("small", K=70, T=3, N=N, O=1500, precision=precision)
    t = np.linspace(0, 2 * np.pi, 6000)
    sc = sc.replace(path=np.stack([6 * np.cos(t), 3 * np.sin(t)], axis=1))
    one, many, _ = _both(lib, sc, 8, monkeypatch)
    _equal(one, many)
    fits = O.gp_fit(sc.X, sc.Y, sc.hyper)
    x0 = sc.x0.astype(np.float32).astype(np.float64)
    check_step(sc, O.rollout(sc, fits, x0, sc.U0, 5), sc.U0, *(x.astype(np.float64) for x in many))
