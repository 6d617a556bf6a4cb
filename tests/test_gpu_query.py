"""The query rollout (mean chain, variances of all queries, stage costs) at the
edges of its tiles, against the FP64 oracle with the trajectory tolerances of
parity.py: training sets around the 128-column blocks and 32-point chunks,
query counts around the 32- and 128-query tiles, sample counts on both sides
of the samples-per-warp rule, and a rollout taken in several pieces."""
import numpy as np
import pytest

import oracle as O
import scenarios as S
from parity import TOL_COST, assert_close, check_trace, gpu_trace, make_ctrl, reconcile_costs

pytestmark = pytest.mark.gpu


def _check_rows(lib, sc, rows, it=3):
    g, ctrl = make_ctrl(lib, sc)
    x0 = sc.x0.astype(np.float32).astype(np.float64)
    tr = gpu_trace(lib, ctrl, sc, x0, sc.U0, it=it)
    fits = O.Ensemble([O.gp_fit(*t) for t in sc.terrains], sc.terrain_w) if sc.terrains else O.gp_fit(sc.X, sc.Y, sc.hyper)
    ro = O.rollout(sc, fits, x0, sc.U0, it, samples=rows)
    check_trace(sc, ro, tr, rows)
    ref, _ = reconcile_costs(sc, ro, tr["costs"][rows], rows)
    assert_close(tr["costs"][rows], ref, TOL_COST, what="costs")


def _rows(K, n=24):
    rng = np.random.default_rng(K)
    r = {0, K - 1, K // 2} | set(rng.integers(0, K, n).tolist())
    return np.array(sorted(r))


@pytest.mark.parametrize("K,T,N", [
    (33, 3, 1), (64, 17, 2), (31, 33, 31), (129, 5, 33), (300, 16, 127), (300, 15, 128), (257, 16, 129),
    (1799, 4, 255), (1800, 4, 257), (3601, 3, 300), (500, 9, 1023), (70, 20, 1025), (40, 6, 4096)])
def test_fp32_tile_edges(lib, K, T, N):
    _check_rows(lib, S.scenario("small", K=K, T=T, N=N, precision=0), _rows(K))


def test_fp32_in_pieces(lib):
    # 2^23 queries are recorded at a time: 5 x 1.7 M samples take two pieces
    sc = S.scenario("small", K=1_700_001, T=5, N=3, precision=0)
    _check_rows(lib, sc, np.array([0, 1, 1_677_720, 1_677_721, 1_677_722, 1_700_000]))


@pytest.mark.parametrize("precision", [1, 2, 3])
@pytest.mark.parametrize("K,T,N", [
    (33, 3, 1), (64, 4, 63), (64, 4, 64), (65, 4, 65), (31, 33, 129), (300, 5, 255), (257, 4, 256), (129, 5, 257),
    (200, 4, 449), (1, 1, 513), (90, 3, 769), (260, 2, 1025)])
def test_split_tile_edges(lib, K, T, N, precision):
    """The tensor-core variances: training sets around the 64-column steps of the
    diagonal, the 256-column passes and the 32- and 64-point stages, query counts
    around the 256 queries of a CTA pair, one pass or several split over the pairs."""
    _check_rows(lib, S.scenario("small", K=K, T=T, N=N, precision=precision), _rows(K))


@pytest.mark.parametrize("N", [1, 31, 127, 128, 129, 300, 1025])
@pytest.mark.parametrize("M", [1, 127, 129])
def test_predict_tile_edges(lib, N, M):
    """gp_predict around the 128-query tiles and the 128-column blocks: the mean
    and variance of the FP64 posterior, within the rounding of their FP32 sums
    (N eps times the sums of magnitudes)."""
    import torch
    sc = S.scenario("small", K=33, T=2, N=N, precision=0)
    g, _ = make_ctrl(lib, sc)
    rng = np.random.default_rng(N * 1000 + M)
    Z = (rng.random((M, 4)) * [2.0, 3.0, 2.0, 3.0] - [0.0, 1.5, 0.0, 1.5]).astype(np.float32)
    mean = torch.empty(M, 2, device="cuda")
    var = torch.empty(M, 2, device="cuda")
    lib.gp_predict(g, torch.tensor(Z, device="cuda"), mean, var)
    torch.cuda.synchronize()
    eps = 2.0 ** -23
    for o in range(2):
        h = sc.hyper[o]
        d = (Z[:, None].astype(np.float64) - sc.X[None]) / np.asarray(h.lengthscale)
        k = h.signal_var * np.exp(-0.5 * (d * d).sum(-1))
        Linv, alpha = lib.gp_factors(g, o)
        Linv = np.asarray(Linv).reshape(N, N)
        v = k @ Linv.T
        # a kernel value is good to a few eps times its exponent's magnitude
        rel = (8.0 + 2.0 * np.max((d * d).sum(-1))) * eps
        tol_m = (rel + np.sqrt(N) * eps) * (np.abs(k) @ np.abs(np.asarray(alpha))) + eps
        tol_v = 2.0 * (np.abs(v) * ((rel + np.sqrt(N) * eps) * (np.abs(k) @ np.abs(Linv).T))).sum(1) + 8 * eps * h.signal_var
        assert np.all(np.abs(mean[:, o].cpu().numpy() - k @ np.asarray(alpha)) <= tol_m)
        assert np.all(np.abs(var[:, o].cpu().numpy() - np.maximum(0.0, h.signal_var - (v * v).sum(1))) <= tol_v)


def test_gradient_ragged_samples(lib):
    """The adjoint over a sample count that is no multiple of its eight-row padding
    and a training set past one block, against the FP64 central differences."""
    sc = S.scenario("small", K=45, T=6, N=150, precision=0)
    h = sc.hyper[0]
    sc = sc.replace(hyper=(h, S.Hyper(tuple(h.lengthscale), h.signal_var, h.noise_var)))
    import torch
    _, ctrl = make_ctrl(lib, sc)
    J, dU, dl = lib.mppi_grad(ctrl, sc.x0, torch.tensor(sc.U0, dtype=torch.float32, device="cuda"), 20.0, None,
                              want_dl=True)
    torch.cuda.synchronize()
    x0, U = sc.x0.astype(np.float32).astype(np.float64), sc.U0.astype(np.float32).astype(np.float64)
    Jo, _ = O.objective(sc, sc.hyper, x0, U, 0, None, 20.0)
    gU, gL = O.fd_gradient(sc, sc.hyper, x0, U, 0, None, 20.0)
    assert abs(float(J.cpu().numpy()[0]) - Jo) <= 1e-4 * abs(Jo)
    for got, ref in ((dU, gU), (dl, gL)):
        got, ref = got.cpu().numpy().ravel().astype(np.float64), np.asarray(ref).ravel()
        floor = 1e-3 * np.max(np.abs(ref))
        assert np.max(np.abs(got - ref) / np.maximum(np.abs(ref), floor)) <= 1e-3


@pytest.mark.parametrize("precision", [0, 2])
def test_prediction_and_step_under_capture(lib, precision):
    """gp_predict, as the first call on a fitted GP, and mppi_step may be captured
    into a CUDA graph: the replay gives what the direct calls give, bit for bit."""
    import torch
    sc = S.scenario("small", K=70, T=5, N=130, precision=precision)
    g, ctrl = make_ctrl(lib, sc)
    x0 = sc.x0.astype(np.float32)
    Z = torch.rand(150, 4, device="cuda")
    U = torch.tensor(sc.U0.astype(np.float32), device="cuda")
    bufs = [torch.zeros(n, device="cuda") for n in (300, 300, U.numel(), 70, 70)]
    mean, var, Un, w, costs = (b.view(-1, 2) if i < 3 else b for i, b in enumerate(bufs))

    def calls(stream):
        lib.gp_predict(g, Z, mean, var, stream=stream)
        lib.mppi_set_iteration(ctrl, 4)
        lib.mppi_step(ctrl, x0, U, Un, w, costs, stream=stream)

    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        calls(s)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    replayed = [b.cpu().numpy().copy() for b in bufs]
    for b in bufs:
        b.zero_()
    calls(None)
    torch.cuda.synchronize()
    for a, b in zip(replayed, bufs):
        assert a.any() and np.array_equal(a, b.cpu().numpy())
