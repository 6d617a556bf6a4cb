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
