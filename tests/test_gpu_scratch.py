"""Scratch that is made by a first call or shrinks on a full device: the results do
not depend on it, and what a first call prepared lets later ones be captured."""
import ctypes

import numpy as np
import pytest

import scenarios as S
from parity import make_ctrl

pytestmark = pytest.mark.gpu


class _Full:
    """All but `left` bytes of the device held by one allocation."""

    def __init__(self, left):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        for more in range(0, 256 << 20, 2 << 20):
            try:
                self.hold = torch.empty(max(0, free - left - more), dtype=torch.uint8, device="cuda")
                return
            except torch.cuda.OutOfMemoryError:
                pass

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        import torch
        del self.hold
        torch.cuda.empty_cache()


def _grad(lib, ctrl, sc, want_dl=True):
    import torch
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    out = lib.mppi_grad(ctrl, sc.x0, U, 20.0, None, want_dl=want_dl)
    return [x.cpu().numpy() for x in out if x is not None]


@pytest.mark.parametrize("K,T,N,left", [
    (4001, 40, 500, 300 << 20),       # 0.7 GB of rows: one piece, and a few with a ragged last one
    (6001, 60, 1000, 500 << 20)])     # 3 GB: one piece, and more than four
def test_gradient_on_a_full_device(lib, K, T, N, left):
    """Fewer samples at a time: J and dU are per-sample terms added in the samples'
    order, the same bits; the lengthscales' Gram sums are FP32 sums of thousands of
    products in another grouping (1e-4 of the largest)."""
    sc = S.scenario("small", K=K, T=T, N=N, precision=0)
    _, ctrl = make_ctrl(lib, sc)
    free = _grad(lib, ctrl, sc)
    _, ctrl = make_ctrl(lib, sc)
    with _Full(left):
        full = _grad(lib, ctrl, sc)
        again = _grad(lib, ctrl, sc)
    assert all(np.all(np.isfinite(x)) for x in free)
    assert np.array_equal(free[0], full[0]) and np.array_equal(free[1], full[1])
    assert np.max(np.abs(free[2] - full[2])) <= 1e-4 * np.max(np.abs(free[2]))
    assert all(np.array_equal(a, b) for a, b in zip(full, again))


def test_gradient_after_a_cost_may_be_captured(lib):
    """A first call for J alone makes what a call for dU needs."""
    import torch
    sc = S.scenario("small", K=70, T=5, N=130, precision=0)
    _, ctrl = make_ctrl(lib, sc)
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    J, dU = torch.zeros(1, device="cuda"), torch.zeros(5, 2, device="cuda")
    lib.mppi_grad(ctrl, sc.x0, U, 20.0, None, J, want_dU=False)
    s = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        lib.mppi_grad(ctrl, sc.x0, U, 20.0, None, J, dU, want_dl=False, stream=s)
    J.zero_()
    graph.replay()
    torch.cuda.synchronize()
    ref = _grad(lib, ctrl, sc, want_dl=False)
    assert np.array_equal(J.cpu().numpy(), ref[0]) and np.array_equal(dU.cpu().numpy(), ref[1]) and ref[1].any()


@pytest.mark.parametrize("K,T,N", [(4096, 50, 500), (16384, 100, 300)])
def test_memory_of_an_fp32_controller(lib, K, T, N):
    """256 MB of rows of v at most, whatever K and T, beside 36 bytes of records and
    the 8 of the perturbed control for every query (and 2 MB granules)."""
    import torch
    sc = S.scenario("small", K=K, T=T, N=N, precision=0)
    g, _ = make_ctrl(lib, S.scenario("small", K=33, T=2, N=N, precision=0))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    _, ctrl = make_ctrl(lib, sc, g)
    assert before - torch.cuda.mem_get_info()[0] <= (256 << 20) + 44 * K * T + (32 << 20)


@pytest.mark.parametrize("shared", [True, False])
@pytest.mark.parametrize("N", [0, 1, 127, 130, 1025])
def test_prediction_in_a_graph_instantiated_twice(lib, N, shared):
    """A captured gp_predict is kernels alone, so that its graph may be instantiated
    as often as one likes: both replays give the direct call's bits."""
    import torch
    cu = ctypes.CDLL("libcuda.so.1")
    sc = S.scenario("small", K=33, T=2, N=N, precision=0)
    h = sc.hyper[0]
    other = h if shared else S.Hyper(tuple(1.3 * x for x in h.lengthscale), 0.7 * h.signal_var, h.noise_var)
    g = lib.gp_fit(sc.X, sc.Y, (h, S.Hyper(tuple(other.lengthscale), other.signal_var, other.noise_var)))
    Z = torch.rand(300, 4, device="cuda") * 2.0
    mean, var = torch.zeros(300, 2, device="cuda"), torch.zeros(300, 2, device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = ctypes.c_void_p(st.cuda_stream)
    graph, execs = ctypes.c_void_p(), [ctypes.c_void_p(), ctypes.c_void_p()]
    assert cu.cuStreamBeginCapture_v2(s, 0) == 0
    lib.gp_predict(g, Z, mean, var, stream=st)
    assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
    for e in execs:
        assert cu.cuGraphInstantiateWithFlags(ctypes.byref(e), graph, ctypes.c_ulonglong(0)) == 0
    got = []
    for e in execs:
        mean.zero_()
        var.zero_()
        torch.cuda.synchronize()
        assert cu.cuGraphLaunch(e, s) == 0
        st.synchronize()
        got.append((mean.cpu().numpy(), var.cpu().numpy()))
    for e in execs:
        cu.cuGraphExecDestroy(e)
    cu.cuGraphDestroy(graph)
    lib.gp_predict(g, Z, mean, var)
    torch.cuda.synchronize()
    for m, v in got:
        assert np.array_equal(m, mean.cpu().numpy()) and np.array_equal(v, var.cpu().numpy()) and v.any()


def test_prediction_on_a_full_device(lib):
    """Smaller pieces, down to no scratch at all: the same bits."""
    import torch
    sc = S.scenario("small", K=33, T=2, N=1025, precision=0)
    g = lib.gp_fit(sc.X, sc.Y, sc.hyper)
    Z = torch.rand(60000, 4, device="cuda") * 2.0
    mean, var = torch.zeros(60000, 2, device="cuda"), torch.zeros(60000, 2, device="cuda")
    small = [torch.zeros(200, 2, device="cuda") for _ in range(2)]
    lib.gp_predict(g, Z, mean, var)
    torch.cuda.synchronize()
    want = mean.cpu().numpy(), var.cpu().numpy()
    del g                                 # (what its predictions left in the pool goes with it)
    g2 = lib.gp_fit(sc.X, sc.Y, sc.hyper)
    for left in (100 << 20, 2 << 20):
        mean.zero_()
        var.zero_()
        with _Full(left):
            lib.gp_predict(g2, Z, mean, var)
            lib.gp_predict(g2, Z[:200], *small)
            torch.cuda.synchronize()
        assert np.array_equal(mean.cpu().numpy(), want[0]) and np.array_equal(var.cpu().numpy(), want[1])
        assert np.array_equal(small[1].cpu().numpy(), want[1][:200])


def test_a_failed_allocation_ends_with_its_call(lib):
    """A controller that does not fit is OOM; the calls after it are not."""
    import torch
    sc = S.scenario("small", K=60, T=4, N=70, precision=0)
    big = S.scenario("small", K=1 << 20, T=64, N=70, precision=0)
    g, ctrl = make_ctrl(lib, sc)
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    want, got = torch.empty_like(U), torch.empty_like(U)
    lib.mppi_step(ctrl, sc.x0, U, want)
    with _Full(64 << 20):
        with pytest.raises(lib.GpmppiError) as ei:
            make_ctrl(lib, big, g)
        assert ei.value.code == lib.GPMPPI_ERR_OOM
        g2, ctrl = make_ctrl(lib, sc)
        lib.mppi_step(ctrl, sc.x0, U, got)
        torch.cuda.synchronize()
    assert torch.equal(got, want)


@pytest.mark.parametrize("precision,terrains", [(2, 1), (3, 1), (3, 2)])
def test_batch_after_a_failed_one(lib, precision, terrains):
    """A batch whose factor tiles do not fit is OOM, whichever of them fails; made again
    with room it steps as the controller does on its own."""
    import torch
    N = 1500
    if terrains == 1:
        sc = S.scenario("small", K=70, T=3, N=N, precision=precision)
    else:
        sc = S.terrain_scenario("small", M=terrains, N=N, K=70, T=3, precision=precision)
    _, ctrl = make_ctrl(lib, sc)
    U = torch.tensor(sc.U0, dtype=torch.float32, device="cuda")
    want, w, c = torch.empty_like(U), torch.empty(70, device="cuda"), torch.empty(70, device="cuda")
    failed = 0
    for left in (2, 6, 10, 14, 18, 24):           # a part is 5 MB, of the stacked factor 18
        with _Full(left << 20):
            try:
                b = lib.mppi_batch_create([ctrl])
                del b
            except lib.GpmppiError as e:
                assert e.code == lib.GPMPPI_ERR_OOM
                failed += 1
    assert failed >= 2
    lib.mppi_set_iteration(ctrl, 4)
    b = lib.mppi_batch_create([ctrl])
    b.state[0].copy_(torch.tensor(sc.x0, dtype=torch.float32))
    b.U_nom[0].copy_(U)
    lib.mppi_step(ctrl, sc.x0.astype(np.float32), U, want, w, c)
    lib.mppi_batch_step(b)
    torch.cuda.synchronize()
    assert torch.equal(b.U_new[0], want) and torch.equal(b.weights[0], w) and want.any()
