"""Products of more than 64 columns (one launch over all of them) against the float64 product of the
masked W, within the tolerance of tests/test_gpu_spmm.py (needs a B200)."""
import numpy as np
import pytest

from paper_2607_08786_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tl3():
    import torch
    assert torch.cuda.is_available()
    from paper_2607_08786_b200 import build, tl3 as mod
    build.build_library()
    mod.lib()
    return mod


def _within(oracle_mod, W, X, Y):
    Yref, bound = oracle_mod.dense_fp64(W, X)
    err, tol = np.abs(Y.astype(np.float64) - Yref), oracle_mod.tolerance(bound)
    assert np.all(err <= tol), f"max err/tol {np.max(err / tol):.3f}"


# Column counts around the edges of a pass (one and two accumulators, one and two passes, a ragged last
# one), shapes with one tile, ragged tiles, many CTAs per row-tile and many row-tiles per CTA, blocks
# so large that fewer buffers fit (dense), every pitch of Y that 16-byte stores can not take, and up to
# 64 columns with many CTAs per row-tile.
@pytest.mark.parametrize("M,K,N,sparsity", [(128, 128, 65, 0.5), (7, 8, 80, 0.5), (300, 2000, 129, 0.6), (1000, 1096, 96, 0.4),
                                            (2048, 4096, 240, 0.5), (2048, 4096, 241, 0.5), (700, 3000, 256, 0.5),
                                            (9000, 640, 257, 0.5), (640, 9000, 300, 0.7), (512, 640, 512, 0.0), (20000, 256, 200, 0.5),
                                            (1024, 1024, 64, 0.5), (1024, 1024, 33, 0.5), (700, 6000, 24, 0.5), (1300, 1300, 32, 0.6)])
def test_wide_products(tl3, oracle_mod, M, K, N, sparsity):
    import torch
    case = wl.Case(0, "wide", M, K, N, 300 + N, sparsity, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.encode(W)
    m.upload()
    ws = m.new_workspace(N)
    Xd = torch.zeros((K, (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = torch.from_numpy(X)
    Xt = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xt[:, :K] = torch.from_numpy(np.ascontiguousarray(X.T))
    results = []
    for pitch in (N, (N + 7) // 8 * 8 + 8):
        buf = torch.full((M, pitch), float("nan"), dtype=torch.float16, device="cuda")
        m.spmm(Xd[:, :N], buf[:, :N], workspace=ws)
        torch.cuda.synchronize()
        assert m.status(ws) == tl3.OK and torch.isnan(buf[:, N:]).all()
        results.append(buf[:, :N].cpu().numpy())
    buf = torch.full((N + 1, M + 3), float("nan"), dtype=torch.float16, device="cuda")
    m.spmm_nt(Xt[:, :K], buf[:N, :M], workspace=ws)
    torch.cuda.synchronize()
    assert m.status(ws) == tl3.OK and torch.isnan(buf[N:]).all() and torch.isnan(buf[:, M:]).all()
    results.append(buf[:N, :M].T.cpu().numpy())
    _within(oracle_mod, W, X, results[0])
    for Y in results[1:]:                                   # same sums in the same order
        assert np.array_equal(Y.view(np.uint16), results[0].view(np.uint16))
    assert int(ws[:4096].sum()) == 0                        # status word and flags are left cleared


def _check_linear(W, Xt, bias, activation, Y, ctas):
    """Y (N x M) against act(Xt W^T + bias) in float64.  The sums are chains of 2 K / 32 MMA steps and then of
    up to `ctas` partial sums in fp32, each addition off by 2^-23 of what it may reach at most, the sum of the
    absolute products; the functions (slope at most 1.13) are off by a few ulp of fp32, which cancellation in
    1 + tanh leaves as 2^-20 of the argument; one rounding to fp16."""
    import torch
    X, D = Xt.double(), torch.from_numpy(W).cuda().double()
    sums = X @ D.T
    bound = X.abs() @ D.abs().T + (0 if bias is None else bias.double().abs())
    if bias is not None:
        sums = sums + bias.double()
    want = {None: lambda v: v, "relu": torch.relu, "silu": torch.nn.functional.silu,
            "gelu_tanh": lambda v: torch.nn.functional.gelu(v, approximate="tanh")}[activation](sums)
    tol = 1.13 * (W.shape[1] / 16 + ctas) * 2.0**-23 * bound + (2.0**-11 + 2.0**-18) * want.abs() + 2.0**-20 * sums.abs() + 2.0**-25
    err = (Y.double() - want).abs()
    assert bool((err <= tol).all()), float((err / tol).max())


@pytest.mark.parametrize("activation", [None, "relu", "silu", "gelu_tanh"])
def test_wide_bias_and_activation(tl3, activation):
    """Both layouts, one of them without an odd column."""
    import torch
    case = wl.Case(0, "wide_act", 1100, 1500, 150, 9, 0.5, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.encode(W)
    m.upload()
    bias = torch.linspace(-0.5, 0.5, 1100, device="cuda").half()
    Xt = torch.zeros((150, 1504), dtype=torch.float16, device="cuda")
    Xt[:, :1500] = torch.from_numpy(np.ascontiguousarray(X.T))
    Y = m.spmm_nt(Xt[:, :1500], bias=bias, activation=activation)
    Z = m.spmm(Xt[:144, :1500].T.contiguous(), bias=bias, activation=activation)
    _check_linear(W, Xt[:, :1500], bias, activation, Y, 9)
    _check_linear(W, Xt[:144, :1500], bias, activation, Z.T, 9)


# Every kind of pass there is beside those of the cases above (which are all for a CTA alone, but for two):
# pairs of CTAs with one and two accumulators, an even and an odd number of row-tiles, row-tiles of their own
# and shared by three pairs, blocks of every size (at 0 % sparsity the rings shrink).  The plan is asserted,
# so that another estimate of the passes cannot leave one of them without a case.
@pytest.mark.parametrize("M,K,N,sparsity,columns,cluster,accumulators", [
    (4300, 1500, 512, 0.5, 256, 2, 1), (4200, 1500, 511, 0.4, 256, 2, 1), (4300, 1530, 512, 0.0, 256, 2, 1),
    (7500, 128, 1000, 0.5, 256, 2, 1), (7000, 2000, 129, 0.5, 160, 2, 2), (6900, 2048, 129, 0.0, 160, 2, 2),
    (6200, 250, 450, 0.4, 160, 2, 2), (20000, 256, 200, 0.4, 224, 2, 2), (1024, 1024, 128, 0.4, 64, 1, 2), (12000, 1000, 128, 0.0, 128, 1, 2)])
def test_every_kind_of_pass(tl3, M, K, N, sparsity, columns, cluster, accumulators):
    import torch
    case = wl.Case(0, "plan", M, K, N, 500 + N, sparsity, "bernoulli")
    W, X = case.make_W(), case.make_X()
    m = tl3.Matrix.encode_on_device(torch.from_numpy(W).cuda(), device_only=True)
    m.upload_packed_on_device()
    ws = m.new_workspace(N)
    Xt = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xt[:, :K] = torch.from_numpy(np.ascontiguousarray(X.T))
    Xd = torch.zeros((K, (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = Xt[:, :K].T
    bias = torch.linspace(-0.5, 0.5, M, device="cuda").half()
    for b, activation in ((None, None), (bias, None), (bias, "gelu_tanh")):
        Y = m.spmm(Xd[:, :N], workspace=ws, bias=b, activation=activation)
        assert m.last_pass() == {"columns": columns, "cluster": cluster, "accumulators": accumulators}
        Yt = m.spmm_nt(Xt[:, :K], workspace=ws, bias=b, activation=activation)
        assert m.last_pass() == {"columns": columns, "cluster": cluster, "accumulators": accumulators}
        _check_linear(W, Xt[:, :K], b, activation, Yt, 9)
        assert torch.equal(Y.T.view(torch.int16), Yt.view(torch.int16))       # same sums in the same order
    assert m.status(ws) == tl3.OK and int(ws[:4096].sum()) == 0


@pytest.mark.parametrize("room", [64, 300])
@pytest.mark.parametrize("way", ["plain", "graph", "streams"])
def test_both_kernels_take_turns_without_a_wait(tl3, way, room):
    """Products of 16 to 300 columns of two matrices, straight after one another on one workspace (made for
    `room` columns): the same bits as one at a time.  Launches overlap the end of the one before, and the
    kernels lay out flags and partial sums differently."""
    import torch
    cases = [wl.Case(0, "turns", 1024, 5120, 300, 1, 0.5, "magnitude"), wl.Case(0, "turns", 9000, 640, 300, 2, 0.4, "bernoulli")]
    matrices = []
    for c in cases:
        m = tl3.Matrix.encode_on_device(torch.from_numpy(c.make_W()).cuda(), device_only=True)
        m.upload_packed_on_device()
        matrices.append((m, torch.from_numpy(c.make_X()).cuda()))
    calls = []                                                     # (matrix, X, bias, activation, Y)
    for N in (16, 300, 64, 128, 16, 257, 8, 300, 24, 72):
        for m, X in matrices:
            x = torch.zeros((X.shape[0], (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
            x[:, :N] = X[:, :N]
            b = torch.linspace(-1, 1, m.shape[0], device="cuda").half() if N % 3 else None
            calls.append((m, x[:, :N], b, "relu" if N == 64 else None, torch.empty((m.shape[0], N), dtype=torch.float16, device="cuda")))

    def run(ws):
        for m, x, b, act, y in calls:
            m.spmm(x, y, workspace=ws, bias=b, activation=act)

    ws = matrices[0][0].new_workspace(room)
    want = []
    for m, x, b, act, y in calls:
        m.spmm(x, y, workspace=ws, bias=b, activation=act)
        torch.cuda.synchronize()
        want.append(y.clone())
        y.fill_(float("nan"))
    spaces = [ws]
    torch.cuda.synchronize()
    if way == "plain":
        for _ in range(20):
            run(ws)
    elif way == "graph":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(ws)
        for _ in range(20):
            graph.replay()
    else:                                                          # forked over streams, each with a workspace and outputs of its own
        streams = [torch.cuda.Stream() for _ in range(3)]
        spaces = [matrices[0][0].new_workspace(room) for _ in streams]
        torch.cuda.synchronize()
        outs = [[torch.full_like(c[4], float("nan")) for c in calls] for _ in streams]
        torch.cuda.synchronize()
        for _ in range(5):
            for i, (m, x, b, act, _y) in enumerate(calls):
                for s, space, out in zip(streams, spaces, outs):
                    m.spmm(x, out[i], workspace=space, stream=s, bias=b, activation=act)
        torch.cuda.synchronize()
        for out in outs[1:]:
            for a, b in zip(out, want):
                assert torch.equal(a.view(torch.int16), b.view(torch.int16))
        for c, o in zip(calls, outs[0]):
            c[4].copy_(o)
    torch.cuda.synchronize()
    for c, w in zip(calls, want):
        assert torch.equal(c[4].view(torch.int16), w.view(torch.int16)), tuple(c[4].shape)
    for space in spaces:
        assert matrices[0][0].status(space) == tl3.OK and int(space[:4096].sum()) == 0


def test_a_workspace_for_fewer_columns_still_serves_wide_products(tl3):
    """One that was made for 64 columns; more of them in test_gpu_workspace.py."""
    import torch
    case = wl.Case(0, "wide_ws", 900, 700, 300, 10, 0.5, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.encode(W)
    m.upload()
    Xd = torch.zeros((700, 304), dtype=torch.float16, device="cuda")
    Xd[:, :300] = torch.from_numpy(X)
    ws = m.new_workspace(64)
    Y = m.spmm(Xd[:, :300], workspace=ws)
    Xt = torch.zeros((300, 704), dtype=torch.float16, device="cuda")
    Xt[:, :700] = Xd[:, :300].T
    Yt = m.spmm_nt(Xt[:, :700], workspace=ws)
    want = m.spmm(Xd[:, :300])
    for got in (Y, Yt.T):                                   # other split of K: fp32 sums in another order, one rounding
        assert (got - want).abs().max() <= 2.0**-9 * want.abs().max()
    assert m.status(ws) == tl3.OK


@pytest.mark.parametrize("M,K,others", [(4608, 1024, 4), (4600, 1000, 4), (4096, 768, 4), (4096, 1024, 4), (4608, 4096, 4), (4096, 4096, 5), (3584, 2048, 5), (3328, 2048, 6),
                                        (1024, 1024, 7), (5120, 5120, 4)])
@pytest.mark.parametrize("N", [33, 64])
def test_where_the_kernels_meet(tl3, M, K, others, N):
    """With four stages at 64 columns and 50 % sparsity, four partial sums besides the reducer's own fit
    them: then the product stays with the other kernel (four stages), from five on it comes here."""
    import torch
    tiles_m, tiles_k = -(-M // 128), -(-K // 128)
    T = tiles_m * tiles_k
    G = min(T, torch.cuda.get_device_properties(0).multi_processor_count)
    owner = [((t + 1) * G - 1) // T for t in range(T)]
    assert max(owner[(r + 1) * tiles_k - 1] - owner[r * tiles_k] for r in range(tiles_m)) == others
    case = wl.Case(0, "meet", M, K, N, 5, 0.5, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.Matrix.encode_on_device(torch.from_numpy(W).cuda(), device_only=True)
    m.upload_packed_on_device()
    Xt = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xt[:, :K] = torch.from_numpy(np.ascontiguousarray(X.T))
    Xd = torch.zeros((K, 64), dtype=torch.float16, device="cuda")
    Xd[:, :N] = Xt[:, :K].T
    Y = m.spmm(Xd[:, :N])
    assert (m.last_launch()["stages"] == 4) == (others <= 4), m.last_launch()
    Yt = m.spmm_nt(Xt[:, :K])
    _check_linear(W, Xt[:, :K], None, None, Yt, 9)
    _check_linear(W, Xt[:, :K], None, None, Y.T, 9)
