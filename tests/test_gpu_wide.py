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


@pytest.mark.parametrize("activation", [None, "relu", "silu", "gelu_tanh"])
def test_wide_bias_and_activation(tl3, activation):
    """Against the same expression in float64, within 2^-10 relative (one rounding to fp16 and the
    fp32 sums) plus 2e-3 of the sums' scale for sums that cancel."""
    import torch
    case = wl.Case(0, "wide_act", 1100, 1500, 150, 9, 0.5, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.encode(W)
    m.upload()
    bias = torch.linspace(-0.5, 0.5, 1100, device="cuda").half()
    Xt = torch.zeros((150, 1504), dtype=torch.float16, device="cuda")
    Xt[:, :1500] = torch.from_numpy(np.ascontiguousarray(X.T))
    ref = Xt[:, :1500].double() @ torch.from_numpy(W).cuda().double().T
    bound = Xt[:, :1500].double().abs() @ torch.from_numpy(W).cuda().double().abs().T
    ref = ref + bias.double()
    ref = {None: lambda v: v, "relu": torch.relu, "silu": torch.nn.functional.silu,
           "gelu_tanh": lambda v: torch.nn.functional.gelu(v, approximate="tanh")}[activation](ref)
    Y = m.spmm_nt(Xt[:, :1500], bias=bias, activation=activation).double()
    Z = m.spmm(Xt[:144, :1500].T.contiguous(), bias=bias, activation=activation).double()
    for got, want in ((Y, ref), (Z.T, ref[:144])):
        assert ((got - want).abs() <= 2.0**-10 * want.abs() + 2e-3 * bound[:len(want)]).all()


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
