"""A workspace made for fewer columns than the product has (needs a B200): every entry point stays inside
it and gives the same product as with one made for that many columns."""
import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3, workloads as wl

pytestmark = pytest.mark.gpu


# Passes of 128 columns or fewer, pairs of CTAs (n_pad 160, 224, 256) with row-tiles shared by several of
# them, an odd number of row-tiles, N beyond one and beyond two passes.
@pytest.mark.parametrize("M,K,N,sparsity", [(900, 700, 300, 0.5), (9000, 640, 257, 0.5), (7001, 2003, 200, 0.6), (12800, 640, 230, 0.4),
                                            (5120, 2048, 512, 0.5), (6400, 700, 777, 0.5)])
def test_workspace_for_64_columns(oracle_mod, M, K, N, sparsity):
    import torch
    build.build_library()
    case = wl.Case(0, "ws", M, K, N, 70 + N, sparsity, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.Matrix.encode_on_device(torch.from_numpy(W).cuda(), device_only=True)
    m.upload_packed_on_device()
    full, small = m.workspace_bytes(N), m.workspace_bytes(64)
    assert full > small
    # all of a full workspace's bytes are there, the last of them as a guard
    room = torch.full((full,), 0xA5, dtype=torch.uint8, device="cuda")
    assert tl3.lib().tl3_workspace_init(room.data_ptr(), small, None) == tl3.OK
    ws = room[:small]
    ld = (N + 7) // 8 * 8
    Xd = torch.zeros((K, ld), dtype=torch.float16, device="cuda")
    Xd[:, :N] = torch.from_numpy(X)
    Xt = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xt[:, :K] = Xd[:, :N].T
    dX, dY = torch.zeros(K * ld, dtype=torch.float16, device="cuda"), torch.empty(M * N, dtype=torch.float16, device="cuda")
    host, later = np.zeros((M, N), dtype=np.float16), np.zeros((M, N), dtype=np.float16)
    Y = m.spmm(Xd[:, :N], workspace=ws)
    Yt = m.spmm_nt(Xt[:, :K], workspace=ws)
    m.spmm_host(X, host, dX, dY, ws)
    m.spmm_host_async(X, later, dX, dY, ws)
    torch.cuda.synchronize()
    assert m.status(ws) == tl3.OK
    assert bool((room[small:] == 0xA5).all())                 # nothing was stored beyond the workspace
    assert int(ws[:4096].sum()) == 0                          # status word and flags are left cleared
    # the fp32 sums of the float64 product, rounded once: from any split of K
    Yref, bound = oracle_mod.dense_fp64(W, X)
    got = Y.cpu().numpy()
    assert np.all(np.abs(got.astype(np.float64) - Yref) <= oracle_mod.tolerance(bound))
    for other in (Yt.T.cpu().numpy(), host, later):
        assert np.array_equal(other.view(np.uint16), got.view(np.uint16))


def test_workspace_that_was_only_zeroed():
    """Zeroed memory without tl3_workspace_init() counts as the smallest that serves any N."""
    import torch
    build.build_library()
    case = wl.Case(0, "ws", 9000, 640, 257, 3, 0.5, "magnitude")
    m = tl3.Matrix.encode_on_device(torch.from_numpy(case.make_W()).cuda(), device_only=True)
    m.upload_packed_on_device()
    X = torch.zeros((640, 264), dtype=torch.float16, device="cuda")
    X[:, :257] = torch.from_numpy(case.make_X())
    ws = torch.zeros(m.workspace_bytes(257), dtype=torch.uint8, device="cuda")
    Y, want = m.spmm(X[:, :257], workspace=ws), m.spmm(X[:, :257])
    assert m.status(ws) == tl3.OK
    assert (Y - want).abs().max() <= 2.0**-9 * want.abs().max()   # sums in another order, one rounding
