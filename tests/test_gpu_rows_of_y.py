"""Rows of Y that 16-byte stores fit, rows that are turned in shared memory first and rows that are stored as
they are, at up to 64 columns and with half a step of the wider kernel at the end (needs a B200): every pitch gives the same bits, nothing beyond the columns is touched, and the values are
those of the float64 product within the tolerance of tests/test_gpu_spmm.py."""
import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 5, 8, 15, 17, 24, 31, 33, 40, 56, 63, 64, 72, 136])
@pytest.mark.parametrize("M,K", [(1100, 500), (130, 1300)])
def test_every_pitch(oracle_mod, M, K, N):
    import torch
    build.build_library()
    case = wl.Case(0, "pitch", M, K, N, 60 + N, 0.5, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.encode(W)
    m.upload()
    Xd = torch.zeros((K, (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = torch.from_numpy(X)
    results = []
    for pitch, shift in ((N, 0), (N + 1, 0), ((N + 7) // 8 * 8 + 8, 0), ((N + 7) // 8 * 8 + 8, 1)):
        room = torch.full((M * pitch + shift,), float("nan"), dtype=torch.float16, device="cuda")
        buf = room[shift:].view(M, pitch)
        m.spmm(Xd[:, :N], buf[:, :N])
        torch.cuda.synchronize()
        assert torch.isnan(buf[:, N:]).all() and torch.isnan(room[:shift]).all()
        results.append(buf[:, :N].cpu().numpy())
    Yref, bound = oracle_mod.dense_fp64(W, X)
    assert np.all(np.abs(results[0].astype(np.float64) - Yref) <= oracle_mod.tolerance(bound))
    for Y in results[1:]:
        assert np.array_equal(Y.view(np.uint16), results[0].view(np.uint16))
