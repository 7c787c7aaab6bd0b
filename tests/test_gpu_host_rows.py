"""Host buffers whose rows the TMA cannot take as they are (N no multiple of eight), pinned and not
(needs a B200): bit for bit what the device entry point gives."""
import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(130, 1, 1), (128, 3, 3), (257, 1031, 5), (300, 640, 63), (500, 700, 129), (128, 128, 8)])
def test_ragged_rows(M, K, N):
    import torch
    build.build_library()
    case = wl.Case(0, "rows", M, K, N, 40 + N, 0.5, "magnitude")
    W, X = case.make_W(), case.make_X()
    m = tl3.encode(W)
    m.upload()
    ld = (N + 7) // 8 * 8
    Xd = torch.zeros((K, ld), dtype=torch.float16, device="cuda")
    Xd[:, :N] = torch.from_numpy(X)
    want = m.spmm(Xd[:, :N]).cpu().numpy()
    ws = m.new_workspace(N)
    dX = torch.zeros(K * ld, dtype=torch.float16, device="cuda")
    dY = torch.empty(M * N, dtype=torch.float16, device="cuda")
    room = torch.empty(K * N + 16, dtype=torch.float16, pin_memory=True)
    for shift in (0, 1, 8, None):                           # pinned: on 16 bytes or not; None: pageable
        x = X.copy() if shift is None else room[shift:shift + K * N].view(K, N).numpy()
        x[:] = X
        Y = np.zeros((M, N), dtype=np.float16)
        dX.zero_()
        m.spmm_host(x, Y, dX, dY, ws)
        assert np.array_equal(Y.view(np.uint16), want.view(np.uint16)), shift
