"""Host buffers in both directions, pinned and not, on 16 bytes or not, of sizes around a thread's 16 bytes,
a block's 4096 and the largest that a kernel copies (needs a B200): bit for bit the device entry point."""
import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(1, 8, 8), (129, 16, 8), (256, 256, 8), (257, 264, 8), (255, 130, 16), (8192, 128, 64), (8193, 128, 64), (130, 8200, 64), (1000, 60, 5), (1536, 1536, 64), (1537, 1544, 64),
                                   # Y ends within a thread's 16 bytes: 2, 14, 18, 50010 bytes, two short of 192 KB and of a megabyte, two more than 192 KB
                                   (1, 8, 1), (7, 8, 1), (9, 16, 1), (5001, 300, 5), (98303, 8, 1), (524287, 8, 1), (98305, 8, 1)])
@pytest.mark.parametrize("x_shift,y_shift", [(0, 0), (8, 8), (1, 0), (0, 1), (None, 0), (0, None)])      # None: pageable
def test_host_copies(M, K, N, x_shift, y_shift):
    import torch
    build.build_library()
    case = wl.Case(0, "copies", M, K, N, 60 + N, 0.5, "magnitude")
    X = case.make_X()
    m = tl3.encode(case.make_W())
    m.upload()
    ld = (N + 7) // 8 * 8
    Xd = torch.zeros((K, ld), dtype=torch.float16, device="cuda")
    Xd[:, :N] = torch.from_numpy(X)
    want = m.spmm(Xd[:, :N]).cpu().numpy()
    ws = m.new_workspace(N)
    dX = torch.zeros(K * ld, dtype=torch.float16, device="cuda")
    dY = torch.empty(M * N, dtype=torch.float16, device="cuda")

    def buffer(rows, cols, shift):
        room = torch.full((rows * cols + 16,), 7.0, dtype=torch.float16, pin_memory=shift is not None)
        return room, room.numpy()[(shift or 0):(shift or 0) + rows * cols].reshape(rows, cols)

    (x_room, x), (y_room, y) = buffer(K, N, x_shift), buffer(M, N, y_shift)
    x[:] = X
    for _ in range(3):                                      # one after another on the same buffers
        y[:] = 0
        m.spmm_host(x, y, dX, dY, ws)
        assert np.array_equal(y.view(np.uint16), want.view(np.uint16))
    before = y_shift or 0
    assert bool((y_room[:before] == 7).all()) and bool((y_room[before + M * N:] == 7).all())
    # two products behind each other on one stream, with the same device buffers
    y2_room, y2 = buffer(M, N, y_shift)
    y[:] = 0
    m.spmm_host_async(x, y, dX, dY, ws)
    m.spmm_host_async(x, y2, dX, dY, ws)
    torch.cuda.synchronize()
    assert np.array_equal(y.view(np.uint16), want.view(np.uint16)) and np.array_equal(y2.view(np.uint16), want.view(np.uint16))


@pytest.mark.parametrize("N", [8, 5])
def test_device_scratch_that_is_too_small_is_refused(N):
    """Pinned X goes to dX by a kernel: only where dX holds it.  Otherwise the runtime's copy gets the call, and refuses."""
    import ctypes
    import torch
    build.build_library()
    case = wl.Case(0, "small", 256, 4096, N, 5, 0.5, "magnitude")
    m = tl3.encode(case.make_W())
    m.upload()
    X = torch.from_numpy(case.make_X()).pin_memory()
    Y = torch.full((256, N), 7.0, dtype=torch.float16, pin_memory=True)
    dY, ws = torch.empty(256 * N, dtype=torch.float16, device="cuda"), m.new_workspace(N)
    cu, d = ctypes.CDLL("libcuda.so.1"), ctypes.c_uint64()
    assert cu.cuMemAlloc_v2(ctypes.byref(d), ctypes.c_size_t(4096)) == 0              # of 65536 bytes
    try:
        stream = torch.cuda.current_stream().cuda_stream
        rc = tl3.lib().tl3_spmm_host(m._h, X.data_ptr(), Y.data_ptr(), N, d.value, dY.data_ptr(), ws.data_ptr(), stream)
        assert rc == tl3.ERR_CUDA and tl3.lib().tl3_last_cuda_error() == 1             # cudaErrorInvalidValue
        torch.cuda.synchronize()
        assert bool((Y == 7).all())
    finally:
        assert cu.cuMemFree_v2(d) == 0
    dX = torch.zeros(4096 * 8, dtype=torch.float16, device="cuda")
    m.spmm_host(X.numpy(), Y.numpy(), dX, dY, ws)
    Xd = torch.zeros((4096, 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = X.cuda()
    assert torch.equal(Y, m.spmm(Xd[:, :N]).cpu())


def test_blocking_calls_from_several_threads():
    """Beside another blocking call large copies go another way than alone: the same bits."""
    import threading
    import torch
    build.build_library()
    case = wl.Case(0, "threads", 2048, 2048, 64, 9, 0.5, "magnitude")
    X = case.make_X()
    m = tl3.encode(case.make_W())
    m.upload()
    want = m.spmm(torch.from_numpy(X).cuda()).cpu()
    calls = []
    for _ in range(4):
        calls.append((torch.from_numpy(X).pin_memory(), torch.zeros((2048, 64), dtype=torch.float16, pin_memory=True),
                      torch.empty(2048 * 64, dtype=torch.float16, device="cuda"), torch.empty(2048 * 64, dtype=torch.float16, device="cuda"),
                      m.new_workspace(64), torch.cuda.Stream()))
    torch.cuda.synchronize()
    wrong, errors = [], []

    def work(x, y, dX, dY, ws, stream):
        try:
            for _ in range(20):
                y.zero_()
                m.spmm_host(x.numpy(), y.numpy(), dX, dY, ws, stream)
                wrong.append(not torch.equal(y, want))
        except Exception as e:                                  # reported below, in the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=c) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors and len(wrong) == 80 and not any(wrong)
