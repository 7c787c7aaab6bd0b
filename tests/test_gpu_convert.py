"""Edges of the conversion kernels on the GPU: byte equality with the host library (needs a B200)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tl3():
    import torch
    assert torch.cuda.is_available()
    from paper_2607_08786_b200 import build, tl3 as mod
    build.build_library()
    mod.lib()
    return mod


def _runs(M, K, run):
    """Full and empty windows in runs of `run`: every boundary costs a dummy byte, so that a tile has
    close to the largest possible number of pairs and more than 4096 code bytes."""
    rng = np.random.default_rng([M, K, run])
    W = (rng.standard_normal((M, K)) * 0.05 + 0.3).astype(np.float16)
    window = np.arange(M)[:, None] * (K // 4) + np.arange(K)[None, :] // 4
    W[(window // run) % 2 == 1] = 0
    return W


def _random(M, K, p):
    rng = np.random.default_rng([M, K])
    W = (rng.standard_normal((M, K)) * 0.02).astype(np.float16)
    return np.where(rng.random((M, K)) < p, W, np.float16(0))


@pytest.mark.parametrize("W,pitch,shift", [(_runs(128, 128, 9), 128, 0),         # code bytes beyond the staging area
                                           (_random(129, 131, 0.5), 131, 0),     # one row and three columns over, odd pitch
                                           (_random(7, 3, 1.0), 3, 0),           # less than a window
                                           (_random(200, 250, 0.6), 252, 1),     # base not on 8 bytes
                                           (_random(200, 250, 0.6), 252, 4),     # 8-byte windows, ragged last one
                                           (_random(130, 900, 0.3), 904, 0)])
def test_conversion_of_awkward_sources(tl3, W, pitch, shift):
    """Container and packed blob, each byte for byte the host library's: tiles at the edges of the
    matrix, sources that 8-byte loads cannot read, a tile with more code bytes than are staged."""
    import torch
    M, K = W.shape
    ref = tl3.encode(W)
    buf = torch.zeros(M * pitch + shift, dtype=torch.float16, device="cuda")
    src = buf[shift:].view(M, pitch)[:, :K]
    src.copy_(torch.from_numpy(W))
    m = tl3.Matrix.encode_on_device(src)
    for name in tl3.CANONICAL:
        assert np.array_equal(m.canonical(name), ref.canonical(name)), name
    assert m.serialize() == ref.serialize()
    want = ref.pack()
    assert np.array_equal(m.upload_packed_on_device().cpu().numpy(), want)
    only = tl3.Matrix.encode_on_device(src, device_only=True)
    assert np.array_equal(only.upload_packed_on_device().cpu().numpy(), want)
    assert only.stats()["canonical_bytes"] == ref.stats()["canonical_bytes"]


def test_conversion_on_a_nearly_full_device(tl3):
    """Room for the container, its bytes and entries as they are, but not for the allocation that serves any
    matrix down to 40 % sparsity at once (29 KB per tile)."""
    import torch
    W = torch.from_numpy(_random(8192, 4096, 0.5)).cuda()
    tiles, MB = 64 * 32, 1 << 20
    ref = tl3.Matrix.encode_on_device(W, device_only=True)
    want = ref.upload_packed_on_device().clone()
    blob = torch.empty_like(want)
    ref.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = 52 * MB
    assert 19200 * tiles + 5 * MB < room < 29000 * tiles
    filler = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    assert abs(torch.cuda.mem_get_info()[0] - room) <= 3 * MB
    m = tl3.Matrix.encode_on_device(W, device_only=True)
    stream = torch.cuda.current_stream().cuda_stream
    assert m.device_bytes() == want.numel()
    assert tl3.lib().tl3_upload_device(m._h, blob.data_ptr(), stream) == tl3.OK
    del filler
    torch.cuda.empty_cache()
    assert torch.equal(blob, want)


@pytest.mark.parametrize("call", ["encode_device_only", "encode_device", "plan_device"])
def test_calls_after_one_that_found_no_memory(tl3, call):
    """A conversion or an upload that the device has no room for reports that, and the calls after it on the same
    thread report themselves: not the failed allocation once more."""
    import torch
    W = torch.from_numpy(_random(8192, 4096, 0.5)).cuda()
    MB = 1 << 20
    ref = tl3.Matrix.encode_on_device(W)
    want = torch.from_numpy(ref.pack()).cuda()
    W2 = torch.from_numpy(_random(300, 260, 0.5)).cuda()
    X = torch.zeros((260, 16), dtype=torch.float16, device="cuda").normal_()
    small = tl3.Matrix.encode_on_device(W2, device_only=True)
    small.upload_packed_on_device()
    ws, Y, again = small.new_workspace(16), small.spmm(X), torch.zeros((300, 16), dtype=torch.float16, device="cuda")
    plan = tl3.Matrix.deserialize(ref.serialize())
    calls = {"encode_device_only": lambda: tl3.Matrix.encode_on_device(W, device_only=True),
             "encode_device": lambda: tl3.Matrix.encode_on_device(W),
             "plan_device": lambda: tl3._check(tl3.lib().tl3_plan_device(plan._h, torch.cuda.current_stream().cuda_stream), "plan")}
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - 24 * MB, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(tl3.Tl3Error) as e:
            calls[call]()
        assert e.value.code == tl3.ERR_CUDA and tl3.lib().tl3_last_cuda_error() == 2  # cudaErrorMemoryAllocation
        small.spmm(X, again, workspace=ws)                                             # (allocates nothing)
    finally:
        del filler
        torch.cuda.empty_cache()
    assert torch.equal(again, Y)
    m = tl3.Matrix.encode_on_device(W, device_only=True)
    assert torch.equal(m.upload_packed_on_device(), want)
    assert torch.equal(plan.upload_packed_on_device(), want)
    assert torch.equal(small.spmm(X, again, workspace=ws), Y)
