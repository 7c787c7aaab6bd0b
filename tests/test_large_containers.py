"""Containers large enough that copying, checking and sending them is shared out over threads."""
import threading

import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3


@pytest.fixture(scope="module")
def matrix():
    build.build_library()
    rng = np.random.default_rng(11)
    W = (rng.standard_normal((2300, 4100)) * 0.02).astype(np.float16)   # value array 9.9 MB, ragged in both sizes
    W[rng.random(W.shape) < 0.45] = 0
    return tl3.encode(W)


@pytest.mark.parametrize("kind", [bytes, bytearray, memoryview, lambda b: np.frombuffer(b, dtype=np.uint8)])
@pytest.mark.parametrize("compact", [False, True])
def test_round_trip(matrix, kind, compact):
    data = matrix.serialize(compact=compact)
    m = tl3.Matrix.deserialize(kind(data))
    assert m.shape == matrix.shape and m.serialize() == matrix.serialize()
    for name in tl3.CANONICAL:
        assert np.array_equal(m.canonical(name), matrix.canonical(name)), name


@pytest.mark.parametrize("M,K", [(4096, 4991), (4096, 5119), (6000, 4200)])
def test_arrays_around_the_size_that_more_threads_copy(M, K):
    """Value arrays a column of tiles short of 20 MB, of 20 MB and of 25."""
    rng = np.random.default_rng(K)
    W = np.zeros((M, K), dtype=np.float16)
    W[rng.random(W.shape) < 0.5] = 0.25
    m = tl3.encode(W)
    data = m.serialize()
    again = tl3.Matrix.deserialize(data)
    assert again.serialize() == data and np.array_equal(again.decode(), W.view(np.uint16))


def test_a_bad_position_in_any_tile_is_found(matrix):
    data = bytearray(matrix.serialize())
    n_tiles = matrix.stats()["n_tiles"]
    header = 8 + 16 + 16 + 48
    at = header
    for name in ("tc_vals", "tc_meta"):
        at += 8 + int.from_bytes(data[at:at + 8], "little")
    at += 8                                                     # chain_tau0: 128 two-byte starts per tile
    for tile in (0, 63, 64, n_tiles // 2, n_tiles - 1):
        spot = at + tile * 256
        saved = bytes(data[spot:spot + 2])
        data[spot:spot + 2] = (8192).to_bytes(2, "little")      # one beyond the last slot of a tile
        with pytest.raises(tl3.Tl3Error) as e:
            tl3.Matrix.deserialize(data)
        assert e.value.code == tl3.ERR_BAD_CONTAINER
        data[spot:spot + 2] = saved
    tl3.Matrix.deserialize(data)
    for wrong in (b"", bytes(data[:-1]), bytes(data[:header])):
        with pytest.raises(tl3.Tl3Error):
            tl3.Matrix.deserialize(wrong)


@pytest.mark.gpu
def test_loading_from_several_threads(matrix):
    """One thread sends through the pinned pieces, the others meanwhile do without."""
    import torch
    data, want = matrix.serialize(), matrix.pack()
    got, errors = [None] * 4, []

    def load(i):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                m = tl3.Matrix.deserialize(data)
                got[i] = m.upload_packed_on_device().cpu().numpy()
        except Exception as e:                                  # reported below, in the main thread
            errors.append(e)

    torch.cuda.init()
    threads = [threading.Thread(target=load, args=(i,)) for i in range(len(got))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for blob in got:
        assert np.array_equal(blob, want)


@pytest.mark.gpu
def test_encoding_on_several_threads(matrix):
    """The way down: one thread's container comes through the pinned pieces, the others' meanwhile without."""
    import torch
    W, want = torch.from_numpy(matrix.decode().view(np.float16)).cuda(), matrix.serialize()
    got, errors = [None] * 4, []
    torch.cuda.synchronize()

    def encode(i):
        try:
            for _ in range(3):
                got[i] = tl3.Matrix.encode_on_device(W, stream=torch.cuda.Stream()).serialize()
        except Exception as e:                                  # reported below, in the main thread
            errors.append(e)

    threads = [threading.Thread(target=encode, args=(i,)) for i in range(len(got))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    assert all(data == want for data in got)
