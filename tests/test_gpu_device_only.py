"""Dense W to packed blob in one pass on the GPU (needs a B200): blob and layer counts against the host
library's, byte for byte, where the pass takes its rarer ways."""
import numpy as np
import pytest

from special_cases import clustered_surplus_tile

pytestmark = pytest.mark.gpu


def _cut(rows, M=128, K=128):
    """Rows of dense weights among 2:4 rows with an empty slot every 115: eight delta bytes per pair, so that the
    first of them is cut at 255, and from the second on surplus weights find no empty slot either."""
    rng = np.random.default_rng(len(rows))
    W = np.zeros((M, K), dtype=np.float16)
    base = (rng.standard_normal((M, K)) * 0.05 + 0.3).astype(np.float16)
    W[:, 0::4], W[:, 1::4] = base[:, 0::4], base[:, 1::4]
    W[rows] = base[rows]
    for k in range(70):
        tau = 64 + k * 115
        if tau // 64 not in rows:
            W[tau // 64, 4 * ((tau % 64) // 2) + (tau & 1)] = 0
    return W


def _random(M, K, p):
    rng = np.random.default_rng([M, K])
    W = (rng.standard_normal((M, K)) * 0.02 + 0.1).astype(np.float16)
    return np.where(rng.random((M, K)) < p, W, np.float16(0))


@pytest.mark.parametrize("W", [_cut([0]), _cut([0, 60]), _cut([5, 6, 127]), np.vstack([_cut([0]), _cut([3, 90])]), clustered_surplus_tile(),
                               _random(128, 128, 1.0),                  # 51840 bytes, which the first allocation has room for; not
                               _random(128, 256, 1.0), _random(640, 900, 1.0),      # for two such tiles, nor for forty: a second pass makes the others
                               _random(640, 900, 0.75), np.zeros((300, 140), dtype=np.float16), _random(1, 1, 1.0)],
                         ids=["cut", "cut_and_beyond", "cut_3", "two_tiles_cut", "clustered", "dense_tile", "two_dense_tiles", "dense", "a_quarter", "zeros", "one_weight"])
def test_device_only(W):
    import torch
    from paper_2607_08786_b200 import build, tl3
    build.build_library()
    ref = tl3.encode(W)
    want, stats = ref.pack(), ref.stats()
    m = tl3.Matrix.encode_on_device(torch.from_numpy(W).cuda(), device_only=True)
    assert m.device_bytes() == want.size
    for key, value in m.stats().items():
        assert value == (-1 if key.startswith("canonical_bytes_compact") else stats[key]), key
    blob = torch.full((want.size,), 0xA5, dtype=torch.uint8, device="cuda")      # every byte of it is written
    assert tl3.lib().tl3_upload_device(m._h, blob.data_ptr(), torch.cuda.current_stream().cuda_stream) == tl3.OK
    assert np.array_equal(blob.cpu().numpy(), want)
