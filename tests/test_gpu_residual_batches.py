"""Tiles with given numbers of Residual entries around the batches that a decode thread takes them in (needs a
B200): a product with the unit matrix gives back W bit for bit, from both kernels, with few and with many
entries per tile on average."""
import numpy as np
import pytest

from paper_2607_08786_b200 import build, tl3

pytestmark = pytest.mark.gpu


def _tile(count, rng):
    """Windows of two weights (no slot is empty), of which `count` surplus weights are added: all of them Residual."""
    W = np.zeros((128 * 32, 4), dtype=np.float16)
    values = (rng.standard_normal(W.shape) * 0.05).astype(np.float16)
    values[values == 0] = np.float16(0.01)
    W[:, :2] = values[:, :2]
    spots = rng.permutation(128 * 32)[:(count + 1) // 2]
    W[spots, 2] = values[spots, 2]
    W[spots[:count - (count + 1) // 2], 3] = values[spots[:count - (count + 1) // 2], 3]
    return W.reshape(128, 128)


@pytest.mark.parametrize("counts", [(512, 512), (511, 513), (511, 512), (1023, 1), (1024, 0), (1025, 127), (2047, 129), (2048, 640), (8192, 0), (8191, 8192), (0, 0), (640, 383)])
def test_residual_counts(counts):
    import torch
    build.build_library()
    rng = np.random.default_rng(list(counts))
    W = np.vstack([_tile(c, rng) for c in counts])
    m = tl3.encode(W)
    m.upload()
    assert m.stats()["n_res"] == sum(counts)
    eye = torch.eye(128, dtype=torch.float16, device="cuda")
    Y = m.spmm(eye)                                                # more than 64 columns: one kernel
    parts = [m.spmm(eye[:, c:c + n].contiguous()) for c, n in ((0, 64), (64, 32), (96, 16), (112, 16))]     # up to 64: the other
    Yt = m.spmm_nt(eye)
    for got in (Y, torch.cat(parts, dim=1), Yt.T):
        assert np.array_equal(got.cpu().numpy().view(np.uint16), W.view(np.uint16))
