"""Where launches of 65 to 128 columns begin to go in pairs of CTAs (needs a B200): both sides of the line, both
layouts, an odd number of row-tiles, a workspace for few columns, against the product in float64."""
import pytest

from paper_2607_08786_b200 import build, tl3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N,columns,cluster", [(128 * 37, 128 * 128, 65, 96, 2), (128 * 37, 128 * 128, 128, 128, 2), (128 * 37 - 5, 128 * 129 - 3, 100, 128, 2),
                                                   (128 * 37, 128 * 127, 100, 112, 1), (128 * 37, 128 * 127, 64, 64, 1)])
def test_pairs_of_few_columns(M, K, N, columns, cluster):
    import torch
    build.build_library()
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the shapes are 31.75 and 32 tiles per CTA of 148")
    g = torch.Generator(device="cuda").manual_seed(M + N)
    W = torch.randn((M, K), generator=g, device="cuda").mul_(0.02).half()
    W[torch.rand((M, K), generator=g, device="cuda") < 0.5] = 0
    m = tl3.Matrix.encode_on_device(W, device_only=True)
    m.upload_packed_on_device()
    Xt = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xt[:, :K] = torch.randn((N, K), generator=g, device="cuda").half()
    Xd = torch.zeros((K, (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = Xt[:, :K].T
    sums = torch.cat([Xt[:, :K].double() @ W[r:r + 1024].double().T for r in range(0, M, 1024)], dim=1)
    bound = torch.cat([Xt[:, :K].double().abs() @ W[r:r + 1024].double().abs().T for r in range(0, M, 1024)], dim=1)
    # chains of 2 K / 32 MMA steps and some partial sums in fp32, each off by 2^-23 of what it may reach at most; one rounding to fp16
    tol = (K / 16 + 9) * 2.0**-23 * bound + (2.0**-11 + 2.0**-18) * sums.abs() + 2.0**-25
    results = []
    for room in (None, 64):
        ws = m.new_workspace(room or N)
        Y, Yt = m.spmm(Xd[:, :N], workspace=ws), m.spmm_nt(Xt[:, :K], workspace=ws)
        if N > 64:
            assert {"columns": columns, "cluster": cluster} == {k: m.last_pass()[k] for k in ("columns", "cluster")}
        assert bool(((Yt.double() - sums).abs() <= tol).all())
        assert torch.equal(Y.T.contiguous().view(torch.int16), Yt.view(torch.int16))
        assert m.status(ws) == tl3.OK
        results.append(Yt)
    small = torch.zeros(m.workspace_bytes(N), dtype=torch.uint8, device="cuda")     # only zeroed: counts as the smallest
    assert bool(((m.spmm_nt(Xt[:, :K], workspace=small).double() - sums).abs() <= tol).all()) and m.status(small) == tl3.OK
    assert torch.equal(results[0].view(torch.int16), results[1].view(torch.int16))


@pytest.mark.parametrize("N", [65, 96, 128])
def test_pairs_of_few_columns_in_a_workspace_that_was_only_zeroed(N):
    """The smallest workspace holds all columns of such a pass: the same passes as with an initialised one, and so
    the same partial sums and the same bits."""
    import torch
    build.build_library()
    M, K = 128 * 42, 128 * 114
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the shape is 32.4 tiles per CTA of 148")
    g = torch.Generator(device="cuda").manual_seed(N)
    W = torch.randn((M, K), generator=g, device="cuda").mul_(0.02).half()
    W[torch.rand((M, K), generator=g, device="cuda") < 0.5] = 0
    m = tl3.Matrix.encode_on_device(W, device_only=True)
    m.upload_packed_on_device()
    Xt = torch.randn((N, K), generator=g, device="cuda").half()
    Xd = torch.zeros((K, (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = Xt.T
    made, zeroed = m.new_workspace(N), torch.zeros(m.workspace_bytes(N), dtype=torch.uint8, device="cuda")
    for product, X in ((m.spmm, Xd[:, :N]), (m.spmm_nt, Xt)):
        want, got = product(X, workspace=made), product(X, workspace=zeroed)
        assert m.last_pass()["cluster"] == 2
        assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    assert m.status(zeroed) == tl3.OK


@pytest.mark.parametrize("row_tiles,N,cluster", [(9, 128, 1), (9, 100, 1), (35, 96, 1), (36, 96, 2), (9, 80, 2), (2, 66, 2), (1, 80, 1)])
def test_few_row_tiles_go_in_pairs_up_to_80_columns_only(row_tiles, N, cluster):
    import torch
    build.build_library()
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the shapes are a little more than 32 tiles per CTA of 148")
    M, K = 128 * row_tiles, 128 * -(-(72 if row_tiles == 2 else 33) * 148 // row_tiles)
    g = torch.Generator(device="cuda").manual_seed(M + N)
    W = torch.randn((M, K), generator=g, device="cuda").mul_(0.02).half()
    W[torch.rand((M, K), generator=g, device="cuda") < 0.5] = 0
    m = tl3.Matrix.encode_on_device(W, device_only=True)
    m.upload_packed_on_device()
    Xt = torch.randn((N, K), generator=g, device="cuda").half()
    Xd = torch.zeros((K, (N + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    Xd[:, :N] = Xt.T
    Y, Yt = m.spmm(Xd[:, :N]), m.spmm_nt(Xt)
    assert m.last_pass()["cluster"] == cluster
    sums, bound = Xt.double() @ W.double().T, Xt.double().abs() @ W.double().abs().T
    # as above: chains of MMA steps and partial sums in fp32, one rounding to fp16
    assert bool(((Yt.double() - sums).abs() <= (K / 16 + 9) * 2.0**-23 * bound + (2.0**-11 + 2.0**-18) * sums.abs() + 2.0**-25).all())
    assert torch.equal(Y.T.contiguous().view(torch.int16), Yt.view(torch.int16))
