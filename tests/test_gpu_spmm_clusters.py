"""Prefill calls whose tiles are shared by the CTAs of a thread-block cluster, which add their sums themselves: 2 to 16 CTAs to a tile, with
equal and unequal slices of its K-blocks, several token blocks, more CTAs than tokens, rows and tokens that end inside a tile.  Small whole numbers,
so that sums are exact in any order and the results have to be equal."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K,N", [(700, 5000, 16), (700, 5000, 3), (513, 1100, 33), (1024, 1024, 16), (1300, 2100, 100), (2048, 2048, 250), (5000, 900, 22),
                                   (11000, 1030, 128), (11008, 1024, 130), (16000, 700, 129), (250, 200, 5), (4000, 4098, 7), (8100, 1600, 60)])
@pytest.mark.parametrize("y", ["f32", "f16"])
def test_whole_numbers_are_exact(M, K, N, y):
    import torch
    from paper_2607_21985_b200 import spdp
    g = torch.Generator(device="cuda").manual_seed(M + K + N)
    W = torch.randint(1, 5, (M, K), generator=g, device="cuda") * (2 * torch.randint(0, 2, (M, K), generator=g, device="cuda") - 1)
    W = (W * (torch.rand(M, K, generator=g, device="cuda") < 0.4)).half()
    X = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    X[:, :K] = torch.randint(-2, 3, (N, K), generator=g, device="cuda").half()
    want = X[:, :K].double() @ W.double().T
    assert want.abs().max() < 2048          # whole numbers of 16 bits too
    h = spdp.spdp_pack_tiled_cbc(W)
    try:
        out = []
        for _ in range(3):                  # calls in a row start beside one another
            Y = torch.full((N, M + 1), float("nan"), dtype=torch.float32 if y == "f32" else torch.float16, device="cuda")[:, :M]
            spdp.spdp_spmm(h, X[:, :K], Y)
            out.append(Y)
        torch.cuda.synchronize()
        assert spdp.spdp_last_device_status(h) == 0
        assert all(torch.equal(Y.double(), want) for Y in out)
    finally:
        spdp.spdp_free(h)
