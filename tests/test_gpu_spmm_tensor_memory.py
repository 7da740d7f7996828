"""Prefill with decoded W in tensor memory (up to 128 tokens a tile): every row of a column tile with every number of values before it, the ends of
K-blocks and row tiles, token counts around the steps of the products and of the stores.  Small whole numbers, so that sums are exact in
any order and the results have to be equal."""
import pytest

pytestmark = pytest.mark.gpu


def _layer(M, K, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    W = torch.randint(1, 8, (M, K), generator=g) * (2 * torch.randint(0, 2, (M, K), generator=g) - 1)
    keep = torch.rand(M, K, generator=g) < torch.linspace(0.0, 1.0, K)[torch.randperm(K, generator=g)]      # empty columns, full ones, all between
    return (W * keep).half()


@pytest.mark.parametrize("M,K", [(256, 64), (1, 1), (255, 31), (300, 33), (513, 130), (1030, 1100), (64, 2049)])
@pytest.mark.parametrize("N", [1, 7, 8, 9, 16, 17, 32, 33, 100, 128, 129])
def test_whole_numbers_are_exact(M, K, N):
    import torch
    from paper_2607_21985_b200 import spdp
    W = _layer(M, K, 7 * M + K)
    ld = (K + 7) // 8 * 8
    X = torch.zeros(N, ld, dtype=torch.float16)
    X[:, :K] = torch.randint(-8, 9, (N, K), generator=torch.Generator().manual_seed(N)).half()
    want = X[:, :K].double() @ W.double().T
    assert want.abs().max() < 2 ** 24
    h = spdp.spdp_pack_tiled_cbc(W.cuda())
    try:
        Xd = X.cuda()
        for ldy, off in ((M, 0), (M + 3, 1)):                   # rows that may be stored two at a time, and rows that may not
            Y = torch.full((N * ldy + off,), 7.0, device="cuda")
            Yv = Y[off:].view(N, ldy)[:, :M]
            spdp.spdp_spmm(h, Xd[:, :K], Yv)
            torch.cuda.synchronize()
            assert torch.equal(Yv.cpu().double(), want)
        assert spdp.spdp_last_device_status(h) == 0
    finally:
        spdp.spdp_free(h)
