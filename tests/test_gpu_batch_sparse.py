"""The batch kernel has two forms of its expansion, chosen by the values of an average column tile: both sides of that line, and
columns of every density inside one layer, give exact sums on integers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", [0, 1, 79, 81, 256])
@pytest.mark.parametrize("M,K,B", [(256, 64, 3), (700, 1000, 8), (1536, 300, 5)])
def test_both_forms_exact_on_integers(values, M, K, B):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp as S
    rng = np.random.Generator(np.random.PCG64(values * 1000 + M))
    # column densities between 0 and twice the average (an average of 256 is a full layer): every nibble pattern at every alignment
    share = np.minimum(values / 256.0 * 2.0 * rng.random(K) if values < 256 else np.ones(K), 1.0)
    W = rng.integers(1, 9, (M, K)).astype(np.float16) * rng.choice([-1, 1], (M, K)).astype(np.float16)
    W[rng.random((M, K)) >= share] = 0
    X = rng.integers(-4, 5, (B, K)).astype(np.float16)
    want = X.astype(np.float64) @ W.astype(np.float64).T                 # |sums| <= 1000 * 32 < 2^24: exact in fp32
    h = S.spdp_pack_tiled_cbc(torch.from_numpy(W).cuda())
    try:
        Y = torch.full((B, M), float("nan"), dtype=torch.float32, device="cuda")
        S.spdp_spmspv_batch(h, torch.from_numpy(X).cuda(), S.SPDP_DP_NONE, 0.0, Y)
        torch.cuda.synchronize()
        assert S.spdp_last_device_status(h) == 0
        assert np.array_equal(Y.cpu().numpy().astype(np.float64), want)
    finally:
        S.spdp_free(h)
