"""The batch kernel has two forms of its expansion, chosen by the values that a full column tile of average density has (of
256): 16-bit loads up to 80, aligned words above.  Both sides of that line, and columns from empty to full in
either form, give exact sums on integers; values that are not finite read the same in both."""
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
    # column densities between 0 and twice the average (an average of 256 is a full layer)
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


def line(M, K):
    """The most values of a layer that takes the 16-bit loads."""
    return 80 * M * K // 256


@pytest.mark.parametrize("beyond", [0, 1])
@pytest.mark.parametrize("M,K,B", [(512, 300, 3), (700, 1001, 8), (256, 64, 5)])
def test_exactly_at_the_line(beyond, M, K, B):
    """A layer with exactly as many values as the 16-bit loads take, and one with one more: full and empty columns (the loads of a
    full one run past its last value) and every count between in both."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp as S
    rng = np.random.Generator(np.random.PCG64(M + K))
    R = (M + 255) // 256
    rows = [min(256, M - 256 * r) for r in range(R)]
    counts = np.stack([rng.integers(0, rows[r] + 1, K) for r in range(R)])
    fixed = np.zeros(K, bool)
    fixed[rng.permutation(K)[:K // 5]] = True
    counts[:, fixed] = np.where(rng.random((R, fixed.sum())) < 0.5, 0, np.array(rows)[:, None])
    want_nnz = line(M, K) + beyond
    while (d := want_nnz - int(counts.sum())) != 0:                     # the other columns make up the rest
        r, k = rng.integers(R), rng.integers(K)
        if not fixed[k]:
            counts[r, k] = min(rows[r], max(0, counts[r, k] + max(-40, min(40, d))))
    W = np.zeros((M, K), np.float16)
    for r in range(R):
        for k in range(K):
            at = 256 * r + rng.permutation(rows[r])[:counts[r, k]]
            W[at, k] = rng.integers(1, 9, len(at)) * rng.choice([-1, 1], len(at))
    X = rng.integers(-4, 5, (B, K)).astype(np.float16)
    want = X.astype(np.float64) @ W.astype(np.float64).T                # |sums| <= 1001 * 32 < 2^24: exact in fp32
    h = S.spdp_pack_tiled_cbc(torch.from_numpy(W).cuda())
    try:
        assert S.spdp_get_info(h).nnz == want_nnz
        for ctas in (0, 2):
            S.spdp_set_num_ctas(h, ctas)
            Y = torch.full((B, M), float("nan"), dtype=torch.float32, device="cuda")
            S.spdp_spmspv_batch(h, torch.from_numpy(X).cuda(), S.SPDP_DP_NONE, 0.0, Y)
            torch.cuda.synchronize()
            assert S.spdp_last_device_status(h) == 0
            assert np.array_equal(Y.cpu().numpy().astype(np.float64), want)
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("density", [0.25, 0.9])
def test_non_finite_values_in_both_forms(density):
    """An infinite weight or a NaN among the weights stays in its row, in the tokens that keep its column; a token that skips
    the column gets NaN there (0 * Inf) where another token makes it fetched; a NaN activation reaches every row of its token."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp as S
    rng = np.random.Generator(np.random.PCG64(int(100 * density)))
    M, K, B = 512, 200, 5
    W = rng.integers(1, 5, (M, K)).astype(np.float16)
    W[rng.random((M, K)) >= density] = 0
    W[5, 50], W[300, 51], W[301, 51] = np.inf, np.nan, 2.0
    X = rng.integers(1, 4, (B, K)).astype(np.float16)
    X[1, 50] = X[2, 51] = 0.0
    X[3, 60] = np.nan
    rule, thr = S.SPDP_DP_ABS_GT, 0.0                                   # skips exact zeros
    finite = np.where(np.isfinite(W), W, 0).astype(np.float64)
    want = np.where(np.isfinite(X), X, 0).astype(np.float64) @ finite.T
    h = S.spdp_pack_tiled_cbc(torch.from_numpy(W).cuda())
    try:
        assert (S.spdp_get_info(h).nnz <= line(M, K)) == (density < 0.3)
        Y = torch.zeros((B, M), dtype=torch.float32, device="cuda")
        S.spdp_spmspv_batch(h, torch.from_numpy(X).cuda(), rule, thr, Y)
        torch.cuda.synchronize()
        Y = Y.cpu().numpy()
    finally:
        S.spdp_free(h)
    assert np.all(Y[[0, 2, 4], 5] == np.inf) and np.isnan(Y[1, 5])
    assert np.all(np.isnan(Y[:, 300]))
    assert np.all(np.isnan(Y[3]))
    rest = np.ones(M, bool)
    rest[[5, 300]] = False
    for b in (0, 1, 2, 4):
        assert np.array_equal(Y[b, rest].astype(np.float64), want[b, rest]), b
