"""The batch kernel has two forms of its expansion, chosen by the values of an average column tile and by how much the
columns differ: 16-bit loads below a line, aligned words above.  Both sides of that line, and columns from empty to full in
either form, give exact sums on integers; values that are not finite read the same in both."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_batch_form import compile_rule, rows_of

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


@pytest.fixture(scope="module")
def one_by_one(tmp_path_factory):
    return compile_rule(tmp_path_factory.mktemp("form"))


# values of a column tile of so many rows, in column k, and whether the layer takes the 16-bit loads
LAYERS = {
    "last before the line": (lambda rows, k, rng: rows * 96 // 256, True),
    "first behind the line": (lambda rows, k, rng: -(-rows * 97 // 256), False),
    "a few full columns among sparse ones": (lambda rows, k, rng: rows if k % 150 == 7 else rng.integers(0, 10), True),
    "from empty to full": (lambda rows, k, rng: (0, rows, rng.integers(0, rows + 1))[k % 3], False),
    "sparse and uneven": (lambda rows, k, rng: rows * (10 if k % 2 else 70) // 256, False),
}


@pytest.mark.parametrize("layer", list(LAYERS))
@pytest.mark.parametrize("M,K,B", [(512, 300, 3), (700, 1001, 8), (256, 200, 5)])
def test_both_sides_of_the_line(one_by_one, layer, M, K, B):
    """Layers on either side of the line, down to one value a tile from it, and full columns in both forms (their loads run past the last
    value)."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp as S
    rng = np.random.Generator(np.random.PCG64(M + K))
    count, loads = LAYERS[layer]
    counts = np.array([[count(rows, k, rng) for k in range(K)] for rows in rows_of(M)])
    assert one_by_one(counts, M) == loads
    W = np.zeros((M, K), np.float16)
    for r, rows in enumerate(rows_of(M)):
        for k in range(K):
            at = 256 * r + rng.permutation(rows)[:counts[r, k]]
            W[at, k] = rng.integers(1, 9, len(at)) * rng.choice([-1, 1], len(at))
    X = rng.integers(-4, 5, (B, K)).astype(np.float16)
    want = X.astype(np.float64) @ W.astype(np.float64).T                # |sums| <= 1001 * 32 < 2^24: exact in fp32
    h = S.spdp_pack_tiled_cbc(torch.from_numpy(W).cuda())
    try:
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
def test_non_finite_values_in_both_forms(one_by_one, density):
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
    assert one_by_one((W.reshape(2, 256, K) != 0).sum(1), M) == (density < 0.3)
    h = S.spdp_pack_tiled_cbc(torch.from_numpy(W).cuda())
    try:
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
