"""Waits of the prefill kernels that run out.  The checked build lets a test set after how many attempts they do; with a few, roles give up all over the
call, each at another place.  What is left then: the kernels end, the status says so, no output is wrong (it is right or unwritten) although the
scratch memory still holds an earlier call's sums, and the next call is whole.  Small whole numbers, so that sums are exact in any order.
Nothing here reads or writes out of range or waits without a limit: a role that gives up touches nothing any more, hands nothing on, and a CTA leaves when
its copies and products have landed."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from device_plan import device_plan

# row tiles, K, tokens, sparsity -> kernel, cut, CTA ranges that cross tiles
ONE = {
    (1, 2600, 1, 0.5): (0, True, False),
    (149, 64, 20, 0.0): (0, False, False),
    (50, 2600, 20, 0.5): (1, True, True),
    (150, 1000, 30, 0.9): (1, True, False),
    (75, 2000, 129, 0.5): (2, True, True),
    (60, 64, 100, 0.5): (2, False, False),
}
# -> kernel, whole tiles, cut tiles (sparse layers have three X tiles in flight for each accumulator)
PAIRS = {
    (75, 640, 400, 0.5): (3, True, True),
    (75, 640, 400, 0.9): (3, True, True),
    (3, 12000, 1024, 0.9): (3, False, True),
    (8, 3000, 150, 0.5): (4, False, True),
    (8, 3000, 150, 0.9): (4, False, True),
    (22, 700, 1024, 0.5): (4, True, False),
    (38, 5000, 257, 0.5): (4, False, True),
}
# -> kernel, CTAs of a cluster: each adds up a share of the tokens, where another's sums are missing if that one gave up
CLUSTERS = {
    (35, 200, 20, 0.5): (0, 2),
    (27, 1000, 2, 0.5): (0, 4),
    (6, 1600, 2, 0.9): (0, 9),
    (26, 640, 250, 0.5): (1, 2),
    (43, 4096, 128, 0.6): (1, 3),
    (15, 9000, 128, 0.5): (1, 9),
}
# 32-bit results, whose K-blocks go to several accumulators in turn -> kernel, CTAs of a cluster, accumulators
SETS = {
    (60, 2176, 30, 0.5): (1, 2, 2),
    (43, 4096, 64, 0.6): (1, 3, 2),
    (10, 6144, 146, 0.5): (4, 1, 2),
    (10, 9216, 219, 0.9): (3, 1, 2),
}


@pytest.mark.parametrize("shape", list(CLUSTERS))
def test_shapes_of_clusters(shape):
    q = device_plan(*shape[:3])
    assert (q["kernel"], q["cluster"]) == CLUSTERS[shape]


@pytest.mark.parametrize("shape", list(SETS))
def test_shapes_of_several_accumulators(shape):
    q = device_plan(*shape[:3], wide=True)
    assert (q["kernel"], q["cluster"], q["sets"]) == SETS[shape]


@pytest.mark.parametrize("shape", list(ONE))
def test_shapes_of_one_cta(shape):
    q = device_plan(*shape[:3])
    assert (q["kernel"], q["cut"], q["crosses"]) == ONE[shape] and q["cluster"] == 1


@pytest.mark.parametrize("shape", list(PAIRS))
def test_shapes_of_pairs(shape):
    q = device_plan(*shape[:3])
    assert (q["kernel"], q["tiles"] > q["rest"], q["cut"]) == PAIRS[shape]


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import build, spdp
    saved = (spdp.LIB_PATH, spdp._lib)
    spdp.LIB_PATH, spdp._lib = build.build_checked(), None
    spdp.lib().spdp_checked_wait_tries.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_uint, ctypes.c_uint, ctypes.c_int]
    yield spdp
    spdp.LIB_PATH, spdp._lib = saved


# attempts of the chosen warps and of the others, chosen warps, chosen CTAs (modulo 16): all at once, then one role at a time, in all CTAs, in every
# second, in one of 16; then only where a warp waits for the products before it stores them (all warps do in a pair).  Warps 0 to 23 decode, the first of them store; behind them
# the tensor-core, copy and X or relay warps.
ALL, LATE = 0xFFFFFFFF, 1 << 12
LIMITS = [(tries, tries, ALL, 0xFFFF, 0) for tries in (0, 1, 2, 4, 8, 16, 32, 64, 128)]
LIMITS += [(tries, LATE, 1 << warp, ctas, 0) for warp in (0, 5, 10, 15, 23, 24, 25, 26, 27) for ctas in (0xFFFF, 0x5555, 0xAAAA, 0x0200) for tries in (0, 2, 16)]
LIMITS += [(0, LATE, warps, ctas, 1) for warps in (1, 1 << 5, 1 << 10, 1 << 23, 1 << 24, ALL) for ctas in (0xFFFF, 0x5555, 0xAAAA, 0x0200)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape,dt", [(shape, "float16") for shape in list(ONE) + list(PAIRS) + list(CLUSTERS)] + [(shape, "float32") for shape in SETS])
def test_nothing_wrong_is_left(S, shape, dt):
    R, K, N, sparsity = shape
    M = 256 * R - 5
    g = torch.Generator(device="cuda").manual_seed(R * K + N)
    W = torch.randint(1, 5, (M, K), generator=g, device="cuda").half() * (2 * torch.randint(0, 2, (M, K), generator=g, device="cuda") - 1).half()
    W[torch.rand(M, K, generator=g, device="cuda") < sparsity] = 0
    X = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    X[:, :K] = torch.randint(1, 3, (N, K), generator=g, device="cuda").half()
    want = (X[:, :K].double() @ W.double().T).to(getattr(torch, dt))
    other = -X                                                  # whose sums are in the scratch memory
    h = S.spdp_pack_tiled_cbc(W)
    limit = S.lib().spdp_checked_wait_tries
    incomplete = 0
    try:
        def call(x):
            Y = torch.full((N, M), float("nan"), dtype=want.dtype, device="cuda")
            S.spdp_spmm(h, x[:, :K], Y)
            return Y, S.spdp_last_device_status(h)
        for tries in LIMITS:
            Y, status = call(other)
            assert status == 0 and torch.equal(Y, -want)
            assert limit(*tries) == 0
            Y, status = call(X)
            assert limit(-1, -1, 0, 0, 0) == 0
            unwritten = torch.isnan(Y)
            assert bool((unwritten | (Y == want)).all()), tries
            assert status == S.SPDP_ERR_TIMEOUT or (status == 0 and not bool(unwritten.any())), tries
            incomplete += bool(unwritten.any())
        assert incomplete > 0                                   # without any attempt nobody gets far
        Y, status = call(X)
        assert status == 0 and torch.equal(Y, want)
    finally:
        limit(-1, -1, 0, 0, 0)
        S.spdp_free(h)
