"""How far 32-bit prefill results are from 64-bit ones.  The tensor cores do not round what they add to an accumulator to nearest, so that the error grows with the
K-blocks (64 columns) that one accumulator adds: 6e-8 to 8e-8 of the results' root mean square for each one, measured from 7 to 166 of them on layers of
30 to 90 % sparsity; the roundings of the sums and of the result are 1e-7 in all.  A shape's bound is 1e-7 for each K-block that its accumulators are to
add, and 1.5e-7."""
import math

import pytest

torch = pytest.importorskip("torch")

from device_plan import device_plan, lib

# row tiles, K, tokens -> K-blocks that one accumulator adds, at most: the root of the mean, over the results, of the cubes' sum over a tile's accumulators by its
# K-blocks.  These are the lengths before clusters and before pairs with W in tensor memory.
SHAPES = {
    (10, 6144, 146): 6.89,          # pairs, half the K-blocks in a second accumulator
    (10, 9216, 219): 10.32,         # pairs of 512 tokens, the same
    (5, 5353, 481): 6.0,
    (28, 5120, 761): 38.5,
    (69, 6272, 221): 40.1,
    (70, 4096, 190): 32.0,
    (72, 6000, 129): 47.0,
    (43, 4096, 128): 17.3,
    (43, 4096, 32): 17.3,           # clusters, two accumulators
    (60, 2176, 30): 12.4,
    (12, 1152, 28): 1.74,
    (4, 1024, 16): 1.0,
    (17, 555, 125): 4.59,
    (11, 1792, 184): 3.61,
    (14, 2304, 702): 12.0,
    (140, 4096, 32): 64.0,          # whole tiles, as long as ever
}


def blocks_added(q, nkb):
    """The same of a plan, counted out."""
    sets, steps = q["sets"], 1 if q["kernel"] >= 3 else 2               # a K-block goes to the accumulators whole, or in halves

    def cubes(blocks):
        n = [(steps * blocks + sets - 1 - s) // sets for s in range(sets)]
        assert sum(n) == steps * blocks
        return sum(x ** 3 for x in n) / steps ** 3

    total = (q["tiles"] - (q["rest"] if q["cut"] else 0)) * cubes(nkb)
    if q["cut"]:
        units = q["rest"] * nkb
        for w in range(q["sharers"]):
            a, b = units * w // q["sharers"], units * (w + 1) // q["sharers"]
            while a < b:
                end = min(b, (a // nkb + 1) * nkb)
                total += cubes(end - a)
                a = end
    return math.sqrt(total / nkb / q["tiles"])


@pytest.mark.parametrize("shape", list(SHAPES))
def test_no_accumulator_adds_more(shape):
    R, K, N = shape
    assert blocks_added(device_plan(R, K, N, wide=True), (K + 63) // 64) <= SHAPES[shape]


def test_plans_of_32_bit_results_hold_together():
    seen = set()
    for R in (1, 2, 7, 16, 43, 73, 75, 112, 149, 400):
        for K in (1, 64, 65, 200, 1000, 4096, 20000):
            for N in (1, 16, 32, 33, 64, 65, 128, 129, 192, 193, 256, 257, 384, 385, 700, 1024, 5000):
                q, nkb = device_plan(R, K, N, wide=True), (K + 63) // 64
                pairs = q["kernel"] >= 3
                slots, tokens = 74 if pairs else 148, lib().shim_pair_tile_tokens(N) if q["kernel"] == 4 else (32, 128, 256, 512)[q["kernel"]]
                seen.add((q["kernel"], q["sets"]))
                # room for the accumulators: of 128 columns, of the second accumulator of a pair, which no tile needs
                assert q["sets"] in (1, 2, 4)
                assert q["sets"] == 1 or (q["kernel"] == 0) or (q["kernel"] == 1 and q["sets"] * N <= 128) or (q["sets"] == 2 and N <= {3: 256, 4: 192}[q["kernel"]])
                assert not q["cut"] or (q["sharers"] <= q["rest"] * nkb and (1 if pairs else 2) * q["sharers"] * min(N, tokens) <= 2 * 148 * 256)
                assert q["kernel"] == 4 or q["sharers"] <= max(slots, q["rest"])
                if pairs:
                    assert not q["cut"] or (q["sharers"] == q["slices"] * q["rest"] and q["slices"] <= nkb)
                else:
                    assert q["tiles"] == q["rounds"] * slots + q["rest"] and 1 <= q["workers"] <= 148
    assert {(0, 1), (1, 1), (1, 2), (1, 4), (2, 1), (3, 1), (3, 2), (4, 1), (4, 2)} <= seen


@pytest.mark.gpu
@pytest.mark.parametrize("shape", list(SHAPES))
def test_error_against_64_bits(shape):
    from paper_2607_21985_b200 import spdp
    R, K, N = shape
    M, g = 256 * R, torch.Generator(device="cuda").manual_seed(R + K + N)
    W = (0.02 * torch.randn(M, K, generator=g, device="cuda") * (torch.rand(M, K, generator=g, device="cuda") < 0.5)).half()
    X = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    X[:, :K] = torch.randn(N, K, generator=g, device="cuda").half()
    Y = torch.full((N, M), float("nan"), device="cuda")
    h = spdp.spdp_pack_tiled_cbc(W)
    try:
        spdp.spdp_spmm(h, X[:, :K], Y)
        torch.cuda.synchronize()
        assert spdp.spdp_last_device_status(h) == 0
    finally:
        spdp.spdp_free(h)
    want = torch.cat([X[:, :K].double() @ W[r:r + 4096].double().T for r in range(0, M, 4096)], 1)
    error = float((Y.double() - want).norm() / want.norm())
    assert error <= 1e-7 * SHAPES[shape] + 1.5e-7
