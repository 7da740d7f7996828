"""How a prefill call is cut on a device that runs thread-block clusters: clusters that add a tile's sums themselves, and CTA pairs with decoded W in
tensor memory.  The rule (csrc/spmm_plan.h) is compiled for the host and held against what its kernels can do, with the
cluster counts of a device of 148 SMs; the products of shapes that take the pairs, whole and cut, run on the GPU."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RESIDENT = [148, 148, 74, 45, 33, 26, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7]

# rows, K, tokens, sparsity of calls of pairs with W in tensor memory
PAIRS = [
    (4001, 4098, 300, 0.3),         # all tiles cut, two accumulators
    (15300, 1000, 256, 0.6),        # whole tiles, one accumulator of 256 tokens
    (15300, 1000, 384, 0.9),        # two accumulators of 192, three X tiles for each
    (15300, 1000, 257, 0.0),        # two of 160, the second with 97 tokens; full columns: the ring holds few K-blocks
    (19100, 1000, 384, 0.5),        # one round and a tile more, cut
    (28672, 8192, 300, 0.7),        # the last tiles in more slices than the device holds at once
    (4096, 4096, 700, 0.5),         # two token blocks
    (3000, 3000, 600, 0.8),
]


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    out = tmp_path_factory.mktemp("plan") / "libplan_device_shim.so"
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"),
                    "-o", str(out), os.path.join(ROOT, "tests", "plan_device_shim.cpp")], check=True)
    L = ctypes.CDLL(str(out))
    L.shim_device_plan.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] + [ctypes.c_void_p] * 2
    L.shim_pair_acc_tokens.argtypes = L.shim_pair_tile_tokens.argtypes = [ctypes.c_longlong]

    def make(R, K, N, sms=148, resident=RESIDENT):
        v = (ctypes.c_longlong * 8)()
        L.shim_device_plan(R, (K + 63) // 64, N, sms, (ctypes.c_int * 17)(*resident), v)
        return dict(zip(("kernel", "workers", "rounds", "sharers", "slices", "tiles", "rest", "cluster"), v))
    make.lib = L
    return make


def test_tokens_of_pairs(plan):
    for N in list(range(1, 1200)) + [4000, 10 ** 6]:
        acc, tile = plan.lib.shim_pair_acc_tokens(N), plan.lib.shim_pair_tile_tokens(N)
        assert acc % 32 == 0 and (tile == acc <= 256 or tile == 2 * acc <= 384)         # units of the instruction, room in tensor memory
        assert -(-N // tile) == -(-N // 384)                                            # no more tiles than there have to be


@pytest.mark.parametrize("resident", [RESIDENT, [0] * 17])
def test_plans_hold_together(plan, resident):
    """Every tile is computed, no CTA has more than it can do, and no more CTAs wait for one another than the device holds at once."""
    seen = set()
    for sms in (2, 3, 148):
        for R in (1, 2, 7, 16, 43, 73, 75, 112, 149, 400):
            for K in (1, 64, 65, 1000, 4096, 20000):
                for N in (1, 16, 33, 100, 128, 129, 200, 256, 300, 384, 385, 512, 700, 1024, 5000):
                    q, nkb = plan(R, K, N, sms, resident if sms == 148 else [0] * 17), (K + 63) // 64
                    pairs = q["kernel"] >= 3
                    tokens = plan.lib.shim_pair_tile_tokens(N) if q["kernel"] == 4 else (32, 128, 256, 512)[q["kernel"]]
                    slots, cut = sms // 2 if pairs else sms, q["rest"] > 0 and q["sharers"] > q["rest"]
                    seen.add((q["kernel"], q["cluster"] > 1))
                    assert q["tiles"] == R * -(-N // tokens)
                    assert not cut or q["sharers"] <= q["rest"] * nkb
                    assert not cut or (1 if pairs else 2) * q["sharers"] * min(N, tokens) <= 2 * 148 * 256       # 77 MB of scratch memory
                    assert q["kernel"] == 4 or q["sharers"] <= max(slots, q["rest"])
                    if pairs:
                        assert q["cluster"] == 1 and q["slices"] >= 1 and (not cut or q["sharers"] == q["slices"] * q["rest"]) and q["slices"] <= max(nkb, 1)
                    else:
                        assert q["tiles"] == q["rounds"] * slots + q["rest"] and 1 <= q["workers"] <= sms
                    if q["cluster"] > 1:
                        c, each = q["cluster"], min(N, tokens)
                        assert q["kernel"] <= 1 and q["rounds"] == 0 and c <= 16 and c <= nkb and q["rest"] <= resident[c]
                        assert q["workers"] == q["sharers"] == c * q["rest"] and (c - 1) * -(-each // c) <= 126
    assert resident is not RESIDENT or {(0, True), (1, True), (4, False)} <= seen
    assert resident is RESIDENT or not any(c for _, c in seen)


def test_every_cta_of_a_cluster_has_a_k_block(plan):
    """Whatever sizes of clusters a device holds, sizes in between not among them."""
    for only in range(2, 17):
        resident = [148, 148] + [7 if c == only else 0 for c in range(2, 17)]
        for R in (1, 2, 3, 5, 7):
            for nkb in range(1, 20):
                for N in (1, 7, 16, 33, 128):
                    assert plan(R, 64 * nkb, N, resident=resident)["cluster"] <= nkb


def test_shapes_take_the_pairs(plan):
    whole, more, cut = 0, 0, 0
    for M, K, N, _ in PAIRS:
        q = plan(-(-M // 256), K, N)
        assert q["kernel"] == 4
        whole += q["tiles"] > q["rest"]
        cut += q["rest"] > 0
        more += q["rest"] > 0 and q["sharers"] > 74
    assert whole >= 3 and cut >= 3 and more >= 1


@pytest.mark.gpu
@pytest.mark.parametrize("M,K,N,sparsity", PAIRS)
def test_products_are_exact(M, K, N, sparsity):
    from paper_2607_21985_b200 import spdp
    g = torch.Generator(device="cuda").manual_seed(M + K + N)
    W = torch.randint(1, 5, (M, K), generator=g, device="cuda").half() * (2 * torch.randint(0, 2, (M, K), generator=g, device="cuda") - 1).half()
    W[torch.rand(M, K, generator=g, device="cuda") < sparsity] = 0
    X = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")
    X[:, :K] = torch.randint(-2, 3, (N, K), generator=g, device="cuda").half()
    want = X[:, :K].double() @ W.double().T                 # |sums| <= 8 * 8192 < 2^24: exact in any order
    h = spdp.spdp_pack_tiled_cbc(W)
    try:
        for ldy in (M, M + 1, (M + 3) // 4 * 4):
            out = []
            for _ in range(3):                              # calls in a row start beside one another
                Y = torch.full((N, ldy), float("nan"), device="cuda")[:, :M]
                spdp.spdp_spmm(h, X[:, :K], Y)
                out.append(Y)
            torch.cuda.synchronize()
            assert spdp.spdp_last_device_status(h) == 0
            assert all(torch.equal(Y.double(), want) for Y in out)
    finally:
        spdp.spdp_free(h)
