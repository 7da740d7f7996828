"""The CTA-pair form of the prefill product.  It has two builds: two X tiles in flight for each accumulator, with barriers of their own, and
three, handed on with their K-block, for layers of few values; and three ways to be cut: whole tiles, whole rounds with the
tiles of the last round cut along K, and all tiles cut.  A test without a GPU compiles the rule that chooses (csrc/spmm_plan.h)
and holds it against what each shape below is there for, on the 148 SMs that the product tests run on."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# row tiles, K, tokens, sparsity -> X tiles in flight, whole tiles, cut tiles, slices of a cut tile
SHAPES = {
    (75, 1000, 300, 0.8): (6, 74, 1, 16),       # two accumulators, the second with 44 tokens
    (75, 1000, 770, 0.8): (6, 148, 2, 8),       # a second token block of 258 tokens
    (75, 2048, 700, 0.8): (6, 148, 2, 16),      # one of 188: one accumulator, the ring of X tiles moves by one per K-block
    (148, 2050, 300, 0.9): (6, 148, 0, 1),      # whole tiles only, K-blocks of two columns at the end
    (16, 4104, 300, 0.9): (6, 0, 16, 4),        # all tiles cut
    (3, 12000, 1024, 0.9): (6, 0, 6, 12),       # enough slices for the second kernel's deeper form
    (75, 1000, 770, 0.5): (4, 148, 2, 8),
    (75, 2048, 700, 0.5): (4, 148, 2, 16),
    (148, 2050, 300, 0.0): (4, 148, 0, 1),      # full columns: the ring of values holds two K-blocks
    (16, 4104, 300, 0.0): (4, 0, 16, 4),
    (3, 12000, 1024, 0.5): (4, 0, 6, 12),
}
IN_A_ROW = [(75, 2048, 300), (16, 4096, 300)]       # a call's launches beside the next call's: whole rounds and a cut rest; all tiles cut
INTO_ANY_Y = (148, 712, 300)


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    out = tmp_path_factory.mktemp("plan") / "libplan_shim.so"
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"),
                    "-o", str(out), os.path.join(ROOT, "tests", "plan_shim.cpp")], check=True)
    L = ctypes.CDLL(str(out))
    L.shim_make_plan.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 2 + [ctypes.c_void_p]
    L.shim_pair_x_tiles.argtypes = [ctypes.c_longlong] * 3

    def make(R, K, N, sms=148, may_cut=True):
        v = (ctypes.c_longlong * 7)()
        L.shim_make_plan(R, (K + 63) // 64, N, sms, may_cut, v)
        return dict(zip(("kernel", "workers", "rounds", "sharers", "slices", "tiles", "rest"), v))
    make.x_tiles = lambda R, K, sparsity: L.shim_pair_x_tiles(int(256 * R * K * (1.0 - sparsity)), R, (K + 63) // 64)
    return make


@pytest.mark.parametrize("shape", list(SHAPES))
def test_shapes_are_what_they_are_there_for(plan, shape):
    R, K, N, sparsity = shape
    q, (x_tiles, whole, cut, slices) = plan(R, K, N), SHAPES[shape]
    assert q["kernel"] == 3 and plan.x_tiles(R, K, sparsity) == x_tiles
    assert (q["tiles"] - q["rest"], q["rest"]) == (whole, cut) and q["slices"] == slices
    assert q["slices"] * q["rest"] == (q["sharers"] if cut else 0)


def test_other_shapes_take_pairs(plan):
    for shape in IN_A_ROW:
        q = plan(*shape)
        assert q["kernel"] == 3 and q["rest"] > 0
        assert plan.x_tiles(*shape[:2], 0.0) == 4 and plan.x_tiles(*shape[:2], 0.9) == 6
    assert plan(*IN_A_ROW[0])["tiles"] > plan(*IN_A_ROW[0])["rest"]
    assert plan(*INTO_ANY_Y)["kernel"] == 3 and plan(*INTO_ANY_Y)["rest"] == 0


def test_plans_hold_together(plan):
    """Every tile is computed: whole rounds and the rest make up the tiles, a cut tile has at least one K-block for each CTA that
    shares it, no cut where none is allowed, no more CTAs than the machine holds at once."""
    for sms in (2, 3, 148):
        for R in (1, 2, 7, 16, 73, 75, 149, 400):
            for K in (1, 64, 65, 1000, 4096, 20000):
                for N in (1, 16, 33, 128, 129, 256, 300, 512, 700, 1024, 5000):
                    for may_cut in (True, False):
                        q, nkb = plan(R, K, N, sms, may_cut), (K + 63) // 64
                        slots, tokens = (sms // 2 if q["kernel"] == 3 else sms), (32, 128, 256, 512)[q["kernel"]]
                        assert q["tiles"] == R * ((N + tokens - 1) // tokens)
                        cut = q["rest"] > 0 and q["sharers"] > q["rest"]
                        assert may_cut or not cut
                        assert q["sharers"] <= max(slots, q["rest"]) and (not cut or q["sharers"] <= q["rest"] * nkb)
                        if q["kernel"] == 3:
                            assert q["slices"] >= 1 and (not cut or q["sharers"] == q["slices"] * q["rest"])
                        else:
                            assert q["tiles"] == q["rounds"] * slots + q["rest"] and 1 <= q["workers"] <= sms


# ---- the products, on the GPU ----

@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp
    spdp.lib()
    return spdp


def integers(M, K, N, sparsity, seed):
    """W, X and their product: |sums| <= 12000 * 8 < 2^24, so that every partial sum is exact."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = torch.randint(1, 5, (M, K), generator=g, device="cuda").half() * (2 * torch.randint(0, 2, (M, K), generator=g, device="cuda") - 1).half()
    W[torch.rand(M, K, generator=g, device="cuda") < sparsity] = 0
    X = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")            # a token starts on a 16-byte boundary
    X[:, :K] = torch.randint(-2, 3, (N, K), generator=g, device="cuda").half()
    return W, X[:, :K], X[:, :K].double() @ W.double().T


@pytest.mark.gpu
@pytest.mark.parametrize("shape", list(SHAPES))
def test_products_are_exact(S, shape):
    R, K, N, sparsity = shape
    M = 256 * R - 37
    W, X, want = integers(M, K, N, sparsity, R * K + N)
    h = S.spdp_pack_tiled_cbc(W)
    try:
        for dt in (torch.float32, torch.float16):
            Y = torch.full((N, M), float("nan"), dtype=dt, device="cuda")
            S.spdp_spmm(h, X, Y)
            torch.cuda.synchronize()
            assert S.spdp_last_device_status(h) == 0
            assert torch.equal(Y, want.to(dt))
    finally:
        S.spdp_free(h)


@pytest.mark.gpu
@pytest.mark.parametrize("R,K,N", IN_A_ROW)
@pytest.mark.parametrize("sparsity", [0.0, 0.9])
def test_calls_in_a_row(S, R, K, N, sparsity):
    """Calls in a row start beside one another; in the second and third pass a copy just before the call makes its input.
    Full columns: the ring of stored values is full before the call ahead has ended."""
    M = 256 * R
    W, X0, want0 = integers(M, K, N, sparsity, R)
    h = S.spdp_pack_tiled_cbc(W)
    try:
        X, want = [X0, -X0, X0.flip(0).contiguous(), (2 * X0).contiguous()], [want0, -want0, want0.flip(0), 2 * want0]
        buf = torch.empty((N, K), dtype=torch.float16, device="cuda")
        Y = torch.empty((4, N, M), dtype=torch.float32, device="cuda")
        for repeat in range(3):
            Y.fill_(float("nan"))
            for x, y in zip(X, Y):
                if repeat:
                    buf.copy_(x)
                S.spdp_spmm(h, buf if repeat else x, y)
            torch.cuda.synchronize()
            for y, ref in zip(Y, want):
                assert torch.equal(y.double(), ref)
        assert S.spdp_last_device_status(h) == 0
    finally:
        S.spdp_free(h)


@pytest.mark.gpu
@pytest.mark.parametrize("dt", [torch.float16, torch.float32])
def test_whole_tiles_into_any_y(S, dt):
    """Whole tiles are stored in fours where Y allows it: a base off the boundary of four elements with a row stride that is a
    multiple of four, a stride that is none, and rows that end inside a four.  Nothing outside Y is written."""
    R, K, N = INTO_ANY_Y
    M = 256 * R - 6
    W, X, want = integers(M, K, N, 0.5, 9)
    want = want.to(dt)
    h = S.spdp_pack_tiled_cbc(W)
    try:
        for pad, at in ((2, 0), (2, 1), (2, 2), (6, 3), (2, 4), (0, 0), (3, 0), (3, 1)):
            buf = torch.full((N * (M + pad) + at + 8,), 7.0, dtype=dt, device="cuda")
            Y = buf[at:at + N * (M + pad)].view(N, M + pad)
            S.spdp_spmm(h, X, Y[:, :M])
            torch.cuda.synchronize()
            assert torch.equal(Y[:, :M], want), (pad, at)
            assert bool((Y[:, M:] == 7.0).all()) and bool((buf[:at] == 7.0).all()) and bool((buf[at + N * (M + pad):] == 7.0).all())
        assert S.spdp_last_device_status(h) == 0
    finally:
        S.spdp_free(h)
