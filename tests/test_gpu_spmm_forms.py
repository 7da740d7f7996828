"""Prefill products by every form and cut that the library takes on a device of 148 SMs: one CTA per tile of 32, 128 or 256 tokens, whole, cut with a second
kernel, with ranges that cross tiles; clusters of every size that the rule chooses; CTA pairs of 512 tokens with both numbers of X tiles in flight and
one or two accumulators in the last token block; pairs with W in tensor memory.  What a shape is there for is held, without a GPU, against the rule with
the cluster counts that the library hands it; that is the rule for 16-bit results (32-bit ones are cut more finely, or added to several accumulators in
turn, and run beside them).  Whole numbers, so that sums are exact in any order and the results have to be equal."""
import pytest

torch = pytest.importorskip("torch")

from device_plan import device_plan, lib, pair_x_tiles

# row tiles, K, tokens, sparsity -> kernel (0, 1, 2: 32, 128, 256 tokens), tiles that are whole, tiles left for the last round, CTAs that share those, ranges cross tiles
ONE = {
    (20, 100, 2, 0.5): (0, 0, 20, 20, False),
    (150, 64, 5, 0.5): (0, 148, 2, 2, False),
    (3, 1900, 31, 0.5): (0, 0, 3, 45, False),
    (8, 1250, 128, 0.9): (0, 0, 32, 128, False),         # four token blocks
    (82, 1000, 100, 0.5): (1, 0, 82, 82, False),
    (250, 1280, 20, 0.0): (1, 148, 102, 148, True),
    (65, 3000, 5, 0.9): (1, 0, 65, 148, True),
    (80, 1700, 250, 0.5): (2, 0, 80, 80, False),
    (8, 1000, 129, 0.5): (2, 0, 8, 64, False),
    (149, 300, 150, 0.0): (2, 148, 1, 5, False),
    (76, 500, 900, 0.5): (2, 296, 8, 32, False),         # four token blocks, the last one of 132 tokens
    (75, 1700, 129, 0.9): (2, 0, 75, 148, True),
    (112, 8192, 250, 0.5): (2, 0, 112, 148, True),
    (230, 1500, 150, 0.5): (2, 148, 82, 148, True),
}
# -> CTAs of a cluster, of 32 (0) or 128 (1) tokens
CLUSTERS = {
    (35, 300, 5, 0.5): (2, 0),
    (4, 300, 100, 0.5): (3, 0),
    (17, 1000, 5, 0.5): (4, 0),
    (17, 600, 31, 0.0): (5, 0),
    (6, 1000, 64, 0.5): (6, 0),
    (10, 1250, 20, 0.5): (7, 0),
    (9, 1000, 31, 0.9): (8, 0),
    (8, 1700, 7, 0.5): (9, 0),
    (7, 1900, 2, 0.5): (10, 0),                         # more CTAs than tokens
    (74, 2000, 128, 0.0): (2, 1),
    (43, 4096, 128, 0.6): (3, 1),
    (6, 700, 800, 0.5): (3, 1),                         # seven token blocks, the last one of 32 tokens
    (33, 3000, 128, 0.9): (4, 1),
    (26, 1900, 100, 0.5): (5, 1),
    (22, 3000, 128, 0.5): (6, 1),
    (14, 4096, 127, 0.5): (8, 1),
    (15, 11008, 112, 0.9): (9, 1),
}
# -> kernel (3: 512 tokens, 4: W in tensor memory), X tiles in flight, whole tiles, cut tiles, slices of a cut tile, accumulators in the last token block
PAIRS = {
    (51, 100, 200, 0.0): (3, 4, 51, 0, 1, 1),
    (51, 100, 200, 0.9): (3, 6, 51, 0, 1, 1),
    (38, 64, 100, 0.5): (3, 4, 38, 0, 1, 1),            # one K-block
    (148, 712, 300, 0.9): (3, 6, 148, 0, 1, 2),
    (37, 5000, 700, 0.0): (3, 4, 74, 0, 1, 1),          # full columns: the ring of values holds two K-blocks
    (37, 5000, 700, 0.8): (3, 6, 74, 0, 1, 1),          # the ring of X tiles moves by one per K-block
    (14, 1250, 150, 0.5): (3, 4, 0, 14, 4, 1),
    (14, 1250, 150, 0.9): (3, 6, 0, 14, 4, 1),
    (27, 2100, 385, 0.0): (3, 4, 0, 27, 2, 2),
    (27, 2100, 385, 0.9): (3, 6, 0, 27, 2, 2),
    (75, 500, 385, 0.5): (3, 4, 74, 1, 8, 2),
    (75, 640, 400, 0.9): (3, 6, 74, 1, 10, 2),
    (92, 2100, 800, 0.5): (3, 4, 148, 36, 2, 2),
    (75, 1000, 770, 0.8): (3, 6, 148, 2, 8, 2),
    (3, 12000, 1024, 0.5): (3, 4, 0, 6, 12, 2),         # enough slices for the second kernel's deeper form
    (3, 12000, 1024, 0.9): (3, 6, 0, 6, 12, 2),
    (75, 1000, 300, 0.8): (4, 6, 74, 1, 8, 2),
    (75, 2048, 700, 0.5): (4, 4, 148, 2, 16, 2),
    (5, 4096, 512, 0.5): (4, 4, 0, 10, 7, 1),
}
# 32-bit results -> kernel, CTAs of a cluster, accumulators that the K-blocks go to in turn (some of the shapes above have two)
SETS = {
    (6, 1000, 40, 0.5): (0, 6, 4),
    (29, 300, 17, 0.0): (0, 2, 4),
    (7, 2500, 31, 0.5): (1, 1, 4),
    (12, 1000, 40, 0.9): (1, 4, 2),
    (14, 1250, 150, 0.9): (3, 1, 2),
    (14, 4096, 127, 0.5): (4, 1, 2),
}


@pytest.mark.parametrize("shape", list(ONE))
def test_shapes_of_one_cta(shape):
    q = device_plan(*shape[:3])
    assert (q["kernel"], q["tiles"] - q["rest"], q["rest"], q["sharers"], q["crosses"]) == ONE[shape] and q["cluster"] == 1


@pytest.mark.parametrize("shape", list(CLUSTERS))
def test_shapes_of_clusters(shape):
    q = device_plan(*shape[:3])
    assert (q["cluster"], q["kernel"]) == CLUSTERS[shape]


@pytest.mark.parametrize("shape", list(PAIRS))
def test_shapes_of_pairs(shape):
    R, K, N, sparsity = shape
    q = device_plan(R, K, N)
    if q["kernel"] == 3:
        last, acc = (N - 1) % 512 + 1, 256
    else:
        tokens, acc = lib().shim_pair_tile_tokens(N), lib().shim_pair_acc_tokens(N)
        last = (N - 1) % tokens + 1
    assert (q["kernel"], pair_x_tiles(R, K, sparsity), q["tiles"] - q["rest"], q["rest"], q["slices"], 2 if last > acc else 1) == PAIRS[shape]


@pytest.mark.parametrize("shape", list(SETS))
def test_shapes_of_several_accumulators(shape):
    q = device_plan(*shape[:3], wide=True)
    assert (q["kernel"], q["cluster"], q["sets"]) == SETS[shape]


# ---- the products, on the GPU ----

@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp
    spdp.lib()
    return spdp


def integers(R, K, N, sparsity, short=0):
    """A packed matrix of 256 R - short rows, X, and their product: |sums| <= 12000 * 8 < 2^24, so that every partial sum is exact."""
    from paper_2607_21985_b200 import spdp
    M, g = 256 * R - short, torch.Generator(device="cuda").manual_seed(R * K + N)
    W = torch.randint(1, 5, (M, K), generator=g, device="cuda").half() * (2 * torch.randint(0, 2, (M, K), generator=g, device="cuda") - 1).half()
    W[torch.rand(M, K, generator=g, device="cuda") < sparsity] = 0
    X = torch.zeros(N, (K + 7) // 8 * 8, dtype=torch.float16, device="cuda")            # a token starts on a 16-byte boundary
    X[:, :K] = torch.randint(-2, 3, (N, K), generator=g, device="cuda").half()
    return spdp.spdp_pack_tiled_cbc(W), X[:, :K], (X[:, :K].double() @ W.double().T).float()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", sorted(set(ONE) | set(CLUSTERS) | set(PAIRS) | set(SETS)))
def test_products_are_exact(S, shape):
    """Calls in a row, which start beside one another and find an earlier call's sums in the scratch memory; in the last ones a copy just before the
    call makes its input."""
    R, K, N, sparsity = shape
    h, X, want = integers(R, K, N, sparsity, short=37)
    M = 256 * R - 37
    try:
        buf, minus = (torch.zeros(N, X.stride(0), dtype=torch.float16, device="cuda")[:, :K] for _ in range(2))
        minus.copy_(-X)
        for dt, ldy in ((torch.float32, M), (torch.float16, M + 3)):
            Y = [torch.full((N, ldy), float("nan"), dtype=dt, device="cuda")[:, :M] for _ in range(4)]
            S.spdp_spmm(h, X, Y[0])
            S.spdp_spmm(h, minus, Y[1])
            for y, sign in ((Y[2], 1), (Y[3], -1)):
                buf.copy_(X if sign > 0 else minus)
                S.spdp_spmm(h, buf, y)
            torch.cuda.synchronize()
            assert S.spdp_last_device_status(h) == 0
            for y, sign in zip(Y, (1, -1, 1, -1)):
                assert torch.equal(y, (sign * want).to(dt))
    finally:
        S.spdp_free(h)


class _DeviceWords:
    """int32 view of device memory at an address."""
    def __init__(self, address, n):
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<i4", data=(address, False), version=3)


# cut tiles that a second kernel or the CTAs of a cluster add up
REFUSED = [(8, 1250, 128, 0.9), (65, 3000, 5, 0.9), (8, 1000, 129, 0.5), (75, 1700, 129, 0.9), (14, 1250, 150, 0.9), (27, 2100, 385, 0.0), (17, 600, 31, 0.0),
           (9, 1000, 31, 0.9), (7, 1900, 2, 0.5), (74, 2000, 128, 0.0), (43, 4096, 128, 0.6), (6, 700, 800, 0.5), (14, 4096, 127, 0.5), (15, 11008, 112, 0.9)]


@pytest.mark.gpu
@pytest.mark.parametrize("dt", ["float16", "float32"])
@pytest.mark.parametrize("shape", REFUSED)
def test_a_refused_tile_stays_unwritten(S, shape, dt):
    """A TileOffset word that cannot be (the kernels' own check refuses the K-blocks at it and copies nothing): the status says so, and the tile's outputs stay
    unwritten although other CTAs have left their partial sums of it and the scratch memory holds an earlier call's."""
    R, K, N, sparsity = shape
    h, X, want = integers(R, K, N, sparsity)
    want = want.to(getattr(torch, dt))
    try:
        def call():
            Y = torch.full((N, 256 * R), float("nan"), dtype=want.dtype, device="cuda")
            S.spdp_spmm(h, X, Y)
            torch.cuda.synchronize()
            return Y, S.spdp_last_device_status(h)
        Y, status = call()
        assert status == 0 and torch.equal(Y, want)
        info, C = S.spdp_get_info(h), (K + 15) // 16
        words = torch.as_tensor(_DeviceWords(info.tileoffset_dev, info.NGT + 1), device="cuda")
        at = 3 * C + 4 * (C // 8)                              # between two K-blocks in the middle of row tile 3
        good = int(words[at])
        words[at] = -1                                         # 2^32 - 1 values: beyond the array
        torch.cuda.synchronize()                               # the kernels may read the matrix ahead of the stream
        Y, status = call()
        words[at] = good
        torch.cuda.synchronize()
        assert status == S.SPDP_ERR_OVERFLOW
        assert bool(torch.isnan(Y[:, 768:1024]).all())
        assert torch.equal(Y[:, :512], want[:, :512]) and torch.equal(Y[:, 1280:], want[:, 1280:])      # a CTA may share the neighbouring tiles, not these
        Y, status = call()
        assert status == 0 and torch.equal(Y, want)
    finally:
        S.spdp_free(h)


# clusters, ranges that cross tiles, cut pairs of both kinds
OTHERWISE = [(35, 300, 5, 0.5), (17, 600, 31, 0.0), (43, 4096, 128, 0.6), (75, 1700, 129, 0.9), (14, 1250, 150, 0.5), (5, 4096, 512, 0.5)]


@pytest.mark.gpu
@pytest.mark.parametrize("dt", [torch.float16, torch.float32])
@pytest.mark.parametrize("shape", OTHERWISE)
def test_in_a_graph_and_on_two_streams(S, shape, dt):
    """A captured pair of calls, whose partial sums are memory of the graph, replayed on new inputs with calls on two streams in between."""
    R, K, N, sparsity = shape
    h, X, want = integers(R, K, N, sparsity)
    want = want.to(dt)
    other = torch.cuda.Stream()
    try:
        buf, minus = (torch.zeros(N, X.stride(0), dtype=torch.float16, device="cuda")[:, :K] for _ in range(2))
        minus.copy_(-X)
        Y, beside = torch.empty_like(want), [torch.empty_like(want) for _ in range(2)]
        S.spdp_spmm(h, buf, Y)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            S.spdp_spmm(h, buf, Y)
            S.spdp_spmm(h, buf, Y)
        for x, sign in ((X, 1), (minus, -1), (X, 1)):
            buf.copy_(x)
            for y in [Y] + beside:
                y.fill_(float("nan"))
            torch.cuda.synchronize()
            graph.replay()
            S.spdp_spmm(h, minus, beside[0])
            S.spdp_spmm(h, X, beside[1], stream=other)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(Y, sign * want) and torch.equal(beside[0], -want) and torch.equal(beside[1], want)
        assert S.spdp_last_device_status(h) == 0
        del graph
    finally:
        S.spdp_free(h)


@pytest.mark.gpu
@pytest.mark.parametrize("dt", [torch.float16, torch.float32])
@pytest.mark.parametrize("shape", OTHERWISE)
def test_into_any_y(S, shape, dt):
    """Rows that end inside a group that is stored at once, a Y whose base and row stride are off that group's boundary: nothing outside Y is written."""
    R, K, N, sparsity = shape
    M = 256 * R - 6
    h, X, want = integers(R, K, N, sparsity, short=6)
    try:
        for pad, at in ((0, 0), (1, 1), (2, 2), (3, 4), (5, 3)):
            buf = torch.full((N * (M + pad) + at + 8,), 7.0, dtype=dt, device="cuda")
            Y = buf[at:at + N * (M + pad)].view(N, M + pad)
            S.spdp_spmm(h, X, Y[:, :M])
            torch.cuda.synchronize()
            assert torch.equal(Y[:, :M], want.to(dt))
            assert bool((Y[:, M:] == 7.0).all()) and bool((buf[:at] == 7.0).all()) and bool((buf[at + N * (M + pad):] == 7.0).all())
        assert S.spdp_last_device_status(h) == 0
    finally:
        S.spdp_free(h)
