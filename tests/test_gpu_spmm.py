"""Prefill product on the packed handle (spdp_spmm, Sec. 4.3) against the oracle's dense fp64 definition."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import spdp_oracle as O
from paper_2607_21985_b200 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp
    spdp.lib()
    return spdp


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def run(S, h, X, M, ydtype=torch.float32):
    Y = torch.full((X.shape[0], M), float("nan"), dtype=ydtype, device="cuda")      # poison: every entry must be written
    S.spdp_spmm(h, dev(X), Y)
    torch.cuda.synchronize()
    assert S.spdp_last_device_status(h) == 0
    return Y.float().cpu().numpy().astype(np.float64)


def check(Y, Y_ref, S_ref):
    err = np.abs(Y - Y_ref)
    tol = O.tolerance(S_ref)                       # |y - y_ref| <= 1e-3 * S + 1e-5
    assert np.all(err <= tol), f"worst error/tolerance {np.nanmax(err / tol):.3g}"


@pytest.mark.parametrize("M,K,sp,seed", [(256, 16, 0.5, 1), (300, 40, 0.3, 2), (1, 8, 0.0, 3), (257, 24, 0.5, 4),
                                         (1024, 1024, 0.5, 5), (768, 4400, 0.7, 6), (2304, 528, 0.9, 7),
                                         (512, 72, 0.0, 8)])
@pytest.mark.parametrize("N", [1, 16, 128, 300])
def test_spmm_matches_oracle(S, M, K, sp, seed, N):
    rw, rx = WL._rngs(seed)
    W = WL.prune_global_magnitude(WL.normal_weights(rw, M, K), sp).astype(np.float16)
    X = rx.standard_normal((N, K), dtype=np.float32).astype(np.float16)
    Y_ref, S_ref = O.spmm_ref(W, X)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        for dt in (torch.float32, torch.float16):
            check(run(S, h, X, M, dt), Y_ref, S_ref)
        assert np.array_equal(run(S, h, X, M), run(S, h, X, M))          # the same bits from call to call
    finally:
        S.spdp_free(h)


def test_spmm_exact_on_integers_and_strided_tensors(S):
    rng = np.random.Generator(np.random.PCG64(61))
    M, K, N = 700, 904, 37
    W = rng.integers(-8, 9, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.6] = 0
    X = rng.integers(-4, 5, (N, K)).astype(np.float16)
    Y_ref, _ = O.spmm_ref(W, X)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        assert np.array_equal(run(S, h, X, M), Y_ref)                     # every partial sum is an exact integer
        Xd = torch.zeros((N, K + 24), dtype=torch.float16, device="cuda")  # padded row strides (a multiple of 8 elements)
        Xd[:, :K] = dev(X)
        Yd = torch.full((N, M + 5), float("nan"), dtype=torch.float32, device="cuda")
        S.spdp_spmm(h, Xd[:, :K], Yd[:, :M])
        torch.cuda.synchronize()
        out = Yd.cpu().numpy()
        assert np.array_equal(out[:, :M].astype(np.float64), Y_ref) and np.all(np.isnan(out[:, M:]))
        # one token agrees with the decode call without dynamic pruning
        y1 = torch.empty(M, dtype=torch.float32, device="cuda")
        S.spdp_spmspv(h, dev(X[3]), O.DP_NONE, 0.0, y1)
        torch.cuda.synchronize()
        assert np.array_equal(y1.cpu().numpy().astype(np.float64), Y_ref[3])
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("R,K,N", [(80, 200, 1), (80, 200, 256), (80, 72, 300), (40, 136, 600), (30, 264, 700), (3, 520, 1100),
                                   (76, 264, 100), (150, 520, 300), (75, 2048, 700)])
def test_spmm_both_kernels(S, R, K, N):
    """The launch chooses among CTAs of 32, 128 and 256 tokens and CTA pairs of 512 by an estimate of each one's time.  On
    148 SMs these shapes reach all four, with one and with several token blocks, ragged in M, K and N, without a cut in the
    one-CTA forms.  The last two take pairs and leave a last round of two: those tiles are cut along K and their slices added by
    a second kernel.  (Cut tiles of the one-CTA forms: test_spmm_work_cuts.)"""
    rw, rx = WL._rngs(100 + R)
    M = 256 * R - 37
    W = WL.prune_global_magnitude(WL.normal_weights(rw, M, K), 0.5).astype(np.float16)
    X = rx.standard_normal((N, K), dtype=np.float32).astype(np.float16)
    Y_ref, S_ref = O.spmm_ref(W, X)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        y = run(S, h, X, M)
        check(y, Y_ref, S_ref)
        check(run(S, h, X, M, torch.float16), Y_ref, S_ref)
        assert np.array_equal(y, run(S, h, X, M))                       # the same bits from call to call
    finally:
        S.spdp_free(h)


def test_spmm_rejects_bad_arguments(S):
    h = S.spdp_pack_tiled_cbc(torch.zeros((256, 32), dtype=torch.float16, device="cuda"))
    try:
        X = torch.zeros((4, 40), dtype=torch.float16, device="cuda")
        Y = torch.zeros((4, 256), dtype=torch.float32, device="cuda")
        with pytest.raises(S.SpdpError, match="INVALID_ARG"):
            S.spdp_spmm(h, X[:, 1:33], Y)                                  # X not 16-byte aligned
        with pytest.raises(S.SpdpError, match="INVALID_ARG"):
            S.spdp_spmm(h, X[:, :32], Y[:, :100].contiguous())             # fewer than M outputs per token
        Xo = torch.zeros((4, 35), dtype=torch.float16, device="cuda")
        with pytest.raises(S.SpdpError, match="INVALID_ARG"):
            S.spdp_spmm(h, Xo[:, :32], Y)                                  # row stride not a multiple of 8 elements
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("R,K,N", [(150, 520, 20), (149, 1000, 30), (5, 5000, 40), (3, 640, 33), (1, 12800, 128), (1, 130, 256),
                                   (7, 3000, 129), (2, 20000, 1), (37, 64, 513), (2, 65, 31),
                                   (50, 1280, 20), (50, 1280, 60), (50, 2000, 200), (250, 1280, 20)])
@pytest.mark.parametrize("sp", [0.0, 0.5, 0.95])
def test_spmm_work_cuts(S, R, K, N, sp):
    """How the work is cut over CTAs: whole rounds plus a shared rest (150, 149 and 250 row tiles), CTA ranges that start in one
    row tile and end in the next (50 and 250 row tiles on 148 SMs, with 32, 128 and 256 tokens per CTA), a whole number of CTAs per
    row tile (5, 7), many on one (1, 2), K-blocks of one column, full columns (the ring of stored values at its fullest)
    and nearly empty ones.  Integers: every partial sum is exact."""
    rng = np.random.Generator(np.random.PCG64(R * 1000 + K))
    M = 256 * R - 3
    W = rng.integers(-4, 5, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < sp] = 0
    X = rng.integers(-2, 3, (N, K)).astype(np.float16)
    Y_ref = X.astype(np.float32) @ W.astype(np.float32).T              # exact: |sums| <= 20000 * 8 < 2^24
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        Xd = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")     # a token starts on a 16-byte boundary
        Xd[:, :K] = dev(X)
        Y = torch.full((N, M), float("nan"), dtype=torch.float32, device="cuda")
        S.spdp_spmm(h, Xd[:, :K], Y)
        torch.cuda.synchronize()
        assert S.spdp_last_device_status(h) == 0
        assert np.array_equal(Y.cpu().numpy(), Y_ref)
    finally:
        S.spdp_free(h)


class _DeviceWords:
    """int32 view of device memory at an address."""
    def __init__(self, address, n):
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<i4", data=(address, False), version=3)


@pytest.mark.parametrize("R,K,N", [(6, 4096, 32), (6, 8192, 40), (5, 4096, 512), (6, 8192, 512), (16, 4098, 300)])
def test_spmm_leaves_a_refused_tile_unwritten(S, R, K, N):
    """A TileOffset word that cannot be (the kernel's own check refuses the K-blocks at it and copies nothing): the status says
    so, and the tile's outputs stay unwritten although other CTAs have left their partial sums of it and the scratch memory
    still holds an earlier call's.  The shapes are cut along K, with 32, 128 and 256 tokens per CTA and with CTA pairs."""
    rng = np.random.Generator(np.random.PCG64(R))
    M, C = 256 * R, (K + 15) // 16
    W = rng.integers(-4, 5, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.5] = 0
    X = torch.zeros((N, (K + 7) // 8 * 8), dtype=torch.float16, device="cuda")
    X[:, :K] = dev(rng.integers(-2, 3, (N, K)).astype(np.float16))
    Y_ref = X[:, :K].float().cpu().numpy() @ W.astype(np.float32).T
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        def call():
            Y = torch.full((N, M), float("nan"), dtype=torch.float32, device="cuda")
            S.spdp_spmm(h, X[:, :K], Y)
            torch.cuda.synchronize()
            return Y.cpu().numpy(), S.spdp_last_device_status(h)
        Y, status = call()
        assert status == 0 and np.array_equal(Y, Y_ref)
        info = S.spdp_get_info(h)
        words = torch.as_tensor(_DeviceWords(info.tileoffset_dev, info.NGT + 1), device="cuda")
        at = 3 * C + 4 * (C // 8)                              # between two K-blocks in the middle of row tile 3
        good = int(words[at])
        words[at] = -1                                         # 2^32 - 1 values: beyond the array
        torch.cuda.synchronize()                               # the kernels may read the matrix ahead of the stream
        Y, status = call()
        words[at] = good
        torch.cuda.synchronize()
        assert status == S.SPDP_ERR_OVERFLOW
        assert np.isnan(Y[:, 768:1024]).all()
        far = np.r_[0:512, 5 * 256:M]
        assert np.array_equal(Y[:, far], Y_ref[:, far])        # a CTA may share the neighbouring tiles, not these
        Y, status = call()
        assert status == 0 and np.array_equal(Y, Y_ref)
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("R,K,N", [(20, 4096, 200), (20, 4096, 30), (37, 1024, 128), (6, 8192, 512)])
@pytest.mark.parametrize("sp", [0.0, 0.9])
def test_spmm_calls_in_a_row(S, R, K, N, sp):
    """Calls in a row start beside one another; in the second and third pass a copy just before the call makes its input.
    Full columns: the ring of stored values holds two K-blocks, so the copies stop before the call ahead has ended."""
    rng = np.random.Generator(np.random.PCG64(R))
    M = 256 * R
    W = rng.integers(1, 5, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < sp] = 0
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        X = [dev(rng.integers(-2, 3, (N, K)).astype(np.float16)) for _ in range(4)]
        buf = torch.empty((N, K), dtype=torch.float16, device="cuda")
        Wd = dev(W).double()
        want = [x.double() @ Wd.T for x in X]
        Y = torch.empty((4, N, M), dtype=torch.float32, device="cuda")
        for repeat in range(3):
            Y.fill_(float("nan"))
            for x, y in zip(X, Y):
                if repeat:
                    buf.copy_(x)
                S.spdp_spmm(h, buf if repeat else x, y)
            torch.cuda.synchronize()
            for y, ref in zip(Y, want):
                assert torch.equal(y.double(), ref)            # integers: every sum is exact
        assert S.spdp_last_device_status(h) == 0
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("R,K,N", [(6, 8192, 512), (43, 4096, 200), (8, 4096, 1024)])
def test_spmm_without_memory_for_partial_sums(S, R, K, N):
    """Shapes whose tiles are cut along K (75, 61 and 34 MB of partial sums), called while the device has less memory than that
    left: whole tiles then, same results."""
    rng = np.random.Generator(np.random.PCG64(R))
    M = 256 * R
    W = rng.integers(-4, 5, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.5] = 0
    X = dev(rng.integers(-2, 3, (N, K)).astype(np.float16))
    want = torch.from_numpy(X.float().cpu().numpy() @ W.astype(np.float32).T)
    h = S.spdp_pack_tiled_cbc(dev(W))
    Y = torch.full((2, N, M), float("nan"), dtype=torch.float32, device="cuda")
    hold = []
    try:
        S.spdp_free(None)                                      # the scratch memory that the library keeps
        torch.cuda.empty_cache()
        for piece in (1 << 30, 64 << 20, 8 << 20):
            while torch.cuda.mem_get_info()[0] > piece + (16 << 20):
                hold.append(torch.empty(min(torch.cuda.mem_get_info()[0] - (16 << 20), 16 << 30) // piece * piece, dtype=torch.uint8, device="cuda"))
        assert torch.cuda.mem_get_info()[0] < 30 << 20
        S.spdp_spmm(h, X, Y[0])
        torch.cuda.synchronize()
        hold.clear()
        torch.cuda.empty_cache()
        S.spdp_spmm(h, X, Y[1])
        torch.cuda.synchronize()
        assert S.spdp_last_device_status(h) == 0
    finally:
        hold.clear()
        torch.cuda.empty_cache()
        S.spdp_free(h)
    assert torch.equal(Y[0].cpu(), want) and torch.equal(Y[1].cpu(), want)


CUT = [(6, 4096, 32), (6, 8192, 40), (43, 4096, 128), (6, 8192, 512), (16, 4104, 300)]      # 32, 128, 128, 256 tokens per CTA, CTA pairs


def _cut_layer(S, R, K, N, count):
    """A layer, `count` inputs and their exact products; on integers every partial sum is exact."""
    rng = np.random.Generator(np.random.PCG64(R + N))
    W = rng.integers(-4, 5, (256 * R, K)).astype(np.float16)
    W[rng.random(W.shape) < 0.5] = 0
    X = [dev(rng.integers(-2, 3, (N, K)).astype(np.float16)) for _ in range(count)]
    Wd = dev(W).double()
    return S.spdp_pack_tiled_cbc(dev(W)), X, [(x.double() @ Wd.T).float() for x in X]


@pytest.mark.parametrize("R,K,N", CUT)
def test_spmm_cut_tiles_in_a_graph(S, R, K, N):
    """A captured call whose partial sums are memory of the graph: replays on new inputs, with direct calls in between."""
    h, X, want = _cut_layer(S, R, K, N, 3)
    try:
        buf, Y = torch.zeros_like(X[0]), torch.empty_like(want[0])
        direct = torch.empty_like(Y)
        S.spdp_spmm(h, buf, Y)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            S.spdp_spmm(h, buf, Y)
            S.spdp_spmm(h, buf, Y)
        for _ in range(2):
            for x, w in zip(X, want):
                buf.copy_(x)
                Y.fill_(float("nan"))
                graph.replay()
                S.spdp_spmm(h, X[0], direct)
                graph.replay()
                torch.cuda.synchronize()
                assert torch.equal(Y, w) and torch.equal(direct, want[0])
        assert S.spdp_last_device_status(h) == 0
        del graph
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("a,b", [(0, 3), (1, 4), (2, 2), (4, 4)])
def test_spmm_cut_tiles_on_two_streams(S, a, b):
    """Calls on two streams that may run side by side, on two handles or on the same one: each has partial sums of its own."""
    layers = [_cut_layer(S, *CUT[a], 2), None]
    layers[1] = layers[0] if a == b else _cut_layer(S, *CUT[b], 2)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    try:
        Y = [[torch.full_like(w, float("nan")) for w in want for _ in range(4)] for _, _, want in layers]
        torch.cuda.synchronize()
        for k in range(len(Y[0])):
            for (h, X, _), s, y in zip(layers, streams, Y):
                S.spdp_spmm(h, X[k // 4], y[k], stream=s)
        torch.cuda.synchronize()
        for (h, _, want), y in zip(layers, Y):
            assert all(torch.equal(y[k], want[k // 4]) for k in range(len(y)))
            assert S.spdp_last_device_status(h) == 0
    finally:
        for h in {layers[0][0], layers[1][0]}:
            S.spdp_free(h)


@pytest.mark.parametrize("R,K,N", [(4, 2048, 30), (4, 2048, 1), (3, 1280, 129), (75, 2048, 700)])
@pytest.mark.parametrize("dt", [torch.float16, torch.float32])
def test_spmm_cut_tiles_into_any_y(S, R, K, N, dt):
    """The second kernel of a cut call stores 4 rows at once where Y allows it: rows that end inside such a group, tokens that
    are no multiple of the block's, and a Y whose base and row stride are off the 8-byte boundary give the same bits as an aligned
    Y, and nothing outside Y is written.  (75 row tiles x 700 tokens: K-slices of CTA pairs, the others ranges of one-CTA forms.)"""
    M = 256 * R - 6
    g = torch.Generator(device="cuda").manual_seed(R * K + N)
    W = torch.randn(M, K, generator=g, device="cuda").half() * (torch.rand(M, K, generator=g, device="cuda") < 0.5)
    X = torch.randn(N, K, generator=g, device="cuda").half()
    h = S.spdp_pack_tiled_cbc(W)
    try:
        want = torch.full((N, M + 2), float("nan"), dtype=dt, device="cuda")[:, :M]       # rows start on 8-byte boundaries
        S.spdp_spmm(h, X, want)
        torch.cuda.synchronize()
        assert S.spdp_last_device_status(h) == 0 and not torch.isnan(want).any()
        err = (want.double() - X.double() @ W.double().T).abs()
        assert bool((err <= 1e-3 * (X.double().abs() @ W.double().abs().T) + 1e-5).all())
        for pad, at in ((0, 0), (1, 1), (3, 2), (5, 3)):
            buf = torch.full((N * (M + pad) + at + 8,), 7.0, dtype=dt, device="cuda")
            Y = buf[at:at + N * (M + pad)].view(N, M + pad)
            S.spdp_spmm(h, X, Y[:, :M])
            torch.cuda.synchronize()
            assert torch.equal(Y[:, :M], want)
            assert bool((Y[:, M:] == 7.0).all()) and bool((buf[:at] == 7.0).all()) and bool((buf[at + N * (M + pad):] == 7.0).all())
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("R,K", [(75, 1000), (3, 712)])
def test_spmm_token_counts_around_the_instructions_units(S, R, K):
    """The tensor-core instructions take a tile's tokens in units of 16 (one CTA) or 32 (CTA pairs, half of them in each CTA's shared
    memory): token counts around those units, around the tiles and around the pairs' second accumulator.  Integers: exact."""
    M = 256 * R - 100
    g = torch.Generator(device="cuda").manual_seed(R)
    W = torch.randint(-4, 5, (M, K), generator=g, device="cuda").half() * (torch.rand(M, K, generator=g, device="cuda") < 0.5)
    h = S.spdp_pack_tiled_cbc(W)
    try:
        for N in (1, 15, 16, 17, 31, 32, 33, 127, 129, 145, 255, 256, 257, 272, 288, 289, 479, 481, 511, 513, 545, 768, 770):
            X = torch.randint(-3, 4, (N, K), generator=g, device="cuda").half()
            Y = torch.full((N, M), float("nan"), dtype=torch.float32, device="cuda")
            S.spdp_spmm(h, X, Y)
            torch.cuda.synchronize()
            assert S.spdp_last_device_status(h) == 0
            assert torch.equal(Y.double(), X.double() @ W.double().T), N            # |sums| <= 1000 * 12 < 2^24
    finally:
        S.spdp_free(h)
