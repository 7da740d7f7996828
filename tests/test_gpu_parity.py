"""Parity of the CUDA library (through the C ABI) with the CPU oracle on the same seeded inputs.

Bars: packed arrays and the active-column set bit-exact; every output within
|y - y_ref| <= 1e-3 * sum_j |W_ij x_j| + 1e-5 (y widened to fp64, no re-rounding); exact
equality where every partial sum is exactly representable.
"""
import numpy as np
import pytest

from oracle import spdp_oracle as O
from paper_2607_21985_b200 import workloads as WL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp
    spdp.lib()
    return spdp


def dev(a):
    a = np.ascontiguousarray(a)
    if a.dtype == np.uint32:
        return torch.from_numpy(a.view(np.int32)).cuda()
    return torch.from_numpy(a).cuda()


def assert_same_packed(got, want):
    for key in ("tileoffset", "colinfo", "bitmap", "values"):
        assert got[key].dtype == want[key].dtype, key
        assert got[key].shape == want[key].shape, key
        assert np.array_equal(got[key], want[key]), key
    assert got["nnz"] == want["nnz"]


def gpu_spmspv(S, h, x, rule, thr, M, ydtype=torch.float32, mask_words=None):
    xd = dev(x)
    y = torch.full((M,), float("nan"), dtype=ydtype, device="cuda")        # poison: every entry must be written
    md = dev(mask_words) if mask_words is not None else None
    S.spdp_spmspv(h, xd, rule, thr, y, mask=md)
    torch.cuda.synchronize()
    assert S.spdp_last_device_status(h) == 0
    return y.cpu().numpy().astype(np.float64)


def gpu_active(S, h, x, rule, thr, K, mask_words=None):
    bits = torch.full(((K + 31) // 32,), -1, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    S.spdp_active_columns(h, dev(x), rule, thr, bits, cnt, mask=dev(mask_words) if mask_words is not None else None)
    torch.cuda.synchronize()
    return bits.cpu().numpy().view(np.uint32), int(cnt.item())


def check_y(y, y_ref, S_ref):
    err = np.abs(y - y_ref)
    tol = O.tolerance(S_ref)
    bad = np.flatnonzero(~(err <= tol))
    assert bad.size == 0, f"{bad.size} outputs out of tolerance, worst ratio {np.nanmax(err / tol):.3g} at {bad[:5]}"
    return float(np.max(err / tol))


# ------------------------------------------------------------------------------------------
# packer / unpacker: bit-exact
# ------------------------------------------------------------------------------------------
@pytest.mark.parametrize("M,K,seed", [(256, 16, 1), (512, 48, 2), (1, 1, 3), (257, 17, 4), (300, 40, 5),
                                      (1000, 200, 6), (2048, 272, 7)])
def test_pack_bit_exact_and_unpack(S, M, K, seed):
    W = WL.special_values_matrix(M, K, seed)
    want = O.pack_fast(W)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        got = S.spdp_export(h)
        assert_same_packed(got, want)
        info = S.spdp_get_info(h)
        assert (info.M, info.K, info.nnz, info.values_len) == (M, K, want["nnz"], len(want["values"]))
        assert info.packed_bytes == O.packed_bytes(want)
        out = torch.full((M, K + 3), -1.0, dtype=torch.float16, device="cuda")[:, :K]   # ldw != K
        S.spdp_unpack(h, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().view(np.uint16), O.canon(W))
    finally:
        S.spdp_free(h)


def test_pack_strided_input_and_storage_formula(S):
    M, K = 512, 96
    W = WL.special_values_matrix(M, K, 9)
    big = torch.zeros((M, K + 24), dtype=torch.float16, device="cuda")
    big[:, :K] = dev(W)
    h8 = S.spdp_pack_tiled_cbc(big[:, :K])
    h1 = S.spdp_pack_tiled_cbc(big[:, :K], pad_elems=1)
    try:
        assert_same_packed(S.spdp_export(h8), O.pack_fast(W))
        got1 = S.spdp_export(h1)
        assert_same_packed(got1, O.pack_fast(W, pad_elems=1))
        nnz = int(np.count_nonzero(W.view(np.uint16) & 0x7FFF))
        # Sec. 4.1 storage formula, exact when nothing is padded
        assert S.spdp_get_info(h1).packed_bytes == O.storage_formula_bytes(M, K, nnz)
        with pytest.raises(S.SpdpError, match="UNSUPPORTED_SHAPE"):
            S.spdp_spmspv(h1, torch.zeros(K, dtype=torch.float16, device="cuda"), 0, 0.0,
                          torch.zeros(M, dtype=torch.float32, device="cuda"))
    finally:
        S.spdp_free(h8)
        S.spdp_free(h1)


def test_pack_empty_and_full(S):
    for fill in (0.0, 1.0):
        W = np.full((512, 32), fill, np.float16)
        h = S.spdp_pack_tiled_cbc(dev(W))
        try:
            assert_same_packed(S.spdp_export(h), O.pack_ref(W))
        finally:
            S.spdp_free(h)


# ------------------------------------------------------------------------------------------
# active-column set: bit-exact
# ------------------------------------------------------------------------------------------
def test_active_set_bit_exact(S):
    K = 1000
    rng = np.random.Generator(np.random.PCG64(11))
    x = rng.standard_normal(K, dtype=np.float32).astype(np.float16)
    thr = float(np.float16(0.5))
    up, dn = np.nextafter(np.float16(0.5), np.float16(9)), np.nextafter(np.float16(0.5), np.float16(0))
    x[:14] = np.asarray([0.0, -0.0, 0.5, -0.5, up, -up, dn, -dn, np.nan, np.inf, -np.inf, 6e-8, -6e-8, 65504], np.float16)
    h = S.spdp_pack_tiled_cbc(dev(np.ones((256, K), np.float16)))
    try:
        for rule, t in ((O.DP_ABS_GT, thr), (O.DP_ABS_GT, 0.0), (O.DP_ABS_GT, -1.0), (O.DP_NONE, 0.0),
                        (O.DP_ABS_GT, 1e30), (O.DP_ABS_GT, float("inf"))):
            want = O.active_ref(x, rule, t)
            bits, cnt = gpu_active(S, h, x, rule, t, K)
            assert np.array_equal(bits, O.active_to_words(want)) and cnt == int(want.sum())
        m = rng.random(K) < 0.3
        bits, cnt = gpu_active(S, h, x, O.DP_MASK, 0.0, K, O.active_to_words(m))
        assert np.array_equal(bits, O.active_to_words(m)) and cnt == int(m.sum())
    finally:
        S.spdp_free(h)


# ------------------------------------------------------------------------------------------
# spMspV against the oracle
# ------------------------------------------------------------------------------------------
@pytest.mark.parametrize("M,K,sp,skip,seed", [
    (256, 16, 0.5, 0.5, 1), (512, 64, 0.5, 0.0, 2), (300, 40, 0.3, 0.25, 3), (1, 1, 0.0, 0.0, 4),
    (257, 17, 0.5, 0.5, 5), (1024, 1024, 0.5, 0.5, 6), (768, 4400, 0.7, 0.9, 7), (2304, 528, 0.9, 0.4, 8),
    (4096, 272, 0.0, 0.1, 9), (256, 8192, 0.6, 0.5, 10),
    # rows longer than one batch of the kernel (pieces carry their sums over) and ragged long rows
    (512, 20000, 0.5, 0.3, 11), (300, 16400, 0.9, 0.0, 12), (1000, 8200, 0.2, 0.6, 13)])
@pytest.mark.parametrize("ydtype", ["f32", "f16"])
def test_spmspv_matches_oracle(S, M, K, sp, skip, seed, ydtype):
    rw, rx = WL._rngs(seed)
    W = WL.prune_global_magnitude(WL.normal_weights(rw, M, K), sp).astype(np.float16)
    x = rx.standard_normal(K, dtype=np.float32).astype(np.float16)
    rule, thr = WL.skip_threshold(x, skip)
    a = O.active_ref(x, rule, thr)
    y_ref, S_ref = O.spmspv_ref(W, x, a)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        bits, cnt = gpu_active(S, h, x, rule, thr, K)
        assert np.array_equal(bits, O.active_to_words(a)) and cnt == int(a.sum())
        yd = torch.float32 if ydtype == "f32" else torch.float16
        y = gpu_spmspv(S, h, x, rule, thr, M, yd)
        check_y(y, y_ref, S_ref)
        y2 = gpu_spmspv(S, h, x, rule, thr, M, yd)
        assert np.array_equal(y, y2)                                   # fixed summation order
        for ctas in (1, 3, 37, 1000):                                  # other split-K layouts
            S.spdp_set_num_ctas(h, ctas)
            check_y(gpu_spmspv(S, h, x, rule, thr, M, yd), y_ref, S_ref)
    finally:
        S.spdp_free(h)


def test_spmspv_exact_on_integers_and_powers_of_two(S):
    """Every product and partial sum is exactly representable: the GPU must match exactly."""
    rng = np.random.Generator(np.random.PCG64(21))
    M, K = 700, 900
    W = rng.integers(-8, 9, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.6] = 0
    x = rng.integers(-4, 5, K).astype(np.float16)
    a = O.active_ref(x, O.DP_ABS_GT, 1.0)
    y_ref, _ = O.spmspv_ref(W, x, a)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        assert np.array_equal(gpu_spmspv(S, h, x, O.DP_ABS_GT, 1.0, M), y_ref)
        Wp = (2.0 ** rng.integers(-6, 3, (M, K))).astype(np.float16) * rng.choice([-1, 1], (M, K)).astype(np.float16)
        Wp[rng.random((M, K)) < 0.5] = 0
        xp = (2.0 ** rng.integers(-3, 3, K)).astype(np.float16)
        hp = S.spdp_pack_tiled_cbc(dev(Wp))
        try:
            yp_ref, _ = O.spmspv_ref(Wp, xp, np.ones(K, bool))
            assert np.array_equal(gpu_spmspv(S, hp, xp, O.DP_NONE, 0.0, M), yp_ref)
        finally:
            S.spdp_free(hp)
    finally:
        S.spdp_free(h)


def test_spmspv_degenerate_cases(S):
    M, K = 600, 100
    rng = np.random.Generator(np.random.PCG64(23))
    W = (rng.standard_normal((M, K), dtype=np.float32) * 0.02).astype(np.float16)
    W[:, 10:20] = 0                                  # empty columns
    W[256:512, :] = 0                                # an empty row tile
    x = rng.standard_normal(K, dtype=np.float32).astype(np.float16)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        # nothing active: y is written as zeros
        y = gpu_spmspv(S, h, x, O.DP_ABS_GT, 1e9, M)
        assert not y.any()
        y = gpu_spmspv(S, h, x, O.DP_MASK, 0.0, M, mask_words=np.zeros(4, np.uint32))
        assert not y.any()
        # a single active column; explicit mask rule
        m = np.zeros(K, bool)
        m[37] = True
        y = gpu_spmspv(S, h, x, O.DP_MASK, 0.0, M, mask_words=O.active_to_words(m))
        y_ref, S_ref = O.spmspv_ref(W, x, m)
        check_y(y, y_ref, S_ref)
        # NaN activation is active and propagates; Inf weight in a skipped column does not
        W2 = W.copy()
        W2[5, 50] = np.inf
        x2 = x.copy()
        x2[50] = 0.0
        x2[60] = np.nan
        h2 = S.spdp_pack_tiled_cbc(dev(W2))
        try:
            y = gpu_spmspv(S, h2, x2, O.DP_ABS_GT, 0.0, M)
            nz60 = O.is_nonzero(W2[:, 60])
            assert np.all(np.isnan(y[nz60])) and not np.isnan(y[~nz60]).any()
        finally:
            S.spdp_free(h2)
    finally:
        S.spdp_free(h)


def test_unaligned_x_and_mask_rule_on_a_long_row(S):
    """x that is only 2-byte aligned takes the kernel's plain-load path; the explicit mask rule on two batches."""
    w = WL.config2(768, 9000, seed=8)
    a = O.active_ref(w.x, w.rule, w.thr)
    y_ref, S_ref = O.spmspv_ref(w.W, w.x, a)
    h = S.spdp_pack_tiled_cbc(dev(w.W))
    try:
        buf = torch.zeros(w.K + 8, dtype=torch.float16, device="cuda")
        for shift in (1, 3, 8):
            xs = buf[shift: shift + w.K]
            xs.copy_(dev(w.x))
            assert xs.data_ptr() % 16 == (2 * shift) % 16
            y = torch.full((w.M,), float("nan"), dtype=torch.float32, device="cuda")
            S.spdp_spmspv(h, xs, w.rule, w.thr, y)
            torch.cuda.synchronize()
            check_y(y.cpu().numpy().astype(np.float64), y_ref, S_ref)
        y = gpu_spmspv(S, h, w.x, O.DP_MASK, 0.0, w.M, mask_words=O.active_to_words(a))
        check_y(y, y_ref, S_ref)
    finally:
        S.spdp_free(h)


def test_spmspv_in_a_cuda_graph(S):
    """spdp_spmspv only launches (no allocation, no synchronisation): it can be captured and replayed."""
    w = WL.config1(1024, 2048, seed=9)
    a = O.active_ref(w.x, w.rule, w.thr)
    y_ref, S_ref = O.spmspv_ref(w.W, w.x, a)
    h = S.spdp_pack_tiled_cbc(dev(w.W))
    try:
        x = dev(w.x)
        y = torch.zeros(w.M, dtype=torch.float32, device="cuda")
        S.spdp_spmspv(h, x, w.rule, w.thr, y)                      # warm-up outside the capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            with torch.cuda.graph(g, stream=side):
                S.spdp_spmspv(h, x, w.rule, w.thr, y, stream=side)
        for _ in range(3):
            y.fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            check_y(y.cpu().numpy().astype(np.float64), y_ref, S_ref)
    finally:
        S.spdp_free(h)


def test_imported_oracle_arrays_give_same_result(S):
    w = WL.config1(768, 640, seed=4)
    p = O.pack_fast(w.W)
    h_imp = S.spdp_import_tiled_cbc(w.M, w.K, p["tileoffset"], p["colinfo"], p["bitmap"], p["values"])
    h_gpu = S.spdp_pack_tiled_cbc(dev(w.W))
    try:
        assert_same_packed(S.spdp_export(h_imp), p)
        y1 = gpu_spmspv(S, h_imp, w.x, w.rule, w.thr, w.M)
        y2 = gpu_spmspv(S, h_gpu, w.x, w.rule, w.thr, w.M)
        assert np.array_equal(y1, y2)
        bad = p["colinfo"].copy()
        bad[3] += 1
        with pytest.raises(S.SpdpError, match="INVALID_ARG"):
            S.spdp_import_tiled_cbc(w.M, w.K, p["tileoffset"], bad, p["bitmap"], p["values"])
    finally:
        S.spdp_free(h_imp)
        S.spdp_free(h_gpu)


def test_host_vector_entry_point(S):
    w = WL.config2(1024, 512, seed=6)
    a = O.active_ref(w.x, w.rule, w.thr)
    y_ref, S_ref = O.spmspv_ref(w.W, w.x, a)
    h = S.spdp_pack_tiled_cbc(dev(w.W))
    try:
        xh = torch.from_numpy(w.x.copy()).pin_memory()
        for dt in (torch.float16, torch.float32):
            yh = torch.full((w.M,), float("nan"), dtype=dt).pin_memory()
            S.spdp_spmspv_host(h, xh, w.rule, w.thr, yh)
            check_y(yh.numpy().astype(np.float64), y_ref, S_ref)
        yn = np.full(w.M, np.nan, np.float32)
        S.spdp_spmspv_host(h, w.x, O.DP_MASK, 0.0, yn, mask_host=O.active_to_words(a))
        check_y(yn.astype(np.float64), y_ref, S_ref)
    finally:
        S.spdp_free(h)


def test_host_vector_entry_point_repeated_calls(S):
    """The same pinned buffers call after call (the library may replay a recorded graph): new contents
    of x must give new results, and a different CTA count, other buffers or pageable memory still work."""
    rng = np.random.Generator(np.random.PCG64(91))
    M, K = 1300, 2100
    W = (rng.standard_normal((M, K)) * (rng.random((M, K)) < 0.5) * 0.05).astype(np.float16)
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        xh = torch.zeros(K, dtype=torch.float16).pin_memory()
        yh = torch.zeros(M, dtype=torch.float32).pin_memory()
        for step in range(6):
            x = rng.standard_normal(K).astype(np.float16)
            xh.copy_(torch.from_numpy(x))
            yh.fill_(float("nan"))
            if step == 4:
                S.spdp_set_num_ctas(h, 37)
            S.spdp_spmspv_host(h, xh, O.DP_ABS_GT, 0.4, yh)
            a = O.active_ref(x, O.DP_ABS_GT, 0.4)
            y_ref, S_ref = O.spmspv_ref(W, x, a)
            check_y(yh.numpy().astype(np.float64), y_ref, S_ref)
        y2 = torch.zeros(M, dtype=torch.float16).pin_memory()          # another output buffer and dtype
        S.spdp_spmspv_host(h, xh, O.DP_ABS_GT, 0.4, y2)
        check_y(y2.numpy().astype(np.float64), y_ref, S_ref)
        yn = np.full(M, np.nan, np.float32)                            # pageable memory
        for _ in range(3):
            S.spdp_spmspv_host(h, x, O.DP_ABS_GT, 0.4, yn)
            check_y(yn.astype(np.float64), y_ref, S_ref)
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("make", [lambda: WL.config1(1024, 1024), lambda: WL.config2(1536, 1024),
                                  lambda: WL.config3(1024, 2752), lambda: WL.config4(3584, 1024),
                                  lambda: WL.config5(0, 0, 1024, 1024), lambda: WL.config5(3, 3, 1024, 1024)])
def test_scaled_down_benchmark_layers(S, make):
    w = make()
    a = O.active_ref(w.x, w.rule, w.thr)
    y_ref, S_ref = O.spmspv_ref(w.W, w.x, a)
    h = S.spdp_pack_tiled_cbc(dev(w.W))
    try:
        assert_same_packed(S.spdp_export(h), O.pack_fast(w.W))
        bits, _ = gpu_active(S, h, w.x, w.rule, w.thr, w.K)
        assert np.array_equal(bits, O.active_to_words(a))
        check_y(gpu_spmspv(S, h, w.x, w.rule, w.thr, w.M, torch.float16), y_ref, S_ref)
        check_y(gpu_spmspv(S, h, w.x, w.rule, w.thr, w.M, torch.float32), y_ref, S_ref)
    finally:
        S.spdp_free(h)


# ------------------------------------------------------------------------------------------
# the single-vector kernel's own DP test (it lists the active columns itself, 8 per thread)
# ------------------------------------------------------------------------------------------
def _striped_identity(M, K):
    """One stored 1.0 per column, at row j % M: y then shows every column's decision by itself."""
    W = torch.zeros((M, K), dtype=torch.float16, device="cuda")
    j = torch.arange(K, device="cuda")
    W[j % M, j] = 1.0
    return W


@pytest.mark.parametrize("thr", [0.5, 0.50006103515625, 0.3, 0.0, -0.0, -1.0, 1e-10, 70000.0, float("inf"),
                                 float("-inf"), float("nan"), 6.1e-5, 5.96e-8])
def test_spmspv_active_set_on_threshold_edges(S, thr):
    """Values at, just below and just above the threshold (in fp16 steps), zeros of both signs, subnormals,
    the largest finite values, NaN and both infinities, under finite, infinite and NaN thresholds: the
    kernel's in-line DP test must take the oracle's decision for every one.  Also with x only 2-byte
    aligned (the plain-load path) and with the probes astride column 8192, where a CTA that owns a long
    stretch of one row tile ends one list of columns and begins the next."""
    base = np.float16(thr) if np.isfinite(thr) and abs(thr) < 65504 else np.float16(1.0)
    around = np.array([base, np.nextafter(base, np.float16(np.inf)), np.nextafter(base, np.float16(-np.inf)),
                       -base, 0.0, -0.0, 6e-8, -6e-8, 6.1e-5, 65504, -65504, 0.25, 0.5, 0.75,
                       np.nan, np.inf, -np.inf], dtype=np.float16)
    rng = np.random.Generator(np.random.PCG64(78))
    for K, ctas, shift in ((64, 0, 0), (16400, 1, 0), (16400, 3, 1), (16400, 0, 3)):
        M = min(K, 256)
        first = 0 if K == 64 else 8192 - 7                     # probes astride the end of the first list
        x = np.zeros(K, dtype=np.float16)
        x[first:first + len(around)] = rng.permutation(around)
        a = O.active_ref(x, O.DP_ABS_GT, thr)
        want = np.zeros(M, dtype=np.float32)
        for p in range(first, first + len(around)):
            if a[p]:
                want[p % M] = np.float32(x[p])
        h = S.spdp_pack_tiled_cbc(_striped_identity(M, K))
        try:
            if ctas:
                S.spdp_set_num_ctas(h, ctas)
            buf = torch.zeros(K + 8, dtype=torch.float16, device="cuda")
            xs = buf[shift:shift + K]
            xs.copy_(dev(x))
            y = torch.full((M,), float("nan"), dtype=torch.float32, device="cuda")
            S.spdp_spmspv(h, xs, O.DP_ABS_GT, thr, y)
            torch.cuda.synchronize()
            assert np.array_equal(y.cpu().numpy(), want, equal_nan=True), (thr, K, ctas, shift)
            bits, cnt = gpu_active(S, h, x, O.DP_ABS_GT, thr, K)
            assert np.array_equal(bits, O.active_to_words(a)) and cnt == int(a.sum())
        finally:
            S.spdp_free(h)


def test_mask_rule_with_the_mask_at_the_end_of_its_allocation(S):
    """Explicit mask whose last word is the last word of its buffer, on shapes where a CTA's range starts at
    an odd GTile column (the list then has padding units between its two pieces, which must not read the
    mask), and a first call issued on a side stream right after packing."""
    for M, K, ctas in ((512, 4096, 3), (768, 4128, 7), (1024, 2080, 5)):
        rw, rx = WL._rngs(40 + ctas)
        W = WL.prune_global_magnitude(WL.normal_weights(rw, M, K), 0.5).astype(np.float16)
        x = rx.standard_normal(K, dtype=np.float32).astype(np.float16)
        m = rx.random(K) < 0.5
        y_ref, S_ref = O.spmspv_ref(W, x, m)
        words = O.active_to_words(m)
        arena = torch.zeros(4096 + len(words), dtype=torch.int32, device="cuda")
        md = arena[4096:]
        md.copy_(dev(words))
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            h = S.spdp_pack_tiled_cbc(dev(W), stream=side)
            try:
                S.spdp_set_num_ctas(h, ctas)
                y = torch.full((M,), float("nan"), dtype=torch.float32, device="cuda")
                S.spdp_spmspv(h, dev(x), O.DP_MASK, 0.0, y, mask=md, stream=side)
                side.synchronize()
                check_y(y.cpu().numpy().astype(np.float64), y_ref, S_ref)
            finally:
                S.spdp_free(h)


def test_row_sharded_handles_reproduce_the_product(S):
    """Row-tile sharding on one GPU: every rank's slice packed as its own matrix, the slices of y side by
    side against the oracle (the collective that joins them is exercised by the two-rank CPU test)."""
    w = WL.config4(2304, 1040, seed=12)
    a = O.active_ref(w.x, w.rule, w.thr)
    y_ref, S_ref = O.spmspv_ref(w.W, w.x, a)
    x = dev(w.x)
    for world in (2, 3, 16):
        y = torch.full((w.M,), float("nan"), dtype=torch.float32, device="cuda")
        for rank in range(world):
            first, rows = S.spdp_row_shard(w.M, world, rank)
            if rows == 0:
                continue
            h = S.spdp_pack_tiled_cbc(dev(w.W[first:first + rows]))
            try:
                S.spdp_spmspv(h, x, w.rule, w.thr, y[first:first + rows])
            finally:
                torch.cuda.synchronize()
                S.spdp_free(h)
        check_y(y.cpu().numpy().astype(np.float64), y_ref, S_ref)


def test_producer_fused_activation_and_mask(S):
    """x = silu(gate) * up with the keep-mask written in the same pass: x within one fp16 step of the fp64
    definition, the mask exactly the set the magnitude rule chooses on the stored x, and the decode call
    with that mask bit-identical to the decode call that tests x itself."""
    rng = np.random.Generator(np.random.PCG64(83))
    M, K = 1536, 3000
    gate = rng.standard_normal(K).astype(np.float16) * np.float16(2.0)
    up = rng.standard_normal(K).astype(np.float16)
    gate[:4] = np.asarray([0.0, -0.0, 30.0, -30.0], np.float16)
    W = (rng.standard_normal((M, K)) * (rng.random((M, K)) < 0.5) * 0.05).astype(np.float16)
    thr = 0.3
    x_out = torch.full((K,), float("nan"), dtype=torch.float16, device="cuda")
    mask = torch.full(((K + 31) // 32,), -1, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), -5, dtype=torch.int32, device="cuda")
    S.spdp_swiglu_dp(dev(gate), dev(up), thr, x_out, mask, cnt)
    torch.cuda.synchronize()
    xg = x_out.cpu().numpy()
    ref = O.swiglu_ref(gate, up)
    step = np.maximum(np.abs(ref), 2.0 ** -14) * 2.0 ** -10                  # one fp16 step at that magnitude
    assert np.all(np.abs(xg.astype(np.float64) - ref) <= step)
    a = O.active_ref(xg, O.DP_ABS_GT, thr)                                   # decided on the kernel's own fp16 x
    assert np.array_equal(mask.cpu().numpy().view(np.uint32), O.active_to_words(a)) and int(cnt.item()) == int(a.sum())
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        y_mask = torch.empty(M, dtype=torch.float32, device="cuda")
        y_test = torch.empty(M, dtype=torch.float32, device="cuda")
        S.spdp_spmspv(h, x_out, O.DP_MASK, 0.0, y_mask, mask=mask)
        S.spdp_spmspv(h, x_out, O.DP_ABS_GT, thr, y_test)
        torch.cuda.synchronize()
        assert np.array_equal(y_mask.cpu().numpy(), y_test.cpu().numpy())
        y_ref, S_ref = O.spmspv_ref(W, xg, a)
        check_y(y_mask.cpu().numpy().astype(np.float64), y_ref, S_ref)
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("pad", [8, 1])
@pytest.mark.parametrize("M,K,ldw,shift", [(256, 64, 64, 0), (257, 63, 64, 0), (255, 65, 72, 0), (300, 128, 131, 0), (512, 130, 136, 1),
                                           (1, 1, 1, 0), (31, 200, 200, 3), (768, 16, 24, 0), (2000, 1100, 1104, 0)])
def test_pack_blocks_round_trip(S, M, K, ldw, shift, pad):
    """The packer handles 256 x 64 blocks: edges of the block, rows that do not start on 16 bytes (odd strides, shifted
    base), both padding units, special values; packed arrays and the way back bit for bit."""
    W = WL.special_values_matrix(M, K, 7 * M + K)
    buf = torch.zeros(M * ldw + shift + 8, dtype=torch.float16, device="cuda")
    Wd = buf[shift:shift + M * ldw].view(M, ldw)[:, :K]
    Wd.copy_(torch.from_numpy(W))
    h = S.spdp_pack_tiled_cbc(Wd, pad_elems=pad)
    try:
        got, want = S.spdp_export(h), O.pack_ref(W, pad_elems=pad) if M * K < 50000 else O.pack_fast(W, pad_elems=pad)
        for key in ("tileoffset", "colinfo", "bitmap", "values"):
            assert np.array_equal(got[key], want[key]), key
        out = torch.full((M * ldw + shift + 8,), 7.0, dtype=torch.float16, device="cuda")
        S.spdp_unpack(h, out[shift:shift + M * ldw].view(M, ldw)[:, :K])
        torch.cuda.synchronize()
        back = out[shift:shift + M * ldw].view(M, ldw).cpu().numpy().view(np.uint16)
        bits = W.view(np.uint16)
        assert np.array_equal(back[:, :K], np.where(bits & 0x7FFF, bits, 0))
        assert np.all(back[:, K:] == np.float16(7.0).view(np.uint16))          # nothing beyond the K columns is written
    finally:
        S.spdp_free(h)


def test_free_of_nothing_gives_kept_memory_back(S):
    h = S.spdp_pack_tiled_cbc(torch.ones((2048, 4096), dtype=torch.float16, device="cuda"))
    S.spdp_free(h)
    kept = torch.cuda.mem_get_info()[0]
    S.spdp_free(None)
    assert torch.cuda.mem_get_info()[0] >= kept + (16 << 20)                    # the layer's 16 MB of values at least


def test_handle_keeps_its_workspace_where_there_is_no_memory_for_a_new_one(S):
    """1024 CTAs need a workspace of 9.4 MB; with less than that free the call is refused and the handle works on as it was."""
    import ctypes
    rt = ctypes.CDLL("libcudart.so.12")
    rng = np.random.Generator(np.random.PCG64(5))
    W = rng.integers(-4, 5, (4096, 1024)).astype(np.float16)                    # 1024 GTiles
    x = rng.integers(-3, 4, 1024).astype(np.float16)
    want = W.astype(np.float32) @ x.astype(np.float32)
    h, xd, y = S.spdp_pack_tiled_cbc(dev(W)), dev(x), torch.empty(4096, dtype=torch.float32, device="cuda")
    hold = []
    try:
        ctas = S.spdp_get_info(h).num_ctas
        S.spdp_free(None)
        torch.cuda.empty_cache()
        free = lambda: torch.cuda.mem_get_info()[0]
        while free() > 8 << 20:
            p = ctypes.c_void_p()
            assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(max((free() - (6 << 20)) >> 21 << 20, 2 << 20))) == 0
            hold.append(p)
        with pytest.raises(S.SpdpError, match="ERR_ALLOC"):
            S.spdp_set_num_ctas(h, 1024)
        assert S.spdp_get_info(h).num_ctas == ctas
        for _ in range(2):
            y.fill_(float("nan"))
            S.spdp_spmspv(h, xd, O.DP_NONE, 0.0, y)
            assert np.array_equal(y.cpu().numpy(), want)
        for p in hold:
            assert rt.cudaFree(p) == 0
        hold = []
        S.spdp_set_num_ctas(h, 1024)
        assert S.spdp_get_info(h).num_ctas == 1024
        S.spdp_spmspv(h, xd, O.DP_NONE, 0.0, y)
        assert np.array_equal(y.cpu().numpy(), want)
    finally:
        for p in hold:
            rt.cudaFree(p)
        S.spdp_free(h)


def test_packed_arrays_can_be_exported_to_another_process(S):
    """What spdp_get_info names are ordinary device allocations: the runtime gives an interprocess handle for them, for a new
    handle and for one that got the memory of a freed one."""
    import ctypes
    rt = ctypes.CDLL("libcudart.so.12")
    W = torch.ones((1024, 2048), dtype=torch.float16, device="cuda")
    for _ in range(2):
        h = S.spdp_pack_tiled_cbc(W)
        try:
            info = S.spdp_get_info(h)
            for p in (info.values_dev, info.bitmap_dev, info.colinfo_dev, info.tileoffset_dev):
                assert rt.cudaIpcGetMemHandle(ctypes.create_string_buffer(64), ctypes.c_void_p(p)) == 0
        finally:
            S.spdp_free(h)


def test_threads_pack_and_free_side_by_side(S):
    """Memory of freed handles goes to the next ones, on other threads and streams too: every layer keeps its own arrays."""
    import concurrent.futures as cf

    def work(seed):
        torch.cuda.set_device(0)
        rng = np.random.Generator(np.random.PCG64(seed))
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            for step in range(12):
                M, K = 256 * int(rng.integers(1, 6)), 16 * int(rng.integers(1, 40))
                W = rng.integers(-4, 5, (M, K)).astype(np.float16)
                W[rng.random((M, K)) < 0.5] = 0
                x = rng.integers(-3, 4, K).astype(np.float16)
                Wd, xd, y = dev(W), dev(x), torch.full((M,), float("nan"), dtype=torch.float32, device="cuda")
                back = torch.empty_like(Wd)
                h = S.spdp_pack_tiled_cbc(Wd, stream=side)
                try:
                    for _ in range(3):
                        S.spdp_spmspv(h, xd, O.DP_NONE, 0.0, y, stream=side)
                    S.spdp_unpack(h, back, stream=side)
                    side.synchronize()
                finally:
                    S.spdp_free(h)
                assert np.array_equal(y.cpu().numpy(), W.astype(np.float32) @ x.astype(np.float32))
                assert np.array_equal(back.cpu().numpy(), np.where(W == 0, np.float16(0), W))
        return seed
    with cf.ThreadPoolExecutor(6) as pool:
        assert list(pool.map(work, range(6))) == list(range(6))


@pytest.mark.parametrize("K", [1, 2, 31, 63, 64, 65, 127, 129, 1023, 3100, 8191, 8193])
@pytest.mark.parametrize("ctas", [0, 1, 2, 5])
def test_active_list_edges(S, K, ctas):
    """The list phase walks pairs of columns in chunks of 64: lists that end anywhere in a chunk, ranges that hold the tail of
    one row tile and the head of the next (CTA counts that do not divide the row tiles), every rule.  Integers: exact."""
    rng = np.random.Generator(np.random.PCG64(K))
    M = 700
    W = rng.integers(-4, 5, (M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.5] = 0
    x = rng.integers(-3, 4, K).astype(np.float16)
    h, h4 = S.spdp_pack_tiled_cbc(dev(W)), S.spdp_pack_tiled_cbc_q4(dev(np.clip(W, -1, 1)))   # scale 1/7: codes -7, 0, 7
    s7 = np.float32(np.float16(1 / 7)) * np.float32(7)
    keep = rng.random(K) < 0.4
    try:
        for hh, Wq, f in ((h, W, 1.0), (h4, np.clip(W, -1, 1), float(s7))):
            S.spdp_set_num_ctas(hh, ctas)
            for rule, thr, act in ((O.DP_NONE, 0.0, np.ones(K, bool)), (O.DP_ABS_GT, 1.0, np.abs(x) > 1), (O.DP_MASK, 0.0, keep)):
                y = torch.full((M,), float("nan"), dtype=torch.float32, device="cuda")
                S.spdp_spmspv(hh, dev(x), rule, thr, y, mask=dev(O.active_to_words(keep).view(np.int32)) if rule == O.DP_MASK else None)
                torch.cuda.synchronize()
                want = Wq.astype(np.float64) @ np.where(act, x, 0).astype(np.float64) * f
                got = y.cpu().numpy().astype(np.float64)
                if f == 1.0:
                    assert np.array_equal(got, want), (rule, ctas)
                else:                                                  # products of code 7 and scale * x: a rounding per sum
                    scale = np.abs(Wq).astype(np.float64) @ np.abs(np.where(act, x, 0)).astype(np.float64) + 1
                    assert np.all(np.abs(got - want) <= 2.0 ** -24 * (K + 32) * scale), (rule, ctas)
            assert S.spdp_last_device_status(hh) == 0
    finally:
        S.spdp_free(h)
        S.spdp_free(h4)


@pytest.mark.parametrize("K", [8, 1000, 4099])
@pytest.mark.parametrize("pin_x,pin_y,shift", [(True, True, 0), (True, True, 1), (True, False, 0), (False, True, 0), (False, False, 3)])
def test_host_vectors_buffers(S, K, pin_x, pin_y, shift):
    """Pinned and pageable buffers in every mix, pinned x that does not start on 16 bytes, mask rule and threshold, both output
    types; first call, recorded call and replays agree with the device-vector call bit for bit."""
    rng = np.random.Generator(np.random.PCG64(K + shift))
    M = 900
    W = rng.standard_normal((M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.5] = 0
    x = rng.standard_normal(K).astype(np.float16)
    words = O.active_to_words(rng.random(K) < 0.5).view(np.int32)
    buf = torch.zeros(K + shift, dtype=torch.float16)
    buf = buf.pin_memory() if pin_x else buf
    xh = buf[shift:]
    xh.copy_(torch.from_numpy(x))
    mh = torch.from_numpy(words.copy())
    mh = mh.pin_memory() if pin_x else mh
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        for rule, mask in ((O.DP_ABS_GT, None), (O.DP_MASK, mh)):
            for dt in (torch.float16, torch.float32):
                want = torch.empty(M, dtype=dt, device="cuda")
                S.spdp_spmspv(h, dev(x), rule, 0.5, want, mask=None if mask is None else mask.cuda())
                for k in range(4):
                    yh = torch.full((M,), float("nan"), dtype=dt)
                    yh = yh.pin_memory() if pin_y else yh
                    for call in range(3):
                        yh.fill_(float("nan"))
                        S.spdp_spmspv_host(h, xh, rule, 0.5, yh, mask_host=mask)
                        assert torch.equal(yh, want.cpu()), (rule, dt, k, call)
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("x_at,gap_y,gap_mask", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 2, 0), (0, 0, 1), (0, 0, 2)])
@pytest.mark.parametrize("dtype", [np.float16, np.float32])
def test_host_vectors_at_any_byte_of_a_pinned_arena(S, x_at, gap_y, gap_mask, dtype):
    """x, y and the mask words one behind the other in one pinned arena, at bytes that are no multiple of their elements'
    size: such buffers are copied (the kernels must not touch them) and give what the device-vector call gives."""
    M, K = 600, 1001
    rng = np.random.Generator(np.random.PCG64(17))
    W = rng.standard_normal((M, K)).astype(np.float16)
    W[rng.random((M, K)) < 0.5] = 0
    x = rng.standard_normal(K).astype(np.float16)
    words = O.active_to_words(rng.random(K) < 0.5)
    arena = torch.zeros(16384, dtype=torch.uint8).pin_memory().numpy()
    y_at = x_at + 2 * K + gap_y
    mask_at = y_at + M * dtype().itemsize + gap_mask
    xh = np.frombuffer(arena, np.float16, K, x_at)
    yh = np.frombuffer(arena, dtype, M, y_at)
    mh = np.frombuffer(arena, np.uint32, words.size, mask_at)
    xh[:], mh[:] = x, words
    h = S.spdp_pack_tiled_cbc(dev(W))
    try:
        for rule, mask in ((O.DP_ABS_GT, None), (O.DP_MASK, mh)):
            want = torch.empty(M, dtype=torch.float16 if dtype == np.float16 else torch.float32, device="cuda")
            S.spdp_spmspv(h, dev(x), rule, 0.5, want, mask=None if mask is None else dev(words))
            for call in range(3):
                yh[:] = np.nan
                S.spdp_spmspv_host(h, xh, rule, 0.5, yh, mask_host=mask)
                assert np.array_equal(yh, want.cpu().numpy()), (rule, call)
                assert np.array_equal(xh, x) and np.array_equal(mh, words)
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("down", ["fp16", "q4", "batch"])
def test_projections_and_producer_overlap_on_one_stream(S, down):
    """A gated MLP as a decode loop runs it: gate and up projection, the producer, the down projection with its mask, token
    after token in the same buffers without a synchronisation, so that every kernel starts beside the one whose results it
    reads.  Bit for bit what the same calls give when each waits for the one before."""
    rng = np.random.Generator(np.random.PCG64(29))
    D, F, steps, tokens = 1000, 2808, 60, 3 if down == "batch" else 1
    sparse = lambda m, k: (rng.standard_normal((m, k)) * (rng.random((m, k)) < 0.5) * 0.1).astype(np.float16)
    hg, hu = S.spdp_pack_tiled_cbc(dev(sparse(F, D))), S.spdp_pack_tiled_cbc(dev(sparse(F, D)))
    Wd = dev(sparse(D, F))
    hd = S.spdp_pack_tiled_cbc_q4(Wd) if down == "q4" else S.spdp_pack_tiled_cbc(Wd)
    X = dev(rng.standard_normal((steps, tokens, D)).astype(np.float16))
    gate, up = (torch.empty(F, dtype=torch.float16, device="cuda") for _ in range(2))
    h = torch.empty((tokens, F), dtype=torch.float16, device="cuda")
    mask = torch.empty((tokens, (F + 31) // 32), dtype=torch.int32, device="cuda")

    def run(wait):
        Y = torch.full((steps, tokens, D), float("nan"), dtype=torch.float32, device="cuda")
        for s in range(steps):
            for b in range(tokens):
                S.spdp_spmspv(hg, X[s, b], O.DP_ABS_GT, 0.7, gate)
                wait()
                S.spdp_spmspv(hu, X[s, b], O.DP_ABS_GT, 0.7, up)
                wait()
                S.spdp_swiglu_dp(gate, up, 0.4, h[b], mask[b])
                wait()
            if down == "batch":
                S.spdp_spmspv_batch(hd, h, O.DP_MASK, 0.0, Y[s], mask=mask)
            else:
                S.spdp_spmspv(hd, h[0], O.DP_MASK, 0.0, Y[s, 0], mask=mask[0])
            wait()
        torch.cuda.synchronize()
        return Y.cpu().numpy()
    try:
        want = run(torch.cuda.synchronize)
        assert np.isfinite(want).all() and len(np.unique(want[:, 0, 0])) == steps
        for _ in range(5):
            assert np.array_equal(run(lambda: None), want)
    finally:
        for x in (hg, hu, hd):
            S.spdp_free(x)
