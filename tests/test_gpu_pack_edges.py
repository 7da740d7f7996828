"""The packer's comparisons and scan at their edges, bit for bit against the oracle's packer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import spdp_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2607_21985_b200 import spdp
    spdp.lib()
    return spdp


def packed_equal(S, W):
    want = O.pack_fast(W)
    h = S.spdp_pack_tiled_cbc(torch.from_numpy(W).cuda())
    try:
        got = S.spdp_export(h)
        for key in ("tileoffset", "colinfo", "bitmap", "values"):
            assert np.array_equal(got[key], want[key]), key
        back = torch.empty(W.shape, dtype=torch.float16, device="cuda")
        S.spdp_unpack(h, back)
        assert np.array_equal(back.cpu().numpy().view(np.uint16), O.canon(W))
    finally:
        S.spdp_free(h)


@pytest.mark.parametrize("shift", [0, 1])
def test_every_bit_pattern_is_stored_or_not(S, shift):
    """All 65536 fp16 bit patterns (zeros of both signs, subnormals, Inf, every NaN), in either half of the words that the
    count pass compares two at a time."""
    W = np.roll(np.arange(65536, dtype=np.uint16), shift).view(np.float16).reshape(512, 128)
    packed_equal(S, np.ascontiguousarray(W.T))
    packed_equal(S, W)


@pytest.mark.parametrize("tiles", [1, 2, 3, 5, 127, 128, 129, 130, 4095, 4097, 8321])
def test_scan_lengths(S, tiles):
    """Numbers of GTiles around the scan's units (4 entries a lane, 128 a warp step, 4096 the CTA's first step)."""
    rng = np.random.Generator(np.random.PCG64(tiles))
    W = (rng.standard_normal((3, 16 * tiles)) * (rng.random((3, 16 * tiles)) < 0.4)).astype(np.float16)
    packed_equal(S, W)


def test_more_calls_at_once_than_page_locked_words(S):
    """The totals of a pack call come back in page-locked words, of which there are 64 pairs; a call that finds none copies
    instead.  80 calls that all wait behind the same work on a stream: whichever came last copied, and all of them have the same
    arrays."""
    import threading
    rng = np.random.Generator(np.random.PCG64(3))
    W = (rng.standard_normal((300, 400)) * (rng.random((300, 400)) < 0.5)).astype(np.float16)
    want = O.pack_fast(W)
    Wd = torch.from_numpy(W).cuda()
    for h in [S.spdp_pack_tiled_cbc(Wd) for _ in range(80)]:             # the words are there, and memory for all handles
        S.spdp_free(h)
    handles, stream = [None] * 80, torch.cuda.current_stream().cuda_stream
    def pack(i):
        handles[i] = S.spdp_pack_tiled_cbc(Wd, stream=stream)
    a = torch.randn(8192, 8192, device="cuda", dtype=torch.float16)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    for _ in range(1000):                                                # about three quarters of a second
        a @ a
    done.record()
    threads = [threading.Thread(target=pack, args=(i,)) for i in range(80)]
    for t in threads:
        t.start()
    started = not done.query()                                           # the work was still on its way when the last one started
    for t in threads:
        t.join()
    try:
        assert started
        for h in handles:
            got = S.spdp_export(h)
            for key in ("tileoffset", "colinfo", "bitmap", "values"):
                assert np.array_equal(got[key], want[key]), key
            info = S.spdp_get_info(h)
            assert (info.nnz, info.values_len) == (np.count_nonzero(W), len(want["values"]))
    finally:
        for h in handles:
            if h is not None:
                S.spdp_free(h)
    S.spdp_free(None)                                                    # nothing uses the words: they go, and come again
    packed_equal(S, W)
