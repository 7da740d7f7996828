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
