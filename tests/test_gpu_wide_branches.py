"""Branches of the large sizes (2^15 to 2^20) that whole-segment inputs of a few segments do not reach,
against the FP64 oracle: more column groups than one wave over the CTAs, with a ragged rest, where a
copied chunk holds several tiles; input off a 16-byte boundary or with such a hop, which tensor maps
cannot describe, with carried samples and an IF without a partner; synchronous host feeds large enough
to go over in pieces, with overlap and code statistics.

Tolerance: the FP32 bar of the parity tests (1e-5 per channel), denominators floored at 5% of the
channel mean because few segments leave some bins nearly empty.  Code counts are equal."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth
from tests.helpers import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    return torch, polaris


def _streams(seed, n_if, n, bits):
    rng = np.random.default_rng(seed)
    return [synth.pack(synth.random_codes(rng, n, bits), bits) for _ in range(n_if)]


# with one CTA per SM a wave is 152 chunks of 16 bytes: 38, 19 and 9.5 pair-segments of 2^18 at 1, 2
# and 4 bits, 38 and 19 of 2^19 at 1 and 2 bits
@pytest.mark.parametrize("logn,bits,n_seg", [(18, 1, 21), (18, 2, 11), (18, 4, 13), (19, 1, 20), (19, 2, 12)])
def test_full_waves_and_a_rest(env, orc, logn, bits, n_seg):
    _, polaris = env
    n = n_seg << logn
    packed = _streams(logn + bits, 3, n, bits)  # (two FFT pairs, one without a second IF)
    with polaris.Spectrometer(3, bits, 1 << logn, pairs=[(0, 2)], window="hann") as sp:
        sp.set_launch_caps(1, 0)
        sp.feed(packed, n)
        got = sp.integrate()
    ref = orc.spectrometer(packed, bits, 1 << logn, n, window_kind=1, pairs=[(0, 2)])
    assert got["n_segments"] == n_seg
    assert_close(got, ref, [(0, 2)], 1e-5, floor_frac=0.05)


@pytest.mark.parametrize("logn,bits,odd_hop", [(17, 4, False), (18, 2, False), (18, 8, True), (19, 1, True), (20, 4, False)])
def test_input_off_a_16_byte_boundary(env, orc, logn, bits, odd_hop):
    torch, polaris = env
    n_fft, spw = 1 << logn, 32 // bits
    hop = n_fft // 2 + (spw if odd_hop else 0)  # (words per hop: odd, or a multiple of four)
    n = n_fft + 4 * hop + 3 * spw
    packed = _streams(3 * logn + bits, 3, n, bits)
    dev = [torch.from_numpy(np.concatenate([np.zeros(1, np.uint32), p]).view(np.int32)).cuda()[1:] for p in packed]
    assert all(d.data_ptr() % 16 == 4 for d in dev)
    cuts = [0, n_fft + 5 * spw, n_fft + 2 * hop, n]  # samples are carried over each cut
    with polaris.Spectrometer(3, bits, n_fft, hop=hop, pairs=[(0, 1)]) as sp:
        for a, b in zip(cuts, cuts[1:]):
            sp.feed([d[a // spw:b // spw] for d in dev], b - a)
        got = sp.integrate()
    ref = orc.spectrometer(packed, bits, n_fft, n, hop=hop, pairs=[(0, 1)])
    assert got["n_segments"] == ref["n_segments"] == 5
    assert_close(got, ref, [(0, 1)], 1e-5, floor_frac=0.05)


@pytest.mark.parametrize("logn,n_feed", [(15, 3 << 21), (16, (1 << 22) + 4096), (18, 1 << 23)])
def test_host_feed_in_pieces(env, orc, logn, n_feed):
    _, polaris = env
    n_fft, bits, n_if = 1 << logn, 8, 4  # (8 MB a piece: 24, 16 and 32 MB of input)
    hop = n_fft // 2
    n = n_feed + hop  # and a second feed that finds samples carried
    packed = _streams(logn, n_if, n, bits)
    with polaris.Spectrometer(n_if, bits, n_fft, hop=hop, code_stats=True) as sp:
        sp.feed([p[:n_feed // 4] for p in packed], n_feed)
        sp.feed([p[n_feed // 4:] for p in packed], hop)
        got = sp.integrate()
        counts = sp.code_histogram()
    ref = orc.spectrometer(packed, bits, n_fft, n, hop=hop)
    assert got["n_segments"] == ref["n_segments"]
    assert_close(got, ref, [(0, 2), (1, 3)], 1e-5, floor_frac=0.05)
    assert np.array_equal(counts, orc.code_histogram(packed, bits, n_fft, n, hop=hop))
