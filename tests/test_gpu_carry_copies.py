"""Streams fed in uneven pieces (all copies of a feed between carry, staging and input in one
kernel): single words, pieces that complete no segment, several segments at once, pieces that
start off a 16-byte boundary, host and device input; against the FP64 oracle.

Tolerance: the FP32 bar of the parity tests (1e-5 per channel), denominators floored at 5% of
the channel mean because few segments leave some bins nearly empty."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth
from tests.helpers import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn,bits,n_if,hop_div", [(4, 8, 1, 1), (9, 2, 3, 2), (10, 1, 8, 4), (12, 4, 3, 1), (13, 8, 2, 2),
                                                    (17, 2, 4, 1)])
@pytest.mark.parametrize("device", [False, True])
def test_uneven_pieces_match_oracle(orc, logn, bits, n_if, hop_div, device):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft, spw = 1 << logn, 32 // bits
    hop = n_fft // hop_div
    seg_words = n_fft // spw
    rng = np.random.default_rng(97 * logn + bits)
    # words per piece: 1, 3, nothing whole, just over one segment, several segments, the rest
    pieces = [1, 3, max(1, seg_words - 5), seg_words + 1, 3 * seg_words + 2, 1, 2 * seg_words]
    n = sum(pieces) * spw
    packed = [synth.pack(synth.random_codes(rng, n, bits), bits) for _ in range(n_if)]
    src = [torch.from_numpy(p.view(np.int32)).cuda() for p in packed] if device else packed
    with polaris.Spectrometer(n_if, bits, n_fft, hop=hop) as sp:
        at = 0
        for m in pieces:
            sp.feed([p[at:at + m] for p in src], m * spw)
            at += m
        got = sp.integrate()
    ref = orc.spectrometer(packed, bits, n_fft, n, hop=hop)
    assert got["n_segments"] == ref["n_segments"]
    pairs = [(i, i + n_if // 2) for i in range(n_if // 2)] if n_if % 2 == 0 else []
    assert_close(got, ref, pairs, 1e-5, floor_frac=0.05)
