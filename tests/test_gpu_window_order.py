"""The window taps in the order phase 1 takes them (N >= 2^13): random taps, every one of them
different, so that a tap in a wrong place shows; against the FP64 oracle.

Tolerance: the FP32 bar of the parity tests (1e-5 per channel), denominators floored at 5% of
the channel mean because three segments leave some bins nearly empty."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth
from tests.helpers import assert_close

pytestmark = pytest.mark.gpu


# the smallest ordered size and the one below it, 16, 32 and 64 rows per lane, 4, 2 and 1 columns
# per warp, unstaged input (1 bit, 2^19 and 2^20)
@pytest.mark.parametrize("logn,bits", [(12, 2), (13, 2), (14, 8), (15, 1), (17, 4), (18, 8), (19, 1), (19, 2), (20, 1),
                                       (20, 8)])
def test_random_taps_match_oracle(orc, logn, bits):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft, n_seg = 1 << logn, 3
    rng = np.random.default_rng(31 * logn + bits)
    packed = [synth.pack(synth.random_codes(rng, n_seg * n_fft, bits), bits) for _ in range(3)]
    taps = rng.uniform(0.2, 1.0, n_fft).astype(np.float32)
    with polaris.Spectrometer(3, bits, n_fft, window=taps, pairs=[(0, 2)]) as sp:
        sp.feed(packed, n_seg * n_fft)
        got = sp.integrate()
    ref = orc.spectrometer(packed, bits, n_fft, n_seg * n_fft, window_kind=2, taps=taps, pairs=[(0, 2)])
    assert_close(got, ref, [(0, 2)], 1e-5, floor_frac=0.05)
