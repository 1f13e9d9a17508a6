"""X does not leak into Y at the sizes that run in one kernel (2^10 to 2^14): two real IFs go through
one complex transform, and the spectra come apart only as far as bin k and bin N - k have had the same
rounding.  An IF of zeros beside a random one: outside the columns k = 0 and 16 (mod 32), which hold
their own mirrors, every operation on a bin is the conjugate of the one on its mirror, so the silent
IF's auto and the cross spectrum are zero to the bit, whatever the window, and for either IF."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn", [10, 11, 12, 13, 14])
@pytest.mark.parametrize("window", ["rect", "hann"])
@pytest.mark.parametrize("silent", [0, 1])
def test_silent_if_stays_silent(logn, window, silent):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft, n_seg = 1 << logn, 21
    rng = np.random.default_rng(logn)
    packed = [synth.pack(synth.random_codes(rng, n_seg * n_fft, 8), 8) for _ in range(2)]
    packed[silent][:] = 0
    with polaris.Spectrometer(2, 8, n_fft, window=window) as sp:
        sp.feed(packed, n_seg * n_fft)
        got = sp.integrate()
    pairs = np.arange(n_fft // 2 + 1) % 16 != 0
    assert np.all(got["autos"][1 - silent] > 0)
    assert np.all(got["autos"][silent][pairs] == 0)
    assert np.all(got["cross"][0][pairs] == 0)
    assert np.all(got["autos"][silent] <= 1e-10 * got["autos"][1 - silent].mean())  # (columns 0 and 16: rounding, squared)
