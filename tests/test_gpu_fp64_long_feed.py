"""FP64 integration accumulators over one long feed at the sizes that run in one kernel (2^10 to
2^14), which sums a few segments in FP32 before it adds to them.  The feed repeats one segment, so
that every term of a bin's sum is the same FP32 value P, which an integration of that segment alone
reports, and what is left of |sum - S P| is the rounding of the summation.

Tolerance: a chain of n additions of equal terms in FP32 is off by at most 2^-24 (n + 1) / 2 of its
sum; n <= 14 segments; the two readouts round to FP32 once each, 2^-24 apiece: 9.5 x 2^-24.  A
cross spectrum's components are such sums too, no larger than sqrt(A_a A_b)."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 9.5 * 2.0 ** -24


@pytest.mark.parametrize("logn", [10, 11, 12, 13, 14])
@pytest.mark.parametrize("n_if,extra", [(2, 0), (3, 5)])  # (3: one IF without a partner; a ragged last round)
def test_long_feed_keeps_fp64_sums(logn, n_if, extra):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft, bits = 1 << logn, 1
    n_seg = (300 * 2432 >> (logn - 10)) + extra  # 300 segments for each of the teams that an SM's warps make up
    rng = np.random.default_rng(logn)
    one = [torch.from_numpy(synth.pack(synth.random_codes(rng, n_fft, bits), bits).view(np.int32)).cuda()
           for _ in range(n_if)]
    pairs = [(0, 1)]
    got = []
    with polaris.Spectrometer(n_if, bits, n_fft, pairs=pairs, accum_fp64=True) as sp:
        for reps in (1, n_seg):
            sp.feed([w.repeat(reps) for w in one], reps * n_fft)
            torch.cuda.synchronize()
            got.append(sp.integrate())
    p, s = got
    assert s["n_segments"] == n_seg
    autos = n_seg * p["autos"].astype(np.float64)
    scale = np.maximum(autos, np.finfo(np.float64).tiny)
    assert np.max(np.abs(s["autos"] - autos) / scale) <= TOL
    for part in ("real", "imag"):
        c = n_seg * getattr(p["cross"][0], part).astype(np.float64)
        err = np.abs(getattr(s["cross"][0], part) - c) / np.sqrt(scale[0] * scale[1])
        assert np.max(err) <= TOL, part
