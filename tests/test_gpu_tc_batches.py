"""The tensor-core passes where a batch (32 MB: 1024 segments of 4096 points, 16 of 2^18) ends: one
segment, part of a tile, just under, at and over one batch, and several batches.  The same segments
fed one at a time give the same FP32 products per segment (whether those are right is checked
against the oracle elsewhere), summed in FP64 instead of by compensated FP32 sums per batch, whose
error is at most 2 u times the sum of the terms' magnitudes (u = 2^-24): 1.2e-7 of an auto spectrum,
and of sqrt(A_a A_b) for a cross spectrum's parts (Cauchy-Schwarz).  The bound 3e-7 leaves a factor
of two for second-order terms."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fft,n_seg", [(4096, 1), (4096, 3), (4096, 1023), (4096, 1025), (4096, 2100), (262144, 1),
                                         (262144, 16), (262144, 17)])
@pytest.mark.parametrize("precision", ["fp16x3", "bf16"])
def test_batches_equal_single_segments(n_fft, n_seg, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    rng = np.random.default_rng(n_fft + n_seg)
    words = rng.integers(-2**31, 2**31, (2, n_seg, n_fft // 16), dtype=np.int64).astype(np.int32)
    dev = torch.from_numpy(words).cuda()
    got = []
    for whole in (True, False):
        with polaris.TensorCoreSpectrometer(2, n_fft, precision, "hann") as tc:
            if whole:
                tc.feed([dev[0], dev[1]], n_seg * n_fft)
            else:
                for s in range(n_seg):
                    tc.feed([dev[0, s], dev[1, s]], n_fft)
            got.append(tc.integrate())
    a, b = got
    assert a["n_segments"] == b["n_segments"] == n_seg
    assert np.all(np.abs(a["autos"] - b["autos"]) <= 3e-7 * b["autos"])
    scale = np.sqrt(b["autos"][0] * b["autos"][1])
    assert np.all(np.abs((a["cross"] - b["cross"]).real) <= 3e-7 * scale)
    assert np.all(np.abs((a["cross"] - b["cross"]).imag) <= 3e-7 * scale)
