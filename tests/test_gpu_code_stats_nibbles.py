"""4-bit code counts where the nibble counters fill up: constant streams (every word of a thread
adds to one code), at word counts around a block's 15 words per thread; counts are exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", [0, 6, 15])
@pytest.mark.parametrize("n_seg", [1, 59, 60, 61, 307])  # 128 words each; a block pass takes 7680
def test_constant_streams_count_exactly(code, n_seg):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft = 1024
    words = np.full(n_seg * n_fft // 8, code * 0x11111111, np.uint32)
    other = np.full(n_seg * n_fft // 8, 0xFEDCBA98, np.uint32)  # codes 8 to 15, one each per word
    with polaris.Spectrometer(2, 4, n_fft, code_stats=True) as sp:
        for _ in range(2):
            sp.feed([words, other], n_seg * n_fft)
        got = sp.code_histogram()
    want = np.zeros((2, 16), np.uint64)
    want[0, code] = 2 * n_seg * n_fft
    want[1, 8:] = 2 * n_seg * n_fft // 8
    assert np.array_equal(got, want)
