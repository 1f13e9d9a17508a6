"""The sizes whose whole path runs in one kernel (2^10 to 2^14) against the FP64 oracle, at its
edges: fewer segments than one team takes, uneven ranges over the teams, groups of staged
segments that end early, one to eight IFs (pairs with and without a second IF, CTAs shared
unevenly between pairs), segments split between staged and new input, launch caps, FP64 sums.

Tolerance: the FP32 bar of the parity tests (1e-5 per channel), denominators floored at 5% of
the channel mean because few segments leave some bins nearly empty."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth
from tests.helpers import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn", [10, 11, 12, 13, 14])
@pytest.mark.parametrize("bits,n_if,n_seg,hop_half,window,kw", [
    (1, 2, 1, False, "rect", {}),
    (1, 5, 37, False, "hann", {"pairs": [(3, 1)]}),
    (2, 1, 9, False, "taps", {}),
    (2, 4, 701, True, "rect", {"accum_fp64": True}),
    (4, 3, 33, False, "taps", {"pairs": [(0, 2)]}),
    (4, 8, 5, True, "hann", {}),
    (8, 2, 2467, False, "hann", {}),
    (8, 6, 13, True, "taps", {"caps": (1, 0)}),
])
def test_one_kernel_sizes_match_oracle(orc, logn, bits, n_if, n_seg, hop_half, window, kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    kw = dict(kw)
    caps = kw.pop("caps", None)
    n_fft = 1 << logn
    hop = n_fft // 2 if hop_half else n_fft
    spw = 32 // bits
    n = (n_seg - 1) * hop + n_fft + 3 * spw  # and a few samples carried
    rng = np.random.default_rng(1000 * logn + 10 * bits + n_if)
    packed = [synth.pack(synth.random_codes(rng, n, bits), bits) for _ in range(n_if)]
    taps = rng.uniform(0.2, 1.0, n_fft).astype(np.float32) if window == "taps" else None
    cut = (n // 3) // spw * spw
    got = []
    for feeds in ([n], [cut, n - cut]):
        with polaris.Spectrometer(n_if, bits, n_fft, hop=hop, window=window if taps is None else taps, **kw) as sp:
            if caps:
                sp.set_launch_caps(*caps)
            at = 0
            for m in feeds:
                sp.feed([p[at // spw:(at + m) // spw] for p in packed], m)
                at += m
            got.append(sp.integrate())
    ref = orc.spectrometer(packed, bits, n_fft, n, hop=hop, window_kind={"rect": 0, "hann": 1, "taps": 2}[window],
                           taps=taps, pairs=kw.get("pairs"))
    pairs = kw.get("pairs", [(i, i + n_if // 2) for i in range(n_if // 2)] if n_if % 2 == 0 else [])
    for r in got:
        assert r["n_segments"] == n_seg
        assert_close(r, ref, pairs, 1e-5, floor_frac=0.05)


def test_second_integration_starts_from_zero(orc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    rng = np.random.default_rng(12)
    packed = [synth.pack(synth.random_codes(rng, 300 * 2048, 4), 4) for _ in range(2)]
    with polaris.Spectrometer(2, 4, 2048) as sp:
        res = []
        for _ in range(2):
            sp.feed(packed, 300 * 2048)
            res.append(sp.integrate())
    ref = orc.spectrometer(packed, 4, 2048, 300 * 2048)
    for r in res:
        assert_close(r, ref, [(0, 1)], 1e-5)
