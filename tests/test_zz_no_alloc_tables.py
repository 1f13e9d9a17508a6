"""The allocation-free entry point builds its twiddle table in its static array on every call.
Calls of different sizes that follow one another in one stream, without a synchronisation between
them and with a rectangular window (the table's writer is then the kernel just before the
transform), each take their own table: against the FP64 oracle at the tolerance of the parity
tests.  Sizes that run in one kernel and sizes that run in two; the default stream and another.
Collected last, like the entry point's other tests."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth
from tests.helpers import assert_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_stream", [False, True])
def test_alternating_sizes_in_one_stream(orc, own_stream):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    calls = []
    for i, logn in enumerate([10, 14, 11, 13, 12, 10, 16, 14, 9, 12, 13, 11]):
        n_fft, bits = 1 << logn, (2, 8, 4, 1)[i % 4]
        n_seg = max(4, (1 << 17) >> logn)  # denominators need a few segments per channel
        packed = [synth.pack(synth.random_codes(np.random.default_rng(60 + 2 * i + k), n_seg * n_fft, bits), bits)
                  for k in range(2)]
        nb = n_fft // 2 + 1
        dev = [torch.from_numpy(p.view(np.int32)).cuda() for p in packed]
        out = [torch.zeros(s, device="cuda") for s in ((2, nb), (1, nb, 2), (1, 4, nb))]
        calls.append((n_fft, bits, n_seg, packed, dev, out))
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    for _ in range(3):
        for n_fft, bits, n_seg, _packed, dev, out in calls:
            assert polaris.run_noalloc(dev, n_seg * n_fft, bits, n_fft, *out, stream=stream) == n_seg
        torch.cuda.synchronize()
        for n_fft, bits, n_seg, packed, _dev, (a, c, s) in calls:
            c = c.cpu().numpy()
            got = {"autos": a.cpu().numpy(), "cross": c[..., 0] + 1j * c[..., 1], "stokes": s.cpu().numpy()}
            ref = orc.spectrometer(packed, bits, n_fft, n_seg * n_fft)
            assert_close(got, ref, [(0, 1)], 1e-5, floor_frac=0.05)
            a.zero_()
