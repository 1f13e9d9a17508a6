"""The leakage calibration's size-specialised segment kernels (2^9 to 2^14) against its kernels for
any N (which a call with unaligned buffers takes) at every size and width: one segment, one more
than the SMs, and enough for several CTAs per SM and more than one segment in each.  With a zero
target the residual is the spectrum itself.  Both sides are FP32 transforms of at most 14 levels,
two per segment in the window's gradient: a relative error (2-norm) of at most 2 * 14 * u = 1.7e-6
(u = 2^-24) each, doubled in the loss, a square: 1e-5 bounds the difference of any output."""
import numpy as np
import pytest

from paper_1412_1256_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn", range(9, 15))
@pytest.mark.parametrize("bits", [1, 2, 4, 8])
def test_sized_kernels_equal_general_ones(logn, bits):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft, nb = 1 << logn, (1 << logn) // 2 + 1
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(100 * logn + bits)
    for nseg in (1, sms + 1, (2 * sms if logn >= 13 else 8 * sms) + 3):
        words = torch.from_numpy(rng.integers(-2**31, 2**31, (2, nseg * n_fft * bits // 32), dtype=np.int64).astype(np.int32)).cuda()
        window = torch.from_numpy(rng.uniform(0.2, 1.0, n_fft).astype(np.float32)).cuda()
        gains = torch.tensor([1.1, 0.2, 0.9, -0.3], device="cuda")
        leak = torch.from_numpy(rng.uniform(-0.03, 0.03, (2, nb, 2)).astype(np.float32)).cuda()
        target = torch.zeros((4, nb), device="cuda")

        def off(x):  # one 4-byte element past a 16-byte boundary
            y = torch.zeros(x.numel() + 1, dtype=x.dtype, device="cuda")[1:]
            y.copy_(x)
            return y

        with polaris.Adjoint(n_fft, bits) as adj:
            a = adj.run([words[0].clone(), words[1].clone()], nseg * n_fft, window, gains, leak, target, grads=True)
            b = adj.run([off(words[0]), off(words[1])], nseg * n_fft, off(window), gains, leak, target, grads=True)
            torch.cuda.synchronize()
        for key in b:
            x, y = a[key].double(), b[key].double()
            assert float((x - y).norm()) <= 1e-5 * float(y.norm()), (nseg, key)


@pytest.mark.parametrize("logn", [5, 6, 7, 8])
@pytest.mark.parametrize("bits", [1, 2, 4, 8])
def test_small_sizes_equal_oracle(orc, logn, bits):
    """N = 2^5 to 2^8 (many segments per CTA) against the FP64 oracle: one segment, a few, one more than the
    groups of the forward pass (eight per SM), and several rounds of a CTA's teams with a ragged end.
    The bound is the one above (one side is exact here)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_1256_gb300 import polaris

    n_fft, nb = 1 << logn, (1 << logn) // 2 + 1
    groups = 8 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(100 * logn + bits)
    window = rng.uniform(0.2, 1.0, n_fft).astype(np.float32)
    gains = np.array([1.1, 0.2, 0.9, -0.3], np.float32)
    leak = rng.uniform(-0.03, 0.03, (2, nb, 2)).astype(np.float32)
    target = np.zeros((4, nb), np.float32)
    dev = [torch.from_numpy(x).cuda() for x in (window, gains, leak, target)]
    for nseg in (1, 3, groups + 1, 5 * groups + 7):
        n = nseg * n_fft
        host = [rng.integers(0, 2**32, n * bits // 32, dtype=np.uint32) for _ in range(2)]
        st, loss = orc.leak_forward(host, bits, n_fft, n, window, gains, leak, target)
        gw, gg, gd = orc.leak_grad(host, bits, n_fft, n, window, gains, leak, target)
        with polaris.Adjoint(n_fft, bits) as adj:
            r = adj.run([torch.from_numpy(h.view(np.int32)).cuda() for h in host], n, *dev, grads=True)
            torch.cuda.synchronize()
        for key, ref in (("stokes", st), ("loss", loss), ("grad_window", gw), ("grad_gains", gg), ("grad_leak", gd)):
            x, y = r[key].cpu().numpy().astype(np.float64).ravel(), np.asarray(ref, np.float64).ravel()
            assert np.linalg.norm(x - y) <= 1e-5 * np.linalg.norm(y), (nseg, key)
