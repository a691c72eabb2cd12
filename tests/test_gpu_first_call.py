"""The first call of a handle, on a stream that is not ordered with the default stream."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dirty_small_allocations(n=2048, size=512):
    """Fills small device blocks and frees every other one (the rest keep the pages), so that the next small
    allocations hold 0x7f bytes; returns what frees the rest."""
    cu = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    ptrs = []
    for _ in range(n):
        p = ctypes.c_uint64()
        assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        assert cu.cuMemsetD8_v2(p, ctypes.c_ubyte(0x7f), ctypes.c_size_t(size)) == 0
        ptrs.append(p)
    torch.cuda.synchronize()
    for p in ptrs[::2]:
        assert cu.cuMemFree_v2(p) == 0
    return lambda: [cu.cuMemFree_v2(p) for p in ptrs[1::2]]


@pytest.mark.parametrize("shape", [(1, 24, 40), (20, 40, 60)])
def test_penalty_as_first_call_while_the_default_stream_is_busy(shape):
    """Fresh handle, small words in dirty memory, default stream busy, penalty on a non-blocking stream, twice:
    both divide by the maximum of their own input (both launch forms, below and above the small-grid limit)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_07627_gb300 import binding, build
    build.build()
    g = torch.Generator().manual_seed(0)
    s0, rho, fbar = (torch.rand(shape, generator=g).cuda() + 0.1 for _ in range(3))
    sec = torch.zeros(shape, dtype=torch.uint8, device="cuda")
    ref = (0.5 * s0.double() / float(s0.max()) + 0.5 * torch.where(rho > 0.5, fbar, torch.zeros_like(fbar)).double()).cpu().numpy()
    stream = torch.cuda.Stream()
    warm = binding.Imf(shape)                     # loads the kernels, which may wait for the device
    warm.penalize(s0.clone(), rho, fbar, sec, w_acc=0.5)
    warm.sync()
    release = _dirty_small_allocations()
    imf = binding.Imf(shape)
    sens = [s0.clone() for _ in range(2)]
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)                # a fifth of a second on the default stream
    with torch.cuda.stream(stream):
        for s in sens:
            imf.penalize(s, rho, fbar, sec, w_acc=0.5, stream=stream)
    torch.cuda.synchronize()
    for s in sens:
        assert np.abs(s.cpu().numpy() - ref).max() <= 4e-7 * max(1.0, np.abs(ref).max())
    imf.close()
    warm.close()
    release()
