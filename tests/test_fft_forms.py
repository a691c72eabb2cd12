"""The launch forms of the copy-fed y and z transforms."""
import ctypes

import numpy as np
import pytest


@pytest.mark.parametrize("big,ws,wide,want", [(0, 0, 0, 16), (0, 0, 1, 16), (0, 1, 0, 8), (0, 1, 1, 8), (1, 0, 0, 8), (1, 0, 1, 16),
                                              (1, 1, 0, 8), (1, 1, 1, 8)])
def test_every_form_that_the_options_ask_for_is_compiled(big, ws, wide, want):
    """Pencils per item by factor above 16, warp-specialised blocks and the wide-pencil option; a form that is not
    compiled falls back to one-shot blocks without a word."""
    from paper_2002_07627_gb300 import build
    build.build()
    assert ctypes.CDLL(build.HOSTLIB).imf_host_tma_pencils(big, ws, wide) == want


@pytest.mark.gpu
@pytest.mark.parametrize("n", [310, 385])
@pytest.mark.parametrize("wide", [0, 1, 2, -1])
def test_wide_and_narrow_pencils_of_a_big_factor_give_the_same(n, wide):
    """y and z lengths of 324 = 18 x 18 and 400 = 20 x 20, where 16 pencils with the factor no longer fit: the one-shot blocks' bits."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_07627_gb300 import binding, build, synth
    build.build()
    tool = synth.cylinder_tool(2, 5, 4, 4, synth.fibonacci_quats(3))
    rho = torch.from_numpy(synth.beam_density((20, n, n), n_beams=5, seed=2)).cuda()
    got = []
    for options in (dict(fft_tma=0), dict(fft_tma=1 | 1 << 2, fft_wide_pencils=wide)):
        imf = binding.Imf(tuple(rho.shape), precision=binding.IMF_FP32_FFT, separate_yx_passes=True, **options)
        imf.set_tools([tool])
        raw = torch.empty_like(rho)
        imf.compute(rho, raw=raw)
        imf.sync()
        got.append(raw.cpu().numpy())
        imf.close()
    assert np.array_equal(*got)
