"""Grids whose padded extents exceed what one block of sixteen pencils (or eight rows) holds in shared memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# padded lengths on both sides of 880 (sixteen pencils), 1709 (eight) and 3228 (four) in y and z, of 2904 (eight rows) and
# 4842 (four) in x
@pytest.mark.parametrize("shape", [(1, 760, 24), (1, 800, 24), (1, 1500, 20), (1, 1720, 20), (1, 3300, 12), (900, 7, 9), (7, 820, 9),
                                   (1, 16, 2600), (1, 16, 2900), (1, 12, 5200), (5, 6, 2950)])
def test_long_axes_match_the_oracle(shape):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_2002_07627_gb300 import binding, build, synth
    build.build()
    nz, ny, nx = shape
    rng = np.random.default_rng(sum(shape))
    rho = (rng.random(shape) * (rng.random(shape) < 0.3)).astype(np.float32)
    rho[..., : nx // 2] = 1.0
    tool = synth.planar_tool(3, 5, 5, 4, n_orient=3) if nz == 1 else synth.cylinder_tool(1, 4, 2, 3, synth.fibonacci_quats(3))
    f = oracle.imf(synth.Design(rho=rho, fixture=None, tools=[tool]))["f"]
    imf = binding.Imf(shape)
    imf.set_tools([tool])
    r = torch.from_numpy(rho).cuda()
    raw = torch.empty_like(r)
    acc = torch.empty(shape, dtype=torch.uint8, device="cuda")
    imf.compute(r, raw=raw, accessible=acc)
    imf.sync()
    assert f.max() > 0
    assert np.abs(raw.cpu().numpy() - f).max() <= 1e-4 * f.max()
    imf.close()
