"""One 2D handle on two streams: calls that shared nothing before share nothing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_update_beside_a_running_sensitivity():
    """The sensitivity's filter (a wide radius on a small grid: milliseconds on a few SMs) is still running on its stream
    while an update of other data runs on another: the sensitivity gives what it
    gives alone, bit for bit, the update to FP32 storage (its sums have no fixed order)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_07627_gb300 import binding, build, synth
    build.build()
    nx, ny = 96, 48
    force, fixed, _ = synth.cantilever2d(nx, ny)
    g = torch.Generator().manual_seed(1)
    xi, other = (torch.rand((ny, nx), generator=g).cuda() for _ in range(2))
    S = torch.rand((ny, nx), generator=g).cuda()
    to = binding.To2d(nx, ny, rmin=60.0)
    rho = torch.empty_like(xi)
    to.project(xi, rho)
    to.analyze(rho, torch.from_numpy(force).cuda(), torch.from_numpy(fixed).cuda())
    sens, new = torch.empty_like(xi), torch.empty_like(xi)
    to.sensitivity(xi, rho, sens)
    torch.cuda.synchronize()
    to.update(other, S, None, 0.5, new)
    want_sens, want_new = sens.clone(), new.clone()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(5):
        sens.zero_()
        torch.cuda.synchronize()
        to.sensitivity(xi, rho, sens, stream=a)
        to.update(other, S, None, 0.5, new, stream=b)
        torch.cuda.synchronize()
        assert torch.equal(sens, want_sens) and float((new - want_new).abs().max()) <= 1e-6
    to.close()


def test_a_huge_grid_leaves_the_device_to_others():
    """2^28 elements: the handle takes its own vectors (six of 2 doubles a node, two of a double an element), and the
    multigrid hierarchy, five times that, is left out."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_07627_gb300 import binding, build
    build.build()
    torch.zeros(1, device="cuda")
    n = 1 << 14
    own = 6 * 16 * (n + 1) ** 2 + 2 * 8 * n * n
    room = torch.cuda.mem_get_info()[0]
    if room < own + (8 << 30):
        pytest.skip("not enough free memory")
    to = binding.To2d(n, n)
    taken = room - torch.cuda.mem_get_info()[0]
    to.close()
    assert own <= taken <= own + room // 16
