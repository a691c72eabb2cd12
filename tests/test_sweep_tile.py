"""The sweep on staged tiles (Eq. eq_conv_A): its plan on the CPU, and its results against the kernel on
dilation levels, bit for bit, on the GPU."""
import ctypes

import numpy as np
import pytest

from paper_2002_07627_gb300 import synth


def _plan(rk, K, kmin, nx):
    from paper_2002_07627_gb300 import build
    build.build()
    L = ctypes.CDLL(build.HOSTLIB)
    c = lambda a: np.ascontiguousarray(a, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    rk, K, kmin = c(np.reshape(rk, (-1, 3))), c(K), c(kmin)
    head, words = np.zeros(12, np.int32), np.zeros(1 << 18, np.int32)
    n = L.imf_host_plan_sweep(p(rk), len(rk), p(K), p(kmin), nx, p(head), len(words), p(words))
    return n, dict(zip("nq nl ppw UP somax planes smem axis eu ew ou ow".split(), head.tolist())), words[:max(n, 0)]


@pytest.mark.parametrize("case", range(8))
@pytest.mark.parametrize("nx", [5, 32, 33, 256, 1200])
def test_sweep_plan_covers_every_cutter_voxel_once_inside_the_tile(case, nx):
    """The slices' shifts and the runs' offsets, decoded with the window origin K alone, are the cutter's
    offsets, each once; the last thread's reads stay inside the staged tile; shifts fall by whole words."""
    from oracle.ref import resample_tool
    rng = np.random.default_rng(case)
    if case < 5:
        t = synth.cylinder_tool(int(rng.integers(1, 7)), int(rng.integers(1, 21)), 8, 6, rng.normal(size=(1, 4)))
        rk = resample_tool(t, t.quats[0])["RK"]
    elif case == 5:
        rk = np.unique(rng.integers(-9, 10, (60, 3)), axis=0)
    elif case == 6:
        rk = np.array([[x, y, z] for x in range(70) for y in range(20) for z in range(2)]) - 4
    else:
        rk = np.array([[0, 0, 0]])
    rk = np.asarray(rk)
    K, kmin = rk.max(0) + rng.integers(0, 4, 3), rk.min(0) - rng.integers(0, 4, 3)
    n, h, words = _plan(rk, K, kmin, nx)
    assert n > 0 and h["nl"] * h["ppw"] <= 32 and h["nl"] == h["nq"] + h["somax"] + 1 and h["UP"] % 2 == 1
    u, w = (1, 2) if h["axis"] == 0 else (2, 1)
    got, i, last = [], 0, 1 << 30
    while i < n:
        s = int(words[i])
        so, sh, c = s & 255, (s >> 8) & 31, s >> 16
        assert so <= last and so <= h["somax"] and c > 0
        last = so
        for d in words[i + 1:i + 1 + c]:
            L, off = int(d) >> 24, int(d) & 0xffffff
            pl, rem = divmod(off, h["nl"] * h["UP"])
            assert rem < h["UP"] and 1 <= L <= 16
            assert rem + 31 + L - 1 < 32 + h["eu"] <= h["UP"] and pl + h["ppw"] * 2 - 1 < h["planes"] and pl <= h["ew"]
            for j in range(L):
                k = np.zeros(3, int)
                k[0], k[u], k[w] = K[0] - (32 * so + sh), K[u] - (h["ou"] + rem + j), K[w] - (h["ow"] + pl)
                got.append(tuple(k))
        i += 1 + c
    assert len(got) == len(set(got)) == len(rk) and set(got) == {tuple(v) for v in rk.tolist()}


@pytest.mark.gpu
@pytest.mark.parametrize("n,r,n_orient", [((32, 32, 6), 2, 5), ((33, 31, 7), 3, 6), ((97, 40, 35), 3, 9), ((250, 12, 20), 6, 4),
                                          ((1100, 9, 5), 2, 3), ((64, 90, 1), 0, 8), ((5, 3, 2), 1, 3)])
@pytest.mark.parametrize("sets", [False, True])
def test_tiled_sweep_equals_the_sweep_on_levels(n, r, n_orient, sets):
    """Word and tile edges, several words per row tile, planar and tiny grids; the union and the
    per-orientation sets: the same bits as the kernel that walks dilation levels (sweep_loop)."""
    torch = pytest.importorskip("torch")
    from paper_2002_07627_gb300 import binding, build
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    if r:
        tool = synth.cylinder_tool(r, 15, r + 2, 5, np.random.default_rng(n_orient).normal(size=(n_orient, 4)))
        rho = synth.beam_density(n, n_beams=6, seed=3)
    else:
        tool = synth.planar_tool(n_orient=n_orient)
        rho = synth.planar_density(n[0], n[1], seed=2)
    rho = torch.from_numpy(rho).cuda()
    got = []
    for loop in (True, False):
        imf = binding.Imf(tuple(rho.shape), accessible_by_sweep=True, sweep_loop=loop, orient_batch=4)
        imf.set_tools([tool])
        acc = torch.empty(rho.shape, dtype=torch.uint8, device="cuda")
        imf.compute(rho, accessible=acc)
        out = [acc]
        if sets:
            s, _, _ = imf.accessible_sets(rho)
            out.append(s)
            # the union of the sets is the accessible output
            bits = np.unpackbits(s.cpu().numpy().view(np.uint8), axis=-1, bitorder="little")[..., :n[0]]
            assert np.array_equal(bits.any(0), acc.cpu().numpy() != 0)
        imf.sync()
        got.append(out)
        imf.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


def _choice(n, tool, nsm=152):
    """(staged or not, runs of the cutter along x) for one batch of all the tool's orientations on an n = (nx, ny, nz)
    grid, from the plan that the library makes."""
    from paper_2002_07627_gb300 import binding, build
    build.build()
    imf = binding.Imf(n[::-1], plan_only=True, precision=binding.IMF_FP32_FFT)
    imf.set_tool(0, tool.holder, tool.cutter, tool.origin, tool.quats)
    info = imf.tool_info(0)
    rk = [imf.offsets(0, o, 1) for o in range(info.n_orient)]
    imf.close()
    count = np.array([len(v) for v in rk], np.int32)
    flat = np.ascontiguousarray(np.concatenate(rk), np.int32)
    K, kmin, runs = np.array(info.kmax, np.int32), flat.min(0).astype(np.int32), ctypes.c_double()
    L = ctypes.CDLL(build.HOSTLIB)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    got = L.imf_host_sweep_faster(p(flat), p(count), len(count), p(K), p(kmin), *n, nsm, ctypes.byref(runs))
    want = np.mean([len({(y, z, x) for x, y, z in v.tolist()} - {(y, z, x + 1) for x, y, z in v.tolist()}) for v in rk])
    assert abs(runs.value - want) <= 1e-9 * want
    return got


@pytest.mark.parametrize("n,r,l,n_orient,want", [
    ((40, 40, 40), 11, 30, 3, 0), ((40, 40, 40), 11, 30, 32, 0), ((200, 100, 8), 8, 20, 64, 0), ((96, 96, 96), 11, 30, 8, 0),
    ((128, 128, 128), 11, 30, 32, 0), ((48, 48, 48), 3, 20, 16, 0), ((40, 40, 40), 1, 1, 8, 0), ((128, 128, 128), 3, 20, 64, 1),
    ((256, 256, 256), 3, 20, 64, 1), ((96, 96, 96), 6, 12, 32, 1), ((400, 60, 32), 11, 3, 64, 1), ((256, 64, 32), 6, 12, 64, 1)])
def test_the_staged_sweep_is_taken_where_it_measured_faster(n, r, l, n_orient, want):
    assert _choice(n, synth.cylinder_tool(r, l, r + 3, 8, synth.fibonacci_quats(n_orient))) == want


@pytest.mark.gpu
@pytest.mark.parametrize("n,r,l,n_orient", [((97, 70, 67), 4, 9, 48), ((33, 63, 65), 5, 9, 96), ((31, 32, 64), 5, 9, 128),
                                             ((65, 97, 31), 6, 5, 96), ((20, 40, 160), 6, 5, 64), ((5, 64, 32), 6, 5, 256),
                                             ((1100, 40, 24), 6, 9, 48)])
def test_tiled_sweep_equals_the_sweep_on_levels_where_it_runs(n, r, l, n_orient):
    """As above, on cases that the rule does give to the staged tiles, at word and tile edges."""
    torch = pytest.importorskip("torch")
    from paper_2002_07627_gb300 import binding, build
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    tool = synth.cylinder_tool(r, l, r + 2, 5, np.random.default_rng(n_orient).normal(size=(n_orient, 4)))
    assert _choice(n, tool, torch.cuda.get_device_properties(0).multi_processor_count) == 1
    rho = torch.from_numpy(synth.beam_density(n, n_beams=6, seed=3)).cuda()
    got = []
    for loop in (True, False):
        imf = binding.Imf(tuple(rho.shape), accessible_by_sweep=True, sweep_loop=loop, orient_batch=n_orient,
                          precision=binding.IMF_FP32_FFT)
        imf.set_tools([tool])
        acc = torch.empty(rho.shape, dtype=torch.uint8, device="cuda")
        imf.compute(rho, accessible=acc)
        sets, _, _ = imf.accessible_sets(rho)
        imf.sync()
        got.append((acc, sets))
        imf.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
