"""The streamed minimum over sharp points (Eq. eq_imf_2): its plan on the CPU, and its results
against the tiled kernel, bit for bit, on the GPU."""
import ctypes

import numpy as np
import pytest

from paper_2002_07627_gb300 import synth


def _plan(sh, K):
    from paper_2002_07627_gb300 import build
    build.build()
    L = ctypes.CDLL(build.HOSTLIB)
    sh = np.ascontiguousarray(np.asarray(sh, np.int32).reshape(-1, 3))
    Ka = np.ascontiguousarray(K, np.int32)
    head, words = np.zeros(15, np.int32), np.zeros(1 << 18, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    n = L.imf_host_plan_stream(p(sh), len(sh), p(Ka), p(head), len(words), p(words))
    names = "P R Q stages tx rows W groups axis lists need quads ox ou ow".split()
    return n, dict(zip(names, head.tolist())), words[:max(n, 0)]


def _points(case):
    from oracle.ref import resample_tool
    rng = np.random.default_rng(case)
    if case < 6:
        t = synth.cylinder_tool(int(rng.integers(1, 7)), int(rng.integers(1, 21)), 8, 6, rng.normal(size=(1, 4)))
        return resample_tool(t, t.quats[0])["sharp"]
    if case == 6:      # scattered points: many runs of length 1
        return np.unique(rng.integers(-9, 10, (60, 3)), axis=0)
    if case == 7:      # runs longer than the longest the kernel has, both ways
        return np.array([[x, y, z] for x in range(2) for y in range(37) for z in range(20)]) - 5
    return np.array([[0, 0, 0]])


@pytest.mark.parametrize("case", range(9))
def test_stream_plan_covers_every_sharp_point_once_inside_the_copied_rows(case):
    """An output's lists, decoded with the tile origin and the window origin K alone, read every
    sharp point exactly once, only from rows and columns that the copies fill, in planes the two
    stages of the list hold; copies start at multiples of four columns, lengths taken two or four at a
    time start at multiples of that, and the lanes of a warp (8 columns, 4 planes) read 32 banks."""
    sh = np.asarray(_points(case))
    K = sh.max(0) + np.random.default_rng(case).integers(0, 6, 3)
    n, h, words = _plan(sh, K)
    assert n > 0 and n % 4 == 0
    P, Q = h["P"], h["Q"]
    assert h["ox"] % 4 == 0 and h["ox"] >= 0 and P % 4 == 0 and Q % 4 == 0 and Q >= P * h["R"]
    assert len({(x + g * Q) % 32 for x in range(8) for g in range(4)}) == 32
    assert h["stages"] >= 3 and h["stages"] * 16 * Q <= 220 * 1024
    assert h["need"] <= h["R"] and 4 * h["quads"] <= P
    u, w = (1, 2) if h["axis"] == 0 else (2, 1)
    got = []
    for m in range(h["lists"]):
        at = int(words[m])
        assert at % 4 == 0
        count = words[at:at + 4].astype(np.uint32).view(np.uint8)
        i = at + 4
        for L in range(1, 17):
            c = int(count[L - 1])
            step = 4 if L == 1 else 2 if L <= 9 else 1
            i += -i % step if c else 0
            offs = words[i:i + c]
            i += c
            for off in offs:
                assert off % 4 == 0
                k, rem = divmod(int(off) // 4, Q)
                row, col = divmod(rem, P)
                assert 0 <= k < 4
                # the last thread row and column of the block stay inside what was copied
                assert row + h["rows"] - 1 + L - 1 < h["need"] and col + h["tx"] - 1 < 4 * h["quads"]
                for j in range(L):
                    # source cell (window index) of the block's first output -> offset k = K - index
                    idx = np.zeros(3, int)
                    idx[0], idx[u], idx[w] = h["ox"] + col, h["ou"] + row + j, h["ow"] + 4 * m + k
                    got.append(tuple(K - idx))
    assert len(got) == len(set(got)) == len(sh) and set(got) == {tuple(v) for v in sh.tolist()}


def test_stream_plan_refuses_cutters_too_wide_for_its_rows():
    wide = np.array([[x, 0, 0] for x in range(60)])
    assert _plan(wide, wide.max(0))[0] == -1


def _producers(steps, stages, late, stop_at=-1):
    from paper_2002_07627_gb300 import build
    build.build()
    L = ctypes.CDLL(build.HOSTLIB)
    threads, total = late.shape
    steps = np.asarray(steps, np.int32)
    late = np.ascontiguousarray(late, np.uint8)
    how, copied = np.full(threads, -1, np.int32), np.full(threads, -1, np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    stuck = L.imf_host_stream_producers(threads, len(steps), p(steps), stages, stop_at, p(late), total, p(how), p(copied))
    return stuck, how.tolist(), copied.tolist()


@pytest.mark.parametrize("stages", [3, 5, 10])
@pytest.mark.parametrize("who", ["none", "first", "last", "all but one", "all", "at different stages"])
def test_producers_leave_together_when_a_wait_runs_out(stages, who):
    """The committed control flow of the producers on host threads, with waits that run out for some of them only:
    nobody is left at the barrier they share, and whoever is not late leaves no later than the next orientation."""
    steps = [4, 3, 6, 3, 5, 4]
    total, threads = sum(steps), 6
    for at in range(stages, total):
        late = np.zeros((threads, total), np.uint8)
        hit = {"none": [], "first": [0], "last": [threads - 1], "all but one": range(1, threads), "all": range(threads),
               "at different stages": range(threads)}[who]
        for t in hit:
            late[t, min(at + (t if who == "at different stages" else 0), total - 1):] = 1
        stuck, how, copied = _producers(steps, stages, late)
        assert not stuck
        ends = np.cumsum(steps)
        first = min((int(np.argmax(late[t])) for t in hit), default=total)
        nxt = int(ends[np.searchsorted(ends, first)]) if hit else total   # where its orientation ends
        for t in range(threads):
            own = int(np.argmax(late[t])) if late[t].any() else total
            assert copied[t] == min(own, nxt)
            assert how[t] == (0 if copied[t] == total else 2)


def test_producers_stop_together_where_no_output_has_work_left():
    stuck, how, copied = _producers([3, 4, 3], 3, np.zeros((4, 10), np.uint8), stop_at=1)
    assert not stuck and how == [1] * 4 and copied == [3] * 4


@pytest.mark.gpu
@pytest.mark.parametrize("n,r,n_orient", [((32, 24, 8), 3, 1900), ((33, 25, 9), 2, 200), ((70, 45, 37), 3, 40),
                                          ((31, 60, 17), 6, 90), ((5, 3, 2), 1, 930), ((97, 2, 30), 2, 160)])
@pytest.mark.parametrize("groups", [0, 1, 7])
def test_streamed_minimum_equals_the_tiled_one(n, r, n_orient, groups):
    """Tile edges, remainders of every axis, many orientations and several groups of them (enough for
    the streamed kernel to be chosen): the minimum of the same values, so the same bits."""
    torch = pytest.importorskip("torch")
    from paper_2002_07627_gb300 import binding, build
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    quats = np.random.default_rng(n_orient).normal(size=(n_orient, 4))
    tool = synth.cylinder_tool(r, 9, r + 2, 4, quats)
    rho = torch.from_numpy(synth.beam_density(n, n_beams=5, seed=3)).cuda()
    got = []
    for xt in (8, 0):
        imf = binding.Imf(tuple(rho.shape), erode_xt=xt, erode_groups=groups, orient_batch=n_orient,
                          precision=binding.IMF_FP32_FFT)
        imf.set_tool(0, tool.holder, tool.cutter, tool.origin, tool.quats)
        raw = torch.empty_like(rho)
        fbar, sec = imf.compute(rho, raw=raw)
        imf.sync()
        got.append((raw.clone(), fbar.clone(), sec.clone()))
        imf.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("n,cut", [((64, 32), (3, 12)), ((65, 33), (1, 1)), ((7, 100), (5, 21)), ((200, 31), (9, 40)),
                                   ((1, 1), (1, 2))])
@pytest.mark.parametrize("groups", [0, 1])
def test_planar_blocks_equal_the_3d_ones(n, cut, groups):
    """One z-plane: the tiled minimum in planar blocks against the 3D blocks (erode_xt 8), at tile edges
    and remainders: the minimum of the same values, so the same bits."""
    torch = pytest.importorskip("torch")
    from paper_2002_07627_gb300 import binding, build
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    tool = synth.planar_tool(cut[0], cut[1], cut[0] + 4, 6, n_orient=11)
    rho = torch.rand((1, n[1], n[0]), generator=torch.Generator().manual_seed(1)).cuda()
    got = []
    for xt in (8, 0):
        imf = binding.Imf(tuple(rho.shape), erode_xt=xt, erode_groups=groups)
        imf.set_tool(0, tool.holder, tool.cutter, tool.origin, tool.quats)
        raw = torch.empty_like(rho)
        imf.compute(rho, raw=raw)
        imf.sync()
        got.append(raw.clone())
        imf.close()
    assert torch.equal(*got)


def _choice(n, tool, nsm=152):
    """(streamed or not, loads of a thread per orientation, orientations with runs along y / z) for one batch of all
    the tool's orientations on an n = (nx, ny, nz) grid, from the plan that the library makes."""
    from paper_2002_07627_gb300 import binding, build
    build.build()
    imf = binding.Imf(n[::-1], plan_only=True, precision=binding.IMF_FP32_FFT)
    imf.set_tool(0, tool.holder, tool.cutter, tool.origin, tool.quats)
    info = imf.tool_info(0)
    sh = [imf.offsets(0, o, 2) for o in range(info.n_orient)]
    imf.close()
    count = np.array([len(v) for v in sh], np.int32)
    flat = np.ascontiguousarray(np.concatenate(sh), np.int32)
    K, cost, kind = np.array(info.kmax, np.int32), ctypes.c_double(), np.zeros(2, np.int32)
    L = ctypes.CDLL(build.HOSTLIB)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    got = L.imf_host_stream_faster(p(flat), p(count), len(count), p(K), *n, nsm, ctypes.byref(cost), p(kind))
    return got, cost.value, kind.tolist()


@pytest.mark.parametrize("n,r,l,n_orient,want", [
    ((200, 100, 8), 1, 1, 16, 0), ((200, 100, 8), 8, 20, 32, 0), ((400, 60, 32), 1, 3, 8, 0), ((40, 40, 40), 2, 5, 64, 0),
    ((60, 40, 90), 2, 5, 32, 0), ((48, 48, 48), 3, 20, 24, 0), ((64, 64, 1), 3, 20, 64, 0), ((128, 128, 128), 3, 20, 64, 1),
    ((96, 96, 96), 3, 20, 32, 1), ((75, 61, 50), 3, 20, 24, 1), ((128, 128, 128), 1, 1, 32, 1), ((40, 40, 40), 8, 20, 64, 1)])
def test_the_streamed_minimum_is_taken_where_it_measured_faster(n, r, l, n_orient, want):
    got, cost, kind = _choice(n, synth.cylinder_tool(r, l, r + 3, 8, synth.fibonacci_quats(n_orient)))
    assert got == want and cost > 8 and sum(kind) == n_orient


@pytest.mark.gpu
@pytest.mark.parametrize("n,r,l,n_orient", [((31, 60, 17), 6, 9, 120), ((40, 48, 40), 11, 3, 64), ((70, 45, 37), 3, 20, 64),
                                            ((97, 2, 30), 4, 9, 160), ((5, 3, 2), 4, 9, 930), ((33, 49, 17), 4, 9, 300),
                                            ((32, 24, 8), 3, 9, 1900)])
@pytest.mark.parametrize("groups", [0, 1, 7])
def test_streamed_minimum_equals_the_tiled_one_where_it_runs(n, r, l, n_orient, groups):
    """As above, on cases that the rule does give to the streamed kernel (long runs, the widest pitch and the fewest
    stages among them); a group that holds more orientations of a kind than a block can goes to the tiled kernel."""
    torch = pytest.importorskip("torch")
    from paper_2002_07627_gb300 import binding, build
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    quats = np.random.default_rng(n_orient).normal(size=(n_orient, 4))
    tool = synth.cylinder_tool(r, l, r + 2, 4, quats)
    chosen, _, kind = _choice(n, tool, torch.cuda.get_device_properties(0).multi_processor_count)
    assert chosen == 1
    assert groups != 1 or (max(kind) > 256) == (n_orient > 512)
    rho = torch.from_numpy(synth.beam_density(n, n_beams=5, seed=3)).cuda()
    got = []
    for xt in (8, 0):
        imf = binding.Imf(tuple(rho.shape), erode_xt=xt, erode_groups=groups, orient_batch=n_orient,
                          precision=binding.IMF_FP32_FFT)
        imf.set_tool(0, tool.holder, tool.cutter, tool.origin, tool.quats)
        raw = torch.empty_like(rho)
        fbar, sec = imf.compute(rho, raw=raw)
        imf.sync()
        got.append((raw.clone(), fbar.clone(), sec.clone()))
        imf.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
