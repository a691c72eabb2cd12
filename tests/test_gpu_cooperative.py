"""The cooperative kernels: the multigrid-preconditioned conjugate gradient and the update of the 2D
optimisation loop against the oracle's, at the sizes where the hierarchy changes shape, and the greedy
process plan."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _need():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2002_07627_gb300 import binding, build
    build.build()
    return binding


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# one element; the coarsest grid alone; one level inside a block; thin strips; odd and even extents on
# both sides of the block-wide and grid-wide levels; clamped dofs anywhere
@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 7), (4, 4), (9, 1), (1, 40), (31, 31), (32, 31), (37, 23), (130, 3),
                                   (64, 64), (101, 67), (256, 128)])
@pytest.mark.parametrize("clamp", ["edge", "scattered"])
def test_multigrid_cg_matches_the_direct_solve(nx, ny, clamp):
    """The residual of the returned displacements is the iteration's 1e-11 |f| plus what its recurrence
    can drift from the true one in FP64, at most about eps |K| |u| an iteration (Greenbaum's bound; on the
    long strips |u| reaches 1e9 |f|, and the direct solve's own residual is 1e-8 |f|); displacements and
    compliance agree with the direct solve."""
    binding = _need()
    from oracle import to2d
    rng = np.random.default_rng(nx * 1000 + ny)
    rho = rng.uniform(0.0, 1.0, (ny, nx)).astype(np.float32)
    ndof = 2 * (nx + 1) * (ny + 1)
    fixed = np.zeros(ndof, np.uint8)
    if clamp == "edge":
        left = np.arange(ny + 1) * (nx + 1)
        fixed[2 * left] = fixed[2 * left + 1] = 1
    else:
        fixed[rng.choice(ndof, max(3, ndof // 9), replace=False)] = 1
        fixed[[0, 1]] = 1                    # no rigid motion left
        fixed[ndof - 1] = 1
    force = rng.standard_normal(ndof)
    to = binding.To2d(nx, ny, cg_tol=1e-11)
    # a force at an odd FP64 offset: the caller's arrays carry no alignment beyond their type
    buf = torch.empty(ndof + 1, dtype=torch.float64, device="cuda")
    f_d = buf[1:]
    f_d.copy_(_dev(force))
    u_d = torch.empty(ndof, dtype=torch.float64, device="cuda")
    c, it, res = to.analyze(_dev(rho), f_d, _dev(fixed), u_d)
    u_o, c_o, K = to2d.fea(rho.astype(np.float64), force, fixed.astype(bool))
    free = fixed == 0
    u = u_d.cpu().numpy()
    assert res <= 1e-11 and it > 0
    r = (K @ u - force)[free]
    drift = it * np.finfo(np.float64).eps * abs(K).sum(0).max() * np.linalg.norm(u)
    assert np.linalg.norm(r) <= 1.1e-11 * np.linalg.norm(force[free]) + drift
    scale = max(np.abs(u_o).max(), 1e-300)
    assert np.abs(u - u_o).max() <= 1e-6 * scale and np.all(u[~free] == 0)
    assert abs(c - c_o) <= 1e-7 * max(abs(c_o), 1e-300)
    to.close()


def test_iteration_cap_is_reported_with_the_last_iterate():
    binding = _need()
    from paper_2002_07627_gb300 import synth
    force, fixed, _ = synth.cantilever2d(48, 24)
    rho = torch.full((24, 48), 0.5, device="cuda")
    to = binding.To2d(48, 24, cg_max_iter=2)
    u = torch.zeros(force.shape, dtype=torch.float64, device="cuda")
    with pytest.raises(binding.ImfError) as e:
        to.analyze(rho, _dev(force), _dev(fixed), u)
    assert e.value.status == 4 and float(u.abs().max()) > 0
    to.close()


@pytest.mark.parametrize("nx,ny,eta", [(1, 1, 0.5), (7, 3, 0.5), (64, 40, 0.3), (256, 128, 0.5), (40, 20, 5.0)])
@pytest.mark.parametrize("passive", [False, True])
def test_update_on_the_device_matches_the_oracle(nx, ny, eta, passive):
    """xi_new to FP32 storage (1e-6 also covers the last step of the bisection, 1e-9 in the multiplier);
    eta = 5 takes the host's bisection."""
    binding = _need()
    from oracle import to2d
    rng = np.random.default_rng(nx + 7 * ny)
    xi = rng.uniform(0.0, 1.0, (ny, nx)).astype(np.float32)
    S = np.exp(rng.standard_normal((ny, nx))).astype(np.float32)
    S[rng.uniform(size=S.shape) < 0.1] = 0.0
    pas = None
    if passive and nx > 1:
        pas = np.zeros((ny, nx), np.uint8)
        pas[:, 0] = 1
        xi[:, 0] = 1.0
    to = binding.To2d(nx, ny)
    out = torch.empty((ny, nx), device="cuda")
    change, vol = to.update(_dev(xi), _dev(S), None if pas is None else _dev(pas), 0.5, out, move=0.2, eta=eta)
    x_o, _, vol_o = to2d.oc_update(xi, S, 0.5, 2.0, pas, 0.2, eta)
    free = np.ones(xi.shape, bool) if pas is None else pas == 0
    assert np.abs(out.cpu().numpy() - x_o).max() <= 1e-6
    assert abs(vol - vol_o) <= 1e-7 and abs(change - np.abs(x_o - xi)[free].mean()) <= 1e-6
    to.close()


@pytest.mark.parametrize("shape,n_sets,max_steps", [((1, 1, 1), 1, None), ((3, 5, 33), 7, None), ((9, 40, 97), 70, None),
                                                    ((9, 40, 97), 70, 3), ((2, 2, 31), 2100, None), ((40, 60, 70), 5, 0)])
def test_greedy_plan_matches_the_oracle_on_given_sets(shape, n_sets, max_steps):
    """Steps, counts and rest on random sets (some empty, some equal, so that ties occur), with and
    without a cap, and with more sets than one pass counts: whole numbers, so equal."""
    binding = _need()
    import oracle
    rng = np.random.default_rng(n_sets)
    nz, ny, nx = shape
    sets = rng.uniform(size=(n_sets,) + shape) < rng.choice([0.0, 0.02, 0.3], n_sets)[:, None, None, None]
    sets[n_sets // 2] = sets[0]
    words = -(-nx // 32)
    padded = np.zeros((n_sets, nz, ny, words * 32), bool)
    padded[..., :nx] = sets
    packed = np.packbits(padded, axis=-1, bitorder="little").view(np.int32)
    rho = rng.uniform(0, 1, shape).astype(np.float32)
    fix = (rng.uniform(size=shape) < 0.1).astype(np.uint8)
    imf = binding.Imf(shape)
    steps, neg, left = imf.process_plan(_dev(packed), _dev(rho), _dev(fix), max_steps)
    want = oracle.process_plan(list(sets), (fix == 0) & (rho <= 0.5), max_steps)
    assert (steps, neg, left) == want
    imf.close()


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 7, 31), (1, 128, 256), (1, 129, 256), (2, 3, 5)])
@pytest.mark.parametrize("fixture", [False, True])
def test_normalisation_and_penalty_around_the_small_grid_limit(shape, fixture):
    """32768 voxels run the maximum and what follows from it in one cluster, more of them in two launches:
    f_bar and Gamma from the raw f by the FP64 formula (whole values equal, f_bar to its last FP32 bit), and
    the penalty twice in a row (its maximum starts from zero again), against NumPy."""
    binding = _need()
    from paper_2002_07627_gb300 import synth
    rng = np.random.default_rng(shape[2])
    rho = rng.uniform(0, 1, shape).astype(np.float32)
    fix = (rng.uniform(size=shape) < 0.2).astype(np.uint8) if fixture else None
    tool = synth.planar_tool(1, 2, 3, 2, n_orient=3)
    imf = binding.Imf(shape)
    imf.set_tools([tool])
    r, f = _dev(rho), None if fix is None else _dev(fix)
    raw = torch.empty_like(r)
    fbar, sec = imf.compute(r, f, raw=raw)
    imf.sync()
    g = raw.cpu().numpy().astype(np.float64)
    omega = np.ones(shape, bool) if fix is None else fix == 0
    M = g[omega].max() if omega.any() else 0.0
    fb = np.where(omega, g * (1.0 / M) if M > 0 else 0.0, 0.0)
    B = fb > 0.01
    want = (fb * B).astype(np.float32)
    assert np.abs(fbar.cpu().numpy() - want).max() <= np.spacing(np.float32(1.0))
    assert np.array_equal(sec.cpu().numpy(), (omega & (rho <= 0.5) & B).astype(np.uint8))
    for scale in (3.0, 0.25):
        s0 = (rng.standard_normal(shape) * scale).astype(np.float32)
        out = imf.penalize(_dev(s0), r, fbar, sec, f, w_acc=0.3).cpu().numpy().astype(np.float64)
        m = np.abs(s0[omega]).max() if omega.any() else 0.0
        s_imf = np.where(rho > 0.5, want, np.where(omega & (rho <= 0.5) & B, 1.0, 0.0))
        ref = 0.7 * (s0 / m if m > 0 else s0) + 0.3 * s_imf
        assert np.abs(out - ref).max() <= 4e-7 * max(1.0, np.abs(ref).max())
    imf.close()


@pytest.mark.parametrize("shape,n_sets,max_steps", [((1, 1, 8192), 9, None), ((1, 3, 8192), 8, None), ((4, 33, 70), 1025, 40),
                                                    ((1, 16, 16), 5000, 12), ((30, 70, 4000), 3, None)])
def test_greedy_plan_splits_words_and_sets_over_the_blocks(shape, n_sets, max_steps):
    """One chunk of words and just over, parts of the sets that do not divide evenly, more sets than blocks and more
    chunks than blocks: whole numbers, so equal to the oracle's."""
    binding = _need()
    import oracle
    rng = np.random.default_rng(n_sets)
    nz, ny, nx = shape
    words = -(-nx // 32)
    packed = rng.integers(0, 2**32, (n_sets, nz, ny, words), np.uint32)
    for _ in range(3):
        packed &= rng.integers(0, 2**32, packed.shape, np.uint32)
    packed[n_sets // 3] = packed[n_sets - 1]
    sets = [np.unpackbits(p.view(np.uint8), axis=-1, bitorder="little")[..., :nx].astype(bool) for p in packed]
    rho = rng.uniform(0, 1, shape).astype(np.float32)
    imf = binding.Imf(shape)
    got = imf.process_plan(_dev(packed.view(np.int32)), _dev(rho), None, max_steps)
    assert got == oracle.process_plan(sets, rho <= 0.5, max_steps)
    imf.close()


@pytest.mark.parametrize("nx,ny,Emin,most", [(256, 128, 1e-9, 1500), (128, 64, 1e-9, 800), (4, 3, 1e-6, 80)])
def test_slow_and_stalled_multigrid(nx, ny, Emin, most):
    """Checkerboards of 2 x 2 cells at high contrast: the multigrid iteration goes on while its residual falls (the
    plain one takes 3700 and 1900 iterations on the larger two), and where its preconditioner is no inverse (the
    smallest) the plain iteration takes over; compliance as the direct solve has it, to what the condition leaves."""
    binding = _need()
    from oracle import to2d
    from paper_2002_07627_gb300 import synth
    force, fixed, _ = synth.cantilever2d(nx, ny)
    rho = (np.add.outer(np.arange(ny) // 2, np.arange(nx) // 2) % 2).astype(np.float32)
    to = binding.To2d(nx, ny, Emin=Emin)
    c, it, res = to.analyze(_dev(rho), _dev(force), _dev(fixed))
    u, c_o, K = to2d.fea(rho.astype(np.float64), force, fixed.astype(bool), Emin=Emin)
    assert it <= most and res <= 1e-8
    assert abs(c - c_o) <= 1e-5 * abs(c_o)
    to.close()
