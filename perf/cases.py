"""Timed cases of the IMF library: what its users run, through the public entry points.

Every case is a call (or the few calls of one step) that a topology-optimisation loop, a batched
run, a served design or a process planner makes on a design whose tools are already set:
`prepare` builds the design on the GPU and keeps the handle with its tool spectra and its output
arrays, `run` is one pass. Kinds:

  step2d    imf_compute + imf_penalize_sensitivity on a small planar grid, a coarse 2D loop
  loop2d    the constraint side of an iteration of the 2D loop: imf_compute with two tools,
            imf_penalize_sensitivity, imf_to2d_update
  fea2d     the mechanics side of that iteration: imf_to2d_project, _analyze, _sensitivity
  graph     a design replayed as a captured graph, as the batched form runs it
  field     imf_compute on a 3D design: f_bar and Gamma, and f and A where asked
  plan      per-orientation accessible sets and the greedy process plan on a finished design
  direct    imf_compute through the BF16 hi/lo tensor-core collision path (small tools)
  host      imf_compute_host: design and results in host memory

`exact` computes the same outputs in 64 bits with numpy and torch alone.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2002_07627_gb300 import binding

LAM, TAU, THETA_REL = 0.01, 0.5, 0.01
VOLFRAC, MOVE, ETA, BETA, W_ACC = 0.5, 0.2, 0.5, 2.0, 0.5


def listed():
    return [
        # the smallest real call: the 64 x 64 planar design of the 2D studies, 8 directions
        {"name": "step2d_64", "kind": "step2d", "nx": 64, "ny": 64, "n_orient": 8},
        # one iteration's constraint side on the 256 x 128 cantilever, a thin and a thick cutter
        {"name": "loop2d_256x128", "kind": "loop2d", "nx": 256, "ny": 128, "n_orient": 8},
        # its mechanics side: projection, finite elements to 1e-8, filtered sensitivity
        {"name": "fea2d_256x128", "kind": "fea2d", "nx": 256, "ny": 128},
        # a coarse 3D loop of the batched / served mixes, as a graph replay
        {"name": "graph_48", "kind": "graph", "nx": 48, "ny": 48, "nz": 48, "n_orient": 24, "r_cut": 2},
        # an odd-sized part with every output asked for
        {"name": "field_75x61x50", "kind": "field", "nx": 75, "ny": 61, "nz": 50, "n_orient": 24, "r_cut": 3,
         "every": True, "sweep": False, "sharp": "all", "sharp_k": 1},
        # the usual 3D design of a loop: f_bar and Gamma only
        {"name": "field_128", "kind": "field", "nx": 128, "ny": 128, "nz": 128, "n_orient": 64, "r_cut": 3,
         "every": False, "sweep": False, "sharp": "all", "sharp_k": 1},
        # a thick cutter (the upper end of the batched mix), many sharp points
        {"name": "field_144_thick", "kind": "field", "nx": 144, "ny": 144, "nz": 144, "n_orient": 96, "r_cut": 6,
         "every": False, "sweep": False, "sharp": "all", "sharp_k": 1},
        # sampled sharp points: the conservative field, with the accessible set by the sweep
        {"name": "field_128_sampled", "kind": "field", "nx": 128, "ny": 128, "nz": 128, "n_orient": 64, "r_cut": 3,
         "every": True, "sweep": False, "sharp": "nearest", "sharp_k": 16},
        # the finished design's process plan
        {"name": "plan_128", "kind": "plan", "nx": 128, "ny": 128, "nz": 128, "n_orient": 64, "r_cut": 3},
        # the largest design: 256^3, 128 directions, every output, the accessible set by the sweep
        {"name": "field_256", "kind": "field", "nx": 256, "ny": 256, "nz": 256, "n_orient": 128, "r_cut": 3,
         "every": True, "sweep": True, "sharp": "all", "sharp_k": 1},
        # a small tool on the tensor-core collision path
        {"name": "direct_64", "kind": "direct", "nx": 64, "ny": 64, "nz": 64, "n_orient": 32},
        # a caller with host arrays
        {"name": "host_96", "kind": "host", "nx": 96, "ny": 96, "nz": 96, "n_orient": 32, "r_cut": 3},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step2d", "loop2d", "fea2d", "graph", "field", "field", "field", "field", "plan", "direct", "host"])
    if kind == "step2d":
        return {"kind": kind, "nx": size(40, 200), "ny": size(40, 200), "n_orient": rng.randint(4, 16)}
    if kind == "loop2d":
        nx = size(64, 256)
        return {"kind": kind, "nx": nx, "ny": max(48, nx // 2 + rng.randint(-3, 3)), "n_orient": rng.randint(4, 12)}
    if kind == "fea2d":
        nx = size(48, 256)
        return {"kind": kind, "nx": nx, "ny": max(24, nx // 2 + rng.randint(-3, 3))}
    if kind == "graph":
        n = size(40, 80)
        return {"kind": kind, "nx": n, "ny": n, "nz": n, "n_orient": rng.randint(16, 48), "r_cut": rng.randint(2, 4)}
    if kind == "field":
        sharp = rng.choice(["all", "all", "all", "boundary", "nearest"])
        c = {"kind": kind, "every": rng.random() < 0.5, "sweep": rng.random() < 0.25, "sharp": sharp,
             "sharp_k": rng.choice([4, 16, 64])}
        form = rng.random()
        if form < 0.45:      # parts of unequal extents
            c.update(nx=size(30, 150), ny=size(30, 150), nz=size(30, 110), n_orient=rng.randint(8, 64),
                     r_cut=rng.randint(2, 5))
        elif form < 0.85:    # cubes of the batched mix
            n = size(64, 176)
            c.update(nx=n, ny=n, nz=n, n_orient=rng.randint(16, 96), r_cut=rng.randint(2, 6 if n < 150 else 4))
        else:
            n = size(180, 250)
            c.update(nx=n, ny=n, nz=n, n_orient=rng.randint(48, 112), r_cut=3)
        return c
    if kind == "plan":
        n = size(48, 140)
        return {"kind": kind, "nx": n, "ny": n, "nz": max(32, n - rng.randint(0, 20)), "n_orient": rng.randint(12, 64),
                "r_cut": rng.randint(2, 4)}
    if kind == "direct":
        n = size(32, 72)
        return {"kind": kind, "nx": n, "ny": n, "nz": n, "n_orient": rng.randint(8, 48)}
    n = size(40, 128)
    return {"kind": "host", "nx": n, "ny": n, "nz": n, "n_orient": rng.randint(12, 48), "r_cut": rng.randint(2, 4)}


# ------------------------------------------------------------------------------------- inputs

def _gauss(a, sigma, axes):
    """Separable Gaussian blur with a reflecting boundary, in a's own type."""
    r = int(4 * sigma + 0.5)
    w = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-r, r + 1)]
    s = sum(w)
    for ax in axes:
        n = a.shape[ax]
        idx = torch.arange(-r, n + r, device=a.device) % (2 * n)
        idx = torch.where(idx >= n, 2 * n - 1 - idx, idx)
        p = a.index_select(ax, idx)
        out = torch.zeros_like(a)
        for i in range(2 * r + 1):
            out += (w[i] / s) * p.narrow(ax, i, n)
        a = out
    return a


def _planar_density(nx, ny, rng, dev):
    """Smooth noise through a logistic: densities of a planar design midway in its loop."""
    a = torch.from_numpy(rng.random((1, ny, nx))).to(dev)
    a = _gauss(a, 3.0, (1, 2))
    a = (a - a.mean()) / (a.std() + 1e-30)
    return torch.sigmoid(4.0 * a).to(torch.float32).contiguous()


def _beam_density(nx, ny, nz, rng, dev):
    """Union of capsules (radius 2-5 voxels) softened by one voxel: a lattice-like 3D part whose
    beams grow in number with the cross-section (40 at 128^3, 160 at 256^3)."""
    n_beams = max(4, int(40 * (nx * ny * nz) ** (2.0 / 3.0) / 128.0 ** 2))
    ind = torch.zeros((nz, ny, nx), dtype=torch.float32, device=dev)
    hi = np.array([nx - 1, ny - 1, nz - 1], np.float64)
    for _ in range(n_beams):
        p0, p1 = rng.random(3) * hi, rng.random(3) * hi
        r = rng.uniform(2.0, 5.0)
        lo_b = np.maximum(np.floor(np.minimum(p0, p1) - r - 1), 0).astype(int)
        hi_b = np.minimum(np.ceil(np.maximum(p0, p1) + r + 1), hi).astype(int)
        ax = [torch.arange(int(lo_b[c]), int(hi_b[c]) + 1, dtype=torch.float32, device=dev) for c in range(3)]
        dx, dy, dz = ax[0][None, None, :] - p0[0], ax[1][None, :, None] - p0[1], ax[2][:, None, None] - p0[2]
        d = p1 - p0
        dd = max(float(d @ d), 1e-12)
        s = ((dx * d[0] + dy * d[1] + dz * d[2]) / dd).clamp_(0.0, 1.0)
        q = (dx - s * d[0]) ** 2 + (dy - s * d[1]) ** 2 + (dz - s * d[2]) ** 2
        sub = ind[lo_b[2]:hi_b[2] + 1, lo_b[1]:hi_b[1] + 1, lo_b[0]:hi_b[0] + 1]
        sub[q <= r * r] = 1.0
    return _gauss(ind, 1.0, (0, 1, 2)).clamp_(0.0, 1.0).contiguous()


def _planar_tool(cut_w, cut_h, hold_w, hold_h, n_orient):
    """A cut_w x cut_h cutter with the origin at its tip and a holder above it; the directions
    spread over half a turn."""
    tx, ty = max(cut_w, hold_w), cut_h + hold_h
    holder, cutter = np.zeros((1, ty, tx), np.uint8), np.zeros((1, ty, tx), np.uint8)
    c0, h0 = (tx - cut_w) // 2, (tx - hold_w) // 2
    cutter[0, :cut_h, c0:c0 + cut_w] = 1
    holder[0, cut_h:, h0:h0 + hold_w] = 1
    ang = [k * math.pi / (n_orient - 1) for k in range(n_orient)]
    quats = np.array([[math.cos(a / 2), 0.0, 0.0, math.sin(a / 2)] for a in ang])
    return holder, cutter, (c0 + cut_w // 2, 0, 0), quats


def _cylinder_tool(r_cut, l_cut, r_hold, l_hold, n_orient):
    """A cutter cylinder with its tip at the origin and a wider holder on it; directions on a
    Fibonacci hemisphere, each the shortest turn from +z."""
    rr = max(r_cut, r_hold)
    k, j, i = np.meshgrid(np.arange(l_cut + l_hold), np.arange(2 * rr + 1), np.arange(2 * rr + 1), indexing="ij")
    d2 = (i - rr) ** 2 + (j - rr) ** 2
    cutter = ((k < l_cut) & (d2 <= r_cut * r_cut)).astype(np.uint8)
    holder = ((k >= l_cut) & (d2 <= r_hold * r_hold)).astype(np.uint8)
    quats = []
    for n in range(n_orient):
        half, phi = math.acos(1.0 - (n + 0.5) / n_orient) / 2, n * math.pi * (3.0 - math.sqrt(5.0))
        quats.append([math.cos(half), -math.sin(phi) * math.sin(half), math.cos(phi) * math.sin(half), 0.0])
    return holder, cutter, (rr, rr, 0), np.array(quats)


def _tools(case):
    k, n = case["kind"], case["n_orient"]
    if k == "step2d":
        return [_planar_tool(3, 12, 9, 10, n)]
    if k == "loop2d":
        return [_planar_tool(1, 12, 7, 10, n), _planar_tool(3, 12, 9, 10, n)]
    if k == "direct":
        return [_cylinder_tool(2, 6, 4, 6, n)]
    r = case["r_cut"]
    return [_cylinder_tool(r, 20, 8 if r == 3 else int(round(2.5 * r)), 16, n)]


def _cantilever(nx, ny):
    """Left edge clamped, a unit load down at the middle of the right edge; the two leftmost
    element columns are the clamping fixture."""
    ndof = 2 * (nx + 1) * (ny + 1)
    force, fixed = np.zeros(ndof), np.zeros(ndof, np.uint8)
    force[2 * ((ny // 2) * (nx + 1) + nx) + 1] = -1.0
    left = np.arange(ny + 1) * (nx + 1)
    fixed[2 * left] = fixed[2 * left + 1] = 1
    return force, fixed


def _design(case, seed, dev):
    """Density and fixture of a case's design, on `dev`: the same values for every reader."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case.get("nz", 1)
    if nz == 1:
        rho = _planar_density(nx, ny, rng, dev)
        fix = torch.zeros(rho.shape, dtype=torch.uint8, device=dev)
        if case["kind"] == "step2d":
            fix[:, :4] = 1
        else:
            fix[:, :, :2] = 1
            rho[fix != 0] = 1.0
    else:
        rho = _beam_density(nx, ny, nz, rng, dev)
        fix = torch.zeros(rho.shape, dtype=torch.uint8, device=dev)
        fix[:max(2, nz // 24)] = 1
    return rho, fix, rng


def _sens(shape, rng, dev):
    """A positive, widely spread sensitivity field, as compliance gives."""
    return torch.from_numpy(np.exp(rng.standard_normal(shape)).astype(np.float32)).to(dev)


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    rho, fix, rng = _design(case, seed, dev)
    s = {"kind": kind, "rho": rho, "fix": fix}
    if kind in ("loop2d", "fea2d"):
        nx, ny = case["nx"], case["ny"]
        s["to"] = binding.To2d(nx, ny)
        s["xi"] = rho[0].clone()
        if kind == "fea2d":
            force, fixed = _cantilever(nx, ny)
            s.update(force=torch.from_numpy(force).to(dev), fixed=torch.from_numpy(fixed).to(dev),
                     rho=torch.empty_like(s["xi"]), sens=torch.empty_like(s["xi"]))
            return s
        s["xi_new"] = torch.empty_like(s["xi"])
    if kind == "field":
        opt = {"accessible_by_sweep": case["sweep"], "sharp_k": case["sharp_k"],
               "sharp_sampling": {"all": binding.IMF_SHARP_ALL, "boundary": binding.IMF_SHARP_BOUNDARY,
                                  "nearest": binding.IMF_SHARP_NEAREST}[case["sharp"]]}
    else:
        opt = {"precision": binding.IMF_BF16_DIRECT} if kind == "direct" else {}
    imf = binding.Imf(tuple(rho.shape), lam=LAM, tau=TAU, theta_rel=THETA_REL, **opt)
    imf.set_tools([SimpleNamespace(holder=h, cutter=c, origin=o, quats=q) for h, c, o, q in _tools(case)])
    s["imf"] = imf
    if kind == "host":
        s.update(rho=rho.cpu().numpy(), fix=fix.cpu().numpy())
        return s
    s.update(fbar=torch.empty_like(rho), sec=torch.empty_like(fix), raw=None, acc=None)
    if kind == "field" and case["every"]:
        s.update(raw=torch.empty_like(rho), acc=torch.empty_like(fix))
    if kind in ("step2d", "loop2d"):
        s.update(s_phi=_sens(tuple(rho.shape), rng, dev), sens=torch.empty_like(rho))
    if kind == "graph":
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        imf.capture_graph(rho, fix, s["fbar"], s["sec"], stream=stream)
        torch.cuda.current_stream().wait_stream(stream)
    return s


def run(s):
    kind = s["kind"]
    if kind == "fea2d":
        to = s["to"]
        to.project(s["xi"], s["rho"])
        c, _, _ = to.analyze(s["rho"], s["force"], s["fixed"])
        to.sensitivity(s["xi"], s["rho"], s["sens"])
        return {"rho": s["rho"], "compliance": c, "sens": s["sens"]}
    imf = s["imf"]
    if kind == "host":
        fbar, sec, raw, acc = imf.compute_host(s["rho"], s["fix"])
        return {"fbar": fbar, "secluded": sec, "raw": raw, "accessible": acc}
    if kind == "graph":
        imf.launch_graph()
        return {"fbar": s["fbar"], "secluded": s["sec"]}
    if kind == "plan":
        sets, fbar, sec = imf.accessible_sets(s["rho"], s["fix"])
        steps, negative, left = imf.process_plan(sets, s["rho"], s["fix"])
        plan = np.full((len(sets), 2), -1, np.int64)       # (set, voxels removed) per step, then -1
        plan[:len(steps)] = np.array(steps, np.int64).reshape(-1, 2)
        return {"fbar": fbar, "secluded": sec, "sets": sets, "plan": plan, "negative": negative, "left": left}
    imf.compute(s["rho"], s["fix"], s["fbar"], s["sec"], s["raw"], s["acc"])
    out = {"fbar": s["fbar"], "secluded": s["sec"]}
    if s["raw"] is not None:
        out.update(raw=s["raw"], accessible=s["acc"])
    if kind in ("step2d", "loop2d"):
        s["sens"].copy_(s["s_phi"])
        out["sens"] = imf.penalize(s["sens"], s["rho"], s["fbar"], s["sec"], s["fix"], w_acc=W_ACC)
    if kind == "loop2d":
        change, vol = s["to"].update(s["xi"], s["sens"][0], s["fix"][0], VOLFRAC, s["xi_new"], move=MOVE, eta=ETA)
        out.update(xi=s["xi_new"], change=change, vol=vol)
    return out


# --------------------------------------------------------------------------------------- work

def work(case):
    nx, ny, nz = case["nx"], case["ny"], case.get("nz", 1)
    n = nx * ny * nz
    if case["kind"] == "fea2d":
        # a local operator carries the load one node a step, so at least two sweeps of the longer
        # side: per step the element operator and the vector updates, about 320 flops an element
        return {"bytes": 4.0 * n * 3, "flops": 2.0 * max(nx, ny) * 320.0 * n}
    flops, bytes_ = 0.0, n * (4 + 1 + 4 + 1.0)
    for holder, cutter, _, quats in _tools(case):
        m, reach = len(quats), max(cutter.shape)
        points = float((nx + reach) * (ny + reach) * (nz + reach if nz > 1 else 1))
        sharp = int(cutter.sum())
        if case.get("sharp") == "nearest":
            sharp = min(sharp, case["sharp_k"])
        # a correlation per direction (one real transform of the padded grid) and one comparison
        # per cell, direction and sharp point
        flops += m * (2.5 * points * math.log2(points) + float(n) * sharp)
    if case.get("every") or case["kind"] == "host":
        bytes_ += n * 5.0
    if case["kind"] in ("step2d", "loop2d"):
        bytes_ += n * 8.0
    if case["kind"] == "plan":
        bytes_ += case["n_orient"] * n / 8.0
    return {"bytes": bytes_, "flops": flops}


# -------------------------------------------------------------------------------------- exact

def _rotation(q):
    w, x, y, z = np.asarray(q, np.float64) / math.sqrt(((q[0] * q[0] + q[1] * q[1]) + q[2] * q[2]) + q[3] * q[3])
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _resample(mask, origin, R):
    """Integer offsets v (x, y, z) with mask at origin + floor(R^T v + 1/2)."""
    tz, ty, tx = mask.shape
    o = np.array(origin)
    ext = np.array([tx, ty, tz])
    corners = np.array([[(-o[c] - 0.5, ext[c] - o[c] - 0.5)[(i >> c) & 1] for c in range(3)] for i in range(8)]) @ R.T
    lo, hi = np.floor(corners.min(0)).astype(int) - 1, np.ceil(corners.max(0)).astype(int) + 1
    z, y, x = np.meshgrid(*[np.arange(lo[c], hi[c] + 1) for c in (2, 1, 0)], indexing="ij")
    v = np.stack([x.ravel(), y.ravel(), z.ravel()], -1)
    vf = v.astype(np.float64)
    u = np.stack([np.floor(((R[0, c] * vf[:, 0] + R[1, c] * vf[:, 1]) + R[2, c] * vf[:, 2]) + 0.5) for c in range(3)],
                 -1).astype(int) + o
    ok = np.all((u >= 0) & (u < ext), 1)
    u = np.where(ok[:, None], u, 0)
    return v[ok & (mask[u[:, 2], u[:, 1], u[:, 0]] != 0)]


def _sharp_mask(cutter, origin, case):
    mode = case.get("sharp", "all")
    if mode == "all":
        return cutter
    p = np.pad(cutter, 1)
    inner = p[1:-1, 1:-1, 2:] & p[1:-1, 1:-1, :-2] & p[1:-1, 2:, 1:-1] & p[1:-1, :-2, 1:-1] & p[2:, 1:-1, 1:-1] & p[:-2, 1:-1, 1:-1]
    edge = ((cutter != 0) & (inner == 0)).astype(np.uint8)
    if mode == "boundary":
        return edge
    at = np.argwhere(edge)                                 # C order: ties keep the linear index
    d2 = ((at[:, ::-1] - np.array(origin)) ** 2).sum(1)
    at = at[np.argsort(d2, kind="stable")[:case["sharp_k"]]]
    out = np.zeros_like(cutter)
    out[at[:, 0], at[:, 1], at[:, 2]] = 1
    return out


def _exact_field(case, rho, fix):
    """f in 64 bits: correlations by the DFT, minimum over the sharp points row by row."""
    dev = rho.device
    nz, ny, nx = rho.shape
    obst = torch.clamp(rho.double() + (fix != 0).double(), max=1.0)
    f = torch.full(rho.shape, math.inf, dtype=torch.float64, device=dev)
    for holder, cutter, origin, quats in _tools(case):
        whole = ((holder != 0) | (cutter != 0)).astype(np.uint8)
        sharp = _sharp_mask(cutter, origin, case)
        sets = []
        for q in quats:
            R = _rotation(q)
            sets.append((_resample(whole, origin, R), _resample(sharp, origin, R)))
        tv = np.concatenate([t for t, _ in sets])
        kv = np.concatenate([k for _, k in sets])
        tlo, thi, klo, khi = tv.min(0), tv.max(0), kv.min(0), kv.max(0)
        n = np.array([nx, ny, nz])
        P = [int(v) for v in np.maximum(n + np.maximum(khi - tlo, thi - klo) + 1, n + khi - klo + 1)]
        rest = lambda m: m if all(m % p for p in (2, 3, 5, 7)) else rest(next(m // p for p in (2, 3, 5, 7) if m % p == 0))
        P = [next(m for m in range(p, 2 * p + 2) if rest(m) == 1) for p in P]
        px, py, pz = P
        spec = torch.fft.rfftn(obst, s=(pz, py, px))
        for T, K in sets:
            if not len(K):
                continue
            ind = torch.zeros((pz, py, px), dtype=torch.float64, device=dev)
            t = torch.from_numpy(T).to(dev)
            ind[t[:, 2] % pz, t[:, 1] % py, t[:, 0] % px] = 1.0
            g = torch.fft.irfftn(spec * torch.fft.rfftn(ind).conj(), s=(pz, py, px))
            # window of the translations x - k, from -khi
            g = torch.roll(g, shifts=(int(khi[2]), int(khi[1]), int(khi[0])), dims=(0, 1, 2))
            win = [int(n[c] + khi[c] - klo[c]) for c in range(3)]
            g = g[:win[2], :win[1], :win[0]].clamp_(min=0.0).contiguous()
            # runs along x, by length, on sliding minima of that length
            runs = {}
            order = np.lexsort((K[:, 0], K[:, 1], K[:, 2]))
            a = None
            for x, y, z in K[order].tolist() + [[1 << 30, 0, 0]]:
                if a is not None and (y, z) == (a[1], a[2]) and x == a[0] + a[3]:
                    a[3] += 1
                    continue
                if a is not None:
                    runs.setdefault(a[3], []).append(a)
                a = [x, y, z, 1]
            m = g
            for L in range(1, max(runs) + 1):
                if L > 1:
                    m = torch.minimum(m[..., :-1], g[..., L - 1:])
                for x, y, z, _ in runs.get(L, ()):
                    sz, sy, sx = int(khi[2]) - z, int(khi[1]) - y, int(khi[0]) - (x + L - 1)
                    torch.minimum(f, m[sz:sz + nz, sy:sy + ny, sx:sx + nx], out=f)
    omega = fix == 0
    M = float(f[omega].max())
    fbar = torch.where(omega, f / M if M > 0 else torch.zeros_like(f), torch.zeros_like(f))
    B = fbar > LAM
    return f, fbar * B, omega & (rho.double() <= TAU) & B


def _element_matrix(nu):
    D = np.array([[1.0, nu, 0.0], [nu, 1.0, 0.0], [0.0, 0.0, (1.0 - nu) / 2.0]]) / (1.0 - nu * nu)
    at = [(0, 0), (1, 0), (1, 1), (0, 1)]
    k = np.zeros((8, 8))
    g = 0.5 / math.sqrt(3.0)
    for s in (0.5 - g, 0.5 + g):
        for t in (0.5 - g, 0.5 + g):
            B = np.zeros((3, 8))
            for i, (x, y) in enumerate(at):
                gx, gy = (1.0 if x else -1.0) * (t if y else 1 - t), (1.0 if y else -1.0) * (s if x else 1 - s)
                B[0, 2 * i], B[1, 2 * i + 1], B[2, 2 * i], B[2, 2 * i + 1] = gx, gy, gy, gx
            k += 0.25 * B.T @ D @ B
    return k


def _exact_fea(case, xi):
    nx, ny = case["nx"], case["ny"]
    dev = xi.device
    x = xi.double()
    rho64 = 1.0 - torch.exp(-BETA * x) + x * math.exp(-BETA)
    rho = rho64.float().double()            # the density the analysis reads is stored in 32 bits
    E = 1e-3 + rho ** 3 * (1.0 - 1e-3)
    k0 = torch.from_numpy(_element_matrix(0.3)).to(dev)
    force, fixed = _cantilever(nx, ny)
    free = torch.from_numpy(fixed == 0).to(dev).double().view(ny + 1, nx + 1, 2)
    b = torch.from_numpy(force).to(dev).view(ny + 1, nx + 1, 2) * free
    slots = [(0, 0), (0, 1), (1, 1), (1, 0)]

    def corners(v):
        return torch.cat([v[j:j + ny, i:i + nx] for j, i in slots], -1)

    def scatter(e):
        out = torch.zeros((ny + 1, nx + 1, 2), dtype=torch.float64, device=dev)
        for c, (j, i) in enumerate(slots):
            out[j:j + ny, i:i + nx] += e[..., 2 * c:2 * c + 2]
        return out

    apply = lambda v: scatter(E[..., None] * (corners(v) @ k0)) * free
    diag = scatter(E[..., None] * torch.diag(k0)) * free + (1.0 - free)
    u, r = torch.zeros_like(b), b.clone()
    z = r / diag
    p, rz, stop = z.clone(), (r * z).sum(), 1e-26 * float((b * b).sum())
    for it in range(12000):
        q = apply(p)
        alpha = rz / (p * q).sum()
        u += alpha * p
        r -= alpha * q
        if it % 64 == 63 and float((r * r).sum()) <= stop:
            break
        z = r / diag
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    ue = corners(u)
    ce = ((ue @ k0) * ue).sum(-1)
    s = 3.0 * rho ** 2 * (1.0 - 1e-3) * ce * (BETA * torch.exp(-BETA * x) + math.exp(-BETA))
    num, den = torch.zeros_like(s), torch.zeros_like(s)
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            w = 1.5 - math.hypot(dx, dy)
            if w <= 0:
                continue
            to = (slice(max(0, -dy), ny - max(0, dy)), slice(max(0, -dx), nx - max(0, dx)))
            of = (slice(max(0, dy), ny - max(0, -dy)), slice(max(0, dx), nx - max(0, -dx)))
            num[to] += w * (x * s)[of]
            den[to] += w
    return {"rho": rho64, "compliance": float((b * u).sum()), "sens": num / (x.clamp(min=1e-3) * den)}


def _exact_update(xi, S, fix):
    x, S, free = xi.double(), S.clamp(min=0.0), fix == 0
    lo_x, hi_x = (x - MOVE).clamp(min=0.0), (x + MOVE).clamp(max=1.0)

    def new(lam):
        return torch.where(free, torch.maximum(torch.minimum(x * (S / lam) ** ETA, hi_x), lo_x), torch.ones_like(x))

    def volume(v):
        return float((1.0 - torch.exp(-BETA * v) + v * math.exp(-BETA))[free].mean())

    lo, hi = 1e-12, 1e12
    while hi / lo > 1.0 + 1e-9:
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if volume(new(mid)) > VOLFRAC else (lo, mid)
    v = new(math.sqrt(lo * hi))
    return v, float((v - x).abs()[free].mean()), volume(v)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind = case["kind"]
    rho, fix, rng = _design(case, seed, dev)
    if kind == "fea2d":
        return _exact_fea(case, rho[0])
    f, fbar, sec = _exact_field(case, rho, fix)
    out = {"fbar": fbar, "secluded": None}
    if kind == "plan":
        out.update(sets=None, plan=None, negative=None, left=None)
    if kind == "host" or (kind == "field" and case["every"]):
        out.update(raw=f, accessible=None)
    if kind in ("step2d", "loop2d"):
        s = _sens(tuple(rho.shape), rng, dev).double()
        s_imf = torch.where(rho.double() > TAU, fbar, sec.double())
        out["sens"] = (1.0 - W_ACC) * s / float(s[fix == 0].abs().max()) + W_ACC * s_imf
    if kind == "loop2d":
        xi, change, vol = _exact_update(rho[0], out["sens"][0], fix[0])
        out.update(xi=xi, change=change, vol=vol)
    return out
