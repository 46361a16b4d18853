"""What the performance of this framework is measured on: the calls its users
make, from one energy gradient of a small cube to a field step of a
polycrystal with three million potential unknowns, and the warm-start network
next to them.

A case names a path ("kind") and its sizes.  Meshes depend on the case alone
and their uploaded handles are kept, as a program that sweeps fields or states
on one magnet keeps them; the magnetisation, the applied field, the network's
weights and its data come from the seed.
"""
import math

import numpy as np
import torch

from paper_1801_03690_gb300 import Batch, MLP, Magnet, Params

MU0 = 4e-7 * math.pi
NM = 1e-9
PERMALLOY = (8.0e5, 1.3e-11, 0.0)          # Ms (A/m), A (J/m), K1 (J/m^3)
ND2FE14B = (1.28e6, 7.7e-12, 4.3e6)
WIDTHS = (16, 128, 128, 128, 4)            # the warm-start network
LR = 2e-3                                  # learning rate of the training loop
TRAINED = 4                                # training steps before the measured one


def listed():
    return [
        # A field step of the 40 nm permalloy cube of 16^3 voxels (29,791
        # unknowns) with the default parameters: barriers and launches.
        {"name": "step_soft16_fp64", "kind": "step", "mesh": "soft", "n": 16, "form": "fp64", "iters": 4},
        # The same call on an 80 nm Nd2Fe14B cube with jittered nodes, 32
        # voxels per edge (250,047 unknowns), plain FP64: the paper's method.
        {"name": "step_hard32_fp64", "kind": "step", "mesh": "hard", "n": 32, "form": "fp64", "iters": 2},
        # The hard cube at its full resolution (857,375 unknowns) in the
        # precision form with the multigrid preconditioner.
        {"name": "step_hard48_multigrid", "kind": "step", "mesh": "hard", "n": 48, "form": "multigrid", "iters": 3},
        # A polycrystal of 37 grains in a graded air box, 100 voxels per edge
        # (3.2 million unknowns): the form and mesh family of the benchmark.
        {"name": "step_grains100_multigrid", "kind": "step", "mesh": "grains", "n": 100, "form": "multigrid",
         "iters": 3},
        # Twelve platelets of 100 to 240 nm in one launch: a parameter study.
        {"name": "batch_platelets12", "kind": "batch", "members": 12, "longest": 240.0, "form": "multigrid",
         "iters": 3},
        # One gradient through host arrays on a small cube: what an outer
        # optimiser or a coupling to other code calls.
        {"name": "gradient_soft10_fp64", "kind": "gradient", "mesh": "soft", "n": 10, "form": "fp64"},
        # The same on a graded polycrystal, precision form.
        {"name": "gradient_grains48_multigrid", "kind": "gradient", "mesh": "grains", "n": 48, "form": "multigrid"},
        # The four linear operators of the energy on host arrays: post-processing.
        {"name": "operators_hard40", "kind": "operators", "mesh": "hard", "n": 40},
        # The network on the nodes of a small magnet ...
        {"name": "mlp_forward_20011", "kind": "forward", "rows": 20011},
        # ... and on those of the largest benchmarked polycrystal.
        {"name": "mlp_forward_3375000", "kind": "forward", "rows": 3375000},
        # One Adam step of its training on the default mini-batch.
        {"name": "mlp_train_16384", "kind": "train", "rows": 16384},
        # Input standardisation and target scales of a training set.
        {"name": "mlp_fit_1200003", "kind": "fit", "rows": 1200003},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "gradient", "operators", "forward", "train", "fit"])
    if kind == "step":
        form = rng.choice(["fp64", "fp32", "multigrid", "multigrid"])
        mesh = rng.choice(["soft", "hard", "grains"])
        return {"kind": kind, "mesh": mesh, "n": _log(rng, 8, 28 if form == "fp64" else 44), "form": form,
                "iters": rng.randint(1, 4)}
    if kind == "batch":
        return {"kind": kind, "members": rng.randint(2, 14), "longest": round(rng.uniform(130.0, 260.0), 1),
                "form": rng.choice(["fp64", "fp32", "multigrid"]), "iters": rng.randint(1, 3)}
    if kind == "gradient":
        return {"kind": kind, "mesh": rng.choice(["soft", "hard", "grains"]), "n": _log(rng, 5, 44),
                "form": rng.choice(["fp64", "fp32", "multigrid"])}
    if kind == "operators":
        return {"kind": kind, "mesh": rng.choice(["soft", "hard", "grains"]), "n": _log(rng, 5, 44)}
    lo, hi = {"forward": (1, 3400000), "train": (64, 65536), "fit": (1000, 3000000)}[kind]
    return {"kind": kind, "rows": _log(rng, lo, hi)}


# ------------------------------------------------------------------- meshes

def _lattice(xs, ys, zs):
    """Nodes of the lattice xs x ys x zs, six positively oriented tetrahedra
    per voxel (one for each order of the axes) and every tetrahedron's voxel."""
    nx, ny, nz = len(xs), len(ys), len(zs)
    z, y, x = np.meshgrid(zs, ys, xs, indexing="ij")
    xyz = np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1)
    k, j, i = np.meshgrid(np.arange(nz - 1), np.arange(ny - 1), np.arange(nx - 1), indexing="ij")
    i, j, k = (v.ravel().astype(np.int32) for v in (i, j, k))
    base = i + nx * (j + ny * k)
    step = (1, nx, nx * ny)
    tets = np.empty((base.size, 6, 4), dtype=np.int32)
    for t, (a, b, c) in enumerate(((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))):
        even = (a, b, c) in ((0, 1, 2), (1, 2, 0), (2, 0, 1))
        mid = (step[a], step[a] + step[b]) if even else (step[a] + step[b], step[a])
        tets[:, t] = base[:, None] + np.array([0, mid[0], mid[1], sum(step)], dtype=np.int32)
    return xyz, tets.reshape(-1, 4), (i, j, k)


def _graded(half, h, box, ratio):
    """Spacing h over [-half, half], then cells that grow by `ratio`."""
    out, x, step = [], half, h
    while x < box - 1e-15:
        step *= ratio
        x = min(x + step, box)
        out.append(x)
    out = np.array(out)
    return np.concatenate([-out[::-1], np.linspace(-half, half, int(round(2 * half / h)) + 1), out])


def _cube_mesh(kind, n):
    """(xyz, tets, region, materials) of a cube of n voxels per edge in a box
    of twice its edge: "soft" permalloy on a uniform lattice, "hard" Nd2Fe14B
    with jittered nodes, "grains" a polycrystal with a grain-boundary phase in
    a graded box."""
    if kind == "grains":
        h = 250e-9 / 149
        ax = _graded(n * h / 2, h, n * h, 1.06)
    else:
        h = (40e-9 if kind == "soft" else 80e-9) / n
        nb = 2 * n if n % 2 == 0 else 2 * n + 1
        ax = (np.arange(nb + 1) - nb / 2.0) * h
    nv = len(ax) - 1
    lo = (nv - n) // 2
    xyz, tets, vox = _lattice(ax, ax, ax)
    inside = np.ones(vox[0].size, dtype=bool)
    for v in vox:
        inside &= (v >= lo) & (v < lo + n)
    region = np.repeat(inside, 6).astype(np.int32)
    air = (0, 0, 0, 0, 0, 1)
    if kind == "soft":
        return xyz, tets, region, np.array([air, (*PERMALLOY, 1, 0, 0)], dtype=np.float64)
    if kind == "hard":
        q = np.arange(nv + 1)
        free = [(q > 0) & (q < nv), (q > lo) & (q < lo + n), (q >= lo) & (q <= lo + n)]
        box, core, hull = ((f[:, None, None] & f[None, :, None] & f[None, None, :]).ravel() for f in free)
        move = core | (box & ~hull)
        shift = np.random.default_rng(2).uniform(-0.07 * h, 0.07 * h, size=xyz.shape)
        xyz[move] += shift[move]
        t = math.radians(1.0)
        return xyz, tets, region, np.array([air, (*ND2FE14B, math.sin(t), 0, math.cos(t))], dtype=np.float64)
    grains = max(2, round(37 * (n / 100.0) ** 3))
    rng = np.random.default_rng(5)
    seeds = rng.uniform(-n * h / 2, n * h / 2, size=(grains, 3))
    c = rng.uniform(math.cos(math.radians(15.0)), 1.0, size=grains)
    az, s = rng.uniform(0.0, 2 * math.pi, size=grains), np.sqrt(1 - c * c)
    sel = np.nonzero(region)[0]
    cen = torch.from_numpy(xyz).cuda()[torch.from_numpy(tets[sel]).cuda().long()].mean(dim=1)
    sd = torch.from_numpy(seeds).cuda()
    lab = torch.empty(len(sel), dtype=torch.int32, device="cuda")
    for a in range(0, len(sel), 1 << 20):
        d = ((cen[a:a + (1 << 20), None] - sd[None]) ** 2).sum(-1)
        two, idx = torch.topk(d, 2, dim=1, largest=False)
        sep = (sd[idx[:, 0]] - sd[idx[:, 1]]).norm(dim=1)
        own = (idx[:, 0] + 1).int()
        lab[a:a + (1 << 20)] = torch.where((two[:, 1] - two[:, 0]) / (2 * sep) < 1e-9, grains + 1, own)
    region[sel] = lab.cpu().numpy()
    rows = [air] + [(*ND2FE14B, s[g] * math.cos(az[g]), s[g] * math.sin(az[g]), c[g]) for g in range(grains)]
    rows.append((0.4 * ND2FE14B[0], ND2FE14B[1], 0.4 * ND2FE14B[2], 0, 0, 1))
    return xyz, tets, region, np.array(rows, dtype=np.float64)


def _platelet_axes(case, k):
    """Axes and half-extents of platelet k: 5 nm of permalloy, ellipse,
    rectangle or disc, in a graded air box."""
    rng = np.random.default_rng(4000 + k)
    long = rng.uniform(100.0, case["longest"]) * NM
    shape = ("ellipse", "rectangle", "disc")[k % 3]
    a = long / 2
    b = a if shape == "disc" else a / rng.uniform(1.0, 3.0)
    h = 2.5e-9
    axes = []
    for half, box in ((a, 1.3 * a), (b, 1.3 * a), (2.5e-9, max(0.65 * a, 15e-9))):
        half = h * max(1, round(half / h))
        axes.append(_graded(half, h, max(box, half + h), 2.0))
    return shape, a, b, axes


def _platelet_mesh(case, k):
    shape, a, b, axes = _platelet_axes(case, k)
    xyz, tets, _ = _lattice(*axes)
    c = xyz[tets].mean(axis=1)
    if shape == "rectangle":
        flat = (np.abs(c[:, 0]) < a) & (np.abs(c[:, 1]) < b)
    else:
        flat = (c[:, 0] / a) ** 2 + (c[:, 1] / b) ** 2 < 1.0
    region = (flat & (np.abs(c[:, 2]) < 2.5e-9)).astype(np.int32)
    return xyz, tets, region, np.array([(0, 0, 0, 0, 0, 1), (*PERMALLOY, 1, 0, 0)], dtype=np.float64)


_HANDLES = {}


def _handle(key, make):
    """The uploaded magnet of a mesh and its node coordinates on the GPU."""
    if key not in _HANDLES:
        xyz, tets, region, mats = make()
        mag = Magnet(device=0)
        mag.upload_mesh(xyz, tets, region, mats)
        _HANDLES[key] = (mag, torch.from_numpy(xyz / np.abs(xyz).max()).cuda())
    return _HANDLES[key]


def _cube(case):
    return _handle((case["mesh"], case["n"]), lambda: _cube_mesh(case["mesh"], case["n"]))


# ------------------------------------------------------------------- inputs

def _state(x, hard, seed):
    """A magnetisation as a field sweep meets it: the remanent direction (z of
    a hard, x of a soft magnet) with a smooth tilt of a few degrees and a
    little node-wise noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    m = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
    m[:, 2 if hard else 0] = 1.0
    tilt = torch.zeros_like(m)
    for _ in range(6):
        k = torch.randn(3, generator=g, device="cuda", dtype=torch.float64) * 3.0
        p = torch.rand(1, generator=g, device="cuda", dtype=torch.float64) * 2 * math.pi
        v = torch.randn(3, generator=g, device="cuda", dtype=torch.float64)
        tilt += torch.sin(x @ k + p)[:, None] * v
    m += 0.04 * tilt + 1e-3 * torch.randn(m.shape, generator=g, device="cuda", dtype=torch.float64)
    return (m / m.norm(dim=1, keepdim=True)).contiguous()


def _field(hard, seed):
    """An applied field of the sweep: 0 to -4 T along z (before a hard magnet
    switches), +-100 mT along x for a soft one."""
    u = np.random.default_rng(seed).uniform()
    return np.array([0.0, 0.0, -4.0 * u]) if hard else np.array([0.1 - 0.2 * u, 0.0, 0.0])


def _params(case):
    # the precision forms at the potential tolerance of the parity tests, so
    # that iterates depend on the inner solver in rounding only
    form = {"fp64": {"poisson_tol": 1e-10}, "fp32": {"precision": 1, "poisson_tol": 1e-12},
            "multigrid": {"precision": 1, "poisson_tol": 1e-12, "amg": 1, "inner_tol": 1e-3}}
    return Params(jmax=4, max_iter=case.get("iters", 10000), **form[case["form"]])


def _weights(seed):
    rng = np.random.default_rng(seed)
    out = []
    for a, b in zip(WIDTHS[:-1], WIDTHS[1:]):
        lim = math.sqrt(6.0 / a)
        out += [rng.uniform(-lim, lim, size=a * b), rng.uniform(-0.1, 0.1, size=b)]
    return np.concatenate(out).astype(np.float32)


def _features(rows, seed):
    """Features as mm_warmstart_features gives them (unit vectors near z,
    fields of order one, a constant field increment, the potential) and
    targets that follow from them: X [rows, 16], T [rows, 4]."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((rows, 16), generator=g, device="cuda")
    X[:, 0:2] *= 0.05
    X[:, 2] = 1.0 - 0.5 * (X[:, 0] ** 2 + X[:, 1] ** 2)
    X[:, 12:15] = torch.randn(3, generator=g, device="cuda") * 0.05
    X[:, 15] *= 20.0
    w = torch.randn((16, 4), generator=g, device="cuda") * 0.3
    w[15] /= 20.0
    T = torch.tanh(X @ w) + 0.05 * torch.randn((rows, 4), generator=g, device="cuda")
    return X.contiguous(), T.contiguous()


def _norms():
    """The input standardisation that such features have."""
    mean, std = np.zeros(16, np.float32), np.ones(16, np.float32)
    mean[2], std[0:2], std[2], std[15] = 0.9975, 0.05, 2.5e-3, 20.0
    return mean, std


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "gradient", "operators"):
        mag, x = _cube(case)
        hard = case["mesh"] != "soft"
        s = {"kind": kind, "mag": mag}
        if kind == "operators":
            g = torch.Generator(device="cuda").manual_seed(seed)
            s["v"] = _state(x, hard, seed).cpu().numpy()
            s["phi"] = (torch.sin(x @ torch.tensor([2.0, 1.0, 3.0], dtype=torch.float64, device="cuda"))
                        + 0.1 * torch.randn(len(x), generator=g, device="cuda", dtype=torch.float64)).cpu().numpy()
            return s
        s.update(b=_field(hard, seed), params=_params(case), m=_state(x, hard, seed))
        if kind == "gradient":
            s["m"] = s["m"].cpu().numpy()
        else:
            s["out"] = torch.empty_like(s["m"])
        return s
    if kind == "batch":
        key = ("batch", case["members"], case["longest"])
        if key not in _HANDLES:
            _HANDLES[key] = [_handle(("platelet", case["longest"], k), lambda k=k: _platelet_mesh(case, k))
                             for k in range(case["members"])]
        mags = _HANDLES[key]
        ms = [_state(x, False, 100 * seed + k) for k, (_, x) in enumerate(mags)]
        return {"kind": kind, "mags": [m for m, _ in mags], "batch": Batch([m for m, _ in mags]), "m": ms,
                "b": [_field(False, 100 * seed + k) for k in range(len(mags))], "params": _params(case),
                "out": [torch.empty_like(m) for m in ms]}
    X, T = _features(case["rows"], seed)
    mlp = MLP(device=0, seed=0)
    s = {"kind": kind, "mlp": mlp, "X": X}
    if kind == "fit":
        s["T"] = 3.0 * T + 0.5
        return s
    mlp.set_params(_weights(seed))
    mlp.set_input_norm(*_norms())
    if kind == "train":
        s["T"] = T
        torch.cuda.synchronize()
        for _ in range(TRAINED):
            mlp.train_step(X, T, LR)
    return s


def run(state):
    kind = state["kind"]
    if kind == "step":
        mag = state["mag"]
        mag.set_magnetization_dev(state["m"])
        mag.set_field(state["b"])
        st = mag.minimize(state["params"])
        mag.get_magnetization_dev(state["out"])
        return {"m": state["out"], "F": st["F_internal"], "M": st["M"]}
    if kind == "batch":
        for mag, m, b in zip(state["mags"], state["m"], state["b"]):
            mag.set_magnetization_dev(m)
            mag.set_field(b)
        st = state["batch"].minimize(state["params"])
        for mag, out in zip(state["mags"], state["out"]):
            mag.get_magnetization_dev(out)
        return {"m": state["out"], "F": [s["F_internal"] for s in st]}
    if kind == "gradient":
        mag = state["mag"]
        mag.set_field(state["b"])
        return mag.gradient(state["m"], projected=False, params=state["params"])
    if kind == "operators":
        mag, v, phi = state["mag"], state["v"], state["phi"]
        return {"local": mag.local_apply(v), "div": mag.divergence(v), "divt": mag.divergence_t(phi),
                "potential": mag.potential_matvec(phi)}
    mlp = state["mlp"]
    if kind == "forward":
        return mlp.forward(state["X"])
    if kind == "train":
        loss = mlp.train_step(state["X"], state["T"], LR, want_loss=True)
        return {"loss": loss, "params": mlp.get_params()}
    mlp.fit_input_norm(state["X"])
    mean, istd = mlp.input_norm()
    Tn, sm, sp = mlp.fit_target_scales(state["T"])
    return {"mean": mean, "istd": istd, "targets": Tn, "scale_m": sm, "scale_phi": sp}


# --------------------------------------------------------- necessary work

def _sizes(case):
    """(nodes, magnetic nodes, potential unknowns) of a cube."""
    n = case["n"]
    if case["mesh"] == "grains":
        h = 250e-9 / 149
        nv = len(_graded(n * h / 2, h, n * h, 1.06)) - 1
    else:
        nv = 2 * n if n % 2 == 0 else 2 * n + 1
    return (nv + 1) ** 3, (n + 1) ** 3, (nv - 1) ** 3


def _evaluation(nm, nphi, couplings):
    """One energy and gradient: the potential stiffness (`couplings` entries a
    row), the exchange stiffness and the divergence coupling (15 entries a
    row, one and three values) read once, the state in, gradient and potential
    out.  The steps of the iterative solve come on top; how many there are is
    the method's affair and not counted."""
    return {"bytes": 8.0 * (couplings * nphi + 15 * 4 * nm) + 8.0 * (nphi + 14 * nm),
            "flops": 2.0 * (couplings * nphi + 15 * 9 * nm)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for k in range(case["members"]):
            shape, a, b, axes = _platelet_axes(case, k)
            area = 4 * a * b if shape == "rectangle" else math.pi * a * b
            one = _evaluation(3 * area / 2.5e-9 ** 2, np.prod([len(v) - 2.0 for v in axes]), 7)
            for q in total:
                total[q] += (1 + 2 * case["iters"]) * float(one[q])
        return total
    if kind in ("step", "gradient", "operators"):
        n, nm, nphi = _sizes(case)
        one = _evaluation(nm, nphi, 15 if case["mesh"] == "hard" else 7)
        if kind == "step":                 # two evaluations per iteration, one before the first
            return {q: (1 + 2 * case["iters"]) * v for q, v in one.items()}
        if kind == "gradient":
            return {"bytes": one["bytes"] + 48.0 * n, "flops": one["flops"]}
        return {"bytes": one["bytes"] + 8.0 * (15 * 3 * nm + 12 * n), "flops": one["flops"] + 2.0 * 15 * 3 * nm}
    rows, params = float(case["rows"]), float(sum(a * b + b for a, b in zip(WIDTHS[:-1], WIDTHS[1:])))
    layers = float(sum(a * b for a, b in zip(WIDTHS[:-1], WIDTHS[1:])))
    if kind == "forward":
        return {"bytes": 80.0 * rows + 4 * params, "flops": 2 * layers * rows}
    if kind == "train":
        return {"bytes": 80.0 * rows + 24 * params, "flops": 6 * layers * rows}
    return {"bytes": (64.0 + 16.0 + 16.0) * rows, "flops": (16 + 4) * 4 * rows}


# ------------------------------------------------- the same in 64 bits

def _assemble(case):
    """The sparse operators of the energy on a cube, in units of nm and
    mu0 Mref^2 nm^3, all over the mesh's nodes, with plain torch in FP64."""
    xyz, tets, region, mats = _cube_mesh(case["mesh"], case["n"])
    x, t = torch.from_numpy(xyz / NM).cuda(), torch.from_numpy(tets).cuda().long()
    mat = torch.from_numpy(mats).cuda()[torch.from_numpy(region).cuda().long()]
    mref = float(mats[:, 0].max())
    N = len(x)
    e = x[t[:, 1:]] - x[t[:, :1]]
    c = torch.stack([torch.linalg.cross(e[:, 1], e[:, 2]), torch.linalg.cross(e[:, 2], e[:, 0]),
                     torch.linalg.cross(e[:, 0], e[:, 1])], dim=1)
    det = (e[:, 0] * c[:, 0]).sum(-1)
    b = torch.cat([-(c.sum(1, keepdim=True)), c], dim=1) / det[:, None, None]
    vol = det.abs() / 6

    def sparse(rows, cols, vals):
        m = torch.sparse_coo_tensor(torch.stack([rows.reshape(-1), cols.reshape(-1)]), vals.reshape(-1), (N, N))
        return m.coalesce().to_sparse_csr()

    def pairs(q):
        return q[:, :, None].expand(-1, 4, 4), q[:, None, :].expand(-1, 4, 4)

    K = sparse(*pairs(t), vol[:, None, None] * (b @ b.transpose(1, 2)))
    on = mat[:, 0] > 0
    tm, bm, vm, mm = t[on], b[on], vol[on], mat[on]
    A = sparse(*pairs(tm), (mm[:, 1] / (MU0 * mref ** 2 * NM ** 2) * vm)[:, None, None] * (bm @ bm.transpose(1, 2)))
    ms = mm[:, 0] / mref * vm / 4
    D = [sparse(*pairs(tm), (ms[:, None] * bm[:, :, q])[:, :, None].expand(-1, 4, 4)) for q in range(3)]
    Dt = [sparse(*pairs(tm), (ms[:, None] * bm[:, :, q])[:, None, :].expand(-1, 4, 4)) for q in range(3)]
    axis = mm[:, 3:6] / mm[:, 3:6].norm(dim=1, keepdim=True)
    ck = -2 * (mm[:, 2] / (MU0 * mref ** 2) * vm / 4)[:, None, None] * axis[:, :, None] * axis[:, None, :]
    CK = torch.zeros((N, 3, 3), dtype=torch.float64, device="cuda")
    w = torch.zeros(N, dtype=torch.float64, device="cuda")
    for q in range(4):
        CK.index_add_(0, tm[:, q], ck)
        w.index_add_(0, tm[:, q], ms)
    lo, hi = x.min(0).values, x.max(0).values
    free = ((x > lo) & (x < hi)).all(dim=1)
    magnetic = torch.zeros(N, dtype=torch.bool, device="cuda")
    magnetic[tm.reshape(-1)] = True
    diag = torch.zeros(N, dtype=torch.float64, device="cuda")
    diag.index_add_(0, t.reshape(-1), (vol[:, None] * (b * b).sum(-1)).reshape(-1))
    return {"K": K, "A": A, "D": D, "Dt": Dt, "CK": CK, "w": w, "free": free, "magnetic": magnetic, "diag": diag,
            "mref": mref}


def _local(P, v):
    return 2 * torch.stack([P["A"] @ v[:, q] for q in range(3)], dim=1) + torch.einsum("iab,ib->ia", P["CK"], v)


def _div(P, v):
    return P["free"] * sum(P["D"][q] @ v[:, q].contiguous() for q in range(3))


def _div_t(P, phi):
    return torch.stack([P["Dt"][q] @ phi for q in range(3)], dim=1)


def _potential(P, rhs):
    """K phi = rhs on the free nodes by conjugate gradients to rounding."""
    free = P["free"].double()
    phi, r = torch.zeros_like(rhs), rhs.clone()
    z = r / P["diag"]
    d, rz, stop = z.clone(), float(r @ z), 1e-14 * float(rhs.norm())
    for it in range(20000):
        q = free * (P["K"] @ d)
        a = rz / float(d @ q)
        phi += a * d
        r -= a * q
        if it % 8 == 0 and float(r.norm()) < stop:
            break
        z = r / P["diag"]
        new = float(r @ z)
        d = z + (new / rz) * d
        rz = new
    return phi


def _net(w, x):
    """The network's layers in 64 bits: the inputs of every layer and the output."""
    acts, o = [], 0
    for a, b in zip(WIDTHS[:-1], WIDTHS[1:]):
        acts.append(x)
        W, c = w[o:o + a * b].reshape(b, a), w[o + a * b:o + a * b + b]
        o += a * b + b
        x = x @ W.T + c
        if b != WIDTHS[-1]:
            x = torch.relu(x)
    return acts, x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("gradient", "operators"):
        P = _assemble(case)
        xyz = _cube(case)[1]
        hard = case["mesh"] != "soft"
        on = P["magnetic"][:, None]
        if kind == "operators":
            s = prepare(case, seed)
            v, phi = torch.from_numpy(s["v"]).cuda() * on, torch.from_numpy(s["phi"]).cuda() * P["free"]
            return {"local": (_local(P, v) * on).cpu(), "div": _div(P, v).cpu(), "divt": (_div_t(P, phi) * on).cpu(),
                    "potential": (P["free"] * (P["K"] @ phi)).cpu()}
        m = _state(xyz, hard, seed) * on
        h = torch.from_numpy(_field(hard, seed) / (MU0 * P["mref"])).cuda()
        g = _local(P, m) + _div_t(P, _potential(P, _div(P, m))) - P["w"][:, None] * h
        return (g * on).cpu()
    if kind in ("step", "batch"):
        return None                        # iterates of the whole minimiser: no value apart from its own path
    X, T = _features(case["rows"], seed)
    if kind == "fit":
        T = (3.0 * T + 0.5).double()
        out = {"mean": X.double().mean(0), "istd": 1 / X.double().std(0)}
        out["istd"][12:15] = 1.0           # constant columns are only centred
        sm, sp = T[:, :3].std(), T[:, 3].std()
        out["targets"] = T / torch.stack([sm, sm, sm, sp])
        return {**out, "scale_m": float(sm), "scale_phi": float(sp)}
    w = torch.from_numpy(_weights(seed)).cuda().double()
    mean, std = (torch.from_numpy(v).cuda().double() for v in _norms())
    if kind == "forward":
        return torch.cat([_net(w, (c.double() - mean) / std)[1] for c in X.split(1 << 18)])
    X, T = (X.double() - mean) / std, T.double()
    m1, m2, b1, b2 = torch.zeros_like(w), torch.zeros_like(w), 0.9, 0.999
    for k in range(1, TRAINED + 2):
        acts, y = _net(w, X)
        d, grads = 2 * (y - T) / T.numel(), []
        o = w.numel()
        for l in range(3, -1, -1):
            a, b = WIDTHS[l], WIDTHS[l + 1]
            W = w[o - b - a * b:o - b].reshape(b, a)
            grads[:0] = [(d.T @ acts[l]).reshape(-1), d.sum(0)]
            o -= a * b + b
            if l:
                d = (d @ W) * (acts[l] > 0)
        g = torch.cat(grads)
        loss = float(((y - T) ** 2).mean())
        m1, m2 = b1 * m1 + (1 - b1) * g, b2 * m2 + (1 - b2) * g * g
        w = w - LR * (m1 / (1 - b1 ** k)) / ((m2 / (1 - b2 ** k)).sqrt() + 1e-8)
    return {"loss": loss, "params": w}
