"""Performance cases of the finite cell Schwarz-PCG library: the calls a user's program makes.

A solve applies the stiffness K and the Schwarz operator S once per iteration, and, with the coarse correction, the
Galerkin operator K_H and a multigrid cycle on the cell grid; a user who writes their own Krylov loop, who trains
the learned correction or who refines locally calls those applies themselves.  So the cases are those applies over
the sizes of the library's workloads, two whole solves, and the network's inference and training step.

`listed()` gives the fixed cases, `draw(rng)` more of the same ranges.  `prepare(case, seed)` builds what a program
holds before the call: the problem's handle (geometry, stiffness, factors; kept between seeds, as a program keeps it
between right-hand sides) and vectors drawn from the seed.  `run(state)` is one pass through the public entry points.
`exact(case, seed)` computes the same outputs in 64 bits with torch and numpy alone.
"""
import collections
import math

import numpy as np
import torch

from paper_1809_00828_gb300 import fcm, inputs

F64, F32 = torch.float64, torch.float32


def listed():
    return [
        # One K and one S on the smallest problem (1,944 free DOFs, FP64): what a user's own Krylov loop pays per
        # iteration where only launches and latency count.
        _grid("ops_4_p2", "ops", 4, 4, 4, 2, geo="single", alpha=1e-8, depth=3, k="fp64", prec="fp64"),
        # The whole plain FP64 solve of that problem to its tolerance: the latency of many short iterations.
        _grid("pcg_4_p2", "pcg", 4, 4, 4, 2, geo="single", alpha=1e-8, depth=3, k="fp64", prec="fp64", tol=1e-10),
        # K x in the default FP64 arithmetic at the cubic order, 2.7M DOFs, 2,006 cut cells (porous40_32_p3).
        _grid("k_fp64_32_p3", "k", 32, 32, 32, 3, voids=40, geo_seed=11, depth=4, k="fp64", prec="mixed"),
        # S r with mixed factors of the same problem: blocks of 375 rows, each cut patch with its own factor.
        _grid("s_mixed_32_p3", "s", 32, 32, 32, 3, voids=40, geo_seed=11, depth=4, k="fp64", prec="mixed"),
        # K x in double-float arithmetic on the largest grid (porous300_80_p2, 11.4M free DOFs, 72,000 cut cells).
        _grid("k_ff_80_p2", "k", 80, 80, 80, 2, voids=300, geo_seed=21, depth=3, k="double_float", prec="mixed"),
        # S r with mixed factors there: half a million blocks of 81 rows, 4.7 GB of factors.
        _grid("s_mixed_80_p2", "s", 80, 80, 80, 2, voids=300, geo_seed=21, depth=3, k="double_float", prec="mixed"),
        # K_H x and one V-cycle on that cell grid: the coarse correction's two operators.
        _grid("coarse_80_p2", "coarse", 80, 80, 80, 2, voids=300, geo_seed=21, depth=3, k="double_float", prec="mixed"),
        # S on the six unit-strain residuals of a trabecular bone cube at once (trabecular_24_p3).
        _grid("s_many6_24_p3", "s", 24, 24, 24, 3, geo="bone", geo_seed=13, depth=3, k="double_float", prec="mixed",
              nrhs=6),
        # The whole flexible solve of a training-sized cube (the porous40_32_p2 voids), run until its answer no
        # longer depends on the rounding of the preconditioner.
        _grid("fpcg_32_p2", "fpcg", 32, 32, 32, 2, voids=40, geo_seed=7, alpha=1e-8, depth=3, k="fp64",
              prec="mixed", coarse="jacobi", coarse_iters=20, tol=1e-12),
        # The network's prediction on the evaluation cube: 4 levels, 16 to 64 channels, 80^3 cells.
        {"name": "unet_fwd_80", "kind": "unet_fwd", "nx": 80, "ny": 80, "nz": 80, "batch": 1, "base": 16, "levels": 4},
        # One training step's forward and backward on four training cubes (32^3 cells), gradients read back.
        {"name": "unet_train_32", "kind": "unet_train", "nx": 32, "ny": 32, "nz": 32, "batch": 4, "base": 16,
         "levels": 4},
        # K and S of the multi-level cube with a small cavity, refined three times (8^3 base cells, p = 3).
        {"name": "mlhp_8_p3_k3", "kind": "mlhp", "nx": 8, "ny": 8, "nz": 8, "p": 3, "levels": 3, "radius": 0.01,
         "prec": "mixed"},
    ]


def _grid(name, kind, nx, ny, nz, p, geo="porous", voids=1, geo_seed=0, alpha=1e-10, depth=3, **more):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "p": p, "geo": geo, "voids": voids, "geo_seed": geo_seed,
         "alpha": alpha, "depth": depth, **more}
    return {"name": name, **c} if name else c


def draw(rng):
    """A case of the listed ranges: any of the calls, grids of unequal sides, every order the call is used with."""
    kind = rng.choice(["ops", "pcg", "k", "k", "s", "s", "s", "many", "coarse", "fpcg", "unet_fwd", "unet_train", "mlhp"])
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    if kind in ("unet_fwd", "unet_train"):
        levels = rng.choice([2, 3, 4])
        d = 1 << (levels - 1)
        top = 64 if kind == "unet_fwd" else 32
        nx, ny, nz = (max(1, log(8, top) // d) * d for _ in range(3))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "batch": rng.choice([1, 2, 3, 4]),
                "base": rng.choice([4, 8, 12, 16]), "levels": levels}
    if kind == "mlhp":
        p = rng.choice([2, 3])
        nx, ny, nz = (rng.choice([4, 5, 6, 7, 8]) for _ in range(3))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "p": p, "levels": rng.choice([1, 2]),
                "radius": round(rng.uniform(0.05, 0.15), 4), "prec": rng.choice(["mixed", "fp64"])}
    seed, depth = rng.randrange(1, 1000), rng.choice([2, 3])
    voids = rng.choice([5, 10, 20, 40])
    small = {"ops": 7, "pcg": 6, "fpcg": 14}.get(kind)
    if kind in ("ops", "pcg"):
        p = rng.choice([1, 2, 2, 3])
        hi = small if p < 3 else 5
        n = [log(2, hi) for _ in range(3)]
        more = {"k": "fp64", "prec": "fp64"}
        if kind == "pcg":
            more["tol"] = 1e-10
        return _grid(None, kind, *n, p, voids=min(voids, 10), geo_seed=seed, alpha=1e-8, depth=depth, **more)
    if kind == "fpcg":
        n = [log(6, small) for _ in range(3)]
        return _grid(None, kind, *n, 2, voids=voids, geo_seed=seed, alpha=1e-8, depth=depth, k="double_float",
                     prec="mixed", coarse=rng.choice(["jacobi", "vcycle", "hybrid"]), coarse_iters=rng.choice([2, 5, 20]),
                     tol=1e-12)
    if kind == "k":
        p = rng.choice([1, 2, 2, 3, 3, 4])
        hi = {1: 64, 2: 56, 3: 28, 4: 14}[p]
        n = [log(5, hi) for _ in range(3)]
        return _grid(None, kind, *n, p, voids=voids, geo_seed=seed, depth=depth, k=rng.choice(["fp64", "double_float"]),
                     prec="mixed")
    if kind == "coarse":
        n = [log(6, 56) for _ in range(3)]
        return _grid(None, kind, *n, rng.choice([1, 2, 3]) if max(n) < 24 else 2, voids=voids, geo_seed=seed, depth=depth,
                     k="double_float", prec="mixed")
    p = rng.choice([2, 2, 3, 3, 4]) if kind == "s" else rng.choice([2, 3])
    hi = {2: 40, 3: 18, 4: 5}[p]
    n = [log(3 if p == 4 else 5, hi) for _ in range(3)]
    more = {"nrhs": rng.choice([2, 3, 6, 8])} if kind == "many" else {}
    return _grid(None, "s", *n, p, voids=voids, geo_seed=seed, depth=depth, k="double_float",
                 prec=rng.choice(["mixed", "mixed", "fp64", "mixed_fp64"]), blocks=rng.choice(["vertex", "vertex", "element"]), **more)


# ---- what a program holds: the handle of a problem, kept between right-hand sides


def _workload(c):
    n = (c["nx"], c["ny"], c["nz"])
    if c["geo"] == "single":
        geo = inputs.single_sphere_void(c["geo_seed"], 0.3, 0.05, octree_depth=c["depth"])
    elif c["geo"] == "bone":
        geo = inputs.gaussian_random_field_voxels(c["geo_seed"], 128, 0.05, 0.25, octree_depth=c["depth"])
    else:
        geo = inputs.random_sphere_voids(c["geo_seed"], c["voids"], 0.02, 0.08, octree_depth=c["depth"])
        if max(n) < 16:  # spheres of cell size, so that small grids have cut cells too
            geo.spheres[:, 3] *= 32.0 / (2 * max(n))
    return inputs.Workload("case", n, c["p"], c["alpha"], geo, c.get("tol", 1e-8))


class _Handle:
    def __init__(self, c):
        self.solver = fcm.Solver(_workload(c))
        self.solver.set_k_precision(c["k"])
        self.built = None

    def with_factors(self, c):
        want = (c["prec"], c.get("blocks", "vertex"))
        if self.built != want:
            self.solver.precond_build(precision=want[0], blocks=want[1])
            self.built = want
        return self.solver


class _Plan:
    """A multi-level plan on the device, with the system and the factors that the set-up calls returned."""

    def __init__(self, c):
        n, lo, hi = (c["nx"], c["ny"], c["nz"]), (0, 0, 0), (1, 1, 1)
        self.plan = fcm.MLHPPlan(n, lo, hi, [(0.5, 0.5, 0.5, c["radius"])], c["p"], c["levels"], octree_depth=3)
        _, self.K, self.rhs, _ = self.plan.assemble(1e-8, "clamp")
        self.blocks, self.factors, _, self.jac = self.plan.factorize("truncated", device=True)
        self.plan.device_setup(precision=c["prec"])
        self.fp32, self.factor_bytes = self.plan.device_info()


_handles = collections.OrderedDict()


def _kept(key, make):
    """The few problems in use, least recently used first to go."""
    if key in _handles:
        _handles.move_to_end(key)
        return _handles[key]
    while len(_handles) >= 6:
        old = _handles.popitem(last=False)[1]
        (old.plan if isinstance(old, _Plan) else old.solver).close()
    _handles[key] = make()
    return _handles[key]


def _handle(c):
    keys = ("nx", "ny", "nz", "p", "geo", "voids", "geo_seed", "alpha", "depth", "k")
    return _kept(tuple(c[k] for k in keys) + (c.get("blocks", "vertex") if c["kind"] == "s" else "vertex",),
                 lambda: _Handle(c))


def _plan(c):
    return _kept(("mlhp",) + tuple(sorted((k, v) for k, v in c.items() if k != "name")), lambda: _Plan(c))


def _normal(seed, n, dtype=F64, which=0):
    g = torch.Generator(device="cuda").manual_seed(1000 * int(seed) + which)
    return torch.randn(n, dtype=dtype, device="cuda", generator=g)


def _lattice(c):
    return [c["p"] * c[a] + 1 for a in ("nx", "ny", "nz")]


def _smooth(c, seed):
    """A displacement-like lattice vector: low waves plus 1e-2 of noise, the shape of iterates and residuals."""
    M = _lattice(c)
    g = np.random.default_rng(seed)
    ax = [torch.linspace(0, 1, m, dtype=F64, device="cuda") for m in M]
    v = torch.zeros((M[2], M[1], M[0], 3), dtype=F64, device="cuda")
    for a in range(3):
        for _ in range(3):
            k, ph = g.uniform(0.5, 3.0, 3), g.uniform(0, 2 * np.pi, 3)
            s = [torch.sin(2 * np.pi * k[i] * ax[i] + ph[i]) for i in range(3)]
            v[..., a] += s[2][:, None, None] * s[1][None, :, None] * s[0][None, None, :]
    return v.reshape(-1) + 1e-2 * _normal(seed, v.numel(), which=7)


def _load(c, seed):
    """A right-hand side: the problem's traction and a seeded mix of its unit-strain loads."""
    s = _handle(c).solver
    g = np.random.default_rng(seed)
    b = s.rhs(0)
    for k in (1, 4):
        b += float(g.uniform(-0.3, 0.3)) * s.rhs(k)
    return b


def _unet_input(c, seed):
    x = _normal(seed, c["batch"] * 4 * c["nz"] * c["ny"] * c["nx"], F32).view(c["batch"], 4, c["nz"], c["ny"], c["nx"])
    x[:, 3] = torch.clamp(1.2 - 0.5 * x[:, 3].abs(), 0.0, 1.0)  # volume fractions, most of them 1
    return x


def _channels(c):
    """(cin, cout) of every convolution: two per level down, two per level up, the output layer."""
    ch = [min(c["base"] << l, 4 * c["base"]) for l in range(c["levels"])]
    conv = []
    for l in range(c["levels"]):
        conv += [(4 if l == 0 else ch[l - 1], ch[l]), (ch[l], ch[l])]
    for l in range(c["levels"] - 2, -1, -1):
        conv += [(ch[l + 1] + ch[l], ch[l]), (ch[l], ch[l])]
    return conv + [(ch[0], 3)]


def _unet_weights(c, seed):
    """Kaiming-uniform weights and small biases for a prediction.  A training step's gradients jump where a ReLU's
    input changes sign, so two roundings of one network can differ by 1e-3: there the weights are smaller and the
    biases (three of four positive) larger, which keeps every ReLU away from its kink."""
    g = np.random.default_rng(seed + 77)
    parts = []
    for k, (ci, co) in enumerate(_channels(c)):
        train = c["kind"] == "unet_train"
        bound = math.sqrt(6.0 / (27 * ci)) * ((0.02 if k == 0 else 0.1) if train else 1.0)
        b = g.uniform(0.8, 1.2, co) * np.where(np.arange(co) % 4 == 3, -1, 1) if train else g.uniform(-0.05, 0.05, co)
        parts += [g.uniform(-bound, bound, co * ci * 27), b]
    return np.concatenate(parts).astype(np.float32)


def prepare(case, seed):
    c = case
    st = {"case": c}
    if c["kind"].startswith("unet"):
        net = fcm.UNet(4, 3, c["base"], c["levels"], seed=0)
        net.set(_unet_weights(c, seed))
        st.update(net=net, x=_unet_input(c, seed))
        shape = (c["batch"], 3, c["nz"], c["ny"], c["nx"])
        st["out"] = torch.empty(shape, dtype=F32, device="cuda")
        if c["kind"] == "unet_train":
            st["gout"] = _normal(seed, st["out"].numel(), F32, 3).view(shape) / st["out"].numel()
        return st
    if c["kind"] == "mlhp":
        h = _plan(c)
        x, r = _normal(seed, len(h.rhs)), _normal(seed, len(h.rhs), which=1)
        return {"case": c, "plan": h.plan, "x": x, "r": r, "y": torch.empty_like(x), "z": torch.empty_like(r)}
    h = _handle(c)
    s = st["solver"] = h.solver
    if c["kind"] != "k" and c["kind"] != "coarse":
        h.with_factors(c)
    nc = 3 * c["nx"] * c["ny"] * c["nz"]
    if c["kind"] in ("ops", "k"):
        st.update(x=_smooth(c, seed), y=s.empty())
    if c["kind"] in ("ops", "s"):
        m = c.get("nrhs", 1)
        st.update(r=torch.cat([_smooth(c, 31 * seed + i) for i in range(m)]), z=s.empty(m))
    if c["kind"] in ("pcg", "fpcg"):
        st.update(b=_load(c, seed), u=s.empty())
    if c["kind"] == "fpcg":
        s.set_coarse_preconditioner(c["coarse"])
    if c["kind"] == "coarse":
        st.update(cx=_normal(seed, nc, F32), cy=torch.empty(nc, dtype=F32, device="cuda"),
                  cf=_normal(seed, nc, F32, 1), cv=torch.empty(nc, dtype=F32, device="cuda"))
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    s = state.get("solver")
    if kind == "ops":
        return {"Kx": s.apply_K(state["x"], out=state["y"]), "Sr": s.apply_S(state["r"], out=state["z"])}
    if kind == "k":
        return {"Kx": s.apply_K(state["x"], out=state["y"])}
    if kind == "s":
        return {"Sr": s.apply_S(state["r"], out=state["z"])}
    if kind == "pcg":
        return {"u": s.pcg_solve(state["b"], c["tol"], 20000, out=state["u"])[0]}
    if kind == "fpcg":
        return {"u": s.fpcg_solve(None, 0.0, state["b"], c["tol"], 20000, out=state["u"],
                                  coarse_iters=c["coarse_iters"])[0]}
    if kind == "coarse":
        return {"KHx": s.coarse_apply(state["cx"], out=state["cy"]), "Vf": s.coarse_vcycle(state["cf"], out=state["cv"])}
    if kind == "mlhp":
        p = state["plan"]
        return {"Kx": p.apply_K(state["x"], out=state["y"]), "Sr": p.apply_S(state["r"], out=state["z"])}
    net = state["net"]
    out = net.forward(state["x"], out=state["out"])
    if kind == "unet_fwd":
        return {"out": out}
    net.zero_grad()
    din = net.backward(state["gout"], want_din=True)
    return {"out": out, "din": din, "grad": net.get(with_grad=True)[1]}


# ---- the work of one pass


def _boxes(c):
    """Lower corners of the cells, [cell, 3] (x fastest), and the cell size."""
    n = [c["nx"], c["ny"], c["nz"]]
    i = torch.arange(n[0] * n[1] * n[2], device="cuda")
    ijk = torch.stack([i % n[0], (i // n[0]) % n[1], i // (n[0] * n[1])], 1)
    return ijk, torch.tensor([1.0 / v for v in n], dtype=F64, device="cuda")


def _classes(c):
    """Per cell: 0 solid, 1 cut by the boundary, 2 void."""
    ijk, h = _boxes(c)
    lo = ijk * h
    geo = _workload(c).geometry
    kind = torch.zeros(len(ijk), dtype=torch.int64, device="cuda")
    if geo.voxels is not None:
        vox = torch.from_numpy(geo.voxels.astype(np.float64)).cuda()
        m = torch.tensor(vox.shape[::-1], dtype=F64, device="cuda")
        s = torch.zeros([v + 1 for v in vox.shape], dtype=F64, device="cuda")
        s[1:, 1:, 1:] = vox.cumsum(0).cumsum(1).cumsum(2)
        a = torch.floor(lo * m + 1e-9).long()
        b = torch.ceil((lo + h) * m - 1e-9).long()
        at = lambda x, y, z: s[z, y, x]  # noqa: E731
        tot = sum((-1.0) ** (3 - i - j - k) * at((a, b)[i][:, 0], (a, b)[j][:, 1], (a, b)[k][:, 2])
                  for i in (0, 1) for j in (0, 1) for k in (0, 1))
        vol = (b - a).prod(1)
        kind[(tot > 0) & (tot < vol)] = 1
        kind[tot == 0] = 2
        return kind
    for x, y, z, r in geo.sphere_array():
        q = torch.tensor([x, y, z], dtype=F64, device="cuda")
        near = torch.clamp(lo - q, min=0) + torch.clamp(q - lo - h, min=0)
        far = torch.maximum((lo - q).abs(), (lo + h - q).abs())
        dmin, dmax = near.norm(dim=1), far.norm(dim=1)
        kind = torch.where(dmax <= r, torch.full_like(kind, 2), torch.where((dmin < r) & (kind == 0), torch.ones_like(kind), kind))
    return kind


def work(case):
    c = case
    if c["kind"].startswith("unet"):
        flops = nbytes = 0.0
        S = [c["batch"] * (c["nx"] >> l) * (c["ny"] >> l) * (c["nz"] >> l) for l in range(c["levels"])]
        L = c["levels"]
        level = [l for l in range(L) for _ in (0, 1)] + [l for l in range(L - 2, -1, -1) for _ in (0, 1)] + [0]
        for (ci, co), l in zip(_channels(c), level):
            flops += 54.0 * ci * co * S[l] * (3 if c["kind"] == "unet_train" else 1)
            nbytes += 2.0 * 27 * ci * co
        return {"bytes": nbytes + 4.0 * S[0] * (7 if c["kind"] == "unet_fwd" else 14), "flops": flops}
    if c["kind"] == "mlhp":
        h = _plan(c)
        rows = sum(len(b) for b in h.blocks)
        return {"bytes": 12.0 * h.K.nnz + h.factor_bytes + 32.0 * len(h.rhs) + 4.0 * rows,
                "flops": 2.0 * h.K.nnz + 2.0 * sum(len(b) ** 2 for b in h.blocks)}
    M, p = _lattice(c), c["p"]
    nlat = 3 * M[0] * M[1] * M[2]
    kind = _classes(c)
    ncut, nsolid = int((kind == 1).sum()), int((kind == 0).sum())
    cells = c["nx"] * c["ny"] * c["nz"]
    ne = 3 * (p + 1) ** 3
    # K: x and y once, the unique entries of every cut cell's matrix; 36 (p+1)^4 multiply-adds per solid cell
    kb, kf = 16.0 * nlat + 4.0 * ne * (ne + 1) * ncut, 2.0 * ncut * ne * ne + 72.0 * (p + 1) ** 4 * nsolid
    # S: r and z once, the unique entries of the factor of every vertex at a cut cell
    cut = torch.zeros((c["nz"] + 1, c["ny"] + 1, c["nx"] + 1), dtype=torch.bool, device="cuda")
    k3 = (kind == 1).view(c["nz"], c["ny"], c["nx"])
    for i in range(8):
        z, y, x = i >> 2, (i >> 1) & 1, i & 1
        cut[z:z + c["nz"], y:y + c["ny"], x:x + c["nx"]] |= k3
    nb = 3 * (2 * p - 1) ** 3
    m = c.get("nrhs", 1)
    size = 8.0 if c["prec"] == "fp64" else 4.0
    sb = 16.0 * nlat * m + 0.5 * size * nb * (nb + 1) * int(cut.sum())
    sf = 2.0 * nb * nb * (c["nx"] + 1) * (c["ny"] + 1) * (c["nz"] + 1) * m
    if c["kind"] == "k":
        return {"bytes": kb, "flops": kf}
    if c["kind"] == "s":
        return {"bytes": sb, "flops": sf}
    if c["kind"] == "ops":
        return {"bytes": kb + sb, "flops": kf + sf}
    if c["kind"] == "coarse":  # K_H x once; the cycle applies K_H twice on the finest level, 8/7 in all
        kh = 63.0 * 9 * 4 * cells
        return {"bytes": kh * (1 + 16.0 / 7), "flops": 2.0 * 125 * 9 * cells * (1 + 16.0 / 7)}
    its = 100.0  # a solve: K, S and the vector updates of about a hundred iterations
    return {"bytes": its * (kb + sb + 100.0 * nlat), "flops": its * (kf + sf)}


# ---- the same outputs in 64 bits, with torch alone


def _legendre(p, t):
    P = [torch.ones_like(t), t]
    for k in range(2, p + 1):
        P.append(((2 * k - 1) * t * P[-1] - (k - 1) * P[-2]) / k)
    return P


def _basis(p, t):
    """Values and d/dt of the cell's 1D functions at t, in lattice order (left hat, bubbles, right hat), [point, p+1]."""
    P = _legendre(p, t)
    val, der = [(1 - t) / 2], [torch.full_like(t, -0.5)]
    for j in range(2, p + 1):
        val.append((P[j] - P[j - 2]) / math.sqrt(2 * (2 * j - 1)))
        der.append(math.sqrt((2 * j - 1) / 2) * P[j - 1])
    return torch.stack(val + [(1 + t) / 2], 1), torch.stack(der + [torch.full_like(t, 0.5)], 1)


class _Exact:
    """K of a grid case, cell by cell by quadrature: (p+1)-point Gauss rules on the 2^depth-fold subdivision of a
    cut cell (the octree's leaves; its larger uncut leaves are integrated exactly either way), alpha per point."""

    def __init__(self, c):
        self.c, self.p = c, c["p"]
        self.n, self.M = [c["nx"], c["ny"], c["nz"]], _lattice(c)
        self.geo = _workload(c).geometry
        self.ijk, self.h = _boxes(c)
        kind = _classes(c)
        self.lam, self.mu = 0.3 / (1.3 * 0.4), 1 / 2.6
        q = self.p + 1
        i = torch.arange(q ** 3, device="cuda")
        loc = torch.stack([i % q, (i // q) % q, i // (q * q)], 1)
        at = self.p * self.ijk[:, None, :] + loc[None]
        self.nodes = at[..., 0] + self.M[0] * (at[..., 1] + self.M[1] * at[..., 2])
        self.solid = torch.nonzero(kind == 0).flatten()
        cut = torch.nonzero(kind == 1).flatten()
        self.chunks = []  # (cells, alpha-weighted points) of the cut cells that hold some solid point
        step = max(1, int(2e7) // ((q << c["depth"]) ** 3))
        for k in range(0, len(cut), step):
            part = cut[k:k + step]
            on = self._inside(part, c["depth"])
            keep = on.flatten(1).any(1)
            if keep.any():
                self.chunks.append((part[keep], on[keep]))
        free = torch.zeros(self.M[0] * self.M[1] * self.M[2], dtype=torch.bool, device="cuda")
        for cells in [self.solid] + [a for a, _ in self.chunks]:
            free[self.nodes[cells].flatten()] = True
        free[: self.M[0] * self.M[1]] = False
        self.free = free[:, None].expand(-1, 3).reshape(-1)

    def _points(self, depth):
        x, w = np.polynomial.legendre.leggauss(self.p + 1)
        m = 1 << depth
        t = ((2 * np.arange(m)[:, None] + 1 + x[None]) / m - 1).reshape(-1)
        return torch.from_numpy(t).cuda(), torch.from_numpy(np.tile(w / m, m)).cuda()

    def _inside(self, cells, depth):
        t, _ = self._points(depth)
        xyz = [((self.ijk[cells, a:a + 1] + (t[None] + 1) / 2) * self.h[a]) for a in range(3)]
        if self.geo.voxels is not None:
            v = torch.from_numpy(self.geo.voxels).cuda()
            i = [torch.clamp((xyz[a] * v.shape[2 - a]).long(), 0, v.shape[2 - a] - 1) for a in range(3)]
            return v[i[2][:, :, None, None], i[1][:, None, :, None], i[0][:, None, None, :]] != 0
        on = torch.ones((len(cells), len(t), len(t), len(t)), dtype=torch.bool, device="cuda")
        lo, hi = self.ijk[cells] * self.h, (self.ijk[cells] + 1) * self.h
        sph = torch.from_numpy(self.geo.sphere_array()).cuda()
        gap = torch.clamp(lo[:, None] - sph[None, :, :3], min=0) + torch.clamp(sph[None, :, :3] - hi[:, None], min=0)
        touch = gap.norm(dim=2) < sph[None, :, 3]
        for j in torch.nonzero(touch.any(0)).flatten().tolist():
            at = torch.nonzero(touch[:, j]).flatten()
            d = [(xyz[a][at] - sph[j, a]) ** 2 for a in range(3)]
            on[at] &= d[2][:, :, None, None] + d[1][:, None, :, None] + d[0][:, None, None, :] >= sph[j, 3] ** 2
        return on

    def _cells(self, x, cells, depth, on):
        """K_e x_e of the cells: gradients at the points, stress, transposed gradients."""
        q = self.p + 1
        u = x.view(-1, 3)[self.nodes[cells]].view(-1, q, q, q, 3)
        t, w = self._points(depth)
        B, D = _basis(self.p, t)
        f = [(D if a == b else B) for a in range(3) for b in range(3)]
        g = [[None] * 3 for _ in range(3)]
        for a in range(3):
            v = torch.einsum("ezyxc,px->ezypc", u, f[3 * a])
            v = torch.einsum("ezypc,qy->ezqpc", v, f[3 * a + 1])
            v = torch.einsum("ezqpc,rz->erqpc", v, f[3 * a + 2]) * (2 / self.h[a])
            for k in range(3):
                g[k][a] = v[..., k]
        wt = w[:, None, None] * w[None, :, None] * w[None, None, :] * (self.h.prod() / 8)
        if on is not None:
            wt = wt[None] * (on + (~on) * self.c["alpha"])
        tr = self.lam * (g[0][0] + g[1][1] + g[2][2])
        out = 0
        for a in range(3):
            s = torch.stack([(self.mu * (g[k][a] + g[a][k]) + (tr if k == a else 0)) * wt for k in range(3)], -1)
            v = torch.einsum("erqpc,rz->ezqpc", s * (2 / self.h[a]), f[3 * a + 2])
            v = torch.einsum("ezqpc,qy->ezypc", v, f[3 * a + 1])
            out = out + torch.einsum("ezypc,px->ezyxc", v, f[3 * a])
        return out.reshape(len(cells), q ** 3, 3)

    def K(self, x):
        x = x * self.free
        y = torch.zeros(len(x) // 3, 3, dtype=F64, device="cuda")
        jobs = [(a, self.c["depth"], on) for a, on in self.chunks]
        jobs += [(self.solid[k:k + 20000], 0, None) for k in range(0, len(self.solid), 20000)]
        for cells, depth, on in jobs:
            y.index_add_(0, self.nodes[cells].flatten(), self._cells(x, cells, depth, on).reshape(-1, 3))
        return y.reshape(-1) * self.free

    def dense(self):
        idx = torch.nonzero(self.free).flatten()
        A = torch.zeros((len(idx), len(idx)), dtype=F64, device="cuda")
        for j, i in enumerate(idx.tolist()):
            e = torch.zeros(len(self.free), dtype=F64, device="cuda")
            e[i] = 1
            A[:, j] = self.K(e)[idx]
        return idx, (A + A.T) / 2

    def S(self, r, idx, A):
        """Sum over the vertices of the pseudo inverses (eigenvalues above 1e-13 of the largest) of their patches."""
        p, z = self.p, torch.zeros_like(r)
        where = torch.full((len(self.free),), -1, dtype=torch.int64, device="cuda")
        where[idx] = torch.arange(len(idx), device="cuda")
        m = [torch.arange(k, device="cuda") for k in self.M]
        for v in np.ndindex(self.n[0] + 1, self.n[1] + 1, self.n[2] + 1):
            a = [m[i][max(0, p * v[i] - p + 1):p * v[i] + p] for i in range(3)]
            nd = a[0][None, None, :] + self.M[0] * (a[1][None, :, None] + self.M[1] * a[2][:, None, None])
            g = (3 * nd.reshape(-1, 1) + torch.arange(3, device="cuda")).flatten()
            g = g[self.free[g]]
            if not len(g):
                continue
            lam, V = torch.linalg.eigh(A[where[g]][:, where[g]])
            inv = torch.where(lam > 1e-13 * lam[-1], 1 / lam, torch.zeros_like(lam))
            z[g] += V @ (inv * (V.T @ r[g]))
        return z

    def prolong(self, cells):
        """P: a free vertex DOF gets an eighth of the sum of the cells around it; its transpose restricts."""
        v = torch.zeros((self.M[2], self.M[1], self.M[0], 3), dtype=F64, device="cuda")
        x = cells.view(3, self.n[2], self.n[1], self.n[0]).permute(1, 2, 3, 0)
        e = [self.p * k for k in self.n]
        for i in range(8):
            o = [self.p * ((i >> a) & 1) for a in range(3)]
            v[o[2]:o[2] + e[2]:self.p, o[1]:o[1] + e[1]:self.p, o[0]:o[0] + e[0]:self.p] += x / 8
        return v.reshape(-1) * self.free

    def restrict(self, y):
        v = (y * self.free).view(self.M[2], self.M[1], self.M[0], 3)
        e = [self.p * k for k in self.n]
        s = 0
        for i in range(8):
            o = [self.p * ((i >> a) & 1) for a in range(3)]
            s = s + v[o[2]:o[2] + e[2]:self.p, o[1]:o[1] + e[1]:self.p, o[0]:o[0] + e[0]:self.p] / 8
        return s.permute(3, 0, 1, 2).reshape(-1)


def _unet_exact(c, seed):
    F = torch.nn.functional
    w = torch.from_numpy(_unet_weights(c, seed)).cuda()
    par, at = [], 0
    for ci, co in _channels(c):  # the layers use BF16 weights and FP32 biases
        par.append((w[at:at + 27 * ci * co].bfloat16().double().view(co, ci, 3, 3, 3).requires_grad_(),
                    w[at + 27 * ci * co:at + 27 * ci * co + co].double().requires_grad_()))
        at += 27 * ci * co + co
    x = _unet_input(c, seed).double().requires_grad_()
    L = c["levels"]
    conv = lambda k, v: F.conv3d(v, par[k][0], par[k][1], padding=1)  # noqa: E731
    skip, v = [], x
    with torch.set_grad_enabled(c["kind"] == "unet_train"), torch.backends.cudnn.flags(enabled=False):
        for l in range(L):
            if l:
                v = F.avg_pool3d(v, 2)
            v = F.relu(conv(2 * l + 1, F.relu(conv(2 * l, v))))
            skip.append(v)
        for k, l in enumerate(range(L - 2, -1, -1)):
            v = torch.cat([F.interpolate(v, scale_factor=2, mode="nearest"), skip[l]], 1)
            v = F.relu(conv(2 * L + 2 * k + 1, F.relu(conv(2 * L + 2 * k, v))))
        out = conv(len(par) - 1, v)
        if c["kind"] == "unet_fwd":
            return {"out": out.detach()}
        g = _normal(seed, out.numel(), F32, 3).view(out.shape) / out.numel()
        out.backward(g.double())
    return {"out": out.detach(), "din": x.grad, "grad": torch.cat([t.grad.flatten() for pair in par for t in pair])}


def exact(case, seed):
    c = case
    if c["kind"].startswith("unet"):
        return _unet_exact(c, seed)
    if c["kind"] == "mlhp":  # the system and the factors are inputs here: what the set-up calls gave the program
        h = _plan(c)
        x, r = (_normal(seed, len(h.rhs), which=k).cpu().numpy() for k in (0, 1))
        z = h.jac * r
        for b, f in zip(h.blocks, h.factors):
            z[b] += f @ r[b]
        return {"Kx": h.K @ x, "Sr": z}
    if c["kind"] in ("k", "ops"):
        e = _Exact(c)
        out = {"Kx": e.K(_smooth(c, seed))}
        if c["kind"] == "ops":
            small = int(e.free.sum()) <= 4000
            out["Sr"] = e.S(_smooth(c, 31 * seed) * e.free, *e.dense()) if small else None
        return out
    if c["kind"] == "pcg":
        e = _Exact(c)
        if int(e.free.sum()) > 4000:
            return None
        idx, A = e.dense()
        u = torch.zeros(len(e.free), dtype=F64, device="cuda")
        u[idx] = torch.linalg.solve(A, _load(c, seed)[idx])
        return {"u": u}
    if c["kind"] == "coarse":
        e = _Exact(c)
        x = _normal(seed, 3 * c["nx"] * c["ny"] * c["nz"], F32).double()
        return {"KHx": e.restrict(e.K(e.prolong(x))), "Vf": None}
    return None  # S with its thousands of eigen-decompositions, and solves that end at a tolerance
