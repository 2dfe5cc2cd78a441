"""What a user of the GGEM slit library has it do, as timed cases.

A case names a workload family, its sizes and the options of the plan; `prepare`
builds the inputs and the plan a program keeps, `run` makes one call (or the
calls of one step) through the public binding, `exact` evaluates the same
discrete operator in FP64 torch without the library.

kinds
  single, double   one layer operator at the mesh nodes (the matvec of Sec. 3.4 / 3.5)
  layers           both, one step of the matvec benchmark
  points           velocity and stress of point forces at free targets
  solve            one time step's Fredholm solve: the moved mesh is set, then (I + kappa/4pi D) q = b
  train            one epoch of the learned warm start's network
"""
import math

import numpy as np
import torch

from paper_1109_6587_gb300 import ggem
from paper_1109_6587_gb300 import workloads as W

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def _layer(name, kind, shape, capsules, level, box, precision, quadrature="element",
           offgrid="lagrange"):
    Lx, W_, Lz, Nx, Ny, Nz = box
    return {"name": name, "kind": kind, "shape": shape, "capsules": capsules, "level": level,
            "radius": 0.97 if capsules == 1 else 1.0,
            "Lx": Lx, "W": W_, "Lz": Lz, "Nx": Nx, "Ny": Ny, "Nz": Nz,
            "precision": precision, "quadrature": quadrature, "offgrid": offgrid}


_BOX_1 = (8.0, 4.0, 8.0, 32, 33, 32)            # workloads.box_single_sphere
_BOX_8 = (16.0, 6.0, 16.0, 32, 33, 32)          # the learned part's small suspension
_BOX_TRAIN = (20.0, 10.0, 20.0, 64, 65, 64)     # workloads.box_training
_BOX_100 = (40.0, 10.0, 40.0, 128, 65, 128)     # workloads.box_100_capsules
_BOX_4000 = (150.0, 30.0, 150.0, 512, 129, 512)  # workloads.box_rbc_4000


def listed():
    return [
        # one 162-node capsule, plain FP64, nodal sources: the smallest configuration, all
        # launches and latency (validation runs, single-particle mobility)
        _layer("capsule1_single_fp64_nodal", "single", "sphere", 1, 2, _BOX_1, "fp64", "nodal"),
        # a few coarse capsules, native FP64 element rule: what small reference runs use
        _layer("capsules8_double_fp64", "double", "sphere", 8, 2, _BOX_8, "fp64"),
        # the same small suspension in mixed precision: the matvec of the learned part's test solves
        _layer("capsules8_double_mixed", "double", "sphere", 8, 2, _BOX_8, "mixed"),
        # flow field (velocity and stress) of a suspension's nodal forces sampled at scattered
        # points, an odd number of them
        dict(_layer("points_field_mixed", "points", "sphere", 48, 2, _BOX_TRAIN, "mixed", "nodal"),
             targets=10007),
        # the 100-capsule suspension (64,200 nodes), the ordinary size: both layer operators in
        # mixed precision ...
        _layer("capsules100_single_mixed", "single", "sphere", 100, 3, _BOX_100, "mixed"),
        _layer("capsules100_double_mixed", "double", "sphere", 100, 3, _BOX_100, "mixed"),
        # ... the FP64-accurate operator that gives a mixed solve its true residuals ...
        _layer("capsules100_double_emulated", "double", "sphere", 100, 3, _BOX_100,
               "fp64_emulated"),
        # ... the spectrally accurate off-grid evaluation ...
        _layer("capsules100_double_spectral", "double", "sphere", 100, 3, _BOX_100, "mixed",
               offgrid="spectral"),
        # ... and a whole Fredholm solve as each time step makes one: moved mesh, then GMRES to 1e-6
        _layer("capsules100_solve_mixed", "solve", "sphere", 100, 3, _BOX_100, "mixed"),
        # the same slit filled to volume fraction 0.1: many neighbours per node
        _layer("capsules382_double_mixed", "double", "sphere", 382, 3, _BOX_100, "mixed"),
        # the largest configuration, 4000 biconcave cells (2,568,000 nodes): one step of the
        # matvec benchmark, single and double layer
        _layer("rbc4000_layers_mixed", "layers", "rbc", 4000, 3, _BOX_4000, "mixed"),
        # training the learned warm start: one epoch over the samples of a small suspension series
        {"name": "train_epoch", "kind": "train", "samples": 65536, "batch": 2048},
    ]


def draw(rng):
    """One more case of the same ranges: slits of 32 to 256 grid intervals, 1 to about
    1000 capsules, every precision, quadrature and off-grid mode."""
    kind = rng.choice(["single", "double", "single", "double", "layers", "points", "solve",
                       "train"])
    if kind == "train":
        return {"kind": "train", "samples": int(2 ** rng.uniform(12, 17)) | 1,
                "batch": rng.choice([512, 1000, 2048])}
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64_emulated"])
    if kind == "solve":
        precision = "mixed"
    quadrature = rng.choice(["element", "element", "nodal"])
    if kind == "points":
        quadrature = "nodal"
    offgrid = rng.choice(["lagrange", "lagrange", "lagrange", "spectral"])
    big = precision == "mixed"
    Nx = rng.choice([32, 64, 128, 256] if big and kind != "solve" else [32, 64])
    Nz = rng.choice([Nx, Nx, max(32, Nx // 2)])
    Ny = rng.choice([33, 49, 65, 97] if Nx > 32 else [33, 49])
    spacing = rng.uniform(0.25, 0.5)
    W_ = rng.uniform(0.9, 1.1) * 0.5 * spacing * (Ny - 1)
    W_ = max(W_, 3.0)
    box = (spacing * Nx, W_, spacing * Nz, Nx, Ny, Nz)
    # capsules: log-uniform up to a volume fraction of 0.15
    most = int(0.15 * box[0] * box[1] * box[2] / (4.0 / 3.0 * math.pi))
    most = max(1, min(most, 1000 if big else 60))
    n = max(1, int(round(math.exp(rng.uniform(0.0, math.log(most))))))
    level = rng.choice([2, 3])
    shape = rng.choice(["sphere", "sphere", "rbc"])
    if precision == "fp64" and quadrature == "element":
        level, n = 2, min(n, 24)
    c = _layer("", kind, shape, n, level, box, precision, quadrature, offgrid)
    c["radius"] = round(rng.uniform(0.9, 1.0), 4)   # no node pair exactly at r_cut
    del c["name"]
    if kind == "solve":
        c["quadrature"] = "element"
    if kind == "points":
        c["targets"] = int(math.exp(rng.uniform(math.log(100), math.log(60000)))) | 1
    # no more than the largest listed case costs: a pair in double or float-pair arithmetic
    # takes tens of FP32 ones, a solve some FP64-accurate residuals
    heavy = 4.0 if kind == "solve" else {"mixed": 1.0, "fp64_emulated": 20.0, "fp64": 60.0}[
        precision]
    while c["capsules"] > 1 and heavy * work(c)["flops"] > 6e12:
        c["capsules"] = int(0.7 * c["capsules"])
    return c


# ------------------------------------------------------------------ inputs
def _suspension(case, seed):
    box = W.Box(Lx=case["Lx"], Lz=case["Lz"], W=case["W"], y0=-0.5 * case["W"], Nx=case["Nx"],
                Ny=case["Ny"], Nz=case["Nz"])
    rng = np.random.default_rng(seed)
    a = case["radius"]
    centres = W.place_centres(case["capsules"], box, a, rng)
    if case["shape"] == "rbc":
        v, t = W.rbc_mesh(case["level"], a)
        rot = W.random_rotations(len(centres), rng)
        v = np.einsum("pij,nj->pni", rot, v)
    else:
        v, t = W.icosphere(case["level"])
        v = np.broadcast_to(a * v, (len(centres),) + v.shape)
    nb = v.shape[1]
    x = (centres[:, None, :] + v).reshape(-1, 3)
    tri = (t[None, :, :] + nb * np.arange(len(centres))[:, None, None]).reshape(-1, 3)
    part = np.repeat(np.arange(len(centres), dtype=np.int32), nb)
    return W.Suspension(box, np.ascontiguousarray(x), tri.astype(np.int32), part, centres, a)


def _inputs(case, seed):
    """The arrays of a case: suspension, density / forces, targets."""
    s = _suspension(case, seed)
    rng = np.random.default_rng([seed, 1])
    n = len(s.x)
    d = {"susp": s, "q": rng.standard_normal((n, 3))}
    if case["kind"] == "points":
        m, b = case["targets"], s.box
        xt = rng.uniform(0.0, 1.0, (m, 3)) * [b.Lx, 0.98 * b.W, b.Lz]
        xt[:, 1] += b.y0 + 0.01 * b.W
        d["xt"] = xt
    if case["kind"] == "solve":
        d["kappa"], d["b"] = W.bie_rhs(s, lam=5.0, seed=seed)
    return d


def _train_inputs(case, seed):
    rng = np.random.default_rng(seed)
    F = rng.standard_normal((case["samples"], 12))
    A = rng.standard_normal((12, 3)) / 4.0
    return F, np.tanh(F @ A) + 0.05 * rng.standard_normal((case["samples"], 3))


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


def prepare(case, seed):
    if case["kind"] == "train":
        F, T = _train_inputs(case, seed)
        P = ggem.Plan.for_box(W.box_single_sphere(), precision="mixed", max_points=1024,
                              max_tris=1024)
        return {"kind": "train", "P": P, "F": F, "T": T, "batch": case["batch"], "seed": seed}
    d = _inputs(case, seed)
    s = d["susp"]
    n = len(s.x)
    P = ggem.Plan.for_box(s.box, precision=case["precision"], quadrature=case["quadrature"],
                          offgrid=case["offgrid"], max_points=max(n, case.get("targets", 0)),
                          max_tris=len(s.tri))
    st = {"kind": case["kind"], "P": P, "x": _dev(s.x), "q": _dev(d["q"])}
    if case["kind"] == "points":
        m = case["targets"]
        st["xt"] = _dev(d["xt"])
        st["u"] = torch.empty((m, 3), dtype=torch.float64, device=DEV)
        st["s"] = torch.empty((m, 6), dtype=torch.float64, device=DEV)
        return st
    st["tri"] = _dev(s.tri)
    st["w"], st["v"] = torch.empty_like(st["q"]), torch.empty_like(st["q"])
    P.mesh_set(st["x"], st["tri"])
    if case["kind"] == "solve":
        st["kappa"], st["b"] = _dev(d["kappa"]), _dev(d["b"])
        # the workspace and the FP64 twin that a time-stepping program's plan holds from its
        # first step on (no iteration is made)
        P.bie_solve(st["kappa"], st["b"], tol=1e-6, maxit=0)
    return st


def run(state):
    P, kind = state["P"], state["kind"]
    if kind == "train":
        loss = P.mlp_train(state["F"], state["T"], init=True, seed=state["seed"], epochs=1,
                           batch=state["batch"], lr=1e-3)
        return {"loss": float(loss), "model": P.mlp_save()}
    if kind == "points":
        u, s = P.point_forces(state["x"], state["q"], state["xt"], want_u=True, want_sigma=True,
                              u=state["u"], sigma=state["s"])
        return {"u": u, "sigma": s}
    if kind == "solve":
        P.mesh_set(state["x"], state["tri"])
        q, _, _, _ = P.bie_solve(state["kappa"], state["b"], tol=1e-6)
        return {"q": q}
    out = {}
    if kind != "double":
        out["w"] = P.single_layer(state["q"], state["w"])
    if kind != "single":
        out["v"] = P.double_layer(state["q"], state["v"])
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def _alpha_rcut(case):
    h = max(case["Lx"] / case["Nx"], case["W"] / (case["Ny"] - 1), case["Lz"] / case["Nz"])
    return 1.0 / (2.0 * h), 8.0 * h


def _mesh_size(case):
    m1 = 20 * 4 ** case["level"]
    n1 = m1 // 2 + 2
    return case["capsules"] * n1, case["capsules"] * m1, n1, m1


def work(case):
    """Inputs read once and results written once; the local pairs within r_cut (from the
    densities of the node's own capsule and of the suspension) and the global part's spread,
    transforms and interpolation."""
    if case["kind"] == "train":
        n = case["samples"]
        weights = 12 * 128 + 2 * 128 * 128 + 128 * 3
        return {"bytes": 15.0 * 8 * n, "flops": 6.0 * weights * n}
    N, M, n1, m1 = _mesh_size(case)
    _, rc = _alpha_rcut(case)
    vol = case["Lx"] * case["W"] * case["Lz"]
    ball = 4.0 / 3.0 * math.pi * rc ** 3
    own = min(1.0, (rc / (2.0 * case["radius"])) ** 2)

    def pairs(nt, src1, src, own_share):
        return nt * (own_share * src1 + (src - src1) / vol * ball)

    grid = case["Nx"] * case["Ny"] * case["Nz"]
    spread = N * min(1.0, ball / vol) * grid * 10.0
    fft = 5.0 * grid * math.log2(case["Nx"] * case["Nz"])
    cheb = 2.0 * grid * case["Ny"]

    def layer(double):
        k = 6 if double else 3
        f = spread + (3 + k) * (fft + cheb) + N * 125 * 2.0 * k
        if case["quadrature"] == "element":
            f += pairs(N, 16 * m1, 16 * M, own) * (72.0 if double else 52.0)
        else:
            f += pairs(N, n1, N, own) * (72.0 if double else 52.0)
        return f, N * 72.0 + (M * 12.0)

    if case["kind"] == "points":
        m = case["targets"]
        f = pairs(m, 0, N, 0.0) * 110.0 + spread + 12 * (fft + cheb) + m * 125 * 18.0
        return {"bytes": N * 48.0 + m * 96.0, "flops": f}
    if case["kind"] == "solve":
        f, b = layer(True)
        return {"bytes": 2 * b, "flops": 14 * f}     # about 14 operator applications
    both = [layer(k) for k in ((False, True) if case["kind"] == "layers"
                               else (case["kind"] == "double",))]
    return {"bytes": sum(b for _, b in both), "flops": sum(f for f, _ in both)}


# ------------------------------------------------------------------ the same in FP64 torch
_PI = math.pi
_SP = math.sqrt(math.pi)


def _kernel_terms(al, d, r2, g, n, layer):
    """sum over the last-but-one axis of G^l g (layer 0), T^l g . n (layer 1) or the six
    components of T^l g (layer 2); d [..., S, 3], r2 [..., S] (0 where the pair is left out)."""
    on = r2 > 0
    r2 = torch.where(on, r2, torch.ones_like(r2))
    r = torch.sqrt(r2)
    ec = torch.where(on, torch.erfc(al * r), torch.zeros_like(r))
    ex = torch.where(on, torch.exp(-al * al * r2), torch.zeros_like(r))
    xg = (d * g).sum(-1)
    if layer == 0:
        A = ec / r - 2 * al / _SP * ex
        B = (ec / r ** 3 + 2 * al / _SP * ex / r2) * xg
        return (A[..., None] * g + B[..., None] * d).sum(-2)
    D = -6 * ec / r ** 5 - 12 * al / _SP * ex / r2 ** 2 - 8 * al ** 3 / _SP * ex / r2
    E = 4 * al ** 3 / _SP * ex
    if layer == 1:
        xn, gn = (d * n).sum(-1), (g * n).sum(-1)
        return ((D * xg * xn + E * gn)[..., None] * d + (E * xn)[..., None] * g
                + (E * xg)[..., None] * n).sum(-2)
    out = []
    for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)):
        t = D * xg * d[..., i] * d[..., j] + E * (g[..., j] * d[..., i] + g[..., i] * d[..., j])
        if i == j:
            t = t + E * xg
        out.append(t.sum(-1))
    return torch.stack(out, -1)


def _local(case, al, rc, xt, nt, xs, gs, layer, skip=None, block=1 << 25):
    """Local sums at targets xt [m, 3] from sources xs [S, 3] with strengths gs, the sources
    gathered per group of nearby targets; skip(rows, cols) marks pairs left out."""
    L = torch.tensor([case["Lx"], 0.0, case["Lz"]], dtype=torch.float64, device=DEV)
    per = torch.tensor([case["Lx"], 1e300, case["Lz"]], dtype=torch.float64, device=DEV)
    m = xt.shape[0]
    out = torch.zeros((m, 6 if layer == 2 else 3), dtype=torch.float64, device=DEV)
    # targets grouped by boxes of about one r_cut
    w = torch.floor(torch.stack([torch.remainder(xt[:, 0], case["Lx"]), xt[:, 1] + case["W"],
                                 torch.remainder(xt[:, 2], case["Lz"])], 1) / rc).long()
    key = (w[:, 0] * 4096 + w[:, 1]) * 4096 + w[:, 2]
    order = torch.argsort(key)
    bounds = torch.unique_consecutive(key[order], return_counts=True)[1].cumsum(0).tolist()
    lo = 0
    for hi in bounds:
        rows = order[lo:hi]
        lo = hi
        c = (w[rows[0]].double() + 0.5) * rc
        c[1] -= case["W"]
        dc = xs - c
        dc = dc - L * torch.round(dc / per)
        near = torch.nonzero((dc.abs() < 1.5 * rc + 1e-9).all(1))[:, 0]
        if len(near) == 0:
            continue
        step = max(1, block // len(near))
        for a in range(0, len(rows), step):
            rr = rows[a:a + step]
            d = xt[rr][:, None, :] - xs[near][None]
            d = d - L * torch.round(d / per)
            r2 = (d * d).sum(-1)
            keep = (r2 > 0) & (r2 < rc * rc)
            if skip is not None:
                keep = keep & ~skip(rr, near)
            r2 = torch.where(keep, r2, torch.zeros_like(r2))
            n = nt[rr][:, None, :] if nt is not None else None
            out[rr] = _kernel_terms(al, d, r2, gs[near][None], n, layer)
    return out


def _geometry(x, tri):
    e2, e3 = x[tri[:, 1]] - x[tri[:, 0]], x[tri[:, 2]] - x[tri[:, 0]]
    c = torch.linalg.cross(e2, e3)
    a2 = c.norm(dim=1)
    Ab = torch.zeros(len(x), dtype=x.dtype, device=x.device)
    nb = torch.zeros_like(x)
    for v in range(3):
        Ab.index_add_(0, tri[:, v], a2 / 6.0)
        nb.index_add_(0, tri[:, v], 0.5 * c)
    return 0.5 * a2, c / a2[:, None], Ab, nb / nb.norm(dim=1, keepdim=True)


def _element_local(case, al, rc, x, tri, q, layer):
    """The 4 x 4 collapsed Gauss rule on every triangle without the node, the polar rule on
    the triangles around it."""
    Ak, nk, _, nb = _geometry(x, tri)
    t, w = np.polynomial.legendre.leggauss(4)
    t, w = 0.5 * (t + 1.0), 0.5 * w
    eta = np.repeat(t, 4)
    s = np.tile(t, 4)
    xi = (1.0 - eta) * s
    wq = np.repeat(w, 4) * np.tile(w, 4) * (1.0 - eta)
    phi = _dev(np.stack([1.0 - xi - eta, xi, eta], 1))                     # [16, 3]
    X, Q = x[tri], q[tri]
    xs = torch.einsum("av,mvc->mac", phi, X).reshape(-1, 3)
    gs = (torch.einsum("av,mvc->mac", phi, Q) * (_dev(wq)[None, :] * 2 * Ak[:, None])[..., None])
    own = torch.arange(len(tri), device=DEV).repeat_interleave(16)

    def skip(rows, cols):
        v = tri[own[cols]]                                               # [S, 3]
        return (v[None] == rows[:, None, None]).any(-1)

    out = _local(case, al, rc, x, nb, xs, gs.reshape(-1, 3), layer, skip)
    th = 0.5 * _PI * t
    rmax = 1.0 / (np.cos(th) + np.sin(th))
    rho = rmax[:, None] * t[None, :]                                     # [angle, radius]
    pxi, pet = rho * np.cos(th)[:, None], rho * np.sin(th)[:, None]
    pw = 0.5 * _PI * w[:, None] * rmax[:, None] * w[None, :] * rho
    pxi, pet, pw = (_dev(v.ravel()) for v in (pxi, pet, pw))
    for v in range(3):
        i1, i2, i3 = tri[:, v], tri[:, (v + 1) % 3], tri[:, (v + 2) % 3]
        e2, e3 = x[i2] - x[i1], x[i3] - x[i1]
        d = -(pxi[None, :, None] * e2[:, None] + pet[None, :, None] * e3[:, None])
        p1 = 1.0 - pxi - pet
        g = (p1[None, :, None] * q[i1][:, None] + pxi[None, :, None] * q[i2][:, None]
             + pet[None, :, None] * q[i3][:, None]) * (pw[None, :] * 2 * Ak[:, None])[..., None]
        n = p1[None, :, None] * nk[:, None] + (pxi + pet)[None, :, None] * nb[i1][:, None]
        r2 = (d * d).sum(-1)
        r2 = torch.where(r2 < rc * rc, r2, torch.zeros_like(r2))
        out.index_add_(0, i1, _kernel_terms(al, d, r2, g, n, layer))
    return out


def _cheb(Ny):
    N = Ny - 1
    n = np.arange(Ny)
    cb = np.ones(Ny)
    cb[0] = cb[N] = 2.0
    c = np.cos(_PI * ((n[:, None] * n[None, :]) % (2 * N)) / N)
    fwd = 2.0 / (N * cb[:, None] * cb[None, :]) * c
    D = np.zeros((Ny, Ny))
    for i in range(Ny):
        for m in range(i + 1, Ny, 2):
            D[i, m] = 2.0 * m / (2.0 if i == 0 else 1.0)
    return fwd, c, D


def _global(case, al, rc, xs, g, stress):
    """Chebyshev-Fourier coefficients [c, Ny, Nz, Nx] of the global velocity (3) and, with
    stress, of the stress (6): spread, wall data, per-mode tau solves."""
    Nx, Ny, Nz = case["Nx"], case["Ny"], case["Nz"]
    Lx, Lz, Wd = case["Lx"], case["Lz"], case["W"]
    y0 = -0.5 * Wd
    dx, dz = Lx / Nx, Lz / Nz
    yj = _dev(y0 + 0.5 * Wd * (1.0 + np.cos(_PI * np.arange(Ny) / (Ny - 1))))
    f = torch.zeros((3, Ny * Nz * Nx), dtype=torch.float64, device=DEV)
    R = int(math.ceil(max(rc / dx, rc / dz))) + 1
    o = torch.arange(-R, R + 2, device=DEV)
    step = max(1, (1 << 25) // (len(o) ** 2 * Ny))
    for a in range(0, len(xs), step):
        x = xs[a:a + step]
        xw, zw = torch.remainder(x[:, 0], Lx), torch.remainder(x[:, 2], Lz)
        ix = torch.floor(xw / dx).long()[:, None] + o
        iz = torch.floor(zw / dz).long()[:, None] + o
        r2 = ((ix * dx - xw[:, None]) ** 2)[:, None, None, :] \
            + ((iz * dz - zw[:, None]) ** 2)[:, None, :, None] \
            + ((yj[None] - x[:, 1:2]) ** 2)[:, :, None, None]
        rho = torch.where(r2 < rc * rc, al ** 3 / _PI ** 1.5 * torch.exp(-al * al * r2)
                          * (2.5 - al * al * r2), torch.zeros_like(r2))
        idx = ((torch.arange(Ny, device=DEV)[None, :, None, None] * Nz
                + torch.remainder(iz, Nz)[:, None, :, None]) * Nx
               + torch.remainder(ix, Nx)[:, None, None, :]).reshape(-1)
        for c in range(3):
            f[c].index_add_(0, idx, -(rho * g[a:a + step, c][:, None, None, None]).reshape(-1))
    f = f.reshape(3, Ny, Nz, Nx)
    gx, gz = torch.arange(Nx, device=DEV) * dx, torch.arange(Nz, device=DEV) * dz
    walls = []
    for y in (y0, y0 + Wd):
        zz, xx = torch.meshgrid(gz, gx, indexing="ij")
        xt = torch.stack([xx.reshape(-1), torch.full((Nx * Nz,), y, dtype=torch.float64,
                                                     device=DEV), zz.reshape(-1)], 1)
        u = _local(case, al, rc, xt, None, xs, g, 0) / (8 * _PI)
        walls.append(-u.T.reshape(3, Nz, Nx))
    fwd, inv, Dm = _cheb(Ny)
    fwd, D = _dev(fwd), _dev(Dm) * (2.0 / Wd)
    Fh = torch.einsum("nj,cjzx->zxcn", fwd.to(torch.complex128),
                      torch.fft.fft2(f) / (Nx * Nz))
    Gb, Gt = (torch.fft.fft2(v).permute(1, 2, 0) / (Nx * Nz) for v in walls)
    lx, mz = np.fft.fftfreq(Nx, 1.0 / Nx), np.fft.fftfreq(Nz, 1.0 / Nz)
    KZ, KX = np.meshgrid(2 * _PI * mz / Lz, 2 * _PI * lx / Lx, indexing="ij")
    MZ, LX = np.meshgrid(mz, lx, indexing="ij")
    k2 = KX ** 2 + KZ ** 2
    ok = (np.abs(LX) != Nx // 2) & (np.abs(MZ) != Nz // 2)
    nc = 9 if stress else 3
    out = torch.zeros((Nz, Nx, nc, Ny), dtype=torch.complex128, device=DEV)
    bot = _dev((-1.0) ** np.arange(Ny))
    top = torch.ones(Ny, dtype=torch.float64, device=DEV)
    D2 = D @ D
    cplx = lambda v: v.to(torch.complex128)  # noqa: E731

    def bc(r, b, t):
        r = r.clone()
        r[..., -2], r[..., -1] = b, t
        return r

    def solve(H, cols):
        """H real [M, Ny, Ny]; cols complex [M, k, Ny]."""
        k = cols.shape[1]
        B = torch.cat([cols.real, cols.imag], 1).transpose(1, 2)
        S = torch.linalg.solve(H, B).transpose(1, 2)
        return torch.complex(S[:, :k], S[:, k:])

    def stresses(u, v, w, p, ikx, ikz):
        Dc = cplx(D).T
        dU, dV, dW = u @ Dc, v @ Dc, w @ Dc
        return [-p + 2 * ikx * u, ikx * v + dU, ikz * u + ikx * w, -p + 2 * dV, ikz * v + dW,
                -p + 2 * ikz * w]

    sel = np.argwhere(ok & (k2 > 0))
    for a in range(0, len(sel), 2048):
        zi, xi = (torch.as_tensor(v, device=DEV) for v in sel[a:a + 2048].T)
        kx, kz = _dev(KX)[zi, xi], _dev(KZ)[zi, xi]
        ikx, ikz = 1j * cplx(kx)[:, None], 1j * cplx(kz)[:, None]
        M = len(kx)
        H = D2[None] - (kx * kx + kz * kz)[:, None, None] * torch.eye(Ny, dtype=torch.float64,
                                                                    device=DEV)
        H[:, -2], H[:, -1] = bot, top
        F = Fh[zi, xi]
        Dc = cplx(D).T
        zero = torch.zeros((M, Ny), dtype=torch.complex128, device=DEV)
        rp = -(ikx * F[:, 0] + F[:, 1] @ Dc + ikz * F[:, 2])
        Pm = solve(H, torch.stack([bc(rp, 0, 0), bc(zero, 1, 0), bc(zero, 0, 1)], 1))
        cols = []
        for c in range(3):
            fs = F if c == 0 else torch.zeros_like(F)
            gb = Gb[zi, xi] if c == 0 else torch.zeros((M, 3), dtype=torch.complex128, device=DEV)
            gt = Gt[zi, xi] if c == 0 else torch.zeros_like(gb)
            p = Pm[:, c]
            cols += [bc(fs[:, 0] + ikx * p, gb[:, 0], gt[:, 0]),
                     bc(fs[:, 1] + p @ Dc, gb[:, 1], gt[:, 1]),
                     bc(fs[:, 2] + ikz * p, gb[:, 2], gt[:, 2])]
        V = solve(H, torch.stack(cols, 1)).reshape(M, 3, 3, Ny)          # [mode, abc, uvw, n]
        div = ikx[:, None] * V[:, :, 0] + V[:, :, 1] @ Dc + ikz[:, None] * V[:, :, 2]
        at = torch.stack([div @ cplx(bot), div @ cplx(top)], 1)          # [mode, wall, abc]
        p12 = torch.linalg.solve(at[:, :, 1:], -at[:, :, :1])[:, :, 0]
        co = torch.cat([torch.ones((M, 1), dtype=torch.complex128, device=DEV), p12], 1)
        uvw = (co[:, :, None, None] * V).sum(1)
        p = (co[:, :, None] * Pm).sum(1)
        u, v, w = uvw[:, 0], uvw[:, 1], uvw[:, 2]
        res = [u, v, w] + (stresses(u, v, w, p, ikx, ikz) if stress else [])
        out[zi, xi] = torch.stack(res, 1)
    # k = 0
    H = D2.clone()
    H[-2], H[-1] = bot, top
    F, gb, gt = Fh[0, 0], Gb[0, 0], Gt[0, 0]
    uw = solve(H[None], torch.stack([bc(F[0], gb[0], gt[0]), bc(F[2], gb[2], gt[2])])[None])[0]
    v = torch.zeros(Ny, dtype=torch.complex128, device=DEV)
    v[0], v[1] = 0.5 * (gb[1] + gt[1]), 0.5 * (gt[1] - gb[1])
    G = -(0.5 * Wd) * F[1]
    p = torch.zeros_like(v)
    for n in range(1, Ny):
        p[n] = ((2.0 if n == 1 else 1.0) * G[n - 1] - (G[n + 1] if n + 1 < Ny else 0.0)) / (2.0 * n)
    for n in range(2, Ny, 2):
        p[0] = p[0] - p[n] / (1.0 - n * n)
    z0 = torch.zeros(1, dtype=torch.complex128, device=DEV)
    res = [uw[0], v, uw[1]] + (stresses(uw[0], v, uw[1], p, z0, z0) if stress else [])
    out[0, 0] = torch.stack(res)
    return out.permute(2, 3, 0, 1)                                       # [c, Ny, Nz, Nx]


def _at_targets(case, coef, xt):
    """The global field at the targets: 5-point Lagrange interpolation of its grid values, or
    its expansion itself."""
    Nx, Ny, Nz = case["Nx"], case["Ny"], case["Nz"]
    Lx, Lz, Wd = case["Lx"], case["Lz"], case["W"]
    y0 = -0.5 * Wd
    nc = coef.shape[0]
    out = torch.empty((len(xt), nc), dtype=torch.float64, device=DEV)
    _, inv, _ = _cheb(Ny)
    if case["offgrid"] == "spectral":
        # Re sum over k_x >= 0 with weight 2 (k_x > 0): the field is real
        half = coef[..., :Nx // 2].reshape(nc, Ny, -1)
        flat = half.permute(1, 0, 2).reshape(Ny, -1)
        flat = torch.cat([flat.real, flat.imag], 1)
        kx = 2 * _PI / Lx * torch.arange(Nx // 2, device=DEV, dtype=torch.float64)
        kz = 2 * _PI / Lz * _dev(np.fft.fftfreq(Nz, 1.0 / Nz))
        wx = torch.full((Nx // 2,), 2.0, dtype=torch.float64, device=DEV)
        wx[0] = 1.0
        step = max(1, (1 << 27) // flat.shape[1])
        for a in range(0, len(xt), step):
            x = xt[a:a + step]
            yb = (2.0 * (x[:, 1] - y0) / Wd - 1.0).clamp(-1, 1)
            T = torch.cos(torch.arange(Ny, device=DEV) * torch.arccos(yb)[:, None])
            S = T @ flat
            h = S.shape[1] // 2
            S = torch.complex(S[:, :h], S[:, h:]).reshape(len(x), nc, Nz, Nx // 2)
            ez = torch.exp(1j * (kz[None] * x[:, 2:3]))
            ex = torch.exp(1j * (kx[None] * x[:, 0:1])) * wx
            S = torch.einsum("tczx,tz->tcx", S, ez)
            out[a:a + step] = torch.einsum("tcx,tx->tc", S, ex).real
        return out
    field = torch.fft.ifft2(torch.einsum("jn,cnzx->cjzx", _dev(inv).to(torch.complex128), coef)
                            * (Nx * Nz)).real
    yj = _dev(y0 + 0.5 * Wd * (1.0 + np.cos(_PI * np.arange(Ny) / (Ny - 1))))
    off = torch.arange(-2, 3, device=DEV)

    def lagrange(nodes, t):
        Lw = torch.ones_like(nodes)
        for p in range(5):
            for q in range(5):
                if q != p:
                    Lw[:, p] *= (t - nodes[:, q]) / (nodes[:, p] - nodes[:, q])
        return Lw

    step = 1 << 14
    for a in range(0, len(xt), step):
        x = xt[a:a + step]
        ux, uz = x[:, 0] / (Lx / Nx), x[:, 2] / (Lz / Nz)
        i0, k0 = torch.round(ux), torch.round(uz)
        of = off.double().expand(len(x), 5).clone()
        wx, wz = lagrange(of, ux - i0), lagrange(of, uz - k0)
        ix = torch.remainder(i0.long()[:, None] + off, Nx)
        iz = torch.remainder(k0.long()[:, None] + off, Nz)
        jn = (x[:, 1:2] - yj[None]).abs().argmin(1)
        jy = (jn - 2).clamp(0, Ny - 5)[:, None] + torch.arange(5, device=DEV)
        wy = lagrange(yj[jy].clone(), x[:, 1])
        vals = field[:, jy[:, :, None, None], iz[:, None, :, None], ix[:, None, None, :]]
        out[a:a + step] = torch.einsum("cnabd,na,nb,nd->nc", vals, wy, wz, wx)
    return out


def exact(case, seed):
    if case["kind"] in ("train", "solve"):
        return None                 # rounding points of its own; many operator applications
    N, M, n1, m1 = _mesh_size(case)
    al, rc = _alpha_rcut(case)
    per_target = (16 * M if case["quadrature"] == "element" else N) * min(
        1.0, 27.0 * rc ** 3 / (case["Lx"] * case["W"] * case["Lz"]))
    modes = case["Nx"] * case["Nz"]
    cost = N * per_target * (2 if case["kind"] == "layers" else 1) + 4e3 * modes * case["Ny"]
    if case["offgrid"] == "spectral":
        cost += 6.0 * N * modes * case["Ny"] / 40.0
    if cost > 4e10 or case["Nx"] * case["Nz"] > 128 * 128:
        return None
    d = _inputs(case, seed)
    s = d["susp"]
    x, q = _dev(s.x), _dev(d["q"])
    if case["kind"] == "points":
        xt = _dev(d["xt"])
        ul = _local(case, al, rc, xt, None, x, q, 0) / (8 * _PI)
        sl = _local(case, al, rc, xt, None, x, q, 2) / (8 * _PI)
        gf = _at_targets(case, _global(case, al, rc, x, q, True), xt)
        return {"u": ul + gf[:, :3], "sigma": sl + gf[:, 3:]}
    tri = _dev(s.tri).long()
    _, _, Ab, nb = _geometry(x, tri)
    g = 8 * _PI * Ab[:, None] * q
    elem = case["quadrature"] == "element"
    out = {}
    gf = _at_targets(case, _global(case, al, rc, x, g, case["kind"] != "single"), x)
    if case["kind"] != "double":
        if elem:
            out["w"] = _element_local(case, al, rc, x, tri, q, 0) + gf[:, :3]
        else:
            out["w"] = (_local(case, al, rc, x, None, x, g, 0) / (8 * _PI) + gf[:, :3]
                        - 4 * al / _SP * g / (8 * _PI))
    if case["kind"] != "single":
        S = gf[:, 3:]
        vg = torch.stack([nb[:, 0] * S[:, 0] + nb[:, 1] * S[:, 1] + nb[:, 2] * S[:, 2],
                          nb[:, 0] * S[:, 1] + nb[:, 1] * S[:, 3] + nb[:, 2] * S[:, 4],
                          nb[:, 0] * S[:, 2] + nb[:, 1] * S[:, 4] + nb[:, 2] * S[:, 5]], 1)
        if elem:
            out["v"] = vg + _element_local(case, al, rc, x, tri, q, 1)
        else:
            out["v"] = vg + _local(case, al, rc, x, nb, x, g, 1) / (8 * _PI)
    return out
