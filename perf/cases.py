"""What this framework is asked to do, as cases to be timed.

Each case is one call of a user's program through the public entry points
(Plan, BatchPlan, UNet): field solves of the particle-in-cell cycle in their
forms (binary64 and mixed, one problem and a batch, annulus, composite domain,
stretched axial mesh), the azimuthal transforms, the steps before and after
the solve (deposit and projection, face field), and the learned warm start's
network (inference, and one gradient step).  Geometry and charge are those of
paper_2609_07172_gb300.workloads; the settings of the large solves are what
the autotuner picks for them.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2609_07172_gb300 import FP64, MIXED, BatchPlan, Plan, query, workloads as W
from paper_2609_07172_gb300.unet import UNet

R_IN, R_OUT, Z_LEN, PHI_Z0 = 0.02, 0.05, 0.03, 300.0     # the annulus of workloads.annulus
EPS0, E_CHARGE = 8.8541878128e-12, 1.602176634e-19
TOL = 1e-10                                              # the solves' relative residual
WEIGHT = 1e8                                             # macro-particle weight

# settings of a solve: as the autotuner reports them for the headline grid (fp64, mixed), the
# channel-plume domain and the stretched axial mesh; "default" leaves every option at its default
SETTINGS = {
    "default": {},
    "fp64": dict(pre_sweeps=2, post_sweeps=1, fmg=1),
    "mixed": dict(precision=MIXED, pre_sweeps=2, post_sweeps=2, inner_cycles=3, smooth_fused=1),
    "plume": dict(pre_sweeps=1, post_sweeps=2, fmg=1),
    "axial": dict(precision=MIXED, pre_sweeps=1, post_sweeps=1, inner_cycles=3, omega=1.2),
}


def listed():
    sizes = ",".join("%dx%dx%d" % (p.nr, p.ntheta, p.nz) for p, _ in W.uneven_batch(3))
    return [
        # the smallest solve, a test problem or a coarse scan of parameters: latency and launches
        dict(name="solve_tiny", kind="solve", nr=32, nt=16, nz=32, use="default", graph=True),
        # a solve out of the box on a grid that is no power of two: every option at its default
        dict(name="solve_ragged", kind="solve", nr=152, nt=32, nz=90, use="default", graph=False),
        # the field solve of every time step on the paper's grid, in binary64
        dict(name="solve_fp64", kind="solve", nr=512, nt=128, nz=400, use="fp64", graph=True),
        # the same in the mixed form
        dict(name="solve_mixed", kind="solve", nr=512, nt=128, nz=400, use="mixed", graph=True),
        # independent problems of uneven sizes in one plan (a study over grids)
        dict(name="batch_uneven", kind="batch", sizes=sizes, use="fp64", graph=True),
        # the channel-plume composite domain: patches, exposed faces, a dense coarsest solve
        dict(name="solve_plume", kind="plume", nr=256, nt=64, nz=192, use="plume", graph=True),
        # a mesh whose cells grow along the axis
        dict(name="solve_axial", kind="axial", nr=512, nt=128, nz=400, ratio=1.002, use="axial", graph=True),
        # charge to modes and modes to potential: diagnostics, and the transforms a caller's own iteration uses
        dict(name="transforms", kind="transforms", nr=512, nt=128, nz=400),
        # the electric field on the faces after every solve
        dict(name="face_field", kind="field", nr=512, nt=128, nz=400),
        # charge deposit of two cell-sorted species and its projection, before every solve
        dict(name="deposit", kind="deposit", nr=512, nt=128, nz=400, ppc=4, sort=True),
        # the learned warm start's network on all modes of a step
        dict(name="unet_infer", kind="unet", n=65, h=200, w=256, train=False),
        # one batch of its training: forward pass, loss and gradients
        dict(name="unet_train", kind="unet", n=16, h=200, w=256, train=True),
    ]


# ------------------------------------------------------------------ drawn cases
def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, cells, multiple=2):
    """nr, nt, nz of at most `cells` cells: nr even (or a multiple), nz any count."""
    while True:
        step = multiple * rng.choice((1, 2, 4))
        nr = max(16, int(_log(rng, 16, 512) / step + 0.5) * step)
        nt = rng.choice((8, 16, 32, 64, 128, 256))
        step = max(1, multiple // 2) * rng.choice((1, 2, 8))
        nz = max(12, int(_log(rng, 12, 400) / step + 0.5) * step)
        if nr * nt * nz <= cells and nr % multiple == 0:
            return nr, nt, nz


def _accepted(case):
    try:
        for p in _problems(case):
            query(p, **SETTINGS[case["use"]])
    except RuntimeError:          # refused: the coarsest level would be too large for the direct solve
        return False
    return True


def draw(rng):
    c1 = 512 * 128 * 400
    kind = rng.choice(("solve", "solve", "solve", "solve", "batch", "plume", "axial", "transforms", "field", "deposit",
                       "unet", "unet"))
    while True:
        if kind == "solve":
            nr, nt, nz = _grid(rng, c1)
            use = rng.choice(("default", "fp64", "mixed"))
            c = dict(kind=kind, nr=nr, nt=nt, nz=nz, use=use, graph=use != "default" or rng.random() < 0.5)
        elif kind == "batch":
            sizes = ["%dx%dx%d" % _grid(rng, c1 // 8) for _ in range(rng.randint(2, 16))]
            c = dict(kind=kind, sizes=",".join(sizes), use=rng.choice(("fp64", "mixed")), graph=True)
        elif kind == "plume":
            c = dict(kind=kind, nr=16 * rng.choice((2, 3, 4, 6, 8, 16)), nt=rng.choice((8, 16, 32, 64)),
                     nz=16 * rng.choice((2, 3, 4, 6, 12)), use=rng.choice(("plume", "default")), graph=True)
        elif kind == "axial":
            nr, nt, nz = _grid(rng, c1 // 2, 8)
            c = dict(kind=kind, nr=nr, nt=nt, nz=nz, ratio=1.0 + rng.uniform(-0.5, 0.5) / nz,
                     use=rng.choice(("axial", "fp64")), graph=True)
        elif kind in ("transforms", "field"):
            nr, nt, nz = _grid(rng, c1)
            return dict(kind=kind, nr=nr, nt=nt, nz=nz) if _accepted(
                dict(kind="solve", nr=nr, nt=nt, nz=nz, use="default")) else draw(rng)
        elif kind == "deposit":
            nr, nt, nz = _grid(rng, c1 // 4)
            c = dict(kind=kind, nr=nr, nt=nt, nz=nz, ppc=rng.randint(1, 12), sort=rng.random() < 0.75)
            if _accepted(dict(c, kind="solve", use="default")):
                return c
            continue
        else:
            train = rng.random() < 0.5
            w = rng.choice((32, 64, 128, 256, 8 * rng.randint(3, 32)))      # mostly the solver's powers of two
            h = 8 * int(_log(rng, 3, 25) + 0.5)
            return dict(kind=kind, n=rng.randint(1, 16) if train else rng.randint(1, 65), h=h, w=w, train=train)
        if _accepted(c):
            return c


# ------------------------------------------------------------------ inputs
def _axial_faces(nz, ratio):
    w = ratio ** np.arange(nz)
    return Z_LEN * np.r_[0.0, np.cumsum(w)] / w.sum()


def _problems(case):
    kind = case["kind"]
    if kind == "batch":
        return [W.annulus(*map(int, s.split("x"))) for s in case["sizes"].split(",")]
    size = (case["nr"], case["nt"], case["nz"])
    if kind == "plume":
        return [W.channel_plume(*size)]
    p = W.annulus(*size)
    return [p.with_z_faces(_axial_faces(p.nz, case["ratio"])) if kind == "axial" else p]


def _species(p, ppc, sort, gen):
    """One species' particles, `ppc` per cell, uniformly inside the cells, cell by cell or shuffled."""
    n = p.nr * p.ntheta * p.nz * ppc
    cell = torch.arange(n, device="cuda", dtype=torch.int32) // ppc
    if not sort:
        cell = cell[torch.randperm(n, device="cuda", generator=gen)]
    u = lambda: torch.rand(n, device="cuda", dtype=torch.float64, generator=gen)  # noqa: E731
    r = (u().add_(cell % p.nr)).mul_((R_OUT - R_IN) / p.nr).add_(R_IN)
    z = (u().add_(cell // (p.nr * p.ntheta))).mul_(Z_LEN / p.nz)
    a = (u().add_((cell // p.nr) % p.ntheta)).mul_(2.0 * math.pi / p.ntheta)
    return r, a, z


LAYERS = (("e0", 16, 16), ("e1", 16, 32), ("e2", 32, 64), ("b1", 64, 128), ("b2", 128, 64),
          ("d2", 128, 32), ("d1", 64, 16), ("d0", 32, 16), ("out", 16, 16))


def _network(case, seed):
    """Weights and biases of the trained network's size and scale, its input x (residual and shift
    channels of every mode) and a target."""
    gen = torch.Generator().manual_seed(1_000 + seed)
    weights = {}
    for name, cin, cout in LAYERS:
        w = torch.randn(9, cout, cin, generator=gen) * math.sqrt(2.0 / (9 * (3 if name == "e0" else cin)))
        b = 0.1 * torch.randn(cout, generator=gen)
        if name == "e0":
            w[:, :, 3:] = 0.0                     # the input's unused channels
        if name == "out":
            w[:, 2:, :] = 0.0                     # the output's unused channels
            b[2:] = 0.0
        weights[name] = (w, b)
    gen = torch.Generator("cuda").manual_seed(seed)
    n, h, w = case["n"], case["h"], case["w"]
    x = torch.zeros(n, h, w, 16, dtype=torch.bfloat16, device="cuda")
    x[..., :2] = torch.randn(n, h, w, 2, device="cuda", generator=gen).to(torch.bfloat16)
    x[..., 2] = torch.rand(n, 1, w, device="cuda", generator=gen).to(torch.bfloat16)
    y = torch.randn(n, h, w, 2, device="cuda", generator=gen)
    return weights, x, y


def prepare(case, seed):
    kind = case["kind"]
    if kind == "unet":
        weights, x, y = _network(case, seed)
        net = UNet(seed=0)
        net.load_state(weights)
        return dict(kind=kind, net=net, x=x, y=y, train=case["train"])
    probs = _problems(case)
    p = probs[0]
    if kind in ("solve", "plume", "axial"):
        return dict(kind=kind, plan=Plan(p, graph=case["graph"], **SETTINGS[case["use"]]), rho=W.rho_plasma_torch(p, seed),
                    phi=torch.empty(p.shape, dtype=torch.float64, device="cuda"))
    if kind == "batch":
        return dict(kind=kind, plan=BatchPlan(probs, graph=case["graph"], **SETTINGS[case["use"]]),
                    rhos=[W.rho_plasma_torch(q, 64 * seed + i) for i, q in enumerate(probs)],
                    phis=[torch.empty(q.shape, dtype=torch.float64, device="cuda") for q in probs])
    state = dict(kind=kind, plan=Plan(p))
    gen = torch.Generator("cuda").manual_seed(seed)
    if kind == "transforms":
        uhat = torch.randn(p.nz, p.nr, p.n_modes, 2, device="cuda", dtype=torch.float64, generator=gen)
        uhat *= (1.0 / (1.0 + torch.arange(p.n_modes, device="cuda", dtype=torch.float64)))[:, None]
        state.update(rho=W.rho_plasma_torch(p, seed), uhat=uhat)
    elif kind == "field":
        z = torch.linspace(PHI_Z0, 0.0, p.nz, device="cuda", dtype=torch.float64)
        state.update(phi=z[:, None, None] + 10.0 * torch.randn(p.shape, device="cuda", dtype=torch.float64, generator=gen))
    else:
        state.update(ions=_species(p, case["ppc"], case["sort"], gen), electrons=_species(p, case["ppc"], case["sort"], gen))
    return state


# ------------------------------------------------------------------ one pass
def run(s):
    kind = s["kind"]
    if kind == "unet":
        y = s["net"].forward(s["x"])
        if not s["train"]:
            return y
        loss = s["net"].loss_backward(s["y"])
        return {"loss": loss, "w": dict(s["net"].gw), "b": dict(s["net"].gb)}
    plan = s["plan"]
    if kind in ("solve", "plume", "axial"):
        phi, info = plan.solve(s["rho"], s["phi"], tol=TOL)
        return {"phi": phi, "status": info["status"]}
    if kind == "batch":
        phis, infos = plan.solve(s["rhos"], s["phis"], tol=TOL)
        return {"phis": phis, "status": [i["status"] for i in infos]}
    if kind == "transforms":
        return {"bhat": plan.forward(s["rho"]), "phi": plan.inverse(s["uhat"])}
    if kind == "field":
        return plan.face_field(s["phi"])
    ions = plan.deposit(*s["ions"], WEIGHT)
    electrons = plan.deposit(*s["electrons"], WEIGHT)
    rho = plan.project(ions, E_CHARGE)
    rho = plan.project(electrons, -E_CHARGE, rho, accumulate=True)
    return {"ions": ions, "electrons": electrons, "rho": rho}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "unet":
        px = {0: case["h"] * case["w"]}
        level = dict(e0=0, e1=1, e2=2, b1=3, b2=3, d2=2, d1=1, d0=0, out=0)
        macs = sum(9 * cin * cout * px[0] / 4 ** level[name] for name, cin, cout in LAYERS) * case["n"]
        weights = sum(9 * cin * cout + cout for _, cin, cout in LAYERS)
        io = case["n"] * px[0]
        if case["train"]:       # input and target in, weights in, gradients out; two more convolutions per layer
            return {"bytes": io * (16 * 2 + 2 * 4) + weights * (2 + 4), "flops": 3 * 2 * macs}
        return {"bytes": io * (16 * 2 + 16 * 4) + weights * 2, "flops": 2 * macs}
    if kind == "deposit":
        n = 2 * case["nr"] * case["nt"] * case["nz"] * case["ppc"]
        nodes = (case["nr"] + 1) * case["nt"] * (case["nz"] + 1)
        cells = case["nr"] * case["nt"] * case["nz"]
        return {"bytes": 8 * (3 * n + 2 * nodes + cells), "flops": 30 * n}
    total = {"bytes": 0, "flops": 0}
    for p in _problems(case):
        cells, modes = p.nr * p.ntheta * p.nz, p.nr * p.nz * p.n_modes
        fft = 2.5 * cells * math.log2(p.ntheta)
        if kind == "transforms":
            total["bytes"] += 2 * (8 * cells + 16 * modes)
            total["flops"] += 2 * fft
        elif kind == "field":
            total["bytes"] += 4 * 8 * cells
            total["flops"] += 6 * cells
        else:                   # two transforms; one application of the operator to check the result
            total["bytes"] += 2 * 8 * cells
            total["flops"] += 2 * fft + 18 * modes
    return total


# ------------------------------------------------------------------ the same in 64 bits, without this framework
def _faces(case, nr, nz):
    rf = np.array([R_IN + (R_OUT - R_IN) * a / nr for a in range(nr + 1)])
    zf = _axial_faces(nz, case["ratio"]) if case["kind"] == "axial" else np.arange(nz + 1) * (Z_LEN / nz)
    return rf, zf


def _geometry(rf, zf):
    """Cell centres, widths, and conductances per unit width: radial faces (nr + 1), axial faces (nz + 1)."""
    rc, zc = 0.5 * (rf[1:] + rf[:-1]), 0.5 * (zf[1:] + zf[:-1])
    gr = rf / np.diff(np.r_[rf[0], rc, rf[-1]])
    gz = 1.0 / np.diff(np.r_[zf[0], zc, zf[-1]])
    return rc, np.diff(rf), np.diff(zf), gr, gz


def _lambda(nt):
    da = 2.0 * math.pi / nt
    return 4.0 / da ** 2 * np.sin(np.pi * np.arange(nt // 2 + 1) / nt) ** 2


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda", dtype=torch.float64)


def _rhs(rho, rc, dr, dz):
    """Mode right-hand sides (nz, nm, nr) without wall terms: s rho_hat."""
    rhat = torch.fft.rfft(rho, dim=1) / rho.shape[1]
    return rhat * (_cuda(dz)[:, None, None] * _cuda(rc * dr)[None, None, :] / EPS0)


def _exact_annulus(case, rho, nr, nt, nz):
    """Direct solve: eigenvectors of the axial operator, one radial tridiagonal system per eigenvector and mode."""
    rc, dr, dz, gr, gz = _geometry(*_faces(case, nr, nz))
    b = _rhs(rho, rc, dr, dz)
    b[0, 0] += _cuda(PHI_Z0 * gz[0] * rc * dr)
    tz = np.diag(gz[:-1] + gz[1:]) - np.diag(gz[1:-1], 1) - np.diag(gz[1:-1], -1)
    iw = 1.0 / np.sqrt(dz)
    theta, q = np.linalg.eigh(tz * iw[:, None] * iw[None, :])
    v = _cuda(q * iw[:, None])                                              # v^T diag(dz) v = 1
    nm = nt // 2 + 1
    w = torch.view_as_real(b).permute(0, 2, 1, 3).reshape(nz, -1)           # (nz, nr nm 2)
    w = (v.T @ w).reshape(nz, nr, nm, 2)
    d = (_cuda(gr[:-1] + gr[1:])[None, :, None] + _cuda(theta)[:, None, None] * _cuda(rc * dr)[None, :, None]
         + _cuda(dr / rc)[None, :, None] * _cuda(_lambda(nt))[None, None, :])
    for i in range(1, nr):
        f = gr[i] / d[:, i - 1]
        d[:, i] -= gr[i] * f
        w[:, i] += f[..., None] * w[:, i - 1]
    w[:, -1] /= d[:, -1, :, None]
    for i in range(nr - 2, -1, -1):
        w[:, i] = (w[:, i] + gr[i + 1] * w[:, i + 1]) / d[:, i, :, None]
    u = (v @ w.reshape(nz, -1)).reshape(nz, nr, nm, 2)
    return torch.fft.irfft(torch.view_as_complex(u).permute(0, 2, 1), n=nt, dim=1, norm="forward")


def _exact_plume(case, rho, nr, nt, nz):
    """Direct solve row by row (block elimination along the axis), cells outside the domain as identities."""
    rc, dr, dz, gr, gz = _geometry(*_faces(case, nr, nz))
    act = np.zeros((nz, nr), dtype=bool)
    act[:nz // 2, nr // 4:nr // 2] = True
    act[nz // 2:] = True
    h = Z_LEN / nz
    half_w, half_e = (rc - 0.5 * dr) / (0.5 * dr), (rc + 0.5 * dr) / (0.5 * dr)   # centre to the cell's own r faces
    b = _rhs(rho, rc, dr, dz)
    b *= _cuda(act)[:, None, :]
    b[0, 0] += _cuda(PHI_Z0 * gz[0] * rc * dr * act[0])
    nm = nt // 2 + 1
    lam = _cuda(_lambda(nt))
    inv, up = [], []
    for k in range(nz):
        a = act[k]
        south = act[k - 1] if k > 0 else np.zeros(nr, dtype=bool)
        north = act[k + 1] if k < nz - 1 else np.zeros(nr, dtype=bool)
        diag = rc * dr * (np.where(south, 1.0 / h, 2.0 / h) + np.where(north, 1.0 / h, 2.0 / h))
        west, east = np.r_[False, a[:-1]], np.r_[a[1:], False]
        diag = diag + h * (np.where(west, gr[:-1], half_w) + np.where(east, gr[1:], half_e))
        m = np.diag(np.where(a, diag, 1.0))
        off = np.where(a[:-1] & a[1:], -h * gr[1:-1], 0.0)
        m = m + np.diag(off, 1) + np.diag(off, -1)
        s = _cuda(m)[None] + torch.diag_embed(lam[:, None] * _cuda(np.where(a, dr * h / rc, 0.0))[None])
        if k > 0:
            c = _cuda(np.where(a & south, rc * dr / h, 0.0))
            s = s - c[:, None] * inv[-1] * c[None, :]
            b[k] += c * torch.einsum("mij,mj->mi", inv[-1].to(b.dtype), b[k - 1])
            up.append(c)
        inv.append(torch.linalg.inv(s))
    u = torch.zeros_like(b)
    for k in range(nz - 1, -1, -1):
        r = b[k] + up[k] * u[k + 1] if k < nz - 1 else b[k]
        u[k] = torch.einsum("mij,mj->mi", inv[k].to(b.dtype), r)
    return torch.fft.irfft(u, n=nt, dim=1, norm="forward")


def _exact_deposit(case, parts):
    nr, nt, nz = case["nr"], case["nt"], case["nz"]
    dr, da, dz = (R_OUT - R_IN) / nr, 2.0 * math.pi / nt, Z_LEN / nz
    nodes = torch.zeros(nz + 1, nt, nr + 1, dtype=torch.float64, device="cuda")
    flat = nodes.view(-1)
    for at in range(0, parts[0].numel(), 1 << 24):
        t = [(parts[0][at:at + (1 << 24)] - R_IN) / dr, parts[1][at:at + (1 << 24)] / da, parts[2][at:at + (1 << 24)] / dz]
        cell = [x.floor() for x in t]
        inside = functools.reduce(torch.logical_and, [(c >= 0) & (c < n) for c, n in zip(cell, (nr, nt, nz))])
        t = [(x - c)[inside] for x, c in zip(t, cell)]
        i, j, k = [c[inside].long() for c in cell]
        for corner in range(8):
            x, y, q = corner & 1, (corner >> 1) & 1, corner >> 2
            wgt = (t[0] if x else 1 - t[0]) * (t[1] if y else 1 - t[1]) * (t[2] if q else 1 - t[2])
            flat.index_add_(0, ((k + q) * nt + (j + y) % nt) * (nr + 1) + i + x, wgt)
    rf = R_IN + dr * np.arange(nr + 1)
    edge = np.r_[rf[0], 0.5 * (rf[1:] + rf[:-1]), rf[-1]]
    lz = np.full(nz + 1, dz)
    lz[0] = lz[-1] = 0.5 * dz
    vr = 0.5 * (edge[1:] ** 2 - edge[:-1] ** 2)
    return nodes * WEIGHT / (_cuda(vr)[None, None, :] * da * _cuda(lz)[:, None, None])


def _exact_project(case, nodes, charge):
    nr, nt = case["nr"], case["nt"]
    dr = (R_OUT - R_IN) / nr
    lo = R_IN + dr * np.arange(nr)
    mid, hi = lo + 0.5 * dr, lo + dr
    flo, fhi = (mid ** 2 - lo ** 2) / (hi ** 2 - lo ** 2), (hi ** 2 - mid ** 2) / (hi ** 2 - lo ** 2)
    n = nodes + nodes.roll(-1, 1)
    n = 0.25 * (n[1:] + n[:-1])
    return charge * (_cuda(flo) * n[..., :-1] + _cuda(fhi) * n[..., 1:])


def _exact_unet(case, seed):
    weights, x, target = _network(case, seed)
    ws = {k: w.to(torch.bfloat16).cuda().double().requires_grad_() for k, (w, _) in weights.items()}
    bs = {k: b.cuda().double().requires_grad_() for k, (_, b) in weights.items()}

    def conv(name, t, relu=True):
        w = ws[name]
        t = F.conv2d(t, w.permute(1, 2, 0).reshape(w.shape[1], w.shape[2], 3, 3), bs[name], padding=1)
        return F.relu(t) if relu else t

    def forward(t):
        up = lambda v: F.interpolate(v, scale_factor=2, mode="nearest")  # noqa: E731
        e0 = conv("e0", t)
        e1 = conv("e1", F.avg_pool2d(e0, 2))
        e2 = conv("e2", F.avg_pool2d(e1, 2))
        b2 = conv("b2", conv("b1", F.avg_pool2d(e2, 2)))
        d2 = conv("d2", torch.cat([up(b2), e2], 1))
        d1 = conv("d1", torch.cat([up(d2), e1], 1))
        d0 = conv("d0", torch.cat([up(d1), e0], 1))
        return conv("out", d0, relu=False).permute(0, 2, 3, 1)

    t = x.double().permute(0, 3, 1, 2)
    if not case["train"]:
        with torch.no_grad():
            return torch.cat([forward(t[i:i + 8]) for i in range(0, case["n"], 8)])
    loss = 0.0
    for i in range(0, case["n"], 4):
        part = (forward(t[i:i + 4])[..., :2] - target[i:i + 4].double()).square().sum() / target.numel()
        part.backward()
        loss = loss + part.detach()
    return {"loss": loss.reshape(1), "w": {k: v.grad for k, v in ws.items()}, "b": {k: v.grad for k, v in bs.items()}}


def exact(case, seed):
    kind = case["kind"]
    if kind == "unet":
        return _exact_unet(case, seed)
    size = None if kind == "batch" else (case["nr"], case["nt"], case["nz"])
    if kind in ("solve", "axial"):
        return {"phi": _exact_annulus(case, W.rho_plasma_torch(_problems(case)[0], seed), *size), "status": None}
    if kind == "plume":
        if case["nr"] ** 3 * case["nt"] * case["nz"] > 3e11:
            return None
        return {"phi": _exact_plume(case, W.rho_plasma_torch(_problems(case)[0], seed), *size), "status": None}
    if kind == "batch":
        probs = _problems(case)
        return {"phis": [_exact_annulus(case, W.rho_plasma_torch(p, 64 * seed + i), p.nr, p.ntheta, p.nz) for i, p in enumerate(probs)],
                "status": None}
    s = prepare(case, seed)
    if kind == "transforms":
        nr, nt, nz = size
        rc, dr, dz, _, gz = _geometry(*_faces(case, nr, nz))
        b = _rhs(s["rho"], rc, dr, dz)
        b[0, 0] += _cuda(PHI_Z0 * gz[0] * rc * dr)
        u = torch.view_as_complex(s["uhat"]).permute(0, 2, 1).clone()
        u[:, 0].imag.zero_()
        u[:, -1].imag.zero_()
        return {"bhat": torch.view_as_real(b.permute(0, 2, 1)).contiguous(),
                "phi": torch.fft.irfft(u, n=nt, dim=1, norm="forward")}
    if kind == "field":
        nr, nt, nz = size
        rc, _, _, gr, gz = _geometry(*_faces(case, nr, nz))
        rf, _ = _faces(case, nr, nz)
        phi = s["phi"]
        zero = phi[..., :1] * 0.0
        er = -torch.diff(torch.cat([zero, phi, zero], 2), dim=2) * _cuda(gr / rf)
        ea = (phi - phi.roll(-1, 1)) / (_cuda(rc) * (2.0 * math.pi / nt))
        wall = phi[:1] * 0.0
        ez = -torch.diff(torch.cat([wall + PHI_Z0, phi, wall], 0), dim=0) * _cuda(gz)[:, None, None]
        return er, ea, ez
    ions, electrons = _exact_deposit(case, s["ions"]), _exact_deposit(case, s["electrons"])
    rho = _exact_project(case, ions, E_CHARGE) + _exact_project(case, electrons, -E_CHARGE)
    return {"ions": ions, "electrons": electrons, "rho": rho}
