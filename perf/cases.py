"""What a user of this framework has it do, as cases that can be timed and compared.

Each case goes through the public binding (paper_2205_08417_gb300.kitrt): time steps of the M_N
system in the closure modes, the S_N step, the discrete adjoint, batch closures (training data of
the learned closure) and a training step of its network. Meshes and media are the repository's own
synthetic ones; initial states are moments of positive angular densities on the solver's
quadrature (a line source some time after its start: a streaming ring plus its scattered part).

`exact` restates the method in 64-bit torch, without the library: quadrature, basis, closure by
damped Newton, kinetic upwind flux (first and second order), the S_N update, the adjoint by the
implicit-function theorem, and the network's loss gradient and Adam step.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2205_08417_gb300 import kitrt, synth

M0 = 1.0 / math.sqrt(4.0 * math.pi)
F64 = torch.float64


# ------------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest runs: a few thousand cells, where launches and round trips count
        dict(name="m2_line_4k_fp64", kind="step", k=45, box="line", degree=2, order=10, mode="fp64", steps=2),
        # the benchmark's configuration: the line source on ~100k triangles, mixed precision
        dict(name="m3_line_100k_tf32", kind="step", k=224, box="line", degree=3, order=20, mode="mixed_tf32", steps=4),
        # the same run in the reference precision
        dict(name="m3_line_100k_fp64", kind="step", k=224, box="line", degree=3, order=20, mode="fp64", steps=2),
        # the learned closure with its Newton fallback, medium mesh
        dict(name="m3_line_25k_learned", kind="step", k=113, box="line", degree=3, order=20, mode="learned", steps=2),
        # the largest run: a million triangles, degree 5, block medium
        dict(name="m5_blocks_1m_tf32", kind="step", k=707, box="blocks", degree=5, order=30, mode="mixed_tf32", steps=2),
        # the checkerboard: second order in space and time, vacuum walls
        dict(name="m3_checker_25k_heun", kind="step", k=113, box="checker", degree=3, order=10, mode="mixed_tf32",
             steps=2, second=True, vacuum=True),
        # continuous slowing down with a tissue density: one call and a dose update per step; an
        # odd quadrature order and a ragged mesh size, BF16 operands
        dict(name="m4_csd_20k_bf16", kind="csd", k=101, box="line", degree=4, order=15, mode="mixed_bf16", steps=2),
        # discrete ordinates: FP32, isotropic scattering, the benchmark's mesh
        dict(name="sn_line_100k_fp32", kind="sn", k=224, box="line", degree=3, order=20, fp32=True, steps=4),
        # discrete ordinates: FP64, anisotropic scattering, odd order
        dict(name="sn_blocks_20k_fp64", kind="sn", k=101, box="blocks", degree=3, order=15, fp32=False, steps=3, g=0.7),
        # sensitivities of the absorbed energy to the block coefficients
        dict(name="m3_adjoint_60k", kind="adjoint", k=173, box="blocks", degree=3, order=10, steps=16, every=8),
        # closing a batch of training densities from the isotropic start, tight tolerance
        dict(name="m3_closure_20k", kind="closure", rows=20001, degree=3, order=20, kappa=20.0),
        # one training step of the network (loss gradient, then Adam), default batch
        dict(name="mlp_train_1k", kind="mlp", rows=1024, degree=3),
    ]


def draw(rng):
    def sizes(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "step", "step", "csd", "sn", "sn", "adjoint", "closure", "mlp"])
    degree = rng.choice([1, 2, 3, 3, 4, 5])
    order = rng.randint(max(6, 2 * degree), 24)
    if kind == "step":
        box = rng.choice(["line", "blocks", "checker"])
        return dict(kind=kind, k=sizes(14, 240), box=box, degree=degree, order=order,
                    mode=rng.choice(["fp64", "mixed_tf32", "mixed_tf32", "mixed_bf16", "learned"]),
                    steps=rng.randint(2, 3), vacuum=box != "line")
    if kind == "csd":
        return dict(kind=kind, k=sizes(14, 160), box="line", degree=degree, order=order,
                    mode=rng.choice(["fp64", "mixed_tf32", "mixed_bf16"]), steps=rng.randint(2, 3))
    if kind == "sn":
        return dict(kind=kind, k=sizes(14, 224), box=rng.choice(["line", "blocks"]), degree=degree, order=order,
                    fp32=rng.random() < 0.5, steps=rng.randint(1, 4), g=rng.choice([0.0, 0.5, 0.8]))
    if kind == "adjoint":
        return dict(kind=kind, k=sizes(14, 120), box="blocks", degree=min(degree, 4), order=order,
                    steps=rng.randint(4, 10), every=rng.randint(2, 6))
    if kind == "closure":
        return dict(kind=kind, rows=sizes(100, 40000), degree=min(degree, 4), order=max(order, 14),
                    kappa=rng.uniform(4.0, 20.0))
    return dict(kind=kind, rows=sizes(128, 8192), degree=degree)


def _cells(case):
    return 2 * (case["k"] - 1) ** 2


def work(case):
    """Bytes: state in and out (u, alpha or ordinates), cell coefficients and geometry, each once
    per step. Flops: per folded point one exponent (2n), one exponential (counted 10), the upwind
    fluctuation (12) and the projection on the basis (2n); the adjoint three such passes per step;
    a batch closure five (a Newton solve from the isotropic start)."""
    n = (case["degree"] + 1) * (case["degree"] + 2) // 2
    if case["kind"] == "mlp":
        d, h, rows = n - 1, 64, case["rows"]
        p = d * h + h + 2 * (h * h + h) + h * d + d
        return {"bytes": 4.0 * (2 * rows * d + 8 * p), "flops": 6.0 * rows * (2 * d * h + 2 * h * h)}
    qf = (case["order"] + 1) // 2 * 2 * case["order"]
    if case["kind"] == "closure":
        return {"bytes": 8.0 * case["rows"] * 3 * n, "flops": 5.0 * case["rows"] * qf * (4 * n + 10)}
    cells, steps, geo = _cells(case), case["steps"], 16 + 48 + 8 + 24
    if case["kind"] == "sn":
        b = 4 if case["fp32"] else 8
        mom = n if case.get("g") else 1
        return {"bytes": float(steps * cells * (2 * qf * b + geo)), "flops": float(steps * cells * qf * (16 + 4 * mom))}
    passes = 2 if case.get("second") else 3 if case["kind"] == "adjoint" else 1
    return {"bytes": float(passes * steps * cells * (4 * 8 * n + geo)),
            "flops": float(passes * steps * cells * qf * (4 * n + 22))}


# ------------------------------------------------------------------------------------------------
# inputs (the same ones for `run` and `exact`)
# ------------------------------------------------------------------------------------------------
_BOX = {"line": (-1.5, 1.5), "blocks": (0.0, 7.0), "checker": (0.0, 7.0)}


@functools.lru_cache(maxsize=3)
def _mesh(k, box):
    return synth.jittered_mesh(k, *_BOX[box], seed=2)


@functools.lru_cache(maxsize=8)
def _rule(order, degree):
    """Folded product rule in the library's point order (rings from the pole to the equator; per
    ring phi = 0, pi, then the mirrored pairs): weights, 2D directions, basis values [Q', n], and
    the degree of every basis function."""
    x, g = np.polynomial.legendre.leggauss(order)
    nphi = 2 * order
    steps = [0, order] + [j for i in range(1, order) for j in (i, nphi - i)]
    phi = 2.0 * math.pi / nphi * np.array(steps)
    mu, w = [], []
    for i in range(order - 1, order // 2 - 1, -1):
        if order % 2 and i == order // 2:
            mu.append(0.0), w.append(g[i])
        else:
            mu.append(x[i]), w.append(2.0 * g[i])
    mu, w = np.array(mu), np.array(w) * 2.0 * math.pi / nphi
    s = np.sqrt(1.0 - mu ** 2)
    om = np.stack([s[:, None] * np.sin(phi), s[:, None] * np.cos(phi)], axis=-1).reshape(-1, 2)
    P = {(0, 0): np.full(mu.shape, math.sqrt(1.0 / (4.0 * math.pi)))}
    for k in range(1, degree + 1):
        P[k, k] = math.sqrt((2 * k + 1) / (2 * k)) * s * P[k - 1, k - 1]
    for k in range(degree):
        P[k + 1, k] = math.sqrt(2 * k + 3) * mu * P[k, k]
    for k in range(degree + 1):
        for l in range(k + 2, degree + 1):
            a = math.sqrt((4 * l * l - 1) / (l * l - k * k))
            b = math.sqrt(((l - 1) ** 2 - k * k) / (4 * (l - 1) ** 2 - 1))
            P[l, k] = a * (mu * P[l - 1, k] - b * P[l - 2, k])
    cols, deg = [], []
    for l in range(degree + 1):
        for k in range(-l, l + 1, 2):
            t = np.ones_like(phi) if k == 0 else math.sqrt(2) * (np.cos(k * phi) if k > 0 else np.sin(-k * phi))
            cols.append((P[l, abs(k)][:, None] * t).reshape(-1))
            deg.append(l)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return dev(np.repeat(w, nphi)), dev(om), dev(np.stack(cols, axis=1)), deg


def _chunks(rows, width):
    step = max(1, int(4e8) // (8 * width))
    return [slice(i, min(rows, i + step)) for i in range(0, rows, step)]


def _density(case, seed):
    """psi(x, Omega) of a line source a while after its start, as a function of cell centroids and
    directions: the streaming part is carried along Omega, the scattered part is isotropic."""
    r = np.random.default_rng(seed)
    lo, hi = _BOX[case["box"]]
    size = hi - lo
    x0 = 0.5 * (lo + hi) + r.uniform(-0.08, 0.08, 2) * size
    t, w, ws = r.uniform(0.08, 0.12) * size, r.uniform(0.035, 0.05) * size, r.uniform(0.06, 0.08) * size
    mix = r.uniform(0.3, 0.5)

    def psi(cen, om):
        at = torch.from_numpy(x0).to(cen)
        d = cen - at
        d2, o2, do = (d * d).sum(1, keepdim=True), (om * om).sum(1)[None], d @ om.T
        ring = torch.exp(-(d2 - 2 * t * do + t * t * o2) / (2 * w * w)) / (2 * math.pi * w * w)
        scat = torch.exp(-d2 / (2 * ws * ws)) / (2 * math.pi * ws * ws)
        return (ring + mix * scat + 1e-3) / (4 * math.pi)
    return psi


def _medium(case, cen, seed):
    """sigma_a, sigma_s, q per cell (numpy), and the block of each cell where there are blocks."""
    C = cen.shape[0]
    if case["box"] == "line":
        return np.zeros(C), np.ones(C), np.zeros(C), None
    if case["box"] == "checker":
        return (*synth.checkerboard_medium(cen), None)
    blk, sa, ss = synth.block_coefficients(cen, 0.0, 7.0, 7, seed)
    q = np.where(blk == 3 * 7 + 3, 1.0, 0.0)
    return sa[blk], ss[blk], q, blk


def _inputs(case, seed):
    m = _mesh(case["k"], case["box"])
    cen = m.centroids()
    w, om, M, _ = _rule(case["order"], case["degree"])
    psi, c = _density(case, seed), torch.from_numpy(cen).cuda()
    sa, ss, q, blk = _medium(case, cen, seed)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    out = dict(mesh=m, cen=cen, sa=dev(sa), ss=dev(ss), q=dev(q), blk=blk)
    if case["kind"] == "sn":
        out["psi"] = torch.empty(m.ncells, w.numel(), dtype=torch.float32 if case["fp32"] else F64, device="cuda")
        for s in _chunks(m.ncells, w.numel()):
            out["psi"][s] = psi(c[s], om)
    else:
        out["u"] = torch.cat([psi(c[s], om) @ (w[:, None] * M) for s in _chunks(m.ncells, w.numel())])
    if case["kind"] == "csd":
        rho = synth.two_tissue_density(cen)
        out["rho"] = dev(rho)
        out["u"] = out["u"] * out["rho"][:, None]
    a, b, d = (m.xy[m.tri[:, i]] for i in range(3))
    area = 0.5 * np.abs((b - a)[:, 0] * (d - a)[:, 1] - (b - a)[:, 1] * (d - a)[:, 0])
    per = sum(np.hypot(*(p - r).T) for p, r in ((a, b), (b, d), (d, a)))
    # the step that the library's CFL rule picks, kept inside the cells' stability limit
    out["dt"] = float(min(0.4 * np.min(2 * area / per), 0.9 / np.max(per / (2 * area) + sa + ss)))
    return out


def _vmf(case, seed):
    """Moments of von Mises-Fisher mixtures (training densities) and the isotropic start."""
    w, om, M, _ = _rule(case["order"], case["degree"])
    c, kap, wt = synth.vmf_mixtures(case["rows"], seed, kappa_hi=case["kappa"])
    scale = np.exp(np.random.default_rng(seed + 1).uniform(-4.0, 3.0, size=case["rows"]))
    c, kap, wt = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (c, kap, wt * scale[:, None]))
    mu = torch.sqrt(torch.clamp(1.0 - (om * om).sum(1), min=0.0))
    rows = []
    for s in _chunks(case["rows"], 8 * w.numel()):
        psi = 0.0
        for sign in (0.5, -0.5):  # the two directions +-mu of a folded point
            x = torch.stack([om[:, 0], om[:, 1], 2 * sign * mu])
            k = kap[s][:, :, None]
            psi = psi + 0.5 * (wt[s][:, :, None] * k / (2 * math.pi * -torch.expm1(-2 * k))
                               * torch.exp(k * (c[s] @ x - 1.0))).sum(1)
        rows.append(psi @ (w[:, None] * M))
    u = torch.cat(rows)
    alpha = torch.zeros_like(u)
    alpha[:, 0] = torch.log(u[:, 0] / (4 * math.pi * M0)) / M0
    return u, alpha


def _network(case, seed):
    """A network's packed parameters (three hidden layers of 64), one batch, and Adam's moments."""
    d, h = (case["degree"] + 1) * (case["degree"] + 2) // 2 - 1, 64
    g = torch.Generator().manual_seed(seed)
    parts = []
    for i, o in [(d, h), (h, h), (h, h), (h, d)]:
        parts += [(torch.rand(i * o, generator=g) * 2 - 1) * math.sqrt(6.0 / (i + o)), 0.05 * torch.randn(o, generator=g)]
    p = torch.cat(parts)
    X, T = (torch.randn(case.get("rows", 1), d, generator=g) for _ in range(2))
    m = 1e-3 * torch.randn(p.numel(), generator=g)
    v = 1e-5 * (0.5 + torch.rand(p.numel(), generator=g))
    return d, h, p.cuda(), X.cuda(), T.cuda(), m.cuda(), v.cuda()


# ------------------------------------------------------------------------------------------------
# what a program has in hand, and one pass
# ------------------------------------------------------------------------------------------------
class _State:
    pass


def _anisotropy(case):
    return np.array([case["g"] ** l for l in range(case["degree"] + 1)]) if case.get("g") else None


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "mlp":
        s.d, s.h, s.p, s.X, s.T, s.m, s.v = _network(case, seed)
        s.work = torch.empty(kitrt._lib().kitrt_mlp_work_floats(case["rows"], s.h, s.d), device="cuda")
        return s
    if case["kind"] == "closure":
        k = 2 + math.isqrt(case["rows"] // 2)
        s.mesh = kitrt.Mesh(*(lambda m: (m.xy, m.tri))(_mesh(k + 1, "line")))
        s.solver = kitrt.MNSolver(s.mesh, case["degree"], case["order"], tau=1e-12)
        s.u, s.alpha0 = _vmf(case, seed)
        s.alpha = s.alpha0.clone()
        s.status = torch.zeros(case["rows"], dtype=torch.int32, device="cuda")
        return s
    s.inp = i = _inputs(case, seed)
    s.mesh = kitrt.Mesh(i["mesh"].xy, i["mesh"].tri)
    opts = dict(tau=1e-10)
    mode = case.get("mode", "fp64")
    if mode != "fp64":
        opts["tau"] = 1e-8
    if case.get("second"):
        opts["order"] = 2
    bc = "vacuum" if case.get("vacuum") or case["kind"] == "adjoint" else "neumann"
    s.solver = kitrt.MNSolver(s.mesh, case["degree"], case["order"], mode=mode, bc=bc, **opts)
    s.dt = i["dt"]
    if case["kind"] == "sn":
        s.psi, s.work = i["psi"].clone(), torch.empty_like(i["psi"])
        return s
    if mode == "learned":
        d, h, p, *_ = _network(dict(degree=case["degree"]), seed)
        one, zero = torch.ones(d, device="cuda"), torch.zeros(d, device="cuda")
        s.solver.set_mlp(p, torch.cat([zero, 0.3 * one, zero, one]))
    s.u = i["u"].clone()
    s.alpha = s.solver.isotropic_alpha(s.u)
    if case["kind"] == "csd":
        s.solver.set_density(i["rho"])
        s.dose = torch.zeros(s.mesh.ncells, dtype=F64, device="cuda")
    if case["kind"] == "adjoint":
        s.blk, s.target = torch.from_numpy(i["blk"]).cuda(), _target(i["blk"])
    return s


def _target(blk):
    return torch.from_numpy(np.isin(blk, [bx * 7 + by for bx in (2, 3, 4) for by in (2, 3, 4)]).astype(np.uint8)).cuda()


def run(s):
    """One pass: the state comes in (as from the host or another model), the call advances it. The
    warm start alpha stays with the solver between passes, as in a time loop."""
    case = s.case
    if case["kind"] == "mlp":
        loss, grad = kitrt.mlp_loss_grad(s.p, s.X, s.T, s.d, s.h, s.d, work=s.work)
        kitrt.mlp_adam(s.p, grad, s.m, s.v, 10, lr=3e-3)
        return loss, grad, s.p, s.m, s.v
    if case["kind"] == "closure":
        s.alpha.copy_(s.alpha0)
        s.solver.closure_batch(s.u, s.alpha, s.status)
        return s.alpha, s.status
    i = s.inp
    if case["kind"] == "sn":
        s.psi.copy_(i["psi"])
        s.solver.sn_step(s.psi, s.work, i["sa"], i["ss"], i["q"], dt=s.dt, nsteps=case["steps"], g=_anisotropy(case))
        return s.psi
    if case["kind"] == "adjoint":
        return s.solver.adjoint(i["u"], s.alpha, i["sa"], i["ss"], i["q"], s.blk, 49, s.target, s.dt,
                                case["steps"], case["every"])
    s.u.copy_(i["u"])
    if case["kind"] == "csd":
        s.dose.zero_()
        for it in range(case["steps"]):
            s.solver.dose_accumulate(s.u, 1.0 + 0.1 * it, s.dt, s.dose)
            s.solver.step(s.u, s.alpha, i["sa"], i["ss"], i["q"], dt=s.dt, nsteps=1)
        return s.u, s.alpha, s.dose
    s.solver.step(s.u, s.alpha, i["sa"], i["ss"], i["q"], dt=s.dt, nsteps=case["steps"])
    return s.u, s.alpha


# ------------------------------------------------------------------------------------------------
# the method in 64 bits
# ------------------------------------------------------------------------------------------------
def _close(u, alpha, w, M):
    """alpha minimising <exp(alpha.m)> - alpha.u, row by row: damped Newton, then two full steps."""
    n = M.shape[1]
    tri = torch.tril_indices(n, n, device=u.device)
    MM = M[:, tri[0]] * M[:, tri[1]]
    out = alpha.clone()
    for s in _chunks(u.shape[0], M.shape[0] * 2):
        rows = torch.arange(s.start, s.stop, device=u.device)
        a, lam, d, f0, gd, left = out[s].clone(), None, None, None, None, None
        ub = u[s]
        left = torch.full((len(rows),), 2, device=u.device)
        lam = torch.zeros(len(rows), dtype=F64, device=u.device)
        d, f0, gd = torch.zeros_like(a), torch.full_like(lam, math.inf), torch.zeros_like(lam)
        for _ in range(200):
            t = a + lam[:, None] * d
            e = torch.exp(t @ M.T) * w
            f = e.sum(1) - (t * ub).sum(1)
            ok = torch.isfinite(f) & ((f <= f0 + 1e-4 * lam * gd + 2e-14 * (e.sum(1) + f.abs())) | (left < 2))
            g = e @ M - ub
            near = ok & (g.norm(dim=1) <= 1e-9 * ub.norm(dim=1))
            left = left - near.int()
            H = torch.zeros(len(rows), n, n, dtype=F64, device=u.device)
            H[:, tri[0], tri[1]] = e @ MM
            L, info = torch.linalg.cholesky_ex(H)
            ok = ok & (info == 0)
            step = -torch.cholesky_solve(g[:, :, None], torch.where((info == 0)[:, None, None], L, torch.eye(n, dtype=F64, device=u.device)))[:, :, 0]
            a = torch.where(ok[:, None], t, a)
            d = torch.where(ok[:, None], step, d)
            gd, f0 = torch.where(ok, (g * step).sum(1), gd), torch.where(ok, f, f0)
            lam = torch.where(ok, torch.ones_like(lam), 0.5 * lam)
            done = left < 0
            if bool(done.any()):
                out[rows[done]] = a[done] + d[done]
                keep = ~done
                if not bool(keep.any()):
                    break
                rows, a, ub, lam, d, f0, gd, left = (v[keep] for v in (rows, a, ub, lam, d, f0, gd, left))
        else:
            out[rows] = a
    return out


def _geometry(m):
    v = np.array(m.tri, dtype=np.int64)
    p = m.xy[v]
    cross = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 1, 1] - p[:, 0, 1]) * (p[:, 2, 0] - p[:, 0, 0])
    v[cross < 0] = v[cross < 0][:, [0, 2, 1]]
    p = m.xy[v]
    nxt = np.roll(p, -1, axis=1)
    nrm = np.stack([nxt[..., 1] - p[..., 1], p[..., 0] - nxt[..., 0]], axis=-1)
    mid = 0.5 * (p + nxt) - p.mean(axis=1, keepdims=True)
    vn = np.roll(v, -1, axis=1)
    key = (np.minimum(v, vn) * len(m.xy) + np.maximum(v, vn)).reshape(-1)
    order = np.argsort(key, kind="stable")
    same = np.nonzero(key[order][1:] == key[order][:-1])[0]
    other = np.full(key.size, -1)
    other[order[same]], other[order[same + 1]] = order[same + 1], order[same]
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    return dict(area=dev(0.5 * np.abs(cross)), nrm=dev(nrm), mid=dev(mid), other=dev(other.reshape(-1, 3)))


def _flux(G, psi, w, om, M, vacuum, second=False):
    """Projected kinetic upwind flux of every cell; psi [C, Q'] as transported."""
    C = psi.shape[0]
    out = torch.empty(C, M.shape[1], dtype=F64, device=psi.device)
    nb = torch.where(G["other"] >= 0, G["other"] // 3, -1)
    parts = _chunks(C, psi.shape[1] * 4)

    def ghost(s, f, own):
        x = psi[nb[s, f].clamp(min=0)]
        return torch.where((nb[s, f] >= 0)[:, None], x, torch.zeros_like(own) if vacuum else own)

    face = None
    if second:
        face = torch.empty(C, 3, psi.shape[1], dtype=F64, device=psi.device)
        for s in parts:
            own = psi[s]
            side = [ghost(s, f, own) for f in range(3)]
            g = sum(0.5 * (own + side[f])[:, None, :] * G["nrm"][s, f][:, :, None] for f in range(3)) / G["area"][s][:, None, None]
            D = [(g * G["mid"][s, f][:, :, None]).sum(1) for f in range(3)]
            lim = torch.ones_like(own)
            for f in range(3):
                room = torch.where(D[f] > 0, torch.maximum(own, side[f]), torch.minimum(own, side[f])) - own
                lim = torch.where(D[f] != 0, torch.minimum(lim, room / torch.where(D[f] != 0, D[f], 1.0)), lim)
            for f in range(3):
                face[s, f] = own + lim * D[f]
        face = face.reshape(C * 3, -1)
    for s in parts:
        own, acc = psi[s], 0.0
        for f in range(3):
            dot = G["nrm"][s, f] @ om.T
            if second:
                mine = face[3 * torch.arange(s.start, s.stop, device=psi.device) + f]
                up = torch.where((nb[s, f] >= 0)[:, None], face[G["other"][s, f].clamp(min=0)],
                                 torch.zeros_like(own) if vacuum else mine)
                acc = acc + dot * (torch.where(dot > 0, mine, up) - own)
            else:
                acc = acc + dot.clamp(max=0.0) * (ghost(s, f, own) - own)
        out[s] = acc @ (w[:, None] * M)
    return out


def _source(u, i, mbar):
    R = -(i["sa"] + i["ss"])[:, None] * u + i["q"][:, None] * mbar
    R[:, 0] += i["ss"] * u[:, 0]
    return R


def _psi(alpha, M):
    return torch.exp(alpha @ M.T)


def _iso(u):
    a = torch.zeros_like(u)
    a[:, 0] = torch.log(u[:, 0] / (4 * math.pi * M0)) / M0
    return a


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    w, om, M, deg = _rule(case["order"], case["degree"])
    if case["kind"] == "closure":
        u, a = _vmf(case, seed)
        return _close(u, a, w, M), None
    i = _inputs(case, seed)
    G, dt, mbar = _geometry(i["mesh"]), i["dt"], w @ M
    vacuum = bool(case.get("vacuum"))
    if case["kind"] == "sn":
        g = _anisotropy(case)
        g = torch.tensor([(g[l] if g is not None else float(l == 0)) for l in deg], dtype=F64, device="cuda")
        psi = i["psi"].double()
        nb = torch.where(G["other"] >= 0, G["other"] // 3, -1)
        for _ in range(case["steps"]):
            new = torch.empty_like(psi)
            for s in _chunks(psi.shape[0], psi.shape[1] * 4):
                own, acc = psi[s], 0.0
                for f in range(3):
                    up = torch.where((nb[s, f] >= 0)[:, None], psi[nb[s, f].clamp(min=0)], own)
                    acc = acc + (G["nrm"][s, f] @ om.T).clamp(max=0.0) * (up - own)
                scat = ((own @ (w[:, None] * M)) * g) @ M.T
                new[s] = (own - dt * (acc / G["area"][s][:, None] + (i["sa"] + i["ss"])[s][:, None] * own
                                      - i["ss"][s][:, None] * scat - i["q"][s][:, None]))
            psi = new
        return psi
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, i, G, w, om, M, mbar)
    u, a = i["u"], _iso(i["u"])
    rho = i.get("rho")
    dose = torch.zeros_like(u[:, 0])

    def rate(v, a):
        a = _close(v, a, w, M)
        psi = _psi(a, M)
        if rho is not None:
            psi /= rho[:, None]
        return a, _source(v, i, mbar) - _flux(G, psi, w, om, M, vacuum, bool(case.get("second"))) / G["area"][:, None]

    for it in range(case["steps"]):
        if rho is not None:
            dose += dt * (1.0 + 0.1 * it) * u[:, 0] / (M0 * rho)
        a, r = rate(u, a)
        if case.get("second"):
            v = u + dt * r
            a, r = rate(v, a)
            u = 0.5 * (u + v + dt * r)
        else:
            u = u + dt * r
    return (u, a, dose) if rho is not None else (u, a)


def _exact_adjoint(case, i, G, w, om, M, mbar):
    dt, blk, tgt = i["dt"], torch.from_numpy(i["blk"]).long().cuda(), _target(i["blk"]).double()
    us, al, u, a, J = [], [], i["u"], _iso(i["u"]), 0.0
    for _ in range(case["steps"]):
        J += float((dt * tgt * G["area"] * i["sa"] * u[:, 0] / M0).sum())
        a = _close(u, a, w, M)
        us.append(u), al.append(a)
        u = u + dt * (_source(u, i, mbar) - _flux(G, _psi(a, M), w, om, M, True) / G["area"][:, None])
    lam = torch.zeros_like(u)
    gsa, gss = (torch.zeros(49, dtype=F64, device="cuda") for _ in range(2))
    nb = torch.where(G["other"] >= 0, G["other"] // 3, -1)
    n = M.shape[1]
    tri = torch.tril_indices(n, n, device="cuda")
    MM = M[:, tri[0]] * M[:, tri[1]]
    for u, a in zip(us[::-1], al[::-1]):
        gsa.index_add_(0, blk, -dt * (lam * u).sum(1) + tgt * dt * G["area"] * u[:, 0] / M0)
        gss.index_add_(0, blk, -dt * (lam[:, 1:] * u[:, 1:]).sum(1))
        Lq = (lam / G["area"][:, None]) @ M.T
        new = torch.empty_like(lam)
        for s in _chunks(u.shape[0], M.shape[0] * 4):
            e = _psi(a[s], M) * w
            acc = 0.0
            for f in range(3):
                out = (G["nrm"][s, f] @ om.T).clamp(min=0.0)
                there = torch.where((nb[s, f] >= 0)[:, None], Lq[nb[s, f].clamp(min=0)], torch.zeros_like(e))
                acc = acc + out * (Lq[s] - there)
            H = torch.zeros(e.shape[0], n, n, dtype=F64, device="cuda")
            H[:, tri[0], tri[1]] = e @ MM
            new[s] = torch.cholesky_solve(((-dt * acc * e) @ M)[:, :, None], torch.linalg.cholesky(H))[:, :, 0]
        back = -(i["sa"] + i["ss"])[:, None] * lam
        back[:, 0] += i["ss"] * lam[:, 0]
        lam = lam + dt * back + new
        lam[:, 0] += tgt * dt * G["area"] * i["sa"] / M0
    return J, gsa.cpu().numpy(), gss.cpu().numpy()


def _exact_mlp(case, seed):
    d, h, p, X, T, m, v = _network(case, seed)
    p, X, T, m, v = (t.double() for t in (p, X, T, m, v))
    q = p.clone().requires_grad_(True)
    x, off = X, 0
    for layer, (i, o) in enumerate([(d, h), (h, h), (h, h), (h, d)]):
        W, b = q[off:off + i * o].view(i, o), q[off + i * o:off + i * o + o]
        off += i * o + o
        x = x @ W + b
        if layer < 3:
            x = torch.where(x > 0, x, torch.zeros_like(x)) + torch.log1p(torch.exp(-x.abs()))
    loss = 0.5 * (x - T).square().sum() / X.shape[0]
    g, = torch.autograd.grad(loss, q)
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    p = p - 3e-3 * (m / (1 - 0.9 ** 10)) / ((v / (1 - 0.999 ** 10)).sqrt() + 1e-8)
    return loss.detach().reshape(1), g, p, m, v
