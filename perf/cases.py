"""Workloads that the library's speed is measured on, each through its public entry points.

Single steps of the operator (steps 2+3 `apply_pairs`, step 1 `apply_precond`, the two together
`apply_operator`, step 1 on device buffers `apply_precond_noalloc`), the flow at points
(`eval_velocity`) and two whole calls (`solve`, `batch_solve_rhs`).  A case is a dict of plain
values; `geometry` seeds the sphere positions, so a case fixes its discretisation, and the seed
given to `prepare` draws the vectors a program brings to it.

Data.  Pair sums get O(1) random strengths and data.  Step 1 gets random data, whose strengths
the truncated pseudo-inverse amplifies by many orders, as it does the rough part of a Krylov
vector.  The operator gets the scaled boundary data of random rigid motions, normalised: the
first Krylov vector of a solve.  The whole calls are solved to 1e-11, where forces, torques and
velocities no longer depend on the path the iteration took.

`exact` evaluates the same formulas with its own discretisation in 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2407_03343_gb300 import mfs, workloads

PRECISION = {"fp64": mfs.FP64, "mixed": mfs.MIXED, "pass": mfs.MIXED_PASS}
EPS_TRUNC = 5e-12
DEV = "cuda" if torch.cuda.is_available() else "cpu"


def listed():
    return [
        # the smallest call: step 1 of two near spheres on buffers the caller owns, as inside a
        # latency-critical time step (native FP64)
        dict(name="precond_noalloc_two", kind="noalloc", shape="two", gap=0.05, P=2, N=300, M0=600, r_proxy=0.63),
        # steps 2+3 of the gap sweep's hardest geometry (20 images per sphere): one GMRES pass on two spheres
        dict(name="pairs_mixed_two", kind="pairs", precision="mixed", shape="two", gap=1e-3, P=2, N=800, M0=1600,
             r_proxy=0.63, geometry=1),
        # steps 2+3 of the fixed cluster of 100 spheres in a background flow (basic method, no images)
        dict(name="pairs_mixed_cluster100", kind="pairs", precision="mixed", shape="cluster", gap=1e-2, P=100, N=686,
             M0=823, r_proxy=0.75, geometry=1),
        # the largest: steps 2+3 of the 200-sphere suspension with ~300 near contacts
        dict(name="pairs_mixed_suspension200", kind="pairs", precision="mixed", shape="suspension", phi=0.2, P=200,
             N=800, M0=1600, r_proxy=0.63, geometry=3),
        # the native FP64 pair sums: the refinement residual of a tight solve, plain FP64 solves
        dict(name="pairs_fp64_suspension20", kind="pairs", precision="fp64", shape="suspension", phi=0.2, P=20, N=686,
             M0=823, r_proxy=0.63, geometry=7),
        # step 1 inside the mixed GMRES passes, one distinct factor per sphere (the sweep's lockstep tail)
        dict(name="precond_pass_two", kind="precond", precision="pass", shape="two", gap=1e-3, P=2, N=800, M0=1600,
             r_proxy=0.63, geometry=1),
        # step 1 of the refinement residual where every sphere shares the basic factor
        dict(name="precond_mixed_cluster100", kind="precond", precision="mixed", shape="cluster", gap=1e-2, P=100,
             N=686, M0=823, r_proxy=0.75, geometry=1),
        # one GMRES operator application of a small suspension with images (the batched suspensions' sizes)
        dict(name="operator_pass_suspension8", kind="operator", precision="pass", shape="suspension", phi=0.2, P=8,
             N=400, M0=800, r_proxy=0.63, geometry=5, far=0.0),
        # the same for a contact-free cluster with the far field: near pairs, equivalent sources, tensor cores
        dict(name="operator_far_cluster150", kind="operator", precision="pass", shape="cluster", gap=1e-2, P=150,
             N=686, M0=823, r_proxy=0.75, geometry=1, far=3.5),
        # the flow on a grid of points around three spheres (the exterior-flow plot: ~16,000 points)
        dict(name="velocity_three_16k", kind="velocity", shape="dilute", phi=0.05, P=3, N=300, M0=400, r_proxy=0.63,
             geometry=2, points=16125),
        # a whole resistance solve of a dilute suspension, with the flow at check points
        dict(name="solve_dilute20", kind="solve", shape="dilute", phi=0.05, P=20, N=300, M0=400, r_proxy=0.63,
             geometry=3, points=500, mobility=False),
        # a sweep of gaps, three motions each, as one lockstep batch with several right-hand sides per geometry
        dict(name="batch_sweep", kind="batch", gaps=6, gap_lo=0.05, gap_hi=1.0, P=2, N=400, M0=800, r_proxy=0.63),
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    """One more case of these ranges: any size between a three-sphere toy and the listed large ones."""
    kind = rng.choice(["noalloc", "pairs", "pairs", "precond", "operator", "velocity", "solve", "batch"])
    geometry = rng.randrange(1, 10000)
    if kind == "pairs":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        P = int(round(_log(rng, 2, 90 if precision == "mixed" else 16)))
        N = int(round(_log(rng, 96, 800)))
        c = dict(kind=kind, precision=precision, P=P, N=N, M0=int(N * rng.uniform(1.2, 2.0)), r_proxy=0.63,
                 geometry=geometry)
        if rng.random() < 0.5:
            return dict(c, shape="suspension", phi=round(rng.uniform(0.05, 0.2), 3))
        return dict(c, shape="cluster", gap=round(_log(rng, 1e-3, 0.3), 5))
    if kind in ("noalloc", "precond"):
        precision = "fp64" if kind == "noalloc" else rng.choice(["fp64", "mixed", "pass"])
        N = int(round(_log(rng, 96, 500)))
        c = dict(kind=kind, N=N, M0=int(N * rng.uniform(1.3, 2.0)), r_proxy=0.63, geometry=geometry)
        if kind == "precond":
            c["precision"] = precision
        if rng.random() < 0.5:
            return dict(c, shape="two", P=2, gap=round(_log(rng, 1e-3, 0.5), 5))
        return dict(c, shape="dilute", P=int(round(_log(rng, 2, 60))), phi=0.05)
    if kind == "operator":
        N = int(round(_log(rng, 96, 400)))
        c = dict(kind=kind, precision=rng.choice(["fp64", "mixed", "pass"]), N=N, M0=int(N * rng.uniform(1.3, 2.0)),
                 r_proxy=0.63, geometry=geometry, far=0.0)
        if rng.random() < 0.5:
            return dict(c, shape="suspension", P=int(round(_log(rng, 2, 8))), phi=round(rng.uniform(0.05, 0.2), 3))
        P = int(round(_log(rng, 2, 60)))
        far = 4.0 if c["precision"] != "fp64" and rng.random() < 0.5 else 0.0
        return dict(c, shape="dilute", P=P, phi=0.05, far=far)
    if kind == "batch":
        N = int(round(_log(rng, 150, 400)))
        return dict(kind=kind, gaps=rng.randrange(1, 7), gap_lo=round(_log(rng, 0.05, 0.2), 4), gap_hi=1.0, P=2, N=N,
                    M0=2 * N + rng.randrange(0, 30), r_proxy=0.63)
    N = int(round(_log(rng, 150, 300)))
    c = dict(kind=kind, shape="dilute", phi=0.05, N=N, M0=int(N * rng.uniform(1.35, 2.0)), r_proxy=0.63,
             geometry=geometry)
    if kind == "velocity":
        return dict(c, P=int(round(_log(rng, 1, 12))), points=int(round(_log(rng, 50, 20000))))
    return dict(c, P=int(round(_log(rng, 2, 20))), points=int(round(_log(rng, 50, 2000))), mobility=rng.random() < 0.5)


# ---------------------------------------------------------------- geometry and parameters
def _centres(case):
    P = case["P"]
    if case["shape"] == "two":
        return workloads.two_spheres(case["gap"])
    if case["shape"] == "cluster":
        return workloads.cluster(P, case["gap"], seed=case["geometry"])
    if case["shape"] == "suspension":
        return workloads.suspension(P, case["phi"], seed=case["geometry"])
    # dilute: every gap at least 0.3, so no images and one shared basic factor
    return workloads.suspension(P, case["phi"], seed=case["geometry"], gap_lo=0.3, gap_hi=1.0, min_gap=0.3)


def _params(case):
    p = dict(n_proxy=case["N"], r_proxy=case["r_proxy"], m_basic=case["M0"])
    if case.get("shape") == "cluster":
        p["nim_fixed"] = 0
    if case.get("far", 0.0) > 0:
        p["far_dist"] = case["far"]
    if case["kind"] == "pairs":
        p["build_factors"] = 0
    return p


def _gaps(case):
    n, lo, hi = case["gaps"], case["gap_lo"], case["gap_hi"]
    return [lo * (hi / lo) ** (i / max(1, n - 1)) for i in range(n)]


def _points(case, centres, rng):
    """Points in the box around the spheres, outside every sphere."""
    lo, hi, got, n = centres.min(0) - 2.0, centres.max(0) + 2.0, [], 0
    while n < case["points"]:
        x = rng.uniform(lo, hi, size=(2 * case["points"] + 64, 3))
        d = np.linalg.norm(x[:, None] - centres[None], axis=2).min(axis=1)
        got.append(x[d > 1.0 + 1e-2])
        n += len(got[-1])
    return np.concatenate(got)[: case["points"]].copy()


def _vectors(case, centres, seed):
    """The random vectors of a case, drawn in one order for prepare and exact alike."""
    rng = np.random.default_rng([seed, 20240703])
    P = len(centres)
    v = {"v": rng.normal(size=(P, 3)), "w": rng.normal(size=(P, 3)), "rng": rng}
    if "points" in case:
        v["x"] = _points(case, centres, rng)
    return v


def _built(case, centres):
    ctx = mfs.Context(0)
    ctx.set_spheres(centres)
    ctx.build(**_params(case))
    return ctx


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        rng = np.random.default_rng([seed, 20240703])
        ctxs, problems = [], []
        for gap in _gaps(case):
            ctx = _built(dict(case, shape="two"), workloads.two_spheres(gap))
            for _ in range(3):
                ctxs.append(ctx)
                problems.append((rng.normal(size=(2, 3)), rng.normal(size=(2, 3))))
        return dict(case=case, ctxs=ctxs, problems=problems)
    centres = _centres(case)
    vec = _vectors(case, centres, seed)
    ctx = _built(case, centres)
    st = dict(case=case, ctx=ctx, **vec)
    s = ctx.sizes()
    if kind == "pairs":
        st["lam"] = vec["rng"].normal(size=s.n_unknowns)
        st["mu"] = vec["rng"].normal(size=3 * s.n_colloc)
    elif kind == "precond":
        st["mu"] = vec["rng"].normal(size=3 * s.n_colloc)
    elif kind == "noalloc":
        st["mu"] = torch.from_numpy(vec["rng"].normal(size=3 * s.n_colloc)).to(DEV)
        st["out"] = torch.zeros(s.n_unknowns, dtype=torch.float64, device=DEV)
        torch.cuda.synchronize()
    elif kind == "operator":
        ctx.set_rigid_velocities(vec["v"], vec["w"])
        b = ctx.rhs()
        st["mu"] = b / np.linalg.norm(b)
    elif kind == "velocity":
        ctx.set_rigid_velocities(vec["v"], vec["w"])
        ctx.solve(precision="mixed", tol=1e-11)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        _, out = mfs.batch_solve_rhs(st["ctxs"], st["problems"], precision="mixed", tol=1e-11)
        return {"F": np.stack([f for f, _ in out]), "T": np.stack([t for _, t in out])}
    ctx = st["ctx"]
    if kind == "pairs":
        return ctx.apply_pairs(st["lam"], st["mu"], PRECISION[case["precision"]])
    if kind == "precond":
        return ctx.apply_precond(st["mu"], PRECISION[case["precision"]])
    if kind == "operator":
        return ctx.apply_operator(st["mu"], PRECISION[case["precision"]])
    if kind == "noalloc":
        ctx.apply_precond_noalloc(st["mu"].data_ptr(), st["out"].data_ptr())
        return st["out"]
    if kind == "velocity":
        return ctx.eval_velocity(st["x"])
    if case["mobility"]:
        ctx.set_forces_torques(st["v"], st["w"])
        ctx.solve(precision="mixed", tol=1e-11)
        V, W = ctx.rigid_velocities()
        return {"V": V, "W": W, "u": ctx.eval_velocity(st["x"])}
    ctx.set_rigid_velocities(st["v"], st["w"])
    ctx.solve(precision="mixed", tol=1e-11)
    F, T = ctx.forces_torques()
    return {"F": F, "T": T, "u": ctx.eval_velocity(st["x"])}


# ---------------------------------------------------------------- the same formulas in 64-bit torch
def _fib(n, cos_t):
    j = np.arange(1, n + 1)
    sin_t = np.sqrt(np.maximum(0.0, 1.0 - cos_t ** 2))
    phi = np.mod(2.0 * math.pi * j / 1.6180339887498948482, 2.0 * math.pi)
    return np.stack([sin_t * np.cos(phi), sin_t * np.sin(phi), cos_t], axis=1)


def _grid(n):
    return _fib(n, 1.0 - (2.0 * np.arange(1, n + 1) - 1.0) / n)


def _images(delta, nim_fixed):
    if delta >= 0.15:
        return 0
    return nim_fixed if nim_fixed >= 0 else min(20, max(0, math.ceil(-8.72 * math.log10(delta) - 6.15)))


def _discretise(case, centres):
    """Per unit sphere: nodes and images relative to the centre, area weights; the proxies are common."""
    proxy, basic = case["r_proxy"] * _grid(case["N"]), _grid(case["M0"])
    t0, nim_fixed = case["r_proxy"] * 1.05, _params(case).get("nim_fixed", -1)
    out = []
    for k in range(len(centres)):
        x, w, img = [basic], [np.full(len(basic), 4 * math.pi / len(basic))], []
        d = centres - centres[k]
        dist = np.linalg.norm(d, axis=1)
        for kp in np.nonzero((dist > 0) & (dist - 2.0 < 0.15))[0]:
            delta = dist[kp] - 2.0
            nim = _images(delta, nim_fixed)
            if nim == 0:
                continue
            e = d[kp] / dist[kp]
            h = np.array([0.0, 0.0, 1.0]) if abs(e[2]) <= 0.9 else np.array([1.0, 0.0, 0.0])
            e1 = h - (h @ e) * e
            e1 /= np.linalg.norm(e1)
            e2 = np.cross(e, e1)
            racc = 1.0 + 0.5 * delta - math.sqrt(delta + 0.25 * delta * delta)
            t = t0 + (racc - t0) * np.cos(np.arange(nim) / (2.0 * nim) * math.pi)
            img.append(t[:, None] * e[None])
            m = 18 * nim
            for beta in (math.pi / 5, math.pi / 60):
                c = _fib(m, 1.0 - np.arange(1, m + 1) * (1.0 - math.cos(beta)) / m)
                x.append(c[:, :1] * e1 + c[:, 1:2] * e2 + c[:, 2:] * e)
                w.append(np.full(m, 2 * math.pi * (1.0 - math.cos(beta)) / m))
        out.append(dict(x=np.concatenate(x), w=np.sqrt(np.concatenate(w)), proxy=proxy,
                        img=np.concatenate(img) if img else np.zeros((0, 3))))
    return out


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


def _field(x, sph, lam, shift):
    """Velocity at targets x (n, 3) of one sphere's strengths; shift: target frame minus sphere centre."""
    N = sph["proxy"].shape[0]
    u = torch.zeros_like(x)
    f = lam[: 3 * N].view(N, 3)
    img = lam[3 * N:].view(-1, 9)
    step = max(1, (1 << 25) // max(1, N))
    for a in range(0, x.shape[0], step):
        xs = x[a: a + step] + shift
        for y, s in ((_t(sph["proxy"]), f), (_t(sph["img"]), img)):
            if len(y) == 0:
                continue
            r = xs[:, None] - y[None]
            ir2 = 1.0 / (r * r).sum(2)
            ir = ir2.sqrt()
            rf = (r * s[None, :, :3]).sum(2)
            v = ir @ s[:, :3] + ((rf * ir * ir2)[..., None] * r).sum(1)
            if s.shape[1] == 9:
                ir3 = ir * ir2
                v += (ir3[..., None] * torch.cross(s[None, :, 3:6].expand_as(r), r, dim=2)).sum(1)
                q = s[:, 6:]
                v += 2.0 * (-(ir3 @ q) + 3.0 * (((r * q[None]).sum(2) * ir3 * ir2)[..., None] * r).sum(1))
            u[a: a + step] += v / (8.0 * math.pi)
    return u


def _matrix(x, sph, shift):
    """Dense (3 n, 3 N_k) block of one sphere's sources at targets x, columns in the strength order."""
    eye = torch.eye(3, dtype=torch.float64, device=DEV)
    r = (x + shift)[:, None] - _t(sph["proxy"])[None]
    ir = (r * r).sum(2).rsqrt()[..., None, None]
    rr = r[..., :, None] * r[..., None, :]
    cols = [((eye * ir + rr * ir ** 3) / (8 * math.pi)).permute(0, 2, 1, 3).reshape(3 * len(x), -1)]
    if len(sph["img"]):
        r = (x + shift)[:, None] - _t(sph["img"])[None]
        ir = (r * r).sum(2).rsqrt()[..., None, None]
        rr = r[..., :, None] * r[..., None, :]
        z = torch.zeros_like(r[..., 0])
        cr = torch.stack([torch.stack([z, r[..., 2], -r[..., 1]], -1), torch.stack([-r[..., 2], z, r[..., 0]], -1),
                          torch.stack([r[..., 1], -r[..., 0], z], -1)], -2)
        blk = torch.cat([(eye * ir + rr * ir ** 3) / (8 * math.pi), cr * ir ** 3 / (8 * math.pi),
                         (-eye * ir ** 3 + 3 * rr * ir ** 5) / (4 * math.pi)], -1)
        cols.append(blk.permute(0, 2, 1, 3).reshape(3 * len(x), -1))
    return torch.cat(cols, 1)


def _pinv(sph):
    """(Sigma^+ U^T, V) of the scaled self block, truncated."""
    b = _t(np.repeat(sph["w"], 3))[:, None] * _matrix(_t(sph["x"]), sph, 0.0)
    q, r = torch.linalg.qr(b)
    if r.is_cuda:
        u, s, vh = torch.linalg.svd(r, full_matrices=False, driver="gesvd")
    else:
        u, s, vh = torch.linalg.svd(r, full_matrices=False)
    k = s >= EPS_TRUNC * s.max()
    return ((q @ u[:, k]) / s[k]).T.contiguous(), vh[k].T.contiguous()


class _System:
    """The preconditioned operator, its parts and the solve, for one geometry."""

    def __init__(self, case, centres, factors=True, dense=False):
        self.case, self.c, self.sph = case, centres, _discretise(case, centres)
        self.P = len(centres)
        self.x = [_t(s["x"]) for s in self.sph]
        self.w = [_t(s["w"]) for s in self.sph]
        self.off = np.cumsum([0] + [3 * len(s["x"]) for s in self.sph])
        self.uoff = np.cumsum([0] + [3 * case["N"] + 9 * len(s["img"]) for s in self.sph])
        self.f = []
        if factors:
            basic = None
            for s in self.sph:
                if len(s["img"]) == 0 and basic is not None:
                    self.f.append(basic)
                    continue
                self.f.append(_pinv(s))
                basic = self.f[-1] if len(s["img"]) == 0 else basic
        self.g = None
        if dense:
            self.g = [torch.cat([torch.zeros(3 * len(self.x[k]), int(self.uoff[q + 1] - self.uoff[q]), dtype=torch.float64,
                                             device=DEV) if q == k else
                                 self.w[k].repeat_interleave(3)[:, None] * _matrix(self.x[k], self.sph[q], self.shift(k, q))
                                 for q in range(self.P)], 1) for k in range(self.P)]

    def shift(self, k, q):
        return _t(self.c[k] - self.c[q])

    def split(self, v):
        return [v[self.off[k]: self.off[k + 1]] for k in range(self.P)]

    def precond(self, mu):
        return torch.cat([f[1] @ (f[0] @ m) for f, m in zip(self.f, self.split(mu))])

    def pairs(self, lam, mu):
        if self.g is not None:
            return mu + torch.cat([g @ lam for g in self.g])
        out = []
        for k, m in enumerate(self.split(mu)):
            u = torch.zeros_like(self.x[k])
            for q in range(self.P):
                if q != k:
                    u += _field(self.x[k], self.sph[q], lam[self.uoff[q]: self.uoff[q + 1]], self.shift(k, q))
            out.append(m + (self.w[k][:, None] * u).reshape(-1))
        return torch.cat(out)

    def rhs(self, v, w):
        out = []
        for k in range(self.P):
            om = _t(w[k])[None].expand_as(self.x[k])
            out.append((self.w[k][:, None] * (_t(v[k]) + torch.cross(om, self.x[k], dim=1))).reshape(-1))
        return torch.cat(out)

    def forces(self, lam):
        F, T = [], []
        for k, s in enumerate(self.sph):
            l, N = lam[self.uoff[k]: self.uoff[k + 1]], self.case["N"]
            f, img = l[: 3 * N].view(N, 3), l[3 * N:].view(-1, 9)
            F.append(f.sum(0) + img[:, :3].sum(0))
            T.append(torch.cross(_t(s["proxy"]), f, dim=1).sum(0) + img[:, 3:6].sum(0) +
                     torch.cross(_t(s["img"]), img[:, :3], dim=1).sum(0))
        return torch.stack(F), torch.stack(T)

    def velocity(self, lam, x):
        x = _t(x)
        return sum(_field(x, self.sph[q], lam[self.uoff[q]: self.uoff[q + 1]], -_t(self.c[q])) for q in range(self.P))

    def solve(self, v, w, mobility):
        """(lambda, V, Omega): resistance for rigid velocities v, w, or mobility for forces v and torques w."""
        n, P = int(self.off[-1]), self.P
        sF, sT = 1.0 / (6 * math.pi), 1.0 / (8 * math.pi)
        if not mobility:
            lam = self.precond(_gmres(lambda m: self.pairs(self.precond(m), m), self.rhs(v, w)))
            return lam, None, None

        def op(z):
            lam, U = self.precond(z[:n]), z[n:].view(P, 6)
            F, T = self.forces(lam)
            return torch.cat([self.pairs(lam, z[:n]) - self.rhs(U[:, :3].cpu().numpy(), U[:, 3:].cpu().numpy()),
                              torch.cat([sF * F, sT * T], 1).reshape(-1)])

        b = torch.cat([torch.zeros(n, dtype=torch.float64, device=DEV), torch.cat([sF * _t(v), sT * _t(w)], 1).reshape(-1)])
        z = _gmres(op, b)
        return self.precond(z[:n]), z[n:].view(P, 6)[:, :3], z[n:].view(P, 6)[:, 3:]


def _gmres(op, b, tol=1e-13, restart=160, cycles=3):
    x = torch.zeros_like(b)
    for _ in range(cycles):
        r = b - op(x)
        beta = float(r.norm())
        if beta <= tol * float(b.norm()):
            break
        V, H = [r / beta], np.zeros((restart + 1, restart))
        for j in range(restart):
            w = op(V[j])
            for _ in range(2):
                h = torch.stack(V) @ w
                w = w - h @ torch.stack(V)
                H[: j + 1, j] += h.cpu().numpy()
            H[j + 1, j] = float(w.norm())
            e = np.zeros(j + 2)
            e[0] = beta
            y, *_ = np.linalg.lstsq(H[: j + 2, : j + 1], e, rcond=None)
            V.append(w / H[j + 1, j])
            if np.linalg.norm(H[: j + 2, : j + 1] @ y - e) <= 0.3 * tol * float(b.norm()):
                break
        x = x + torch.stack(V[:-1]).T @ _t(y)
    return x


def _pair_count(sph):
    """(node, proxy) pairs and (node, image node) triples of one application, self blocks left out."""
    nodes, imgs = [len(s["x"]) for s in sph], [len(s["img"]) for s in sph]
    N = len(sph[0]["proxy"])
    return sum(nodes) * (len(sph) - 1) * N, sum(m * (sum(imgs) - i) for m, i in zip(nodes, imgs))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        rng = np.random.default_rng([seed, 20240703])
        F, T = [], []
        for gap in _gaps(case):
            s = _System(dict(case, shape="two"), workloads.two_spheres(gap), dense=True)
            for _ in range(3):
                f, t = s.forces(s.solve(rng.normal(size=(2, 3)), rng.normal(size=(2, 3)), False)[0])
                F.append(f)
                T.append(t)
        return {"F": torch.stack(F), "T": torch.stack(T)}
    centres = _centres(case)
    vec = _vectors(case, centres, seed)
    if kind in ("pairs", "operator") and _pair_count(_discretise(case, centres))[0] > 1.4e10:
        return None  # minutes in 64 bits
    if kind in ("solve", "velocity"):
        s = _System(case, centres, dense=True)
        lam, V, W = s.solve(vec["v"], vec["w"], case.get("mobility", False))
        u = s.velocity(lam, vec["x"])
        if kind == "velocity":
            return u
        if case["mobility"]:
            return {"V": V, "W": W, "u": u}
        F, T = s.forces(lam)
        return {"F": F, "T": T, "u": u}
    s = _System(case, centres, factors=kind != "pairs")
    if kind == "pairs":
        lam = _t(vec["rng"].normal(size=int(s.uoff[-1])))
        return s.pairs(lam, _t(vec["rng"].normal(size=int(s.off[-1]))))
    if kind == "operator":
        mu = s.rhs(vec["v"], vec["w"])
        mu = mu / mu.norm()
        return s.pairs(s.precond(mu), mu)
    return s.precond(_t(vec["rng"].normal(size=int(s.off[-1]))))


# ---------------------------------------------------------------- work that cannot be avoided
def _step1_elements(case, sph):
    """Entries of the distinct factors Sigma^+ U^T and V (full rank) and of all spheres' products."""
    a = v = pa = pv = 0
    seen = False
    for s in sph:
        cols, rows = 3 * case["N"] + 9 * len(s["img"]), 3 * len(s["x"])
        pa, pv = pa + cols * rows, pv + cols * cols
        if len(s["img"]) == 0:
            if seen:
                continue
            seen = True
        a, v = a + cols * rows, v + cols * cols
    return a, v, pa, pv


def work(case):
    """Bytes and flops of one pass.  A (node, Stokeslet) pair counts 28 flops and a (node, image)
    triple 63, the paths' own convention; factors are read once in the form their mode stores
    (8 bytes an entry, 4 for Sigma^+ U^T inside the passes).  The whole calls count the
    operator applications that a solve to 1e-11 of such a geometry needs (~50 for the dilute
    suspensions, ~35 for the pairs)."""
    kind = case["kind"]
    if kind == "batch":
        n = f = 0
        for gap in _gaps(case):
            sph = _discretise(dict(case, shape="two"), workloads.two_spheres(gap))
            a, v, pa, pv = _step1_elements(case, sph)
            pp, pi = _pair_count(sph)
            n += 35 * (4 * a + 8 * v)
            f += 35 * 3 * (2 * (pa + pv) + 28 * pp + 63 * pi)
        return {"bytes": n, "flops": f}
    centres = _centres(case)
    sph = _discretise(case, centres)
    nodes = sum(len(s["x"]) for s in sph)
    unk = sum(3 * case["N"] + 9 * len(s["img"]) for s in sph)
    pp, pi = _pair_count(sph)
    a, v, pa, pv = _step1_elements(case, sph)
    per_a = 4 if case.get("precision") == "pass" else 8
    if kind == "pairs":
        return {"bytes": 8 * (6 * nodes + unk), "flops": 28 * pp + 63 * pi}
    if kind in ("precond", "noalloc"):
        return {"bytes": per_a * a + 8 * v + 8 * (3 * nodes + unk), "flops": 2 * (pa + pv)}
    if kind == "operator":
        return {"bytes": per_a * a + 8 * v + 8 * 6 * nodes, "flops": 2 * (pa + pv) + 28 * pp + 63 * pi}
    points = {"bytes": 48 * case["points"] + 8 * unk, "flops": 28 * case["points"] * case["P"] * case["N"]}
    if kind == "velocity":
        return points
    return {"bytes": points["bytes"] + 50 * (4 * a + 8 * v),
            "flops": points["flops"] + 50 * (2 * (pa + pv) + 28 * pp + 63 * pi)}
