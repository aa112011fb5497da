"""Performance cases of the rigid-particle mobility library: what its users call, and how much it costs.

A case is one call (or a short sequence) of the public entry points in paper_1606_07428_gb300.rbs on
seeded particles: mobility solves in each precision and far-field option over the range of sizes, one
time step, the magnetic forces, one operator application, and a solve on a new geometry with its
set-up.  `exact` restates the discretisation in float64 torch, independently of the library, so that the
error of every result can be told.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1606_07428_gb300 import rbs

TOL = 1e-10  # rbs_advance's default tolerance in the binding; the full-size parity tests solve to it too
H0 = 10.0 / math.sqrt(3.0) * np.array([1.0, -1.0, -1.0])  # the field of the magnetorheological set-up
MU_RATIO = 2.0
DT = 0.01
DF_DEFAULTS = {"df_theta": 0.4, "df_degree": 12}


def listed():
    return [
        # the smallest call: a handful of spheres, where launches and latency are the time (the
        # repository's 8-sphere workload)
        _case("spheres_8", kind="solve", body="spheres", n=8, p=8),
        # the plain float64 solve, which users without a need for speed (and references) run
        _case("float64_60", kind="solve", n=60, p=8, precision="float64"),
        # an ordinary suspension with the float32 treecode and exact double-float passes (400 ellipsoids,
        # the repository's profiling size)
        _case("ellipsoids_400", kind="solve", n=400, p=8, far="tree"),
        # finer grids, with both treecodes at the library's default accuracy
        _case("ellipsoids_700_p12", kind="solve", n=700, p=12, far="tree-df"),
        # a dense suspension at the benchmark's grid, fraction and treecode settings; the largest case
        _case("dense_1500", kind="solve", n=1500, p=8, fill=0.145, far="tree-df", df_theta=0.45, df_degree=11),
        # many independent suspensions of mixed sizes and orders in one context
        _case("batch_24", kind="solve", n=24, p=0, batch=24, far="direct"),
        # particles of one shape with float16 self blocks: the tensor-core block path
        _case("same_shape_600_fp16", kind="solve", body="same", n=600, p=8, precision="mixed-fp16", far="tree"),
        # general surfaces given by spherical-harmonic coefficients (full self blocks)
        _case("surfaces_40_p10", kind="solve", body="surfaces", n=40, p=10),
        # one RK4 step of sedimenting ellipsoids through the host-buffer call, each stage from the last
        # density (odd particle count, the sedimentation workloads' 11 x 22 grid)
        _case("step_101_p10", kind="step", n=101, p=10, nphi=22),
        # magnetic forces on paramagnetic particles in a uniform field (the set-up of the paper's Fig. 1;
        # ellipsoids, since a sphere's torque is zero)
        _case("magnetic_216", kind="magnetic", n=216, p=8),
        # one double-float application of the system operator, as a residual check does it
        _case("operator_500_p10", kind="operator", n=500, p=10, nphi=22),
        # a suspension never seen before: set-up of every shape's blocks, then one solve
        _case("new_geometry_64_p12", kind="geometry", n=64, p=12),
    ]


def _case(name, kind, n, p, nphi=0, body="ellipsoids", fill=0.10, precision="mixed", far="direct", batch=0,
          df_theta=0.4, df_degree=12):
    c = dict(kind=kind, body=body, n=n, p=p, nphi=nphi or 2 * p, fill=fill, precision=precision, far=far,
             batch=batch, df_theta=df_theta, df_degree=df_degree)
    if name:
        c["name"] = name
    return c


def draw(rng):
    """A case of the same ranges: sizes over their logarithm, odd counts among them, p of the grids that
    the workloads use."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["small", "tree", "tree", "tree-df", "tree-df", "batch", "fp16", "surfaces", "step",
                       "magnetic", "operator", "geometry", "float64"])
    if kind == "small":
        return _case("", "solve", n=logint(2, 90), p=rng.choice([6, 8, 10, 12]), fill=rng.choice([0.05, 0.10, 0.14]))
    if kind == "tree":
        return _case("", "solve", n=logint(100, 700), p=rng.choice([6, 8, 10]), far="tree")
    if kind == "tree-df":
        p = rng.choice([6, 8, 10, 12])
        return _case("", "solve", n=logint(250, 1200 if p <= 8 else 500), p=p, far="tree-df",
                     fill=rng.choice([0.06, 0.10, 0.14]), **rng.choice([DF_DEFAULTS, {"df_theta": 0.45, "df_degree": 11}]))
    if kind == "batch":
        k = logint(4, 40)
        return _case("", "solve", n=k, p=0, batch=k, far=rng.choice(["direct", "tree"]))
    if kind == "fp16":
        return _case("", "solve", body="same", n=logint(64, 900), p=rng.choice([6, 8]), precision="mixed-fp16", far="tree")
    if kind == "surfaces":
        return _case("", "solve", body="surfaces", n=logint(4, 60), p=rng.choice([6, 8, 10]))
    if kind == "step":
        return _case("", "step", n=logint(9, 160), p=10, nphi=22)
    if kind == "magnetic":
        return _case("", "magnetic", n=logint(8, 343), p=8)
    if kind == "operator":
        p = rng.choice([6, 8, 10, 12])
        return _case("", "operator", n=logint(30, 600), p=p, nphi=2 * p + rng.choice([0, 2]))
    if kind == "geometry":
        return _case("", "geometry", n=logint(8, 80), p=rng.choice([6, 8, 10, 12]))
    return _case("", "solve", n=logint(6, 90), p=rng.choice([6, 8]), precision="float64")


# ---------------------------------------------------------------------------------------------- inputs

def _quaternions(rng, n):
    q = rng.normal(size=(n, 4))
    return q / np.linalg.norm(q, axis=1, keepdims=True)


def _lattice(rng, n, fill, radius):
    """Centres on a randomly occupied cubic lattice of the given volume fraction (particles of mean volume
    4 pi / 3), moved by as much as keeps bounding spheres of the given radius 0.2 apart."""
    m = math.ceil(n ** (1 / 3) - 1e-9)
    need = 2 * radius + 0.2
    spacing = max(need + 0.02, (4 * math.pi / 3 / fill) ** (1 / 3))
    sites = np.stack(np.meshgrid(*[np.arange(m) * spacing] * 3, indexing="ij"), -1).reshape(-1, 3)
    sites = sites[np.sort(rng.permutation(m ** 3)[:n])]
    jitter = 0.5 * (spacing - need)
    return sites - sites.mean(0) + rng.uniform(-jitter, jitter, size=(n, 3))


def _particles(case, seed):
    """Everything a user's program knows of the particles, as numpy arrays."""
    rng = np.random.default_rng([seed, 7])
    body, n = case["body"], case["n"]
    if case["batch"]:  # sizes and orders as in the batched workload, the same ones for every seed
        layout = np.random.default_rng(case["batch"])
        sizes = np.floor(np.exp(layout.uniform(math.log(4), math.log(49), size=case["batch"]))).astype(int)
        sid = np.repeat(np.arange(case["batch"]), sizes)
        n = len(sid)
        p = layout.choice(np.array([6, 8, 12, 16], np.int32), size=n).astype(np.int32)
        nphi = (2 * p).astype(np.int32)
    else:
        sid, sizes = None, [n]
        p = np.full(n, case["p"], np.int32)
        nphi = np.full(n, case["nphi"], np.int32)
    s = {"p": p, "nphi": nphi, "sid": sid, "n": n, "quats": _quaternions(rng, n), "shapes": None, "shape_of": None}
    radius = 1.4
    if body == "spheres":
        s["axes"], s["quats"], radius = np.ones((n, 3)), np.tile([1.0, 0, 0, 0], (n, 1)), 1.0
    elif body == "same":  # the shape of the paper's ellipsoid lattices
        s["axes"], radius = np.tile([1.0, 0.5, 0.5], (n, 1)), 1.0
    elif body == "surfaces":  # a few smooth shapes, each carried by several particles
        s["shapes"] = [_surface(rng) for _ in range(1 + n // 8)]
        s["shape_of"] = rng.integers(0, len(s["shapes"]), n).astype(np.int32)
        s["axes"] = None
    else:
        s["axes"] = rng.uniform(0.6, 1.4, size=(n, 3))
    s["centres"] = np.concatenate([_lattice(rng, int(k), case["fill"], radius) for k in sizes])
    if case["kind"] == "step":
        s["F"], s["T"] = np.tile([0.0, 0.0, -1.0], (n, 1)), np.zeros((n, 3))
    else:
        s["F"], s["T"] = rng.normal(size=(n, 3)), rng.normal(size=(n, 3))
    return s


def _surface(rng):
    """Coefficients (3, 16) of a degree-3 surface in the library's basis order: an ellipsoid with small
    random harmonics of degree 2 and 3."""
    order = [(d, m) for m in range(4) for d in range(m, 4) for _ in range(1 if m == 0 else 2)]
    degree = np.array([d for d, _ in order])
    coef = np.where(degree[None, :] >= 2, 0.02 * rng.normal(size=(3, 16)), 0.0)
    unit = math.sqrt(4 * math.pi / 3)
    axes = rng.uniform(0.8, 1.2, 3)
    at = {(1, 0): order.index((1, 0)), (1, 1): order.index((1, 1))}
    coef[0, at[1, 1]] = axes[0] * unit
    coef[1, at[1, 1] + 1] = axes[1] * unit
    coef[2, at[1, 0]] = axes[2] * unit
    return coef, 3


PRECISION = {"float64": rbs.RBS_PREC_FP64, "mixed": rbs.RBS_PREC_MIXED, "mixed-fp16": rbs.RBS_PREC_MIXED_FP16}
FAR = {"direct": rbs.RBS_FAR_DIRECT, "tree": rbs.RBS_FAR_TREECODE, "tree-df": rbs.RBS_FAR_TREECODE_DF}


def _set_geometry(ctx, s):
    if s["shapes"] is not None:
        ctx.set_shapes(s["shapes"], s["shape_of"], s["p"], s["nphi"], s["centres"], s["quats"], s["sid"])
    else:
        ctx.set_geometry(s["axes"], s["p"], s["nphi"], s["centres"], s["quats"], s["sid"])


def prepare(case, seed):
    """The context with its geometry (but for a new geometry, which `run` sets), forces, and the buffers
    that results go to."""
    s = _particles(case, seed)
    kw = {"warm_start": rbs.RBS_WARM_PREVIOUS} if case["kind"] == "step" else {}
    ctx = rbs.Context(precision=PRECISION[case["precision"]], far_field=FAR[case["far"]],
                      tree_df_theta=case["df_theta"], tree_df_degree=case["df_degree"], **kw)
    nodes = int(((s["p"] + 1) * s["nphi"]).sum())
    s |= {"case": case, "ctx": ctx, "nodes": nodes}
    if case["kind"] != "geometry":
        _set_geometry(ctx, s)
    if case["kind"] in ("solve", "geometry"):
        s["F_dev"], s["T_dev"] = torch.tensor(s["F"], device="cuda"), torch.tensor(s["T"], device="cuda")
        s["v"], s["omega"] = torch.empty_like(s["F_dev"]), torch.empty_like(s["F_dev"])
        s["mu"] = torch.empty((nodes, 3), dtype=torch.float64, device="cuda")
    elif case["kind"] == "operator":
        s["x"] = _density(case, seed, nodes)
        s["y"] = torch.empty_like(s["x"])
    torch.cuda.synchronize()
    return s


def _density(case, seed, nodes):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((nodes, 3), dtype=torch.float64, device="cuda", generator=g)


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"].ctx
    if kind in ("solve", "geometry"):
        if kind == "geometry":
            _set_geometry(s["ctx"], s)
        rbs.rbs_mobility_solve_device(ctx, s["F_dev"], s["T_dev"], TOL, s["v"], s["omega"], s["mu"])
        return {"v": s["v"], "omega": s["omega"], "mu": s["mu"]}
    if kind == "step":
        rbs.rbs_advance(ctx, s["F"], s["T"], DT, 1, rbs.RBS_RK4, TOL)
        centres, quats = rbs.rbs_get_state(ctx, s["n"])
        return {"centres": centres, "quats": quats}
    if kind == "magnetic":
        F, T, q, _ = rbs.rbs_magnetic_forces(ctx, H0, MU_RATIO, TOL, s["n"], s["nodes"])
        return {"F": F, "T": T, "q": q}
    rbs.rbs_apply_operator_device(ctx, rbs.RBS_OP_A, rbs.RBS_PREC_DF, s["x"], s["y"])
    return {"y": s["y"]}


# ---------------------------------------------------------------------------------------------- work

def work(case):
    """Bytes: inputs read and results written once, and each distinct shape's self block once.  Flops: the
    pair sums and the block products of the fewest operator applications that a solve to the tolerance takes
    (about 15 of the traction operator and one of the Stokeslet), direct sums over all nodes of a suspension, or,
    with a treecode, over a target's neighbourhood of 27 particles and a dozen clusters per level."""
    if case["batch"]:
        n, nodes_of = 18 * case["batch"], 220.0
        targets, sources = n * nodes_of, 30 * nodes_of
    else:
        n, nodes_of = case["n"], float((case["p"] + 1) * case["nphi"])
        targets, sources = n * nodes_of, n * nodes_of
        if case["far"] != "direct":
            sources = min(sources, 27 * nodes_of + 512 * 12 * math.log2(max(2, n)))
    block = (3 * nodes_of) ** 2
    shapes = 1 if case["body"] in ("spheres", "same") else (1 + n // 8 if case["body"] == "surfaces" else n)
    entry = {"float64": 8, "mixed": 4, "mixed-fp16": 2}[case["precision"]]
    one = targets * sources * 29 + n * 2 * block
    kind = case["kind"]
    if kind == "operator":
        return {"bytes": targets * (24 + 24 + 56) + shapes * block / 6 * 8, "flops": one}
    if kind == "magnetic":
        return {"bytes": targets * 56 + n * 48, "flops": 8 * targets * (sources * 14 + 2 * nodes_of)}
    solves = 4 if kind == "step" else 1
    flops = solves * 16 * one
    if kind == "geometry":  # singular quadrature of two kernels at a sixth of the targets, interpolated to the grid
        p = case["p"]
        flops += n * nodes_of / 6 * 18 * (2 * p + 1) * (4 * p + 2) * 2 * (p + 1) ** 2
    return {"bytes": solves * (n * 96 + targets * (24 + 56)) + shapes * block / 6 * entry * 2, "flops": flops}


# ---------------------------------------------------------------------------------------------- float64 restatement

def exact(case, seed):
    s = _particles(case, seed)
    per = (s["p"] + 1) * s["nphi"]
    nodes = int(per.sum())
    pairs = float((np.bincount(s["sid"], per) ** 2).sum()) if s["sid"] is not None else float(nodes) ** 2
    if pairs > (2e10 if case["kind"] == "operator" else 5e9):
        return None  # over 20 seconds
    ref = _Reference(s)
    kind = case["kind"]
    if kind in ("solve", "geometry"):
        v, omega, mu = ref.solve(s["F"], s["T"])
        return {"v": v, "omega": omega, "mu": mu}
    if kind == "operator":
        x = _density(case, seed, nodes)
        return {"y": ref.apply("K", x, half=0.5, with_L=True)}
    if kind == "magnetic":
        F, T, q = ref.magnetic(H0, MU_RATIO)
        return {"F": F.cpu().numpy(), "T": T.cpu().numpy(), "q": q.cpu().numpy()}
    c = torch.tensor(s["centres"], device="cuda")
    q = torch.tensor(s["quats"], device="cuda")
    kc, kq, x0 = [], [], None
    for a in (0.0, 0.5, 0.5, 1.0):  # classical RK4 of dc/dt = v, dq/dt = (0, omega) q / 2
        cs, qs = (c + DT * a * kc[-1], q + DT * a * kq[-1]) if kc else (c, q)
        ref.place(cs, qs)
        v, w, x0 = ref.solve(s["F"], s["T"], x0)
        kc.append(v)
        kq.append(0.5 * torch.cat([-(w * qs[:, 1:]).sum(1, keepdim=True),
                                   w * qs[:, :1] + torch.linalg.cross(w, qs[:, 1:])], 1))
    c = c + DT / 6 * (kc[0] + 2 * kc[1] + 2 * kc[2] + kc[3])
    q = q + DT / 6 * (kq[0] + 2 * kq[1] + 2 * kq[2] + kq[3])
    return {"centres": c.cpu().numpy(), "quats": (q / q.norm(dim=1, keepdim=True)).cpu().numpy()}


def _harmonics(p, mmax, u):
    """Real orthonormal harmonics at unit vectors u (M, 3) and their derivatives d/dtheta and
    (d/dphi) / sin(theta): three (B, M) tensors in the order m = 0.., n = m.., cosine then sine."""
    ct = u[:, 2]
    st = torch.hypot(u[:, 0], u[:, 1])
    phi = torch.atan2(u[:, 1], u[:, 0])
    P = {}  # P[n, m] / sin(theta) for m >= 1, P[n, 0] itself
    P[0, 0] = torch.full_like(ct, 1 / math.sqrt(4 * math.pi))
    for m in range(0, p + 1):
        if m == 1:
            P[1, 1] = math.sqrt(1.5) * P[0, 0]
        elif m > 1:
            P[m, m] = math.sqrt((2 * m + 1) / (2 * m)) * st * P[m - 1, m - 1]
        for n in range(m + 1, p + 1):
            a = math.sqrt((4 * n * n - 1) / (n * n - m * m))
            low = P[n - 2, m] * math.sqrt(((n - 1) ** 2 - m * m) / (4 * (n - 1) ** 2 - 1)) if n > m + 1 else 0
            P[n, m] = a * (ct * P[n - 1, m] - low)
    Y, Yt, Yp = [], [], []
    for m in range(0, mmax + 1):
        for n in range(m, p + 1):
            if m == 0:
                Y.append(P[n, 0])
                Yt.append(-math.sqrt(n * (n + 1)) * st * P[n, 1] if n else torch.zeros_like(ct))
                Yp.append(torch.zeros_like(ct))
                continue
            c, s = math.sqrt(2) * torch.cos(m * phi), math.sqrt(2) * torch.sin(m * phi)
            low = math.sqrt((2 * n + 1) / (2 * n - 1) * (n * n - m * m)) * P[n - 1, m] if n > m else 0
            dt = n * ct * P[n, m] - low
            Y += [st * P[n, m] * c, st * P[n, m] * s]
            Yt += [dt * c, dt * s]
            Yp += [-m * P[n, m] * s, m * P[n, m] * c]
    return torch.stack(Y), torch.stack(Yt), torch.stack(Yp)


def _dev(a):
    return torch.tensor(np.asarray(a, np.float64), device="cuda")


def _sphere_grid(p, nphi):
    """Unit vectors (N, 3) and solid-angle weights of the Gauss-Legendre x uniform grid."""
    t, lam = np.polynomial.legendre.leggauss(p + 1)
    st = np.sqrt(1 - t * t)
    phi = 2 * math.pi * np.arange(nphi) / nphi
    u = np.stack([np.outer(st, np.cos(phi)), np.outer(st, np.sin(phi)), np.outer(t, np.ones(nphi))], -1)
    return _dev(u.reshape(-1, 3)), _dev(np.repeat(lam, nphi) * 2 * math.pi / nphi)


class _Grid:
    """One (p, n_phi) grid: nodes, analysis, upsampled grid and the rotated-pole rule of every node."""

    def __init__(self, p, nphi):
        self.p, self.nphi, self.np = p, nphi, (p + 1) * nphi
        self.mmax = min(p, (nphi - 1) // 2)
        self.u, q = _sphere_grid(p, nphi)
        self.q = q
        self.Y, self.Yt, self.Yp = _harmonics(p, self.mmax, self.u)
        self.An = self.Y * q
        self.u_up, self.q_up = _sphere_grid(2 * p, nphi + 2 * p)
        self.up = _harmonics(p, self.mmax, self.u_up)[0].T @ self.An
        ps, nb = 2 * p, 4 * p + 2
        x, lam = np.polynomial.legendre.leggauss(ps + 1)
        th, ph = 0.5 * math.pi * (x + 1), 2 * math.pi * np.arange(nb) / nb
        pole = np.stack([np.outer(np.sin(th), np.cos(ph)), np.outer(np.sin(th), np.sin(ph)),
                         np.outer(np.cos(th), np.ones(nb))], -1).reshape(-1, 3)
        self.rule = _dev(np.repeat(0.5 * math.pi * lam * np.sin(th) * 2 * math.pi / nb, nb))
        self.pole = _dev(pole)

    def rotated(self):
        """Per node t: the rule's points (M, 3) around it and their interpolation matrix (M, N).  The nodes of
        one latitude share the matrix but for a shift of its columns."""
        for j in range(self.p + 1):
            z = float(self.u[j * self.nphi, 2])
            st = math.sqrt(1 - z * z)
            interp = _harmonics(self.p, self.mmax, self.pole @ _dev([[z, 0, -st], [0, 1, 0], [st, 0, z]]))[0].T @ self.An
            for k in range(self.nphi):
                c, s = math.cos(2 * math.pi * k / self.nphi), math.sin(2 * math.pi * k / self.nphi)
                rot = _dev([[c * z, -s, c * st], [s * z, c, s * st], [-st, 0.0, z]])
                shifted = interp.reshape(-1, self.p + 1, self.nphi).roll(k, dims=2)
                yield j * self.nphi + k, self.pole @ rot.T, shifted.reshape(interp.shape)


class _Reference:
    """The discretised operators on the particles of _particles, in float64."""

    def __init__(self, s):
        self.s, self.n = s, s["n"]
        self.sid = np.zeros(self.n, int) if s["sid"] is None else s["sid"]
        keys = list(zip(s["p"].tolist(), s["nphi"].tolist()))
        self.grids = {k: _Grid(*k) for k in set(keys)}
        self.grid = [self.grids[k] for k in keys]
        self.off = np.concatenate([[0], np.cumsum([g.np for g in self.grid])])
        self.members = {k: [i for i in range(self.n) if keys[i] == k] for k in self.grids}
        self.blocks = {}
        # body frames
        self.shift = torch.zeros((self.n, 3), dtype=torch.float64, device="cuda")
        if s["axes"] is None:
            for k, ids in self.members.items():
                x, J, _ = self._surface(ids, self.grids[k].u)
                w = J * self.grids[k].q
                self.shift[ids] = (w[..., None] * x).sum(1) / w.sum(1, keepdim=True)
        self.radius = np.zeros(self.n)
        self.body = [None] * self.n
        self.body_up = [None] * self.n
        for k, ids in self.members.items():
            g = self.grids[k]
            x, J, nrm = self._surface(ids, g.u)
            xu, Ju, _ = self._surface(ids, g.u_up)
            for a, i in enumerate(ids):
                self.body[i] = (x[a], J[a] * g.q, nrm[a])
                self.body_up[i] = (xu[a], Ju[a] * g.q_up)
                self.radius[i] = s["axes"][i].max() if s["axes"] is not None else float(xu[a].norm(dim=1).max())
        self.place(_dev(s["centres"]), _dev(s["quats"]))

    def _surface(self, ids, u):
        """Body points (k, M, 3), area per solid angle (k, M) and normals at parameter points u."""
        if self.s["axes"] is not None:
            ax = _dev(self.s["axes"][ids])[:, None, :]
            cof = torch.stack([ax[..., 1] * ax[..., 2], ax[..., 0] * ax[..., 2], ax[..., 0] * ax[..., 1]], -1) * u
            J = cof.norm(dim=-1)
            return ax * u, J, cof / J[..., None]
        Y, Yt, Yp = _harmonics(3, 3, u)
        coef = _dev(np.stack([self.s["shapes"][self.s["shape_of"][i]][0] for i in ids]))
        a, b = (coef @ Yt).transpose(1, 2), (coef @ Yp).transpose(1, 2)
        cr = torch.linalg.cross(a, b)
        J = cr.norm(dim=-1)
        return (coef @ Y).transpose(1, 2) - self.shift[ids][:, None, :], J, cr / J[..., None]

    def place(self, centres, quats):
        q = quats / quats.norm(dim=1, keepdim=True)
        w, x, y, z = q.T
        self.R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                              2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                              2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
        self.c = centres
        self.r = torch.cat([b[0] @ self.R[i].T for i, b in enumerate(self.body)])
        self.w = torch.cat([b[1] for b in self.body])
        self.nrm = torch.cat([b[2] @ self.R[i].T for i, b in enumerate(self.body)])
        self.pid = torch.tensor(np.repeat(np.arange(self.n), np.diff(self.off)), device="cuda")
        self.x = self.r + self.c[self.pid]
        cen = centres.cpu().numpy()
        self.near = []
        for i in range(self.n):
            d = np.linalg.norm(cen - cen[i], axis=1)
            hit = (d < self.radius + self.radius[i] + 1.0) & (self.sid == self.sid[i])
            hit[i] = False
            self.near.append(np.flatnonzero(hit))
        self.xup = [b[0] @ self.R[i].T + centres[i] for i, b in enumerate(self.body_up)]
        self.area = self.sum(self.w[:, None])[:, 0]
        r2 = self.sum((self.w * (self.r ** 2).sum(1))[:, None])[:, 0]
        outer = self.sum((self.w[:, None, None] * self.r[:, :, None] * self.r[:, None, :]).reshape(-1, 9))
        self.tau = r2[:, None, None] * torch.eye(3, dtype=torch.float64, device="cuda") - outer.reshape(-1, 3, 3)

    def sum(self, f):
        """Per-particle sums of a node field."""
        out = torch.zeros((self.n, f.shape[1]), dtype=torch.float64, device="cuda")
        return out.index_add_(0, self.pid, f)

    def sl(self, i):
        return slice(int(self.off[i]), int(self.off[i + 1]))

    def self_blocks(self, kind):
        """Body-frame singular-rule blocks: per grid (k, N, c, N, c), c = 3, or 1 for the Laplace kernels."""
        if kind in self.blocks:
            return self.blocks[kind]
        c = 1 if kind.startswith("laplace") else 3
        self.blocks[kind] = {}
        for k, ids in self.members.items():
            g = self.grids[k]
            out = torch.empty((len(ids), g.np, c, g.np, c), dtype=torch.float64, device="cuda")
            x = torch.stack([self.body[i][0] for i in ids])
            nrm = torch.stack([self.body[i][2] for i in ids])
            for t, u, interp in g.rotated():
                y, J, _ = self._surface(ids, u)
                d = x[:, t, None, :] - y
                inv = 1 / d.norm(dim=-1)
                wt = g.rule * J
                dn = (d * nrm[:, t, None, :]).sum(-1)
                if kind == "K":
                    ker = (-3 / (4 * math.pi) * wt * dn * inv ** 5)[..., None, None] * d[..., :, None] * d[..., None, :]
                elif kind == "S":
                    ker = d[..., :, None] * d[..., None, :] * (inv ** 3)[..., None, None]
                    ker = ker + torch.eye(3, dtype=torch.float64, device="cuda") * inv[..., None, None]
                    ker = ker * (wt / (8 * math.pi))[..., None, None]
                elif kind == "laplace-K":
                    ker = (-wt * dn * inv ** 3 / (4 * math.pi))[..., None, None]
                else:
                    ker = (wt * inv / (4 * math.pi))[..., None, None]
                out[:, t] = torch.einsum("kmab,ms->kasb", ker, interp)
            self.blocks[kind][k] = out
        return self.blocks[kind]

    def apply(self, kind, f, half=0.0, with_L=False):
        """half f + (operator of kind) f (+ L f) on node fields (N, 3), or (N, 1) for the Laplace kernels."""
        y = half * f
        laplace = kind.startswith("laplace")
        for k, ids in self.members.items():
            g, blk = self.grids[k], self.self_blocks(kind)[k]
            z = torch.stack([f[self.sl(i)] for i in ids])
            if not laplace:
                z = torch.einsum("ksb,kbc->ksc", z, self.R[ids])
            z = torch.bmm(blk.reshape(len(ids), g.np * f.shape[1], -1), z.reshape(len(ids), -1, 1)).reshape(z.shape)
            if not laplace:
                z = torch.einsum("ksb,kcb->ksc", z, self.R[ids])
            for a, i in enumerate(ids):
                y[self.sl(i)] += z[a]
        if with_L:
            total = self.sum(self.w[:, None] * f)
            moment = self.sum(self.w[:, None] * torch.linalg.cross(self.r, f))
            y = y + total[self.pid] + torch.linalg.cross(moment[self.pid], self.r)
        up = [self.grid[j].up @ f[self.sl(j)] for j in range(self.n)]
        wf = self.w[:, None] * f
        for i in range(self.n):
            group = np.flatnonzero(self.sid == self.sid[i])
            lo, hi = int(self.off[group[0]]), int(self.off[group[-1] + 1])
            q = wf[lo:hi].clone()
            own = slice(int(self.off[i]) - lo, int(self.off[i + 1]) - lo)
            skip = torch.zeros(hi - lo, dtype=torch.bool, device="cuda")
            for j in [i, *self.near[i]]:
                skip[int(self.off[j]) - lo:int(self.off[j + 1]) - lo] = True
            q[skip] = 0
            src = torch.cat([self.x[lo:hi]] + [self.xup[j] for j in self.near[i]]) - self.c[i]
            q = torch.cat([q] + [self.body_up[j][1][:, None] * up[j] for j in self.near[i]])
            xt, nt = self.r[self.sl(i)], self.nrm[self.sl(i)]
            r2 = (xt ** 2).sum(1)[:, None] + (src ** 2).sum(1)[None, :] - 2 * xt @ src.T
            r2[:, own] = 1.0
            inv = torch.rsqrt(r2)
            if kind == "laplace-S":
                y[self.sl(i)] += inv @ q / (4 * math.pi)
                continue
            dn = (xt * nt).sum(1)[:, None] - nt @ src.T
            if kind == "laplace-K":
                y[self.sl(i)] -= (dn * inv ** 3) @ q / (4 * math.pi)
                continue
            dq = xt @ q.T - (src * q).sum(1)[None, :]
            c = dq * inv ** 3 if kind == "S" else dn * dq * inv ** 5
            acc = xt * c.sum(1, keepdim=True) - c @ src
            if kind == "S":
                y[self.sl(i)] += (acc + inv @ q) / (8 * math.pi)
            else:
                y[self.sl(i)] += -3 / (4 * math.pi) * acc
        return y

    def solve(self, F, T, x0=None, tol=1e-13):
        F, T = _dev(F), _dev(T)
        spin = torch.linalg.solve(self.tau, T)
        rho = (F / self.area[:, None])[self.pid] + torch.linalg.cross(spin[self.pid], self.r)
        b = -self.apply("K", rho, half=0.5)
        mu = _gmres(lambda z: self.apply("K", z, half=0.5, with_L=True), b, tol, x0)
        u = self.apply("S", rho + mu)
        v = self.sum(self.w[:, None] * u) / self.area[:, None]
        omega = torch.linalg.solve(self.tau, self.sum(self.w[:, None] * torch.linalg.cross(self.r, u)))
        return v, omega, mu

    def magnetic(self, field, ratio):
        field, eta = _dev(field), (ratio - 1) / (ratio + 1)
        hn = self.nrm @ field
        q = _gmres(lambda z: 0.5 * z + eta * self.apply("laplace-K", z), eta * hn[:, None], 1e-13)
        phi = self.apply("laplace-S", q)[:, 0] - self.x @ field
        Hn = hn + 0.5 * q[:, 0] - self.apply("laplace-K", q)[:, 0]
        H = Hn[:, None] * self.nrm
        for i in range(self.n):
            g, sl = self.grid[i], self.sl(i)
            coef = g.An @ phi[sl]
            ft, fp = g.Yt.T @ coef, g.Yp.T @ coef
            ax = _dev(self.s["axes"][i])
            st, ct = torch.hypot(g.u[:, 0], g.u[:, 1]), g.u[:, 2]
            cp, sp = g.u[:, 0] / st, g.u[:, 1] / st
            a = torch.stack([ct * cp, ct * sp, -st], 1) * ax @ self.R[i].T
            b = torch.stack([-sp, cp, torch.zeros_like(sp)], 1) * ax @ self.R[i].T
            aa, bb, ab = (a * a).sum(1), (b * b).sum(1), (a * b).sum(1)
            det = aa * bb - ab * ab
            H[sl] -= ((bb * ft - ab * fp) / det)[:, None] * a + ((aa * fp - ab * ft) / det)[:, None] * b
        f = (H * self.nrm).sum(1, keepdim=True) * H - 0.5 * (H * H).sum(1, keepdim=True) * self.nrm
        return self.sum(self.w[:, None] * f), self.sum(self.w[:, None] * torch.linalg.cross(self.r, f)), q[:, 0]


def _gmres(apply, b, tol, x0=None, most=150):
    """Unrestarted GMRES with reorthogonalised Gram-Schmidt."""
    shape = b.shape
    x = torch.zeros_like(b) if x0 is None else x0
    r = b if x0 is None else b - apply(x0)
    beta, goal = float(r.norm()), tol * float(b.norm())
    if beta <= goal:
        return x
    V, H = [(r / beta).reshape(-1)], np.zeros((most + 1, most))
    for k in range(most):
        w = apply(V[k].reshape(shape)).reshape(-1)
        basis = torch.stack(V)
        for _ in range(2):
            h = basis @ w
            w = w - h @ basis
            H[:k + 1, k] += h.cpu().numpy()
        H[k + 1, k] = float(w.norm())
        rhs = np.zeros(k + 2)
        rhs[0] = beta
        y = np.linalg.lstsq(H[:k + 2, :k + 1], rhs, rcond=None)[0]
        if np.linalg.norm(rhs - H[:k + 2, :k + 1] @ y) <= goal:
            break
        V.append(w / H[k + 1, k])
    return x + (_dev(y) @ torch.stack(V[:len(y)])).reshape(shape)
