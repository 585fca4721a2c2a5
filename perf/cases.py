"""Performance cases of the meshfree BGK library: what its users have it do.

Each case is one kind of run at a size of its range: time steps of a single cavity (2D and
3D, fixed points and moving points, FP64 / FP32 / BF16 storage, linear and quadratic
stencils, first and second order in time, with a moving disc), steps of a sweep of small
cavities in one context, and the adjoint gradient.  ``prepare`` builds the point cloud, the
solver and the initial distribution; ``run`` steps it through the public entry points;
``exact`` is the same computation in plain FP64 torch.

The initial state is not an equilibrium: a Maxwellian of smooth rho, U and T times
(1 + 0.1 u), u uniform in [-1, 1] for every point and velocity.
"""
import math
import random

import numpy as np
import torch

import paper_2408_02350_gb300 as bgk
from paper_2408_02350_gb300 import adjoint

TORCH = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
CODE = {"f64": bgk.BGK_F64, "f32": bgk.BGK_F32, "bf16": bgk.BGK_BF16}


def _case(name=None, kind="step", dim=2, n=41, nv=16, vmax=5.0, kn=0.1, lid=0.1, storage="f32", ale=False,
          wls=1, order=1, body=False, steps=2, count=1):
    c = dict(kind=kind, dim=dim, n=n, nv=nv, vmax=vmax, kn=kn, lid=lid, storage=storage, ale=ale, wls=wls,
             order=order, body=body, steps=steps, count=count)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest calls: an interactive run of the small cavity, bound by latency
        _case("cavity2d_small_f32", n=41, nv=16, lid=0.1),
        # the same cavity by the plain FP64 method, with the moments read every second step
        _case("cavity2d_f64", n=41, nv=16, storage="f64"),
        # the flagship: the moving-point cavity at its benchmark size
        _case("ale2d_f32", n=201, nv=32, vmax=6.0, lid=0.02, ale=True),
        # the same with 16-bit storage (half the memory)
        _case("ale2d_bf16", n=201, nv=32, vmax=6.0, lid=0.02, ale=True, storage="bf16"),
        # the second-order Taylor stencils on moving points, rarefied gas
        _case("ale2d_quadratic_f32", n=181, nv=24, kn=1.0, lid=0.02, ale=True, wls=2),
        # a disc moving through the gas
        _case("body2d_f32", n=201, nv=28, vmax=6.0, lid=0.02, ale=True, body=True),
        # fixed points with an odd velocity grid (no aligned velocity rows), state read back
        _case("fixed2d_odd_f32", n=133, nv=27, kn=0.03),
        # second order in time at the benchmark size
        _case("fixed2d_order2_f32", n=201, nv=32, vmax=6.0, order=2),
        # a parameter sweep: 24 cavities of different sizes in one context
        _case("sweep2d_f32", kind="sweep", n=121, nv=32, steps=4, count=24),
        # the 3D cavity at its benchmark size, the largest single run
        _case("cavity3d_f32", dim=3, n=41, nv=16),
        # a 3D cavity with moving points
        _case("ale3d_f32", dim=3, n=27, nv=12, lid=0.02, ale=True),
        # the gradient of the lid flux over a few steps, at the adjoint workload's size
        _case("adjoint2d_f32", kind="adjoint", n=101, nv=24, steps=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kn = 10.0 ** rng.uniform(-2.0, 0.0)
    what = rng.choice(["fixed", "fixed", "f64", "ale", "ale", "body", "quadratic", "order2", "sweep", "3d", "3d",
                       "ale3d", "adjoint"])
    fl = rng.choice(["f32", "f32", "bf16"])
    if what == "fixed":
        return _case(n=_log(rng, 41, 401), nv=rng.randint(12, 32), kn=kn, lid=rng.uniform(0.05, 0.2), storage=fl)
    if what == "f64":
        return _case(n=_log(rng, 31, 101), nv=rng.randint(8, 20), kn=kn, storage="f64", ale=False)
    if what == "ale":
        return _case(n=rng.randint(181, 301), nv=rng.choice([24, 27, 28, 30, 32]), vmax=6.0, kn=kn, lid=0.02,
                     ale=True, storage=fl)
    if what == "body":
        return _case(n=rng.randint(181, 281), nv=rng.choice([24, 28, 32]), vmax=6.0, kn=kn, lid=0.02, ale=True,
                     body=True)
    if what == "quadratic":
        return _case(n=rng.randint(161, 221), nv=rng.randint(20, 32), kn=kn, lid=0.02, ale=True, wls=2)
    if what == "order2":
        return _case(n=_log(rng, 61, 241), nv=rng.randint(12, 32), kn=kn, order=2)
    if what == "sweep":
        return _case(kind="sweep", n=rng.randint(81, 121), nv=rng.randint(24, 32), steps=4, count=rng.randint(8, 32))
    if what == "3d":
        return _case(dim=3, n=rng.randint(15, 37), nv=rng.randint(8, 16), kn=kn, storage=fl)
    if what == "ale3d":
        return _case(dim=3, n=rng.randint(21, 31), nv=rng.choice([10, 12, 16]), kn=kn, lid=0.02, ale=True)
    return _case(kind="adjoint", n=_log(rng, 51, 121), nv=4 * rng.randint(3, 6), kn=kn, steps=rng.randint(4, 8))


# ---- inputs ----


def _params(c):
    dim, dx = c["dim"], 1.0 / (c["n"] - 1)
    p = {"dim": dim, "nv": c["nv"], "vmax": c["vmax"], "kn": c["kn"], "tau_mode": 0,
         "dt": 0.5 * dx / (c["vmax"] * math.sqrt(dim)), "h": 2.5 * dx, "alpha": 6.25, "wall_T": 1.0,
         "lid_u": [c["lid"], 0.0, 0.0], "lid_wall": 2 * dim, "ale": int(c["ale"]), "periodic": 0, "guard": 0.1 * dx,
         "storage": c["storage"], "max_nbrs": 48 if dim == 2 else 160, "wls_order": c["wls"],
         "time_order": c["order"]}
    if c["body"]:
        p.update(body_wall=2 * dim + 2, body_u=[0.02, 0.0, 0.0], body_centre=[0.4, 0.5, 0.0], body_radius=0.1)
    return p


def _cloud(c, p, seed):
    """A lattice on the unit square or cube, interior points jittered by 0.1 dx."""
    dim, n = c["dim"], c["n"]
    dx = 1.0 / (n - 1)
    idx = np.indices((n,) * dim).reshape(dim, -1)[::-1].T
    x = idx * dx
    x[idx == n - 1] = 1.0
    lo, hi = idx == 0, idx == n - 1
    walls = (lo | hi).sum(axis=1)
    kind = np.zeros(len(x), dtype=np.int32)
    normal = lo.astype(np.float64) - hi.astype(np.float64)
    for a in range(dim):
        kind[(walls == 1) & lo[:, a]] = 2 * a + 1
        kind[(walls == 1) & hi[:, a]] = 2 * a + 2
    kind[walls >= 2] = 2 * dim + 1
    length = np.sqrt((normal * normal).sum(axis=1))
    normal[length > 0] /= length[length > 0, None]
    lattice = x.copy()
    jitter = np.random.RandomState(seed % (1 << 31)).uniform(-0.1 * dx, 0.1 * dx, x.shape)
    x[kind == 0] += jitter[kind == 0]
    if c["body"]:
        centre, radius = np.array(p["body_centre"][:2]), p["body_radius"]
        far = np.sqrt(((lattice - centre) ** 2).sum(axis=1)) >= radius + 0.5 * dx
        keep = (kind != 0) | far
        m = max(8, round(2.0 * math.pi * radius / dx))
        angle = 2.0 * math.pi * np.arange(m) / m
        out = np.stack([np.cos(angle), np.sin(angle)], axis=1)
        x = np.concatenate([x[keep], centre + radius * out])
        kind = np.concatenate([kind[keep], np.full(m, p["body_wall"], dtype=np.int32)])
        normal = np.concatenate([normal[keep], out])
    return {"x": x, "kind": kind, "normal": normal}


def _velocities(p, dev):
    """[NV][dim] nodes, the first axis fastest, and the node spacing."""
    nv, dim = p["nv"], p["dim"]
    dv = 2.0 * p["vmax"] / (nv - 1)
    v = (torch.arange(nv, dtype=torch.float64, device=dev) - 0.5 * (nv - 1)) * dv
    k = torch.arange(nv**dim, device=dev)
    return torch.stack([v[(k // nv**a) % nv] for a in range(dim)], dim=1), dv


def _maxwell(rho, U, T, v):
    """[n][ncomp][NV] Maxwellian (3D) or its two Chu reductions (2D)."""
    dim = v.shape[1]
    c2 = sum((v[None, :, a] - U[:, a, None]) ** 2 for a in range(dim))
    M = (rho / (2.0 * math.pi * T) ** (0.5 * dim))[:, None] * torch.exp(-c2 / (2.0 * T)[:, None])
    return torch.stack([M, T[:, None] * M], dim=1) if dim == 2 else M[:, None]


def _initial(c, p, cloud, seed, dev):
    """The initial f in the storage type."""
    x = torch.from_numpy(cloud["x"]).to(dev)
    n, dim, amp = x.shape[0], c["dim"], 0.02 if c["ale"] else 0.2
    s, k = torch.sin(math.pi * x), torch.cos(math.pi * x)
    U = torch.zeros_like(x)
    U[:, 0], U[:, 1] = amp * s[:, 0] ** 2 * 2 * s[:, 1] * k[:, 1], -amp * s[:, 1] ** 2 * 2 * s[:, 0] * k[:, 0]
    rho, T = 1.0 + 0.1 * k[:, 0] * k[:, -1], 1.0 + 0.05 * k[:, 1]
    v, _ = _velocities(p, dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    f = torch.empty((n, 2 if dim == 2 else 1, v.shape[0]), dtype=TORCH[c["storage"]], device=dev)
    for a in range(0, n, 8192):  # in blocks of points, to keep the FP64 intermediates small
        b = slice(a, min(n, a + 8192))
        M = _maxwell(rho[b], U[b], T[b], v)
        u = torch.rand(M.shape, generator=gen, dtype=torch.float32, device=dev)
        f[b] = (M * (1.0 + 0.1 * (2.0 * u.double() - 1.0))).to(f.dtype)
    return f


def _members(c, seed):
    """(case, seed) of each cavity of a sweep, or of the one cavity; a sweep draws sides
    from 41 up to n, velocity nodes from 16 up to nv, Kn and the lid speed."""
    if c["kind"] != "sweep":
        return [(c, seed)]
    rng = random.Random(1000 * c["n"] + c["count"])  # the sizes are the case's, the values the seed's
    out = []
    for k in range(c["count"]):
        m = dict(c, n=rng.randint(41, c["n"]), nv=rng.randint(16, c["nv"]))
        r = random.Random(seed + k)
        out.append((dict(m, kn=10.0 ** r.uniform(-2.0, 0.0), lid=r.uniform(0.05, 0.2)), seed + 7919 * k))
    return out


def prepare(c, seed):
    dev = torch.device("cuda")
    members = _members(c, seed)
    params = [_params(m) for m, _ in members]
    clouds = [_cloud(m, p, s) for (m, s), p in zip(members, params)]
    solver = bgk.Solver(params, clouds)
    fs = [_initial(m, p, cl, s, dev) for (m, s), p, cl in zip(members, params, clouds)]
    st = {"c": c, "solver": solver, "f": fs, "code": CODE[c["storage"]]}
    st["bound"] = c["kind"] == "step" and fs[0].shape[2] % 4 == 0
    for k, f in enumerate(fs):
        if st["bound"]:  # the solver's state lives in the caller's tensor
            fs[k] = torch.empty_like(f)
            solver.bind_f(fs[k], k)
            fs[k].copy_(f)
        solver.set_f(fs[k], k)
    if c["ale"]:
        st["x"] = torch.empty(clouds[0]["x"].shape, dtype=torch.float64, device=dev)
    if c["storage"] == "f64":
        n, d = clouds[0]["x"].shape
        st["mom"] = [torch.empty(s, dtype=torch.float64, device=dev) for s in ((n,), (n, d), (n,))]
    return st


def run(st):
    c, s = st["c"], st["solver"]
    if c["kind"] == "adjoint":
        J, du, dkn, lam = adjoint.gradient(s, c["steps"], f0=st["f"][0])
        return {"J": J, "du": float(du[0]), "dkn": dkn, "lam": lam}
    s.step(c["steps"])
    if not st["bound"]:
        for k, f in enumerate(st["f"]):
            bgk.bgk_get_f(s.ctx, k, f, st["code"])
    out = {"f": st["f"]}
    if "x" in st:
        bgk.bgk_get_positions(s.ctx, 0, st["x"])
        out["x"] = st["x"]
    if "mom" in st:
        bgk.bgk_moments(s.ctx, 0, *st["mom"])
        out["mom"] = st["mom"]
    return out


def work(c):
    """f read and written once per step (and once more where it is read back); per update and
    neighbour the projections, their minima, the sums."""
    size = {"f64": 8, "f32": 4, "bf16": 2}[c["storage"]]
    updates = sum(float(m["n"] ** m["dim"] * m["nv"] ** m["dim"]) for m, _ in _members(c, 0))
    comp, nbrs, ops = (2, 20, 12) if c["dim"] == 2 else (1, 80, 14)
    passes = 2.0 * c["steps"] * c["order"]
    flops = updates * nbrs * ops * c["steps"] * c["order"]
    if c["kind"] == "adjoint":
        # forward, its segment again, and the reverse sweep (read f and lambda, write lambda)
        passes, flops = 7.0 * c["steps"], 4.0 * flops
    elif c["kind"] == "sweep" or c["nv"] ** c["dim"] % 4:
        passes += 2.0
    return {"bytes": updates * comp * size * passes, "flops": flops}


# ---- the same in plain FP64 ----


def _neighbours(x, h):
    """Padded lists: idx [n][K] and valid [n][K], ascending."""
    n = x.shape[0]
    rows, cols = [], []
    for a in range(0, n, 1024):
        d2 = 0.0
        for k in range(x.shape[1]):
            d = x[None, :, k] - x[a:a + 1024, None, k]
            d2 = d2 + d * d
        r, j = torch.nonzero(d2 <= h * h, as_tuple=True)
        rows.append(r + a)
        cols.append(j)
    r, j = torch.cat(rows), torch.cat(cols)
    r, j = r[r != j], j[r != j]
    cnt = torch.bincount(r, minlength=n)
    start = torch.cumsum(cnt, 0) - cnt
    slot = torch.arange(len(r), device=x.device) - start[r]
    idx = torch.zeros((n, int(cnt.max())), dtype=torch.int64, device=x.device)
    valid = torch.zeros(idx.shape, dtype=torch.bool, device=x.device)
    idx[r, slot], valid[r, slot] = j, True
    return idx, valid


def _projected(p, x, idx, valid):
    """P [m][K][dim][dim]: the projected WLS coefficients times their frame vectors (rows d)
    of the points whose lists are given, x their own positions and xj = x[idx]."""
    own, xj = x
    dim = own.shape[1]
    dr = torch.where(valid[..., None], xj - own[:, None], torch.ones_like(xj))
    r2 = (dr * dr).sum(-1)
    w = torch.where(valid, torch.exp(-p["alpha"] * r2 / p["h"] ** 2), torch.zeros_like(r2))
    s = dr / p["h"]  # scaled, for the conditioning of the fit
    basis = [s[..., a] for a in range(dim)]
    if p["wls_order"] == 2:
        basis += [s[..., a] * s[..., b] * (0.5 if a == b else 1.0) for a in range(dim) for b in range(a, dim)]
    b = torch.stack(basis, dim=-1)
    A = torch.einsum("mk,mka,mkb->mab", w, b, b)
    G = torch.linalg.inv(A)[:, :dim]
    coef = torch.einsum("mk,mab,mkb->mka", w, G, b) / p["h"]
    nrm = dr / torch.sqrt(r2)[..., None]
    if dim == 2:
        E = torch.stack([nrm, torch.stack([-nrm[..., 1], nrm[..., 0]], dim=-1)], dim=-2)
    else:
        rxy = torch.sqrt(dr[..., 0] ** 2 + dr[..., 1] ** 2)
        on = rxy > 0.0
        cp = torch.where(on, dr[..., 0] / rxy, torch.ones_like(rxy))
        sp = torch.where(on, dr[..., 1] / rxy, torch.zeros_like(rxy))
        ct, sn = nrm[..., 2], rxy / torch.sqrt(r2)
        E = torch.stack([nrm, torch.stack([ct * cp, ct * sp, -sn], dim=-1),
                         torch.stack([-sp, cp, torch.zeros_like(sp)], dim=-1)], dim=-2)
    return (E * coef[..., None, :]).sum(-1, keepdim=True) * E


class _Upwind(torch.autograd.Function):
    """sum_j m_ij(v) (f_j - f_i) with the transposed sum as its derivative; m and the lists
    are those of the points `inner`."""

    @staticmethod
    def forward(ctx, f, inner, idx, coef):
        ctx.geom = (inner, idx, coef)
        ctx.shape = f.shape
        out = torch.zeros((len(inner),) + f.shape[1:], dtype=f.dtype, device=f.device)
        for a, m in coef():
            own = f[inner[a]]
            for s, ms in enumerate(m):
                out[a] += ms[:, None] * (f[idx[a, s]] - own)
        return out

    @staticmethod
    def backward(ctx, g):
        inner, idx, coef = ctx.geom
        back = torch.zeros(ctx.shape, dtype=g.dtype, device=g.device)
        for a, m in coef():
            for s, ms in enumerate(m):
                t = ms[:, None] * g[a]
                back.index_add_(0, idx[a, s], t)
                back.index_add_(0, inner[a], -t)
        return back, None, None, None


class _Plain:
    """One cavity stepped in FP64 torch: the scheme of arXiv 2408.02350 as the library reads it."""

    def __init__(self, c, seed, dev):
        self.c, self.p = c, _params(c)
        cl = _cloud(c, self.p, seed)
        self.f = _initial(c, self.p, cl, seed, dev).double()
        self.x, self.kind, self.normal = (torch.from_numpy(cl[k]).to(dev) for k in ("x", "kind", "normal"))
        self.v, self.dv = _velocities(self.p, dev)
        self.inner, self.wall = torch.nonzero(self.kind == 0)[:, 0], torch.nonzero(self.kind != 0)[:, 0]
        self.lid_u = torch.tensor(self.p["lid_u"][:c["dim"]], dtype=torch.float64, device=dev)
        self.kn = torch.tensor(self.p["kn"], dtype=torch.float64, device=dev)
        self.body_u = torch.tensor(self.p.get("body_u", [0.0] * 3)[:c["dim"]], dtype=torch.float64, device=dev)
        self.body_c = torch.tensor(self.p.get("body_centre", [0.0] * 3)[:c["dim"]], dtype=torch.float64, device=dev)
        self.listed = False
        self.mom = self.moments(self.f)

    def moments(self, f):
        wv = self.dv ** self.c["dim"]
        g = f[:, 0]
        rho = g.sum(1) * wv
        U = (g @ self.v) * wv / rho[:, None]
        E = g @ (self.v * self.v).sum(1)
        if f.shape[1] == 2:
            E = E + f[:, 1].sum(1)
        return rho, U, (E * wv / rho - (U * U).sum(1)) / 3.0

    def lists(self):
        p, dim = self.p, self.c["dim"]
        idx, valid = _neighbours(self.x, p["h"])
        self.idx = idx[self.inner]
        self.P = torch.zeros(self.idx.shape + (dim, dim), dtype=torch.float64, device=self.x.device)
        for a in range(0, len(self.inner), 16384):
            b = slice(a, a + 16384)
            on = valid[self.inner[b]]
            P = _projected(p, (self.x[self.inner[b]], self.x[self.idx[b]]), self.idx[b], on)
            self.P[b] = torch.where(on[..., None, None], P, torch.zeros_like(P))
        # walls: linear reconstruction from interior neighbours, the constant fit below dim + 1
        wi = idx[self.wall]
        on = valid[self.wall] & (self.kind[wi] == 0)
        dr = self.x[wi] - self.x[self.wall][:, None]
        w = torch.where(on, torch.exp(-p["alpha"] * (dr * dr).sum(-1) / p["h"] ** 2), torch.zeros_like(dr[..., 0]))
        b = torch.cat([torch.ones_like(dr[..., :1]), dr / p["h"]], dim=-1)
        few = on.sum(1) <= dim
        B = torch.einsum("mk,mka,mkb->mab", w, b, b)
        B[few] = torch.eye(dim + 1, dtype=torch.float64, device=B.device)
        z = torch.linalg.inv(B)[:, 0]
        self.recon = torch.where(few[:, None], w / w.sum(1, keepdim=True), w * torch.einsum("mb,mkb->mk", z, b))
        self.wi, self.listed = wi, True

    def coefficients(self):
        """Blocks of points and their m_ij(v) = sum_d min(c.P_d, 0), one neighbour slot at a time."""
        U = self.mom[1][self.inner].detach() if self.c["ale"] else None
        size = max(1, (1 << 25) // self.v.shape[0])

        def block(b):
            for s in range(self.idx.shape[1]):
                m = 0.0
                for d in range(self.c["dim"]):
                    q = self.P[b, s, d] @ self.v.T
                    if U is not None:
                        q = q - (U[b] * self.P[b, s, d]).sum(1, keepdim=True)
                    m = m + torch.clamp(q, max=0.0)
                yield m

        for a in range(0, len(self.inner), size):
            b = slice(a, min(len(self.inner), a + size))
            yield b, block(b)

    def transport(self, f):
        """f~ of the interior points."""
        return f[self.inner] - 2.0 * self.p["dt"] * _Upwind.apply(f, self.inner, self.idx, self.coefficients)

    def relaxed(self, ft, exact_h=None):
        """The relaxation of rows ft (implicit over dt, or exactly over exact_h) and their moments."""
        rho, U, T = self.moments(ft)
        tau = math.sqrt(2.0 / math.pi) * self.kn / (rho * torch.sqrt(T))
        a = tau / (tau + self.p["dt"]) if exact_h is None else torch.exp(-exact_h / tau)
        M = _maxwell(rho, U, T, self.v)
        return a[:, None, None] * ft + (1.0 - a)[:, None, None] * M, (rho, U, T)

    def walls(self, f):
        """f with the rows of the wall points from its interior rows (diffuse reflection)."""
        p, kb = self.p, self.kind[self.wall]
        uw = torch.zeros((len(self.wall), self.c["dim"]), dtype=torch.float64, device=f.device)
        uw = torch.where((kb == p["lid_wall"])[:, None], self.lid_u, uw)
        if "body_wall" in p:
            uw = torch.where((kb == p["body_wall"])[:, None], self.body_u, uw)
        g = torch.zeros((len(self.wall),) + f.shape[1:], dtype=torch.float64, device=f.device)
        for s in range(self.wi.shape[1]):
            g = g + self.recon[:, s, None, None] * f[self.wi[:, s]]
        cn = 0.0
        for a in range(self.c["dim"]):
            cn = cn + (self.v[None, :, a] - uw[:, a, None]) * self.normal[self.wall][:, a, None]
        one = torch.ones(len(self.wall), dtype=torch.float64, device=f.device)
        M = _maxwell(one, uw, p["wall_T"] * one, self.v)
        out = cn > 0.0
        rho = torch.where(out, 0.0, -cn * g[:, 0]).sum(1) / torch.where(out, cn * M[:, 0], 0.0).sum(1)
        return f.index_copy(0, self.wall, torch.where(out[:, None], rho[:, None, None] * M, g))

    def move(self):
        p = self.p
        y = self.x[self.inner] + p["dt"] * self.mom[1][self.inner]
        y = torch.clamp(y, min=p["guard"], max=1.0 - p["guard"])
        if self.c["body"]:
            self.body_c = self.body_c + p["dt"] * self.body_u
            d = y - self.body_c
            r, rg = torch.sqrt((d * d).sum(1, keepdim=True)), p["body_radius"] + p["guard"]
            y = torch.where(r < rg, self.body_c + d * (rg / r), y)
        x = self.x.clone()
        x[self.inner] = y
        if self.c["body"]:
            x[self.kind == p["body_wall"]] += p["dt"] * self.body_u
        self.x, self.listed = x, False

    def step(self):
        if not self.listed:
            self.lists()
        f, dt = self.f, self.p["dt"]
        if self.c["order"] == 2:
            a = f.index_copy(0, self.inner, self.relaxed(f[self.inner], 0.5 * dt)[0])
            b = self.walls(a.index_copy(0, self.inner, self.transport(a)))
            ft = 0.5 * (a[self.inner] + self.transport(b))
            y, m = self.relaxed(ft, 0.5 * dt)
            f = a
        else:
            y, m = self.relaxed(self.transport(f))
        self.f = self.walls(f.index_copy(0, self.inner, y))
        whole = self.moments(self.f)
        self.mom = tuple(w.index_copy(0, self.inner, q) for w, q in zip(whole, m))
        if self.c["ale"]:
            self.move()

    def flux(self):
        """The x-momentum flux through the lid."""
        lid = torch.nonzero(self.kind == self.p["lid_wall"])[:, 0]
        w = self.v[:, 0] * self.v[:, -1] * self.dv ** self.c["dim"]
        return (self.f[lid, 0] @ w).mean()


def exact(c, seed):
    dev = torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")
    if c["kind"] == "adjoint":
        s = _Plain(c, seed, dev)
        f0 = s.f.requires_grad_()
        s.lid_u.requires_grad_()
        s.kn.requires_grad_()
        J = 0.0
        for _ in range(c["steps"]):
            s.step()
            J = J + s.flux() / c["steps"]
        df, du, dkn = torch.autograd.grad(J, (f0, s.lid_u, s.kn))
        return {"J": float(J.detach()), "du": float(du[0]), "dkn": float(dkn), "lam": df}
    out = {"f": []}
    for m, sd in _members(c, seed):
        s = _Plain(m, sd, dev)
        with torch.no_grad():
            for _ in range(c["steps"]):
                s.step()
        out["f"].append(s.f)
    if c["ale"]:
        out["x"] = s.x
    if c["storage"] == "f64":
        out["mom"] = list(s.mom)
    return out
