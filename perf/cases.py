"""Performance cases of the framework: what a user of the library has it do.

A case is one call (or one short sequence of calls) of the public binding on a mesh of a
stated kind and size:

  residual, jvp (FP64 / FP32), vjp   the operator entry points, Q1 (uniform and adaptive octrees,
                                     with hanging nodes) and Q2 (uniform octrees);
  newton                             one implicit step (the main call of a simulation);
  rollout                            a differentiable rollout: loss, d loss / d U0, d loss / d Cn;
  setup                              discrete mu0, mass and energy of a state (after remeshing or a
                                     restart, and as diagnostics).

`exact` evaluates the same discrete operators with plain torch in FP64, from the leaf list
alone (its own node numbering, hanging constraints and quadrature).
"""
import math

import numpy as np
import torch

import paper_2009_06628_gb300 as chns
from paper_2009_06628_gb300 import autograd as chns_autograd

# dimensionless groups of the synthetic workloads (drop in 2D / 3D, two drops, layer)
CONFIGS = {
    "drop2d": dict(dim=2, Re=100.0, We=10.0, Pe=100.0, Cn=0.05, Fr=0.0, rho_ratio=1.0, eta_ratio=1.0, dt=1e-3),
    "drop3d": dict(dim=3, Re=100.0, We=10.0, Pe=100.0, Cn=0.02, Fr=1.0, rho_ratio=10.0, eta_ratio=10.0, dt=5e-4),
    "twodrops3d": dict(dim=3, Re=100.0, We=10.0, Pe=100.0, Cn=0.02, Fr=1.0, rho_ratio=100.0, eta_ratio=50.0,
                       dt=5e-4),
    "layer3d": dict(dim=3, Re=1000.0, We=1000.0, Pe=1000.0, Cn=0.01, Fr=1.0, rho_ratio=3.0, eta_ratio=1.0, dt=2e-4),
}

# double operations per element that the operators cannot do without (Q1: 2^d Gauss points of
# the pointwise map, its tangent or adjoint, and the sum-factorised basis products)
FLOPS = {("residual", 2): 1500, ("residual", 3): 5500, ("jvp", 2): 2800, ("jvp", 3): 10000,
         ("vjp", 2): 3300, ("vjp", 3): 12000}


def _op(name, op, config, lmin, level, order=1, precision=64, hi=1.0, pin=2, pc=1, degree=16, steps=1):
    """lmin == level: uniform octree of that level; lmin < level: a band of finest leaves around
    the interface, 2:1 graded down to lmin."""
    return dict(name=name, op=op, config=config, lmin=lmin, level=level, order=order, precision=precision, hi=hi,
                pin=pin, pc=pc, degree=degree, steps=steps)


def listed():
    return [
        _op("jvp64_2d_l5", "jvp", "drop2d", 5, 5),
        _op("jvp32_3d_l6", "jvp", "drop3d", 6, 6, precision=32),
        _op("jvp32_two_drops_l4-8", "jvp", "twodrops3d", 4, 8, precision=32),
        _op("residual_two_drops_l3-7", "residual", "twodrops3d", 3, 7),
        _op("vjp_layer_l4-6", "vjp", "layer3d", 4, 6, pin=1),
        _op("q2_jvp32_3d_l5", "jvp", "drop3d", 5, 5, order=2, precision=32),
        _op("q2_vjp_3d_l4", "vjp", "drop3d", 4, 4, order=2),
        _op("setup_two_drops_l3-7", "setup", "twodrops3d", 3, 7),
        _op("newton64_2d_l5", "newton", "drop2d", 5, 5, precision=64),
        _op("newton32_3d_l6", "newton", "drop3d", 6, 6, precision=32),
        _op("newton32_mg_two_drops_l3-6", "newton", "twodrops3d", 3, 6, precision=32, pc=4, degree=2),
        _op("rollout_3d_l3", "rollout", "drop3d", 3, 3, precision=64, steps=2),
    ]


def draw(rng):
    op = rng.choice(["residual", "jvp", "jvp", "jvp", "vjp", "setup", "newton", "q2", "q2"])
    hi = rng.choice([1.0, 1.0, round(rng.uniform(0.7, 1.6), 3)])
    pin = rng.choice([0, 1, 2])
    if op == "q2":
        kind = rng.choice(["residual", "jvp", "jvp", "vjp"])
        config = rng.choice(["drop2d", "drop3d"])
        level = rng.randint(3, 7) if config == "drop2d" else rng.randint(2, 5 if kind == "jvp" else 4)
        return _drop_name(_op("", kind, config, level, level, order=2, hi=hi, pin=rng.choice([0, 2]),
                              precision=rng.choice([32, 64]) if kind == "jvp" and level < 5 else
                              (32 if kind == "jvp" else 64)))
    if op == "newton":
        config = rng.choice(["drop2d", "drop3d", "twodrops3d"])
        pc = rng.choice([1, 1, 3, 4])
        if config == "drop2d":
            level = rng.randint(4, 7)
            return _drop_name(_op("", "newton", config, level, level, precision=rng.choice([32, 64]), pc=1))
        if config == "drop3d":
            level = rng.randint(3, 5)
            return _drop_name(_op("", "newton", config, level, level, precision=32, pc=pc,
                                  degree=16 if pc < 3 else rng.choice([2, 3])))
        return _drop_name(_op("", "newton", config, rng.randint(2, 3), rng.randint(4, 6), precision=32, pc=pc,
                              degree=16 if pc < 3 else rng.choice([2, 3])))
    config = rng.choice(["drop2d", "drop3d", "twodrops3d", "layer3d"])
    precision = rng.choice([32, 32, 64]) if op == "jvp" else 64
    if config == "drop2d":
        level = rng.randint(3, 9)
        lmin = rng.choice([level, max(1, level - rng.randint(1, 4))])
    elif config == "drop3d":
        level = rng.randint(2, 6)
        lmin = rng.choice([level, max(1, level - rng.randint(1, 3))])
    else:
        level = rng.randint(4, 7)
        lmin = max(2, level - rng.randint(1, 4))
    return _drop_name(_op("", op, config, lmin, level, precision=precision, hi=hi, pin=pin))


def _drop_name(c):
    c.pop("name")
    return c


# ---------------------------------------------------------------------------------
# leaves: a band of finest leaves around the interface, graded so that it is 2:1 balanced
# ---------------------------------------------------------------------------------
def _spread(v, dim):
    v = v.astype(np.uint64)
    if dim == 2:
        for s, m in ((16, 0x0000FFFF0000FFFF), (8, 0x00FF00FF00FF00FF), (4, 0x0F0F0F0F0F0F0F0F),
                     (2, 0x3333333333333333), (1, 0x5555555555555555)):
            v = (v | (v << np.uint64(s))) & np.uint64(m)
    else:
        for s, m in ((32, 0x001F00000000FFFF), (16, 0x001F0000FF0000FF), (8, 0x100F00F00F00F00F),
                     (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
            v = (v | (v << np.uint64(s))) & np.uint64(m)
    return v


def _morton(c, dim):
    k = _spread(c[:, 0], dim)
    for i in range(1, dim):
        k = k | (_spread(c[:, i], dim) << np.uint64(i))
    return k


def _distance(config):
    """Signed distance (positive inside the phi = +1 phase) of the configuration's interface in the
    unit cube, as a function of coordinates x (N, d) of either numpy or torch.  The mesh follows
    it, so it is the same for every seed; `_state` moves the interface within the band."""
    r = np.random.default_rng(3)

    def drop(x, c, R):
        d2 = 0.0
        for k in range(x.shape[1]):
            d2 = d2 + (x[:, k] - c[k]) ** 2
        return R - d2 ** 0.5

    if config in ("drop2d", "drop3d"):
        c = 0.5 + 0.02 * r.uniform(-1.0, 1.0, 3)
        R = 0.25 if config == "drop2d" else 0.2
        return lambda x: drop(x, c, R)
    if config == "twodrops3d":
        u = r.normal(size=3)
        u /= np.linalg.norm(u)
        c1, c2 = 0.5 - 0.175 * u, 0.5 + 0.175 * u
        mx = lambda a, b: torch.maximum(a, b) if isinstance(a, torch.Tensor) else np.maximum(a, b)
        return lambda x: mx(drop(x, c1, 0.12), drop(x, c2, 0.15))
    phase = r.uniform(0.0, 2.0 * math.pi)

    def layer(x):
        cos = torch.cos if isinstance(x, torch.Tensor) else np.cos
        return x[:, -1] - (0.5 + 0.05 * cos(2.0 * math.pi * x[:, 0] + phase))
    return layer


def _leaves(case):
    cfg = CONFIGS[case["config"]]
    dim, lmin, L = cfg["dim"], case["lmin"], case["level"]
    n = 1 << lmin
    g = np.meshgrid(*[np.arange(n, dtype=np.int64) << (L - lmin)] * dim, indexing="ij")
    a = np.stack([x.reshape(-1) for x in g], axis=1)
    dist = _distance(case["config"])
    done_a, done_l = [], []
    # a leaf of size h is split when its centre is within band + 2 sqrt(d) h of the interface: the
    # margin of a size covers that of the next one plus the centre offset of a touching leaf
    # (<= (3/4) sqrt(d) h, interface slope factor 1.05), so touching leaves differ by one level
    for lev in range(lmin, L):
        h = 0.5 ** lev
        mid = (a + (1 << (L - lev - 1))) / float(1 << L)
        flag = np.abs(dist(mid)) <= 0.5 * h + 2.0 * math.sqrt(dim) * h * 1.05
        done_a.append(a[~flag])
        done_l.append(np.full(int((~flag).sum()), lev, dtype=np.int64))
        p = a[flag]
        s = 1 << (L - lev - 1)
        off = np.array([[(c >> k) & 1 for k in range(dim)] for c in range(1 << dim)], dtype=np.int64) * s
        a = (p[:, None, :] + off[None]).reshape(-1, dim)
    done_a.append(a)
    done_l.append(np.full(a.shape[0], L, dtype=np.int64))
    a, l = np.concatenate(done_a), np.concatenate(done_l)
    o = np.argsort(_morton(a, dim))
    out = np.zeros((a.shape[0], 4), dtype=np.int32)
    out[:, :dim] = a[o]
    out[:, 3] = l[o]
    return out


# ---------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------
def _config(case):
    return dict(CONFIGS[case["config"]], pin_pressure=case["pin"])


def _state(case, seed, x):
    """(U_old, U_new, x / w vector) on the GPU for unit-cube node coordinates x (N, d)."""
    cfg = CONFIGS[case["config"]]
    d, Cn = cfg["dim"], cfg["Cn"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 13)
    rnd = lambda *s: torch.randn(*s, dtype=torch.float64, device="cuda", generator=gen)
    N = x.shape[0]
    r = np.random.default_rng(seed)
    shift = 0.3 * Cn * r.uniform(-1.0, 1.0)
    U = torch.zeros(N, d + 3, dtype=torch.float64, device="cuda")
    U[:, d + 1] = torch.tanh((_distance(case["config"])(x) + shift) / (math.sqrt(2.0) * Cn))
    vel = torch.zeros(N, d, dtype=torch.float64, device="cuda")
    for _ in range(4):   # curls of products of sin^2: divergence free, zero on the boundary
        k = r.integers(1, 4, size=d)
        s = [torch.sin(math.pi * int(k[i]) * x[:, i]) for i in range(d)]
        c = [torch.cos(math.pi * int(k[i]) * x[:, i]) for i in range(d)]
        grad = []
        for j in range(d):
            g = 2.0 * math.pi * float(k[j]) * s[j] * c[j]
            for m in range(d):
                if m != j:
                    g = g * s[m] ** 2
            grad.append(g)
        amp = float(r.normal())
        ax = int(r.integers(0, 3)) if d == 3 else 2
        if d == 2:
            vel[:, 0] += amp * grad[1]
            vel[:, 1] -= amp * grad[0]
        else:
            i, j = (ax + 1) % 3, (ax + 2) % 3
            vel[:, i] += amp * grad[j]
            vel[:, j] -= amp * grad[i]
    U[:, :d] = 0.1 * vel / vel.norm(dim=1).max()
    if case["op"] in ("newton", "rollout"):
        return U, None, None
    U[:, d + 1] += 1e-3 * (2.0 * torch.rand(N, dtype=torch.float64, device="cuda", generator=gen) - 1.0)
    if case["op"] == "setup":
        return U, None, None
    U[:, d] = 0.01 * torch.cos(math.pi * x[:, 0]) * torch.cos(2.0 * math.pi * x[:, d - 1]) + 1e-3 * rnd(N)
    U[:, d + 2] = U[:, d + 1] ** 3 - U[:, d + 1] + 1e-3 * rnd(N)
    Un = U + 1e-3 * rnd(N, d + 3)
    edge = ((x <= 0.0) | (x >= 1.0)).any(dim=1)
    U[edge, :d] = 0.0
    Un[edge, :d] = 0.0
    return U, Un, rnd(N, d + 3)


def prepare(case, seed):
    cfg = _config(case)
    d, hi = cfg["dim"], case["hi"]
    prm = chns.Params.make(**cfg)
    if case["order"] == 2:
        mesh = chns.MeshQ2(d, case["level"], 0.0, hi)
    else:
        mesh = chns.Mesh(d, case["level"], _leaves(case), 0.0, hi)
    x = torch.tensor(mesh.node_coords(), device="cuda").double() / float(1 << mesh.max_level)
    U, Un, v = _state(case, seed, x)
    st = dict(case=case, mesh=mesh, prm=prm, U=U)
    if case["op"] == "jvp":
        dt = torch.float32 if case["precision"] == 32 else torch.float64
        st.update(U=U.to(dt), Un=Un.to(dt), x=v.to(dt))
    elif case["op"] in ("residual", "vjp"):
        st.update(Un=Un, x=v)
    elif case["op"] == "newton":
        chns.initial_mu(mesh, prm, U)
        mixed = case["precision"] == 32
        st["opts"] = chns.SolverOpts.make(rtol=1e-10 if mixed else 1e-12, atol=1e-14 if mixed else 1e-16,
                                          krylov_rtol=1e-3 if mixed else 1e-6, precision=1 if mixed else 0,
                                          restart=30 if d == 3 else 100, max_krylov=3000, pc_type=case["pc"],
                                          pc_degree=case["degree"])
    elif case["op"] == "rollout":
        st["opts"] = chns.SolverOpts.make(rtol=1e-12, atol=1e-13, krylov_rtol=1e-12, precision=0, restart=256,
                                          max_krylov=4000, max_newton=20)
        st["adj"] = chns.SolverOpts.make(krylov_rtol=1e-12, restart=256, max_krylov=4000, precision=0)
        st["U"] = U.requires_grad_(True)
        st["Cn"] = torch.tensor(cfg["Cn"], dtype=torch.float64, device="cuda", requires_grad=True)
    return st


def run(s):
    op, mesh, prm = s["case"]["op"], s["mesh"], s["prm"]
    if op == "residual":
        return chns.residual(mesh, prm, s["U"], s["Un"])
    if op == "jvp":
        return chns.jvp(mesh, prm, s["U"], s["Un"], s["x"])
    if op == "vjp":
        return chns.vjp(mesh, prm, s["U"], s["Un"], s["x"])
    if op == "newton":
        return chns.newton_step(mesh, prm, s["opts"], s["U"])[0]
    if op == "setup":
        chns.initial_mu(mesh, prm, s["U"])
        return s["U"], chns.mass(mesh, s["U"]), chns.energy(mesh, prm, s["U"])
    loss = chns_autograd.rollout(mesh, prm, s["opts"], s["adj"], s["U"], s["Cn"], s["case"]["steps"], 5)
    gU, gCn = torch.autograd.grad(loss, [s["U"], s["Cn"]])
    return loss.detach(), gU, gCn


def work(case):
    d = CONFIGS[case["config"]]["dim"]
    nf = d + 3
    if case["order"] == 2:
        E = 1 << (d * case["level"])
        N = ((2 << case["level"]) + 1) ** d
        per = (3 ** d) / (2 ** d) * 1.5     # more Gauss points, second-derivative terms
        conn = 4 * 3 ** d
    else:
        lv = _leaves(case)
        E = lv.shape[0]
        N = ((1 << case["level"]) + 1) ** d if case["lmin"] == case["level"] else int(E * 1.06)
        per = 1.0
        conn = 4 * 2 ** d + 1
    vec = N * nf * (4 if case["op"] == "jvp" and case["precision"] == 32 else 8)
    op = case["op"]
    if op == "residual":
        return dict(bytes=3 * vec + E * conn, flops=E * per * FLOPS[op, d])
    if op == "jvp":
        return dict(bytes=4 * vec + E * conn, flops=E * per * FLOPS[op, d])
    if op == "vjp":
        return dict(bytes=5 * vec + N + E * conn, flops=E * per * FLOPS[op, d])
    if op == "setup":
        # right-hand side, about 40 conjugate-gradient iterations of the mass matrix (FP64
        # vectors of one field), mass and energy
        return dict(bytes=3 * vec + 43 * E * conn + 40 * 10 * N * 8, flops=40.0 * E * 100 + E * 1500)
    if op == "newton":
        # about 5 residuals, and 150 operator applications with their orthogonalisation
        ob = 4 if case["precision"] == 32 else 8
        return dict(bytes=5 * (3 * vec + E * conn) + 150 * (4 * N * nf * ob + E * conn + 16 * vec),
                    flops=E * (5.0 * FLOPS["residual", d] + 150.0 * FLOPS["jvp", d]))
    k = case["steps"]
    return dict(bytes=k * 600 * (4 * vec + E * conn), flops=k * 600.0 * E * FLOPS["jvp", d])


# ---------------------------------------------------------------------------------
# the same operators in plain torch, FP64, from the leaf list alone
# ---------------------------------------------------------------------------------
class _Plain:
    def __init__(self, case):
        self.cfg = _config(case)
        d = self.d = self.cfg["dim"]
        self.order = case["order"]
        dev = "cuda"
        if self.order == 2:
            n = 1 << case["level"]
            g = np.meshgrid(*[np.arange(n, dtype=np.int64)] * d, indexing="ij")
            a = 2 * np.stack([q.reshape(-1) for q in g], axis=1)
            loc = np.array([[(i // 3 ** k) % 3 for k in range(d)] for i in range(3 ** d)], dtype=np.int64)
            corner = a[:, None, :] + loc[None]
            side = 2 * n
            size = np.full(a.shape[0], 2, dtype=np.int64)
        else:
            lv = _leaves(case)
            L = case["level"]
            side = 1 << L
            a = lv[:, :d].astype(np.int64)
            size = np.int64(1) << (L - lv[:, 3].astype(np.int64))
            loc = np.array([[(c >> k) & 1 for k in range(d)] for c in range(1 << d)], dtype=np.int64)
            corner = a[:, None, :] + loc[None] * size[:, None, None]
        nc = loc.shape[0]
        flat = corner.reshape(-1, d)
        key = _morton(flat, d)
        uk, first, inv, cnt = np.unique(key, return_index=True, return_inverse=True, return_counts=True)
        pts = flat[first]
        if self.order == 1:
            # a point is independent when every leaf touching it has it as a corner
            on = ((pts == 0) | (pts == side)).sum(axis=1)
            indep = cnt == (1 << (d - on))
        else:
            indep = np.ones(pts.shape[0], dtype=bool)
        num = np.cumsum(indep) - 1
        self.N = int(indep.sum())
        npts = pts[indep]
        # parents: along the axes where a hanging corner is an odd multiple of the leaf size it sits
        # at the middle of an edge or face of a leaf twice that size
        P = np.zeros((flat.shape[0], 4), dtype=np.int64)
        W = np.zeros((flat.shape[0], 4))
        own = indep[inv]
        P[own, 0] = num[inv[own]]
        W[own, 0] = 1.0
        hg = np.nonzero(~own)[0]
        if hg.size:
            s = np.repeat(size, nc)[hg]
            p = flat[hg]
            odd = (p // s[:, None]) % 2 == 1
            axes = np.argsort(~odd, axis=1, kind="stable")       # odd axes first
            m = odd.sum(axis=1)
            for j in range(4):
                use = j < (1 << m)
                q = p.copy()
                for t in range(min(2, d)):
                    mv = use & (t < m)
                    sg = 1 if (j >> t) & 1 else -1
                    q[mv, axes[mv, t]] += sg * s[mv]
                idx = np.searchsorted(uk, _morton(q[use], d))
                P[hg[use], j] = num[idx]
                W[hg[use], j] = 1.0 / (1 << m[use])
        T = lambda v, dt=torch.float64: torch.tensor(v, device=dev, dtype=dt)
        self.P, self.W = T(P.reshape(-1, nc, 4), torch.int64), T(W.reshape(-1, nc, 4))
        span = case["hi"]
        self.h = T(size) * (span / side)
        self.x = T(npts) / side                                  # unit cube
        self.edge = ((self.x <= 0) | (self.x >= 1)).any(dim=1)
        self.volume = span ** d
        # 1D tables
        if self.order == 1:
            gp = np.array([-1.0, 1.0]) / math.sqrt(3.0)
            w1 = np.ones(2)
            L0 = np.stack([(1 - gp) / 2, (1 + gp) / 2], 1)
            L1 = np.stack([np.full(2, -0.5), np.full(2, 0.5)], 1)
            L2 = np.zeros((2, 2))
        else:
            gp = np.array([-math.sqrt(0.6), 0.0, math.sqrt(0.6)])
            w1 = np.array([5.0, 8.0, 5.0]) / 9.0
            L0 = np.stack([gp * (gp - 1) / 2, 1 - gp ** 2, gp * (gp + 1) / 2], 1)
            L1 = np.stack([gp - 0.5, -2 * gp, gp + 0.5], 1)
            L2 = np.stack([np.ones(3), -2 * np.ones(3), np.ones(3)], 1)

        def tensor(tabs):
            out = np.ones((nc, nc))
            for k in range(d):
                out = out * tabs[k][np.ix_(loc[:, k], loc[:, k])]
            return T(out)
        der = lambda *ax: tensor([(L0, L1, L2)[ax.count(k)] for k in range(d)])
        self.Nq = der()
        self.dN = torch.stack([der(k) for k in range(d)], -1)
        self.HN = torch.stack([torch.stack([der(k, l) for l in range(d)], -1) for k in range(d)], -2)
        self.wq = T(np.prod(w1[loc], axis=1))
        self.gq = T(gp[loc])
        self.anchor = T(corner[:, 0, :]) * (span / side)
        self.detJ = (0.5 * self.h) ** d

    def gather(self, U):
        w = self.W.reshape(self.W.shape + (1,) * (U.dim() - 1))
        return (w * U[self.P]).sum(2)

    def scatter(self, r):
        tail = tuple(r.shape[2:])
        c = self.W.reshape(self.W.shape + (1,) * len(tail)) * r.unsqueeze(2)
        out = torch.zeros((self.N,) + tail, dtype=r.dtype, device=r.device)
        return out.index_add(0, self.P.reshape(-1), c.reshape((-1,) + tail))

    def val(self, u):
        return torch.einsum("qa,ea...->eq...", self.Nq, u)

    def grad(self, u):
        s = (2.0 / self.h).reshape((-1, 1) + (1,) * (u.dim() - 1))
        return torch.einsum("qak,ea...->eq...k", self.dN, u) * s

    def hess(self, u):
        s = (4.0 / self.h ** 2).reshape((-1, 1) + (1,) * u.dim())
        return torch.einsum("qakl,ea...->eq...kl", self.HN, u) * s

    def test(self, f0, f1):
        """sum_q w_q |J| (N_a f0 + grad N_a . f1), at the nodes."""
        sc = (self.detJ.reshape(-1, 1) * self.wq)
        tail = (1,) * (f0.dim() - 2)
        f0 = f0 * sc.reshape(sc.shape + tail)
        f1 = f1 * (sc * (2.0 / self.h).reshape(-1, 1)).reshape(sc.shape + tail + (1,))
        r = torch.einsum("qa,eq...->ea...", self.Nq, f0) + torch.einsum("qak,eq...k->ea...", self.dN, f1)
        return self.scatter(r)

    def residual(self, Uo, Un, Cn=None):
        c, d = self.cfg, self.d
        Cn = c["Cn"] if Cn is None else Cn
        Re, We, Pe, dt = c["Re"], c["We"], c["Pe"], c["dt"]
        fr = 1.0 / c["Fr"] if c["Fr"] > 0 else 0.0
        rm, em = 1.0 / c["rho_ratio"], 1.0 / c["eta_ratio"]
        Ut = 0.5 * (Uo + Un)
        u, du, un = self.gather(Ut), self.gather(Un - Uo), self.gather(Un[:, :d])
        ps = self.gather(Ut[:, d + 1].clamp(-1.0, 1.0))
        V, G, H = self.val(u), self.grad(u), self.hess(u)
        v, gv, phi, gphi, gmu, gp = V[..., :d], G[..., :d, :], V[..., d + 1], G[..., d + 1, :], G[..., d + 2, :], G[..., d, :]
        hphi = H[..., d + 1, :, :]
        tr = lambda m: torch.diagonal(m, dim1=-2, dim2=-1).sum(-1)
        dV = self.val(du) / dt
        vdt, pdt = dV[..., :d], dV[..., d + 1]
        s, gs = self.val(ps), self.grad(ps)
        rho = (1 - rm) / 2 * s + (1 + rm) / 2
        eta = (1 - em) / 2 * s + (1 + em) / 2
        geta = (1 - em) / 2 * gs
        J = (rm - 1.0) / (2.0 * Cn) * gmu
        conv = (gv * v.unsqueeze(-2)).sum(-1)
        Jg = (gv * J.unsqueeze(-2)).sum(-1)
        cap = (hphi * gphi.unsqueeze(-2)).sum(-1) + gphi * tr(hphi).unsqueeze(-1)
        visc = (gv * geta.unsqueeze(-2)).sum(-1) + eta.unsqueeze(-1) * tr(H[..., :d, :, :])
        up = torch.zeros(d, dtype=torch.float64, device=s.device)
        up[d - 1] = fr
        grav = rho.unsqueeze(-1) * up
        mom = rho.unsqueeze(-1) * (vdt + conv) + Jg / Pe + grav
        Rm = mom + Cn / We * cap + gp / We - visc / Re
        Rc = tr(gv)
        Rp = pdt + phi * Rc + (v * gphi).sum(-1) - tr(H[..., d + 2, :, :]) / (Pe * Cn)
        g = (4.0 / self.h ** 2).reshape(-1, 1)
        vv, vJ = (v * v).sum(-1), (v * J).sum(-1)
        tm = (4 / dt ** 2 + g * vv + g * vJ / (rho * Pe) + 6.0 * (eta / (rho * Re)) ** 2 * d * g * g) ** -0.5
        tc = 1.0 / (d * g * tm)
        tp = (4 / dt ** 2 + g * vv + 6.0 * (1.0 / (Pe * Cn)) ** 2 * d * g * g) ** -0.5
        tr_ = (tm / rho).unsqueeze(-1)
        e1 = lambda t: t.unsqueeze(-1)
        a = e1(tm) * v - e1(tm) * tr_ * Rm + tr_ * J / Pe
        f0m = mom - e1(tm) * (gv * Rm.unsqueeze(-2)).sum(-1)
        eye = torch.eye(d, dtype=torch.float64, device=s.device)
        f1m = (Rm.unsqueeze(-1) * a.unsqueeze(-2) - Cn / We * gphi.unsqueeze(-1) * gphi.unsqueeze(-2)
               + eta.unsqueeze(-1).unsqueeze(-1) * gv / Re
               + ((rho * tc * Rc - V[..., d]) / We).unsqueeze(-1).unsqueeze(-1) * eye)
        f0 = torch.cat([f0m, e1(tr(self.grad(un))), e1(pdt), e1(phi ** 3 - phi - V[..., d + 2])], -1)
        f1 = torch.cat([f1m, (tr_ * Rm).unsqueeze(-2),
                        (v * e1(tp * Rp - phi) + tr_ * e1(phi) * Rm + gmu / (Pe * Cn)).unsqueeze(-2),
                        (Cn * Cn * gphi).unsqueeze(-2)], -2)
        R = self.test(f0, f1)
        keep = torch.ones_like(R)
        keep[self.edge, :d] = 0.0
        repl = torch.zeros_like(R)
        repl[:, :d] = self.edge.double().unsqueeze(-1)
        R = R * keep + Un * repl
        if c["pin_pressure"] == 1:
            k2 = torch.ones_like(R)
            k2[0, d] = 0.0
            r2 = 1.0 - k2
            R = R * k2 + (Un - Uo) * r2
        return R

    def mass_apply(self, y):
        v = self.val(self.gather(y))
        return self.test(v, torch.zeros(v.shape + (self.d,), dtype=v.dtype, device=v.device))

    def initial_mu(self, phi):
        Cn = self.cfg["Cn"]
        u = self.gather(phi)
        p = self.val(u)
        b = self.test(p ** 3 - p, Cn * Cn * self.grad(u))
        dg = self.mass_apply(torch.ones_like(b))
        x, r = torch.zeros_like(b), b.clone()
        z = r / dg
        q, rz, bb = z.clone(), (r * z).sum(), float(b.norm())
        for _ in range(400):
            Aq = self.mass_apply(q)
            al = rz / (q * Aq).sum()
            x, r = x + al * q, r - al * Aq
            if float(r.norm()) <= 1e-15 * bb:
                break
            z = r / dg
            rz2 = (r * z).sum()
            q, rz = z + rz2 / rz * q, rz2
        return x

    def integral(self, f):
        return float((f * self.detJ.reshape(-1, 1) * self.wq).sum())

    def energy(self, U):
        c, d = self.cfg, self.d
        u = self.gather(U)
        v, phi, gphi = self.val(u[..., :d]), self.val(u[..., d + 1]), self.grad(u[..., d + 1])
        s = self.val(self.gather(U[:, d + 1].clamp(-1.0, 1.0)))
        rm = 1.0 / c["rho_ratio"]
        rho = (1 - rm) / 2 * s + (1 + rm) / 2
        z = self.anchor[:, d - 1:d] + self.h.reshape(-1, 1) * (self.gq[:, d - 1] + 1.0) / 2.0
        fr = 1.0 / c["Fr"] if c["Fr"] > 0 else 0.0
        Cn = c["Cn"]
        return (self.integral(0.5 * rho * (v * v).sum(-1)),
                self.integral((0.25 * (phi * phi - 1) ** 2 + 0.5 * Cn * Cn * (gphi * gphi).sum(-1)) / (Cn * c["We"])),
                self.integral(fr * rho * z))


def exact(case, seed):
    op = case["op"]
    if op == "rollout" or (op == "newton" and (case["config"] != "drop2d" or case["level"] > 5)):
        return None      # a nonlinear solve with a direct factorisation, or several, per value
    M = _Plain(case)
    U, Un, v = _state(case, seed, M.x)
    if op == "setup":
        d = M.d
        U[:, d + 2] = M.initial_mu(U[:, d + 1])
        return U, M.integral(M.val(M.gather(U[:, d + 1]))), M.energy(U)
    if op == "residual":
        return M.residual(U, Un)
    if op == "jvp":
        if case["precision"] == 32:
            U, Un, v = (t.float().double() for t in (U, Un, v))
        return torch.func.jvp(lambda t: M.residual(U, t), (Un,), (v,))[1]
    if op == "vjp":
        Uo, Un = U.requires_grad_(True), Un.requires_grad_(True)
        Cn = torch.tensor(M.cfg["Cn"], dtype=torch.float64, device="cuda", requires_grad=True)
        gn, go, gc = torch.autograd.grad(M.residual(Uo, Un, Cn), [Un, Uo, Cn], v)
        return gn, go, gc.reshape(1)
    # Newton with a dense Jacobian, the pressure update bordered by its mean
    d = M.d
    U[:, d + 2] = M.initial_mu(U[:, d + 1])
    Uk, X = U, U.clone()
    n = X.numel()
    mass = torch.zeros_like(X)
    mass[:, d] = M.mass_apply(torch.ones(M.N, dtype=torch.float64, device="cuda"))
    for _ in range(8):
        R = M.residual(Uk, X)
        rows = []
        lin = lambda t: torch.func.jvp(lambda y: M.residual(Uk, y), (X,), (t,))[1]
        for i in range(0, n, 256):
            k = min(256, n - i)
            t = torch.zeros(k, n, dtype=torch.float64, device="cuda")
            t[torch.arange(k), torch.arange(i, i + k)] = 1.0
            rows.append(torch.func.vmap(lin)(t.reshape((k,) + tuple(X.shape))).reshape(k, n))
        A = torch.zeros(n + 1, n + 1, dtype=torch.float64, device="cuda")
        A[:n, :n] = torch.cat(rows).T
        A[n, :n] = mass.reshape(-1)
        A[:n, n] = mass.reshape(-1)
        sc = A.abs().max(dim=1).values
        rhs = torch.cat([-R.reshape(-1), torch.zeros(1, dtype=torch.float64, device="cuda")])
        dX = torch.linalg.solve(A / sc.unsqueeze(1), rhs / sc)[:n].reshape(X.shape)
        X = X + dX
        if float(dX.norm()) <= 1e-13 * float(X.norm()):
            break
    return X
