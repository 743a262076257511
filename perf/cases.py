"""What a user of this library has it compute: whole moving-mesh steps, mesh redistributions, shock-tube batches and
training steps, at the sizes of the repository's configurations, tests and benchmark.

A case is a dict of plain values:
  kind "steps"  full steps of one problem through es_steps, from a given state (problem, n, form, steps)
  kind "mesh"   one mesh redistribution through es_mesh_redistribute (n1, n2, form, passes, sweeps)
  kind "tubes"  a batch of 1D shock tubes through es_batch_set_prim / steps / get (tubes, lmin, lmax, steps)
  kind "train"  one training step of the warm-start network (batch, n)

exact() restates the method in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_2407_05568_gb300 import es, learned
from paper_2407_05568_gb300 import perfmodel
from paper_2407_05568_gb300 import workloads as wl

FOREVER = 1e30                       # end time: the number of steps is the unit of work


# ------------------------------------------------------------------------------------------------ the cases

def listed():
    return [
        # 1D contact advection on the fixed mesh: the first configuration, the smallest calls
        dict(name="sine1d-200-fp64", kind="steps", problem="sine1d", n=200, form="fp64", steps=8),
        # 1D Riemann problem on the moving mesh (Example 5.2): every kernel of a step on 100 nodes
        dict(name="rp1-100-moving-fp64", kind="steps", problem="rp1", n=100, form="fp64", steps=8),
        # the benchmark's workload in the plain form, several steps to a call as a run makes them
        dict(name="riemann2d-200-fp64", kind="steps", problem="riemann2d", n=200, form="fp64", steps=4),
        # the same in the mixed form, one step to a call as a caller that looks at the state in between makes them
        dict(name="riemann2d-200-mixed", kind="steps", problem="riemann2d", n=200, form="mixed", steps=1),
        # Mach reflection on 200 x 100 nodes (Example 5.4): walls, a monitor with one gradient term, ten sweeps
        dict(name="mach-200x100-fp64", kind="steps", problem="mach", n=200, form="fp64", steps=4),
        # isentropic vortex of the convergence sweep: ideal gas, periodic, fixed mesh
        dict(name="vortex-256-fp64", kind="steps", problem="vortex", n=256, form="fp64", steps=2),
        # the precision configuration's size: 2D sine wave, mixed form
        dict(name="sine2d-1024-mixed", kind="steps", problem="sine2d", n=1024, form="mixed", steps=2),
        # 3D sine wave on the moving mesh (Example 5.6) in both forms
        dict(name="sine3d-96-fp64", kind="steps", problem="sine3d", n=96, form="fp64", steps=1),
        dict(name="sine3d-96-mixed", kind="steps", problem="sine3d", n=96, form="mixed", steps=1),
        # the mesh redistribution alone on the benchmark's large mesh
        dict(name="mesh-4096-fp64", kind="mesh", n1=4096, n2=4096, form="fp64", passes=5, sweeps=5),
        # the batched configuration: 4096 tubes of 200 to 8000 nodes
        dict(name="tubes-4096", kind="tubes", tubes=4096, lmin=200, lmax=8000, steps=10),
        # a training step of the warm-start network on four 512 x 512 snapshots
        dict(name="train-4x512", kind="train", batch=4, n=512),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["1d", "1d", "2d", "2d", "2d", "3d", "3d", "mesh", "mesh", "tubes", "train"])
    form = rng.choice(["fp64", "mixed"])
    if kind == "1d":
        problem = rng.choice(["sine1d", "rp1"])
        steps = 1 if problem == "rp1" and form == "mixed" else rng.randint(4, 8)
        return dict(kind="steps", problem=problem, n=size(40, 1600), form=form, steps=steps)
    if kind == "2d":
        problem = rng.choice(["riemann2d", "mach", "sine2d", "vortex"])
        if problem == "mach":                                   # walls: the FP64 form only
            return dict(kind="steps", problem=problem, n=size(60, 600), form="fp64", steps=rng.randint(1, 4))
        if problem == "riemann2d":
            n = size(40, 512 if form == "mixed" else 400)
            return dict(kind="steps", problem=problem, n=n, form=form, steps=1 if form == "mixed" else rng.randint(1, 4))
        return dict(kind="steps", problem=problem, n=size(48, 1024 if form == "mixed" else 384), form=form,
                    steps=rng.randint(1, 2))
    if kind == "3d":
        problem = rng.choice(["sine3d", "octant"])
        if problem == "octant":                                 # symmetry planes: the FP64 form only
            return dict(kind="steps", problem=problem, n=size(12, 80), form="fp64", steps=1)
        return dict(kind="steps", problem=problem, n=size(12, 96), form=form, steps=1)
    if kind == "mesh":
        return dict(kind="mesh", n1=size(100, 4096), n2=size(100, 4096), form=form, passes=5,
                    sweeps=rng.choice([5, 5, 10]))
    if kind == "tubes":
        return dict(kind="tubes", tubes=size(4, 2048), lmin=rng.randint(40, 400), lmax=rng.randint(500, 8000),
                    steps=rng.randint(1, 10))
    return dict(kind="train", batch=rng.randint(1, 4), n=size(64, 512))


def _workload(case, seed):
    """The workload of a "steps" case with the seed's own states: a phase, a strength or a position drawn from it."""
    rng = np.random.default_rng(seed)
    u = rng.uniform(-1.0, 1.0)
    n, problem = case["n"], case["problem"]
    if problem == "sine1d":
        w = wl.sine_1d(n)
        w["rho"] = 0.5 + 0.2 * np.sin(2 * np.pi * (w["x"][0] + u))
    elif problem == "sine2d":
        w = wl.sine_2d(n)
        w["rho"] = 0.5 + 0.2 * np.sin(2 * np.pi * (w["x"][0] + w["x"][1] + u))
    elif problem == "sine3d":
        w = wl.sine_3d(n, moving=True)
        w["rho"] = 0.5 + 0.2 * np.sin(2 * np.pi * (w["x"].sum(axis=0) + u))
    elif problem == "rp1":
        w = wl.riemann_1d("RP1", n)
        w["p"] = np.where(w["x"][0] < 0.5, w["p"] * (1.0 + 0.02 * u), w["p"])
    elif problem == "octant":
        w = wl.spherical_shock_3d(n)
        w["p"] = np.where(w["rho"] > 1.0, w["p"] * (1.0 + 0.02 * u), w["p"])
    elif problem == "mach":
        w = wl.mach_reflection("D1", n, n // 2, "MM", foot=0.4 + 0.03 * u)
        w["rho"] = w["rho"] * (1.0 + 1e-3 * u)
    elif problem == "vortex":
        w = wl.isentropic_vortex(n, eps_v=5.0 + 0.3 * u)
    else:
        w = wl.riemann_2d(n, seed=int(rng.integers(1 << 30)))
    return w


def _mesh_inputs(case, seed, device):
    """Primitive fields and a smoothly moved mesh on n1 x n2 nodes: four seeded quadrant states with a ripple."""
    rng = np.random.default_rng(seed)
    st = torch.tensor(np.array(wl.quadrant_states(int(rng.integers(1 << 30)))), dtype=torch.float64, device=device)
    ph = rng.uniform(0.0, 2.0 * np.pi, 2)
    n1, n2 = case["n1"], case["n2"]
    X = torch.linspace(0.0, 1.0, n1, dtype=torch.float64, device=device)[None, :].expand(n2, n1)
    Y = torch.linspace(0.0, 1.0, n2, dtype=torch.float64, device=device)[:, None].expand(n2, n1)
    q = torch.where(X > 0.5, torch.where(Y > 0.5, 0, 3), torch.where(Y > 0.5, 1, 2))
    rho = st[q, 0] * (1.0 + 0.01 * torch.sin(6 * np.pi * X + ph[0]) * torch.sin(4 * np.pi * Y + ph[1]))
    v = torch.stack([st[q, 1], st[q, 2]])
    p = st[q, 3]
    bump = 0.02 * torch.sin(np.pi * X) * torch.sin(np.pi * Y)
    x = torch.stack([X + bump * torch.cos(2 * np.pi * Y), Y + bump * torch.sin(2 * np.pi * X)])
    w = dict(gas=wl.UNITS_A, dim=2, n=(n2, n1), dxi=(1.0 / (n1 - 1), 1.0 / (n2 - 1)), bc=("outflow", "outflow"),
             period=(1.0, 1.0), cfl=0.4, moving=True,
             mesh=dict(monitor="vdw", alphas=(1200.0, 1200.0, 1200.0), kappa=2, filter_passes=case["passes"],
                       sweeps=case["sweeps"], eps=0.0))
    return w, rho.contiguous(), v.contiguous(), p.contiguous(), x.contiguous()


MESH_DT = 1e-4                       # the step a redistribution's velocity belongs to


def _tube_batch(case, seed):
    # the lengths belong to the case (they are the plan's), the states to the seed
    lengths = np.random.default_rng(12345).integers(case["lmin"], case["lmax"] + 1, size=case["tubes"])
    return wl.shock_tube_batch(lengths=lengths, seed=seed)


def _snapshots(case, seed, device):
    """Features [B][4][n][n] and target displacements [B][2][n][n]: smooth random fields of the sizes that ln omega,
    G/(1 + |G|) and displacements in cells take."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    B, n = case["batch"], case["n"]

    def smooth(c, scale):
        a = torch.randn((B, c, 18, 18), generator=g, device=device, dtype=torch.float32)
        a = torch.nn.functional.interpolate(a, size=(n, n), mode="bicubic", align_corners=True)
        return a * torch.tensor(scale, device=device, dtype=torch.float32)[None, :, None, None]

    return smooth(4, (1.5, 0.4, 4.0, 4.0)).contiguous(), smooth(2, (1.0, 1.0)).contiguous()


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "steps":
        w = _workload(case, seed)
        ctx, JU, J, x = es.setup_workload(w, case["form"], dev)
        parts = (JU, J, x)
        # one buffer with the three arrays in a row, so that going back to the first state is one copy
        flat0 = torch.cat([a.reshape(-1).view(torch.float64) for a in parts])
        flat = flat0.clone()
        views, at = [], 0
        for a in parts:
            m = a.numel() * a.element_size() // 8
            views.append(flat[at:at + m].view(a.dtype).view(a.shape))
            at += m
        return dict(case=case, ctx=ctx, flat=flat, flat0=flat0, state=views)
    if case["kind"] == "mesh":
        w, rho, v, p, x = _mesh_inputs(case, seed, dev)
        ctx = es.es_create(es.make_params(w, precision=case["form"]))
        J = es.state_empty(ctx, x.shape[1:], dev)
        es.es_init_mesh(ctx, x, J)
        JU = es.state_empty(ctx, (4,) + tuple(x.shape[1:]), dev)
        es.es_prim_to_cons(ctx, rho, v, p, J, JU)
        return dict(case=case, ctx=ctx, JU=JU, J=J, x=x, xdot=torch.empty_like(x))
    if case["kind"] == "tubes":
        batch = _tube_batch(case, seed)
        b = es.es_batch_create(es.batch_params(batch["gas"]), batch["lengths"])
        prim = [torch.tensor(a, dtype=torch.float64, device=dev) for a in wl.batch_fields(batch)]
        out = [torch.empty((3, b.ntot), dtype=torch.float64, device=dev)] + \
              [torch.empty(b.ntot, dtype=torch.float64, device=dev) for _ in range(2)]
        return dict(case=case, b=b, prim=prim, out=out)
    feats, tgts = _snapshots(case, seed, dev)
    net = learned.WarmStartNet(hidden=32, layers=4, seed=seed, in_scale=learned.feature_scale(feats), device=dev)
    return dict(case=case, net=net, feats=feats, tgts=tgts)


def run(state):
    case = state["case"]
    if case["kind"] == "steps":
        JU, J, x = state["state"]
        state["flat"].copy_(state["flat0"])
        es.es_steps(state["ctx"], JU, J, x, case["steps"], FOREVER)
        return dict(JU=JU, J=J, x=x)
    if case["kind"] == "mesh":
        es.es_mesh_redistribute(state["ctx"], state["JU"], state["J"], state["x"], MESH_DT, state["xdot"], stats=False)
        return dict(xdot=state["xdot"])
    if case["kind"] == "tubes":
        es.es_batch_set_prim(state["b"], *state["prim"])
        es.es_batch_steps(state["b"], case["steps"], FOREVER)
        es.es_batch_get(state["b"], *state["out"])
        return dict(zip(("JU", "J", "x"), state["out"]))
    net = state["net"]
    loss = net.train_step(state["feats"], state["tgts"], 2e-3)
    return dict(loss=loss, gw=net.gw, gb=net.gb)


#: operations per node and RK stage of the 3D operator: three directions of three pair fluxes and one face (the 2D
#: count for its two directions, with the fifth component's reconstructions and the 3D frame)
STAGE_FLOPS_3D = 8500


def _mesh_flops(dim, passes, sweeps):
    return 60 + 20 * dim + passes * 2 * 3 ** dim + sweeps * 10 * dim


def work(case):
    if case["kind"] == "steps":
        dim = {"sine1d": 1, "rp1": 1, "sine3d": 3, "octant": 3}.get(case["problem"], 2)
        n = case["n"]
        nodes = n * (n // 2) if case["problem"] == "mach" else n ** dim
        stage = STAGE_FLOPS_3D if dim == 3 else perfmodel.flops_per_node_stage(dim)
        mesh = {"rp1": (5, 10), "riemann2d": (5, 5), "mach": (5, 10), "sine3d": (20, 10), "octant": (5, 10)}
        flops = 3 * stage + 40 * dim
        if case["problem"] in mesh:
            flops += _mesh_flops(dim, *mesh[case["problem"]])
        return dict(bytes=2 * 8 * (2 * dim + 3) * nodes, flops=flops * nodes * case["steps"])
    if case["kind"] == "mesh":
        nodes = case["n1"] * case["n2"]
        return dict(bytes=8 * (7 + 2) * nodes, flops=_mesh_flops(2, case["passes"], case["sweeps"]) * nodes)
    if case["kind"] == "tubes":
        nodes = case["tubes"] * 0.5 * (case["lmin"] + case["lmax"])
        per = 3 * perfmodel.flops_per_node_stage(1) + 40 + _mesh_flops(1, 5, 5)
        return dict(bytes=8 * (3 + 5) * nodes, flops=per * nodes * case["steps"])
    pixels = case["batch"] * case["n"] ** 2
    macs = 9 * (4 * 32 + 2 * 32 * 32 + 32 * 2)
    return dict(bytes=4 * (4 + 2) * pixels, flops=2 * pixels * (3 * macs - 9 * 4 * 32))


# ------------------------------------------------------------------------------------------------ in 64 bits

ALPHA = (1.5, -0.3, 1.0 / 30.0)      # weights of the 6th-order combination


def _logmean(a, b):
    f = (a - b) / (a + b)
    u = f * f
    series = 1 + u * (1 / 3 + u * (1 / 5 + u * (1 / 7 + u * (1 / 9 + u / 11))))
    F = torch.where(f.abs() < 1e-2, series, torch.atanh(f) / torch.where(f == 0, torch.ones_like(f), f))
    return (a + b) / (2 * F)


def _mean(a, b):
    return 0.5 * (a + b)


class _Scheme:
    """The scheme on one mesh: fields are [n3][n2][n1] tensors, direction k is the axis -1 - k."""

    def __init__(self, w, sign_tol):
        g = w["gas"]
        self.a, self.b, self.R, self.cv = g["a"], g["b"], g["R"], g["cv"]
        self.delta = self.R / self.cv
        self.dim, self.bc, self.dxi, self.period = w["dim"], w["bc"], w["dxi"], w["period"]
        self.gam = w.get("weno_gammas", (0.005, 0.045, 0.95))
        self.cfl, self.moving, self.m = w["cfl"], w.get("moving", False), w.get("mesh", {})
        self.tol = sign_tol

    # ---- ghosts: wrap, copy / odd reflection at outflow ends, mirror at walls
    def pad(self, f, k, g, odd=False, shift=0.0, along=True, flip=False):
        ax = f.dim() - 1 - k
        n = f.shape[ax]
        bc = self.bc[k]
        if bc == "periodic":
            return torch.cat([f.narrow(ax, n - g, g) - shift, f, f.narrow(ax, 0, g) + shift], ax)

        def end(first, inner, mirror):
            if odd and not (mirror and along):
                return 2 * first - inner
            if mirror:
                return -inner if flip else inner
            return first.expand(inner.shape)

        lo = end(f.narrow(ax, 0, 1), f.narrow(ax, 1, g).flip(ax), bc in ("reflect", "symmetry_lo"))
        hi = end(f.narrow(ax, n - 1, 1), f.narrow(ax, n - 1 - g, g).flip(ax), bc == "reflect")
        return torch.cat([lo, f, hi], ax)

    def pad_all(self, x, g, shift):
        out = [x[c] for c in range(self.dim)]
        for k in range(self.dim):
            out = [self.pad(out[c], k, g, odd=True, shift=self.period[k] if shift and c == k else 0.0, along=c != k)
                   for c in range(self.dim)]
        return out

    def diff(self, f, k):
        """6th-order central difference along k, on the nodes with three neighbours each side."""
        ax = f.dim() - 1 - k
        n = f.shape[ax] - 6
        return sum(0.5 * al * (f.narrow(ax, 3 + m, n) - f.narrow(ax, 3 - m, n)) for m, al in enumerate(ALPHA, 1))

    def cut(self, f, k, t=3):
        ax = f.dim() - 1 - k
        return f.narrow(ax, t, f.shape[ax] - 2 * t)

    def metrics(self, x, xdot, k):
        """(n_j, J xi_t) of direction k on its nodes with three ghosts along k."""
        xd = self.pad_all(xdot, 3, False)
        xd = [self._only(v, k) for v in xd]
        if self.dim == 1:
            n = [torch.ones_like(xd[0])]
        else:
            xp = self.pad_all(x, 3, True)
            if self.dim == 2:
                o = 1 - k
                d = [self.diff(xp[c], o) / self.dxi[o] for c in range(2)]
                n = [d[1], -d[0]] if k == 0 else [-d[1], d[0]]
            else:
                l, m = (k + 1) % 3, (k + 2) % 3
                n = []
                for j in range(3):
                    p, q = (j + 1) % 3, (j + 2) % 3
                    t1 = self.diff(self.diff(xp[p], l) * self.cut(xp[q], l), m)
                    t2 = self.diff(self.diff(xp[p], m) * self.cut(xp[q], m), l)
                    n.append((t1 - t2) / (self.dxi[l] * self.dxi[m]))
        return n, -sum(a * b for a, b in zip(xd, n))

    def _only(self, f, k):
        for o in range(self.dim):
            if o != k:
                f = self.cut(f, o)
        return f

    def jacobian(self, x):
        xp = self.pad_all(x, 3, True)
        D = [[self._only(self.diff(xp[c], k), k) / self.dxi[k] for k in range(self.dim)] for c in range(self.dim)]
        if self.dim == 1:
            return D[0][0]
        if self.dim == 2:
            return D[0][0] * D[1][1] - D[0][1] * D[1][0]
        return sum(D[0][i] * (D[1][(i + 1) % 3] * D[2][(i + 2) % 3] - D[1][(i + 2) % 3] * D[2][(i + 1) % 3])
                   for i in range(3))

    # ---- gas
    def cons(self, rho, v, p):
        T = (p + self.a * rho ** 2) * (1 - self.b * rho) / (self.R * rho)
        E = rho * (self.cv * T - self.a * rho) + 0.5 * rho * (v ** 2).sum(0)
        return torch.cat([rho[None], rho * v, E[None]])

    def prim(self, U):
        rho = U[0]
        v = U[1:-1] / rho
        T = (U[-1] / rho - 0.5 * (v ** 2).sum(0) + self.a * rho) / self.cv
        return rho, v, T, rho * self.R * T / (1 - self.b * rho) - self.a * rho ** 2

    def sound2(self, rho, T):
        return (1 + self.delta) * self.R * T / (1 - self.b * rho) ** 2 - 2 * self.a * rho

    def fundamental(self, rho, T):
        nu = 1 / rho
        pnn = (1 + self.delta) * (2 + self.delta) * self.R * T / (nu - self.b) ** 3 - 6 * self.a * rho ** 4
        return nu ** 3 * pnn / (2 * self.sound2(rho, T))

    def entropy_vars(self, rho, v, T):
        s = self.cv * T.log() + self.R * ((1 - self.b * rho) / rho).log()
        V0 = self.cv - s - 2 * self.a * rho / T + self.R / (1 - self.b * rho) - 0.5 * (v ** 2).sum(0) / T
        return torch.cat([V0[None], v / T, -1 / T[None]])

    # ---- two-point flux through the mean metrics
    def pair(self, L, R, n, xt):
        (rl, vl, Tl), (rr, vr, Tr) = L, R
        oml, omr = 1 - self.b * rl, 1 - self.b * rr
        Tm, rm = _mean(Tl, Tr), _mean(rl, rr)
        coef = self.R * self.b / (oml * omr) - self.a / Tm
        D = self.R / _logmean(rl, rr) + coef - self.a / Tm
        if self.b > 0:
            D = D + self.R * self.b / _logmean(oml, omr)
        gm = _mean(self.R / oml - self.a * rl / Tl, self.R / omr - self.a * rr / Tr)
        rT, vm, vT = _mean(rl / Tl, rr / Tr), _mean(vl, vr), _mean(vl / Tl, vr / Tr)
        rv = _mean(rl * vl, rr * vr)
        B0 = 0.5 * _mean((vl ** 2).sum(0) / Tl, (vr ** 2).sum(0) / Tr) - self.cv * Tm / _logmean(Tl, Tr) + 2 * self.a * rT
        nn = torch.stack(n)
        Q = xt * (rm * coef + gm) / D + (nn * (rv * coef + gm * vm)).sum(0) / D
        P = rm * Tm * gm
        mom = vm * Q + nn * P
        en = (self.a * rT * (xt * rm + (nn * rv).sum(0)) - B0 * Q + (vT * mom).sum(0)) / _mean(1 / Tl, 1 / Tr)
        return torch.cat([Q[None], mom, en[None]])

    # ---- multi-resolution WENO value at the face right of the middle node of five
    def weno(self, w):
        g1, g2, g3 = self.gam
        e = [a - w[2] for a in w]
        p2 = ((-e[1] + 2 * e[3]) / 6) * (g1 + g2) / g2
        p3 = ((2 * e[0] - 13 * e[1] + 27 * e[3] - 3 * e[4]) / 60 - g2 * p2) / g3
        b1 = torch.minimum(e[1] ** 2, e[3] ** 2)
        b2 = 13 / 12 * (e[1] + e[3]) ** 2 + 0.25 * (e[3] - e[1]) ** 2
        o1, o2, a1, a2 = (e[3] - e[1]) / 2, (e[4] - e[0]) / 2, (e[3] + e[1]) / 2, (e[4] + e[0]) / 2
        c3, c1 = (o2 - 2 * o1) / 6, (34 * o1 - 5 * o2) / 24
        c4, c2 = (a2 - 4 * a1) / 12, (12 * a1 - a2) / 8
        b3 = (c1 * (c1 + 0.5 * c3) + c2 * (13 / 3 * c2 + 4.2 * c4) + 3129 / 80 * c3 ** 2 + 87617 / 140 * c4 ** 2)
        tau = (0.5 * ((b3 - b1).abs() + (b3 - b2).abs())) ** 2
        k = [g * (1 + tau / (b + 1e-6)) for g, b in zip(self.gam, (b1, b2, b3))]
        return w[2] + (k[1] * p2 + k[2] * p3) / (k[0] + k[1] + k[2])

    def frame(self, nf):
        """|n| and the rows of the rotation to the face normal."""
        L = torch.sqrt(sum(a * a for a in nf))
        one, zero = torch.ones_like(L), torch.zeros_like(L)
        if self.dim == 1:
            return L, [[nf[0] / L]]
        if self.dim == 2:
            c, s = nf[0] / L, nf[1] / L
            return L, [[c, s], [-s, c]]
        r = torch.sqrt(nf[0] ** 2 + nf[1] ** 2)
        flat = r <= 1e-12 * L
        safe = torch.where(flat, one, r)
        ct, st = torch.where(flat, one, nf[0] / safe), torch.where(flat, zero, nf[1] / safe)
        cp, sp = r / L, nf[2] / L
        return L, [[cp * ct, cp * st, sp], [-st, ct, zero], [-sp * ct, -sp * st, cp]]

    def faces(self, U, n, xt):
        """Fluxes of JU and J at the N + 1 faces of lines with three ghosts each side (last axis)."""
        d, N = self.dim, xt.shape[-1] - 6

        def at(f, o):
            return f[..., 2 + o:3 + o + N]

        rho, v, T, p = self.prim(U)
        F, FJ = 0.0, 0.0
        for m, al in enumerate(ALPHA, 1):
            for s in range(m):
                l, r = -s, m - s
                x_m = _mean(at(xt, l), at(xt, r))
                F = F + al * self.pair((at(rho, l), at(v, l), at(T, l)), (at(rho, r), at(v, r), at(T, r)),
                                       [_mean(at(c, l), at(c, r)) for c in n], x_m)
                FJ = FJ + al * x_m
        rf = _logmean(at(rho, 0), at(rho, 1))
        q = rho / p
        pf = rf / _logmean(at(q, 0), at(q, 1))
        vf = _mean(at(v, 0), at(v, 1))
        L, rot = self.frame([_mean(at(c, 0), at(c, 1)) for c in n])
        xf = _mean(at(xt, 0), at(xt, 1))
        vr = [sum(a * b for a, b in zip(row, vf)) for row in rot]
        Tf = (pf + self.a * rf ** 2) * (1 - self.b * rf) / (self.R * rf)
        c2 = self.sound2(rf, Tf)
        c = c2.sqrt()
        E = rf * (self.cv * Tf - self.a * rf) + 0.5 * rf * sum(a * a for a in vr)
        H = (E + pf) / rf
        mid = H - c2 * (1 - self.b * rf) / self.delta
        sA = torch.sqrt(rf * Tf / (2 * c2))
        sE = torch.sqrt(self.R * self.delta * rf * Tf ** 2 /
                        ((self.R * Tf - 2 * self.a * rf * (1 - self.b * rf) ** 2) * c2))
        sT = torch.sqrt(rf * Tf)
        one, zero = torch.ones_like(rf), torch.zeros_like(rf)
        vn, vt = vr[0], vr[1:]
        cols = [[one, vn - c, *vt, H - vn * c], [one, vn, *vt, mid]]
        scal = [sA, sE]
        for i in range(d - 1):
            cols.append([zero, zero] + [one if j == i else zero for j in range(d - 1)] + [vt[i]])
            scal.append(sT)
        cols.append([one, vn + c, *vt, H + vn * c])
        scal.append(sA)
        V = self.entropy_vars(rho, v, T)
        TV = []
        for o in range(-2, 4):
            a = at(V, o)
            TV.append([a[0]] + [sum(r * a[1 + j] for j, r in enumerate(row)) for row in rot] + [a[-1]])
        lam = (xf + L * vn).abs() + L * c
        inc = [torch.zeros_like(rf) for _ in range(d + 2)]
        mag = [TV[2][i].abs() + TV[3][i].abs() for i in range(d + 2)]
        for m, (col, sc) in enumerate(zip(cols, scal)):
            W = [sc * sum(a * b for a, b in zip(col, tv)) for tv in TV]
            jw = self.weno(W[5:0:-1]) - self.weno(W[0:5])
            size = sc * sum(a.abs() * b for a, b in zip(col, mag))
            if 2 <= m <= d:
                size = size + sc * c * mag[-1]
            j = W[3] - W[2]
            keep = (jw * j > 0) & (j.abs() > self.tol * size)
            y = torch.where(keep, sc * jw, zero)
            inc = [i + a * y for i, a in zip(inc, col)]
        mom = [sum(rot[r][j] * inc[1 + r] for r in range(d)) for j in range(d)]
        return F - 0.5 * lam * torch.stack([inc[0], *mom, inc[-1]]), FJ

    def rhs(self, JU, J, x, xdot):
        U = JU / J
        dU, dJ = 0.0, 0.0
        for k in range(self.dim):
            Up = torch.stack([self.pad(U[c], k, 3, flip=c == 1 + k) for c in range(self.dim + 2)])
            n, xt = self.metrics(x, xdot, k)
            ax = -1 - k
            FU, FJ = self.faces(Up.movedim(ax, -1), [a.movedim(ax, -1) for a in n], xt.movedim(ax, -1))
            dU = dU - ((FU[..., 1:] - FU[..., :-1]) / self.dxi[k]).movedim(-1, ax)
            dJ = dJ - ((FJ[..., 1:] - FJ[..., :-1]) / self.dxi[k]).movedim(-1, ax)
        return dU, dJ

    def time_step(self, JU, J, x, xdot):
        rho, v, T, _ = self.prim(JU / J)
        c = self.sound2(rho, T).sqrt()
        tot = 0.0
        for k in range(self.dim):
            n, xt = self.metrics(x, xdot, k)
            n, xt = [self.cut(a, k) for a in n], self.cut(xt, k)
            L = torch.sqrt(sum(a * a for a in n))
            tot = tot + ((xt + sum(a * b for a, b in zip(n, v))).abs() + L * c) / J / self.dxi[k]
        return self.cfl / float(tot.max())

    # ---- mesh redistribution
    def nb(self, f, k, s, **how):
        fp = self.pad(f, k, 1, **how)
        ax = f.dim() - 1 - k
        return fp.narrow(ax, 1 + s, f.shape[ax])

    def monitor(self, JU, J):
        rho, _, T, _ = self.prim(JU / J)
        G = self.fundamental(rho, T)

        def grad(f):
            return sum(((self.nb(f, k, 1) - self.nb(f, k, -1)) / (2 * self.dxi[k])) ** 2 for k in range(self.dim))

        def second(f):
            return sum(((self.nb(f, k, 1) - 2 * f + self.nb(f, k, -1)) / self.dxi[k] ** 2) ** 2
                       for k in range(self.dim))

        al = self.m["alphas"]
        if self.m["monitor"] == "smooth":
            terms = [(al[0], grad(rho).sqrt()), (al[1], second(rho).sqrt())]
        elif self.m["kappa"] == 2:
            terms = [(al[0], grad(rho)), (al[1], grad(G)), (al[2], second(G))]
        else:
            terms = [(al[0], grad(rho)), (al[1], second(G))]
        om = torch.sqrt(1 + sum(a * t / t.max() if float(t.max()) > 0 else 0 * t for a, t in terms))
        for _ in range(self.m["filter_passes"]):
            for k in range(self.dim):
                om = 0.25 * self.nb(om, k, -1) + 0.5 * om + 0.25 * self.nb(om, k, 1)
        return om

    def redistribute(self, JU, J, x, dt):
        om = self.monitor(JU, J)
        D = range(self.dim)
        wp = [0.5 * (om + self.nb(om, k, 1)) / self.dxi[k] ** 2 for k in D]
        wm = [0.5 * (om + self.nb(om, k, -1)) / self.dxi[k] ** 2 for k in D]
        den = sum(a + b for a, b in zip(wp, wm))
        fixed = torch.zeros_like(x, dtype=torch.bool)
        for k in D:
            ax = x.dim() - 2 - k
            for end, mirror in ((0, self.bc[k] in ("reflect", "symmetry_lo")), (-1, self.bc[k] == "reflect")):
                if self.bc[k] != "periodic":
                    for c in [k] if mirror else D:
                        fixed[c].select(ax, end).fill_(True)

        def beside(y, c, k, s):
            return self.nb(y[c], k, s, odd=True, shift=self.period[k] if c == k else 0.0, along=c != k)

        y = x
        for _ in range(self.m["sweeps"]):
            y = torch.stack([torch.where(fixed[c], y[c], sum(wp[k] * beside(y, c, k, 1) + wm[k] * beside(y, c, k, -1)
                                                             for k in D) / den) for c in D])
        gam = 1.0
        for k in D:
            dx = y[k] - x[k]
            for s in (-1, 1):
                on = dx * s > 0
                room = (beside(x, k, k, s) - x[k]) / (2 * dx)
                if bool(on.any()):
                    gam = min(gam, float(room[on].min()))
        return gam * (y - x) / dt

    def step(self, JU, J, x):
        still = torch.zeros_like(x)
        dt, xdot = self.time_step(JU, J, x, still), still
        if self.moving:
            xdot = self.redistribute(JU, J, x, dt)
            dt = min(dt, self.time_step(JU, J, x, xdot))
        U, G = JU, J
        for a, b, c in ((0.0, 1.0, 0.0), (0.75, 0.25, 1.0), (1 / 3, 2 / 3, 0.5)):
            dU, dG = self.rhs(U, G, x + c * dt * xdot, xdot)
            U, G = a * JU + b * (U + dt * dU), a * J + b * (G + dt * dG)
        return U, G, x + dt * xdot


def _planes(a):
    """A state array as the mixed form's planes: the float nearest to the value, and what is left of it."""
    hi = a.float().double()
    return torch.stack([hi, a - hi])


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    with torch.no_grad():
        if case["kind"] == "steps":
            w = _workload(case, seed)
            sch = _Scheme(w, 1e-12 if case["form"] == "fp64" else 4e-7)
            x, rho, v, p = (torch.tensor(np.ascontiguousarray(w[k]), dtype=torch.float64, device=dev)
                            for k in ("x", "rho", "v", "p"))
            J = sch.jacobian(x)
            JU = sch.cons(rho, v, p) * J
            for _ in range(case["steps"]):
                JU, J, x = sch.step(JU, J, x)
            if case["form"] == "mixed":
                JU, J = _planes(JU), _planes(J)
            return dict(JU=JU, J=J, x=x)
        if case["kind"] == "mesh":
            w, rho, v, p, x = _mesh_inputs(case, seed, dev)
            sch = _Scheme(w, 1e-12)
            J = sch.jacobian(x)
            return dict(xdot=sch.redistribute(sch.cons(rho, v, p) * J, J, x, MESH_DT))
        if case["kind"] == "tubes":
            if case["tubes"] * case["steps"] > 200:             # one tube and step takes about 0.05 s
                return None
            batch = _tube_batch(case, seed)
            got = []
            for k in range(case["tubes"]):
                w = wl.batch_problem(batch, k)
                sch = _Scheme(w, 4e-7)
                x, rho, v, p = (torch.tensor(np.ascontiguousarray(w[q]), dtype=torch.float64, device=dev)
                                for q in ("x", "rho", "v", "p"))
                J = sch.jacobian(x)
                JU = sch.cons(rho, v, p) * J
                for _ in range(case["steps"]):
                    JU, J, x = sch.step(JU, J, x)
                got.append((JU, J, x[0]))
            return dict(JU=torch.cat([a[0] for a in got], 1), J=torch.cat([a[1] for a in got]),
                        x=torch.cat([a[2] for a in got]))
    feats, tgts = _snapshots(case, seed, dev)
    net = learned.WarmStartNet(hidden=32, layers=4, seed=seed, in_scale=learned.feature_scale(feats), device=dev)
    wo, bo = net._offsets()
    ws = [net.w[wo[l]:wo[l + 1]].bfloat16().double().view(net.shapes[l]).requires_grad_() for l in range(net.layers)]
    bs = [net.b[bo[l]:bo[l + 1]].double().requires_grad_() for l in range(net.layers)]
    loss = torch.zeros(1, dtype=torch.float64, device=dev)
    for i in range(case["batch"]):                              # one image at a time: double activations are large
        a = feats[i:i + 1].double()
        for l in range(net.layers):
            # the correlation as nine shifted products
            H, W = a.shape[-2:]
            ap = torch.nn.functional.pad(a, (1, 1, 1, 1))
            z = bs[l][None, :, None, None]
            for t in range(9):
                z = z + torch.einsum("oi,bihw->bohw", ws[l][:, :, t // 3, t % 3],
                                     ap[:, :, t // 3:t // 3 + H, t % 3:t % 3 + W])
            a = torch.tanh(z) if l < net.layers - 1 else z
        part = ((a - tgts[i:i + 1].double()) ** 2).sum() / tgts.numel()
        part.backward()
        loss = loss + part.detach()
    return dict(loss=loss, gw=torch.cat([g.grad.reshape(-1) for g in ws]), gb=torch.cat([g.grad for g in bs]))
