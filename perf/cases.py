"""Performance cases: the work a user of the framework has it do, through the
package's public entry points.

A case is a dict with a "kind":
  step         an advance of the stored state by `steps` SSP-RK3 steps, then the
               new state on the device (Solver.step, Solver.get_state);
  stage        one Runge--Kutta stage on the caller's device arrays (Solver.stage);
  rhs          one residual of a caller's device array (Solver.rhs);
  diagnostics  a state set from outside (a checkpoint) and its macroscopic
               fields, moments, totals and entropy;
  infer        a batch through the learned guess's network (Solver.mlp_infer);
  train        a training of that network on logged pairs (Solver.mlp_train).
The solver kinds name a problem: one of workloads.py's, with its mesh, order
and velocity grid; "octant" is the Taylor--Green box between symmetry planes.

exact() restates the method in FP64 with plain torch operations (the box and
the curvilinear mesh both through the mapped flux form).
"""
import math

import numpy as np
import torch

from paper_2312_06567_gb300 import bgk
from paper_2312_06567_gb300 import workloads as W

EXACT_VALUES = 1.2e9        # state values up to which exact() runs within its time


# ---- cases -------------------------------------------------------------------
def _solver_case(kind, problem, n, p, v, precision="mixed", delta=None, **kw):
    c = {"kind": kind, "problem": problem, "n1": n[0], "n2": n[1], "n3": n[2], "p": p,
         "v1": v[0], "v2": v[1], "v3": v[2], "precision": precision,
         "delta": delta if delta is not None else (2.0 if problem in ("shock", "ogrid") else 0.0),
         "tensor": False, "learned": False, "tune": False, "graphs": False, "steps": 1}
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return dict(c, name=name)
    return [
        # the small plain case at its own size and length: launches and latency
        named("sine_box_10_steps", _solver_case("step", "sine", (4, 4, 4), 1, (8, 8, 8), graphs=True, steps=10)),
        # the throughput case (16 elements along the first axis, full velocity grid; a quarter of
        # its box), set up as in the user guide: tuned, trained guess, graph replay
        named("taylor_green_learned", _solver_case("step", "taylor_green", (16, 16, 4), 3, (24, 24, 24), learned=True,
                                                   tune=True, graphs=True)),
        # the hypersonic normal shock: F and G, p = 2, Dirichlet ends; half its cross-section
        named("normal_shock", _solver_case("step", "shock", (64, 2, 4), 2, (32, 32, 32), tune=True, graphs=True)),
        # the blunt body: curvilinear O-grid, diffuse wall, poles, farfield; 40^3 velocities
        named("sphere_ogrid", _solver_case("step", "ogrid", (6, 12, 12), 1, (40, 40, 40), tune=True, graphs=True)),
        # full double precision, the form results are checked with
        named("taylor_green_fp64", _solver_case("step", "taylor_green", (4, 4, 4), 3, (24, 24, 24), "fp64", tune=True,
                                                graphs=True)),
        # a program with its own integrator: one stage on its own arrays, default settings
        named("stage_call", _solver_case("stage", "taylor_green", (8, 8, 4), 3, (24, 24, 24))),
        # symmetry planes on a reduced domain, default settings, ragged sizes
        named("octant_specular", _solver_case("step", "octant", (7, 6, 5), 2, (24, 22, 20))),
        # a smooth curvilinear mesh, monatomic, residual evaluation
        named("wavy_rhs", _solver_case("rhs", "wavy", (6, 5, 6), 2, (20, 20, 20))),
        # the tensor variant of the ES equilibrium
        named("es_tensor", _solver_case("step", "taylor_green", (6, 5, 4), 3, (20, 20, 20), tensor=True, graphs=True)),
        # restart from a checkpoint and write the monitored quantities
        named("diagnostics", _solver_case("diagnostics", "taylor_green", (8, 8, 4), 3, (24, 24, 24))),
        # the learned guess on its own: a batch of the size it is quoted at, and a training run
        {"name": "mlp_infer_1e6", "kind": "infer", "points": 1000000},
        {"name": "mlp_train", "kind": "train", "n1": 4, "n2": 4, "n3": 4, "p": 3, "epochs": 64},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["stage", "rhs", "diagnostics", "infer", "train"])
    if kind == "infer":
        return {"kind": "infer", "points": _log_int(rng, 1000, 4000000)}
    if kind == "train":
        return {"kind": "train", "n1": rng.randint(1, 6), "n2": rng.randint(2, 6), "n3": rng.randint(1, 6),
                "p": rng.randint(1, 3), "epochs": rng.randint(20, 80)}
    problem = rng.choice(["sine", "taylor_green", "taylor_green", "shock", "ogrid", "octant", "wavy"]) \
        if kind != "diagnostics" else rng.choice(["sine", "taylor_green", "shock"])
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    delta = 2.0 if problem in ("shock", "ogrid") else rng.choice([0.0, 0.0, 2.0])
    p = rng.randint(1, 2) if problem in ("ogrid",) else rng.randint(1, 3) if problem == "wavy" else rng.randint(1, 4)
    while True:
        if problem == "shock":
            n = (_log_int(rng, 8, 48), rng.randint(1, 3), rng.randint(1, 3))
            v = (rng.randint(30, 36), rng.randint(24, 32), rng.randint(24, 32))
        elif problem == "ogrid":
            n = (rng.randint(1, 5), rng.randint(4, 8), rng.randint(4, 9))
            v = tuple(rng.randint(36, 42) for _ in range(3))
        else:
            n = tuple(_log_int(rng, 2, 12) for _ in range(3))
            v = tuple(rng.randint(8, 25) for _ in range(3))
        values = n[0] * n[1] * n[2] * (p + 1) ** 3 * v[0] * v[1] * v[2] * (2 if delta else 1)
        wide = problem in ("shock", "ogrid")         # whose velocity grids cannot be small
        most = (6e7 if wide else 1.5e7) if precision == "fp64" else 1.2e8 if problem in ("ogrid", "octant") else 2e8
        if values <= most:
            break
    return _solver_case(kind, problem, n, p, v, precision, delta,
                        tensor=kind == "step" and delta == 0.0 and rng.random() < 0.15,
                        graphs=kind == "step" and rng.random() < 0.5, steps=rng.randint(1, 3) if kind == "step" else 1)


# ---- problems ------------------------------------------------------------------
def _workload(c):
    n, v = (c["n1"], c["n2"], c["n3"]), (c["v1"], c["v2"], c["v3"])
    name = c["problem"]
    if name == "wavy":
        wl = W.wavy_periodic_box(p=c["p"], n=n, vel_n=v, Pr=0.72)
    elif name == "ogrid":
        wl = W.sphere_ogrid(n=n, p=c["p"]).replace(vel_n=v)
    else:
        base = {"sine": W.periodic_sine_box, "taylor_green": W.taylor_green_box, "octant": W.taylor_green_box,
                "shock": W.normal_shock_tube}[name]()
        wl = W.reduced(base, mesh_n=n, vel_n=v).replace(p=c["p"])
        if name == "octant":
            half = tuple(0.5 * h for h in wl.mesh_hi)
            wl = wl.replace(mesh_hi=half, periodic=(False,) * 3,
                            specular=tuple((d, s) for d in range(3) for s in (-1, 1)))
    return wl.replace(delta=c["delta"], es_tensor=c["tensor"])


def _fields(wl, x, seed):
    """The problem's initial (rho, U, theta) at the nodes with a seeded smooth
    perturbation of a few percent: q[P, 5]."""
    rng = np.random.default_rng(seed)
    P = x.shape[0] * x.shape[1]
    rho, U, theta = wl.init(x)
    rho = np.broadcast_to(rho, x.shape[:-1]).reshape(P)
    U = np.broadcast_to(U, x.shape).reshape(P, 3)
    theta = np.broadcast_to(theta, x.shape[:-1]).reshape(P)
    xs = x.reshape(P, 3)
    span = xs.max(axis=0) - xs.min(axis=0) + 1e-12
    t = 2.0 * math.pi * (xs - xs.min(axis=0)) / span

    def wave():
        k, phase = rng.integers(1, 3, 3), rng.uniform(0.0, 2.0 * math.pi, 3)
        return np.sin(k[0] * t[:, 0] + phase[0]) * np.sin(k[1] * t[:, 1] + phase[1]) * np.sin(k[2] * t[:, 2] + phase[2])
    rho = rho * (1.0 + 0.03 * wave())
    U = U + 0.03 * np.sqrt(theta)[:, None] * np.stack([wave() for _ in range(3)], axis=1)
    theta = theta * (1.0 + 0.03 * wave())
    return np.ascontiguousarray(np.concatenate([rho[:, None], U, theta[:, None]], axis=1))


def _velocities(wl, device):
    """Nodes u[Nu, 3] and trapezoid weights w[Nu], k = k1 + n1 (k2 + n2 k3)."""
    ax, wt = [], []
    for d in range(3):
        ax.append(np.linspace(wl.vel_lo[d], wl.vel_hi[d], wl.vel_n[d]))
        h = (wl.vel_hi[d] - wl.vel_lo[d]) / (wl.vel_n[d] - 1)
        wt.append(np.full(wl.vel_n[d], h))
        wt[d][0] *= 0.5
        wt[d][-1] *= 0.5
    u3, u2, u1 = np.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    w = wt[2][:, None, None] * wt[1][None, :, None] * wt[0][None, None, :]
    u = np.stack([u1.ravel(), u2.ravel(), u3.ravel()], axis=1)
    return torch.from_numpy(u).to(device), torch.from_numpy(w.ravel()).to(device)


def _chunks(n, per, most=2.0e7):
    step = max(1, int(most // max(1, per)))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _maxwellian(u, q):
    """[K, P] isotropic Maxwellian of q[P, 5] at u[K, 3]."""
    c2 = sum((u[:, d:d + 1] - q[None, :, 1 + d]) ** 2 for d in range(3))
    return (q[:, 0] / (2.0 * math.pi * q[:, 4]) ** 1.5)[None, :] * torch.exp(-0.5 * c2 / q[None, :, 4])


def _state_of(wl, q, seed, dtype, device):
    """A state away from equilibrium around q: two Maxwellians per node with
    seeded drifts and temperatures, G = delta theta / 2 F modulated."""
    rng = np.random.default_rng([seed, 1])
    P = q.shape[0]
    qa, qb = q.copy(), q.copy()
    drift = 0.4 * np.sqrt(q[:, 4])[:, None] * rng.uniform(-1.0, 1.0, (P, 3))
    qa[:, 0] *= 0.7
    qa[:, 1:4] -= 0.3 * drift
    qa[:, 4] *= 1.0 + 0.2 * rng.uniform(-1.0, 1.0, P)
    qb[:, 0] *= 0.3
    qb[:, 1:4] += 0.7 * drift
    qb[:, 4] *= 1.2
    ta, tb = torch.from_numpy(qa).to(device), torch.from_numpy(qb).to(device)
    g = torch.from_numpy(0.5 * wl.delta * q[:, 4] * (1.0 + 0.1 * rng.uniform(-1.0, 1.0, P))).to(device)
    u, _ = _velocities(wl, device)
    f = torch.empty((wl.n_comp, wl.n_vel, P), dtype=dtype, device=device)
    for k0, k1 in _chunks(wl.n_vel, P):
        F = _maxwellian(u[k0:k1], ta) + _maxwellian(u[k0:k1], tb)
        f[0, k0:k1] = F
        if wl.n_comp == 2:
            f[1, k0:k1] = g[None, :] * F
    return f.reshape(wl.n_comp, wl.n_vel, wl.n_elem, wl.n_sol)


# ---- preparing and running -------------------------------------------------------
def _network(seed):
    """Weights, normalisation and the scale of features as the solver logs them."""
    rng = np.random.default_rng([seed, 2])
    params = []
    for fan, shape in ((9, (9, 64)), (0, (64,)), (64, (64, 64)), (0, (64,)), (64, (64, 5)), (0, (5,))):
        params.append((rng.standard_normal(shape) * (math.sqrt(2.0 / fan) if fan else 0.1)).astype(np.float32))
    mean = np.array([1.0, 0.0, 0.0, 0.0, 1.0, 3.0, 3.0, 1.0, 0.01])
    std = np.array([0.01, 0.06, 0.06, 0.06, 0.02, 0.01, 0.02, 0.01, 1e-4])
    norm = np.concatenate([mean, std, rng.normal(0.0, 1e-5, 5), 1e-5 * rng.uniform(0.5, 2.0, 5)]).astype(np.float32)
    return params, norm, mean, std


def _features(c, seed):
    _, _, mean, std = _network(seed)
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    x = torch.randn((c["points"], 9), generator=g) * torch.from_numpy(std).float() + torch.from_numpy(mean).float()
    return x.contiguous()


def _dtype(c):
    return torch.float64 if c["precision"] == "fp64" else torch.float32


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "infer":
        s = bgk.Solver(W.reduced(W.periodic_sine_box(), mesh_n=(1, 1, 1)), bgk.BGK_MIXED)
        params, norm, _, _ = _network(seed)
        s.mlp_weights(load=(params, norm))
        x = _features(c, seed).cuda()
        return {"case": c, "solver": s, "x": x, "out": torch.empty((c["points"], 5), dtype=torch.float32, device="cuda")}
    if c["kind"] == "train":
        # every point's pair of one stage (as many pairs as the batch: every run sees the same batches)
        wl = W.reduced(W.taylor_green_box(), mesh_n=(c["n1"], c["n2"], c["n3"]), vel_n=(12, 12, 12)).replace(p=c["p"])
        s = bgk.Solver(wl, bgk.BGK_MIXED)
        s.set_maxwellian(torch.from_numpy(_fields(wl, W.node_positions(wl), seed)).cuda())
        s.mlp_log(True, s.n_points)
        s.step(wl.dt(), 1)
        s.mlp_log(False)
        return {"case": c, "solver": s, "pairs": s.n_points, "seed": int(seed)}
    wl = _workload(c)
    q = _fields(wl, W.node_positions(wl), seed)
    s = bgk.Solver(wl, bgk.BGK_FP64 if c["precision"] == "fp64" else bgk.BGK_MIXED)
    st = {"case": c, "solver": s, "dt": wl.dt()}
    if c["kind"] == "step":
        s.set_maxwellian(torch.from_numpy(q).cuda())
        if c["tune"]:
            s.tune_stage(wl.dt(), reps=1)
        if c["learned"]:
            s.mlp_log(True, 3 * s.n_points)
            s.step(wl.dt(), 1)
            s.mlp_log(False)
            s.mlp_train(epochs=8, batch=4096, lr=2e-3, seed=0)
            s.set_guess(1)
            s.set_maxwellian(torch.from_numpy(q).cuda())
        s.set_graphs(c["graphs"])
        st["out"] = torch.empty(s.shape, dtype=_dtype(c), device="cuda")
        return st
    st["f"] = _state_of(wl, q, seed, _dtype(c), "cuda")
    if c["kind"] == "stage":
        st["fn"] = _state_of(wl, q, seed + 1, _dtype(c), "cuda")
    if c["kind"] in ("stage", "rhs"):
        st["out"] = torch.empty(s.shape, dtype=_dtype(c), device="cuda")
    else:
        st["macro"] = torch.empty((s.n_points, 10), dtype=torch.float64, device="cuda")
        st["moments"] = torch.empty((s.n_points, 11), dtype=torch.float64, device="cuda")
    return st


def run(state):
    c, s = state["case"], state["solver"]
    if c["kind"] == "infer":
        return s.mlp_infer(state["x"], state["out"])
    if c["kind"] == "train":
        loss = s.mlp_train(epochs=c["epochs"], batch=state["pairs"], lr=2e-3, seed=state["seed"])
        params, norm = s.mlp_weights()
        return {"loss": loss, "params": params, "norm": norm}
    if c["kind"] == "step":
        s.step(state["dt"], c["steps"])
        return s.get_state(state["out"])
    if c["kind"] == "stage":
        s.stage(state["fn"], state["f"], state["out"], 0.75, 0.25, 0.25 * state["dt"])
        return state["out"]
    if c["kind"] == "rhs":
        return s.rhs(state["f"], state["out"])
    s.set_state(state["f"])
    return {"macro": s.macro(state["macro"]), "moments": s.moments(state["moments"]), "totals": s.totals(),
            "entropy": s.entropy()}


def work(case):
    """Bytes and operations the path cannot do without.  A stage reads its input
    and f^n (not in a first stage) and writes its output; per state value it
    costs the FR derivative in three directions, the equilibrium, source and
    update, and the moments of the result, and the Q' solve one evaluation."""
    c = case
    if c["kind"] == "infer":
        return {"bytes": 4.0 * 14 * c["points"], "flops": 2.0 * (9 * 64 + 64 * 64 + 64 * 5) * c["points"]}
    if c["kind"] == "train":
        n = float(c["n1"] * c["n2"] * c["n3"] * (c["p"] + 1) ** 3)
        return {"bytes": 4.0 * 14 * n * c["epochs"], "flops": 6.0 * (9 * 64 + 64 * 64 + 64 * 5) * n * c["epochs"]}
    q, comp = c["p"] + 1, 2 if c["delta"] else 1
    dof = float(c["n1"] * c["n2"] * c["n3"] * q ** 3) * c["v1"] * c["v2"] * c["v3"]
    size = 8 if c["precision"] == "fp64" else 4
    stage = dof * (comp * (6.0 * q + 23.0 + 9.0 / q) + 26.0 + 22.0 + 16.0)
    if c["kind"] == "step":
        return {"bytes": 8.0 * dof * comp * size * c["steps"], "flops": 3.0 * stage * c["steps"]}
    if c["kind"] == "stage":
        return {"bytes": 3.0 * dof * comp * size, "flops": stage}
    if c["kind"] == "rhs":
        return {"bytes": 2.0 * dof * comp * size, "flops": stage}
    return {"bytes": dof * comp * size, "flops": 40.0 * dof}


# ---- the method in FP64, plain torch ---------------------------------------------
def _fr(p, device):
    leg = np.polynomial.legendre
    xi, wq = leg.leggauss(p + 1)

    def lag(src, dst):
        return np.array([[np.prod([(t - src[m]) / (src[j] - src[m]) for m in range(len(src)) if m != j])
                          for j in range(len(src))] for t in dst])

    def dlag(src, dst):
        return np.array([[sum(1.0 / (src[j] - src[k]) * np.prod([(t - src[m]) / (src[j] - src[m])
                                                                 for m in range(len(src)) if m not in (j, k)])
                              for k in range(len(src)) if k != j) for j in range(len(src))] for t in dst])
    gr = leg.Legendre.basis(p + 1) + leg.Legendre.basis(p)
    gl = (leg.Legendre.basis(p) - leg.Legendre.basis(p + 1)) * (-1.0) ** p
    one = np.array([-1.0, 1.0])
    ends = lag(xi, one)
    lob = np.array([-1.0, 1.0]) if p == 1 else np.concatenate([[-1.0], np.sort(leg.Legendre.basis(p).deriv().roots().real),
                                                               [1.0]])
    t = {"D": dlag(xi, xi), "lm": ends[0], "lp": ends[1], "dgL": 0.5 * gl.deriv()(xi), "dgR": 0.5 * gr.deriv()(xi),
         "w": wq, "to_lob": lag(xi, lob), "Dlob": dlag(lob, lob), "lob_to_gl": lag(lob, xi), "lob_to_end": lag(lob, one)}
    return {k: torch.from_numpy(np.ascontiguousarray(v)).to(device) for k, v in t.items()}


def _line(M, f, ax):
    """Apply M[a, i] along axis ax of f."""
    return torch.movedim(torch.tensordot(f, M, dims=([ax], [1])), -1, ax)


class _Exact:
    """One problem in FP64: states f[C, Nu, n3, n2, n1, q, q, q] (i3, i2, i1)."""

    def __init__(self, c, device):
        self.wl = wl = _workload(c)
        self.dev = device
        self.q = wl.p + 1
        self.fr = _fr(wl.p, device)
        self.u, self.w = _velocities(wl, device)
        self.es = c["tensor"]
        q, n = self.q, wl.mesh_n
        self.grid = (n[2], n[1], n[0], q, q, q)
        self.eax, self.nax = (2, 1, 0), (5, 4, 3)            # element and node axes of direction d in `grid`
        x = W.node_positions(wl) if wl.mapping is not None else None
        if x is None:
            h = [(wl.mesh_hi[d] - wl.mesh_lo[d]) / n[d] for d in range(3)]
            J = h[0] * h[1] * h[2] / 8.0
            self.J = torch.full(self.grid, J, dtype=torch.float64, device=device)
            self.S = [[torch.full(self.grid, 2.0 * J / h[d] if i == d else 0.0, dtype=torch.float64, device=device)
                       for i in range(3)] for d in range(3)]
        else:
            self._metrics(torch.from_numpy(x).to(device))
        self.face = {}
        for d in range(3):
            for side, end in ((0, "lm"), (1, "lp")):
                if x is None:
                    v = [_line(self.fr[end][None], self.S[d][i], self.nax[d]).squeeze(self.nax[d]) for i in range(3)]
                else:
                    v = self.ends[d][side]
                self.face[d, side] = v
            if x is not None:                                  # the two sides' traces of a shared face, averaged
                for i in range(3):
                    L, R = self.face[d, 0][i], self.face[d, 1][i]
                    m = 0.5 * (R + torch.roll(L, -1, self.eax[d]))
                    keep = torch.zeros(L.shape[self.eax[d]], dtype=torch.bool, device=device)
                    keep[-1] = not wl.periodic[d]
                    sh = [1] * L.ndim
                    sh[self.eax[d]] = -1
                    keep = keep.reshape(sh)
                    R2 = torch.where(keep, R, m)
                    L2 = torch.where(torch.roll(keep, 1, self.eax[d]), L, torch.roll(m, 1, self.eax[d]))
                    self.face[d, 0][i], self.face[d, 1][i] = L2, R2

    def _metrics(self, x):
        """Conservative curl form of S^d = J grad xi_d on the Gauss--Lobatto points."""
        fr = self.fr
        X = [x[:, :, i].reshape(self.grid) for i in range(3)]

        def all3(M, f):
            for a in self.nax:
                f = _line(M, f, a)
            return f
        G = [all3(fr["to_lob"], Xi) for Xi in X]
        dG = [[_line(fr["Dlob"], g, self.nax[d]) for d in range(3)] for g in G]
        Sl = [[None] * 3 for _ in range(3)]
        for n in range(3):
            m, l = (n + 1) % 3, (n + 2) % 3
            V = [G[l] * dG[m][d] for d in range(3)]
            for i in range(3):
                j, k = (i + 1) % 3, (i + 2) % 3
                Sl[i][n] = -(_line(fr["Dlob"], V[k], self.nax[j]) - _line(fr["Dlob"], V[j], self.nax[k]))
        self.S = [[all3(fr["lob_to_gl"], Sl[d][i]) for i in range(3)] for d in range(3)]
        a = [[_line(fr["D"], Xi, self.nax[d]) for d in range(3)] for Xi in X]
        self.J = (a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) - a[0][1] * (a[1][0] * a[2][2] - a[1][2] * a[2][0])
                  + a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]))
        self.ends = {}
        for d in range(3):
            self.ends[d] = [[], []]
            for side in (0, 1):
                for i in range(3):
                    v = Sl[d][i]
                    for e in range(3):
                        v = _line(fr["lob_to_end"][side:side + 1] if e == d else fr["lob_to_gl"], v, self.nax[e])
                    self.ends[d][side].append(v.squeeze(self.nax[d]))

    # -- moments and the equilibrium --
    def moments(self, f):
        P = self.J.numel()
        u, w = self.u, self.w
        cols = [torch.ones_like(w), u[:, 0], u[:, 1], u[:, 2], u[:, 0] ** 2, u[:, 1] ** 2, u[:, 2] ** 2,
                u[:, 0] * u[:, 1], u[:, 0] * u[:, 2], u[:, 1] * u[:, 2]]
        B = torch.stack([w * c for c in cols])
        m = torch.zeros((11, P), dtype=torch.float64, device=self.dev)
        for k0, k1 in _chunks(len(w), P):
            m[:10] += B[:, k0:k1] @ f[0, k0:k1].reshape(k1 - k0, P).double()
            if self.wl.n_comp == 2:
                m[10] += w[k0:k1] @ f[1, k0:k1].reshape(k1 - k0, P).double()
        return m

    def macroscopic(self, m):
        wl = self.wl
        rho = m[0]
        U = m[1:4] / rho
        E = 0.5 * (m[4] + m[5] + m[6]) + m[10]
        gamma = (5.0 + wl.delta) / (3.0 + wl.delta)
        pres = (gamma - 1.0) * (E - 0.5 * rho * (U * U).sum(0))
        theta = pres / rho
        mu = wl.mu_ref * torch.ones_like(theta)
        if wl.theta_S >= 0:
            r = theta / wl.theta_ref
            mu = wl.mu_ref * r ** 1.5 * (wl.theta_ref + wl.theta_S) / (theta + wl.theta_S)
        return rho, U, E, gamma, pres, theta, mu

    def equilibrium(self, m):
        """(c0, V[3], A[3, 3], G factor, 1/tau) per point: g = exp(c0 - c^T A c / 2), c = u - V."""
        wl = self.wl
        rho, U, E, _, pres, theta, mu = self.macroscopic(m)
        Pi = torch.empty((len(rho), 3, 3), dtype=torch.float64, device=self.dev)
        for j, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            Pi[:, a, b] = Pi[:, b, a] = m[4 + j] - rho * U[a] * U[b]
        B = (1.0 - 1.0 / wl.Pr) * Pi / rho[:, None, None]
        eye = torch.eye(3, dtype=torch.float64, device=self.dev)
        x = torch.cat([rho[None], U, theta[None]]).T.contiguous()
        Q = torch.stack([rho, m[1], m[2], m[3], E], dim=1)
        c0 = torch.empty_like(rho)
        A = torch.empty_like(Pi)
        for p0, p1 in _chunks(len(rho), len(self.w), 4.0e6):
            y = x[p0:p1]
            for it in range(14):
                T = B[p0:p1] + (y[:, 4] / wl.Pr)[:, None, None] * eye
                Ai = torch.linalg.inv(T)
                lc = torch.log(y[:, 0]) - 0.5 * torch.log(torch.linalg.det(2.0 * math.pi * T))
                c = self.u[:, None, :] - y[None, :, 1:4]
                Ac = torch.einsum("pij,kpj->kpi", Ai, c)
                g = torch.exp(lc[None] - 0.5 * (c * Ac).sum(-1)) * self.w[:, None]
                psi = torch.cat([torch.ones_like(self.u[:, :1]), self.u, 0.5 * (self.u ** 2).sum(1, keepdim=True)], dim=1)
                tr = Ai[:, 0, 0] + Ai[:, 1, 1] + Ai[:, 2, 2]
                cols = [g / y[None, :, 0]] + [g * Ac[:, :, d] for d in range(3)] + [g * ((Ac * Ac).sum(-1) - tr) / (2.0 * wl.Pr)]
                R = (psi.T @ g).T - Q[p0:p1]
                M0 = g.sum(0)
                hd = 0.5 * wl.delta
                R[:, 4] += hd * y[:, 4] * M0
                Jm = torch.stack([(psi.T @ col).T for col in cols], dim=2)
                Jm[:, 4, :] += hd * y[:, 4:5] * torch.stack([col.sum(0) for col in cols], dim=1)
                Jm[:, 4, 4] += hd * M0
                sc = torch.maximum(torch.maximum(R[:, 0].abs() / rho[p0:p1], R[:, 4].abs() / E[p0:p1].abs()),
                                   R[:, 1:4].abs().amax(1) / (rho[p0:p1] * theta[p0:p1].sqrt()))
                if it == 13 or float(sc.max()) < 2e-14:
                    break
                dy = torch.linalg.solve(Jm, -R)
                lam = torch.ones_like(rho[p0:p1])
                for _ in range(20):
                    bad = (y[:, 0] + lam * dy[:, 0] <= 0) | (y[:, 4] + lam * dy[:, 4] <= 0.1 * y[:, 4])
                    lam = torch.where(bad, 0.5 * lam, lam)
                y = y + lam[:, None] * dy
            x[p0:p1], c0[p0:p1], A[p0:p1] = y, lc, Ai
        V = x[:, 1:4]
        if self.es:
            c0, V, A = self._tensor(rho, U, theta, Pi, c0, V, A)
        return c0, V, A, 0.5 * wl.delta * x[:, 4], wl.Pr * pres / mu

    def _tensor(self, rho, U, theta, Pi, c0, V, A):
        """The discrete Gaussian with the full target stress: Newton on its ten natural parameters."""
        ex = ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1))
        Pr = self.wl.Pr
        t = torch.zeros((len(rho), 10), dtype=torch.float64, device=self.dev)
        t[:, 0] = rho
        for j, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            t[:, 4 + j] = (1.0 - 1.0 / Pr) * Pi[:, a, b] + (rho * theta / Pr if a == b else 0.0)
        d = V - U.T
        Ad = torch.einsum("pij,pj->pi", A, d)
        b = torch.stack([c0 - 0.5 * (d * Ad).sum(1), Ad[:, 0], Ad[:, 1], Ad[:, 2], -0.5 * A[:, 0, 0], -0.5 * A[:, 1, 1],
                         -0.5 * A[:, 2, 2], -A[:, 0, 1], -A[:, 0, 2], -A[:, 1, 2]], dim=1)
        for p0, p1 in _chunks(len(rho), len(self.w), 2.0e6):
            ut = self.u[:, None, :] - U.T[None, p0:p1]
            phi = torch.stack([ut[..., 0] ** e[0] * ut[..., 1] ** e[1] * ut[..., 2] ** e[2] for e in ex], dim=-1)
            phi = phi.permute(1, 0, 2).contiguous()            # [P, K, 10]
            y = b[p0:p1]
            for _ in range(8):
                g = torch.exp((phi @ y[:, :, None])[:, :, 0]) * self.w[None]
                wp = phi * g[:, :, None]
                R = wp.sum(1) - t[p0:p1]
                y = y + torch.linalg.solve(wp.transpose(1, 2) @ phi, -R)
            b[p0:p1] = y
        A = torch.empty_like(A)
        for j, (i, k) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
            A[:, i, k] = A[:, k, i] = -b[:, 4 + j] * (2.0 if i == k else 1.0)
        d = torch.linalg.solve(A, b[:, 1:4])
        return b[:, 0] + 0.5 * (b[:, 1:4] * d).sum(1), U.T + d, A

    # -- advection --
    def _dirichlet(self, d, side, k0, k1):
        """Exterior value per component and velocity, or None."""
        wl, s = self.wl, -1 if side == 0 else 1
        if (d, s) in wl.dirichlet:
            r, U, th = wl.dirichlet[(d, s)]
        elif (d, s) in wl.diffuse:
            (U, th), r = wl.diffuse[(d, s)], 1.0
        else:
            return None
        M = _maxwellian(self.u[k0:k1], torch.tensor([[r, U[0], U[1], U[2], th]], dtype=torch.float64, device=self.dev))[:, 0]
        return [M, 0.5 * wl.delta * th * M][:wl.n_comp]

    def _edge(self, f, d, side):
        """The trace of f[..., grid] on the face `side` of the elements at that end of axis d."""
        o = f.ndim - 6
        e = f.narrow(o + self.eax[d], 0 if side == 0 else f.shape[o + self.eax[d]] - 1, 1)
        return _line(self.fr["lm" if side == 0 else "lp"][None], e, o + self.nax[d]).squeeze(o + self.nax[d])

    def wall_density(self, f):
        out = {}
        for (d, s) in self.wl.diffuse:
            side = 0 if s < 0 else 1
            sel = [v.narrow(self.eax[d], 0 if side == 0 else v.shape[self.eax[d]] - 1, 1) for v in self.face[d, side]]
            num = torch.zeros_like(sel[0])
            den = torch.zeros_like(sel[0])
            for k0, k1 in _chunks(len(self.w), self.J.numel()):
                u = self.u[k0:k1]
                un = sum(u[:, i].reshape((-1,) + (1,) * 5) * sel[i][None] for i in range(3)) * s
                wk = self.w[k0:k1].reshape((-1,) + (1,) * 5)
                tr = self._edge(f[0, k0:k1].double(), d, side)
                M = self._dirichlet(d, side, k0, k1)[0].reshape((-1,) + (1,) * 5)
                num += (wk * un.clamp(min=0.0) * tr).sum(0)
                den += (wk * un.clamp(max=0.0) * M).sum(0)
            out[d, side] = -num / den
        return out

    def residual(self, f, n=None, a=0.0, b=0.0, c=1.0):
        """a f^n + b f + c R(f), a new FP64 tensor shaped as f."""
        wl, fr = self.wl, self.fr
        P = self.J.numel()
        c0, V, A, gfac, itau = self.equilibrium(self.moments(f))
        rho_w = self.wall_density(f)
        n1, n2 = wl.vel_n[0], wl.vel_n[1]
        ks = torch.arange(len(self.w), device=self.dev)
        idx = [ks % n1, (ks // n1) % n2, ks // (n1 * n2)]
        out = torch.empty(f.shape, dtype=torch.float64, device=self.dev)
        one = (-1,) + (1,) * 6
        for k0, k1 in _chunks(len(self.w), P):
            u = self.u[k0:k1]
            cc = [u[:, i:i + 1] - V[None, :, i] for i in range(3)]
            ex = sum(A[None, :, i, j] * cc[i] * cc[j] for i in range(3) for j in range(3))
            g = torch.exp(c0[None] - 0.5 * ex)
            for comp in range(wl.n_comp):
                F = f[comp, k0:k1].double()
                div = torch.zeros_like(F)
                for d in range(3):
                    ea, na = self.eax[d] + 1, self.nax[d] + 1
                    Ft = F * sum(u[:, i].reshape(one) * self.S[d][i][None] for i in range(3) if wl.mapping is not None or i == d)
                    trL, trR = (_line(fr[e][None], F, na).squeeze(na) for e in ("lm", "lp"))
                    FI = []
                    for side in (0, 1):
                        un = sum(u[:, i].reshape(one[:-1]) * self.face[d, side][i][None] for i in range(3))
                        ext = torch.roll(trR, 1, ea) if side == 0 else torch.roll(trL, -1, ea)
                        own = trL if side == 0 else trR
                        flux_own = un < 0 if side == 0 else un > 0
                        s = -1 if side == 0 else 1
                        if not wl.periodic[d]:
                            at = 0 if side == 0 else F.shape[ea] - 1
                            if (d, s) in wl.closed:
                                un = un.clone()
                                un.narrow(ea, at, 1).zero_()
                            elif (d, s) in wl.specular:
                                m = list(idx)
                                m[d] = wl.vel_n[d] - 1 - m[d]
                                km = (m[0] + n1 * (m[1] + n2 * m[2]))[k0:k1]
                                ext.narrow(ea, at, 1).copy_(self._edge(f[comp][km].double(), d, side))
                            else:
                                e = self._dirichlet(d, side, k0, k1)[comp].reshape(one[:-1])
                                ext.narrow(ea, at, 1).copy_(e * rho_w[d, side][None] if (d, side) in rho_w
                                                            else e.expand_as(ext.narrow(ea, at, 1)))
                        FI.append(un * torch.where(flux_own, own, ext))
                    tL, tR = (_line(fr[e][None], Ft, na).squeeze(na) for e in ("lm", "lp"))
                    sh = [1] * F.ndim
                    sh[na] = -1
                    div += _line(fr["D"], Ft, na)
                    div += (FI[1] - tR).unsqueeze(na) * fr["dgR"].reshape(sh) + (FI[0] - tL).unsqueeze(na) * fr["dgL"].reshape(sh)
                eq = g if comp == 0 else g * gfac[None]
                R = (eq.reshape(F.shape) - F) * itau.reshape(self.grid)[None] - div / self.J[None]
                o = c * R + b * F
                if a:
                    o += a * n[comp, k0:k1].double()
                out[comp, k0:k1] = o
        return out

    def step(self, f, dt):
        f1 = self.residual(f, None, 0.0, 1.0, dt)
        f2 = self.residual(f1, f, 0.75, 0.25, 0.25 * dt)
        del f1
        return self.residual(f2, f, 1.0 / 3.0, 2.0 / 3.0, 2.0 / 3.0 * dt)

    def diagnostics(self, f):
        wl, fr = self.wl, self.fr
        m = self.moments(f)
        rho, U, E, gamma, pres, theta, mu = self.macroscopic(m)
        lam = mu / rho * torch.sqrt(math.pi / (2.0 * theta))
        r = rho.reshape(self.grid)
        g2 = torch.zeros_like(r)
        for d in range(3):
            ea, na = self.eax[d], self.nax[d]
            trL, trR = (_line(fr[e][None], r, na).squeeze(na) for e in ("lm", "lp"))
            oL, oR = torch.roll(trR, 1, ea), torch.roll(trL, -1, ea)
            if not wl.periodic[d]:
                oL.narrow(ea, 0, 1).fill_(wl.dirichlet[(d, -1)][0])
                oR.narrow(ea, r.shape[ea] - 1, 1).fill_(wl.dirichlet[(d, 1)][0])
            sh = [1] * 6
            sh[na] = -1
            der = _line(fr["D"], r, na) + (0.5 * (oL - trL)).unsqueeze(na) * fr["dgL"].reshape(sh) \
                + (0.5 * (oR - trR)).unsqueeze(na) * fr["dgR"].reshape(sh)
            g2 += (2.0 * wl.mesh_n[d] / (wl.mesh_hi[d] - wl.mesh_lo[d]) * der) ** 2
        gn = torch.sqrt(g2).reshape(-1)
        mach = torch.sqrt((U * U).sum(0) / (gamma * theta))
        macro = torch.stack([rho, U[0], U[1], U[2], theta, pres, mach, lam, gn, lam * gn / rho], dim=1)
        w3 = self.fr["w"]
        Wq = (w3[:, None, None] * w3[None, :, None] * w3[None, None, :]).reshape(-1)
        Wp = (Wq[None] * self.J.reshape(wl.n_elem, -1)).reshape(-1)
        tot = np.array([float((Wp * v).sum()) for v in (rho, m[1], m[2], m[3], E)])
        H = torch.zeros_like(rho)
        for k0, k1 in _chunks(len(self.w), len(rho)):
            F = f[0, k0:k1].reshape(k1 - k0, -1).double()
            H += self.w[k0:k1] @ (F * torch.log(F))
        return {"macro": macro, "moments": m.T.contiguous(), "totals": tot, "entropy": float((Wp * H).sum())}


def exact(case, seed):
    c = dict(case)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if c["kind"] == "train":
        return None                      # many optimiser steps on BF16 operands have no 64-bit value of their own
    if c["kind"] == "infer":
        if c["points"] > 20000000:
            return None
        params, norm, _, _ = _network(seed)

        def bf16(t):
            return t.float().to(torch.bfloat16).double()
        p = [torch.from_numpy(v).to(device).double() for v in params]
        nm = torch.from_numpy(norm).to(device)
        x = _features(c, seed).to(device)
        h = bf16((x - nm[:9]) / nm[9:18])
        for k in (0, 2):
            z = h @ bf16(p[k]) + p[k + 1]
            h = bf16(z * torch.sigmoid(z))
        return (h @ bf16(p[4]) + p[5]) * nm[23:28].double() + nm[18:23].double()
    wl = _workload(c)
    if wl.dof * wl.n_comp > EXACT_VALUES or (c["tensor"] and wl.dof * c["steps"] > EXACT_VALUES / 8):
        return None
    ex = _Exact(c, device)
    q = _fields(wl, W.node_positions(wl), seed)
    shape = (wl.n_comp, wl.n_vel) + ex.grid
    if c["kind"] == "step":
        qt = torch.from_numpy(q).to(device)
        f = torch.empty((wl.n_comp, wl.n_vel, len(q)), dtype=_dtype(c), device=device)
        for k0, k1 in _chunks(wl.n_vel, len(q)):
            f[0, k0:k1] = _maxwellian(ex.u[k0:k1], qt)
            if wl.n_comp == 2:
                f[1, k0:k1] = 0.5 * wl.delta * qt[None, :, 4] * _maxwellian(ex.u[k0:k1], qt)
        f = f.reshape(shape)
        for _ in range(c["steps"]):
            f = ex.step(f, wl.dt())
        return f.reshape(wl.n_comp, wl.n_vel, wl.n_elem, wl.n_sol)
    f = _state_of(wl, q, seed, _dtype(c), device).reshape(shape)
    if c["kind"] == "diagnostics":
        return ex.diagnostics(f)
    if c["kind"] == "rhs":
        return ex.residual(f).reshape(wl.n_comp, wl.n_vel, wl.n_elem, wl.n_sol)
    fn = _state_of(wl, q, seed + 1, _dtype(c), device).reshape(shape)
    return ex.residual(f, fn, 0.75, 0.25, 0.25 * wl.dt()).reshape(wl.n_comp, wl.n_vel, wl.n_elem, wl.n_sol)
