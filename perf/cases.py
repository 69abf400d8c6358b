"""The calls whose speed matters to a user of this package, from the smallest to the largest.

A case is a scene (what cloth, how many nodes, what obstacles, which solver
options) and a call on it:
  step      one time step of one cloth (``Cloth.step``)
  solve     the global-step solve P^-1 rhs on its own (``global_solve``)
  rollout   several steps forward (``rollout``)
  grad      a rollout and its adjoint (``rollout`` + ``backward``)
  autograd  the same through ``rollout_fn`` and torch's autograd
  fit       new material parameters, a rollout, and the adjoint of a trajectory
            loss: one evaluation of a parameter fit (``set_params`` + ``rollout`` +
            ``backward`` with per-step gradients)
  serve     a round of requests through a ``Server``
Scene families: "hang" (two pinned corners, over a sphere), "drape" (unpinned,
over a sphere and the ground), "capsules" (eight random capsules and the ground,
h = 1/240 s), "slide" (on an incline past its friction angle), and with more than
one cloth a batch of "drape" cloths of random grid sizes in one context.

The material and the obstacles follow from the case's ``scene`` number; the
positions, velocities and loss gradients follow from the seed.  The cloth starts
2 mm above the highest obstacle, moves down at about 1 m/s and expands at about
1 per second (in tension: a compressed cloth's adjoint systems are near singular),
so that contact, sticking and slipping set in within the first steps.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2106_05306_gb300 as dc

GRAVITY = (0.0, -9.8, 0.0)
DENSITY, MARGIN, PD_ITERS = 0.1, 1e-6, 20

# ---------------------------------------------------------------------- cases

_DEFAULTS = dict(call="rollout", family="drape", n=16, n_hi=0, cloths=1, scene=0, steps=1, solver=0, every=1,
                 graphs=False, layout="node_major", tol=1e-12, gpu_factor=False, slots=4, pack=8)


def _case(name=None, **kw):
    case = dict(_DEFAULTS, **kw)
    if name is not None:
        case["name"] = name
    return case


def listed():
    return [
        # one step of a small pinned cloth: an interactive or control loop that
        # reads the state back after every step
        _case("step_hang16", call="step", family="hang", n=16),
        # the gradient of a short rollout of the same cloth through autograd: one
        # iteration of a trajectory optimisation
        _case("autograd_hang16", call="autograd", family="hang", n=16, steps=8),
        # one evaluation of a parameter fit on a small sliding cloth: new stiffness,
        # 24 steps, the adjoint of a loss on every step's positions
        _case("fit_slide8", call="fit", family="slide", n=8, steps=24),
        # the global solve alone, odd size, explicit inverse rows
        _case("solve_drape61", call="solve", n=61),
        # the draped cloth forward (data generation), replayed as a graph
        _case("rollout_drape61", n=61, steps=10, graphs=True),
        # the same with supernodal substitution, plain launches, an even ragged size
        _case("rollout_drape100_sn", n=100, steps=4, solver=1, scene=3),
        # the draped cloth's gradient with checkpoints (recomputed forward steps)
        _case("grad_drape61", call="grad", n=61, steps=4, every=2),
        # the large cloth on capsules, forward, component-major arrays
        _case("rollout_capsules200", family="capsules", n=200, steps=3, solver=1, layout="component_major"),
        # the large cloth's gradient
        _case("grad_capsules200", call="grad", family="capsules", n=200, steps=2, solver=1),
        # many cloths of ragged sizes in one context, forward: dataset generation
        _case("rollout_batch96", n=16, n_hi=64, cloths=96, steps=6, solver=1, graphs=True),
        # many cloths, forward and adjoint: batched training or fitting
        _case("grad_batch96", call="grad", n=16, n_hi=64, cloths=96, steps=2, solver=1, graphs=True),
        # a round of independent requests of different sizes and lengths
        _case("serve12", call="serve", n=18, n_hi=48, cloths=12, steps=3, solver=1, gpu_factor=True,
              tol=1e-10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    call = rng.choice(["step", "solve", "rollout", "rollout", "grad", "grad", "autograd", "batch", "batch", "fit",
                       "serve"])
    scene = rng.randrange(1, 100000)
    solver = rng.randrange(2)
    if call == "fit":
        return _case(call="fit", family="slide", n=rng.randint(5, 16), steps=rng.randint(8, 24), scene=scene)
    if call == "serve":
        return _case(call="serve", n=18, n_hi=rng.randint(24, 48), cloths=rng.randint(3, 12), steps=rng.randint(1, 3),
                     solver=1, gpu_factor=True, tol=1e-10, scene=scene, slots=rng.randint(1, 4), pack=rng.choice([1, 4, 8]))
    if call == "batch":
        lo = rng.randint(8, 24)
        return _case(call=rng.choice(["rollout", "grad"]), n=lo, n_hi=lo + rng.randint(4, 40),
                     cloths=_log_int(rng, 3, 64), steps=rng.randint(1, 2), solver=solver, every=rng.choice([1, 1, 2]),
                     graphs=rng.random() < 0.5, scene=scene)
    family = rng.choice(["hang", "drape", "drape", "capsules"])
    n = _log_int(rng, 8, 120)
    if n > 72:
        solver = 1
    return _case(call=call, family=family, n=n, steps=1 if call in ("step", "solve") else rng.randint(1, 4 if call == "rollout" else 3),
                 solver=solver, every=rng.choice([1, 1, 2, 3]), graphs=rng.random() < 0.5, scene=scene,
                 layout=rng.choice(["node_major", "component_major"]) if call != "autograd" else "node_major")


# ---------------------------------------------------------------------- scenes

def _grid(n, side, height, x0, z0):
    """Rest positions of a flat n x n grid (node (i, j) at j n + i) and its triangles,
    every quad split along its (i, j)-(i + 1, j + 1) diagonal."""
    a = side / (n - 1)
    j, i = np.divmod(np.arange(n * n), n)
    pos = np.stack([x0 + a * i, np.full(n * n, height), z0 + a * j], axis=1)
    jq, iq = np.divmod(np.arange((n - 1) ** 2), n - 1)
    v = jq * n + iq
    tris = np.stack([np.stack([v, v + 1, v + n + 1], axis=1), np.stack([v, v + n + 1, v + n], axis=1)], axis=1)
    return pos, np.ascontiguousarray(tris.reshape(-1, 3).astype(np.int32))


def _log_uniform(rng, lo, hi):
    return float(math.exp(rng.uniform(math.log(lo), math.log(hi))))


# The largest stretch stiffness of a call's cloths: the stiffer decade (up to 1e4) goes
# through the forward calls; there the adjoint's systems are so ill-conditioned that a
# gradient says little about the code that computed it.
_STIFFEST = dict(step=1e4, solve=1e4, rollout=1e4, serve=3e2)


def _cloths(case):
    """The cloths of a case: dicts of rest, tris, pins, normal (of the incline, or up), params."""
    out = []
    for c in range(case["cloths"]):
        rng = np.random.default_rng([case["scene"], c, 0xC107])
        n = case["n"] if not case["n_hi"] else int(rng.integers(case["n"], case["n_hi"] + 1))
        p = dict(k_stretch=1e3, k_bend=1e-3, mu=0.3, density=DENSITY, h=1.0 / 120.0, gravity=GRAVITY,
                 contact_margin=MARGIN, n_pd_iters=PD_ITERS, adj_tol=case["tol"], global_solver=case["solver"],
                 checkpoint_every=case["every"], factor_on_gpu=int(case["gpu_factor"]))
        ground = dict(kind="plane", normal=(0.0, 1.0, 0.0), offset=0.0)
        pins = np.zeros(0, np.int32)
        up = np.array([0.0, 1.0, 0.0])
        if case["family"] == "slide":
            th = math.atan(0.5) + 0.15
            rest, tris = _grid(n, 0.4, 0.0, 0.0, 0.0)
            cs, sn = math.cos(th), math.sin(th)
            rot = np.array([[cs, -sn, 0.0], [sn, cs, 0.0], [0.0, 0.0, 1.0]])
            rest = rest @ rot.T
            up = rot @ up
            p.update(k_stretch=_log_uniform(rng, 500.0, 2000.0), mu=float(rng.uniform(0.3, 0.5)), h=0.01,
                     obstacles=[dict(kind="plane", normal=tuple(up), offset=0.0)])
        elif case["family"] == "capsules":
            obst, top = [ground], 0.0
            for _ in range(8):
                mid = np.array([rng.uniform(-0.4, 0.4), rng.uniform(0.1, 0.35), rng.uniform(0.1, 0.9)])
                ang, half, r = rng.uniform(0, math.pi), rng.uniform(0.05, 0.2), float(rng.uniform(0.02, 0.1))
                d = np.array([math.cos(ang), 0.0, math.sin(ang)]) * half
                obst.append(dict(kind="capsule", a=tuple(mid - d), b=tuple(mid + d), radius=r))
                top = max(top, mid[1] + r)
            rest, tris = _grid(n, 1.0, top + 0.002, -0.5, 0.0)
            p.update(mu=0.4, h=1.0 / 240.0, obstacles=obst)
        else:
            r, cy, cz = 0.3, 0.35, 0.5
            if case["cloths"] > 1:
                r = float(rng.uniform(0.2, 0.5))
                cy = r + float(rng.uniform(0.0, 0.2))
            if case["family"] == "hang":
                cz = 0.55
                pins = np.array([0, n - 1], dtype=np.int32)
            else:
                p.update(k_stretch=_log_uniform(rng, 1e2, _STIFFEST.get(case["call"], 1e3)), k_bend=_log_uniform(rng, 1e-4, 1e-2),
                         mu=float(rng.uniform(0.1, 0.6)))
            rest, tris = _grid(n, 1.0, cy + r + 0.002, -0.5, 0.0)
            p.update(obstacles=[ground, dict(kind="sphere", center=(0.0, cy, cz), radius=r)])
        out.append(dict(rest=rest, tris=tris, pins=pins, up=up, params=p))
    return out


def _waves(rng, rest, normal, amplitude):
    """A smooth random displacement or velocity field over the cloth: six plane waves
    of at least a third of a metre along its normal, with a hundredth of it in the plane."""
    out = np.zeros_like(rest)
    for _ in range(6):
        k = rng.uniform(-3.0, 3.0, 3)
        d = rng.standard_normal() * normal + 0.01 * rng.standard_normal(3)
        out += np.sin(2.0 * math.pi * (rest @ k) + rng.uniform(0, 2 * math.pi))[:, None] * d
    return amplitude / 6.0 * out


def _motion(case, cloth, rng):
    """Initial positions and velocities of one cloth."""
    rest, up = cloth["rest"], cloth["up"]
    out = rest - rest.mean(axis=0)        # from the cloth's centre, in its plane
    if case["family"] == "slide":
        x0 = rest + 0.0
        v0 = rng.uniform(0.3, 0.6) * out + 0.02 * rng.standard_normal(3)
        v0 -= np.outer(v0 @ up, up)
    else:
        x0 = rest + 0.003 * out + _waves(rng, rest, up, 0.003)
        v0 = rng.uniform(0.8, 1.2) * (out - up) + _waves(rng, rest, up, 0.2)
    x0[cloth["pins"]] = rest[cloth["pins"]]
    v0[cloth["pins"]] = 0.0
    return x0, v0


def _inputs(case, seed):
    """(cloths, arrays): per-node arrays over all cloths, node-major."""
    rng = np.random.default_rng([seed, 0x1D])
    cloths = _cloths(case)
    xs, vs = zip(*[_motion(case, c, rng) for c in cloths])
    x0, v0 = np.concatenate(xs), np.concatenate(vs)
    a = dict(x0=x0, v0=v0, gx=rng.standard_normal(x0.shape), gv=0.01 * rng.standard_normal(x0.shape))
    if case["call"] == "fit":
        a["gtraj"] = rng.standard_normal((case["steps"] + 1,) + x0.shape)
    return cloths, a


# ---------------------------------------------------------------------- calls

class _State:
    pass


def _request_steps(case, k):
    return max(1, case["steps"] - k % 3)


def prepare(case, seed):
    cloths, a = _inputs(case, seed)
    s = _State()
    s.case = case
    if case["call"] == "serve":
        s.server = dc.Server(n_slots=case["slots"], n_prep_threads=4, max_batch=case["pack"],
                             hbm_budget_bytes=20 << 30)
        s.requests, lo = [], 0
        for k, c in enumerate(cloths):
            hi = lo + len(c["rest"])
            s.requests.append((c["rest"], c["tris"], c["pins"], a["x0"][lo:hi], a["v0"][lo:hi], a["gx"][lo:hi],
                               _request_steps(case, k), c["params"]))
            lo = hi
        return s
    s.stream = torch.cuda.Stream() if case["graphs"] else torch.cuda.current_stream()
    with torch.cuda.stream(s.stream):
        if case["cloths"] > 1:
            s.obj = dc.ClothBatch([(c["rest"], c["tris"], c["pins"]) for c in cloths])
            s.obj.set_params([c["params"] for c in cloths])
        else:
            s.obj = dc.Cloth(cloths[0]["rest"], cloths[0]["tris"], cloths[0]["pins"])
            s.obj.set_params(**cloths[0]["params"])
            s.params = cloths[0]["params"]
        if case["graphs"]:
            s.obj.set_graphs(True)
        if case["layout"] != "node_major":
            s.obj.set_layout(case["layout"])
            a = {k: np.ascontiguousarray(np.swapaxes(v, -1, -2)) for k, v in a.items()}
        for k, v in a.items():
            setattr(s, k, torch.tensor(v, device="cuda"))
        if case["call"] == "autograd":
            s.obj.allow_nonconverged = True
            p = cloths[0]["params"]
            s.theta = torch.tensor([p["k_stretch"], p["k_bend"], p["mu"]], dtype=torch.float64)
    s.stream.synchronize()
    return s


def run(s):
    case = s.case
    call = case["call"]
    if call == "serve":
        tickets = [s.server.submit(*req) for req in s.requests]
        done = [s.server.wait(t) for t in tickets]
        # (a request whose adjoint stopped above its tolerance brings no arrays back)
        return {k: [r[k] for r in done if r["status"] == "DC_OK"] for k in ("x_final", "v_final", "dL_dx0", "dL_dv0", "dL_dparams")}
    with torch.cuda.stream(s.stream):
        if call == "step":
            return s.obj.step(s.x0, s.v0)
        if call == "solve":
            return s.obj.global_solve(s.gx)
        if call == "rollout":
            return s.obj.rollout(s.x0, s.v0, case["steps"])
        if call == "grad":
            x, v = s.obj.rollout(s.x0, s.v0, case["steps"])
            return (x, v) + s.obj.backward(s.gx, s.gv, allow_nonconverged=True)
        if call == "fit":
            s.obj.set_params(**s.params)
            x, v, traj = s.obj.rollout(s.x0, s.v0, case["steps"], traj=True)
            return (x, v, traj) + s.obj.backward(s.gx, s.gv, s.gtraj, allow_nonconverged=True)
        x0 = s.x0.detach().requires_grad_(True)
        v0 = s.v0.detach().requires_grad_(True)
        theta = s.theta.detach().requires_grad_(True)
        x, v = dc.rollout_fn(s.obj, x0, v0, theta, case["steps"])
        ((s.gx * x).sum() + (s.gv * v).sum()).backward()
        return x.detach(), v.detach(), x0.grad, v0.grad, theta.grad


# ---------------------------------------------------------------------- work

def work(case):
    """Bytes: the call's node arrays, the mesh (56 bytes a triangle) and the Cholesky
    factor of P, about 6 m log2 m values for these grids, each once a call.  Flops:
    per PD iteration 150 a triangle, 100 a node and 12 a factor entry (two
    substitutions on three columns); per adjoint step the factorisation of the
    adjoint matrix, 27 times a scalar factorisation of 100 m^1.5 flops, and five
    applications of 36 flops a factor entry."""
    call = case["call"]
    total = dict(bytes=0.0, flops=0.0)
    for k, c in enumerate(_cloths(case)):
        m, t = len(c["rest"]), len(c["tris"])
        nnz = 6.0 * m * math.log2(m)
        steps = _request_steps(case, k) if call == "serve" else case["steps"]
        arrays = {"solve": 2, "step": 4, "rollout": 4}.get(call, 8) + (2 * (steps + 1) if call == "fit" else 0)
        total["bytes"] += 24.0 * m * arrays + (56.0 * t if call != "solve" else 0.0) + 8.0 * nnz
        if call == "solve":
            total["flops"] += 12.0 * nnz
            continue
        total["flops"] += steps * (PD_ITERS * (150.0 * t + 100.0 * m + 12.0 * nnz) + 12.0 * nnz)
        if call not in ("step", "rollout"):
            total["flops"] += steps * (27.0 * 100.0 * m ** 1.5 + 5.0 * 36.0 * nnz)
    return total


# ---------------------------------------------------------------------- the same in plain torch, 64 bits, dense matrices

def _phi(ob, x):
    """Signed distance, its gradient and the gradient's Jacobian at points x (m, 3)."""
    eye = torch.eye(3, dtype=x.dtype, device=x.device)
    if ob["kind"] == "plane":
        n = torch.tensor(ob["normal"], dtype=x.dtype, device=x.device)
        n = n / n.norm()
        return x @ n - ob["offset"], n.expand_as(x), torch.zeros(len(x), 3, 3, dtype=x.dtype, device=x.device)
    if ob["kind"] == "sphere":
        d = x - torch.tensor(ob["center"], dtype=x.dtype, device=x.device)
        ee = torch.zeros(len(x), 3, 3, dtype=x.dtype, device=x.device)
    else:
        a = torch.tensor(ob["a"], dtype=x.dtype, device=x.device)
        ab = torch.tensor(ob["b"], dtype=x.dtype, device=x.device) - a
        t = (x - a) @ ab / (ab @ ab)
        d = x - (a + t.clamp(0.0, 1.0)[:, None] * ab)
        ee = torch.outer(ab, ab) / (ab @ ab) * ((t > 0) & (t < 1)).to(x.dtype)[:, None, None]
    r = d.norm(dim=1)
    n = d / r[:, None]
    return r - ob["radius"], n, (eye - n[:, :, None] * n[:, None, :] - ee) / r[:, None, None]


class _Dense:
    """One cloth: rest operators, P^-1 and the step, dense, float64."""

    def __init__(self, cloth):
        p = cloth["params"]
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        f = dict(dtype=torch.float64, device=dev)
        self.f, self.h, self.mu, self.obst = f, p["h"], p["mu"], p["obstacles"]
        X = torch.tensor(cloth["rest"], **f)
        tri = torch.tensor(cloth["tris"].astype(np.int64), device=dev)
        m = self.m = len(X)
        self.tri = tri
        free = torch.ones(m, dtype=torch.bool, device=dev)
        free[torch.tensor(cloth["pins"].astype(np.int64), device=dev)] = False
        self.free = free.nonzero()[:, 0]
        self.g = torch.tensor(p["gravity"], **f)
        e1, e2 = X[tri[:, 1]] - X[tri[:, 0]], X[tri[:, 2]] - X[tri[:, 0]]
        cr = torch.linalg.cross(e1, e2)
        self.area = 0.5 * cr.norm(dim=1)
        u = e1 / e1.norm(dim=1, keepdim=True)
        w = torch.linalg.cross(cr / cr.norm(dim=1, keepdim=True), u)
        Dm = torch.stack([torch.stack([(e1 * u).sum(1), (e2 * u).sum(1)], 1),
                          torch.stack([(e1 * w).sum(1), (e2 * w).sum(1)], 1)], 1)
        E = torch.tensor([[-1.0, -1.0], [1.0, 0.0], [0.0, 1.0]], **f)
        self.G = E @ torch.linalg.inv(Dm)                                  # (T, 3, 2)
        Wc = torch.zeros(m * m, **f)
        self.abar = torch.zeros(m, **f)
        for k in range(3):
            o, i, j = tri[:, k], tri[:, (k + 1) % 3], tri[:, (k + 2) % 3]
            a, b = X[i] - X[o], X[j] - X[o]
            cot = 0.5 * (a * b).sum(1) / torch.linalg.cross(a, b).norm(dim=1)
            Wc.index_add_(0, i * m + j, cot)
            Wc.index_add_(0, j * m + i, cot)
            self.abar.index_add_(0, o, self.area / 3.0)
        Wc = Wc.view(m, m)
        self.L = (Wc - torch.diag(Wc.sum(1))) / self.abar[:, None]
        self.mass = p["density"] * self.abar
        self.wt, self.wb = p["k_stretch"] * self.area, p["k_bend"] * self.abar
        self.q_rest = self.L @ X
        self.s = self.q_rest.norm(dim=1)
        scale = self.L.abs().sum(1) * (X - X.mean(0)).norm(dim=1).max()
        self.s[self.s <= 1e-9 * scale] = 0.0
        S = torch.zeros(m * m, **f)
        GG = (self.G @ self.G.transpose(1, 2)) * self.wt[:, None, None]
        S.index_add_(0, (tri[:, :, None] * m + tri[:, None, :]).reshape(-1), GG.reshape(-1))
        P = torch.diag(self.mass) + self.h ** 2 * (S.view(m, m) + self.L.T @ (self.wb[:, None] * self.L))
        self.Pinv = torch.cholesky_inverse(torch.linalg.cholesky(P[self.free][:, self.free]))

    def solve(self, rhs):
        out = torch.zeros_like(rhs)
        out[self.free] = self.Pinv @ rhs[self.free]
        return out

    def grad_F(self, x):
        return torch.einsum("tac,tak->tck", x[self.tri], self.G)

    def polar(self, F):
        C = F.transpose(1, 2) @ F
        sd = torch.linalg.cross(F[:, :, 0], F[:, :, 1]).norm(dim=1)
        t = (C[:, 0, 0] + C[:, 1, 1] + 2.0 * sd).sqrt()
        S = (C + sd[:, None, None] * torch.eye(2, **self.f)) / t[:, None, None]
        Si = torch.linalg.inv(S)
        return F @ Si, Si, t

    def bend(self, q):
        nq = q.norm(dim=1, keepdim=True)
        p = torch.where(nq > 1e-14 * self.s[:, None], self.s[:, None] * q / nq.clamp_min(1e-300), self.q_rest)
        return torch.where(self.s[:, None] > 0, p, torch.zeros_like(q))

    def step(self, x, v):
        h, m = self.h, self.m
        v = v.clone()
        fixed = torch.ones(m, dtype=torch.bool, device=x.device)
        fixed[self.free] = False
        v[fixed] = 0.0
        phis = torch.stack([_phi(ob, x + h * v)[0] for ob in self.obst])
        best, ob = phis.min(dim=0)
        nodes = ((best <= MARGIN) & ~fixed).nonzero()[:, 0]
        ob = ob[nodes]
        at = [_phi(o, x[nodes]) for o in self.obst]
        pick = torch.arange(len(nodes), device=x.device)
        phi0, nrm, Dn = (torch.stack([a[k] for a in at])[ob, pick] for k in range(3))
        beta = phi0 / h
        ind = torch.zeros(m, 1, **self.f)
        ind[nodes] = 1.0
        c = (h * self.solve(ind))[nodes]
        f = torch.zeros(len(nodes), 3, **self.f)
        kind = torch.zeros(len(nodes), dtype=torch.int64, device=x.device)
        My = self.mass[:, None] * (v + h * self.g)
        Fn, qn = self.grad_F(x), self.L @ x
        for _ in range(PD_ITERS):
            xk = x + h * v
            R, _, _ = self.polar(self.grad_F(xk))
            D = (R - Fn) * self.wt[:, None, None]
            rhs = My.clone()
            rhs.index_add_(0, self.tri.reshape(-1),
                           h * torch.einsum("tck,tak->tac", D, self.G).reshape(-1, 3))
            rhs += h * (self.L.T @ (self.wb[:, None] * (self.bend(self.L @ xk) - qn)))
            rhs[nodes] += h * f
            v = self.solve(rhs)
            vt = v[nodes] - c * f
            vn = (nrm * vt).sum(1)
            uN = vn + beta
            uT = vt - vn[:, None] * nrm
            nt = uT.norm(dim=1)
            kind = torch.where(uN >= 0, 0, torch.where(nt <= -self.mu * uN, 1, 2))
            fN = -uN[:, None] / c
            slip = fN * nrm - self.mu * fN / nt.clamp_min(1e-300)[:, None] * uT
            stick = (-beta[:, None] * nrm - vt) / c
            f = torch.where(kind[:, None] == 1, stick, torch.where(kind[:, None] == 2, slip, torch.zeros_like(slip)))
            v[nodes] = torch.where(kind[:, None] == 1, -beta[:, None] * nrm, vt + c * f)
        return x + h * v, v, dict(nodes=nodes, nrm=nrm, Dn=Dn, beta=beta, f=f, kind=kind)

    def adjoint(self, x, x1, v1, rec, gx, gv):
        """dL at step n + 1 -> dL at step n, and dL / d(k_stretch, k_bend, mu) of the step."""
        h, m, mu = self.h, self.m, self.mu
        eye3, eye2 = torch.eye(3, **self.f), torch.eye(2, **self.f)
        F = self.grad_F(x1)
        R, Si, t = self.polar(F)
        T = len(F)
        # dR for each unit dF[c, k], as (T, 3, 2, 3, 2): [.., c', k', c, k]
        RtE = torch.einsum("tcl,kn->tlnck", R, eye2)                         # R^T dF, entry (l, n)
        om = (RtE[:, 1, 0] - RtE[:, 0, 1]) / t[:, None, None]
        J = torch.tensor([[0.0, -1.0], [1.0, 0.0]], **self.f)
        dR = torch.einsum("tcl,ln,tdk->tcndk", R, J, om)
        Pn = eye3 - R @ R.transpose(1, 2)
        dR = dR + torch.einsum("tcd,tkn->tcndk", Pn, Si)
        K = torch.einsum("cd,kn->cndk", eye3, eye2)[None] - dR               # d(F - R)
        blk = torch.einsum("tan,tcndk,tbk->tacbd", self.G, K, self.G) * self.wt[:, None, None, None, None]
        dof = (3 * self.tri[:, :, None] + torch.arange(3, device=x.device)).reshape(T, 9)
        W = torch.zeros(9 * m * m, **self.f)
        W.index_add_(0, (dof[:, :, None] * (3 * m) + dof[:, None, :]).reshape(-1), blk.reshape(-1))
        W = W.view(m, 3, m, 3)
        q = self.L @ x1
        nq = q.norm(dim=1).clamp_min(1e-300)
        kap = torch.where((self.s > 0) & (nq > 1e-14 * self.s), self.s / nq, torch.zeros_like(nq))
        qh = q / nq[:, None]
        for a in range(3):
            for b in range(3):
                d = self.wb * ((1.0 - kap) * float(a == b) + kap * qh[:, a] * qh[:, b])
                if bool((d != 0).any()):
                    W[:, a, :, b] += self.L.T @ (d[:, None] * self.L)
        W = W.reshape(3 * m, 3 * m)
        nodes, nrm, kind = rec["nodes"], rec["nrm"], rec["kind"]
        st, sl = nodes[kind == 1], nodes[kind == 2]
        n2, f2 = nrm[kind == 2], rec["f"][kind == 2]
        v2 = v1[sl]
        vn = (n2 * v2).sum(1, keepdim=True)
        uT = v2 - vn * n2
        nt = uT.norm(dim=1, keepdim=True)
        th = uT / nt
        bh = torch.linalg.cross(n2, th)
        fN = (f2 * n2).sum(1)
        H = h * h * W
        H.diagonal().add_(self.mass.repeat_interleave(3))
        slip_blk = (h * mu * fN / nt[:, 0])[:, None, None] * bh[:, :, None] * bh[:, None, :]
        H.view(m, 3, m, 3)[sl, :, sl, :] += slip_blk
        keep = torch.zeros(m, dtype=torch.bool, device=x.device)
        keep[self.free] = True
        keep[st] = False
        keep[sl] = False
        fd = (3 * keep.nonzero() + torch.arange(3, device=x.device)).reshape(-1)
        Q = torch.stack([bh, th + mu * n2], 2)                                # (s, 3, 2), null space of n - mu t
        Rm = torch.stack([th, bh], 2)                                        # null space of n
        sd = (3 * sl[:, None] + torch.arange(3, device=x.device)).reshape(-1)
        ns = len(sl)
        cols = torch.cat([H[:, fd], torch.einsum("nsc,scp->nsp", H[:, sd].view(3 * m, ns, 3), Q).reshape(3 * m, 2 * ns)], 1)
        A = torch.cat([cols[fd], torch.einsum("scn,scp->spn", cols[sd].view(ns, 3, cols.shape[1]), Rm)
                       .reshape(2 * ns, cols.shape[1])])
        g = gv + h * gx
        gf = g.reshape(-1)
        rhs = torch.cat([gf[fd], torch.einsum("sc,scp->sp", g[sl], Rm).reshape(-1)])
        y = torch.linalg.solve(A, rhs)
        z = torch.zeros(3 * m, **self.f)
        z[fd] = y[:len(fd)]
        z[sd] = torch.einsum("scp,sp->sc", Q, y[len(fd):].view(ns, 2)).reshape(-1)
        res = (gf - H @ z).view(m, 3)
        ox = gx - h * (W @ z).view(m, 3)
        z = z.view(m, 3)
        ov = self.mass[:, None] * z
        n1, D1, b1 = nrm[kind == 1], rec["Dn"][kind == 1], rec["beta"][kind == 1]
        r1 = res[st]
        ox[st] -= b1[:, None] * torch.einsum("sba,sb->sa", D1, r1) + n1 * (n1 * r1).sum(1, keepdim=True) / h
        D2 = rec["Dn"][kind == 2]
        psi = (n2 * res[sl]).sum(1, keepdim=True)
        dPv = -(vn[:, :, None] * eye3 + n2[:, :, None] * v2[:, None, :]) @ D2
        Dt = (eye3 - th[:, :, None] * th[:, None, :]) @ dPv / nt[:, :, None]
        ox[sl] += h * fN[:, None] * torch.einsum("sba,sb->sa", D2 - mu * Dt, z[sl])
        ox[sl] -= (torch.einsum("sba,sb->sa", D2, v2) + n2 / h) * psi
        dks = -h * (self.area * (self.grad_F(z) * (F - R)).sum((1, 2))).sum()
        dkb = -h * (self.abar * ((self.L @ z) * (q - self.bend(q))).sum(1)).sum()
        dmu = -h * (fN * (th * z[sl]).sum(1)).sum()
        return ox, ov, torch.stack([dks, dkb, dmu])


def exact(case, seed):
    cloths, a = _inputs(case, seed)
    call = case["call"]
    sizes = [len(c["rest"]) for c in cloths]
    steps = [_request_steps(case, k) if call == "serve" else case["steps"] for k in range(len(cloths))]
    if max(sizes) > 12000 or sum(float(m) ** 2 * 8 * (25 * s + 20) for m, s in zip(sizes, steps)) > 4e13:
        return None
    grads = call in ("grad", "autograd", "fit", "serve") and max(sizes) <= 4100 and \
        sum((3.0 * m) ** 3 * s for m, s in zip(sizes, steps)) < 8e12
    out = dict(x=[], v=[], dx=[], dv=[], dth=[], traj=[], sol=[])
    lo = 0
    for c, m, n_steps in zip(cloths, sizes, steps):
        hi = lo + m
        D = _Dense(c)
        x, v, gx, gv = (torch.tensor(a[k][lo:hi], **D.f) for k in ("x0", "v0", "gx", "gv"))
        if call == "solve":
            out["sol"].append(D.solve(gx))
            lo = hi
            continue
        if call == "serve":
            gv = torch.zeros_like(gv)
        hist = []
        traj = [x]
        for _ in range(n_steps):
            x1, v1, rec = D.step(x, v)
            hist.append((x, x1, v1, rec))
            x, v = x1, v1
            traj.append(x)
        out["x"].append(x)
        out["v"].append(v)
        out["traj"].append(torch.stack(traj))
        if grads:
            gt = torch.tensor(a["gtraj"][:, lo:hi], **D.f) if call == "fit" else None
            gv[[i for i in range(m) if i in set(c["pins"].tolist())]] = 0.0
            dth = torch.zeros(3, **D.f)
            for n in range(n_steps - 1, -1, -1):
                if gt is not None:
                    gx = gx + gt[n + 1]
                gx, gv, d = D.adjoint(*hist[n], gx, gv)
                dth = dth + d
            if gt is not None:
                gx = gx + gt[0]
            out["dx"].append(gx)
            out["dv"].append(gv)
            out["dth"].append(dth)
        lo = hi

    def whole(k):
        if not out[k]:
            return None
        t = torch.cat(out[k]) if k != "traj" else torch.cat(out[k], 1)
        return t.transpose(-1, -2).contiguous() if case["layout"] != "node_major" else t

    if call == "solve":
        return whole("sol")
    if call in ("step", "rollout"):
        return whole("x"), whole("v")
    if call == "serve":
        none = [None] * len(cloths)
        return dict(x_final=out["x"], v_final=out["v"], dL_dx0=out["dx"] or none, dL_dv0=out["dv"] or none,
                    dL_dparams=out["dth"] or none)
    dth = None if not out["dth"] else out["dth"][0] if case["cloths"] == 1 else torch.stack(out["dth"])
    lead = (whole("x"), whole("v")) + ((whole("traj"),) if call == "fit" else ())
    return lead + (whole("dx"), whole("dv"), dth)
