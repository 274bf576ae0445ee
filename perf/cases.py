"""The work a user of this library has it do, as timed cases.

Each case is one call (or one burst of calls) through the public Python entry
points -- ``ucn.Solver`` and ``serving.Server`` -- on seeded problems of the
shapes in ``workloads``: whole SCP solves of one problem, of batches and of
scenario groups, in both precisions and all four models; the stand-alone
linearisation and ADMM calls; and a burst of served requests.

Whole solves run a fixed number of SCP iterations (``stop = 0``), as a planner
with a fixed time budget does: the work of a case then depends on its sizes
alone.  Their status uses the success gate of such a budget (a defect of 1e-2),
the descent batches, which converge, the library's own 1e-5.

FP32_REFINE computes in single precision, so a program that asks for it takes
the trajectories in single precision too; FP64 results stay doubles.
"""
import math

import numpy as np
import torch

import workloads as W
from paper_2603_10711_gb300 import serving, ucn

F64, F32 = ucn.UCN_PREC_FP64, ucn.UCN_PREC_FP32_REFINE
PREC = {"fp64": F64, "fp32": F32}
NX = {"quad": 12, "mars": 7, "quat": 13, "mars6": 14}
NU = {"quad": 4, "mars": 3, "quat": 4, "mars6": 3}


def listed():
    return [
        # one plan of the quadrotor obstacle task in plain FP64: the smallest call, one instance on the device
        dict(name="quad_one_fp64", kind="scp", model="quad", prec="fp64", B=1, N=50, N_max=50, obs=5, scp=15, admm=200, rho=1.0),
        # the same vehicle replanned on the fast path: latency of a single FP32 solve
        dict(name="quad_one_fp32", kind="scp", model="quad", prec="fp32", B=1, N=50, N_max=50, obs=5, scp=10, admm=200, rho=10.0),
        # batched planning with uneven horizons and 10 to 30 obstacles (an odd batch size)
        dict(name="quad_uneven_fp32", kind="scp", model="quad", prec="fp32", B=1023, N=40, N_max=120, obs=30, scp=10, admm=200, rho=10.0),
        # the same in plain FP64, for users who need its accuracy; about one instance per SM
        dict(name="quad_uneven_fp64", kind="scp", model="quad", prec="fp64", B=149, N=40, N_max=120, obs=30, scp=10, admm=200, rho=10.0),
        # scenario robust MPC: 64 problems of 16 scenarios that share their first control
        dict(name="scenario_mpc_fp32", kind="scp", model="quad", prec="fp32", B=1024, N=40, N_max=40, obs=8, scp=8, admm=200, rho=10.0, group=16),
        # Monte-Carlo batch of Mars powered descents: the headline workload
        dict(name="mars_batch_fp32", kind="scp", model="mars", prec="fp32", B=1024, N=100, N_max=100, obs=0, scp=60, admm=40, rho=1.0),
        # a quarter of it in plain FP64
        dict(name="mars_batch_fp64", kind="scp", model="mars", prec="fp64", B=256, N=100, N_max=100, obs=0, scp=60, admm=40, rho=1.0),
        # Monte-Carlo batch of the 6-DOF lander
        dict(name="mars6_batch_fp32", kind="scp", model="mars6", prec="fp32", B=1000, N=30, N_max=30, obs=0, scp=40, admm=100, rho=1.0),
        # the quaternion quadrotor's parameter study
        dict(name="quat_study_fp32", kind="scp", model="quat", prec="fp32", B=256, N=50, N_max=50, obs=3, scp=20, admm=100, rho=1.0),
        # a user's own SCP loop: linearise every node, then one ADMM call on the result
        dict(name="linearize_quad_fp64", kind="linearize", model="quad", prec="fp64", B=2048, N=40, N_max=120, obs=10),
        dict(name="admm_quad_fp32", kind="admm", model="quad", prec="fp32", B=511, N=40, N_max=120, obs=10, admm=100, rho=10.0),
        # a burst of 70% quadrotor and 30% descent requests at a server, sizes mixed
        dict(name="serve_burst_fp32", kind="serve", model="quad", prec="fp32", B=64, N=30, N_max=120, obs=30, scp=10, admm=200, rho=10.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["scp"] * 7 + ["linearize", "admm", "serve"])
    model = rng.choice(["quad", "quad", "quad", "mars", "mars", "mars6", "quat"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    c = dict(kind=kind, model=model, prec=prec)
    if kind == "serve":
        n = rng.randint(31, 72)
        c.update(model="quad", prec="fp32", B=log_int(2, 96), N=n - 20, N_max=n + 40, obs=rng.randint(5, 30), scp=8, admm=100, rho=10.0)
    elif kind == "linearize":
        lo = rng.randint(5, 60)
        c.update(B=log_int(1, 1500), N=lo, N_max=lo + (rng.randint(0, 60) if model == "quad" else 0), obs=rng.randint(1, 12))
    elif kind == "admm":
        lo = rng.randint(5, 60)
        c.update(B=log_int(1, 400 if prec == "fp32" else 48), N=lo, N_max=lo + (rng.randint(0, 60) if model == "quad" else 0),
                 obs=rng.randint(0, 12) if model != "quat" else 3, admm=rng.randint(20, 120), rho=10.0 if model == "quad" else 1.0)
    elif model == "quad" and rng.random() < 0.3:
        k = rng.choice([3, 8, 16, 32])
        p = log_int(1, (640 if prec == "fp32" else 160) // k)
        n = rng.randint(17, 47)
        c.update(B=p * k, N=n, N_max=n, obs=rng.randint(1, 10), scp=rng.randint(3, 8), admm=rng.choice([100, 200]), rho=10.0, group=k)
    elif model == "quad":
        lo = rng.randint(15, 60)
        c.update(B=log_int(1, 512 if prec == "fp32" else 96), N=lo, N_max=lo + rng.randint(0, 60), obs=rng.randint(1, 30),
                 scp=rng.randint(3, 10), admm=rng.choice([100, 200]), rho=10.0)
    elif model == "mars":
        n = rng.randint(31, 150)
        c.update(B=log_int(1, (1024 if prec == "fp32" else 192) * 100 // max(n, 100)), N=n, N_max=n, obs=0, scp=60, admm=40, rho=1.0)
    elif model == "mars6":
        n = rng.randint(15, 40)
        c.update(B=log_int(1, 1000 if prec == "fp32" else 48), N=n, N_max=n, obs=0, scp=rng.randint(10, 40), admm=100, rho=1.0)
    else:
        n = rng.randint(25, 60)
        c.update(B=log_int(1, 256 if prec == "fp32" else 48), N=n, N_max=n, obs=3, scp=20, admm=100, rho=1.0)
    return c


def _settings(c):
    s = dict(admm_iters=c.get("admm", 1), scp_iters=c.get("scp", 1), stop=0)
    rho = c.get("rho", 1.0)
    s.update(rho_eq=rho, rho_dyn=rho, rho_geo=rho)
    s["defect_tol"] = 1e-5 if c["model"] == "mars" else 1e-2
    return s


def _merge(ps):
    """Several problems as one batch."""
    most = max(p.max_obs for p in ps)
    f = {}
    for name, v in vars(ps[0]).items():
        if name in ("model", "nx", "nu", "settings"):
            f[name] = v
        elif name in ("obs_c", "obs_r"):
            rows = [getattr(p, name) for p in ps]
            f[name] = np.concatenate([np.pad(r, [(0, 0), (0, most - r.shape[1])] + [(0, 0)] * (r.ndim - 2)) for r in rows])
        else:
            f[name] = np.concatenate([getattr(p, name) for p in ps])
    return W.Problem(**f)


def _problem(c, seed):
    s = _settings(c)
    if c["model"] == "mars":
        return W.mars_batch(c["B"], seed=seed, N=c["N"], settings=s)
    if c["model"] == "mars6":
        return W.mars6_batch(c["B"], seed=seed, N=c["N"], tf=c["N"] / 6.0, settings=s)
    if c["model"] == "quat":
        return W.quat_study(c["B"], seed=seed, N=c["N"], tf=0.12 * c["N"], n_obs=c["obs"], settings=s)
    if c.get("group", 1) > 1:
        return W.scenario_mpc(c["B"] // c["group"], c["group"], seed=seed, N=c["N"], n_obs=c["obs"], settings=s)
    if c["B"] == 1 and c["N"] == c["N_max"]:
        return W.quad_path(1, seed=seed, N=c["N"], n_obs=min(c["obs"], 5), settings=s)
    # horizons mixed over [N, N_max], the same ones for every seed
    span = c["N_max"] - c["N"] + 1
    N = c["N"] + np.arange(c["B"]) * 37 % span
    parts, of = [], []
    for n in np.unique(N):
        idx = np.nonzero(N == n)[0]
        parts.append(W.quad_box(len(idx), seed=seed * 256 + int(n), N_range=(n, n), obs_range=(min(c["obs"], 10), c["obs"]), settings=s))
        of.append(idx)
    return _merge(parts).subset(np.argsort(np.concatenate(of)))


def _nominal(p, seed):
    """A nominal off the straight-line guess, as in the middle of an SCP solve."""
    r = np.random.default_rng(seed)
    x = p.xguess + 0.02 * r.standard_normal(p.xguess.shape)
    u = p.uguess + 0.02 * r.standard_normal(p.uguess.shape)
    x[p.xoff] = p.xinit
    return x, u


BUCKETS = {1: (40, 72, 120), 2: (100, 200)}   # horizons of the servers, one per model and bucket


def _requests(c, seed):
    out = []
    for k in range(c["B"]):
        v = W.uniform(4, 90, np.arange(3 * k, 3 * k + 3))   # the same mix for every seed
        if v[0] < 0.7:
            n = c["N"] + int(v[1] * (c["N_max"] - c["N"] + 1))
            o = min(5, c["obs"]) + int(v[2] * (c["obs"] - min(5, c["obs"]) + 1))
            out.append(W.quad_box(1, seed=seed * 1000 + k, N_range=(n, n), obs_range=(o, o), settings=_settings(c)))
        else:
            s = _settings(dict(model="mars", admm=40, scp=60))
            out.append(W.mars_batch(1, seed=seed * 1000 + k, N=50 + int(v[1] * 101), settings=s))
    return out


def prepare(case, seed):
    c, prec = case, PREC[case["prec"]]
    if c["kind"] == "serve":
        reqs = _requests(c, seed)
        route = serving.horizon_route(BUCKETS)
        count = {}
        for p in reqs:
            count[route(p)] = count.get(route(p), 0) + 1
        first = {route(p): p for p in reversed(reqs)}
        servers = {key: serving.Server(key[0], prec, max_slots=n, max_horizon=key[1], max_obs=c["obs"] if key[0] == 1 else 0,
                                       lanes=4, settings=first[key].settings) for key, n in count.items()}
        return dict(kind="serve", reqs=[(route(p), p) for p in reqs], servers=servers)
    p = _problem(c, seed)
    s = ucn.Solver(p, precision=prec)
    st = dict(kind=c["kind"], solver=s, single=c["prec"] == "fp32")
    if c["kind"] == "scp":
        st.update(x=s.tensor(p.xguess), u=s.tensor(p.uguess))
        return st
    x, u = _nominal(p, seed)
    st.update(x=s.tensor(x), u=s.tensor(u))
    if c["kind"] == "admm":
        lin = ucn.Solver(p, precision=F64)
        st["lin"] = lin.linearize(st["x"], st["u"])
        torch.cuda.synchronize()
        lin.close()
        st.update(radius=s.tensor(np.full(p.batch, 0.7)), iters=c["admm"])
    return st


def _serve(st):
    servers, waiting, tickets, done = st["servers"], list(enumerate(st["reqs"])), {}, {}
    while len(done) < len(st["reqs"]):
        left = []
        for k, (key, p) in waiting:
            rc, ticket = servers[key].submit(p)
            if rc == ucn.UCN_OK:
                tickets[k] = (key, ticket, int(p.N[0]))
            else:
                left.append((k, (key, p)))
        waiting = left
        for srv in servers.values():
            srv.pump()
        for k, (key, ticket, n) in list(tickets.items()):
            rc, res = servers[key].poll(ticket, horizon=n)
            if rc == ucn.UCN_OK:
                done[k] = res
                del tickets[k]
    got = [done[k] for k in range(len(st["reqs"]))]
    return {"x": np.concatenate([r["x"].ravel() for r in got]).astype(np.float32),
            "u": np.concatenate([r["u"].ravel() for r in got]).astype(np.float32),
            "status": np.array([r["stats"]["status"] for r in got], np.int32)}


def run(st):
    if st["kind"] == "serve":
        return _serve(st)
    s = st["solver"]
    out = (lambda t: t.float()) if st["single"] else (lambda t: t)
    if st["kind"] == "scp":
        x, u = s.scp_solve(st["x"], st["u"])
        return {"x": out(x), "u": out(u), "status": s.status}
    if st["kind"] == "linearize":
        A, B, d = s.linearize(st["x"], st["u"])
        return {"A": out(A), "B": out(B), "d": out(d)}
    xh, uh, res, status = s.admm_solve(st["x"], st["u"], *st["lin"], st["radius"], st["iters"])
    return {"x": out(xh), "u": out(uh), "res": out(res), "status": status}


def work(case):
    """Bytes: the call's inputs and outputs.  Flops: the dense per-node products
    of the method -- linearisation (a value and nx + nu tangents of four stages
    of the dynamics), assembly, factorisation and inverse, and per ADMM
    iteration [A B]^T w, H^-1 g, [A B] xi and the projections."""
    c = case
    nx, nu = NX[c["model"]], NU[c["model"]]
    n = nx + nu
    nodes = c["B"] * (c["N"] + c["N_max"]) / 2.0
    jac = 4 * 60.0 * (n + 1)
    iteration = 4.0 * nx * n + 2.0 * n * n + 12.0 * nx + 6.0 * nu + (10.0 * c["obs"] if c["model"] in ("quad", "quat") else 60.0)
    setup = 2.0 * nx * n * n / 2 + n ** 3
    if c["kind"] == "linearize":
        return {"bytes": nodes * 8 * (n + nx * n + nx), "flops": nodes * (jac + 2.0 * nx * n)}
    if c["kind"] == "admm":
        return {"bytes": nodes * 8 * (2 * n + nx * n + nx), "flops": nodes * (setup + c["admm"] * iteration)}
    return {"bytes": nodes * 8 * 2 * n, "flops": nodes * c["scp"] * (jac + setup + c["admm"] * iteration)}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch
def _dynamics(model, p):
    """x-dot of a model as a function of (x, u); p [B, 1, 8] its constants."""
    k = [p[..., j] for j in range(8)]

    def quad(x, u):
        m, jx, jy, jz, arm, km, cd, g = k
        vx, vy, vz, ph, th, ps, wx, wy, wz = [x[..., j] for j in range(3, 12)]
        a, b, c, d = [u[..., j] for j in range(4)]
        f = (a + b + c + d) / m
        sph, cph, sth, cth, sps, cps = ph.sin(), ph.cos(), th.sin(), th.cos(), ps.sin(), ps.cos()
        return torch.stack([
            vx, vy, vz,
            f * (cph * sth * cps + sph * sps) - cd / m * vx,
            f * (cph * sth * sps - sph * cps) - cd / m * vy,
            f * cph * cth - g - cd / m * vz,
            wx + (sph * wy + cph * wz) * sth / cth,
            cph * wy - sph * wz,
            (sph * wy + cph * wz) / cth,
            (arm * (b - d) - (jz - jy) * wy * wz) / jx,
            (arm * (c - a) - (jx - jz) * wz * wx) / jy,
            (km * (a - b + c - d) - (jy - jx) * wx * wy) / jz], -1)

    def spin(q, w):   # q' = q (x) (0, w) / 2
        qw, qx, qy, qz = q
        wx, wy, wz = w
        return [(-qx * wx - qy * wy - qz * wz) / 2, (qw * wx + qy * wz - qz * wy) / 2,
                (qw * wy - qx * wz + qz * wx) / 2, (qw * wz + qx * wy - qy * wx) / 2]

    def quat(x, u):
        m, jx, jy, jz, _, _, cd, g = k
        vx, vy, vz, qw, qx, qy, qz, wx, wy, wz = [x[..., j] for j in range(3, 13)]
        t, tx, ty, tz = [u[..., j] for j in range(4)]
        return torch.stack([
            vx, vy, vz,
            2 * (qx * qz + qw * qy) * t / m - cd / m * vx,
            2 * (qy * qz - qw * qx) * t / m - cd / m * vy,
            (qw * qw - qx * qx - qy * qy + qz * qz) * t / m - g - cd / m * vz,
            *spin((qw, qx, qy, qz), (wx, wy, wz)),
            (tx - (jz - jy) * wy * wz) / jx, (ty - (jx - jz) * wz * wx) / jy, (tz - (jy - jx) * wx * wy) / jz], -1)

    def mars(x, u):
        g, alpha = k[0], k[1]
        acc = u / x[..., 6:7]
        up = torch.stack([g, 0 * g, 0 * g], -1)
        return torch.cat([x[..., 3:6], acc - up, -(alpha * u.square().sum(-1).sqrt())[..., None]], -1)

    def mars6(x, u):
        alpha, g, jx, jy, jz, lever = k[:6]
        m, qw, qx, qy, qz, wx, wy, wz = [x[..., j] for j in (0, 7, 8, 9, 10, 11, 12, 13)]
        a, b, c = [u[..., j] for j in range(3)]
        fx = (qw * qw + qx * qx - qy * qy - qz * qz) * a + 2 * (qx * qy - qw * qz) * b + 2 * (qx * qz + qw * qy) * c
        fy = 2 * (qx * qy + qw * qz) * a + (qw * qw - qx * qx + qy * qy - qz * qz) * b + 2 * (qy * qz - qw * qx) * c
        fz = 2 * (qx * qz - qw * qy) * a + 2 * (qy * qz + qw * qx) * b + (qw * qw - qx * qx - qy * qy + qz * qz) * c
        return torch.stack([
            -alpha * u.square().sum(-1).sqrt(), x[..., 4], x[..., 5], x[..., 6],
            fx / m - g, fy / m, fz / m, *spin((qw, qx, qy, qz), (wx, wy, wz)),
            -(jz - jy) * wy * wz / jx, (lever * c - (jx - jz) * wz * wx) / jy, (-lever * b - (jy - jx) * wx * wy) / jz], -1)

    return {"quad": quad, "quat": quat, "mars": mars, "mars6": mars6}[model]


def _ball(v, r):
    n = v.norm(dim=-1, keepdim=True)
    return torch.where(n > r, v * (r / n), v)


def _cone(v, tau):
    """Onto {(t, y): |y| <= tau t}."""
    t, y = v[..., :1], v[..., 1:]
    s = y.norm(dim=-1, keepdim=True)
    c = (t + s * tau) / (1 + tau * tau)
    edge = torch.cat([c, tau * c * y / s.clamp_min(1e-300)], -1)
    return torch.where(s <= tau * t, v, torch.where(tau * s <= -t, torch.zeros_like(v), edge))


class _Exact:
    """The method on a batch padded to its longest horizon: node i of an instance
    is live while i <= N, and has a control while i < N."""

    def __init__(self, model, p, group=1):
        dev = "cuda" if torch.cuda.is_available() else "cpu"

        def t(a):
            return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)

        self.model, self.p, self.group, self.t = model, p, group, t
        self.nx, self.nu, self.B, self.M = p.nx, p.nu, p.batch, int(p.N.max()) + 1
        N = torch.as_tensor(p.N.astype(np.int64), device=dev)[:, None]
        i = torch.arange(self.M, device=dev)[None, :]
        self.live, self.hasu, self.term, self.later = i <= N, i < N, i == N, (i >= 1) & (i <= N)
        self.one = {k: v.double()[..., None] for k, v in dict(live=self.live, hasu=self.hasu, term=self.term, later=self.later).items()}
        self.h = t(p.dt)[:, None, None]
        self.f = _dynamics(model, t(p.params)[:, None, :])
        self.sets = t(p.sets)[:, None, None, :]
        self.Q = torch.where(self.term[..., None], t(p.QNd)[:, None], t(p.Qd)[:, None])
        self.R = t(p.Rd)[:, None].expand(-1, self.M, -1)
        self.lin = self.Q * t(p.xref)[:, None] - self.one["term"] * t(p.qN)[:, None]
        self.linu = self.R * t(p.uref)[:, None]
        self.xi_ref = t(p.xref)[:, None], t(p.uref)[:, None]
        self.w_d = p.settings["w_d"]

    def pad(self, x, u):
        X = torch.zeros(self.B, self.M, self.nx, dtype=torch.float64, device=self.live.device)
        U = torch.zeros(self.B, self.M, self.nu, dtype=torch.float64, device=self.live.device)
        X[self.live], U[self.hasu] = self.t(x), self.t(u)
        for dead, filled in ((~self.live, X), (~self.hasu, U)):   # any regular point: its results are masked
            filled[dead] = (filled[:, :1].expand_as(filled))[dead]
        return X, U

    def rk4(self, x, u):
        h, f = self.h, self.f
        a = f(x, u)
        b = f(x + h / 2 * a, u)
        c = f(x + h / 2 * b, u)
        d = f(x + h * c, u)
        return x + h / 6 * (a + 2 * b + 2 * c + d)

    def linearize(self, X, U):
        """[A B] and d of every node (zero where a node has no control)."""
        cols = []
        for j in range(self.nx + self.nu):
            ex, eu = torch.zeros_like(X), torch.zeros_like(U)
            (ex if j < self.nx else eu)[..., j if j < self.nx else j - self.nx] = 1
            cols.append(torch.func.jvp(self.rk4, (X, U), (ex, eu))[1])
        AB = torch.stack(cols, -1)
        d = self.rk4(X, U) - (AB @ torch.cat([X, U], -1)[..., None])[..., 0]
        return AB * self.one["hasu"][..., None], d * self.one["hasu"]

    def mirrors(self, X, U):
        """G of the non-box sets as linear maps of (x, u), and their projection."""
        B, M, nx, n = self.B, self.M, self.nx, self.nx + self.nu
        if self.model in ("quad", "quat"):
            c, r = self.t(self.p.obs_c)[:, None], self.t(self.p.obs_r)[:, None]
            used = torch.arange(r.shape[-1], device=X.device)[None, None] < torch.as_tensor(self.p.nobs, device=X.device)[:, None, None]
            v = X[..., None, :3] - c
            nv = v / v.norm(dim=-1, keepdim=True)
            G = nv * (used & self.live[..., None]).double()[..., None]
            low = (nv * c).sum(-1) + r
            return slice(0, 3), G, lambda s: torch.maximum(s, low)
        tmin, tmax, tau, tgim, rtilt, wmax = [self.sets[..., 0, j:j + 1] for j in range(6)]
        pos = 1 if self.model == "mars6" else 0
        rows = [pos, pos + 1, pos + 2] + ([9, 10, 11, 12, 13] if pos else []) + [nx, nx + 1, nx + 2]
        G = torch.zeros(B, M, len(rows) + 1 + (3 if pos else 0), n, dtype=torch.float64, device=X.device)
        for k, r in enumerate(rows):
            G[..., k, r] = 1
        k = len(rows)
        G[..., k, nx:nx + 3] = U / U.norm(dim=-1, keepdim=True)
        for j in range(3 if pos else 0):
            G[..., k + 1 + j, nx + j] = 1
        on = torch.where(torch.tensor([bool((G[0, 0, r, nx:] != 0).any()) for r in range(G.shape[2])], device=X.device),
                         self.one["hasu"], self.one["live"])
        G = G * on[..., None]

        def project(s):
            parts = [_cone(s[..., 0:3], tau)]
            if pos:
                parts += [_ball(s[..., 3:5], rtilt), _ball(s[..., 5:8], wmax)]
            parts += [_ball(s[..., k - 3:k], tmax), torch.maximum(s[..., k:k + 1], tmin)]
            if pos:
                parts.append(_cone(s[..., k + 1:k + 4], tgim))
            return torch.cat(parts, -1)

        return slice(0, n), G, project

    def box(self, X, U, radius):
        p, r = self.p, radius[:, None, None]
        lo, hi = torch.maximum(self.t(p.xlo)[:, None], X - r), torch.minimum(self.t(p.xhi)[:, None], X + r)
        end = self.term[..., None] & (self.t(p.tmask)[:, None] != 0)
        lo, hi = (torch.where(end, self.t(p.xtarget)[:, None], v) for v in (lo, hi))
        lo[:, 0], hi[:, 0] = self.t(p.xinit), self.t(p.xinit)
        ulo, uhi = torch.maximum(self.t(p.ulo)[:, None], U - r), torch.minimum(self.t(p.uhi)[:, None], U + r)
        return torch.cat([lo, ulo], -1), torch.cat([hi, uhi], -1)

    def start(self, X, U):
        xi = torch.cat([X, U], -1)
        return dict(z=X.clone(), lam=torch.zeros_like(X), mu=torch.zeros_like(X), hat=xi, nu=torch.zeros_like(xi), nus=None)

    def admm(self, S, X, U, AB, d, radius, rho, iters):
        """`iters` iterations of Steps 1-4 on the state S; the last one's residuals."""
        re, rd, rg = rho
        nx, live, hasu, later = self.nx, self.one["live"], self.one["hasu"], self.one["later"]
        cols, G, project = self.mirrors(X, U)
        GT, ABT = G.transpose(-1, -2).contiguous(), AB.transpose(-1, -2).contiguous()
        H = rd * (ABT @ AB)
        H[..., cols, cols] += rg * (GT @ G)
        diag = torch.cat([self.Q + rg + re * later, (self.R + rg) * hasu + (1 - hasu)], -1)
        H.diagonal(dim1=-2, dim2=-1).add_(torch.where(self.live[..., None], diag, torch.ones_like(diag)))
        Hi = torch.linalg.inv(H)
        lin = torch.cat([self.lin * live, self.linu * hasu], -1)
        keep = torch.cat([live.expand(-1, -1, nx), hasu.expand(-1, -1, self.nu)], -1)
        lo, hi = self.box(X, U, radius)

        def mul(m, v):
            return (m @ v[..., None])[..., 0]

        def shift(v, by):
            out = torch.zeros_like(v)
            if by > 0:
                out[:, 1:] = v[:, :-1]
            else:
                out[:, :-1] = v[:, 1:]
            return out

        s = project(mul(G, S["hat"][..., cols]))
        nus = torch.zeros_like(s) if S["nus"] is None else S["nus"]
        z, lam, mu, hat, nu = S["z"], S["lam"], S["mu"], S["hat"], S["nu"]
        res = None
        for it in range(iters):
            g = lin + rg * hat - nu + mul(ABT, shift(mu + rd * z, -1) - rd * d)
            g[..., :nx] += later * (re * z - lam)
            g[..., cols] += mul(GT, rg * s - nus)
            xi = mul(Hi, g * keep)
            x = xi[..., :nx]
            dd = shift(mul(AB, xi) + d, 1)
            zn = (re * x + lam + rd * dd - mu) / (re + rd)
            lam, mu = later * (lam + re * (x - zn)), later * (mu + rd * (zn - dd))
            arg, l, h = xi + nu / rg, lo, hi
            if self.group > 1:   # the scenarios' first control: the mean, within every box
                a, l, h = (v.clone() for v in (arg, lo, hi))
                of = (self.B // self.group, self.group, self.nu)
                for v, how in ((a, torch.mean), (l, torch.amax), (h, torch.amin)):
                    v[:, 0, nx:] = how(v[:, 0, nx:].reshape(of), 1, keepdim=True).expand(of).reshape(self.B, self.nu)
                arg = a
            hn = torch.minimum(torch.maximum(arg, l), h)
            nu = nu + rg * (xi - hn)
            y = mul(G, xi[..., cols])
            sn = project(y + nus / rg)
            nus = nus + rg * (y - sn)
            if it + 1 == iters:
                used = (G != 0).any(-1).double()
                dz = later * (zn - z)
                pr = (keep * (xi - hn)).square().sum((1, 2)) + (used * (y - sn)).square().sum((1, 2)) + \
                    (later * (x - zn)).square().sum((1, 2)) + (later * (zn - dd)).square().sum((1, 2))
                dv = rg * (hn - hat) + rd * mul(ABT, shift(dz, -1))
                dv[..., :nx] += re * dz
                dv[..., cols] += rg * mul(GT, sn - s)
                res = torch.stack([pr.sqrt(), (keep * dv).square().sum((1, 2)).sqrt()], -1)
            z, hat, s = zn, hn, sn
        S.update(z=z, lam=lam, mu=mu, hat=hat, nu=nu, nus=nus)
        return res

    def cost(self, X, U):
        ex, eu = X - self.xi_ref[0], U - self.xi_ref[1]
        c = self.one["live"] * self.Q * ex * ex / 2 + self.one["term"] * self.t(self.p.qN)[:, None] * X
        return c.sum((1, 2)) + (self.one["hasu"] * self.R * eu * eu / 2).sum((1, 2))

    def by_group(self, v, how):
        if self.group <= 1:
            return v
        return how(v.reshape(-1, self.group), 1, keepdim=True).expand(-1, self.group).reshape(-1)

    def scp(self, iters, admm, rho, rho_final):
        p, st = self.p, self.p.settings
        X, U = self.pad(p.xguess, p.uguess)
        S = self.start(X, U)
        nxt = lambda v: torch.cat([v[:, 1:], v[:, -1:]], 1)  # noqa: E731
        gap = lambda x, u: self.one["hasu"] * (self.rk4(x, u) - nxt(x))  # noqa: E731
        radius = torch.full((self.B,), float(st["tr_init"]), dtype=torch.float64, device=X.device)
        J = self.cost(X, U) + self.w_d * gap(X, U).abs().sum((1, 2))
        for k in range(iters):
            f = (rho_final / rho) ** (k / (iters - 1)) if rho_final > 0 and iters > 1 else 1.0
            AB, d = self.linearize(X, U)
            self.admm(S, X, U, AB, d, radius, (rho * f,) * 3, admm)
            Xc, Uc = S["hat"][..., :self.nx], S["hat"][..., self.nx:]
            Xc, Uc = torch.where(self.live[..., None], Xc, X), torch.where(self.hasu[..., None], Uc, U)
            cost = self.cost(Xc, Uc)
            Jc = cost + self.w_d * gap(Xc, Uc).abs().sum((1, 2))
            model = self.one["hasu"] * ((AB @ S["hat"][..., None])[..., 0] + d - nxt(Xc))
            L = cost + self.w_d * model.abs().sum((1, 2))
            den, num = self.by_group(J, torch.sum) - self.by_group(L, torch.sum), self.by_group(J, torch.sum) - self.by_group(Jc, torch.sum)
            tiny, ratio = den <= 1e-12, num / den
            radius = torch.where(~tiny & (ratio < 0.25), radius / 2, torch.where(~tiny & (ratio > 0.75), (2 * radius).clamp_max(st["tr_max"]), radius))
            radius = radius.clamp_min(st["tr_min"])
            yes = tiny | (ratio > 0)
            J = torch.where(yes, Jc, J)
            X, U = torch.where(yes[:, None, None], Xc, X), torch.where(yes[:, None, None], Uc, U)
        defect = gap(X, U).abs().amax((1, 2))
        status = torch.where(defect <= st["defect_tol"], ucn.UCN_OK, ucn.UCN_ENOTCONV).to(torch.int32)
        return {"x": X[self.live], "u": U[self.hasu], "status": status}


def exact(case, seed):
    c = case
    if c["kind"] == "serve":
        reqs = _requests(c, seed)
        got = [None] * len(reqs)
        for model, code in (("quad", W.MODEL_QUAD12), ("mars", W.MODEL_MARS7)):
            of = [k for k, p in enumerate(reqs) if p.model == code]
            if of:
                p = _merge([reqs[k] for k in of])
                e = _Exact(model, p).scp(p.settings["scp_iters"], p.settings["admm_iters"], p.settings["rho_geo"], p.settings["rho_final"])
                for j, k in enumerate(of):
                    xo, uo, n = p.xoff[j], p.uoff[j], int(p.N[j])
                    got[k] = {"x": e["x"][xo:xo + n + 1], "u": e["u"][uo:uo + n], "status": e["status"][j:j + 1]}
        return {k: torch.cat([g[k].reshape(-1) for g in got]) for k in ("x", "u", "status")}
    p = _problem(c, seed)
    e = _Exact(c["model"], p, c.get("group", 1))
    if c["kind"] == "scp":
        return e.scp(c["scp"], c["admm"], c["rho"], p.settings["rho_final"])
    X, U = e.pad(*_nominal(p, seed))
    AB, d = e.linearize(X, U)
    if c["kind"] == "linearize":
        AB = AB[e.hasu]
        return {"A": AB[..., :p.nx].contiguous(), "B": AB[..., p.nx:].contiguous(), "d": d[e.hasu]}
    S = e.start(X, U)
    res = e.admm(S, X, U, AB, d, torch.full((e.B,), 0.7, dtype=torch.float64, device=X.device), (c["rho"],) * 3, c["admm"])
    return {"x": S["hat"][..., :p.nx][e.live], "u": S["hat"][..., p.nx:][e.hasu], "res": res,
            "status": torch.zeros(e.B, dtype=torch.int32, device=X.device)}
