"""Performance cases: the calls that programs built on this package spend their time in.

Every case is one pass through the public Python entry points of
``paper_2303_11767_gb300.dgswe``.  The kinds:

* ``advance``   a resident state on the sphere advanced by a block of time steps and
                read back on the device (what a simulation does between two outputs);
                with ``cfl`` set, the step size is taken from the state first and the
                total mass is read afterwards, as a program that controls its step does;
* ``ensemble``  a batch of meshes of uneven sizes and degrees advanced together, the
                members' states read back to the host;
* ``plane``     shallow water on the periodic f-plane (the geostrophic adjustment set-up);
* ``learned``   the coarse degree-1 solver with the per-element network attached;
* ``train``     one Adam step of that network on a batch, the parameters read back;
* ``start``     the start of a run: point values on the host projected onto the basis,
                the state set, the CFL step and the total mass taken, the state read back.

``exact`` evaluates the same calls in 64 bits with plain torch, from the definitions.
"""
import math

import numpy as np
import torch

R, G, OMEGA = 6.37122e6, 9.80616, 7.292e-5
CFL = 0.1
CMAX = 275.0           # bound of sqrt(u^2 + v^2) + sqrt(g h) over the initial fields below
PLANE_L, PLANE_F = 1.0e7, 1.0e-4
BYTES = {"fp64": 8}    # bytes of one stored value; every other precision stores 32 bits
# Relative error of a state, about four times the largest seen against exact() over meshes of 16..1010
# columns, every degree and up to 60 steps (FP32 4e-8, BF16 5e-4, FP16 8e-5, split pairs 1e-6 and 2e-7).
REL = {"fp64": 5e-14, "fp32": 1.6e-7, "fp32_tc_bf16": 2e-3, "fp32_tc_fp16": 3e-4, "fp32_tc_bf16x3": 4e-6,
       "fp32_tc_fp16x3": 8e-7}


def _advance(nlon, nlat, p, prec, steps, rk=3, cfl=0):
    return {"kind": "advance", "nlon": nlon, "nlat": nlat, "degree": p, "precision": prec, "rk": rk, "steps": steps,
            "cfl": cfl}


def listed():
    return [
        # a teaching-size FP64 run (the default precision): launches and latency only
        dict(_advance(20, 10, 1, "fp64", 100), name="sphere_20x10_p1_fp64"),
        # a 2-degree mesh in FP32: one wave of tiles per stage
        dict(_advance(180, 90, 3, "fp32", 50), name="sphere_180x90_p3_fp32"),
        # the benchmark's headline mesh, production precision
        dict(_advance(360, 180, 4, "fp32", 20), name="sphere_360x180_p4_fp32"),
        # a quarter-degree mesh: state arrays far larger than the caches
        dict(_advance(1440, 720, 4, "fp32", 4), name="sphere_1440x720_p4_fp32"),
        # odd sizes, CFL-controlled step, mass diagnostic each block
        dict(_advance(241, 121, 2, "fp32", 8, 3, 1), name="sphere_241x121_p2_fp32_cfl"),
        # the default precision on an ordinary mesh, the classical RK4
        dict(_advance(180, 90, 3, "fp64", 5, 4), name="sphere_180x90_p3_fp64_rk4"),
        # the tensor-core precision on the headline mesh
        dict(_advance(360, 180, 4, "fp32_tc_bf16", 20), name="sphere_360x180_p4_tc_bf16"),
        # uneven meshes of every degree together
        {"name": "ensemble_12", "kind": "ensemble", "members": 12, "lo": 20, "hi": 60, "steps": 50},
        # the planar timing set-up of the paper: 50 x 50, degree 3, RK4
        {"name": "plane_50x50_p3", "kind": "plane", "nx": 50, "ny": 50, "degree": 3, "rk": 4, "steps": 10},
        # the learned coarse solver between two outputs
        {"name": "learned_72x36", "kind": "learned", "nlon": 72, "nlat": 36, "steps": 20},
        # one optimiser step at the training batch
        {"name": "train_4096", "kind": "train", "batch": 4096},
        # a run's start on an ordinary mesh
        {"name": "start_180x90_p3", "kind": "start", "nlon": 180, "nlat": 90, "degree": 3, "precision": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["advance"] * 6 + ["ensemble", "plane", "learned", "train", "start"])
    if kind == "advance":
        nlon = _log_int(rng, 16, 1100)
        nlat = max(8, nlon // 2 + rng.choice([-3, -1, 0, 0, 1, 2]))
        p = rng.choice([0, 1, 1, 2, 2, 3, 3, 4, 4])
        prec = rng.choice(["fp32"] * 5 + ["fp64"] * 3 + ["fp32_tc_bf16", "fp32_tc_fp16", "fp32_tc_bf16x3", "fp32_tc_fp16x3"])
        dof = nlon * nlat * 3 * (p + 1) ** 2
        most = {"fp64": 1.0e7}.get(prec, 1.0e8)   # value updates of a pass
        steps = max(1, min(rng.randint(2, 60), int(most / (3 * dof))))
        return _advance(nlon, nlat, p, prec, steps, rng.choice([3, 3, 3, 3, 1, 2, 4]), int(rng.random() < 0.3))
    if kind == "ensemble":
        return {"kind": kind, "members": rng.randint(2, 24), "lo": rng.randint(9, 30), "hi": rng.randint(31, 75),
                "steps": rng.randint(4, 40)}
    if kind == "plane":
        nx = _log_int(rng, 10, 160)
        return {"kind": kind, "nx": nx, "ny": max(4, int(nx * rng.uniform(0.6, 1.4))), "degree": rng.choice([0, 1, 2, 3, 3, 4]),
                "rk": rng.choice([3, 4]), "steps": rng.randint(1, 10)}
    if kind == "learned":
        nlat = rng.randint(10, 90)
        return {"kind": kind, "nlon": 2 * nlat + rng.choice([-1, 0, 0, 1]), "nlat": nlat, "steps": rng.randint(5, 40)}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 32, 8192)}
    nlon = _log_int(rng, 20, 260)
    return {"kind": kind, "nlon": nlon, "nlat": max(8, nlon // 2 + rng.choice([-1, 0, 1])), "degree": rng.randint(0, 4),
            "precision": rng.choice(["fp32", "fp64"])}


# ---------------------------------------------------------------- the inputs


def _rule(k):
    x, w = np.polynomial.legendre.leggauss(k)
    return torch.tensor(x, device="cuda"), torch.tensor(w, device="cuda")


def _legendre(n, x):
    """Orthonormal Legendre polynomials L_0..L_{n-1} and derivatives at x: two [n, len(x)] tables."""
    x = x.cpu().numpy()
    out = np.zeros((2, n, len(x)))
    for k in range(n):
        q = math.sqrt((2 * k + 1) / 2.0) * np.polynomial.legendre.Legendre.basis(k)
        out[0, k], out[1, k] = q(x), q.deriv(1)(x) if k else 0.0
    return torch.tensor(out[0], device="cuda"), torch.tensor(out[1], device="cuda")


def _points(count, lo, step, x):
    """Coordinates of the points x of [-1, 1] in each of `count` intervals."""
    i = torch.arange(count, dtype=torch.float64, device="cuda")
    return (lo + (i[:, None] + 0.5 * (1.0 + x)) * step).reshape(-1)


def _field(rng, amp, lam, th):
    """A smooth field |f| <= amp on the sphere: a few broad waves and some finer, weaker ones."""
    waves = [(m, 1.0) for m in (0, 1, 2, 3, 4)] + [(rng.integers(5, 13), 0.1) for _ in range(3)]
    c = np.array([a * rng.uniform(-1, 1) for _, a in waves])
    c *= amp / np.abs(c).sum()
    a, b = [], []
    for (m, _), ck in zip(waves, c):
        a.append(ck * torch.cos(int(m) * lam + rng.uniform(0, 2 * math.pi)))
        b.append(torch.cos(th).clamp(min=0) ** int(m) * torch.sin(rng.integers(1, 5) * th + rng.uniform(0, 2 * math.pi)))
    return torch.stack(b).T @ torch.stack(a)


def _sphere_values(lam, th, seed):
    """(h, hu, hv) on the grid th x lam: a 6 km layer with 200 m waves and at most 20 m/s per component."""
    rng = np.random.default_rng(seed)
    h = 5960.0 + _field(rng, 200.0, lam, th)
    u, v = (_field(rng, 20.0, lam, th) * torch.cos(th)[:, None] for _ in range(2))
    return h, h * u, h * v


def _sphere_state(nlon, nlat, p, seed):
    """[nlat, nlon, 3, (p+1)^2] modal coefficients of the fields, n-point projection."""
    n = p + 1
    x, w = _rule(n)
    P = _legendre(n, x)[0] * w
    lam, th = _points(nlon, 0.0, 2 * math.pi / nlon, x), _points(nlat, -math.pi / 2, math.pi / nlat, x)
    out = torch.empty(nlat, nlon, 3, n * n, dtype=torch.float64, device="cuda")
    for f, v in enumerate(_sphere_values(lam, th, seed)):
        s = (v.reshape(-1, n) @ P.T).reshape(nlat, n, nlon, n)                  # [j][q][i][a]
        out[:, :, f] = torch.einsum("bq,jqia->jiba", P, s).reshape(nlat, nlon, n * n)
    return out


def _sphere_dt(nlon, nlat, p, cfl=CFL):
    x = np.polynomial.legendre.leggauss(p + 1)[0]
    H = R * min(math.pi / nlat, math.cos(-math.pi / 2 + 0.5 * (1 + x[0]) * math.pi / nlat) * 2 * math.pi / nlon)
    return cfl * H / (max(p, 1) * CMAX)


def _plane_state(c, seed):
    """Broad height waves and slow flow on the square [0, L]^2."""
    nx, ny, n = c["nx"], c["ny"], c["degree"] + 1
    rng = np.random.default_rng(seed)
    x, w = _rule(n)
    P = _legendre(n, x)[0] * w
    X, Y = _points(nx, 0.0, PLANE_L / nx, x), _points(ny, 0.0, PLANE_L / ny, x)
    f = []
    for amp in (5.0, 0.2, 0.2):
        v = 0.0
        for _ in range(4):
            kx, ky = rng.integers(0, 4, 2) * 2 * math.pi / PLANE_L
            v = v + amp / 4 * torch.outer(torch.sin(ky * Y + rng.uniform(0, 6)), torch.cos(kx * X + rng.uniform(0, 6)))
        f.append(v)
    h = 1000.0 + f[0]
    out = torch.empty(ny, nx, 3, n * n, dtype=torch.float64, device="cuda")
    for k, v in enumerate((h, h * f[1], h * f[2])):
        s = (v.reshape(-1, n) @ P.T).reshape(ny, n, nx, n)
        out[:, :, k] = torch.einsum("bq,jqia->jiba", P, s).reshape(ny, nx, n * n)
    return out


def _plane_dt(c):
    return 0.2 * PLANE_L / max(c["nx"], c["ny"]) / ((2 * c["degree"] + 1) * 100.0)


def _members(c, seed):
    """Mesh sizes and degrees of an ensemble: part of the case and not of its inputs."""
    rng = np.random.default_rng(1000 * c["members"] + c["lo"] + c["hi"])
    nlat = [int(v) for v in rng.integers(c["lo"], c["hi"] + 1, c["members"])]
    deg = [1 + k % 4 for k in range(c["members"])]
    return [2 * v for v in nlat], nlat, deg


def _network(seed):
    """60-128-128-12 parameters in the library's order, He-uniform with small biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for rows, cols in ((128, 60), (128, 128), (12, 128)):
        a = math.sqrt(6.0 / cols)
        parts += [rng.uniform(-a, a, rows * cols), rng.uniform(-0.1, 0.1, rows)]
    return np.concatenate(parts).astype(np.float32)


def _gather(u):
    """[nlat, nlon, 3, 4] modes -> [nlat * nlon, 60]: the element, then W, E, S, N (zeros across a pole)."""
    e = u.reshape(u.shape[0], u.shape[1], 12)
    zero = torch.zeros_like(e[:1])
    s, n = torch.cat([zero, e[:-1]]), torch.cat([e[1:], zero])
    return torch.cat([e, e.roll(1, 1), e.roll(-1, 1), s, n], -1).reshape(-1, 60)


def _learned_norm(u):
    """Input statistics of the state, and output scales of a slow drift."""
    x = _gather(u)
    std = x.std(0)
    std[std == 0] = 1.0
    ys = 1e-8 * u.abs().reshape(-1, 12).amax(0) + 1e-20
    return [v.float().cpu().numpy() for v in (x.mean(0), std, torch.zeros(12), ys)]


def _train_batch(c, seed):
    """Network inputs at the magnitudes of modal states and targets at those of tendencies."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    scale = torch.tensor([100.0, 10.0, 10.0, 1.0] + [4e4, 4e3, 4e3, 4e2] * 2, device="cuda").repeat(5)
    mean = torch.tensor([1.2e4] + [0.0] * 11, device="cuda").repeat(5)
    x = mean + scale * torch.randn(c["batch"], 60, generator=g, device="cuda")
    tscale = 1e-4 * scale[:12]
    t = tscale * (0.7 * torch.tanh(((x - mean) / scale)[:, 12:24]) + 0.3 * torch.randn(c["batch"], 12, generator=g, device="cuda"))
    norm = [v.cpu().numpy() for v in (mean, scale, torch.zeros(12), tscale)]
    return x, t, norm


def _nodal(c, seed):
    """Point values on the tensor grid of p + 9 points per element and direction, [j][i][f][q][r] on the host."""
    nlon, nlat, nm = c["nlon"], c["nlat"], c["degree"] + 9
    x, _ = _rule(nm)
    lam, th = _points(nlon, 0.0, 2 * math.pi / nlon, x), _points(nlat, -math.pi / 2, math.pi / nlat, x)
    v = torch.stack([f.reshape(nlat, nm, nlon, nm).permute(0, 2, 1, 3) for f in _sphere_values(lam, th, seed)], 2)
    return v.contiguous().cpu().numpy()


# ----------------------------------------------------------------- the calls


def prepare(case, seed):
    from paper_2303_11767_gb300 import dgswe

    kind, st = case["kind"], {"case": case}
    if kind == "advance":
        s = dgswe.Solver(case["nlon"], case["nlat"], case["degree"], precision=case["precision"], rk_order=case["rk"])
        u = _sphere_state(case["nlon"], case["nlat"], case["degree"], seed)
        torch.cuda.synchronize()
        s.set_state_device(u)
        st.update(solver=s, dt=_sphere_dt(case["nlon"], case["nlat"], case["degree"]), out=torch.empty_like(u))
    elif kind == "ensemble":
        nlon, nlat, deg = _members(case, seed)
        e = dgswe.Ensemble(nlon, nlat, deg)
        for m in range(e.members):
            e.set_state(m, _sphere_state(nlon[m], nlat[m], deg[m], seed + 1000 * m).cpu().numpy())
        e.set_dt([_sphere_dt(a, b, d) for a, b, d in zip(nlon, nlat, deg)])
        st.update(ensemble=e)
    elif kind == "plane":
        s = dgswe.Solver.plane_swe(case["nx"], case["ny"], case["degree"], L=PLANE_L, f=PLANE_F, rk_order=case["rk"])
        u = _plane_state(case, seed)
        torch.cuda.synchronize()
        s.set_state_device(u)
        st.update(solver=s, dt=_plane_dt(case), out=torch.empty_like(u))
    elif kind == "learned":
        s = dgswe.Solver(case["nlon"], case["nlat"], 1, precision="fp32")
        u = _sphere_state(case["nlon"], case["nlat"], 1, seed)
        net = dgswe.MLP()
        net.set_params(_network(seed))
        net.set_normalization(*_learned_norm(u))
        torch.cuda.synchronize()
        s.set_state_device(u)
        s.attach_mlp(net)
        st.update(solver=s, net=net, dt=_sphere_dt(case["nlon"], case["nlat"], 1), out=torch.empty_like(u))
    elif kind == "train":
        x, t, norm = _train_batch(case, seed)
        net = dgswe.MLP()
        net.set_params(_network(seed))
        net.set_normalization(*norm)
        st.update(net=net, x=x, t=t)
    else:
        s = dgswe.Solver(case["nlon"], case["nlat"], case["degree"], precision=case["precision"])
        st.update(solver=s, values=_nodal(case, seed))
    torch.cuda.synchronize()
    return st


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind in ("advance", "plane", "learned"):
        s, out = state["solver"], state["out"]
        if not c.get("cfl"):
            s.step(c["steps"], state["dt"])
            s.get_state_device(out)
            return {"state": out}
        dt = s.max_dt(CFL)
        s.step(c["steps"], dt)
        s.get_state_device(out)
        return {"state": out, "dt": dt, "mass": s.total_mass()}
    if kind == "ensemble":
        e = state["ensemble"]
        e.step(c["steps"])
        return [e.get_state(m) for m in range(e.members)]
    if kind == "train":
        loss = state["net"].train_step(state["x"], state["t"], 1e-3)
        return {"loss": loss, "params": state["net"].get_params()}
    s = state["solver"]
    u = s.project_nodal(state["values"])
    s.set_state(u)
    return {"projected": u, "dt": s.max_dt(CFL), "mass": s.total_mass(), "state": s.get_state()}


def _stage_work(elements, p, stages, word):
    """One stage: the state read and written with the increments of the scheme (8/3 words per value at
    least), and the sum-factorised operations with a multiply-add as two."""
    n = p + 1
    return 8.0 / 3.0 * word * elements * 3 * n * n * stages, (40 * n ** 3 + 117 * n ** 2 + 100 * n) * elements * stages


def work(case):
    c, kind = case, case["kind"]
    if kind == "advance":
        b, f = _stage_work(c["nlon"] * c["nlat"], c["degree"], c["steps"] * c["rk"], BYTES.get(c["precision"], 4))
    elif kind == "plane":
        b, f = _stage_work(c["nx"] * c["ny"], c["degree"], c["steps"] * c["rk"], 8)
    elif kind == "ensemble":
        parts = [_stage_work(a * b, d, c["steps"] * 3, 4) for a, b, d in zip(*_members(c, 0))]
        b, f = (sum(x) for x in zip(*parts))
    elif kind == "learned":
        e = c["nlon"] * c["nlat"]
        b, f = _stage_work(e, 1, c["steps"] * 3, 4)
        f += 2.0 * (60 * 128 + 128 * 128 + 128 * 12) * e * c["steps"] * 3
    elif kind == "train":
        macs = 60 * 128 + 128 * 128 + 128 * 12
        b, f = 4.0 * (72 * c["batch"] + 8 * macs), 6.0 * macs * c["batch"]
    else:
        e, n, nm = c["nlon"] * c["nlat"] * 3, c["degree"] + 1, c["degree"] + 9
        b, f = 8.0 * e * (nm * nm + 2 * n * n), 2.0 * e * (nm * nm * n + nm * n * n + n ** 3)
    return {"bytes": b, "flops": f}


def tolerance(case):
    kind = case["kind"]
    if kind == "advance":
        rel = REL[case["precision"]]
        return {"rel": rel, "max": min(0.5, 10 * rel if case["precision"].startswith("fp32") else 40 * rel)}
    if kind == "ensemble":
        return {"rel": REL["fp32"], "max": 10 * REL["fp32"]}
    if kind == "plane":
        return {"rel": 3e-13, "max": 3e-12}
    if kind == "learned":
        return {"rel": 4e-8, "max": 6e-7}
    if kind == "train":
        # where a gradient is near Adam's epsilon its rounding decides the size of that parameter's step
        return {"rel": 2e-6, "max": 1e-3}
    # the FP32 CFL step reads the rounded state
    return {"rel": 2e-8 if case["precision"] == "fp32" else 1e-13}


# ------------------------------------------------------- the same in 64 bits


class _Exact:
    """The semi-discrete operator in 64 bits: dense point maps of the orthonormal Legendre basis, the Rusanov
    flux with the larger one-sided speed, the cos(theta)-weighted mass matrix of each row, explicit RK."""

    def __init__(self, nx, ny, p, plane=False):
        self.nx, self.ny, self.n, self.plane = nx, ny, p + 1, plane
        n = self.n
        x, w = _rule(n)
        L, D = _legendre(n, x)
        lo, hi = _legendre(n, torch.tensor([-1.0]))[0][:, 0], _legendre(n, torch.tensor([1.0]))[0][:, 0]
        kr = lambda b, a: torch.einsum("bq,ar->baqr", b, a).reshape(n * n, -1)  # noqa: E731  modes x points
        self.eval = torch.cat([kr(L, L), kr(L, lo[:, None]), kr(L, hi[:, None]), kr(lo[:, None], L), kr(hi[:, None], L)], 1)
        wl, wd = w * L, w * D
        self.lift = torch.cat([kr(wl, wd), kr(wd, wl), kr(wl, wl), kr(wl, lo[:, None]), -kr(wl, hi[:, None]),
                               kr(lo[:, None], wl), -kr(hi[:, None], wl)], 1).T.contiguous()
        if plane:
            self.cF, self.cG = 2 * nx / PLANE_L, 2 * ny / PLANE_L
            return
        self.dth = math.pi / ny
        self.dlam = 2 * math.pi / nx
        self.cF, self.cG = 2 / (R * self.dlam), 2 / (R * self.dth)
        th = _points(ny, -math.pi / 2, self.dth, x).reshape(ny, 1, n, 1).expand(ny, 1, n, n).reshape(ny, 1, n * n)
        self.cos, self.sin = torch.cos(th), torch.sin(th)
        edge = torch.cos(-math.pi / 2 + torch.arange(ny + 1, dtype=torch.float64, device="cuda") * self.dth)
        edge[0] = edge[-1] = 0.0
        self.edge = edge.reshape(-1, 1, 1)
        xm, wm = _rule(n + 12)
        M = _legendre(n, xm)[0]
        self.C = torch.einsum("q,bq,cq,jq->jbc", wm, M, M, torch.cos(_points(ny, -math.pi / 2, self.dth, xm)).reshape(ny, -1))
        self.Ci = torch.linalg.inv(self.C)

    def rhs(self, u):
        n, NP = self.n, self.n ** 2
        v = u @ self.eval
        q, e = v[..., :NP], v[..., NP:].reshape(*v.shape[:-1], 4, n)   # edge values W, E, S, N
        h, hu, hv = q.unbind(2)
        ux, uy, P = hu / h, hv / h, 0.5 * G * h * h
        if self.plane:
            c, S = 1.0, torch.stack([0 * h, PLANE_F * hv, -PLANE_F * hu], 2)
        else:
            c = self.cos
            K = self.sin * (2 * OMEGA * c + ux / R)
            S = torch.stack([0 * h, K * hv, -(P * self.sin / R) - K * hu], 2)
        F = self.cF * torch.stack([hu, hu * ux + P, hu * uy], 2)
        Gx = self.cG * torch.stack([c * hv, c * (hv * ux), c * (hv * uy + P)], 2)
        west = self._face(e[..., 1, :].roll(1, 1), e[..., 0, :], 1)
        if self.plane:
            south = self._face(e[..., 3, :].roll(1, 0), e[..., 2, :], 2)
            north = south.roll(-1, 0)
        else:
            inner = self._face(e[:-1, ..., 3, :], e[1:, ..., 2, :], 2) * self.edge[1:-1, :, :, None]
            zero = torch.zeros_like(e[:1, ..., 2, :])
            south, north = torch.cat([zero, inner]), torch.cat([inner, zero])
        flux = torch.cat([F, Gx, S, self.cF * west, self.cF * west.roll(-1, 1), self.cG * south, self.cG * north], -1)
        k = flux @ self.lift
        if self.plane:
            return k
        return torch.einsum("jbc,jifca->jifba", self.Ci, k.reshape(*k.shape[:3], n, n)).reshape(k.shape)

    @staticmethod
    def _face(lo, hi, d):
        """Rusanov flux between the states lo (west / south) and hi in direction d (1: hu, 2: hv)."""
        def one(q):
            h, m = q[:, :, 0], q[:, :, d]
            s = m / h
            f = [m, q[:, :, 1] * s, q[:, :, 2] * s]
            f[d] = f[d] + 0.5 * G * h * h
            return torch.stack(f, 2), s.abs() + torch.sqrt(G * h)
        fl, al = one(lo)
        fh, ah = one(hi)
        return 0.5 * (fl + fh) - 0.5 * torch.maximum(al, ah)[:, :, None] * (hi - lo)

    def step(self, u, dt, rk, source=None):
        f = self.rhs if source is None else lambda v: self.rhs(v) + source(v)
        k1 = f(u)
        if rk == 1:
            return u + dt * k1
        if rk == 2:
            return u + 0.5 * dt * (k1 + f(u + dt * k1))
        if rk == 3:
            k2 = f(u + dt * k1)
            return u + dt / 6 * (k1 + k2 + 4 * f(u + 0.25 * dt * (k1 + k2)))
        k2 = f(u + 0.5 * dt * k1)
        k3 = f(u + 0.5 * dt * k2)
        return u + dt / 6 * (k1 + 2 * k2 + 2 * k3 + f(u + dt * k3))

    def max_dt(self, u):
        NP = self.n ** 2
        h, hu, hv = (u @ self.eval[:, :NP]).unbind(2)
        c = (torch.hypot(hu / h, hv / h) + torch.sqrt(G * h)).max().item()
        H = R * min(self.dth, self.cos.min().item() * self.dlam)
        return CFL * H / (max(self.n - 1, 1) * c)

    def mass(self, u):
        n = self.n
        hb = u[:, :, 0].reshape(self.ny, self.nx, n, n)[..., 0].sum(1)          # [j][b], a = 0
        return R * R * 0.5 * self.dlam * self.dth * (self.C[:, 0] * hb).sum().item()


def _layers(params):
    p, out, at = torch.tensor(params, device="cuda"), [], 0
    for rows, cols in ((128, 60), (128, 128), (12, 128)):
        w, at = p[at:at + rows * cols].reshape(rows, cols), at + rows * cols
        b, at = p[at:at + rows], at + rows
        out.append((w.bfloat16().double(), b.double()))    # the products use 16-bit weights
    return out


def _gelu(z):
    return 0.5 * z * (1 + torch.erf(z / math.sqrt(2.0)))


def _source(ex, params, norm):
    (w1, b1), (w2, b2), (w3, b3) = _layers(params)
    im, istd, om, ostd = (torch.tensor(v, device="cuda").double() for v in norm)
    area = ex.C[:, 0, 0].sum() * ex.nx

    def source(u):
        a = _gelu(_gelu(((_gather(u) - im) / istd) @ w1.T + b1) @ w2.T + b2)
        s = ((a @ w3.T + b3) * ostd + om).reshape(ex.ny, ex.nx, 12)
        added = (ex.C[:, 0, 0] * s[..., 0].sum(1) + ex.C[:, 0, 1] * s[..., 2].sum(1)).sum()
        s[..., 0] -= added / area
        return s.reshape(ex.ny, ex.nx, 3, 4)
    return source


def _exact_train(case, seed):
    x, t, norm = _train_batch(case, seed)
    params = _network(seed)
    im, istd, om, ostd = (torch.tensor(v, device="cuda").double() for v in norm)
    leaves = [v.requires_grad_() for pair in _layers(params) for v in pair]
    a = (x.double() - im) / istd
    for k in (0, 2):
        a = _gelu(a @ leaves[k].T + leaves[k + 1])
    y = a @ leaves[4].T + leaves[5]
    loss = ((y - (t.double() - om) / ostd) ** 2).mean()
    loss.backward()
    g = torch.cat([v.grad.reshape(-1) for v in leaves])
    # Adam's first step: the bias-corrected moments are g and g^2
    p = torch.tensor(params, device="cuda").double() - 1e-3 * g / (g.abs() + 1e-8)
    return {"loss": loss.item(), "params": p.cpu().numpy()}


def _exact_start(case, seed):
    n, nm = case["degree"] + 1, case["degree"] + 9
    ex = _Exact(case["nlon"], case["nlat"], case["degree"])
    x, w = _rule(nm)
    P = _legendre(n, x)[0] * w
    cos = torch.cos(_points(ex.ny, -math.pi / 2, ex.dth, x)).reshape(ex.ny, nm)
    r = torch.einsum("bq,jq,jifqr,ar->jifba", P, cos, torch.tensor(_nodal(case, seed), device="cuda"), P)
    u = torch.einsum("jbc,jifca->jifba", ex.Ci, r).reshape(ex.ny, ex.nx, 3, n * n)
    return {"projected": u, "dt": ex.max_dt(u), "mass": ex.mass(u), "state": u}


def _exact_ensemble(case, seed):
    out = []
    for m, (nlon, nlat, d) in enumerate(zip(*_members(case, seed))):
        ex, u = _Exact(nlon, nlat, d), _sphere_state(nlon, nlat, d, seed + 1000 * m)
        for _ in range(case["steps"]):
            u = ex.step(u, _sphere_dt(nlon, nlat, d), 3)
        out.append(u)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "start":
        return _exact_start(case, seed)
    if kind == "ensemble":
        return _exact_ensemble(case, seed)
    if kind == "plane":
        ex, u, dt, rk = _Exact(case["nx"], case["ny"], case["degree"], True), _plane_state(case, seed), _plane_dt(case), case["rk"]
        for _ in range(case["steps"]):
            u = ex.step(u, dt, rk)
        return {"state": u}
    nlon, nlat, p = case["nlon"], case["nlat"], case.get("degree", 1)
    ex, u, dt, source = _Exact(nlon, nlat, p), _sphere_state(nlon, nlat, p, seed), _sphere_dt(nlon, nlat, p), None
    if kind == "learned":
        source = _source(ex, _network(seed), _learned_norm(u))
    if case.get("cfl"):
        dt = ex.max_dt(u)
    for _ in range(case["steps"]):
        u = ex.step(u, dt, case.get("rk", 3), source)
    out = {"state": u}
    if case.get("cfl"):
        out.update(dt=dt, mass=ex.mass(u))
    return out
