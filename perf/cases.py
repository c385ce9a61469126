"""Performance cases of the solver: the calls a user makes, over the sizes they are made at.

Every case goes through the public Python API (binding.Solver, binding.Batch, autograd.rollout).
A pass starts from the same seeded state each time, as one evaluation of a rollout, a gradient
or a training window does, and returns everything it computes: states, step sizes, adjoints,
parameter and weight gradients.

`exact` is an independent plain-torch FP64 statement of the same equations (WENO5 of the
primitive variables, HLLC, Navier-Stokes fluxes, ghost-cell immersed body, SSP-RK3, the neural
flux), differentiated by torch's autograd.  It shares nothing with the package but the inputs.
"""
import math

import numpy as np
import torch

from paper_2601_04400_gb300 import autograd as A
from paper_2601_04400_gb300 import binding as B
from paper_2601_04400_gb300 import inverse as I
from paper_2601_04400_gb300 import neural as N
from paper_2601_04400_gb300 import workloads as W

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # 1D shock tube at the paper's 200 cells: the smallest call, bound by launches
        dict(name="sod_200", do="steps", flow="sod", nx=200, ny=1, steps=10),
        # small viscous body flow (parameter studies, tests, gradient checks)
        dict(name="cylinder_128x64", do="steps", flow="cylinder", nx=128, ny=64, steps=10),
        # the right-hand side alone, odd sizes, viscosity and artificial viscosity (a caller with
        # its own time integrator)
        dict(name="rhs_periodic_701x517", do="rhs", flow="periodic", nx=701, ny=517),
        # four-quadrant Riemann problem at the throughput size, device CFL steps
        dict(name="riemann_1024", do="steps", flow="riemann", nx=1024, ny=1024, steps=2),
        # the benchmark: viscous Mach-2 shock over the immersed cylinder
        dict(name="cylinder_2048x1024", do="steps", flow="cylinder", nx=2048, ny=1024, steps=1),
        # the paper's largest run, Mach-5 Euler on its odd-sized 8.4e6-cell grid, given step size
        dict(name="mach5_4347x1932", do="fixed", flow="mach5", nx=4347, ny=1932, steps=1),
        # reverse of one step at the adjoint configuration's grid
        dict(name="vjp_512", do="vjp", flow="cylinder", nx=512, ny=512),
        # gradient of a multi-step loss through a checkpointed rollout (parameter recovery)
        dict(name="rollout_grad_250x190", do="rollout", flow="cylinder", nx=250, ny=190, steps=6),
        # a batch of uneven shock-cylinder instances, forward (an eighth of the 256-instance sweep)
        dict(name="batch_32", do="batch", count=32, mix=0, steps=2),
        # one reverse step of such a batch
        dict(name="batch_vjp_16", do="batch_vjp", count=16, mix=1, split=1),
        # a solver step with the trained flux correction, BF16 network
        dict(name="neural_bf16_1024", do="neural", flow="riemann", nx=1024, ny=1024, steps=1, precision="bf16"),
        # one training window of the neural flux on a coarse grid, FP32 network
        dict(name="neural_train_128x96", do="train", flow="periodic", nx=128, ny=96, steps=4),
    ]


def _size(rng, lo, hi):
    """A cell count along one axis, spread over the logarithm; odd ones as often as even ones."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["steps", "steps", "steps", "fixed", "rhs", "vjp", "vjp", "rollout", "batch", "batch_vjp", "neural",
                     "train"])
    if do == "batch":
        return dict(do=do, count=rng.randint(4, 32), mix=rng.randint(2, 10 ** 6), steps=rng.randint(1, 3))
    if do == "batch_vjp":
        return dict(do=do, count=rng.randint(2, 16), mix=rng.randint(2, 10 ** 6), split=rng.randint(0, 1))
    if do == "vjp":
        return dict(do=do, flow=rng.choice(["cylinder", "riemann", "periodic"]), nx=_size(rng, 64, 900),
                    ny=_size(rng, 64, 600))
    if do == "rollout":
        return dict(do=do, flow=rng.choice(["cylinder", "riemann"]), nx=_size(rng, 64, 300), ny=_size(rng, 64, 200),
                    steps=rng.randint(2, 6))
    if do == "train":
        return dict(do=do, flow="periodic", nx=_size(rng, 48, 160), ny=_size(rng, 48, 120), steps=rng.randint(2, 5))
    if do == "neural":
        return dict(do=do, flow=rng.choice(["riemann", "periodic"]), nx=_size(rng, 96, 1100), ny=_size(rng, 96, 1000),
                    steps=1, precision=rng.choice(["bf16", "fp32"]))
    flow = rng.choice(["sod", "cylinder", "riemann", "periodic"])
    if do == "rhs":
        flow = rng.choice(["cylinder", "riemann", "periodic"])
    if flow == "sod":
        return dict(do="steps", flow=flow, nx=_size(rng, 64, 4000), ny=1, steps=rng.randint(2, 12))
    nx, ny = _size(rng, 72, 2600), _size(rng, 64, 1400)
    if do == "rhs":
        return dict(do=do, flow=flow, nx=nx, ny=ny)
    return dict(do=do, flow=flow, nx=nx, ny=ny, steps=max(1, min(8, 2000000 // (nx * ny))))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _problem(flow, nx, ny):
    if flow == "sod":
        return W.sod(nx)
    if flow == "riemann":
        return W.riemann2d(nx, ny=ny)
    if flow == "mach5":
        return W.mach5_cylinder(nx, ny)
    if flow == "cylinder":
        return W.shock_cylinder(nx=nx, ny=ny)
    return W.random_periodic(nx, ny, seed=3, mu=2e-3, nu=1e-3)


def _gen(seed):
    return torch.Generator().manual_seed(int(seed))


def _modes(gen, ny, nx, n=6):
    """A smooth seeded field of unit order on the grid."""
    f = torch.zeros(ny, nx, dtype=F64, device=DEV)
    x = (torch.arange(nx, dtype=F64, device=DEV) + 0.5) / nx
    y = (torch.arange(ny, dtype=F64, device=DEV) + 0.5) / ny
    for _ in range(n):
        kx, ky = (int(v) for v in torch.randint(1, 9, (2,), generator=gen))
        a, ph = (float(v) for v in torch.rand(2, generator=gen, dtype=F64))
        ay = 2 * math.pi * (ky * y + ph) if ny > 1 else torch.zeros_like(y)
        f += (0.2 + 0.8 * a) * torch.sin(2 * math.pi * kx * x[None, :] + ay[:, None] + 6.0 * ph)
    return f / n


def _state(prob, gen, amp=0.06):
    """Primitive state: the problem's initial condition with a seeded smooth disturbance; gas at
    rest ahead of a shock stays at rest, as it does until the shock arrives."""
    w = torch.as_tensor(prob.W0, device=DEV).clone()
    ny, nx = w.shape[1:]
    on = (w[1].abs() + w[2].abs() > 0).to(F64) if "x_shock" in prob.meta else torch.ones(ny, nx, dtype=F64, device=DEV)
    w[0] *= 1.0 + amp * on * _modes(gen, ny, nx)
    w[1] += amp * on * _modes(gen, ny, nx)
    if ny > 1:
        w[2] += amp * on * _modes(gen, ny, nx)
    w[3] *= 1.0 + amp * on * _modes(gen, ny, nx)
    return w


def _cons(w, gamma):
    """Conserved state of a primitive one."""
    return torch.stack([w[0], w[0] * w[1], w[0] * w[2], w[3] / (gamma - 1.0) + 0.5 * w[0] * (w[1] ** 2 + w[2] ** 2)])


def _weights(gen):
    """Network parameters of a trained size: He-uniform ReLU layers, a small output layer."""
    w = torch.zeros(B.JS_NN_NPARAM, dtype=F64)
    for k, (cin, cout, off) in enumerate(N.LAYERS):
        n = cout * cin * 9
        w[off:off + n] = (torch.rand(n, generator=gen, dtype=F64) * 2 - 1) * math.sqrt(6.0 / (cin * 9)) * (0.2 if k == 2 else 1)
        w[off + n:off + n + cout] = 0.05 * (torch.rand(cout, generator=gen, dtype=F64) * 2 - 1)
    return w.to(DEV)


def prepare(case, seed):
    gen = _gen(seed)
    do = case["do"]
    if do in ("batch", "batch_vjp"):
        return _prepare_batch(case, gen)
    prob = _problem(case["flow"], case["nx"], case["ny"])
    s = B.Solver.from_problem(prob)
    U0 = _cons(_state(prob, gen), prob.gamma).contiguous()
    st = dict(case=case, do=do, prob=prob, solver=s, U0=U0, cfl=prob.cfl)
    n = case.get("steps", 1)
    if do == "steps":
        st.update(U=U0.clone(), dts=torch.zeros(n, dtype=F64, device=DEV))
    elif do == "rhs":
        st.update(out=torch.empty_like(U0))
    else:
        st["dt"] = 0.8 * s.max_dt(U0, prob.cfl)
    if do in ("fixed", "neural"):
        st["U"] = U0.clone()
    if do in ("neural", "train"):
        st["w"] = _weights(gen)
        st["norm"] = N.frame_norm(U0, scale=0.02)
    if do == "neural":
        s.set_neural(st["w"], st["norm"], precision=case["precision"])
    if do == "vjp":
        st["lam"] = torch.randn(U0.shape, generator=gen, dtype=F64).to(DEV)
        st["lam_n"] = torch.empty_like(U0)
        st["p_bar"] = torch.zeros(B.JS_NPARAM, dtype=F64, device=DEV)
    if do in ("rollout", "train"):
        st["theta"] = A.theta_of(s)
        st["outputs"] = list(range(1, n + 1))
        st["targets"] = torch.stack([U0 * (1.0 + 0.01 * _modes(gen, *U0.shape[1:])) for _ in range(n)])
    return st


def _prepare_batch(case, gen):
    probs = W.batched_cases(case["count"], seed=case["mix"])
    b = B.Batch(probs)
    U0 = [_cons(_state(p, gen), p.gamma).contiguous() for p in probs]
    st = dict(case=case, do=case["do"], probs=probs, batch=b, U0=U0, cfl=0.5)
    if case["do"] == "batch":
        st.update(U=[u.clone() for u in U0], dts=torch.zeros(case["steps"], len(probs), dtype=F64, device=DEV))
        st["t"] = torch.zeros(len(probs), dtype=F64, device=DEV)
        b.set_states(st["U"])
    else:
        b.set_states(U0)
        b.set_reverse_launch(case["split"])
        st["dt"] = [0.4 * p.cfl * min(p.dx, p.dy) / (1.0 + p.meta["mach"]) for p in probs]
        st["lam"] = [torch.randn(u.shape, generator=gen, dtype=F64).to(DEV) for u in U0]
        st["lam_n"] = [torch.empty_like(u) for u in U0]
        st["p_bar"] = [torch.zeros(B.JS_NPARAM, dtype=F64, device=DEV) for _ in U0]
    return st


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def run(st):
    do = st["do"]
    if do == "steps":
        st["U"].copy_(st["U0"])
        st["solver"].step_cfl(st["U"], st["cfl"], st["case"]["steps"], dt_log=st["dts"])
        return {"U": st["U"], "dt": st["dts"]}
    if do in ("fixed", "neural"):
        st["U"].copy_(st["U0"])
        return {"U": st["solver"].step(st["U"], st["dt"], st["case"]["steps"])}
    if do == "rhs":
        return {"L": st["solver"].rhs(st["U0"], st["out"])}
    if do == "vjp":
        st["p_bar"].zero_()
        lam, pb = st["solver"].step_vjp(st["U0"], st["dt"], st["lam"], st["lam_n"], st["p_bar"])
        return {"lam": lam, "p_bar": pb}
    if do in ("rollout", "train"):
        U0 = st["U0"].detach().requires_grad_(True)
        theta = st["theta"].detach().requires_grad_(True)
        w = st["w"].detach().requires_grad_(True) if do == "train" else None
        states = A.rollout(st["solver"], U0, theta, [st["dt"]] * st["case"]["steps"], outputs=st["outputs"],
                           weights=w, norm=st.get("norm"), fp32=do == "train")
        loss = I.multistep_loss(states, st["targets"])
        g = torch.autograd.grad(loss, [U0, theta] + ([w] if w is not None else []))
        out = {"states": states.detach(), "gU": g[0], "gtheta": g[1]}
        if w is not None:
            out["gw"] = g[2]
        return out
    if do == "batch":
        torch._foreach_copy_(st["U"], st["U0"])
        st["t"].zero_()
        st["batch"].step(st["cfl"], st["case"]["steps"], st["t"], st["dts"])
        return {"U": st["U"], "dt": st["dts"], "t": st["t"]}
    torch._foreach_zero_(st["p_bar"])
    st["batch"].step_vjp(st["U0"], st["dt"], st["lam"], st["lam_n"], st["p_bar"])
    return {"lam": st["lam_n"], "p_bar": st["p_bar"]}


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------
# FP64 operations of one cell in one stage (add, multiply, divide, square root each 1; every face
# once), counted on the plain formulation: Euler and Navier-Stokes in 2D; 1D has one direction
EULER, VISCOUS, ONE_D = 1281, 1357, 660
NETWORK = 25344  # multiply-adds x 2 of the neural flux per cell and stage (two faces)


def work(case):
    do = case["do"]
    if do in ("batch", "batch_vjp"):
        cells = sum(p.nx * p.ny for p in _batch_sizes(case))
        per, flow = VISCOUS, "cylinder"
    else:
        cells, flow = case["nx"] * case["ny"], case["flow"]
        per = ONE_D if case["ny"] == 1 else VISCOUS if flow in ("cylinder", "periodic") else EULER
    n = case.get("steps", 1)
    if do == "rhs":
        return {"bytes": 64 * cells, "flops": per * cells}
    if do in ("steps", "fixed", "batch"):
        return {"bytes": 64 * cells, "flops": 3 * n * per * cells}
    if do == "neural":
        return {"bytes": 64 * cells, "flops": 3 * n * (per + NETWORK) * cells}
    if do in ("vjp", "batch_vjp"):
        # two stage states recomputed, three stages reversed (a reverse is twice its forward)
        return {"bytes": 96 * cells, "flops": (2 + 6) * per * cells}
    both = per + (NETWORK if do == "train" else 0)
    return {"bytes": (64 * (n + 1) + 32) * cells, "flops": 3 * n * 3 * both * cells}


def _batch_sizes(case):
    """Grid sizes of a batch (its states are not built)."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["count"]):
        nx, ny = int(rng.choice(tuple(range(128, 513, 64)))), int(rng.choice((128, 192, 256)))
        rng.uniform(1.5, 3.0), rng.uniform(0.3, 0.7)
        out.append(W.Problem("size", nx, ny, 0.0, 0.0, 1.0, 1.0))
    return out


# ---------------------------------------------------------------------------------------
# the same results in plain torch
# ---------------------------------------------------------------------------------------
def _weno(a, b, c, d, e):
    b0 = 13.0 / 12.0 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    b1 = 13.0 / 12.0 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    b2 = 13.0 / 12.0 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    a0, a1, a2 = 0.1 / (1e-6 + b0) ** 2, 0.6 / (1e-6 + b1) ** 2, 0.3 / (1e-6 + b2) ** 2
    p0, p1, p2 = (2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6
    return (a0 * p0 + a1 * p1 + a2 * p2) / (a0 + a1 + a2)


def _hllc(L, R, gamma):
    """Flux of face states (rho, normal velocity, tangential velocity, p)."""
    def energy(q):
        return q[3] / (gamma - 1.0) + 0.5 * q[0] * (q[1] ** 2 + q[2] ** 2)

    aL, aR = torch.sqrt(gamma * L[3] / L[0]), torch.sqrt(gamma * R[3] / R[0])
    xL, xR, zL, zR = L[1] - aL, R[1] - aR, L[1] + aL, R[1] + aR
    sL, sR = torch.where(xR < xL, xR, xL), torch.where(zL < zR, zR, zL)
    mL, mR = L[0] * (sL - L[1]), R[0] * (sR - R[1])
    ss = (R[3] - L[3] + L[1] * mL - R[1] * mR) / (mL - mR)

    def branch(q, s, m, spm):
        E = energy(q)
        rs = m / (s - ss)
        Es = (s - q[1]) / (s - ss) * (E + (ss - q[1]) * (q[0] * ss + q[3] / (s - q[1])))
        mom = q[0] * q[1]
        return torch.stack([mom + spm * (rs - q[0]), mom * q[1] + q[3] + spm * (rs * ss - mom),
                            mom * q[2] + spm * (rs * q[2] - q[0] * q[2]), (E + q[3]) * q[1] + spm * (Es - E)])

    zero = torch.zeros_like(ss)
    FL = branch(L, sL, mL, torch.where(sL < 0, sL, zero))
    FR = branch(R, sR, mR, torch.where(sR > 0, sR, zero))
    return torch.where(ss > 0, FL, torch.where(ss < 0, FR, 0.5 * (FL + FR)))


def _ib(prob):
    """Immersed body: fluid mask, and per ghost cell its flat index, four interpolation cells,
    their weights and the wall normal (flat indices into [ny, nx])."""
    if prob.sdf is None:
        return None
    sdf = np.asarray(prob.sdf)
    ny, nx = sdf.shape
    solid = sdf < 0.0
    pad = np.zeros((ny + 6, nx + 6), bool)
    pad[3:-3, 3:-3] = ~solid
    near = np.zeros_like(solid)
    for b in range(7):
        for a in range(7):
            near |= pad[b:b + ny, a:a + nx]
    j, i = np.nonzero(solid & near)
    il, ir, jl, jr = np.maximum(i - 1, 0), np.minimum(i + 1, nx - 1), np.maximum(j - 1, 0), np.minimum(j + 1, ny - 1)
    gx = (sdf[j, ir] - sdf[j, il]) / ((ir - il) * prob.dx)
    gy = (sdf[jr, i] - sdf[jl, i]) / ((jr - jl) * prob.dy)
    gn = np.sqrt(gx * gx + gy * gy)
    n = np.stack([gx / gn, gy / gn])
    phi = sdf[j, i]
    fx = (prob.x0 + (i + 0.5) * prob.dx - 2 * phi * n[0] - prob.x0) / prob.dx - 0.5
    fy = (prob.y0 + (j + 0.5) * prob.dy - 2 * phi * n[1] - prob.y0) / prob.dy - 0.5
    i0 = np.clip(np.floor(fx).astype(int), 0, nx - 2)
    j0 = np.clip(np.floor(fy).astype(int), 0, ny - 2)
    tx, ty = fx - i0, fy - j0
    src = np.stack([j0 * nx + i0, j0 * nx + i0 + 1, (j0 + 1) * nx + i0, (j0 + 1) * nx + i0 + 1])
    w = np.stack([(1 - tx) * (1 - ty), tx * (1 - ty), (1 - tx) * ty, tx * ty]) * ~solid.reshape(-1)[src]
    w = w / w.sum(0)
    t = lambda v: torch.as_tensor(v, device=DEV)  # noqa: E731
    return dict(fluid=t(~solid), dst=t(j * nx + i), src=t(src), w=t(w), n=t(n))


def _pad(X, kinds, inflow, axis):
    """Three ghost layers on both sides of an axis (2: x, 1: y) of a conserved state."""
    n, mom = X.shape[axis], 1 if axis == 2 else 2
    k0 = 0 if axis == 2 else 2
    idx = {0: ([0] * 3, [n - 1] * 3), 1: ([2, 1, 0], [n - 1, n - 2, n - 3]), 2: ([n - 3, n - 2, n - 1], [0, 1, 2])}
    flip = torch.ones(4, 1, 1, dtype=F64, device=DEV)
    flip[mom] = -1.0
    parts = []
    for side in (0, 1):
        kind = kinds[k0 + side]
        shape = [4, X.shape[1], X.shape[2]]
        shape[axis] = 3
        if kind == 3:
            parts.append(inflow[k0 + side].view(4, 1, 1).expand(shape))
        else:
            g = X.index_select(axis, torch.tensor(idx[kind][side], device=DEV))
            parts.append(g * flip if kind == 1 else g)
    return torch.cat([parts[0], X, parts[1]], dim=axis)


def _network(X, w):
    """Three 3x3 layers with zero padding on one image [4, H, W]."""
    for k, (cin, cout, off) in enumerate(N.LAYERS):
        n = cout * cin * 9
        X = torch.nn.functional.conv2d(X[None], w[off:off + n].view(cout, cin, 3, 3), w[off + n:off + n + cout], padding=1)[0]
        X = torch.tanh(X) if k == 2 else torch.relu(X)
    return X


class _Exact:
    """The solver's step on one grid: theta = (gamma, mu, Pr, nu, inflow states)."""

    def __init__(self, prob, theta=None, w=None, norm=None):
        self.p, self.ib = prob, _ib(prob)
        self.th = torch.as_tensor(prob.theta(), device=DEV) if theta is None else theta
        self.w = w
        self.norm = None if norm is None else torch.as_tensor(norm, device=DEV).view(3, 4, 1, 1)
        q = self.th[4:].view(4, 4)
        self.inflow = [torch.stack([r[0], r[0] * r[1], r[0] * r[2],
                                    r[3] / (self.th[0] - 1.0) + 0.5 * r[0] * (r[1] ** 2 + r[2] ** 2)]) for r in q]

    def prim(self, U):
        u, v = U[1] / U[0], U[2] / U[0]
        return torch.stack([U[0], u, v, (self.th[0] - 1.0) * (U[3] - 0.5 * U[0] * (u * u + v * v))])

    def fill(self, U):
        if self.ib is None:
            return U
        f = U.reshape(4, -1)
        b = self.ib
        q = (self.prim(f[:, b["src"].reshape(-1)]).view(4, 4, -1) * b["w"]).sum(1)
        vn = q[1] * b["n"][0] + q[2] * b["n"][1]
        u, v = q[1] - 2 * vn * b["n"][0], q[2] - 2 * vn * b["n"][1]
        g = torch.stack([q[0], q[0] * u, q[0] * v, q[3] / (self.th[0] - 1.0) + 0.5 * q[0] * (u * u + v * v)])
        return f.index_copy(1, b["dst"], g).view_as(U)

    def direction(self, Q, d):
        """Face fluxes along x (d = 0) or y (d = 1), y transposed so that the line is the last axis."""
        p, th = self.p, self.th
        gy = 3 if p.ny > 1 else 0
        q = Q if d == 0 else Q.transpose(1, 2)[[0, 2, 1, 3]]
        full, cut = q, q[:, gy:-gy] if gy or d else q
        if d == 1:
            cut = q[:, 3:-3]
        hn, ht = (p.dx, p.dy) if d == 0 else (p.dy, p.dx)
        m = cut.shape[2] - 6  # cells; faces 0 .. m
        c = [cut[:, :, k:k + m + 1] for k in range(6)]
        L, R = _weno(*c[:5]), _weno(*c[:0:-1])
        net = None
        if self.w is not None:
            mean = 0.5 * (_cons(L, th[0]) + _cons(R, th[0]))
            net = self.norm[2] * _network((mean - self.norm[0]) / self.norm[1], self.w)
        ok = (L[0] > 0) & (L[3] > 0) & (R[0] > 0) & (R[3] > 0)
        F = _hllc(torch.where(ok, L, c[2]), torch.where(ok, R, c[3]), th[0])
        if p.mu > 0:
            lo, hi = c[2], c[3]
            dn = (hi - lo) / hn
            dT = (hi[3] / hi[0] - lo[3] / lo[0]) / hn
            unt = utt = 0.0
            if p.ny > 1:
                up, dn_ = full[:, 4:-2] if d == 0 else full[:, 4:-2], full[:, 2:-4]
                diff = up - dn_
                s = diff[:, :, 2:2 + m + 1] + diff[:, :, 3:3 + m + 1]
                unt, utt = s[1] / (4 * ht), s[2] / (4 * ht)
            tnn = th[1] * (4.0 / 3.0 * dn[1] - 2.0 / 3.0 * utt)
            tnt = th[1] * (dn[2] + unt)
            kap = th[1] * th[0] / ((th[0] - 1.0) * th[2])
            e = 0.5 * (lo[1] + hi[1]) * tnn + 0.5 * (lo[2] + hi[2]) * tnt + kap * dT
            F = F - torch.stack([torch.zeros_like(e), tnn, tnt, e])
        if net is not None:
            F = F + net
        D = (F[:, :, 1:] - F[:, :, :-1]) / hn
        return D if d == 0 else D[[0, 2, 1, 3]].transpose(1, 2)

    def rhs(self, U):
        """L(U) of a filled state (zero in the body)."""
        p = self.p
        X = _pad(U, p.bc, self.inflow, 2)
        if p.ny > 1:
            X = _pad(X, p.bc, self.inflow, 1)
        Q = self.prim(X)
        out = -self.direction(Q, 0)
        if p.ny > 1:
            out = out - self.direction(Q, 1)
        if p.nu > 0:
            g = 3 if p.ny > 1 else 0
            Y = X[:, g:-g] if g else X
            lap = (Y[:, :, 4:-2] - 2 * U + Y[:, :, 2:-4]) / p.dx ** 2
            if g:
                Z = X[:, :, 3:-3]
                lap = lap + (Z[:, 4:-2] - 2 * U + Z[:, 2:-4]) / p.dy ** 2
            out = out + self.th[3] * lap
        return out if self.ib is None else torch.where(self.ib["fluid"], out, torch.zeros_like(out))

    def step(self, U, dt):
        X, a, b = U, (0.0, 0.75, 1.0 / 3.0), (1.0, 0.25, 2.0 / 3.0)
        for k in range(3):
            X = self.fill(X)
            Y = b[k] * (X + dt * self.rhs(X)) + (a[k] * U if k else 0.0)
            X = Y if self.ib is None else torch.where(self.ib["fluid"], Y, X)
        return X

    def dt(self, U, cfl):
        p, q = self.p, self.prim(U)
        a = torch.sqrt(self.th[0] * q[3] / q[0])
        rate = (q[1].abs() + a) / p.dx
        if p.ny > 1:
            rate = rate + (q[2].abs() + a) / p.dy
        on = torch.ones_like(rate, dtype=torch.bool) if self.ib is None else self.ib["fluid"]
        dt = cfl / rate[on].max()
        if p.mu > 0:
            h = min(p.dx, p.dy) if p.ny > 1 else p.dx
            dt = torch.minimum(dt, cfl * h * h * q[0][on].min() / (2 * p.mu * max(4.0 / 3.0, p.gamma / p.Pr)))
        return dt

    def run(self, U, cfl, n):
        dts = []
        for _ in range(n):
            dts.append(self.dt(U, cfl))
            U = self.step(U, dts[-1])
        return U, torch.stack(dts)


def _exact_vjp(prob, U0, dt, lam):
    """Adjoints of one step by autograd, with the parameter entries the solver reports."""
    U = U0.clone().requires_grad_(True)
    th = torch.as_tensor(prob.theta(), device=DEV).requires_grad_(True)
    gU, gt = torch.autograd.grad(_Exact(prob, th).step(U, dt), (U, th), grad_outputs=lam, allow_unused=True)
    return gU, _theta_entries(prob, gt)


def _theta_entries(prob, g):
    """The gradient entries the solver forms: mu and Pr with viscosity, nu with artificial
    viscosity, inflow states of inflow sides."""
    g = g.clone()
    if not prob.mu > 0:
        g[1:3] = 0.0
    if not prob.nu > 0:
        g[3] = 0.0
    return g


def exact(case, seed):
    do = case["do"]
    cells = 0 if "nx" not in case else case["nx"] * case["ny"]
    if do == "vjp" and cells > 400000:
        return None  # autograd's saved tensors would take a large part of the card
    st = prepare(case, seed)
    if do in ("batch", "batch_vjp"):
        if do == "batch":
            r = [_Exact(p).run(u, st["cfl"], case["steps"]) for p, u in zip(st["probs"], st["U0"])]
            dts = torch.stack([d for _, d in r], dim=1)
            return {"U": [u for u, _ in r], "dt": dts, "t": dts.sum(0)}
        r = [_exact_vjp(p, u, dt, lam) for p, u, dt, lam in zip(st["probs"], st["U0"], st["dt"], st["lam"])]
        return {"lam": [a for a, _ in r], "p_bar": [b for _, b in r]}
    prob, U0 = st["prob"], st["U0"]
    if do == "steps":
        U, dts = _Exact(prob).run(U0, st["cfl"], case["steps"])
        return {"U": U, "dt": dts}
    if do in ("fixed", "neural"):
        e, U = _Exact(prob, w=st.get("w"), norm=st["norm"].reshape(3, 4) if do == "neural" else None), U0
        for _ in range(case["steps"]):
            U = e.step(U, st["dt"])
        return {"U": U}
    if do == "rhs":
        e = _Exact(prob)
        return {"L": e.rhs(e.fill(U0))}
    if do == "vjp":
        lam, pb = _exact_vjp(prob, U0, st["dt"], st["lam"])
        return {"lam": lam, "p_bar": pb}
    U = U0.clone().requires_grad_(True)
    th = torch.as_tensor(prob.theta(), device=DEV).requires_grad_(True)
    w = st["w"].clone().requires_grad_(True) if do == "train" else None
    e = _Exact(prob, th, w, None if w is None else st["norm"].reshape(3, 4))
    states, X = [], U
    for _ in range(case["steps"]):
        X = e.step(X, st["dt"])
        states.append(X)
    states = torch.stack(states)
    loss = ((states - st["targets"]) ** 2).sum() / case["steps"]
    g = torch.autograd.grad(loss, [U, th] + ([w] if w is not None else []))
    out = {"states": states.detach(), "gU": g[0], "gtheta": _theta_entries(prob, g[1]).cpu()}
    if w is not None:
        out["gw"] = g[2]
    return out
