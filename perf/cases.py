"""The work that users of this framework have it do, as cases that can be timed and checked.

A case is one call of a public entry point of ``paper_1907_04839_gb300`` on synthetic
shape-like landmarks (``landmark_synth``): an ellipsoid surface and a copy of it deformed by
Gaussian bumps.  The momenta are those of a registration under way: the displacement to the
target divided by the kernel's row sum, with noise, so that the flow carries the template
most of the way.

``exact`` evaluates the same formulas in FP64 with torch alone:
    Hp_i = sum_j g_ij p_j,   Hq_i = -s sum_j c_ij g_ij d_ij,
    dalpha_i = s sum_j g_ij (c_ij e_ij - (u_ij + s c_ij e_ij.d_ij) d_ij),
    dbeta_i  = sum_j g_ij (alpha_j + s e_ij.d_ij p_j),
with g_ij = exp(-|d_ij|^2 / (2 sigma^2)), s = 1 / sigma^2, d = q_i - q_j, e = beta_i - beta_j,
c = p_i.p_j and u = alpha_i.p_j + alpha_j.p_i.
"""
import math

import numpy as np
import torch

import landmark_synth as ls
import paper_1907_04839_gb300 as gsh

LAMBDA = 10.0
#: |surface| of the ellipsoid with semi-axes 1.0 / 0.8 / 0.6, and the length of the ellipse 1.0 / 0.6
AREA, LENGTH = 7.9, 5.1


def listed():
    return [
        # one gradient of the smallest registration: 40 launches' latency and little else
        dict(name="gradient_256", kind="gradient", n=256, T=10, sigma=0.2),
        # the paper's own size (1847 landmarks, 40 steps), one gradient of its optimisation
        dict(name="gradient_1847", kind="gradient", n=1847, T=40, sigma=0.1),
        # the metric of the benchmark: 4096 landmarks, 20 steps
        dict(name="gradient_4096", kind="gradient", n=4096, T=20, sigma=0.1),
        # the differentiation workload: 16384 landmarks, 40 steps, a narrow kernel
        dict(name="gradient_16384", kind="gradient", n=16384, T=40, sigma=0.05),
        # a large served request, with the trajectory checkpointed every 8 steps
        dict(name="gradient_38785_ckpt", kind="gradient", n=38785, T=20, sigma=0.1, ckpt=8),
        # RK4 steps with the kinetic term at t = 1, a ragged size
        dict(name="gradient_rk4_3001", kind="gradient", n=3001, T=5, sigma=0.1, integrator="rk4", h_at="end"),
        # planar contours
        dict(name="gradient_planar_2000", kind="gradient", n=2000, T=20, sigma=0.05, dim=2),
        # a deformation applied: the forward flow alone
        dict(name="forward_5000", kind="forward", n=5000, T=20, sigma=0.1),
        # one adjoint pair sum for a caller with a time loop of its own
        dict(name="step_backward_3001", kind="step_backward", n=3001, sigma=0.05),
        # the velocity of a deformation on a 101^3 grid
        dict(name="velocity_grid_4096", kind="velocity", n=4096, m=1030301, sigma=0.1),
        # the first iterations of a small registration from host arrays: L-BFGS around small gradients
        dict(name="register_256", kind="register", n=256, T=10, sigma=0.2, iters=8),
        # a packed batch of registrations of mixed size and kernel width, the first iterations
        dict(name="batch_16", kind="batch", count=16, n_lo=500, n_hi=4000, T=20, iters=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gradient", "gradient", "gradient", "variant", "planar", "forward", "step_forward",
                       "step_backward", "velocity", "flow", "register", "batch"])
    sigma = rng.choice([0.05, 0.1, 0.2])
    T = rng.choice([5, 10, 20, 40])
    if kind == "gradient":
        c = dict(kind="gradient", n=_log(rng, 60, 20000), T=T, sigma=sigma)
        if rng.random() < 0.25:
            c["ckpt"] = rng.choice([2, 4, 8])
        return c
    if kind == "variant":
        integ, h_at = rng.choice([("rk4", "start"), ("rk4", "end"), ("euler", "end")])
        return dict(kind="gradient", n=_log(rng, 60, 10000), T=rng.choice([5, 10]), sigma=sigma, integrator=integ,
                    h_at=h_at)
    if kind == "planar":
        return dict(kind="gradient", n=_log(rng, 60, 10000), T=T, sigma=rng.choice([0.05, 0.1]), dim=2)
    if kind == "forward":
        return dict(kind="forward", n=_log(rng, 60, 20000), T=T, sigma=sigma)
    if kind in ("step_forward", "step_backward"):
        return dict(kind=kind, n=_log(rng, 60, 40000), sigma=sigma)
    if kind == "velocity":
        return dict(kind="velocity", n=_log(rng, 60, 10000), m=_log(rng, 1000, 1000000), sigma=sigma)
    if kind == "flow":
        return dict(kind="flow", n=_log(rng, 60, 5000), m=_log(rng, 1000, 200000), T=rng.choice([5, 10, 20]), sigma=sigma)
    if kind == "register":
        return dict(kind="register", n=_log(rng, 60, 3000), T=rng.choice([5, 10, 20]), sigma=rng.choice([0.1, 0.2]),
                    iters=rng.randint(3, 8))
    lo = _log(rng, 100, 1000)
    return dict(kind="batch", count=rng.randint(3, 24), n_lo=lo, n_hi=4 * lo, T=rng.choice([10, 20]), iters=rng.randint(2, 4))


def _shapes(case, seed):
    """(template, target, momenta) as float32 numpy arrays."""
    n, dim, sigma = case["n"], case.get("dim", 3), case["sigma"]
    if dim == 2:
        pr, rows = ls.ellipse_pair(n, seed=seed), 1.0 + n * math.sqrt(2.0 * math.pi) * sigma / LENGTH
    else:
        pr, rows = ls.ellipsoid_pair(n, seed=seed), 1.0 + n * 2.0 * math.pi * sigma ** 2 / AREA
    rng = np.random.default_rng((seed, 7))
    p0 = (pr.target - pr.q0) / rows
    p0 = p0 + rng.normal(0.0, 0.05 * math.sqrt(float(np.mean(p0 ** 2))), size=p0.shape)
    return [np.ascontiguousarray(x, dtype=np.float32) for x in (pr.q0, pr.target, p0)]


def _points(case, seed):
    """Query points: a regular grid around the shape when m is a cube, else points near the surface."""
    m = case["m"]
    side = round(m ** (1.0 / 3.0))
    if side ** 3 == m:
        rng = np.random.default_rng((seed, 9))
        g = [np.linspace(-1.2, 1.2, side) + o for o in rng.uniform(-0.01, 0.01, 3)]
        x = np.stack(np.meshgrid(*g, indexing="ij"), axis=-1).reshape(-1, 3)
    else:
        x = ls.ellipsoid_pair(m, seed=seed + 1, jitter=0.1).q0
    return np.ascontiguousarray(x, dtype=np.float32)


def _batch_sizes(case):
    """Sizes spread evenly over the logarithm, in an order that is not ascending."""
    ns = np.exp(np.linspace(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"]))
    return [int(round(x)) for x in np.concatenate([ns[::2], ns[1::2]])]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        rng = np.random.default_rng((seed, 11))
        s["problems"] = []
        for k, n in enumerate(_batch_sizes(case)):
            pr = ls.ellipsoid_pair(n, seed=int(rng.integers(1 << 30)))
            s["problems"].append(dict(q0=pr.q0.astype(np.float32), target=pr.target.astype(np.float32),
                                      sigma=(0.05, 0.1, 0.2)[k % 3], lam=LAMBDA))
        return s
    q0, target, p0 = _shapes(case, seed)
    if kind == "register":  # a user's arrays on the host
        s.update(q0=q0, target=target)
        return s
    put = lambda x: torch.from_numpy(x).to("cuda")  # noqa: E731
    s.update(q0=put(q0), target=put(target), p0=put(p0))
    if kind == "step_backward":  # the adjoint where the reverse sweep starts its last step
        s["alpha"] = 2.0 * LAMBDA * (s["q0"] - s["target"])
        s["beta"] = torch.from_numpy(np.random.default_rng((seed, 5)).normal(0.0, 0.5, size=p0.shape).astype(np.float32)).to("cuda") + s["alpha"]
    if kind in ("velocity", "flow"):
        s["x"] = put(_points(case, seed))
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "gradient":
        loss, gp, gq = gsh.shoot_gradient(s["q0"], s["p0"], s["target"], c["T"], c["sigma"], LAMBDA,
                                          ckpt_every=c.get("ckpt", 0), integrator=c.get("integrator", "euler"),
                                          h_at=c.get("h_at", "start"))
        return dict(loss=loss, grad_p0=gp, grad_q0=gq)
    if kind == "forward":
        q1, p1, h0 = gsh.shoot_forward(s["q0"], s["p0"], c["T"], c["sigma"])
        return dict(q1=q1, p1=p1, h0=h0)
    if kind == "step_forward":
        hq, hp = gsh.step_forward(s["q0"], s["p0"], c["sigma"])
        return dict(hq=hq, hp=hp)
    if kind == "step_backward":
        da, db = gsh.step_backward(s["q0"], s["p0"], s["alpha"], s["beta"], c["sigma"])
        return dict(dalpha=da, dbeta=db)
    if kind == "velocity":
        return dict(v=gsh.velocity_field(s["q0"], s["p0"], s["x"], c["sigma"]))
    if kind == "flow":
        return dict(x1=gsh.flow_points(s["q0"], s["p0"], s["x"], c["T"], c["sigma"]))
    if kind == "register":
        p0, info = gsh.register(s["q0"], s["target"], c["T"], c["sigma"], LAMBDA, max_iter=c["iters"], grad_tol=0.0)
        return dict(p0=p0, loss=info["loss"], avg_dist=info["avg_dist"])
    got = gsh.register_batch(s["problems"], c["T"], max_iter=c["iters"], grad_tol=0.0)
    return dict(p0=[p for p, _ in got], loss=np.array([i["loss"] for _, i in got], np.float32))


def work(case):
    """27 flops a pair for the forward sums and 63 for the adjoint (planar 18 and 42; the velocity alone 15), the exponential not counted."""
    kind, dim = case["kind"], case.get("dim", 3)
    fwd, bwd = (27.0, 63.0) if dim == 3 else (18.0, 42.0)
    if kind == "batch":
        ns = np.array(_batch_sizes(case), np.float64)
        evals = (case["iters"] + 1) * case["T"]
        return dict(bytes=float(3 * 12 * ns.sum()), flops=float(evals * (fwd + bwd) * (ns ** 2).sum()))
    n, arr = float(case["n"]), 4.0 * dim * case["n"]
    stages = case.get("T", 1) * (4 if case.get("integrator") == "rk4" else 1)
    if kind == "gradient":
        return dict(bytes=5 * arr, flops=(stages * (fwd + bwd) + (fwd if case.get("h_at") == "end" else 0.0)) * n * n)
    if kind == "forward":
        return dict(bytes=4 * arr, flops=stages * fwd * n * n)
    if kind == "step_forward":
        return dict(bytes=4 * arr, flops=fwd * n * n)
    if kind == "step_backward":
        return dict(bytes=6 * arr, flops=bwd * n * n)
    if kind == "velocity":
        return dict(bytes=2 * arr + 24.0 * case["m"], flops=15.0 * n * case["m"])
    if kind == "flow":
        return dict(bytes=2 * arr + 24.0 * case["m"], flops=stages * (15.0 * n * case["m"] + fwd * n * n))
    return dict(bytes=3 * arr, flops=(case["iters"] + 1) * stages * (fwd + bwd) * n * n)


# ---------------------------------------------------------------- FP64

ROWS = 1 << 26  # pairs evaluated at a time


def _chunks(m, n):
    k = max(1, ROWS // n)
    return [slice(i, min(i + k, m)) for i in range(0, m, k)]


def _kernel(x, q, sigma):
    d2 = torch.zeros((x.shape[0], q.shape[0]), dtype=torch.float64, device=q.device)
    for k in range(q.shape[1]):
        d2 += (x[:, k, None] - q[None, :, k]) ** 2
    return torch.exp_(d2.mul_(-0.5 / sigma ** 2))


def _ham(q, p, sigma):
    """(Hq, Hp)."""
    hq, hp = torch.empty_like(q), torch.empty_like(p)
    for r in _chunks(q.shape[0], q.shape[0]):
        g = _kernel(q[r], q, sigma)
        hp[r] = g @ p
        w = g.mul_(p[r] @ p.T)
        hq[r] = -(q[r] * w.sum(1, keepdim=True) - w @ q) / sigma ** 2
    return hq, hp


def _adjoint(q, p, a, b, sigma):
    """(dalpha, dbeta)."""
    s = 1.0 / sigma ** 2
    da, db = torch.empty_like(q), torch.empty_like(q)
    for r in _chunks(q.shape[0], q.shape[0]):
        g = _kernel(q[r], q, sigma)
        c = p[r] @ p.T
        u = a[r] @ p.T + p[r] @ a.T
        t = torch.zeros_like(g)
        for k in range(q.shape[1]):
            t += (b[r, k, None] - b[None, :, k]) * (q[r, k, None] - q[None, :, k])
        db[r] = g @ a + s * ((g * t) @ p)
        h = (u + s * c * t) * g
        c *= g
        da[r] = s * (b[r] * c.sum(1, keepdim=True) - c @ b - q[r] * h.sum(1, keepdim=True) + h @ q)
    return da, db


def _flow(q, p, T, sigma, rk4):
    """The states that the reverse sweep needs, and the end state."""
    dt, kept = 1.0 / T, []
    f = lambda y: (lambda h: (h[1], -h[0]))(_ham(y[0], y[1], sigma))  # noqa: E731
    at = lambda y, k, c: (y[0] + c * k[0], y[1] + c * k[1])  # noqa: E731
    y = (q, p)
    for _ in range(T):
        k1 = f(y)
        if not rk4:
            kept.append([y])
            y = at(y, k1, dt)
            continue
        y2 = at(y, k1, dt / 2)
        k2 = f(y2)
        y3 = at(y, k2, dt / 2)
        k3 = f(y3)
        y4 = at(y, k3, dt)
        k4 = f(y4)
        kept.append([y, y2, y3, y4])
        y = tuple(y[i] + dt / 6 * (k1[i] + 2 * k2[i] + 2 * k3[i] + k4[i]) for i in (0, 1))
    return kept, y


def _gradient(q0, p0, target, T, sigma, rk4, end):
    dt = 1.0 / T
    kept, (q1, p1) = _flow(q0, p0, T, sigma, rk4)
    w = (2 * LAMBDA * (q1 - target), torch.zeros_like(p0))
    loss = LAMBDA * ((q1 - target) ** 2).sum()
    hq, hp = _ham(q1, p1, sigma) if end else _ham(q0, p0, sigma)
    loss = loss + 0.5 * ((p1 if end else p0) * hp).sum()
    if end:
        w = (w[0] + hq, hp)
    back = lambda y, k: _adjoint(y[0], y[1], k[0], k[1], sigma)  # noqa: E731
    lin = lambda a, x, b, v: tuple(a * x[i] + b * v[i] for i in (0, 1))  # noqa: E731
    for ys in reversed(kept):
        if not rk4:
            w = lin(1.0, w, dt, back(ys[0], w))
            continue
        v4 = back(ys[3], lin(dt / 6, w, 0.0, w))
        v3 = back(ys[2], lin(dt / 3, w, dt, v4))
        v2 = back(ys[1], lin(dt / 3, w, dt / 2, v3))
        v1 = back(ys[0], lin(dt / 6, w, dt / 2, v2))
        w = tuple(w[i] + v1[i] + v2[i] + v3[i] + v4[i] for i in (0, 1))
    if end:
        return dict(loss=loss, grad_p0=w[1], grad_q0=w[0])
    return dict(loss=loss, grad_p0=w[1] + hp, grad_q0=w[0] + hq)


def _velocity(q, p, x, sigma):
    v = torch.empty_like(x)
    for r in _chunks(x.shape[0], q.shape[0]):
        v[r] = _kernel(x[r], q, sigma) @ p
    return v


def exact(case, seed):
    kind = case["kind"]
    if kind in ("register", "batch"):
        return None  # an optimisation's iterates
    stages = case.get("T", 1) * (4 if case.get("integrator") == "rk4" else 1)
    if stages * float(case["n"]) * case.get("m", case["n"]) > 2.5e10:
        return None  # more pairs than FP64 does in 20 seconds
    s = prepare(case, seed)
    d = {k: v.double() for k, v in s.items() if isinstance(v, torch.Tensor)}
    sigma, T = case["sigma"], case.get("T", 1)
    if kind == "gradient":
        return _gradient(d["q0"], d["p0"], d["target"], T, sigma, case.get("integrator") == "rk4", case.get("h_at") == "end")
    if kind == "forward":
        _, (q1, p1) = _flow(d["q0"], d["p0"], T, sigma, False)
        return dict(q1=q1, p1=p1, h0=0.5 * (d["p0"] * _ham(d["q0"], d["p0"], sigma)[1]).sum())
    if kind == "step_forward":
        hq, hp = _ham(d["q0"], d["p0"], sigma)
        return dict(hq=hq, hp=hp)
    if kind == "step_backward":
        da, db = _adjoint(d["q0"], d["p0"], d["alpha"], d["beta"], sigma)
        return dict(dalpha=da, dbeta=db)
    if kind == "velocity":
        return dict(v=_velocity(d["q0"], d["p0"], d["x"], sigma))
    kept, _ = _flow(d["q0"], d["p0"], T, sigma, False)
    x = d["x"]
    for (y,) in kept:
        x = x + _velocity(y[0], y[1], x, sigma) / T
    return dict(x1=x)
