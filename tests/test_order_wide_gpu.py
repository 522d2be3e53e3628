"""Ordered sweeps where nearly all pairs are in reach (the culling kernels stream
every source and grow no boxes), against the same sweeps in the caller's order
with every pair evaluated; and register over ordered sweeps.

The bar is that of the narrow kernels (test_order_gpu.py): 2e-6 normwise for
the FP32 sums, and the rounding of a prescaled position to FP32, which moves a
Gaussian by up to 2^-24 |q~|.
"""
import numpy as np
import pytest

import landmark_synth as ls

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def gs():
    import paper_1907_04839_gb300 as m
    return m


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


def put(*arrays):
    return [torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda") for a in arrays]


def every_pair(fn):
    lib = gs().load()
    gs().check(lib.gs_set_step_config(0, 128, 1, 1, 8))
    gs().check(lib.gs_set_step_config(1, 64, 1, 1, 8))
    try:
        return fn()
    finally:
        lib.gs_set_step_config(0, 0, 0, 0, 0)
        lib.gs_set_step_config(1, 0, 0, 0, 0)


@pytest.mark.parametrize("n,dim,T,sigma,kw", [
    (5001, 3, 40, 0.2, {}),
    (16385, 3, 8, 0.2, {}),
    (11201, 3, 9, 0.2, {"ckpt_every": 4}),
    (8255, 3, 4, 0.2, {"integrator": "rk4", "h_at": "end"}),
    (12000, 2, 8, 0.2, {}),
    (9001, 2, 4, 0.2, {"integrator": "rk4", "ckpt_every": 3}),
    (12001, 3, 8, 0.1, {}),   # between the two
])
def test_wide_ordered_gradient_equals_every_pair(n, dim, T, sigma, kw):
    pr = ls.ellipse_pair(n, seed=2) if dim == 2 else ls.ellipsoid_pair(n, seed=2)
    q, p, t = put(pr.q0, np.random.default_rng(n).normal(0.0, 2.0 / n, size=(n, dim)), pr.target)
    run = lambda: gs().shoot_gradient(q, p, t, T, sigma, 10.0, **kw)  # noqa: E731
    a, b = run(), every_pair(run)
    e = abs(a[0] - b[0]) / abs(b[0]), rel(a[1], b[1]), rel(a[2], b[2])
    print("N=%d dim %d sigma %g: loss %.2e grad_p0 %.2e grad_q0 %.2e" % ((n, dim, sigma) + e))
    assert max(e) < 2e-6 + 2.0 ** -24 * float(q.abs().max()) * 0.85 / sigma


@pytest.mark.parametrize("sigma", [0.05, 0.2])
def test_register_distances_over_ordered_sweeps(sigma):
    """avg_dist and max_dist pair each landmark's end with its own target (a
    wrong pairing would give distances of the shape's size, about 1).  The
    momenta come back rounded to FP32 and flow in another order: positions agree
    to the bar above, and so do distances."""
    n, T = 10300, 10
    pr = ls.ellipsoid_pair(n, seed=7)
    q, t = put(pr.q0, pr.target)
    p0, info = gs().register(q, t, T, sigma, 10.0, max_iter=2, grad_tol=0.0)
    q1, _, _ = gs().shoot_forward(q, p0, T, sigma)
    d = (q1.double() - t.double()).norm(dim=1)
    bar = 2e-6 + 2.0 ** -24 * float(q.abs().max()) * 0.85 / sigma
    print("sigma=%g avg %.6g / %.6g max %.6g / %.6g" % (sigma, info["avg_dist"], d.mean(), info["max_dist"], d.max()))
    assert info["evals"] >= 2 and 0.0 < info["avg_dist"] < 0.5
    assert abs(info["avg_dist"] - float(d.mean())) < bar and abs(info["max_dist"] - float(d.max())) < bar
