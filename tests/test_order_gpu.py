"""Ordered sweeps (of 8 evaluations and 10^9 pairs and more: landmarks packed along a space-filling
curve, runs of sources whose Gaussian is exactly zero left out) against
the same sweeps with every pair evaluated, which a launch-shape override selects.

Both sum the same non-zero FP32 terms in another order, so each result carries
the rounding of its FP32 sums: sqrt(128) 2^-24 = 7e-7 of the terms' size per
128-source block, less over the many blocks of a sum: 2e-6 normwise.  After the
first step the two states differ in their last bits, so a prescaled position
q~ may round to the neighbouring FP32 value, which moves a Gaussian by up to
2^-24 |q~| more.
"""
import numpy as np
import pytest

import landmark_synth as ls

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BAR = 2e-6


def gs():
    import paper_1907_04839_gb300 as m
    return m


def rel(a, b):
    a, b = (x.double().cpu().numpy().ravel() for x in (a, b))
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def every_pair(fn):
    lib = gs().load()
    gs().check(lib.gs_set_step_config(0, 128, 1, 1, 8))
    gs().check(lib.gs_set_step_config(1, 64, 1, 1, 8))
    try:
        return fn()
    finally:
        lib.gs_set_step_config(0, 0, 0, 0, 0)
        lib.gs_set_step_config(1, 0, 0, 0, 0)


def case(n, kind, dim):
    rng = np.random.default_rng(n)
    if kind == "surface":
        pr = ls.ellipse_pair(n, seed=2) if dim == 2 else ls.ellipsoid_pair(n, seed=2)
        q = pr.q0
    elif kind == "islands":  # out of each other's reach; the largest case far from the origin
        q = rng.normal(0.0, 0.2, size=(n, dim)) + 1.5 * rng.integers(0, 5, size=(n, 1)) + (300.0 if n > 65536 else 0.0)
    else:  # "points": many landmarks at the same place
        q = np.repeat(rng.uniform(-1, 1, size=(7, dim)), (n + 6) // 7, axis=0)[:n]
    p = rng.normal(0.0, 20.0 / n, size=(n, dim))
    t = q + rng.normal(0.0, 0.05, size=(n, dim))
    return [torch.tensor(np.ascontiguousarray(x), dtype=torch.float32, device="cuda") for x in (q, p, t)]


@pytest.mark.parametrize("n,kind,dim,T,kw", [
    (16384, "surface", 3, 8, {}),
    (12289, "islands", 3, 8, {"ckpt_every": 3}),
    (18433, "points", 3, 8, {}),
    (8255, "surface", 3, 4, {"integrator": "rk4", "h_at": "end"}),
    (16001, "surface", 2, 8, {}),
    (16385, "islands", 2, 2, {"integrator": "rk4", "ckpt_every": 1}),
    (16500, "surface", 3, 8, {"h_at": "end"}),
    (70001, "islands", 3, 8, {}),
])
def test_ordered_gradient_equals_every_pair(n, kind, dim, T, kw):
    q, p, t = case(n, kind, dim)
    run = lambda: gs().shoot_gradient(q, p, t, T, 0.05, 10.0, **kw)  # noqa: E731
    a, b = run(), every_pair(run)
    e = abs(a[0] - b[0]) / abs(b[0]), rel(a[1], b[1]), rel(a[2], b[2])
    print("N=%d %s dim %d: loss %.2e grad_p0 %.2e grad_q0 %.2e" % ((n, kind, dim) + e))
    assert max(e) < BAR + (0.0 if T == 1 else 2.0 ** -24 * float(q.abs().max()) * 0.85 / 0.05)


@pytest.mark.parametrize("n,dim", [(16511, 3), (16001, 2)])
def test_flow_comes_back_in_the_callers_order(n, dim):
    q, p, _ = case(n, "surface", dim)
    run = lambda: gs().shoot_forward(q, p, 8, 0.05)  # noqa: E731
    a, b = run(), every_pair(run)
    bar = BAR + 2.0 ** -24 * float(q.abs().max()) * 0.85 / 0.05
    assert rel(a[0], b[0]) < bar and rel(a[1], b[1]) < bar and abs(a[2] - b[2]) < BAR * abs(b[2])


@pytest.mark.parametrize("points", ["grid", "scattered"])
def test_large_velocity_field_equals_its_slices(points):
    """A field of many points orders its landmarks and leaves runs out of reach
    out; fields of its slices (under 64 points a landmark) do not."""
    n, sigma = 4097, 0.05
    q, p, _ = case(n, "surface", 3)
    if points == "grid":
        g = torch.linspace(-1.2, 1.2, 65, device="cuda")
        x = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), dim=-1).reshape(-1, 3).contiguous()
    else:
        x = torch.rand((262300, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(5)) * 2 - 1
    v = gs().velocity_field(q, p, x, sigma)
    parts = torch.cat([gs().velocity_field(q, p, c.contiguous(), sigma) for c in x.split(60001)])
    assert rel(v, parts) < BAR


def test_large_velocity_field_reports_a_nan_point():
    q, p, _ = case(4097, "surface", 3)
    x = np.random.default_rng(0).uniform(-1, 1, size=(262300, 3)).astype(np.float32)
    x[100000, 2] = np.nan
    with pytest.raises(gs().GShootError) as e:
        gs().velocity_field(q.cpu().numpy(), p.cpu().numpy(), x, 0.05)
    assert e.value.status == -5
