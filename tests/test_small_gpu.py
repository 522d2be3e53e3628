"""Small problems run a whole flow or gradient in one launch (up to 512 padded
landmarks): parity with the FP64 oracle at the edges of its range and in every
variant, and agreement of its flow with its gradient's.

Tolerances: the normwise bars of the parity tests (1e-5, gradients 1e-4).
"""
import numpy as np
import pytest

import landmark_synth as ls
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def gs():
    import paper_1907_04839_gb300 as m
    return m


def rel(a, b):
    a = np.asarray(a.cpu().numpy() if hasattr(a, "cpu") else a, np.float64).ravel()
    b = np.asarray(b, np.float64).ravel()
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("integrator,h_at", [("euler", "start"), ("euler", "end"), ("rk4", "start"), ("rk4", "end")])
@pytest.mark.parametrize("n,T,dim", [(1, 3, 3), (2, 1, 2), (63, 4, 3), (64, 1, 3), (65, 5, 2), (130, 2, 3), (449, 3, 3),
                                     (511, 2, 2), (512, 4, 3)])
def test_small_sweeps_match_the_oracle(n, T, dim, integrator, h_at):
    rng = np.random.default_rng(1000 * n + T)
    f32 = lambda x: np.ascontiguousarray(x, np.float32).astype(np.float64)  # noqa: E731
    q = f32(rng.uniform(-0.5, 0.5, size=(n, dim)))
    p = f32(rng.normal(0.0, 0.3 / max(1.0, 0.1 * n), size=(n, dim)))
    t = f32(q + rng.normal(0.0, 0.1, size=(n, dim)))
    sigma, lam = 0.25, 10.0
    d = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda")  # noqa: E731
    loss, gp, gq = gs().shoot_gradient(d(q), d(p), d(t), T, sigma, lam, integrator=integrator, h_at=h_at)
    r = oracle.shoot_gradient_v(q, p, t, T, sigma, lam, integrator, h_at)
    assert abs(loss - r["loss"]) < 1e-5 * abs(r["loss"])
    assert rel(gp, r["grad_p0"]) < 1e-4 and rel(gq, r["grad_q0"]) < 1e-4
    if h_at == "start":
        q1, p1, h0 = gs().shoot_forward(d(q), d(p), T, sigma, integrator=integrator)
        o1, o2 = oracle.shoot_forward_v(q, p, T, sigma, integrator)
        assert rel(q1, o1) < 1e-5 and rel(p1, o2) < 1e-5
        assert abs(h0 - r["H"]) < 1e-5 * abs(r["H"])
        # host arrays are staged and give the same bits
        hq1, hp1, hh0 = gs().shoot_forward(q.astype(np.float32), p.astype(np.float32), T, sigma, integrator=integrator)
        assert np.array_equal(hq1, q1.cpu().numpy()) and np.array_equal(hp1, p1.cpu().numpy()) and hh0 == h0


def test_small_sweep_reports_nonfinite_inputs():
    pr = ls.ellipsoid_pair(200, seed=3)
    q = torch.tensor(pr.q0, dtype=torch.float32, device="cuda")
    p = torch.zeros_like(q)
    p[7, 1] = float("inf")
    with pytest.raises(gs().GShootError) as e:
        gs().shoot_gradient(q, p, q, 4, 0.2, 10.0)
    assert e.value.status == -5
