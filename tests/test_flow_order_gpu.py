"""Points that follow a flow whose landmarks lie in spatial order (8 steps,
10^9 pairs a sweep and 16 points a landmark at least), where all pairs are in
reach and where few are: parity with the FP64 oracle on a sample of the points.

Tolerances: those of the other flow_points tests (1e-5, displacements 1e-4).
"""
import math

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
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


def f32(x):
    return np.ascontiguousarray(x, np.float32).astype(np.float64)


@pytest.mark.parametrize("n,m,T,sigma", [
    (5000, 80000, 40, 0.2),    # nearly all pairs in reach
    (5000, 80000, 40, 0.05),   # few
    (16400, 262401, 8, 0.2),   # the other line of "nearly all"
])
def test_points_follow_an_ordered_flow(n, m, T, sigma):
    pr = ls.ellipsoid_pair(n, seed=4)
    q, p = f32(pr.q0), f32((pr.target - pr.q0) / (1.0 + n * 2.0 * math.pi * sigma ** 2 / 7.9))
    x = f32(ls.ellipsoid_pair(m, seed=5, jitter=0.1).q0)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    x1 = gs().flow_points(dev(q), dev(p), dev(x), T, sigma).cpu().numpy().astype(np.float64)
    at = np.random.default_rng(6).permutation(m)[:300]
    r = oracle.flow_points(q, p, x[at], T, sigma)
    assert rel(oracle.flow_points(q, p * (1 + 1e-7), x[at], T, sigma), r) < 1e-6  # well conditioned
    e, disp = rel(x1[at], r), rel(x1[at] - x[at], r - x[at])
    print("N=%d M=%d T=%d sigma=%g flow_points rel err %.2e (displacement %.2e)" % (n, m, T, sigma, e, disp))
    assert e < 1e-5 and disp < 1e-4
