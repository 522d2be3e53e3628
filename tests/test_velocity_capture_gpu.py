"""velocity_field recorded into a CUDA graph by its caller: every size that fits
the workspace can be, also one that would order its landmarks had it the room."""
import numpy as np
import pytest

import landmark_synth as ls

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


def test_velocity_field_in_a_graph_capture():
    import paper_1907_04839_gb300 as gsh
    put = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")  # noqa: E731
    state = lambda n: (put(ls.ellipsoid_pair(n, seed=3).q0),  # noqa: E731
                       put(np.random.default_rng(n).normal(0.0, 20.0 / n, size=(n, 3))))
    x = put(np.random.default_rng(4).uniform(-1, 1, size=(262300, 3)))
    gsh.load().gs_release_workspace()
    gsh.velocity_field(*state(8000), x, 0.05)  # room for the landmarks and points below, no order yet
    q, p = state(4000)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        v = gsh.velocity_field(q, p, x, 0.05)
    for k in (1.0, 2.0):
        p.mul_(k)
        g.replay()
        torch.cuda.synchronize()
        # FP32 sums in another order: 2e-6 normwise
        assert rel(v, gsh.velocity_field(q, p, x, 0.05)) < 2e-6
