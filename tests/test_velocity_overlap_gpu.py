"""velocity_field with its output in the memory of its points: the same values as
with an array apart, whatever the offset between the two."""
import ctypes

import numpy as np
import pytest

import landmark_synth as ls

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,m", [(300, 5000), (4100, 262500)])
@pytest.mark.parametrize("offset", [0, -300, 300, 1])  # floats from the points to the velocities
def test_velocities_over_their_points(n, m, offset):
    import paper_1907_04839_gb300 as gsh
    put = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda")  # noqa: E731
    q, p = put(ls.ellipsoid_pair(n, seed=3).q0), put(np.random.default_rng(n).normal(0.0, 20.0 / n, size=(n, 3)))
    x = put(np.random.default_rng(4).uniform(-1, 1, size=(m, 3)))
    want = gsh.velocity_field(q, p, x, 0.05)
    room = torch.zeros(3 * m + 600, device="cuda")
    xs, vs = room[300:300 + 3 * m], room[300 + offset:300 + offset + 3 * m]
    xs.copy_(x.view(-1))
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    gsh.check(gsh.load().velocity_field(n, m, 0.05, ptr(q), ptr(p), ptr(xs), ptr(vs), stream))
    assert torch.equal(vs.view(m, 3), want)
