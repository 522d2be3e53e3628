"""One pair sum of more landmarks than a grid of the fused step kernels has room
for (65535 tiles of 64; the forward step's tiles of 128 set to 64): sampled rows
against the FP64 oracle, at the normwise bar of the other parity tests (1e-5)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N, SIGMA = 65535 * 64 + 1, 0.05
ROWS = np.array([0, 63, N // 2, N - 65, N - 2, N - 1])


def gs():
    import paper_1907_04839_gb300 as m
    return m


def rel(a, b):
    return float(np.linalg.norm(a.cpu().numpy()[ROWS] - b) / np.linalg.norm(b))


def arrays(*ranges):
    rng = np.random.default_rng(0)
    arr = [rng.uniform(lo, hi, size=(N, 3)).astype(np.float32) for lo, hi in ranges]
    return [torch.from_numpy(a).cuda() for a in arr], [a.astype(np.float64) for a in arr]


def test_step_forward_past_the_tile_grid():
    dev, ref = arrays((-1, 1), (0.5e-3, 1.5e-3))
    lib = gs().load()
    gs().check(lib.gs_set_step_config(0, 64, 1, 1, 1))
    try:
        hq, hp = gs().step_forward(*dev, SIGMA)
    finally:
        lib.gs_set_step_config(0, 0, 0, 0, 0)
    rq, rp = oracle.step_forward_rows(*ref, SIGMA, ROWS)
    e = rel(hq, rq), rel(hp, rp)
    print("N=%d Hq %.2e Hp %.2e" % ((N,) + e))
    assert max(e) < 1e-5


def test_step_backward_past_the_tile_grid():
    dev, ref = arrays((-1, 1), (0.5e-3, 1.5e-3), (0.5, 1.5), (0.5, 1.5))
    da, db = gs().step_backward(*dev, SIGMA)
    ra, rb = oracle.step_backward_rows(*ref, SIGMA, ROWS)
    e = rel(da, ra), rel(db, rb)
    print("N=%d dalpha %.2e dbeta %.2e" % ((N,) + e))
    assert max(e) < 1e-5
