"""A small gradient that asks for checkpoints holds little memory, also in a
workspace that has served many landmarks and in one that will."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_small_checkpointed_gradient_holds_little_memory():
    import paper_1907_04839_gb300 as gsh
    rng = np.random.default_rng(1)

    def gradient(n, T, **kw):
        q = torch.tensor(rng.uniform(-1, 1, size=(n, 3)), dtype=torch.float32, device="cuda")
        return gsh.shoot_gradient(q, torch.zeros_like(q), q, T, 0.2, 10.0, **kw)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    gsh.load().gs_release_workspace()
    gradient(16384, 2)
    f0 = free()
    # 4000 slots of 64 landmarks are 6 MB; of the workspace's 16384, 1.6 GB.
    gradient(64, 4000, ckpt_every=8)
    f1 = free()
    gradient(32768, 16, ckpt_every=8)
    f2 = free()
    gsh.load().gs_release_workspace()
    print("bytes held: %d, then %d" % (f0 - f1, f1 - f2))
    assert f0 - f1 < 256 << 20 and f1 - f2 < 256 << 20


@pytest.mark.parametrize("n,dim,integrator,h_at", [(1, 3, "euler", "start"), (65, 2, "rk4", "end"), (512, 3, "rk4", "start")])
def test_small_checkpointed_gradient_is_the_plain_one(n, dim, integrator, h_at):
    """The same sums in the same order: the same bits, at any workspace size."""
    import paper_1907_04839_gb300 as gsh
    rng = np.random.default_rng(n)
    put = lambda s: torch.tensor(rng.normal(0.0, s, size=(n, dim)), dtype=torch.float32, device="cuda")  # noqa: E731
    q, p, t = put(0.3), put(0.01), put(0.3)
    run = lambda **kw: gsh.shoot_gradient(q, p, t, 7, 0.2, 10.0, integrator=integrator, h_at=h_at, **kw)  # noqa: E731
    a = run()
    for _ in range(2):
        for c in (1, 3, 6):
            b = run(ckpt_every=c)
            assert a[0] == b[0] and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
        big = torch.zeros((5000, 3), device="cuda")
        gsh.shoot_gradient(big, big, big, 2, 0.2, 10.0)  # wider slots in the workspace from here on
