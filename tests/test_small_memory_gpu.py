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
