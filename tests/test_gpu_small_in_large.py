"""Small builds in a context made for many stars: the same tree, and no time
lost to the context's size."""
import numpy as np
import pytest

from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu


def _times(contexts, stars):
    """us a build for each context, the best of runs taken in turn."""
    import torch
    best = [1e9] * len(contexts)
    for _ in range(8):
        for k, ctx in enumerate(contexts):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            for _ in range(5):
                ctx.build_tree(*stars)
            a.record()
            for _ in range(50):
                ctx.build_tree(*stars)
            b.record()
            torch.cuda.synchronize()
            best[k] = min(best[k], a.elapsed_time(b) * 20.0)
    return best


@pytest.mark.parametrize("n,n_leaf", [(1000, 64), (4096, 16), (4097, 1), (30000, 16)])
def test_build_in_a_large_context(n, n_leaf):
    import torch
    from paper_1507_01009_gb300 import rv
    p32, m32 = hernquist32(n, 23)
    stars = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p32, m32)]
    large, own = (rv.Context(k, n_leaf=n_leaf, group=32) for k in (1 << 22, n))
    big = [torch.rand(1 << 22, device="cuda") for _ in range(4)]
    large.build_tree(*big)   # leave a large tree's words behind
    large.sync_status()
    for _ in range(2):
        large.build_tree(*stars)
        own.build_tree(*stars)
        a, b = large.tree_view(), own.tree_view()
        for k in ("keys", "perm", "cbox", "clink", "cmom", "groups"):
            assert torch.equal(a[k], b[k]), k
        for u, v in zip(large.tree_forces(), own.tree_forces()):
            assert torch.equal(u, v)
    large.sync_status()
    t_large, t_own = _times((large, own), stars)
    assert t_large <= 1.1 * t_own, (t_large, t_own)
