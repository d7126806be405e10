"""Cell moments of large builds (from 2^20 stars, where a leaf's stars and a cell's
children are taken one by one): the same bits as those of small builds (all in
flight at once), which the parity tests compare with the oracle."""
import numpy as np
import pytest

from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_leaf,group", [(16, 32), (24, 64), (1, 64)])
def test_large_build_has_the_small_builds_moments(n_leaf, group):
    """Members of 1 040 000 and 9 000 stars together (a large build) and alone (small ones)."""
    import torch
    from paper_1507_01009_gb300 import rv
    sizes = [1_040_000, 9_000]
    if n_leaf == 1:
        sizes = [1_040_000, 8_577]   # 2^20 + 1 in all
    assert max(sizes) < 1 << 20 <= sum(sizes)
    parts = [hernquist32(n, 50 + k) for k, n in enumerate(sizes)]
    stars = [[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p, m)] for p, m in parts]
    ctx = rv.Context(sum(sizes), n_leaf=n_leaf, group=group)
    ctx.build_tree_members([0, sizes[0], sum(sizes)], *[torch.cat(t) for t in zip(*stars)])
    v = ctx.tree_view()
    ctx.sync_status()
    first = v["clink"][:, 2]
    for k, s in enumerate((0, sizes[0])):
        own = (first >= s) & (first < s + sizes[k])
        one = rv.Context(sizes[k], n_leaf=n_leaf, group=group)
        one.build_tree(*stars[k])
        w = one.tree_view()
        one.sync_status()
        assert torch.equal(v["cbox"][own], w["cbox"])
        assert torch.equal(v["cmom"].reshape(-1, 12)[own], w["cmom"].reshape(-1, 12))
