"""A part of a group's walk that ends early (a link that points outside the tree, which the
walk checks before it follows it): the group's stars get no forces, whatever its other
parts found, and the next walk of a sound tree is whole."""
import ctypes as C

import numpy as np
import pytest

from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,group", [(4000, 64), (20000, 32), (150000, 64)])
def test_group_with_a_failed_part_is_not_written(n, group):
    import torch
    from paper_1507_01009_gb300 import rv
    p32, m32 = hernquist32(n, 71)
    stars = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p32, m32)]
    ctx = rv.Context(n, theta=0.6, eps_star=0.005, n_leaf=8, group=group, tile=64)
    ctx.build_tree(*stars)
    want = ctx.tree_forces()
    ctx.sync_status()
    v = rv.rv_tree_view()
    ctx._check(ctx.L.rv_get_tree(ctx.h, C.byref(v), rv._stream()))
    at = v.clink - ctx.ws.data_ptr()
    links = ctx.ws[at:at + 16 * v.ncell].view(torch.int32).view(v.ncell, 4)
    leaves = torch.nonzero(links[:, 0] == links[:, 1]).flatten()
    leaf = int(leaves[len(leaves) // 2])
    end = int(links[leaf, 3])
    out = [torch.full((n,), 7.0, device="cuda") for _ in range(4)]
    links[leaf, 3] = n + 1   # its end star, beyond the last one
    ctx.tree_forces(out=out)
    with pytest.raises(rv.RvError) as e:
        ctx.sync_status()
    assert e.value.status == rv.RV_E_STACK
    missing = out[0] == 7.0
    assert 0 < int(missing.sum()) < n   # the groups that open the leaf, or come to it, and only those
    for a, b in zip(out, want):
        assert bool((a[missing] == 7.0).all()) and torch.equal(a[~missing], b[~missing])
    links[leaf, 3] = end
    assert all(torch.equal(a, b) for a, b in zip(ctx.tree_forces(), want))
    ctx.sync_status()
