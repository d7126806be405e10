"""The split of small builds' walks into parts (walk.cu, Part): forces and
interaction counts against the oracle's walk on both sides of every change of
the number of parts, group masks and queue orders that leave the sums alone, and
members of an ensemble that share its split."""
import numpy as np
import pytest

import oracle
from gpu_helpers import err_stats, gpu_tree, hernquist32

pytestmark = pytest.mark.gpu

MED_TOL, MAX_TOL = 1e-5, 1e-4   # the GPU-versus-oracle-tree tolerances of the force tests


@pytest.fixture(scope="module")
def rvmod():
    from paper_1507_01009_gb300 import rv
    rv.load()
    return rv


def last_n(P, group, items=16384):
    """The largest build walked in P parts: P (n / group + 1) <= items (integer division); items doubles for a
    single system of 2^17 to 2^19 stars."""
    return (items // P) * group - 1


# one star, groups smaller than the parts, both sides of 16 / 8 parts (groups of 1, 7, 32 and 64 stars), a ragged middle
@pytest.mark.parametrize("n,group,n_leaf,quad", [(1, 64, 24, True), (17, 64, 4, True), (130, 7, 3, False),
                                                 (last_n(16, 1), 1, 8, True), (last_n(16, 7) + 1, 7, 5, True),
                                                 (last_n(16, 32), 32, 16, True), (last_n(16, 32) + 1, 32, 16, True),
                                                 (50021, 64, 24, False)])
def test_split_walk_vs_oracle(rvmod, n, group, n_leaf, quad):
    p32, m32 = hernquist32(n, 90 + group)
    eps = float(np.float32(0.005))
    ctx = rvmod.Context(n, theta=0.5, eps_star=eps, n_leaf=n_leaf, group=group, quadrupole=quad, tile=32)
    gpu_tree(ctx, p32, m32)
    a = np.stack([t.cpu().numpy() for t in ctx.tree_forces()[:3]]).astype(np.float64)
    ctx.sync_status()
    T = oracle.Tree(p32, m32, n_leaf, group)
    ao, _, _, _, cnt = T.forces(0.5, eps, quad, counts=True)
    # the GPU also counts each star's own pair
    assert ctx.walk_stats() == (int(cnt[:, 0].sum()) + n, int(cnt[:, 1].sum()))
    if n > 1:
        med, _, mx = err_stats(a, ao)
        assert med <= MED_TOL and mx <= MAX_TOL, (med, mx)


@pytest.mark.parametrize("n", [last_n(8, 64), last_n(8, 64) + 1, last_n(8, 64, 32768) + 1])
def test_split_walk_repeats_and_masks(rvmod, n):
    """Cost-ordered, volume-ordered and masked walks of a split build give the same bits."""
    import torch
    p32, m32 = hernquist32(n, 12)
    kw = dict(theta=0.5, eps_star=float(np.float32(0.005)), n_leaf=24, group=64, tile=96)
    ctx = rvmod.Context(n, **kw)
    gpu_tree(ctx, p32, m32)
    first = ctx.tree_forces()
    again = ctx.tree_forces()
    assert all(torch.equal(u, v) for u, v in zip(first, again))
    lv = (np.linalg.norm(p32.astype(np.float64), axis=0) < 0.3).astype(np.int8)
    S = rvmod.System(p32, np.zeros_like(p32), m32)
    B = rvmod.Blocks(n, 1e-9, 1, adapt=False, level=lv)   # the stars do not move within rounding
    ctx.block_start(S, B)
    full = [t.clone() for t in (S.ax, S.ay, S.az)]
    x0 = S.state[:3].clone()
    S.state[6:10] = 0
    S.state[3:6] = 0
    ctx.block_steps(S, B, 1)
    ctx.sync_status()
    act = torch.from_numpy(lv == 1).cuda()
    assert torch.equal(S.state[:3], x0)
    for u, v in zip(full, (S.ax, S.ay, S.az)):
        assert torch.equal(u[act], v[act])


def test_members_of_a_split_build(rvmod):
    """Members walked with the parts of their build's size: each member's forces match its own oracle walk,
    and the counts add up."""
    import torch
    sizes = [700, 0, 33001, 1, 5000]
    eps = float(np.float32(0.005))
    parts = [hernquist32(k, 60 + i) if k else None for i, k in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    p32 = np.ascontiguousarray(np.concatenate([p[0] for p in parts if p], axis=1))
    m32 = np.concatenate([p[1] for p in parts if p])
    ctx = rvmod.Context(int(off[-1]), theta=0.5, eps_star=eps, n_leaf=24, group=32, tile=64)
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (*p32, m32)]
    ctx.build_tree_members(off, *dev)
    a = np.stack([t.cpu().numpy() for t in ctx.tree_forces_members()[:3]]).astype(np.float64)
    ctx.sync_status()
    counts = np.zeros(2, dtype=np.int64)
    for i, k in enumerate(sizes):
        if not k:
            continue
        ao, _, _, _, cnt = oracle.Tree(*parts[i], 24, 32).forces(0.5, eps, counts=True)
        counts += (int(cnt[:, 0].sum()) + k, int(cnt[:, 1].sum()))
        if k > 1:
            med, _, mx = err_stats(a[:, off[i]:off[i + 1]], ao)
            assert med <= MED_TOL and mx <= MAX_TOL, (k, med, mx)
    assert ctx.walk_stats() == tuple(counts)
