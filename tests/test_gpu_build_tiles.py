"""The build's single-pass sort, scan and group kernels at the edges of their
tiles and of their size classes: keys, order, cells and groups bit for bit the
oracle's; the selections' own use of the sort and the scan against numpy."""
import numpy as np
import pytest

import oracle
from gpu_helpers import gpu_cells_as_oracle, gpu_tree, hernquist32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rvmod():
    from paper_1507_01009_gb300 import rv
    rv.load()
    return rv


# one block sorts up to 1024 and up to 4096 stars, then tiles of 1024; tiles of
# 2048 and 4096 from 2^17 and 2^18 stars; n_leaf 1 gives
# the most cells (many group tiles), n_leaf 64 the fewest
@pytest.mark.parametrize("n,n_leaf,G", [(2, 1, 1), (31, 4, 4), (1023, 1, 3), (1024, 8, 32), (1025, 64, 64), (4095, 2, 7),
                                        (4096, 1, 1), (4097, 16, 32), (8191, 1, 1), ((1 << 17) - 1, 24, 64),
                                        (1 << 17, 4, 8), ((1 << 18) - 1, 64, 64), ((1 << 18) + 4097, 16, 32),
                                        ((1 << 19) + 1, 24, 64)])
def test_tree_bits_at_tile_edges(rvmod, n, n_leaf, G):
    p32, m32 = hernquist32(n, 300 + n_leaf)
    ctx = rvmod.Context(n + 5, theta=0.5, eps_star=0.005, n_leaf=n_leaf, group=G)
    T = oracle.Tree(p32, m32, n_leaf, G)
    for _ in range(2):   # the second build starts from the first one's words
        gpu_tree(ctx, p32, m32)
        ctx.sync_status()
        v = ctx.tree_view()
        np.testing.assert_array_equal(v["keys"].cpu().numpy().view(np.uint64), T.key)
        np.testing.assert_array_equal(v["perm"].cpu().numpy(), T.perm)
        np.testing.assert_array_equal(v["pos"].cpu().numpy()[:, :3], p32.T[T.perm])
        np.testing.assert_array_equal(gpu_cells_as_oracle(v), T.cells)
        g, go = v["groups"].cpu().numpy(), np.asarray(T.groups, dtype=np.int64).reshape(-1, 8)
        np.testing.assert_array_equal(g[np.argsort(g[:, 0], kind="stable")], go[np.argsort(go[:, 0], kind="stable")])


def test_coincident_stars_sort_in_caller_order(rvmod):
    """All keys equal: every element of every pass in one digit, one cell per level."""
    n = 70001
    p32 = np.repeat(np.array([[1.0], [2.0], [-3.0]], dtype=np.float32), n, axis=1)
    p32[0, 0] = 0.0   # a bounding cube of side 1
    ctx = rvmod.Context(n, theta=0.5, eps_star=0.005)
    gpu_tree(ctx, p32, np.full(n, 1.0 / n, dtype=np.float32))
    ctx.sync_status()
    np.testing.assert_array_equal(ctx.tree_view()["perm"].cpu().numpy(), np.arange(n))


@pytest.mark.parametrize("n", [1, 2047, 2049, (1 << 17) + 1, (1 << 18) + 3])
def test_selections_at_tile_edges(rvmod, n):
    import torch
    p32, _ = hernquist32(n, 7)
    x, y, z = (torch.from_numpy(np.ascontiguousarray(p32[a])).cuda() for a in range(3))
    ctx = rvmod.Context(n)
    d2 = (p32[0] * p32[0] + p32[1] * p32[1]) + p32[2] * p32[2]   # FP32, one rounding per operation
    for k in (1, min(n, 33), min(n, 5000), 5000):
        idx, cnt = ctx.select_perturbers(x, y, z, (0.0, 0.0, 0.0), 2, k=k)
        kk = min(k, n)
        assert int(cnt.item()) == kk
        np.testing.assert_array_equal(idx[:kk].cpu().numpy(), np.argsort(d2, kind="stable")[:kk])
    r2 = np.float32(0.3) * np.float32(0.3)   # the radius rule: its FP32 square
    inside = np.flatnonzero(d2 < r2)
    idx, cnt = ctx.select_perturbers(x, y, z, (0.0, 0.0, 0.0), 1, radius=0.3, cap=max(1, len(inside)))
    assert int(cnt.item()) == len(inside)
    np.testing.assert_array_equal(idx[:len(inside)].cpu().numpy(), inside)


@pytest.mark.parametrize("n,k", [(9000, 3000), (9000, 5000), (70001, 1), (70001, 4999)])
def test_nearest_of_many_equal_distances(rvmod, n, k):
    """Candidates that do not fit one block's shared memory: all stars at one
    distance (ties by index), and half of them, beside distances of 0, infinity and
    far below the bins' resolution."""
    import torch
    rng = np.random.default_rng(n + k)
    for kind in range(3):
        x = np.full(n, 2.0, dtype=np.float32)
        if kind == 1:
            x[rng.permutation(n)[: n // 2]] = np.float32(3.0)
        if kind == 2:
            x[:] = np.float32(2.0) + rng.integers(0, 3, n).astype(np.float32) * np.float32(2.0 ** -22)
            x[rng.permutation(n)[:5]] = [0.0, np.inf, -np.inf, 1e-30, 2.0]
        y, z = np.zeros_like(x), np.zeros_like(x)
        d2 = (x * x + y * y) + z * z
        ctx = rvmod.Context(n)
        xs = [torch.from_numpy(v).cuda() for v in (x, y, z)]
        for _ in range(2):
            idx, cnt = ctx.select_perturbers(*xs, (0.0, 0.0, 0.0), 2, k=k)
            assert int(cnt.item()) == k
            np.testing.assert_array_equal(idx[:k].cpu().numpy(), np.argsort(d2, kind="stable")[:k])


def test_nearest_per_member(rvmod):
    """Perturbers of every member of an ensemble (empty, smaller than k, large), by the forces they make: the
    selection of each member equals the one of its stars alone."""
    import torch
    sizes, k = [40, 0, 5000, 1, 70001], 64
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    p32, m32 = hernquist32(int(off[-1]), 5)
    M = len(sizes)
    cm = np.full(2 * M, 0.005)
    cx = np.tile(np.array([[0.0055, 0, 0], [-0.0055, 0, 0]]), (M, 1))
    ctx = rvmod.Context(int(off[-1]), theta=0.5, eps_star=0.005)
    S = rvmod.System(p32, np.zeros_like(p32), m32, chain_m=cm, chain_x=cx, chain_v=np.zeros_like(cx), pert_mode=2,
                     pert_k=k, member_offsets=off)
    ctx.system_forces(S)
    at = torch.from_numpy(cx).cuda()
    a, pot = ctx.chain_perturber_forces(S, 0.0, at)
    ctx.sync_status()
    a, pot = a.cpu().numpy().reshape(-1, 3), pot.cpu().numpy()
    for i in range(M):
        p = p32[:, off[i]:off[i + 1]]
        d2 = (p[0] * p[0] + p[1] * p[1]) + p[2] * p[2]
        near = np.argsort(d2, kind="stable")[:k]
        q, w = p[:, near].astype(np.float64), m32[off[i]:off[i + 1]][near].astype(np.float64)
        for b in (2 * i, 2 * i + 1):
            d = q - cx[b][:, None]
            r = np.sqrt((d * d).sum(0))
            ref = (w * d / r ** 3).sum(1)
            assert np.allclose(a[b], ref, rtol=1e-11, atol=1e-12 * max(1.0, np.abs(w / r ** 2).sum()))
            assert np.isclose(pot[b], -(w / r).sum(), rtol=1e-12, atol=1e-14)
