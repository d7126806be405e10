"""What a member of an ensemble shares with the same stars built and walked alone:
the tree and the interactions always, the bits of the forces when both walks
are split into the same number of parts (which follows from the build's star
count), and otherwise the forces up to the rounding of their sums."""
import numpy as np
import pytest

from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu

TILE = 96


def test_members_across_a_change_of_parts():
    """Members walked whole (the build has more than 2^19 stars) against 16 parts alone (the
    small ones) and whole alone (the large one: the same bits).

    Tolerance: a star's terms are the same FP32 numbers in both walks, and both
    add tile sums with compensation, so the two differ by the rounding inside the
    tiles: at most TILE / 2 + 2 additions in a row of partial sums no larger than
    the sum of the terms' sizes A, each off by 2^-24 of it, on either side, and
    the last rounding. A: the potential's is |phi| and the own pair's m / eps; of
    an acceleration's, the direct sum of the terms' sizes (a multipole's terms are
    no larger to within its 10 % of higher orders)."""
    import torch
    from paper_1507_01009_gb300 import rv
    eps = np.float32(0.005)
    sizes = [8192, 0, 530000, 3001]
    kw = dict(theta=0.5, eps_star=float(eps), n_leaf=24, group=64, tile=TILE)
    off = np.concatenate([[0], np.cumsum(sizes)])
    parts = {k: [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p, m)]
             for k, (p, m) in ((k, hernquist32(n, 80 + k)) for k, n in enumerate(sizes) if n)}
    ens = rv.Context(int(off[-1]), **kw)
    ens.build_tree_members(off, *[torch.cat(t) for t in zip(*parts.values())])
    f = ens.tree_forces_members()
    counts = np.array(ens.walk_stats())
    v = ens.tree_view()
    ens.sync_status()
    first = v["clink"][:, 2]
    for k, stars in parts.items():
        s, e = int(off[k]), int(off[k + 1])
        one = rv.Context(e - s, **kw)
        one.build_tree(*stars)
        g = one.tree_forces()
        counts -= one.walk_stats()
        w = one.tree_view()
        one.sync_status()
        own = (first >= s) & (first < e)
        assert torch.equal(v["keys"][s:e], w["keys"]) and torch.equal(v["perm"][s:e] - s, w["perm"])
        assert torch.equal(v["cbox"][own], w["cbox"]) and torch.equal(v["cmom"].reshape(-1, 12)[own], w["cmom"].reshape(-1, 12))
        if e - s > 1 << 19:
            assert all(torch.equal(a[s:e], b) for a, b in zip(f, g))
            continue
        x, m = torch.stack(stars[:3]).double(), stars[3].double()
        bound = 2 * (TILE / 2 + 2) * 2.0 ** -24 + 2.0 ** -23
        same = True
        for i in range(0, e - s, 1024):
            d = x[:, None, :] - x[:, i:i + 1024, None]
            r2 = (d * d).sum(0) + float(eps) ** 2
            at = slice(s + i, min(s + i + 1024, e))
            phi = (m / r2.sqrt()).sum(1)   # with the own pair's m / eps
            assert bool(((f[3][at] - g[3][i:i + 1024]).abs() <= bound * phi).all())
            for a in range(3):
                size = (m * d[a].abs() / r2 ** 1.5).sum(1)
                assert bool(((f[a][at] - g[a][i:i + 1024]).abs() <= 1.1 * bound * size).all())
                same &= torch.equal(f[a][at], g[a][i:i + 1024])
        assert not same   # (the case the tolerance is for: the parts differ)
    assert not counts.any()
