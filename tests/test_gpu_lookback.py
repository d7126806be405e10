"""Look-back waits that give up (rv_lookback_selftest withholds a tile's sum and
limits the polls: no GPU fault): nothing that the wait left unwritten is used,
the status says so, and the context's next call is whole."""
import numpy as np
import pytest

import ics
from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu

SORT, SCAN, GROUPS = 1, 9, 10   # the stages' numbers in include/rv.h
N = 60000                       # several tiles of every stage


@pytest.fixture(scope="module")
def rvmod():
    from paper_1507_01009_gb300 import rv
    rv.load()
    return rv


def _dev(p32, m32):
    import torch
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p32, m32)]


def _gave_up(rvmod, ctx):
    with pytest.raises(rvmod.RvError) as e:
        ctx.sync_status()
    assert e.value.status == rvmod.RV_E_TIMEOUT
    assert "look-back" in str(e.value)   # not the network's completion wait


@pytest.mark.parametrize("members", [1, 3])
@pytest.mark.parametrize("stage", [SORT, SORT + 3, SORT + 6, SORT + 7, SCAN, GROUPS])
def test_build_that_gave_up_writes_no_forces(rvmod, stage, members):
    import torch
    if stage == SORT + 7 and members == 1:
        pytest.skip("no pass over the members")
    stars = _dev(*hernquist32(N, 5))
    off = [0, 20011, 20011, N][:members] + [N]

    def build(c):
        c.build_tree_members(off, *stars) if members > 1 else c.build_tree(*stars)

    ctx = rvmod.Context(N)
    ctx.lookback_selftest(stage, 50)
    build(ctx)
    out = [torch.full((N,), 7.0, device="cuda") for _ in range(4)]
    ctx.tree_forces_members(out=out)
    _gave_up(rvmod, ctx)
    assert all(bool((o == 7.0).all()) for o in out)
    _, ncell, ngroup = ctx.tree_sizes()
    assert ngroup == 0 and (ncell > 0) == (stage == GROUPS)
    build(ctx)
    got = ctx.tree_forces_members()
    ctx.sync_status()
    fresh = rvmod.Context(N)
    build(fresh)
    for a, b in zip(got, fresh.tree_forces_members()):
        assert torch.equal(a, b)


@pytest.mark.parametrize("what,stage", [("radius", SCAN), ("tidal", SCAN), ("absorb", SCAN), ("nearest", SORT),
                                        ("nearest", SORT + 3), ("start", SORT + 1)])
def test_search_that_gave_up_selects_nothing(rvmod, what, stage):
    import torch
    x, y, z, m = _dev(*hernquist32(N, 6))
    ctx = rvmod.Context(N)

    def search():
        if what == "radius":
            return ctx.select_perturbers(x, y, z, (0, 0, 0), 1, radius=0.1)
        if what == "tidal":
            return ctx.select_perturbers_tidal(x, y, z, m, (0, 0, 0), 1e-2, 0.1, 1.0)
        if what == "absorb":
            return ctx.chain_absorb(x, y, z, [1.0, 1.0], [[0.1, 0, 0], [-0.1, 0, 0]])[:2]
        if what == "nearest":   # more than the selection by leading bits takes: a sort
            return ctx.select_perturbers(x, y, z, (0, 0, 0), 2, k=6000, cap=6000)
        r = ctx.chain_start_radius((x, y, z), (x, y, z), m, (0, 0, 0), 1e-3, 1.0, 1.0, 1e-3)
        return r, torch.ones(1)

    ctx.lookback_selftest(stage, 50)
    if what == "start":
        with pytest.raises(rvmod.RvError) as e:
            search()
        assert e.value.status == rvmod.RV_E_TIMEOUT
    else:
        assert int(search()[1]) == 0
    _gave_up(rvmod, ctx)
    assert int(search()[1]) > 0
    ctx.sync_status()


def test_member_search_that_gave_up_has_no_perturbers(rvmod):
    """Radius search of several members (a sort): the pass goes on with no
    perturbers, and the next one equals a fresh context's."""
    sizes = [20000, 15000]
    pos, vel, mass = (np.concatenate(a, -1) for a in zip(*[(w.pos, w.vel, w.mass) for w in
                                                           (ics.hernquist(n, 90 + n) for n in sizes)]))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    b = ics.central_binary()

    def system():
        return rvmod.System(pos, vel, mass, chain_m=np.tile(b.mass, 2), chain_x=np.tile(b.pos, (2, 1)),
                            chain_v=np.tile(b.vel, (2, 1)), pert_mode=1, pert_radius=0.05, member_offsets=off)

    ctx, S = rvmod.Context(sum(sizes), eps_star=0.005), system()
    ctx.lookback_selftest(SORT + 1, 50)
    ctx.system_forces(S)
    a, _ = ctx.chain_perturber_forces(S, 0.0, S.chain_x)
    _gave_up(rvmod, ctx)
    assert float(a.abs().max()) == 0.0
    ctx.system_forces(S)
    ctx.sync_status()
    fresh, F = rvmod.Context(sum(sizes), eps_star=0.005), system()
    fresh.system_forces(F)
    for f in ("ax", "pot", "chain_a", "chain_pot"):
        np.testing.assert_array_equal(getattr(S, f).cpu().numpy(), getattr(F, f).cpu().numpy())


def test_arguments(rvmod):
    ctx = rvmod.Context(10)
    for bad in ((-1, 0), (11, 0), (1, -1), (1, (1 << 20) + 1)):
        with pytest.raises(rvmod.RvError):
            ctx.lookback_selftest(*bad)
    ctx.lookback_selftest(0, 0)
