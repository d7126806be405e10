"""Captured steps and what other calls on the same context leave behind: a
replay must not depend on the builds in between, and the tree it leaves is its
own. Systems on both sides of 4096 stars (one-block builds) and of members."""
import numpy as np
import pytest

import ics
from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rvmod():
    from paper_1507_01009_gb300 import rv
    rv.load()
    return rv


def _stars(n, seed):
    import torch
    p32, m32 = hernquist32(n, seed)
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p32, m32)]


def _system(rvmod, sizes):
    ws = [ics.hernquist(n, 70 + k) for k, n in enumerate(sizes)]
    pos, vel, mass = (np.concatenate(a, -1) for a in zip(*[(w.pos, w.vel, w.mass) for w in ws]))
    b, M = ics.central_binary(), len(sizes)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64) if M > 1 else None
    return rvmod.System(pos, vel, mass, chain_m=np.tile(b.mass, M), chain_x=np.tile(b.pos, (M, 1)),
                        chain_v=np.tile(b.vel, (M, 1)), pert_mode=2, pert_k=16, member_offsets=off)


@pytest.mark.parametrize("other", ["none", "build", "members", "search"])
@pytest.mark.parametrize("sizes", [[3000], [9000], [18000], [2000, 3500, 5000]])   # [18000]: a cluster searches
def test_replay_after_other_builds(rvmod, sizes, other):
    import torch
    n, n_max = sum(sizes), 20000
    st = torch.cuda.Stream()
    between = [_stars(k, 3) for k in (1000, 4097, 20000)]
    dx = [0.0] * (3 * 2 * len(sizes))

    def step(ctx, S, energy, graph):
        if graph:
            ctx.kdk_step_graph(S, 1e-3, 1, energy_out=energy, stream=st)
        else:
            ctx.kdk_step(S, 1e-3, 1, stream=st)
            ctx.energy(S, out=energy, stream=st)

    out = []
    for graph in (True, False):
        ctx, S = rvmod.Context(n_max, theta=0.5, eps_star=0.005), _system(rvmod, sizes)
        energy = torch.zeros(10 * len(sizes), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.system_forces(S, stream=st)
        for k in range(3):
            step(ctx, S, energy, graph)
            if graph and other == "build":
                ctx.build_tree(*between[k], stream=st)
            if graph and other == "members":
                ctx.build_tree_members([0, 300, len(between[k][0])], *between[k], stream=st)
            if graph and other == "search":
                ctx.select_perturbers(*between[k][:3], (0, 0, 0), 2, k=10, stream=st)
        step(ctx, S, energy, graph)
        pull = ctx.chain_perturber_forces(S, 1e-4, torch.tensor(dx, dtype=torch.float64, device="cuda"), stream=st)
        forces = [torch.empty(n, device="cuda") for _ in range(4)]
        torch.cuda.synchronize()
        ctx.tree_forces_members(out=forces, stream=st)
        view = ctx.tree_view(stream=st)
        st.synchronize()
        ctx.sync_status(stream=st)
        out.append([S.state, S.chain_x, S.chain_a, energy, *pull, *forces, view["keys"], view["perm"], view["pos"],
                    view["cbox"]])
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n,n_other", [(3000, 1000), (3000, 9000), (9000, 3000), (9000, 20000)])
def test_callers_graph_replayed_after_another_build(rvmod, n, n_other):
    """A build captured by the caller reads the offsets of the last build: the
    replay is refused in the status and writes nothing, until they fit again."""
    import torch
    ctx = rvmod.Context(20000, theta=0.5, eps_star=0.005)
    stars, others = _stars(n, 8), _stars(n_other, 9)
    out = [torch.zeros(n, device="cuda") for _ in range(4)]
    ctx.build_tree(*stars)
    want = ctx.tree_forces()
    ctx.sync_status()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.build_tree(*stars)
        ctx.tree_forces(out=out)
    g.replay()
    ctx.sync_status()
    assert all(torch.equal(a, b) for a, b in zip(out, want))
    ctx.build_tree(*others)
    ctx.sync_status()
    for o in out:
        o.fill_(7.0)
    g.replay()
    with pytest.raises(rvmod.RvError) as e:
        ctx.sync_status()
    assert e.value.status == rvmod.RV_E_INVAL and "offsets" in str(e.value)
    assert all(bool((o == 7.0).all()) for o in out)
    ctx.build_tree(*stars)
    g.replay()
    ctx.sync_status()
    assert all(torch.equal(a, b) for a, b in zip(out, want))


def test_workspace_is_clear_before_the_first_call(rvmod):
    """The words a context expects to find zero are, on whichever stream its first
    call comes and whatever was queued on the memory before."""
    import torch
    n = 20000
    stars = _stars(n, 10)
    ref = rvmod.Context(n)
    ref.build_tree(*stars)
    want = ref.tree_forces()
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    # the clear waits behind the default stream's work, the build comes on another stream
    ctx = rvmod.Context(n)
    torch.cuda._sleep(200_000_000)
    ctx.ws.fill_(255)
    ctx._check(ctx.L.rv_set_workspace(ctx.h, ctx.ws.data_ptr() + ctx._ws_off, ctx.ws.numel() - 256))
    ctx.build_tree(*stars, stream=st)
    out = [torch.empty(n, device="cuda") for _ in range(4)]
    st.wait_stream(torch.cuda.current_stream())
    ctx.n = n
    ctx.tree_forces(out=out, stream=st)
    ctx.sync_status(stream=st)
    assert all(torch.equal(a, b) for a, b in zip(out, want))
    # the memory's last owner still writes on the context's own stream
    with torch.cuda.stream(st):
        old = torch.empty(ctx.ws.numel(), dtype=torch.uint8, device="cuda")
        at = old.data_ptr()
        torch.cuda._sleep(200_000_000)
        old.fill_(255)
        del old
        other = rvmod.Context(n)
        same = other.ws.data_ptr() == at
        other.build_tree(*stars)
        got = other.tree_forces()
        other.sync_status()
    assert same and all(torch.equal(a, b) for a, b in zip(got, want))
