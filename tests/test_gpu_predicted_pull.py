"""The predicted perturbers' pull on chains of few members (prediction and pull in
one kernel) and of more (in two)."""
import numpy as np
import pytest

from gpu_helpers import hernquist32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [0, 1, 300, 5000])
@pytest.mark.parametrize("n_chain", [1, 8, 9, 40])
def test_predicted_pull(n_chain, k):
    """Against the same sums in numpy's FP64: positions predicted with one rounding
    an operation are equal, the sums of at most 5000 terms differ by their order
    and by fused operations, some 10^-13 of the sum of the terms' sizes."""
    import torch
    from paper_1507_01009_gb300 import rv
    n, dt = 20000, 1.5e-3
    p32, m32 = hernquist32(n, 61)
    g = np.random.default_rng(62 + n_chain)
    v32 = g.normal(0, 0.3, (3, n)).astype(np.float32)
    cm = g.uniform(0.5, 1.5, n_chain) * 1e-3
    cx = g.normal(0, 1e-3, (n_chain, 3))
    S = rv.System(p32, v32, m32, chain_m=cm, chain_x=cx, chain_v=np.zeros((n_chain, 3)), pert_mode=2, pert_k=k)
    ctx = rv.Context(n)
    ctx.system_forces(S)
    at = cx + g.normal(0, 1e-3, (n_chain, 3))
    a, pot = ctx.chain_perturber_forces(S, dt, torch.from_numpy(at).cuda())
    ctx.sync_status()
    centre = ((cm[:, None] * cx).sum(0) / cm.sum()).astype(np.float32)
    d = p32 - centre[:, None]
    near = np.argsort((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2], kind="stable")[:k]
    xp = p32[:, near].astype(np.float64) + v32[:, near].astype(np.float64) * dt
    m = m32[near].astype(np.float64)
    for j in range(n_chain):
        r = xp - at[j][:, None]
        d = np.sqrt((r * r).sum(0))
        t = m * r / d ** 3
        assert np.all(np.abs(a.cpu().numpy()[3 * j:3 * j + 3] - t.sum(1)) <= 1e-12 * np.abs(t).sum(1))
        assert abs(float(pot[j]) + (m / d).sum()) <= 1e-12 * (m / d).sum()
