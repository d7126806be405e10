"""The network's gradient kernel: its activations' rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rvmod():
    from paper_1507_01009_gb300 import rv
    rv.load()
    return rv


def test_activations_are_the_rounded_quotient(rvmod):
    """Layer 1's activations are SiLU(z) = z / (1 + e^-z) in FP32, rounded to
    bfloat16, not z times a rounded 1 / (1 + e^-z): at 64 values of z where the two
    fall on different sides of a bfloat16 rounding. One row of zeros, so z is the
    bias; dW2[k][j] / db2[j] is activation k up to one FP32 rounding, which its
    eight bits survive."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    z = torch.rand(1 << 25, generator=g, device="cuda") * 12.0 - 6.0
    e = 1.0 + torch.exp(-z)
    want, product = (z / e).bfloat16(), (z * (1.0 / e)).bfloat16()
    at = torch.nonzero(want != product).flatten()[:64]
    assert at.numel() == 64
    mlp = rvmod.Mlp(seed=3)
    mlp.master()["b1"].copy_(z[at])
    grad, _ = mlp.gradient(torch.zeros(1, 16, device="cuda"), torch.full((1, 3), 0.5, device="cuda"))
    o, part = 0, {}
    for name, shape in rvmod.MLP_LAYOUT:
        size = int(np.prod(shape))
        part[name] = grad[o:o + size].view(*shape).double()
        o += size
    j = int(part["b2"].abs().argmax())
    got = (part["W2"][:, j] / part["b2"].flatten()[j]).float().bfloat16()
    assert torch.equal(got, want[at])


@pytest.mark.parametrize("n", [1, 64, 65, 1025, "tile more than SMs", 65533])
def test_gradient_over_several_tiles_a_block(rvmod, n):
    """One row, tiles of 64 rows and a ragged one, more than one block's partials a
    run of the reduction (from 1025 rows), several tiles a block (one row more
    than 64 for every SM; 65533). Against the FP64 oracle on the same bfloat16
    weights. The two differ by the FP32 sums (about 1e-7 of the norm) and by
    activations that fall on different sides of a bfloat16 rounding: 2^-8 of an
    activation, at most one in some 10^4 of them, 10^-6 on average and for one row
    (64 + 64 activations, one of them moving) up to 2^-8 / 8 in the worst case."""
    import torch

    import ics
    import oracle
    if n == "tile more than SMs":
        n = 64 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    mlp = rvmod.Mlp(seed=16)
    g = ics.rng(n)
    X = np.zeros((n, 16), dtype=np.float32)
    X[:, :14] = g.normal(0, 1, (n, 14))
    T = g.normal(0, 0.5, (n, 3)).astype(np.float32)
    params = {k: v.detach().cpu().numpy().astype(np.float64) for k, v in mlp.master().items()}
    lo, go = oracle.mlp_loss_grad(params, X.astype(np.float64), T.astype(np.float64))
    want = np.concatenate([go[k].ravel() for k, _ in rvmod.MLP_LAYOUT])
    x, t = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    grad, loss = mlp.gradient(x, t)
    again, _ = mlp.gradient(x, t)
    assert torch.equal(grad, again)   # a fixed order of sums
    got = grad.cpu().numpy().astype(np.float64)
    tol = 1e-4 if n > 1000 else 1e-3
    assert abs(float(loss) / lo - 1) <= tol
    assert np.linalg.norm(got - want) <= tol * np.linalg.norm(want)
    assert np.all(got[want == 0.0] == 0.0)
    o, part = 0, {}
    for name, shape in rvmod.MLP_LAYOUT:
        size = int(np.prod(shape))
        part[name] = got[o:o + size].reshape(shape)
        o += size
    # the padding has no gradient
    assert not part["W1"][14:].any() and not part["W3"][:, 3:].any() and not part["b3"].ravel()[3:].any()
