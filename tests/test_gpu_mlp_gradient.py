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
