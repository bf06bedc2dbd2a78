"""GPU tests of the weight gradient whose second product adds up T = U^T G for itself: rank times consumers at and above the
limit of that kernel, one and several groups of four columns, d inside a 128-byte column tile and ragged."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2509_23472_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    entry.build()
    B.lib()
    return torch.device("cuda:0")


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n,d,r,g", [(16, 16, 16, 4), (40, 40, 16, 8), (700, 776, 64, 16), (700, 520, 64, 24),
                                     (700, 520, 64, 28), (513, 392, 384, 4), (300, 200, 16, 96), (300, 136, 16, 100),
                                     (5000, 264, 48, 20), (9000, 72, 16, 12), (2000, 1000, 96, 16), (700, 520, 32, 19)])
def test_small_weight_gradient(dev, n, d, r, g, dtype):
    gen = torch.Generator(device=dev)
    gen.manual_seed(n + g)
    U, V, G = ((torch.randn(*s, generator=gen, device=dev)).to(dtype) for s in ((n, r), (r, d), (n, (g + 7) // 8 * 8)))
    G = G[:, :g]
    want = V.double().t() @ (U.double().t() @ G.double())
    # two sums in fp32, of n and of r terms, against the sum of the terms' sizes
    bound = 2.0 ** -23 * (4.0 + n ** 0.5 + r ** 0.5) * (V.double().abs().t() @ (U.double().abs().t() @ G.double().abs()))
    dW = B.weight_grad(U, V, G)
    assert bool(((dW.double() - want).abs() <= bound).all())
    again = B.weight_grad(U, V, G, dW=dW.clone(), accumulate=True)
    assert bool(((again.double() - 2 * want).abs() <= 2 * bound + 2.0 ** -23 * 2 * want.abs()).all())
