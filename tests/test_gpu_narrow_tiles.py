"""GPU tests of products whose tiles are as narrow as one round of the SMs allows: few rows and many columns (the test matrix
L^-1 T), row counts on either side of the one-CTA and two-CTA kernels, column counts on either side of where 64, 128 and
256 columns take over, ragged ends; and small results in partial sums (Gram matrices), split counts on either side of the same lines.
Reference: the product in float64."""
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


@pytest.mark.parametrize("m,n", [(16, 264), (64, 1000), (64, 9472), (64, 9480), (96, 776), (128, 11008), (136, 4736), (136, 4744),
                                 (248, 5120), (256, 264), (256, 9472), (256, 9480), (336, 1000), (336, 4744), (512, 11008)])
def test_tiles_of_few_rows(dev, m, n):
    g = torch.Generator(device=dev)
    g.manual_seed(m + n)
    L = torch.randn(m, m, generator=g, device=dev).tril()
    hi = L.bfloat16()
    lo = (L - hi.float()).bfloat16()
    T = torch.randn(m, n, generator=g, device=dev).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    want = (hi.double() + lo.double()) @ T.double()
    got = B.debug_gemm([hi, lo], [T, T], m, n, m, False, True, out_mode=B.OUT_BF16, engine=1, status=status).double()
    assert int(status.item()) == 0
    # one rounding to bf16 (2^-9 of the value); the sum over m products in fp32 is far below 1e-3 of the row's size
    assert float(((got - want).abs() - 2.0 ** -8 * want.abs()).max()) <= 1e-3 * m ** 0.5
    assert float((got - want).norm() / want.norm()) <= 2.5e-3


@pytest.mark.parametrize("mn_major", [False, True])
@pytest.mark.parametrize("l,splits", [(16, 3), (48, 2), (64, 148), (64, 74), (96, 40), (128, 37), (128, 38), (128, 75), (160, 20),
                                      (192, 12), (256, 9), (256, 18), (256, 37), (256, 38), (272, 4), (336, 4), (336, 7), (400, 6), (512, 4),
                                      (512, 9), (512, 10)])
def test_partial_sums_of_small_results(dev, l, splits, mn_major):
    g = torch.Generator(device=dev)
    g.manual_seed(l + splits)
    k = 64 * 2 * splits - 40
    a = torch.randn(*((k, l) if mn_major else (l, (k + 7) // 8 * 8)), generator=g, device=dev).bfloat16()
    k = a.shape[0] if mn_major else a.shape[1]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    parts = B.debug_gemm([a], [a], l, l, k, mn_major, mn_major, engine=1, splits=splits, status=status)
    assert int(status.item()) == 0
    x = a.double().t() if mn_major else a.double()
    per = (k + 63) // 64
    per = (per + splits - 1) // splits * 64
    for s in (0, splits - 1):                                  # K range s of the contraction
        want = x[:, s * per:(s + 1) * per] @ x[:, s * per:(s + 1) * per].t()
        # products of bf16 are exact in fp32; at most 128 of them are added, each addition off by 2^-23 of the running sum
        assert float((parts[s].double() - want).abs().max()) <= 128 * 2.0 ** -23 * float(want.diagonal().max())
