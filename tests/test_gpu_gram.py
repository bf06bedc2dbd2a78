"""GPU tests of the Gram product above 256 columns: widths and row counts around the edges of its tiles, panels and ranges,
against float64, and the application of a triangular factor whose zero blocks are left out."""
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


@pytest.mark.parametrize("n,l", [(264, 264), (320, 320), (512, 512), (600, 336), (1000, 384), (4095, 448), (5003, 336),
                                 (9408, 512), (16384, 320), (32768, 512), (40001, 504)])
def test_gram_above_256_columns(dev, n, l):
    g = torch.Generator(device=dev)
    g.manual_seed(n + l)
    Y = torch.randn(n, l, generator=g, device=dev) * torch.logspace(0, -2, l, device=dev)   # columns of different norms
    Yh = Y.bfloat16()
    Yl = (Y - Yh.float()).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    W = B.debug_gram(Yh, Yl, status)
    assert int(status.item()) == 0
    assert torch.equal(W, W.t())
    Yd = Yh.double() + Yl.double()
    want = Yd.t() @ Yd
    scale = want.diagonal().sqrt()
    # a chain is at most sixteen instructions of 2^-23, the partial sums of every 64 rows are added in fp32 (2^-24 each; of
    # them at most 1 / 22 in one running sum, and the sums of the ranges): bounded against |Y|^T |Y|, relative to the diagonal
    err = ((W.double() - want).abs() / (scale[:, None] * scale[None, :])).max()
    assert float(err) <= (16 + n / 64 / 22 + 32) * 2.0 ** -23


@pytest.mark.parametrize("n,l", [(264, 264), (600, 336), (5003, 336), (4095, 448), (16384, 512), (40001, 504)])
def test_every_product_of_the_gram_matrix_counts(dev, n, l):
    g = torch.Generator(device=dev)
    g.manual_seed(n + 2 * l)
    # two independent matrices of one size: each of the four products, the halved sum and the mirrored tile are of order one
    A, Bm = (torch.randn(n, l, generator=g, device=dev).bfloat16() for _ in range(2))
    W = B.debug_gram(A, Bm).double()
    Yd = A.double() + Bm.double()
    size = (A.double().abs() + Bm.double().abs())
    err = ((W - Yd.t() @ Yd).abs() / (size.t() @ size)).max()
    assert float(err) <= (16 + n / 64 / 22 + 32) * 2.0 ** -23


@pytest.mark.parametrize("n,l", [(4096, 272), (16384, 320), (32768, 512)])
def test_diagonal_of_the_gram_matrix_has_no_bias(dev, n, l):
    g = torch.Generator(device=dev)
    g.manual_seed(n + 3 * l)
    Y = torch.randn(n, l, generator=g, device=dev)
    Yh = Y.bfloat16()
    Yl = (Y - Yh.float()).bfloat16()
    want = (Yh.double() + Yl.double()).square().sum(0)
    bias = ((B.debug_gram(Yh, Yl).diagonal().double() - want) / want).mean()
    # twelve instructions of a block truncate a running sum that grows from nothing: at most half of 12 * 2^-23 = 7.2e-7 of it.
    # Without the product of the low parts it would be 2.8e-6, with chains of thirty blocks 4e-6
    assert abs(float(bias)) <= 8e-7


@pytest.mark.parametrize("n,d,r", [(4096, 768, 272), (16384, 768, 512), (9000, 640, 448), (700, 11008, 512)])
def test_steps_with_a_triangular_factor_in_two_tiles(dev, n, d, r):
    """Shapes at which the application of L^-T (many rows) or the test matrix (many columns) takes two tiles per CTA pair."""
    g = torch.Generator(device=dev)
    g.manual_seed(r)
    X = (torch.randn(n, 600, generator=g, device=dev) * torch.logspace(0, -2, 600, device=dev) @
         torch.randn(600, d, generator=g, device=dev) + 1e-2 * torch.randn(n, d, generator=g, device=dev)).bfloat16()
    U, V, idx = B.compress(X, r, seed=5)
    Xd = X.double()
    S = Xd[idx.long()]
    Q = torch.linalg.solve_triangular(torch.linalg.cholesky(S @ S.t()), S @ Xd.t(), upper=False).t()
    for _ in range(2):
        Q = torch.linalg.solve_triangular(torch.linalg.cholesky(Q.t() @ Q), Q.t(), upper=False).t()
    P = Q @ (Q.t() @ Xd)
    err = float((P - Xd).norm() / Xd.norm())
    # two roundings of 2^-9 and a small slope for the trailing directions, as in the parity tests
    assert float((U.double() @ V.double() - P).norm() / Xd.norm()) <= 2.0 ** -8 + err / 100
