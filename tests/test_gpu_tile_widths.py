"""The width of a tile of a product, which depends on its shape alone: few rows and many columns (the test matrix L^-1 T, the
projection of few rows, Reconstruct of few tiles), small results in partial sums (Gram matrices, T = U^T G), row, column and split
counts on either side of every line; on the GPU, the products that the same rules reach beside the test matrix and the Gram matrices, and
every K range of the partial sums, against float64."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2509_23472_b200 import binding as B


@pytest.fixture(scope="module")
def built():
    entry.build()
    B.lib()


@pytest.fixture(scope="module")
def dev(built):
    return torch.device("cuda:0")


@pytest.mark.parametrize("m,n,width", [
    (16, 264, 64), (64, 1000, 64), (64, 9472, 64), (64, 9480, 128), (96, 776, 64), (128, 11008, 128), (136, 4736, 64), (136, 4744, 128),
    (248, 5120, 128), (256, 264, 128), (256, 9472, 128), (256, 9480, 192), (336, 1000, 128), (336, 4744, 192), (512, 11008, 256)])
def test_width_of_few_rows(built, m, n, width):
    assert B.debug_tile_width(m, n, m, False, True, 2, B.OUT_BF16) == width


# Rows of A of less than 128 bytes (rank 16, 32 or 48: A = U or L^-1), one CTA a tile: up to 64 tiles of 64 columns side by
# side, up to 80 of 128.
@pytest.mark.parametrize("m,n,k,mn_major,terms,width", [
    (16, 4096, 512, True, 1, 64), (16, 4104, 512, True, 1, 128), (48, 5120, 192, True, 1, 128), (16, 10240, 448, True, 1, 128),
    (16, 10248, 448, True, 1, 192), (32, 11008, 64, True, 1, 256), (64, 9472, 448, True, 1, 64),
    (96, 4096, 16, False, 1, 64), (96, 5120, 16, False, 1, 128), (200, 4096, 32, False, 1, 64), (200, 4104, 32, False, 1, 128),
    (200, 9472, 48, False, 1, 128), (128, 11008, 48, False, 1, 256), (128, 9472, 64, False, 1, 64), (255, 5120, 16, False, 1, 128),
    (256, 9472, 16, False, 1, 128), (16, 4096, 16, False, 2, 64), (16, 9472, 16, False, 2, 128), (32, 11008, 32, False, 2, 256)])
def test_width_where_rows_of_a_are_short(built, m, n, k, mn_major, terms, width):
    assert B.debug_tile_width(m, n, k, mn_major, True, terms, B.OUT_BF16) == width


# One term and the other operand orders and results that reach the same rule: Reconstruct (A K-major) and U^T X (both MN-major, bf16 or
# fp32); a pair of bf16 results.  (No product that the rule reaches adds to what is there.)
@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k,mn_major,out,width", [
    (64, 4096, 32, False, B.OUT_BF16, 64), (200, 4736, 96, False, B.OUT_BF16, 64), (200, 4744, 96, False, B.OUT_BF16, 128),
    (384, 4096, 128, False, B.OUT_BF16, 128), (384, 4744, 192, False, B.OUT_BF16, 192), (1000, 1000, 496, False, B.OUT_BF16, 128),
    (4090, 512, 256, False, B.OUT_BF16, 128), (9000, 264, 128, False, B.OUT_BF16, 192), (300, 776, 72, False, B.OUT_SPLIT, 128),
    (100, 1000, 72, False, B.OUT_SPLIT, 64), (100, 1000, 72, False, B.OUT_F32, 64),
    (64, 4096, 200, True, B.OUT_BF16, 64), (96, 9472, 448, True, B.OUT_F32, 64), (96, 9480, 448, True, B.OUT_F32, 128),
    (240, 1000, 500, True, B.OUT_F32, 64), (256, 768, 511, True, B.OUT_BF16, 128), (496, 3000, 510, True, B.OUT_F32, 128),
    (16, 1360, 500, True, B.OUT_BF16, 64), (16, 5120, 500, True, B.OUT_BF16, 128), (48, 9472, 192, True, B.OUT_F32, 128),
    (96, 5120, 16, False, B.OUT_BF16, 128)])
def test_other_products_of_few_tiles(dev, m, n, k, mn_major, out, width):
    assert B.debug_tile_width(m, n, k, mn_major, True, 1, out) == width
    g = torch.Generator(device=dev)
    g.manual_seed(m + n + k)
    up = (k + 7) // 8 * 8
    a = torch.randn(k, m, generator=g, device=dev).bfloat16() if mn_major else \
        torch.randn(m, up, generator=g, device=dev).bfloat16()[:, :k]
    b = torch.randn(k, n, generator=g, device=dev).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    got = B.debug_gemm([a], [b], m, n, k, mn_major, True, out_mode=out, engine=1, status=status)
    assert int(status.item()) == 0
    got = got[0].double() + got[1].double() if out == B.OUT_SPLIT else got.double()
    want = (a.double().t() if mn_major else a.double()) @ b.double()
    # exact products, k additions each off by 2^-23 of the running sum, at most the sum of the magnitudes; one rounding of the result
    sums = (a.double().abs().t() if mn_major else a.double().abs()) @ b.double().abs()
    rounding = {B.OUT_F32: 2.0 ** -23, B.OUT_BF16: 2.0 ** -8, B.OUT_SPLIT: 2.0 ** -16}[out]
    assert bool(((got - want).abs() <= k * 2.0 ** -23 * sums + rounding * want.abs()).all())


# (the width with both operands K-major, and with both MN-major)
@pytest.mark.gpu
@pytest.mark.parametrize("mn_major", [False, True])
@pytest.mark.parametrize("l,splits,widths", [
    (16, 3, (16, 16)), (48, 2, (48, 48)), (64, 148, (64, 64)), (64, 74, (32, 64)), (96, 40, (32, 96)), (96, 50, (96, 96)),
    (128, 37, (32, 64)), (128, 38, (64, 64)), (128, 74, (64, 64)), (128, 75, (128, 128)), (160, 14, (32, 160)), (160, 15, (160, 160)), (192, 12, (32, 64)),
    (256, 9, (32, 128)), (256, 18, (64, 128)), (256, 37, (128, 128)), (256, 38, (256, 256)), (272, 4, (32, 192)), (336, 4, (64, 192)),
    (336, 7, (128, 192)), (400, 6, (128, 256)), (512, 4, (64, 256)), (512, 9, (128, 256)), (512, 10, (256, 256))])
def test_partial_sums_of_small_results(dev, l, splits, widths, mn_major):
    g = torch.Generator(device=dev)
    g.manual_seed(l + splits)
    k = 64 * 2 * splits - 40
    a = torch.randn(*((k, l) if mn_major else (l, (k + 7) // 8 * 8)), generator=g, device=dev).bfloat16()
    k = a.shape[0] if mn_major else a.shape[1]
    assert B.debug_tile_width(l, l, k, mn_major, mn_major, 1, B.OUT_F32, splits) == widths[mn_major]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    parts = B.debug_gemm([a], [a], l, l, k, mn_major, mn_major, engine=1, splits=splits, status=status)
    assert int(status.item()) == 0
    x = a.double().t() if mn_major else a.double()
    per = (k + 63) // 64
    per = (per + splits - 1) // splits * 64
    for s in range(splits):                                    # K range s of the contraction
        want = x[:, s * per:(s + 1) * per] @ x[:, s * per:(s + 1) * per].t()
        # products of bf16 are exact in fp32; at most 128 of them are added, each addition off by 2^-23 of the running sum
        assert float((parts[s].double() - want).abs().max()) <= 128 * 2.0 ** -23 * float(want.diagonal().max())


# Rectangular results (the split sketch, T = U^T G) and three terms, the first two halved (the tall Gram matrix).
@pytest.mark.gpu
@pytest.mark.parametrize("m,n,splits,mn_major,terms,halve,width", [
    (500, 96, 4, False, 1, 0, 32), (512, 160, 7, False, 1, 0, 32), (512, 160, 8, False, 1, 0, 160), (520, 96, 4, False, 1, 0, 96),
    (200, 64, 5, False, 1, 0, 32), (256, 96, 16, True, 1, 0, 96), (64, 256, 30, True, 1, 0, 64), (64, 256, 40, True, 1, 0, 128),
    (200, 128, 37, True, 1, 0, 64), (200, 128, 38, True, 1, 0, 128), (256, 256, 37, True, 3, 2, 128), (128, 128, 64, True, 3, 2, 64),
    (64, 64, 20, True, 3, 2, 64)])
def test_partial_sums_rectangular_and_of_three_terms(dev, m, n, splits, mn_major, terms, halve, width):
    k = 64 * 2 * splits - 24
    assert B.debug_tile_width(m, n, k, mn_major, mn_major, terms, B.OUT_F32, splits) == width
    g = torch.Generator(device=dev)
    g.manual_seed(m + n + splits)
    a = [torch.randn(*((k, m) if mn_major else (m, k)), generator=g, device=dev).bfloat16() for _ in range(terms)]
    b = [torch.randn(*((k, n) if mn_major else (n, k)), generator=g, device=dev).bfloat16() for _ in range(terms)]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    parts = B.debug_gemm(a, b, m, n, k, mn_major, mn_major, engine=1, splits=splits, status=status, halve_at_term=halve)
    assert int(status.item()) == 0
    a64, b64 = ([x.double().t() if mn_major == (i == 0) else x.double() for x in t] for i, t in enumerate((a, b)))
    per = ((k + 63) // 64 + splits - 1) // splits * 64
    for s in range(splits):
        r = slice(s * per, (s + 1) * per)
        factor = [0.5 if t < halve else 1.0 for t in range(terms)]
        want = sum(f * (x[:, r] @ y[r]) for f, x, y in zip(factor, a64, b64))
        sums = sum(x[:, r].abs() @ y[r].abs() for x, y in zip(a64, b64))
        # 128 exact products a term, each addition off by 2^-23 of the running sum, at most the sum of the magnitudes
        assert bool(((parts[s].double() - want).abs() <= 128 * terms * 2.0 ** -23 * sums).all())
