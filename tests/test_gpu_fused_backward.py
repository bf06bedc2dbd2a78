"""GPU tests of the backward kernels that combine a rebuilt tile with another matrix (activation backward, pre-norm
backward) at the edges of their tiles: fewer rows or columns than one tile, ragged rows and columns, one and many tiles per
SM pair, the shortest and the longest contraction, a row stride wider than the row.  Reference: the gradient equations in
float64 from the same factors."""
import pytest
import torch

import __graft_entry__ as entry
from paper_2509_23472_b200 import binding as B

pytestmark = pytest.mark.gpu

SHAPES = [(16, 16, 16), (40, 264, 16), (127, 136, 64), (257, 1000, 80), (300, 2056, 256), (1024, 520, 512),
          (5003, 776, 128), (2500, 4104, 512), (9000, 1032, 16)]


@pytest.fixture(scope="module")
def dev():
    entry.build()
    B.lib()
    return torch.device("cuda:0")


def draw(dev, n, d, r, seed):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    U = (torch.randn(n, r, generator=g, device=dev) / n ** 0.5).bfloat16()
    V = (torch.randn(r, d, generator=g, device=dev) * (2.0 * n / r) ** 0.5).bfloat16()    # rebuilt entries of a few units
    wide = torch.full((n, d + 24), 7.0, device=dev, dtype=torch.bfloat16)
    wide[:, :d] = torch.randn(n, d, generator=g, device=dev).bfloat16()
    return U, V, wide[:, :d], g


def check(got, want, terms_rms):
    """One rounding to bf16 (2^-9 of the value at most), and the fp32 arithmetic before it."""
    err = (got.double() - want).abs()
    assert float((err - 2.0 ** -8 * want.abs()).max()) <= 1e-3 * terms_rms
    assert float(err.norm() / want.norm()) <= 2.5e-3


@pytest.mark.parametrize("n,d,r", SHAPES)
@pytest.mark.parametrize("kind", [B.ACT_SILU, B.ACT_GELU])
def test_activation_backward_at_tile_edges(dev, n, d, r, kind):
    U, V, gZ, _ = draw(dev, n, d, r, n + d + r)
    got = B.activation_backward(U, V, gZ, kind)
    a = U.double() @ V.double()
    if kind == B.ACT_SILU:
        s = torch.sigmoid(a)
        f = s * (1 + a * (1 - s))
    else:
        f = 0.5 * (1 + torch.erf(a / 2 ** 0.5)) + a * torch.exp(-a * a / 2) / (2 * torch.pi) ** 0.5
    check(got, gZ.double() * f, 1.0)
    again = B.activation_backward(U, V, gZ, kind)
    assert torch.equal(again, got)


@pytest.mark.parametrize("n,d,r", SHAPES)
def test_prenorm_backward_at_tile_edges(dev, n, d, r):
    U, V, gA, g = draw(dev, n, d, r, 3 * n + d + r)
    gamma = (1.0 + 0.2 * torch.randn(d, generator=g, device=dev)).bfloat16()
    rstd = torch.rand(n, generator=g, device=dev) + 0.5
    got = B.prenorm_backward(U, V, gamma, rstd, gA)
    A, gm, ga = U.double() @ V.double(), gamma.double(), gA.double()
    inner = (ga * A).mean(dim=1, keepdim=True)
    want = rstd.double()[:, None] * (ga * gm - A / gm * inner)
    assert bool(torch.isfinite(got).all())
    # two terms of opposite sign: the fp32 error is that of the larger one
    check(got, want, float((ga * gm).square().mean().sqrt() + (A / gm * inner).square().mean().sqrt()))


def test_nothing_is_written_past_the_row(dev):
    n, d, r = 300, 264, 32
    U, V, gZ, _ = draw(dev, n, d, r, 5)
    gX = torch.empty(n, d + 24, device=dev, dtype=torch.bfloat16).fill_(3.0)
    desc = B.Desc(n, d, d + 24, r, 0, B.BF16, 0, 0, 0)
    import ctypes
    B._check(B.lib().loract_activation_backward(ctypes.byref(desc), B._ptr(U), B._ptr(V), B._ptr(gZ), B.ACT_SILU,
                                                B._ptr(gX), B._stream(dev)), "loract_activation_backward")
    torch.cuda.synchronize()
    assert bool((gX[:, d:] == 3.0).all())
    assert torch.equal(gX[:, :d], B.activation_backward(U, V, gZ, B.ACT_SILU))


# up to 64 rows the one-CTA kernel loads half tiles of A; the kernel of the fused epilogues takes whole ones at every size
@pytest.mark.parametrize("n", [16, 40, 63, 64, 65])
@pytest.mark.parametrize("d,r", [(136, 16), (1000, 16)])
def test_few_rows(dev, n, d, r):
    U, V, gZ, g = draw(dev, n, d, r, 5 * n + d)
    a = U.double() @ V.double()
    s = torch.sigmoid(a)
    check(B.activation_backward(U, V, gZ, B.ACT_SILU), gZ.double() * s * (1 + a * (1 - s)), 1.0)
    gelu = 0.5 * (1 + torch.erf(a / 2 ** 0.5)) + a * torch.exp(-a * a / 2) / (2 * torch.pi) ** 0.5
    check(B.activation_backward(U, V, gZ, B.ACT_GELU), gZ.double() * gelu, 1.0)
    gamma = (1.0 + 0.2 * torch.randn(d, generator=g, device=dev)).bfloat16()
    rstd = torch.rand(n, generator=g, device=dev) + 0.5
    ws = B.alloc_workspace(B.make_desc(gZ, r), dev)
    got = B.prenorm_backward(U, V, gamma, rstd, gZ, ws=ws)
    assert B.read_device_status(ws) == 0
    gm, ga = gamma.double(), gZ.double()
    inner = (ga * a).mean(dim=1, keepdim=True)
    check(got, rstd.double()[:, None] * (ga * gm - a / gm * inner),
          float((ga * gm).square().mean().sqrt() + (a / gm * inner).square().mean().sqrt()))
