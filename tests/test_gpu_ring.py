"""GPU tests of the operand ring of the tensor-core kernels: numbers of K blocks around the number of stages, operands that
come in whole panels of 64 columns (one load for all) and in single boxes, and loads that are issued ahead of the wait for
the previous kernel."""
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


@pytest.mark.parametrize("a_mn,b_mn", [(False, False), (False, True), (True, True)])
@pytest.mark.parametrize("m,n", [(64, 64), (64, 320), (96, 192), (128, 72), (320, 256), (256, 328), (448, 512), (600, 384)])
@pytest.mark.parametrize("k", [8, 200, 832, 1600])     # 1, 4, 13 and 25 K blocks: one stage, a part of the ring, more than it holds
def test_panels_and_stages(dev, m, n, k, a_mn, b_mn):
    g = torch.Generator(device=dev)
    g.manual_seed(m + 3 * n + 7 * k)
    a = torch.randn(*((k, m) if a_mn else (m, k)), generator=g, device=dev).bfloat16()
    b = torch.randn(*((k, n) if b_mn else (n, k)), generator=g, device=dev).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    C = B.debug_gemm([a], [b], m, n, k, a_mn, b_mn, out_mode=B.OUT_F32, engine=1, status=status).double()
    assert int(status.item()) == 0
    a, b = (a.t() if a_mn else a).double(), (b if b_mn else b.t()).double()
    # fp32 accumulation with truncation: 2^-23 of the running sum per instruction of sixteen products
    assert float((C - a @ b).abs().max() / (a.abs() @ b.abs()).max()) <= (k / 16 + 1) * 2.0 ** -23 + 1e-6


# up to 64 rows half a tile of A is loaded; the accumulator's other rows come from what the stage held
@pytest.mark.parametrize("m", [8, 40, 56, 64, 72])
@pytest.mark.parametrize("k", [72, 640, 1600])
@pytest.mark.parametrize("a_mn,b_mn", [(False, False), (True, True)])
def test_products_of_few_rows(dev, m, k, a_mn, b_mn):
    g = torch.Generator(device=dev)
    g.manual_seed(m + k)
    n = 152
    a = torch.randn(*((k, m) if a_mn else (m, k)), generator=g, device=dev).bfloat16()
    b = torch.randn(*((k, n) if b_mn else (n, k)), generator=g, device=dev).bfloat16()
    ad, bd = (a.t() if a_mn else a).double(), (b if b_mn else b.t()).double()
    for splits in (1, 3):
        status = torch.zeros(1, dtype=torch.int32, device=dev)
        C = B.debug_gemm([a], [b], m, n, k, a_mn, b_mn, out_mode=B.OUT_F32, engine=1, splits=splits, status=status).double()
        assert int(status.item()) == 0
        C = C.sum(0) if splits > 1 else C
        # fp32 accumulation with truncation: 2^-23 of the running sum per instruction of sixteen products
        assert float((C - ad @ bd).abs().max() / (ad.abs() @ bd.abs()).max()) <= (k / 16 + 4) * 2.0 ** -23


@pytest.mark.parametrize("m", [72, 136, 1000, 1024])   # (1024: whole panels, one term after the other)
@pytest.mark.parametrize("n", [16, 24, 48, 96, 112])
@pytest.mark.parametrize("k", [200, 256, 336, 512, 1600])
def test_terms_that_share_their_first_operand(dev, m, n, k):
    g = torch.Generator(device=dev)
    g.manual_seed(m + 3 * n + 7 * k)
    a = torch.randn(k, m, generator=g, device=dev).bfloat16()
    b = [torch.randn(k, n, generator=g, device=dev).bfloat16() for _ in range(3)]   # of one size: each term counts in full
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    C = B.debug_gemm([a, a, a], b, m, n, k, True, True, out_mode=B.OUT_F32, engine=1, status=status).double()
    assert int(status.item()) == 0
    want = a.t().double() @ (b[0].double() + b[1].double() + b[2].double())
    size = a.t().double().abs() @ (b[0].double().abs() + b[1].double().abs() + b[2].double().abs())
    # fp32 accumulation with truncation: 2^-23 of the running sum per instruction of sixteen products
    assert float((C - want).abs().max() / size.max()) <= (3 * k / 16 + 3) * 2.0 ** -23


@pytest.mark.parametrize("n,d,r,t", [(1024, 768, 64, 0), (5003, 1000, 336, 0), (4096, 2048, 128, 1), (16384, 1024, 256, 0)])
def test_inputs_written_right_before_the_call(dev, n, d, r, t):
    """X, V and grad_A are written by a kernel of the same stream right in front of the call, over other values: the results
    have the bits of a call that starts on an idle device."""
    g = torch.Generator(device=dev)
    g.manual_seed(n + r)
    make = lambda *s: torch.randn(*s, generator=g, device=dev).bfloat16()
    X0, G, E0, gamma = make(n, d), make(n, 64), make(n, d), make(d)
    X, E = torch.empty_like(X0), torch.empty_like(E0)
    ws = B.alloc_workspace(B.make_desc(X, r), dev)

    def run(wait):
        E.copy_(E0)
        X.copy_(X0)
        if wait:
            torch.cuda.synchronize()
        U, V, _ = B.compress(X, r, seed=3, ws=ws, power_iters=t)
        V.mul_(0.5)
        if wait:
            torch.cuda.synchronize()
        dW = B.weight_grad(U, V, G, ws=ws)
        rstd = torch.full((n,), 0.5, device=dev)
        if wait:
            torch.cuda.synchronize()
        return U, V, dW, B.prenorm_backward(U, V, gamma, rstd, E, ws=ws)

    want = run(True)
    for _ in range(5):
        X.fill_(7.0)
        E.fill_(7.0)
        for x, y in zip(run(False), want):
            assert torch.equal(x, y)


@pytest.mark.parametrize("out", [B.OUT_BF16, B.OUT_SPLIT, B.OUT_F32])
@pytest.mark.parametrize("n", [16, 48, 80, 96, 176, 240, 264, 336, 488, 1000])
@pytest.mark.parametrize("m", [40, 130, 300, 1111])
def test_output_widths(dev, m, n, out):
    """Widths that fill no staging box: the box is clipped at the edge of the matrix, or the tile is widened to whole boxes."""
    g = torch.Generator(device=dev)
    g.manual_seed(m + n)
    k = 200
    a = torch.randn(m, k, generator=g, device=dev).bfloat16()
    b = torch.randn(n, k, generator=g, device=dev).bfloat16()
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    C = B.debug_gemm([a], [b], m, n, k, False, False, out_mode=out, engine=1, status=status)
    assert int(status.item()) == 0
    pair = out == B.OUT_SPLIT
    C = C[0].double() + C[1].double() if pair else C.double()
    want, scale = a.double() @ b.double().t(), a.double().abs() @ b.double().abs().t()
    unit = 2.0 ** -8 if out == B.OUT_BF16 else (2.0 ** -16 if pair else 0.0)
    # fp32 accumulation with truncation (2^-23 of the running sum per instruction), then the rounding of the output
    assert float(((C - want).abs() - unit * want.abs()).max() / scale.max()) <= (k / 16 + 1) * 2.0 ** -23 + 1e-6
