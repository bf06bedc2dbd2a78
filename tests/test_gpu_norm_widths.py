"""GPU tests of the pre-norm forward at the widths where its form changes (how many 16-byte chunks a lane keeps in
registers, and none), with row counts that do not fill a block and a row stride wider than the row."""
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


@pytest.mark.parametrize("dtype,n,d", [(torch.bfloat16, n, d) for n, d in (
    (37, 16), (37, 504), (16, 512), (19, 520), (33, 1024), (21, 1032), (35, 2048), (17, 2056), (19, 4096), (18, 4104),
    (17, 8192), (16, 8200), (19, 16384), (17, 16392))] + [(torch.float32, n, d) for n, d in (
        (37, 20), (19, 256), (18, 260), (21, 1024), (17, 2052), (16, 4100))])
@pytest.mark.parametrize("kind", [B.NORM_RMS, B.NORM_LAYER])
def test_norm_forward_widths(dev, dtype, n, d, kind):
    g = torch.Generator(device=dev)
    g.manual_seed(n + d)
    wide = torch.randn(n, d + 16, generator=g, device=dev) * 3 + 1.5
    X = wide.to(dtype)[:, :d]
    gamma = (1 + 0.2 * torch.randn(d, generator=g, device=dev)).to(dtype)
    beta = (0.3 * torch.randn(d, generator=g, device=dev)).to(dtype) if kind == B.NORM_LAYER else None
    A, rstd, mean, *_ = B.compress_prenorm(X, gamma, beta, 1e-5, kind, 16)
    x = X.double()
    mu = x.mean(1, keepdim=True) if kind == B.NORM_LAYER else torch.zeros(n, 1, dtype=torch.float64, device=dev)
    rs = 1 / torch.sqrt((x - mu).square().mean(1, keepdim=True) + 1e-5)
    want = (x - mu) * rs * gamma.double() + (beta.double() if beta is not None else 0)
    # fp32 statistics over d entries, then one rounding of the result (bf16: 2^-9 of the value)
    tol = 1e-5
    assert float((rstd.double() - rs[:, 0]).abs().max() / rs.max()) <= tol
    if kind == B.NORM_LAYER:
        assert float((mean.double() - mu[:, 0]).abs().max()) <= tol
    err = (A.double() - want).abs() - (2.0 ** -8 if dtype == torch.bfloat16 else 0.0) * want.abs()
    assert float(err.max()) <= 1e-4
