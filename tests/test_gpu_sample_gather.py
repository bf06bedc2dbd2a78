"""GPU tests of the kernel that samples rows and gathers them: one and several rounds of 256 candidates, a rank at the edge
of a round, samples that are a permutation of all rows, copies smaller and larger than one sweep of the grid (592 CTAs of 256
threads, four 16-byte pieces each).  Indices and gathered bytes are exact."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
from oracle import loract_oracle as orc
from paper_2509_23472_b200 import binding as B, joint

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    entry.build()
    B.lib()
    return torch.device("cuda:0")


@pytest.mark.parametrize("n,d,r", [(16, 64, 16), (300, 16, 16), (256, 264, 256), (100000, 256, 256), (300, 280, 272),
                                   (512, 520, 512), (9000, 2376, 512), (2000, 11008, 448)])
def test_indices_and_rows_are_exact(dev, n, d, r):
    g = torch.Generator(device=dev)
    g.manual_seed(n + d)
    X = torch.randn(n, d, generator=g, device=dev).bfloat16()
    want = orc.sample_indices(n, r, seed=5, call_id=n)
    shard = joint.JointShard(X, n, 0, r, seed=5, call_id=n)
    S = shard.sample_rows()
    torch.cuda.synchronize()
    assert np.array_equal(shard.idx.cpu().numpy().astype(np.int64), want)
    assert torch.equal(S.view(torch.int16), X[torch.as_tensor(want, device=dev)].view(torch.int16))
    row0, rows = n // 3, n // 2
    part = joint.JointShard(X[row0:row0 + rows].contiguous(), n, row0, r, seed=5, call_id=n) if rows >= r else None
    if part is not None:
        Sp = part.sample_rows()
        inside = torch.as_tensor((want >= row0) & (want < row0 + rows), device=dev)
        assert torch.equal(Sp.view(torch.int16), torch.where(inside[:, None], S, torch.zeros_like(S)).view(torch.int16))
