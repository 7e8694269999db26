"""Kernels that run as thread-block clusters, at the edges of their dispatch rules (through the C ABI)."""
import pytest
import torch

import paper_2609_34272_b200 as g

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,d", [(1, 64), (7, 128), (8, 64), (513, 64), (4095, 64), (4097, 64), (2049, 128), (9000, 64)])
def test_key_smoothing_at_the_edges_of_its_row_split(rows, d):
    # one row, fewer rows than CTAs, the last row kept in registers, the first rows read twice.  FP32 sums of n values in
    # any order lie within n 2^-24 of each other relative to the sum of magnitudes; one BF16 step of the output covers it.
    gen = torch.Generator().manual_seed(rows + d)
    X = (torch.randn(3, rows, d, generator=gen) + 4.0 * torch.randn(3, 1, d, generator=gen)).to(torch.bfloat16)
    want = (X.float() - X.double().mean(dim=1, keepdim=True).float())
    buf = X.cuda()
    g.gproj_key_smooth(buf, Y=buf, cu_seqlens=[0, 0, rows, rows])
    got = buf.float().cpu()
    assert torch.all((got - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -20 * X.float().abs().max())
