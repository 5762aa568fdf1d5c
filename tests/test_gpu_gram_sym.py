"""The Gram matrix of a block with itself forms the groups on and above the diagonal and mirrors
them: the same bits as with a copy of the block for the second operand, whose groups are all
formed.  One group, a partial second one, the eigensolver's three, the widest basis."""
import pytest
import torch

from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edge", [16, 40])
@pytest.mark.parametrize("rows", [3, 16, 17, 33, 48, 64])
def test_symmetric_groups_give_the_general_bits(edge, rows):
    need_gpu()
    ctx = rsx.Context((edge,) * 3, 0.3, "fp32")
    g = torch.Generator(device="cuda").manual_seed(rows)
    a = torch.randn((rows,) + (edge,) * 3, device="cuda", generator=g)
    S, G = ctx.gram(a, a), ctx.gram(a, a.clone())
    ctx.sync()
    assert torch.equal(S, G) and torch.equal(S, S.T)
