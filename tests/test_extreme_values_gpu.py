"""Values at the ends of the number range: MoE intermediates whose requantisation scale underflows."""
import pytest
import torch

import oracle
from paper_2604_18616_b200 import inputs

from test_moe_gpu import check as check_moe, run_gpu as run_moe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shrink", [1e-21, 1e-22, 1e-23])
def test_moe_groups_whose_scale_underflows(shrink):
    """Intermediates of about shrink^2 / 2: the largest of a group over 448 is a subnormal or zero in fp32."""
    args = list(inputs.make_moe_inputs(inputs.MoeWorkload("tiny", 40, 256, 256, 4, 2, 3)))
    args[1] = args[1] * shrink
    y = run_moe(args)
    assert torch.isfinite(y).all()
    check_moe(y, oracle.moe_fwd(*[t.numpy() for t in args]), args, "shrink %g" % shrink)
