"""Values at the ends of the number range: MoE intermediates whose requantisation scale underflows, gates far below the point
where exp(-gate) overflows, and infinities among the values of a split-KV call."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_18616_b200 import inputs

from test_moe_gpu import check as check_moe, run_gpu as run_moe
from test_splitkv_gpu import rand_qkv, run_split

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shrink", [1e-21, 1e-22, 1e-23])
def test_moe_groups_whose_scale_underflows(shrink):
    """Intermediates of about shrink^2 / 2: the largest of a group over 448 is a subnormal or zero in fp32."""
    args = list(inputs.make_moe_inputs(inputs.MoeWorkload("tiny", 40, 256, 256, 4, 2, 3)))
    args[1] = args[1] * shrink
    y = run_moe(args)
    assert torch.isfinite(y).all()
    check_moe(y, oracle.moe_fwd(*[t.numpy() for t in args]), args, "shrink %g" % shrink)


@pytest.mark.parametrize("sign", [-1.0, 1.0])
def test_moe_gates_of_any_size(sign):
    """silu(z) = z / (1 + exp(-z)) vanishes for large negative z, however large.  The up value of a token is the size of its
    gate, brought back to the order of 1 by the scale of the up half's weights, so that a token tests one size of gate."""
    one, half = oracle.e4m3_encode(1.0), oracle.e4m3_encode(0.5)
    for size in (1e-3, 1.0, 20.0, 60.0, 86.5, 87.5, 88.5, 89.0, 104.0, 1e3, 1e10, 1e30, 1e38):
        T, C, F = 3, 128, 128
        xq = torch.zeros((T, C), dtype=torch.uint8)
        xq[:, 5] = one
        sx = torch.full((T, 1), size, dtype=torch.float32)
        w13q = torch.full((1, 2 * F, C), one, dtype=torch.uint8)
        w13q[0, :F] = oracle.e4m3_encode(sign)
        w13q[0, :F:3] = oracle.e4m3_encode(0.5 * sign)
        w13q[0, F::5] = half
        s13 = torch.tensor([1.0, 1.0 / size], dtype=torch.float32).view(1, 2, 1)
        w2q = torch.full((1, C, F), one, dtype=torch.uint8)
        s2 = torch.full((1, 1, 1), 1.0 / 128, dtype=torch.float32)
        ids, wts = torch.zeros((T, 1), dtype=torch.int32), torch.ones((T, 1), dtype=torch.float32)
        args = [xq, sx, w13q, s13, w2q, s2, ids, wts]
        ref = oracle.moe_fwd(*[t.numpy() for t in args])
        y = run_moe(args).double().numpy()
        # three roundings (an E4M3 code where two fp32 values straddle a tie: 2^-4; bf16: 2^-9); values below 1e-35 are
        # zero to fp32's exp(-z), which overflows
        assert np.all(np.abs(y - ref) <= 2.0 ** -4 * np.abs(ref) + 1e-35), "gates of %g: %g, oracle %g" % (
            sign * size, y[0, 0], ref[0, 0])


def test_infinite_value_in_the_last_of_an_odd_number_of_ranges():
    B, H, Sq, Sk, D, n_splits = 1, 2, 3, 384, 64, 3
    q, k, v = rand_qkv(11, B, H, H, Sq, Sk, D)
    v[0, :, Sk - 1, 7] = float("inf")
    o, lse = run_split(q, k, v, False, 0.125, n_splits)
    assert torch.isfinite(lse).all()
    assert torch.all(o[..., 7] == float("inf"))
    rest = [c for c in range(D) if c != 7]
    assert torch.isfinite(o[..., rest].float()).all()


@pytest.mark.parametrize("H,Hkv,Sq,Sk", [(2, 2, 200, 150), (16, 16, 200, 150), (4, 2, 60, 40)])  # row-wise merge; packed heads
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("n_splits", [1, 2])
def test_rows_without_keys_are_zero_whatever_the_values_are(n_splits, D, H, Hkv, Sq, Sk):
    # Sq > Sk, causal: the first rows see no key, but share their tile with rows that see infinite values
    q, k, v = rand_qkv(12, 1, H, Hkv, Sq, Sk, D)
    v[0, :, 10, 3] = float("inf")
    o, lse = run_split(q, k, v, True, 0.1, n_splits)
    assert torch.all(lse[:, :, :Sq - Sk] == float("-inf")) and torch.all(o[:, :, :Sq - Sk] == 0)
    assert torch.isfinite(lse[:, :, Sq - Sk:]).all() and torch.all(o[:, :, Sq - Sk + 10:, 3] == float("inf"))
