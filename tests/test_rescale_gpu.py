"""Scores that rise from key to key, so that the running maximum moves, and the accumulator in TMEM is rescaled, at nearly every key
tile: in both attention kernels, through every entry point, at every width of the accumulator.  Oracle and tolerances are those of
the parity tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_18616_b200 import binding

import parity
from test_splitkv_gpu import rand_qkv, run_split

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(params=[binding.KERNEL_TWO_SUBTILES, binding.KERNEL_ONE_SUBTILE], autouse=True)
def kernel(request):
    assert binding.select_kernel(request.param) == binding.AVE_OK
    yield
    assert binding.select_kernel(binding.KERNEL_AUTO) == binding.AVE_OK


def rising(seed, B, H, Hkv, Sq, Sk, D, sign=1.0):
    """16 score units a key tile, more than the maximum may lag behind."""
    q, k, v = rand_qkv(seed, B, H, Hkv, Sq, Sk, D)
    q[..., 0] = sign * 4.0
    k[..., 0] = (torch.arange(Sk, dtype=torch.float32) * (D ** 0.5 / 32)).to(k.dtype)
    return q, k, v


@pytest.mark.parametrize("D", [64, 96, 128, 192, 256])
@pytest.mark.parametrize("Sq,Sk,causal", [(300, 700, False), (300, 300, True), (130, 900, True)])
def test_contiguous(Sq, Sk, causal, D):
    q, k, v = rising(Sq + Sk + D, 1, 4, 2, Sq, Sk, D)
    parity.check_full(q, k, v, causal, D ** -0.5, "rising scores %s" % ((Sq, Sk, causal, D),))
    q, k, v = rising(Sq + Sk + D, 1, 2, 2, Sq, Sk, D, sign=-1.0)
    parity.check_full(q, k, v, causal, -D ** -0.5, "rising scores, negative scale %s" % ((Sq, Sk, causal, D),))


@pytest.mark.parametrize("D", [64, 128, 256])
@pytest.mark.parametrize("causal", [False, True])
def test_variable_lengths(causal, D):
    lens, H, Hkv = [300, 1, 0, 513, 129], 4, 2
    parts = [rising(n + D, 1, H, Hkv, n, n, D) for n in lens]
    q, k, v = (torch.cat([p[i][0].permute(1, 0, 2) for p in parts]).contiguous() for i in range(3))
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32)
    o, lse = binding.ave_attn_fwd_varlen(q.to(DEV), k.to(DEV), v.to(DEV), cu.to(DEV), cu.to(DEV), max(lens), max(lens), causal=causal)
    assert binding.device_status() == (binding.AVE_OK, 0)
    for b, n in enumerate(lens):
        if n:
            o_ref, lse_ref = oracle.attn_fwd(*parts[b], causal, D ** -0.5)
            rows = slice(int(cu[b]), int(cu[b]) + n)
            parity.compare(o[rows].permute(1, 0, 2)[None].cpu(), lse[:, rows][None].cpu(), o_ref, lse_ref, "sequence %d" % b)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("Sq,causal", [(1, True), (100, False), (300, True)])
def test_split_keys(Sq, causal, D):
    q, k, v = rising(Sq + D, 1, 4, 2, Sq, 1500, D)
    o, lse = run_split(q, k, v, causal, D ** -0.5, 3)
    o_ref, lse_ref = oracle.attn_fwd(q, k, v, causal, D ** -0.5)
    parity.compare(o, lse, o_ref, lse_ref, "rising scores, split %s" % ((Sq, causal, D),))
