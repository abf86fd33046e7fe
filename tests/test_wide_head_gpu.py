"""Head dimensions above 128: two score buffers and a ring of half K and V tiles.  Key counts around the half and whole tiles,
tiles of one, two and more steps one after the other on the same SM, and scores whose maximum moves at every step, so that
the accumulator is rescaled between the products that overlap it.  In the single-sub-tile kernel and on CTA pairs, whichever of
them a call would choose by itself.  Oracle and tolerances are those of the parity tests."""
import math

import pytest
import torch

import parity
from paper_2604_18616_b200 import binding
from test_splitkv_gpu import rand_qkv
from test_varlen_gpu import _run_and_check

pytestmark = pytest.mark.gpu


@pytest.fixture(params=[binding.KERNEL_ONE_SUBTILE, binding.KERNEL_TWO_SUBTILES], autouse=True)
def kernel(request):
    assert binding.select_kernel(request.param) == binding.AVE_OK
    yield
    assert binding.select_kernel(binding.KERNEL_AUTO) == binding.AVE_OK


@pytest.mark.parametrize("D", [136, 192, 256])
@pytest.mark.parametrize("Sq,Sk,causal", [(1, 1, False), (128, 63, False), (129, 65, False), (7, 128, True), (200, 129, False),
                                          (130, 193, True), (257, 256, False), (385, 385, True), (64, 1100, True)])
def test_edges_of_half_tiles(D, Sq, Sk, causal):
    q, k, v = rand_qkv(Sq + Sk + D, 2, 4, 2, Sq, Sk, D)
    parity.check_full(q, k, v, causal, 1.0 / math.sqrt(D), "%s" % ((D, Sq, Sk, causal),))


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_maximum_moves_at_every_step(sign):
    q, k, v = rand_qkv(11, 1, 2, 2, 150, 1000, 256)
    q[..., 0], k[..., 0] = 4.0, sign * 0.25 * torch.arange(1000, dtype=torch.float32).to(k.dtype)
    parity.check_full(q, k, v, False, sign / math.sqrt(256), "rising scores, sign %g" % sign)


def test_many_tiles_of_different_lengths():
    lens = [1, 140, 0, 260, 390, 128, 520, 64, 256, 700, 129, 3]
    _run_and_check(lens, lens, 16, 4, 256, True, 3)
