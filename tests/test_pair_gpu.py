"""The CTA-pair kernel of head dimensions above 128, in force for every shape: sub-tiles of unequal numbers of key steps, tiles of
which one CTA has no rows or no visible key, tails of keys, rows and columns, many tiles per pair, and values that must not
reach the rows that do not see them.  Oracle and tolerances are those of the parity tests."""
import math

import pytest
import torch

import parity
from paper_2604_18616_b200 import binding
from test_splitkv_gpu import rand_qkv
from test_varlen_gpu import _run_and_check

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def pairs():
    assert binding.select_kernel(binding.KERNEL_TWO_SUBTILES) == binding.AVE_OK
    yield
    assert binding.select_kernel(binding.KERNEL_AUTO) == binding.AVE_OK


@pytest.mark.parametrize("D", [136, 192, 256])
@pytest.mark.parametrize("B,H,Hkv,Sq,Sk,causal", [
    (1, 1, 1, 1, 1, False), (1, 3, 3, 300, 300, True), (1, 2, 1, 129, 257, True),     # one CTA with a row; odd blocks; paired heads
    (2, 4, 2, 384, 200, True), (1, 3, 1, 300, 130, True), (1, 2, 2, 256, 128, False),  # rows without keys, of both CTAs or of one
    (40, 8, 8, 260, 200, False), (20, 8, 2, 200, 390, True), (3, 8, 8, 130, 1000, True)])  # many tiles a pair; long tiles
def test_pairs(B, H, Hkv, Sq, Sk, causal, D):
    q, k, v = rand_qkv(Sq + Sk + D, B, H, Hkv, Sq, Sk, D)
    parity.check_full(q, k, v, causal, 1.0 / math.sqrt(D), "%s" % ((B, H, Hkv, Sq, Sk, causal, D),))


@pytest.mark.parametrize("scale", [-0.07, 0.0, 0.3])
def test_signs_of_the_scale_and_a_maximum_that_moves(scale):
    q, k, v = rand_qkv(9, 1, 2, 2, 150, 700, 256)
    q[..., 0], k[..., 0] = 4.0, 0.25 * torch.arange(700, dtype=torch.float32).to(k.dtype)
    parity.check_full(q, k, v, False, scale, "scale %g" % scale)


@pytest.mark.parametrize("Hkv", [2, 4])
def test_lengths(Hkv):
    lens = [1, 140, 0, 260, 390, 128, 520, 64, 256, 700, 129, 3]
    _run_and_check(lens, lens, 4, Hkv, 200, True, 3)
    _run_and_check(lens, [n + 70 for n in lens], 4, Hkv, 256, False, 4)


def test_values_that_only_the_other_sub_tile_sees():
    # rows 0..127 see keys 0..127 at most; an infinite value at key 200 is in a step that only rows 128..255 have
    q, k, v = rand_qkv(13, 1, 1, 1, 256, 256, 256)
    v[0, 0, 200, 5] = float("inf")
    o, lse = binding.ave_attn_fwd(q.cuda(), k.cuda(), v.cuda(), causal=True)
    assert torch.isfinite(lse).all() and torch.isfinite(o[:, :, :128]).all() and torch.all(o[:, :, 200:, 5] == float("inf"))


@pytest.mark.parametrize("B,H,Sq,Sk", [(1, 2, 300, 640), (1, 2, 300, 641), (3, 33, 300, 512), (3, 33, 300, 384), (2, 33, 300, 512),
                                       (1, 49, 300, 641), (1, 50, 300, 641)])
def test_sides_of_the_kernel_choice(B, H, Sq, Sk):
    # five and six key tiles; three and four with 297 and 198 tiles; 147 and 150 tiles, which pairs make 196 and 200 CTAs of
    assert binding.select_kernel(binding.KERNEL_AUTO) == binding.AVE_OK
    q, k, v = rand_qkv(H + Sk, B, H, H, Sq, Sk, 144)
    parity.check_full(q, k, v, False, 1.0 / 12, "%s" % ((B, H, Sq, Sk),))
