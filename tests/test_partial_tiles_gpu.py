"""Launches in which much of the tile grid, of a tile, or of a hand-over is empty: variable-length batches of mostly short
sequences (the tile scheduler passes over tiles beyond a sequence's end), tiles in which whole softmax warps have no query row,
split-KV merges with one and with several warps per row, the fused MoE layer with many row tiles per expert, with more experts
than rows and with very small activations.  Oracles and tolerances are those of the neighbouring parity tests."""
import math

import pytest
import torch

import oracle
from paper_2604_18616_b200 import binding, inputs

import parity
from test_moe_gpu import check as check_moe, run_gpu as run_moe
from test_splitkv_gpu import rand_qkv, run_split
from test_varlen_gpu import _run_and_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,causal", [(64, False), (64, True), (128, False), (128, True), (256, True)])
def test_variable_length_batch_of_mostly_empty_blocks(D, causal):
    lens = [1, 0, 5, 700, 0, 0, 129, 3, 0, 128, 2, 64]
    _run_and_check(lens, lens, 4, 2, D, causal, 5)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("Sq", [1, 32, 33, 64, 96, 97, 128])
def test_softmax_warps_without_a_row(D, Sq):
    q, k, v = rand_qkv(Sq + D, 2, 2, 1, Sq, 391, D)
    parity.check_full(q, k, v, True, 1.0 / math.sqrt(D), "Sq = %d, D = %d" % (Sq, D))


@pytest.mark.parametrize("B,H,Hkv,Sq,Sk,D,n_splits", [
    (1, 2, 2, 1, 9000, 64, 64),      # 2 rows: eight warps each, two ranges at a time
    (1, 2, 2, 1, 4300, 128, 33),     # one range beyond a warp's 32
    (4, 16, 16, 40, 700, 64, 5),     # 2560 rows: one warp each
    (1, 3, 1, 1, 1500, 128, 4),      # a last CTA with rows beyond the end
    (2, 4, 2, 100, 500, 128, 1),     # a single range, packed heads on 256-row tiles
    (2, 4, 1, 3, 500, 64, 1),        # a single range, packed heads on 128-row tiles
    (1, 8, 8, 1000, 2600, 64, 19), (1, 8, 8, 1000, 2600, 64, 20),    # the last number of ranges merged row-wise, and the next
    (1, 3, 3, 275, 600, 128, 4), (1, 3, 3, 276, 600, 128, 4),        # the same at 13200 threads; a last CTA in part
    (1, 7, 7, 586, 300, 128, 3), (1, 3, 3, 2731, 300, 64, 3),        # 8 columns for each of more than 65536 threads
])
def test_split_merge_shapes(B, H, Hkv, Sq, Sk, D, n_splits):
    q, k, v = rand_qkv(H + Sk, B, H, Hkv, Sq, Sk, D)
    scale = 1.0 / math.sqrt(D)
    o, lse = run_split(q, k, v, True, scale, n_splits)
    o_ref, lse_ref = oracle.attn_fwd(q, k, v, True, scale)
    parity.compare(o, lse, o_ref, lse_ref, "split %d" % n_splits)


@pytest.mark.parametrize("T,C,F,E,K,shrink", [
    (1100, 128, 128, 1, 1, 1.0),      # nine row tiles of one expert: two groups of tiles
    (20, 256, 128, 1000, 3, 1.0),     # most experts empty
    (33, 640, 384, 3, 2, 1.0),        # odd numbers of weight blocks both ways
    (40, 256, 256, 4, 2, 1e-10),      # requantisation groups far below fp32's reciprocal range of 448
])
def test_moe_edges(T, C, F, E, K, shrink):
    args = list(inputs.make_moe_inputs(inputs.MoeWorkload("edge", T, C, F, E, K, T + E)))
    args[1] = args[1] * shrink
    y_ref = oracle.moe_fwd(*[t.numpy() for t in args])
    check_moe(run_moe(args), y_ref, args, "moe %s" % ((T, C, F, E, K, shrink),))


@pytest.mark.parametrize("H,Sq,Sk,causal", [
    (74, 256, 400, False), (75, 256, 400, False),    # 148 / 150 tiles of 128 rows: one per SM, and more
    (74, 512, 512, True), (75, 512, 512, True),      # 296 / 300: two per SM, both in the two-sub-tile kernel
    (148, 400, 384, False), (148, 400, 385, False),  # 592 tiles of three / four key steps
])
def test_sides_of_the_kernel_choice(H, Sq, Sk, causal):
    q, k, v = rand_qkv(H + Sk, 1, H, H, Sq, Sk, 64)
    parity.check_full(q, k, v, causal, 0.125, "%s" % ((H, Sq, Sk, causal),))


@pytest.mark.parametrize("B,H,Hkv,Sq,Sk,D", [
    (1, 16, 4, 1408, 1408, 128), (1, 16, 4, 1408, 4001, 128),    # 176 tiles, grouped heads: one, and two sub-tiles
    (1, 7, 7, 3201, 3300, 64), (1, 7, 7, 3201, 12000, 64),       # 182 tiles
    (1, 8, 8, 4700, 4700, 128), (1, 8, 8, 4700, 9001, 128),      # 296 tiles, 152 of 256 rows: two, and one sub-tile
    (3, 32, 16, 168, 3000, 96),
])
def test_sides_of_the_kernel_choice_for_prompts_after_cached_keys(B, H, Hkv, Sq, Sk, D):
    q, k, v = rand_qkv(H + Sk, B, H, Hkv, Sq, Sk, D)
    scale = 1.0 / math.sqrt(D)
    o, lse = parity.run_gpu(q, k, v, True, scale)
    g = torch.Generator().manual_seed(Sk)
    rows = torch.stack([torch.randint(0, n, (300,), generator=g) for n in (B, H, Sq)], dim=1)
    rows[:8, 2] = torch.tensor([0, 127, 128, 255, 256, Sq - 129, Sq - 128, Sq - 1]).clamp(0, Sq - 1)
    parity.check_rows(o, lse, q, k, v, rows.numpy(), True, scale, "%s" % ((B, H, Hkv, Sq, Sk, D),))


@pytest.mark.parametrize("lens", [[700, 3, 400], [900, 650, 5, 500]])   # 16 heads: 176 and 320 tiles by the rule's count
def test_sides_of_the_kernel_choice_for_variable_lengths(lens):
    _run_and_check(lens, lens, 16, 4, 128, True, 6)


@pytest.mark.parametrize("Hkv", [1, 2])   # (1: paired heads in the causal two-sub-tile kernel; 2: 256-row tiles)
@pytest.mark.parametrize("kernel", [binding.KERNEL_TWO_SUBTILES, binding.KERNEL_ONE_SUBTILE])
def test_scheduler_passes_over_long_runs_of_empty_tiles(kernel, Hkv):
    """One sequence of 2100 tokens among 300 of at most three: nearly every tile of the grid lies beyond its sequence's end, so
    that each CTA's scheduler asks for the next tile many times over before it has one to hand on."""
    lens = [i % 4 for i in range(150)] + [2100] + [3 - i % 4 for i in range(150)]
    assert binding.select_kernel(kernel) == binding.AVE_OK
    try:
        _run_and_check(lens, lens, 2, Hkv, 64, True, 8)
    finally:
        assert binding.select_kernel(binding.KERNEL_AUTO) == binding.AVE_OK
