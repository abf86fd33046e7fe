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


def _both(call):
    """The call's results on pairs and in the single-sub-tile kernel."""
    r = [t.clone() for t in call()]
    assert binding.select_kernel(binding.KERNEL_ONE_SUBTILE) == binding.AVE_OK
    try:
        return r, [t.clone() for t in call()]
    finally:
        assert binding.select_kernel(binding.KERNEL_TWO_SUBTILES) == binding.AVE_OK


@pytest.mark.parametrize("B,H,Hkv,Sq,Sk,D,causal", [(2, 4, 2, 300, 1100, 256, True), (1, 3, 3, 385, 900, 192, True), (1, 2, 1, 200, 777, 136, False),
                                                    (3, 4, 4, 90, 1500, 256, False), (20, 8, 8, 400, 400, 256, True)])
def test_results_are_those_of_the_single_sub_tile_kernel_to_the_bit(B, H, Hkv, Sq, Sk, D, causal):
    # the same products in the same order: keys in steps of 128, sums of a step's probabilities in four groups
    q, k, v = [t.cuda() for t in rand_qkv(Sq + D, B, H, Hkv, Sq, Sk, D)]
    a, b = _both(lambda: binding.ave_attn_fwd(q, k, v, causal=causal))
    assert binding.device_status() == (binding.AVE_OK, 0)
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("B,H,Hkv,S,D,causal", [(2, 4, 2, 900, 256, True), (1, 3, 3, 777, 192, False), (1, 2, 2, 1025, 136, True)])
def test_views_of_a_packed_buffer(B, H, Hkv, S, D, causal):
    # Q, K and V as slices of one [B, S, H + 2 Hkv, D] buffer; O in rows that are wider than it, whose gaps stay as they are
    q, k, v = rand_qkv(S, B, H, Hkv, S, S, D)
    packed = torch.cat([t.permute(0, 2, 1, 3) for t in (q, k, v)], dim=2).contiguous().cuda()
    heads = packed.transpose(1, 2)
    o_store = torch.full((B, S, H, D + 24), 777.0, dtype=torch.bfloat16, device="cuda")
    ov = o_store[..., :D].transpose(1, 2)
    ov.fill_(float("nan"))
    _, lse = binding.ave_attn_fwd_strided(heads[:, :H], heads[:, H:H + Hkv], heads[:, H + Hkv:], ov, causal=causal)
    assert binding.device_status() == (binding.AVE_OK, 0)
    o2, lse2 = binding.ave_attn_fwd(q.cuda(), k.cuda(), v.cuda(), causal=causal)
    assert torch.equal(ov, o2) and torch.equal(lse, lse2) and torch.all(o_store[..., D:] == 777.0)
    rows = [(b, h, i) for b in range(B) for h in range(H) for i in (0, 127, 128, 255, 256, S - 1)]
    parity.check_rows(ov.contiguous().cpu(), lse.cpu(), q, k, v, rows, causal, D ** -0.5, "packed %s" % ((B, H, Hkv, S, D),))


def test_dependent_calls_without_waits_and_as_a_graph():
    # the output of a call is the query of the next, and a product in between is on CTA pairs as well
    q, k, v = [t.cuda() for t in rand_qkv(21, 1, 4, 4, 384, 1300, 256)]
    w = (torch.randn(1024, 1024, generator=torch.Generator().manual_seed(3)) / 32).to(torch.bfloat16).cuda()
    o, y, lse = torch.empty_like(q), torch.empty_like(q), torch.empty((1, 4, 384), dtype=torch.float32, device="cuda")

    def run(after=lambda: None):
        y.copy_(q)
        for _ in range(8):
            binding.ave_attn_fwd(y, k, v, o=o, lse=lse, causal=True)
            after()
            binding.ave_gemm_bf16_tn(o.view(384, 1024), w, c=y.view(384, 1024))
            after()

    def results():
        torch.cuda.synchronize()
        assert binding.device_status() == (binding.AVE_OK, 0)
        return o.clone(), y.clone(), lse.clone()

    run(after=torch.cuda.synchronize)
    want = results()
    assert all(torch.isfinite(t).all() for t in want)
    for _ in range(3):
        run()
        assert all(torch.equal(a, b) for a, b in zip(results(), want))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            run()
        for _ in range(3):
            o.zero_()
            lse.zero_()
            graph.replay()
        s.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(results(), want))


def test_nothing_is_written_while_the_status_word_is_set():
    # both CTAs of a pair read the word and have to agree
    q, k, v = [t.cuda() for t in rand_qkv(22, 4, 8, 8, 500, 700, 256)]
    want = binding.ave_attn_fwd(q, k, v)
    o, lse = torch.full_like(q, 3.0), torch.full((4, 8, 500), 3.0, dtype=torch.float32, device="cuda")
    assert binding.device_status() == (binding.AVE_OK, 0)
    assert binding.selftest_wait_timeout(16) == binding.AVE_OK
    binding.ave_attn_fwd(q, k, v, o=o, lse=lse)
    torch.cuda.synchronize()
    assert torch.all(o == 3.0) and torch.all(lse == 3.0)
    assert binding.device_status() == (binding.AVE_ERR_DEVICE_TIMEOUT, binding.STATUS_BIT_SELFTEST)
    binding.ave_attn_fwd(q, k, v, o=o, lse=lse)
    assert binding.device_status() == (binding.AVE_OK, 0)
    assert torch.equal(o, want[0]) and torch.equal(lse, want[1])
