"""Calls that depend on one another, enqueued without a wait in between: most kernels of the library are launched so that their
set-up overlaps the end of the kernel before them, and have to wait for its results by themselves.  Every kernel of the
library is deterministic, so a chain must give, bit for bit, what the same calls give one at a time; as a CUDA graph too."""
import math

import pytest
import torch

from paper_2604_18616_b200 import binding, inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
STEPS = 6


def _normal(seed, *shape):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=g)


class Chain:
    """x [256, 512] -> three products (Q, K, V of 4 heads x 256 rows) -> attention -> split-KV attention (scratch shared by all
    steps) -> a product of many columns -> one with a long K -> x again; every step overwrites what the one before used."""

    def __init__(self):
        w = lambda seed, n, k: (_normal(seed, n, k) / math.sqrt(k)).to(torch.bfloat16).to(DEV)
        self.w = [w(i, 512, 512) for i in range(3)]       # tn: few tiles, single CTAs
        self.wide = w(3, 19000, 512)                      # 128 x 256 tiles
        self.long = w(4, 512, 19000)                      # a cluster of eight CTAs shares K
        self.back = w(5, 256, 128)                        # nn, back to [256, 512]
        self.big = w(6, 5000, 512)                        # CTA pairs, several tiles each
        e = lambda *s: torch.empty(s, dtype=torch.bfloat16, device=DEV)
        self.x, self.qkv = e(256, 512), [e(256, 512) for _ in range(3)]
        self.o1, self.o2 = e(1, 4, 256, 128), e(1, 4, 256, 128)
        self.lse = torch.empty((1, 4, 256), dtype=torch.float32, device=DEV)
        self.ws = torch.empty(binding.splitkv_workspace_bytes(1, 4, 256, 128, 2), dtype=torch.uint8, device=DEV)
        self.y, self.z = e(128, 19000), e(128, 512)
        self.a = e(5120, 512)
        self.out = [e(5120, 5000) for _ in range(STEPS)]
        self.copies = [e(256, 512) for _ in range(STEPS)]
        self.one = torch.eye(512, dtype=torch.bfloat16, device=DEV)

    def set_input(self, seed):
        self.x.copy_(_normal(seed, 256, 512))
        self.a.copy_(_normal(seed + 1, 5120, 512))

    def run(self, after=lambda: None):
        heads = [t.view(1, 4, 256, 128) for t in self.qkv]
        for i in range(STEPS):
            for w, t in zip(self.w, self.qkv):
                binding.ave_gemm_bf16_tn(self.x, w, c=t)
                after()
            binding.ave_attn_fwd(*heads, o=self.o1, lse=self.lse, causal=True)
            after()
            binding.ave_attn_fwd_splitkv(self.o1, heads[1], heads[2], 2, workspace=self.ws, o=self.o2, lse=self.lse)
            after()
            o2 = self.o2.view(256, 512)
            binding.ave_gemm_bf16_tn(o2[:128], self.wide, c=self.y)
            after()
            binding.ave_gemm_bf16_tn(self.y, self.long, c=self.z)
            after()
            binding.ave_gemm_bf16_nn(self.back, self.z, c=self.x)
            after()
            binding.ave_gemm_bf16_nn(self.x, self.one, c=self.a[:256])
            after()
            binding.ave_gemm_bf16_tn(self.a, self.big, c=self.out[i])
            after()
            binding.ave_gemm_bf16_nn(self.x, self.one, c=self.copies[i])
            after()

    def results(self):
        torch.cuda.synchronize()
        assert binding.device_status() == (binding.AVE_OK, 0)
        return [t.clone() for t in self.out + self.copies + [self.o1, self.o2, self.lse]]


@pytest.fixture(scope="module")
def chain():
    return Chain()


@pytest.fixture(scope="module")
def one_at_a_time(chain):
    def run(seed):
        chain.set_input(seed)
        chain.run(after=torch.cuda.synchronize)
        return chain.results()
    return {seed: run(seed) for seed in (1, 50)}


def _same(got, want):
    for i, (a, b) in enumerate(zip(got, want)):
        assert torch.isfinite(b).all()
        assert torch.equal(a, b), "result %d differs from the calls one at a time" % i


def test_dependent_calls_without_waits(chain, one_at_a_time):
    for seed in (1, 50, 1):
        chain.set_input(seed)
        chain.run()
        _same(chain.results(), one_at_a_time[seed])


def test_dependent_calls_as_a_cuda_graph(chain, one_at_a_time):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        chain.set_input(1)
        chain.run()                       # (kernels are prepared before the capture)
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            chain.run()
        for seed in (50, 1):
            chain.set_input(seed)
            graph.replay()
            graph.replay()                # (reads x and a as the first replay left them)
            chain.set_input(seed)
            graph.replay()
            _same(chain.results(), one_at_a_time[seed])


def test_expert_layers_that_share_a_workspace():
    w = [inputs.MoeWorkload("chain%d" % i, T, 512, 256, 8, 2, 40 + i) for i, T in enumerate((300, 17, 120))]
    d = [[t.to(DEV) for t in inputs.make_moe_inputs(x)] for x in w]
    ws = torch.empty(max(binding.moe_workspace_bytes(x.T, 512, 256, 8, 2) for x in w), dtype=torch.uint8, device=DEV)
    ys = [torch.empty((x.T, 512), dtype=torch.bfloat16, device=DEV) for x in w]

    def run(after=lambda: None):
        for _ in range(4):
            for args, y in zip(d, ys):
                binding.ave_moe_fused_fwd(*args, y=y, workspace=ws)
                after()
        torch.cuda.synchronize()
        assert binding.device_status() == (binding.AVE_OK, 0)
        return [y.clone() for y in ys]

    want = run(after=torch.cuda.synchronize)
    for y in ys:
        y.fill_(float("nan"))
    _same(run(), want)
