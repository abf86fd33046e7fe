"""The binding's C++ calls: the same results, bit for bit, as the Python wrappers' own way (which a given output tensor selects), and
None, with nothing launched, for every call that is not an ordinary one."""
import pytest
import torch

from paper_2604_18616_b200 import binding

from test_splitkv_gpu import rand_qkv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [None, 0.3])
@pytest.mark.parametrize("causal", [False, True])
def test_results_are_those_of_the_python_way(causal, scale):
    q, k, v = [t.cuda() for t in rand_qkv(3, 2, 6, 2, 70, 130, 64)]
    o, lse = binding.ave_attn_fwd(q, k, v, causal=causal, scale=scale)
    o2, lse2 = binding.ave_attn_fwd(q, k, v, o=torch.empty_like(q), causal=causal, scale=scale)
    assert torch.equal(o, o2) and torch.equal(lse, lse2) and o.shape == q.shape and lse.shape == (2, 6, 70)
    ws = torch.empty(binding.splitkv_workspace_bytes(2, 6, 70, 64, 2), dtype=torch.uint8, device="cuda")
    o, lse = binding.ave_attn_fwd_splitkv(q, k, v, 2, workspace=ws, causal=causal, scale=scale)
    o2, lse2 = binding.ave_attn_fwd_splitkv(q, k, v, 2, workspace=ws, o=torch.empty_like(q), causal=causal, scale=scale)
    assert torch.equal(o, o2) and torch.equal(lse, lse2)
    a, b = q.reshape(-1, 64), k.reshape(-1, 64)
    assert torch.equal(binding.ave_gemm_bf16_tn(a, b), binding.ave_gemm_bf16_tn(a, b, c=a.new_empty(a.shape[0], b.shape[0])))
    b = b.t().contiguous()[:, :512].contiguous()
    assert torch.equal(binding.ave_gemm_bf16_nn(a, b), binding.ave_gemm_bf16_nn(a, b, c=a.new_empty(a.shape[0], b.shape[1])))


def test_calls_out_of_the_ordinary_are_left_to_the_python_way():
    q, k, v = [t.cuda() for t in rand_qkv(4, 1, 2, 2, 8, 16, 64)]
    binding.lib()
    fast, n0 = binding._fast, binding.launch_count()
    for args in [(q.cpu(), k, v), (q, k.cpu(), v), (q.float(), k, v), (q[0], k, v), (q.transpose(1, 2), k, v), (q, k, v[:, :, :8]),
                 (q, k[:, :1], v), (q.data_ptr(), k, v)]:
        assert fast.attn_fwd(*args, False, None) is None
        with pytest.raises((ValueError, AttributeError)):
            binding.ave_attn_fwd(*args)
    assert fast.attn_fwd(q, k, v, False, "1") is None and fast.attn_fwd(q, k, v, False) is None
    assert fast.attn_fwd_splitkv(q, k, v, 2, None, False, None) is None
    assert fast.gemm_tn(q[0, 0], k[0, 0].t()) is None and fast.gemm_nn(q[0, 0], k[0, 0]) is None
    assert binding.launch_count() == n0


def test_errors_of_the_library_raise():
    q, k, v = [t.cuda() for t in rand_qkv(5, 1, 3, 2, 8, 16, 64)]   # three heads on two
    with pytest.raises(binding.AveAttnError) as e:
        binding.ave_attn_fwd(q, k, v)
    assert e.value.status == binding.AVE_ERR_BAD_SHAPE
    with pytest.raises(binding.AveAttnError) as e:
        binding.ave_gemm_bf16_tn(q[0, 0, :, :60].contiguous(), k[0, 0, :, :60].contiguous())
    assert e.value.status != binding.AVE_OK


def test_other_streams_and_capture():
    q, k, v = [t.cuda() for t in rand_qkv(6, 1, 2, 2, 128, 128, 64)]
    want = binding.ave_attn_fwd(q, k, v)[0]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        got = binding.ave_attn_fwd(q, k, v)[0]
    s.synchronize()
    assert torch.equal(got, want)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        o = binding.ave_attn_fwd(q, k, v)[0]
    o.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(o, want)
