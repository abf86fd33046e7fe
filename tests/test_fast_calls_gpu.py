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


def test_ordinary_calls_take_the_short_way():
    """Each extension function launches by itself and its results are those of the Python way; the wrappers ask it first."""
    q, k, v = [t.cuda() for t in rand_qkv(7, 2, 6, 2, 70, 130, 64)]
    binding.lib()
    fast = binding._fast
    assert fast is not None
    ws = torch.empty(binding.splitkv_workspace_bytes(2, 6, 70, 64, 2), dtype=torch.uint8, device="cuda")
    a, b = q.reshape(-1, 64), k.reshape(-1, 64)
    bt = b.t().contiguous()[:, :512].contiguous()
    new = lambda r, c: torch.empty(r, c, dtype=torch.bfloat16, device="cuda")
    for got, want in [
            (lambda: fast.attn_fwd(q, k, v, True, None), lambda: binding.ave_attn_fwd(q, k, v, o=torch.empty_like(q), causal=True)),
            (lambda: fast.attn_fwd(q, k, v, 0, 0.3), lambda: binding.ave_attn_fwd(q, k, v, o=torch.empty_like(q), scale=0.3)),
            (lambda: fast.attn_fwd_splitkv(q, k, v, 2, ws, True, None),
             lambda: binding.ave_attn_fwd_splitkv(q, k, v, 2, workspace=ws, o=torch.empty_like(q), causal=True)),
            (lambda: (fast.gemm_tn(a, b),), lambda: (binding.ave_gemm_bf16_tn(a, b, c=new(a.shape[0], b.shape[0])),)),
            (lambda: (fast.gemm_nn(a, bt),), lambda: (binding.ave_gemm_bf16_nn(a, bt, c=new(a.shape[0], 512)),))]:
        n0 = binding.launch_count()
        r = got()
        assert r is not None and all(isinstance(t, torch.Tensor) for t in r)
        torch.cuda.synchronize()
        assert binding.launch_count() > n0, "nothing was launched"
        assert all(torch.equal(x, y) for x, y in zip(r, want()))
    # a status of the library comes back as an int: three heads on two
    assert fast.attn_fwd(q[:, :3].contiguous(), k, v, False, None) == binding.AVE_ERR_BAD_SHAPE
    assert fast.gemm_tn(a[:, :60].contiguous(), b[:, :60].contiguous()) == binding.AVE_ERR_MISALIGNED


@pytest.mark.parametrize("call,args", [("attn_fwd", 3), ("attn_fwd_splitkv", 3), ("gemm_tn", 2), ("gemm_nn", 2)])
def test_wrappers_return_what_the_short_way_gave(call, args, monkeypatch):
    seen = []

    class Fast:
        def __getattr__(self, name):
            return lambda *a: seen.append(name) or "result"

    binding.lib()
    monkeypatch.setattr(binding, "_fast", Fast())
    x = [torch.empty(0)] * args
    wrapper = getattr(binding, "ave_attn_fwd" + call[8:] if call.startswith("attn") else "ave_gemm_bf16" + call[4:])
    assert (wrapper(*x, 2) if call == "attn_fwd_splitkv" else wrapper(*x)) == "result" and seen == [call]


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
