"""What this library is timed on: passes through its public entry points as a user's program makes them.

``listed()`` names the cases, ``draw(rng)`` gives further ones of the same ranges, ``prepare`` builds on the GPU what a
program has in hand before the call, ``run`` makes the call, ``work`` counts what the pass cannot do without and
``tolerance`` says how far two correct results may lie apart.

Kinds of pass: attention over contiguous tensors ("fwd"), over views of a packed QKV buffer ("packed"), over sequences of
different lengths ("varlen"), one decode step with split keys ("decode"); a bf16 matrix product ("gemm", both layouts of
B); the block-quantised FP8 mixture-of-experts layer ("moe").
"""
import math

import torch

from paper_2604_18616_b200 import binding


def _attn(name, kind, B, H, Hkv, Sq, Sk, D, causal, dist="normal", peaked=0):
    return {"name": name, "kind": kind, "B": B, "H": H, "Hkv": Hkv, "Sq": Sq, "Sk": Sk, "D": D, "causal": causal,
            "dist": dist, "peaked": peaked}


def _gemm(name, layout, M, N, K):
    return {"name": name, "kind": "gemm", "layout": layout, "M": M, "N": N, "K": K}


def _moe(name, T, C=7168, F=2048, E=32, K=4):
    return {"name": name, "kind": "moe", "T": T, "C": C, "F": F, "E": E, "K": K}


def listed():
    return [
        # the smallest call: one head pair, one key tile; what counts is the launch
        _attn("attn_tiny", "fwd", 1, 2, 2, 128, 128, 64, False),
        # ordinary causal prefill with as many key/value heads as query heads
        _attn("attn_mha_prefill", "fwd", 4, 32, 32, 2048, 2048, 128, True),
        # long-context prefill, grouped queries, every 64th key peaked (attention sinks, separators): the largest
        _attn("attn_gqa_long", "fwd", 1, 32, 8, 16384, 16384, 128, True, peaked=64),
        # bidirectional encoder reading Q, K and V in place from the projection's packed output
        _attn("attn_encoder_packed", "packed", 8, 16, 16, 8192, 8192, 64, False, dist="uniform"),
        # prefill of a model with wide heads
        _attn("attn_wide_head", "fwd", 2, 32, 8, 4096, 4096, 256, True),
        # a batch of prompts of different lengths, packed without padding (Sq, Sk: the longest)
        _attn("attn_varlen", "varlen", 24, 32, 8, 2500, 2500, 128, True),
        # decode step of a full batch against caches of an odd length
        _attn("decode_batch", "decode", 64, 32, 8, 1, 4001, 128, True),
        # decode step of a single sequence with a long cache
        _attn("decode_long", "decode", 1, 32, 8, 1, 65536, 128, True),
        # square product, both operands K-contiguous (activations times a weight matrix)
        _gemm("gemm_square", "tn", 4096, 4096, 4096),
        # the other layout of B, ragged in every dimension
        _gemm("gemm_nn_ragged", "nn", 3001, 5112, 2056),
        # expert layer of a decode batch: bound by reading the weights
        _moe("moe_decode", 256),
        # expert layer of a prefill chunk
        _moe("moe_prefill", 4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges; nothing drawn costs more than the largest listed case."""
    kind = rng.choice(["fwd", "fwd", "packed", "varlen", "decode", "decode", "gemm", "gemm", "moe"])
    if kind == "gemm":
        while True:
            m, n, k = _log_int(rng, 128, 9000), 8 * _log_int(rng, 32, 1100), 8 * _log_int(rng, 32, 1100)
            if 2.0 * m * n * k <= 1.1e12:
                return {"kind": kind, "layout": rng.choice(["tn", "nn"]), "M": m, "N": n, "K": k}
    if kind == "moe":
        k = rng.choice([2, 4, 4, 4, 8])
        return {"kind": kind, "T": _log_int(rng, 16, 16384 // k), "C": 7168, "F": 2048, "E": 32, "K": k}
    hkv = rng.choice([1, 2, 4, 8, 8, 16])
    group = rng.choice([1, 1, 2, 4, 4, 8])
    causal = rng.random() < 0.7
    if kind == "decode":
        while True:
            b, sk = _log_int(rng, 1, 128), _log_int(rng, 256, 65536)
            if b * hkv * sk <= 8 * 32 * 8192:
                return {"kind": kind, "B": b, "H": hkv * group, "Hkv": hkv, "Sq": rng.choice([1, 1, 1, 2, 4]), "Sk": sk,
                        "D": rng.choice([64, 128, 128]), "causal": True, "dist": "normal", "peaked": 0}
    d = rng.choice([64, 64, 96, 128, 128, 128, 192, 256])
    while True:
        b, sq = _log_int(rng, 1, 16), _log_int(rng, 64, 16384)
        sk = sq if kind != "fwd" or rng.random() < 0.7 else sq + _log_int(rng, 64, 8192)  # a chunk after cached keys
        c = {"kind": kind, "B": b, "H": hkv * group, "Hkv": hkv, "Sq": sq, "Sk": sk, "D": d, "causal": causal,
             "dist": rng.choice(["normal", "normal", "uniform"]), "peaked": rng.choice([0, 0, 64]) if causal else 0}
        if work(c)["flops"] <= 2.0e12:
            return c


def _lengths(case):
    """Lengths of a variable-length batch: spread from a few tokens to the longest, fixed by the case's sizes alone."""
    n, top = case["B"], case["Sq"]
    lens = [max(1, int(top * (((i * 0.6180339887) % 1.0) ** 1.5))) for i in range(n)]
    lens[n // 2] = top
    return lens


def _filled(shape, dist, g):
    x = torch.empty(shape, dtype=torch.float32, device="cuda")
    if dist == "uniform":
        return x.uniform_(-2.0, 2.0, generator=g)
    return x.normal_(generator=g)


def _quantise_rows(x):
    """E4M3 codes and fp32 scales of x [rows, cols], one scale per row and 128 columns."""
    rows, cols = x.shape
    grp = x.view(rows, cols // 128, 128)
    s = grp.abs().amax(dim=2).clamp_min(1e-20) / 448.0
    return (grp / s[:, :, None]).to(torch.float8_e4m3fn).view(torch.uint8).view(rows, cols), s.contiguous()


def _quantise_weights(E, rows, cols, g):
    """Codes [E, rows, cols] and one scale per 128 x 128 block of weights drawn from N(0, 1/cols)."""
    q = torch.empty((E, rows, cols), dtype=torch.uint8, device="cuda")
    s = torch.empty((E, rows // 128, cols // 128), dtype=torch.float32, device="cuda")
    for e in range(E):
        w = torch.empty((rows // 128, 128, cols // 128, 128), dtype=torch.float32, device="cuda")
        w.normal_(0.0, cols ** -0.5, generator=g)
        s[e] = w.abs().amax(dim=(1, 3)) / 448.0
        w /= s[e][:, None, :, None]
        q[e] = w.to(torch.float8_e4m3fn).view(torch.uint8).view(rows, cols)
    return q, s


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    c = dict(case)
    if c["kind"] == "gemm":
        a = torch.empty((c["M"], c["K"]), dtype=torch.float32, device="cuda").normal_(generator=g).bfloat16()
        shape = (c["N"], c["K"]) if c["layout"] == "tn" else (c["K"], c["N"])
        b = torch.empty(shape, dtype=torch.float32, device="cuda").normal_(generator=g).bfloat16()
        return c, (a, b)
    if c["kind"] == "moe":
        T, C, F, E, K = c["T"], c["C"], c["F"], c["E"], c["K"]
        xq, sx = _quantise_rows(torch.empty((T, C), dtype=torch.float32, device="cuda").normal_(generator=g))
        w13q, s13 = _quantise_weights(E, 2 * F, C, g)
        w2q, s2 = _quantise_weights(E, C, F, g)
        ids = torch.rand((T, E), device="cuda", generator=g).argsort(dim=1)[:, :K].to(torch.int32).contiguous()
        raw = 0.1 + torch.rand((T, K), device="cuda", generator=g)
        wts = (raw / raw.sum(dim=1, keepdim=True)).contiguous()
        ws = torch.empty(binding.moe_workspace_bytes(T, C, F, E, K), dtype=torch.uint8, device="cuda")
        return c, (xq, sx, w13q, s13, w2q, s2, ids, wts), ws
    B, H, Hkv, Sq, Sk, D = (c[k] for k in ("B", "H", "Hkv", "Sq", "Sk", "D"))
    if c["kind"] == "varlen":
        lens = _lengths(c)
        total = sum(lens)
        q = _filled((total, H, D), c["dist"], g).bfloat16()
        k = _filled((total, Hkv, D), c["dist"], g)
        if c["peaked"]:
            k[:: c["peaked"]] *= 4.0
        v = _filled((total, Hkv, D), c["dist"], g).bfloat16()
        cu = torch.tensor([0] + [sum(lens[: i + 1]) for i in range(B)], dtype=torch.int32, device="cuda")
        return c, (q, k.bfloat16(), v, cu)
    if c["kind"] == "packed":
        qkv = torch.empty((B, Sq, (H + 2 * Hkv) * D), dtype=torch.bfloat16, device="cuda")
        for b in range(B):
            x = _filled((Sq, H + 2 * Hkv, D), c["dist"], g)
            if c["peaked"]:
                x[:: c["peaked"], H:H + Hkv] *= 4.0
            qkv[b] = x.view(Sq, -1).bfloat16()
        return c, (qkv,)
    q = _filled((B, H, Sq, D), c["dist"], g).bfloat16()
    k = _filled((B, Hkv, Sk, D), c["dist"], g)
    if c["peaked"]:
        k[:, :, :: c["peaked"]] *= 4.0
    k = k.bfloat16()
    v = _filled((B, Hkv, Sk, D), c["dist"], g).bfloat16()
    if c["kind"] == "decode":
        n = binding.splitkv_default_splits(B, H, Hkv, Sq, Sk, D)
        ws = torch.empty(max(256, binding.splitkv_workspace_bytes(B, H, Sq, D, n)), dtype=torch.uint8, device="cuda")
        return c, (q, k, v), n, ws
    return c, (q, k, v)


def run(state):
    c, x = state[0], state[1]
    if c["kind"] == "gemm":
        return (binding.ave_gemm_bf16_tn if c["layout"] == "tn" else binding.ave_gemm_bf16_nn)(*x)
    if c["kind"] == "moe":
        return binding.ave_moe_fused_fwd(*x, workspace=state[2])
    if c["kind"] == "varlen":
        q, k, v, cu = x
        return binding.ave_attn_fwd_varlen(q, k, v, cu, cu, c["Sq"], c["Sk"], causal=c["causal"])
    if c["kind"] == "packed":
        B, H, Hkv, S, D = c["B"], c["H"], c["Hkv"], c["Sq"], c["D"]
        heads = x[0].view(B, S, H + 2 * Hkv, D).transpose(1, 2)
        o = torch.empty((B, S, H, D), dtype=torch.bfloat16, device=heads.device)  # token-major, for the output projection
        _, lse = binding.ave_attn_fwd_strided(heads[:, :H], heads[:, H:H + Hkv], heads[:, H + Hkv:], o.transpose(1, 2),
                                              causal=c["causal"])
        return o, lse
    if c["kind"] == "decode":
        return binding.ave_attn_fwd_splitkv(*x, state[2], workspace=state[3], causal=c["causal"])
    return binding.ave_attn_fwd(*x, causal=c["causal"])


def _pairs(sq, sk, causal):
    """(query, key) pairs that the mask leaves visible: key j to query i iff j <= i + (sk - sq)."""
    if not causal:
        return sq * sk
    first = min(sq, max(0, sq - sk))  # queries that see no key
    n = sq - first
    return n * (sk - sq + first + 1) + n * (n - 1) // 2


def work(case):
    c = case
    if c["kind"] == "gemm":
        M, N, K = c["M"], c["N"], c["K"]
        return {"bytes": 2 * (M * K + N * K + M * N), "flops": 2 * M * N * K}
    if c["kind"] == "moe":
        T, C, F, E, K = c["T"], c["C"], c["F"], c["E"], c["K"]
        used = E * (1.0 - (1.0 - K / E) ** T)  # experts that some token of the batch is routed to
        return {"bytes": used * 3 * F * C * (1 + 4 / 128 / 128) + T * C * (1 + 4 / 128) + 8 * T * K + 2 * T * C,
                "flops": 2 * T * K * 3 * F * C}
    B, H, Hkv, D = c["B"], c["H"], c["Hkv"], c["D"]
    seqs = [(n, n) for n in _lengths(c)] if c["kind"] == "varlen" else [(c["Sq"], c["Sk"])] * B
    rows, keys = sum(s[0] for s in seqs), sum(s[1] for s in seqs)
    return {"bytes": rows * H * (4 * D + 4) + keys * Hkv * 4 * D,
            "flops": 4 * D * H * sum(_pairs(a, b, c["causal"]) for a, b in seqs)}


def tolerance(case):
    """About four times what the passes show against the same computation in fp64 (2-norm / largest element):
    products 1.7e-3 / 3.9e-3, the expert layer 1.7e-3 / 5.4e-3 (an intermediate that rounds to the neighbouring E4M3 code
    moves single elements further), attention 2.4e-3 / 3.1e-2 (probabilities and results rounded to bf16; the first rows
    of a causal mask are far larger than the root mean square)."""
    if case["kind"] == "gemm":
        return {"rel": 7e-3, "max": 0.016}
    if case["kind"] == "moe":
        return {"rel": 7e-3, "max": 0.04}
    return {"rel": 1e-2, "max": 0.12}
