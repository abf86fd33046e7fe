"""GPU parity of the matrix product where few output tiles make clusters of CTAs share K, and where the CTA pairs' tile is
narrower than 256 columns, against the fp64 oracle.

Tolerance as for the other product tests: products of bf16 values are exact in fp32, the fp32 accumulation of K unit-variance
products (in up to eight parts here, which changes the order of the sum only) errs by about K 2^-24, and the one rounding of C
to bf16 by at most 2^-9 relative: |C - oracle| <= 2^-8 |oracle| + 1e-3 sqrt(K)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2604_18616_b200 import binding, inputs

pytestmark = pytest.mark.gpu

CASES = [
    # M, N, K: few 128 x 128 tiles and a long K (clusters of 8, 8, 2, 4), CTA pairs with tiles of 64 columns (N-contiguous B: a
    # cluster of 4), single CTAs, CTA pairs with tiles of 64, 192 (N-contiguous B: 256) and 128 columns; ragged edges
    (200, 512, 2056),     # a last slice of 8
    (257, 136, 4096),
    (1939, 440, 2416),
    (300, 1000, 3000),    # 24 tiles
    (130, 264, 1000),     # edges just past a tile, a last slice of 40
    (1, 8, 2048),         # a single row and one group of columns (clusters of 8)
    (128, 128, 256),
    (700, 1000, 712),
    (300, 2000, 520),
    (1100, 1096, 328),
    (420, 6544, 840),
    (1711, 2600, 32),
    (1300, 2600, 392),
]


@pytest.mark.parametrize("layout", ["tn", "nn"])
@pytest.mark.parametrize("M,N,K", CASES)
def test_shared_k_and_narrow_tiles(layout, M, N, K):
    a, b = inputs.make_gemm_inputs(M, N, K, M + 3 * N + 7 * K)
    dev = torch.device("cuda:0")
    guard = 512
    buf = torch.full((M * N + 2 * guard,), 777.0, dtype=torch.bfloat16, device=dev)
    c = buf[guard:guard + M * N].view(M, N)
    c.fill_(float("nan"))
    if layout == "tn":
        binding.ave_gemm_bf16_tn(a.to(dev), b.to(dev), c)
    else:
        binding.ave_gemm_bf16_nn(a.to(dev), b.t().contiguous().to(dev), c)
    assert binding.device_status() == (binding.AVE_OK, 0)
    assert torch.all(buf[:guard] == 777.0) and torch.all(buf[guard + M * N:] == 777.0), "guard band touched"
    ref = oracle.gemm_tn(a, b)
    err = np.abs(c.cpu().double().numpy() - ref)
    tol = 2.0 ** -8 * np.abs(ref) + 1e-3 * math.sqrt(K)
    assert np.all(err <= tol), "max error %.3g" % err.max()


def test_clusters_write_nothing_while_the_status_word_is_set():
    """200 x 512 x 2048 runs as clusters of eight CTAs; all of them leave C alone until the word is read, and work after."""
    M, N, K = 200, 512, 2048
    a, b = inputs.make_gemm_inputs(M, N, K, 5)
    dev = torch.device("cuda:0")
    ad, bd = a.to(dev), b.to(dev)
    c = torch.full((M, N), 7.0, dtype=torch.bfloat16, device=dev)
    assert binding.device_status() == (binding.AVE_OK, 0)
    assert binding.selftest_wait_timeout(16) == binding.AVE_OK
    binding.ave_gemm_bf16_tn(ad, bd, c)
    torch.cuda.synchronize()
    assert torch.all(c == 7.0)
    assert binding.device_status() == (binding.AVE_ERR_DEVICE_TIMEOUT, binding.STATUS_BIT_SELFTEST)
    binding.ave_gemm_bf16_tn(ad, bd, c)
    assert binding.device_status() == (binding.AVE_OK, 0)
    ref = oracle.gemm_tn(a, b)
    assert np.all(np.abs(c.cpu().double().numpy() - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-3 * math.sqrt(K))
