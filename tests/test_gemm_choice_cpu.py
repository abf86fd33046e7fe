"""Which matrix-product kernel a product runs (csrc/gemm_choice.cuh), built with the host compiler."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WIDE = 0


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    out = os.path.join(str(tmp_path_factory.mktemp("gc")), "libgemm_choice_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-o", out, os.path.join(ROOT, "tests", "gemm_choice_host.cc")],
                   check=True)
    L = ctypes.CDLL(out)
    L.gc_choose.argtypes = [ctypes.c_int] * 5
    return lambda layout, M, N, K, sms=148: L.gc_choose(int(layout == "nn"), M, N, K, sms)


@pytest.mark.parametrize("M,N,K,tn,nn", [
    # measured: pairs / 128 x 256 tiles / single CTAs of 128 x 128 (us)
    (1, 65536, 512, WIDE, WIDE),       # 25.9 / 17.1 / 27.1
    (128, 19000, 2048, WIDE, WIDE),    # 28.0 / 21.2 / 26.1
    (128, 28672, 4096, WIDE, WIDE),    # 60.1 / 48.1 / 56.2
    (600, 14336, 4096, WIDE, WIDE),    # 67.8 / 60.5
    (64, 14336, 2048, 1, 1),           # 19.2 / 19.8 / 15.8
    (128, 9472, 512, 1, 1),            # 9.2 / 8.3 / 6.4
    (128, 4096, 4096, 4, 4),           # 24.5 / 27.7 / 20.0; clusters of four 13.2
    (200, 512, 8192, 8, 8),
    (1939, 440, 2416, 2, 2),
    (4096, 4096, 4096, -256, -256),    # 113 against 122
    (3001, 5112, 2056, -256, -256),
    (420, 6544, 3840, -192, -256),     # a tile width that fills the last wave
])
def test_choices_at_measured_sizes(choose, M, N, K, tn, nn):
    assert choose("tn", M, N, K) == tn and choose("nn", M, N, K) == nn


def test_every_choice_can_be_launched(choose):
    rng = random.Random(4)
    seen = set()
    for _ in range(20000):
        M, N, K = (int(2 ** rng.uniform(0, 14)) for _ in range(3))
        N, K, sms, layout = 8 * N, 8 * K, rng.choice([148, 148, 132, 2]), rng.choice(["tn", "nn"])
        c = choose(layout, M, N, K, sms)
        seen.add(c)
        slices, tiles = -(-K // 64), -(-M // 128) * -(-N // 128)
        if c > 0:
            assert c in (1, 2, 4, 8) and c * tiles <= sms and c <= slices   # all clusters resident, a slice for each CTA
        elif c < 0:
            assert M > 128 and -c in ((128, 256) if layout == "nn" else (64, 128, 192, 256))
    assert seen == {1, 2, 4, 8, WIDE, -64, -128, -192, -256}                   # no choice that nothing reaches
