"""Compile the CUDA library for sm_100a with nvcc and the binding's C++ part with g++, in-tree.

``python -m paper_2604_18616_b200.build`` (or ``build_cuda()``) writes
``libave_attn.so`` and ``_fastcall.so`` next to this file.  nvcc cross-compiles without a GPU.

The build reads ptxas' resource report and refuses an image in which an
attention kernel got fewer registers per thread than its warp roles' register
split draws on (``setmaxnreg.inc`` beyond the CTA's allocation never returns),
or a kernel spills more than a pair of registers.
The library repeats the check at run time on the loaded image.
"""
from __future__ import annotations

import os
import re
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB_PATH = os.path.join(_HERE, "libave_attn.so")
FAST_PATH = os.path.join(_HERE, "_fastcall.so")
INCLUDE = os.path.join(os.path.dirname(_HERE), "include")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-shared", "-Xcompiler", "-fPIC",
    "-Xptxas", "-v",
]

# Register split of the attention kernel (WsCfg in csrc/attn_fwd_ws.cuh): 384 threads, of which one
# warpgroup keeps 64 registers per thread and two take 216 (72 and 208, which is less in all, in some instantiations).
ATTN_THREADS = 384
ATTN_REGS_NEEDED = 128 * 64 + 256 * 216
# The single-sub-tile kernel (OneCfg in csrc/attn_fwd_1t.cuh): 256 threads, 48 and 208 registers, or 56 and 200.
ONE_THREADS = 256
ONE_REGS_NEEDED = 128 * 48 + 128 * 208
# The MoE GEMM (MoeGemmCfg in csrc/moe_fp8.cuh): 384 threads, 56 and 224 registers.
MOE_THREADS = 384
MOE_REGS_NEEDED = 128 * 56 + 256 * 224
# What a kernel may spill, in bytes a thread: one pair of registers.  (The split-KV form of the two-sub-tile kernel at D = 128 and
# the MoE GEMM do.)
SPILL_BYTES_ALLOWED = 8


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))) + \
        [os.path.join(INCLUDE, h) for h in sorted(os.listdir(INCLUDE)) if h.endswith(".h")]


def kernel_registers(ptxas_report: str) -> dict:
    """{mangled kernel name: registers per thread} from ``-Xptxas -v`` output."""
    regs = {}
    current = None
    for line in ptxas_report.splitlines():
        m = re.search(r"Compiling entry function '([^']+)'", line)
        if m:
            current = m.group(1)
            continue
        m = re.search(r"Used (\d+) registers", line)
        if m and current:
            regs[current] = int(m.group(1))
            current = None
    return regs


def check_register_split(ptxas_report: str) -> dict:
    """Raise if an attention kernel of the report cannot satisfy its register split."""
    regs = {k: v for k, v in kernel_registers(ptxas_report).items() if ("attn_fwd" in k and "attn_fwd_pair" not in k) or "moe_gemm" in k}
    if not regs:
        raise RuntimeError("ptxas reported no attention kernel: cannot verify the register split")
    for name, n in regs.items():
        threads, needed = (ONE_THREADS, ONE_REGS_NEEDED) if "attn_fwd_1t" in name else \
            (MOE_THREADS, MOE_REGS_NEEDED) if "moe_gemm" in name else (ATTN_THREADS, ATTN_REGS_NEEDED)
        if threads * n < needed:
            raise RuntimeError("%s was compiled with %d registers per thread; its warp roles need %d x %d >= %d" % (
                name, n, threads, n, needed))
    return regs


def check_spills(ptxas_report: str) -> dict:
    """{mangled kernel name: bytes spilled}; raise if a kernel spills more than SPILL_BYTES_ALLOWED."""
    spills, current = {}, None
    for line in ptxas_report.splitlines():
        m = re.search(r"Compiling entry function '([^']+)'", line)
        if m:
            current = m.group(1)
        m = re.search(r"(\d+) bytes spill stores", line)
        if m and current:
            spills[current] = int(m.group(1))
    for name, n in spills.items():
        if n > SPILL_BYTES_ALLOWED:
            raise RuntimeError("%s spills %d bytes of registers" % (name, n))
    return spills


def fastcall_stamp() -> str:
    """What the extension is built for: it uses the C++ interface of this torch and the C interface of this Python."""
    import sysconfig

    import torch
    return "%s %s" % (torch.__version__, sysconfig.get_config_var("SOABI"))


def build_fastcall(force: bool = False) -> str:
    """The C++ part of the binding: a Python extension over torch's C++ library."""
    import sysconfig

    import torch
    src = os.path.join(CSRC, "fastcall.cc")
    tdir = os.path.dirname(torch.__file__)
    stamp, stamp_path = fastcall_stamp(), FAST_PATH + ".stamp"
    if not force and os.path.exists(FAST_PATH) and os.path.getmtime(FAST_PATH) >= os.path.getmtime(src) and os.path.exists(stamp_path):
        with open(stamp_path) as f:
            if f.read() == stamp:
                return FAST_PATH
    cuda_home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = FAST_PATH + ".tmp%d" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-I" + os.path.join(tdir, "include"), "-I" + os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           "-I" + os.path.join(cuda_home, "include"), "-I" + sysconfig.get_paths()["include"], "-o", tmp, src,
           "-L" + os.path.join(tdir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout)
        raise subprocess.CalledProcessError(r.returncode, cmd)
    os.replace(tmp, FAST_PATH)
    with open(stamp_path, "w") as f:
        f.write(stamp)
    return FAST_PATH


def build_cuda(force: bool = False, verbose: bool = False) -> str:
    build_fastcall(force)
    newest = max(os.path.getmtime(s) for s in _sources())
    if not force and os.path.exists(LIB_PATH) and os.path.getmtime(LIB_PATH) >= newest:
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB_PATH + ".tmp%d" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + ["-o", tmp, os.path.join(CSRC, "ave_attn.cu")]
    r = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout)
    if r.returncode != 0:
        raise subprocess.CalledProcessError(r.returncode, cmd)
    try:
        check_register_split(r.stdout)
        check_spills(r.stdout)
    except Exception:
        if os.path.exists(tmp):
            os.remove(tmp)
        raise
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build_cuda(force="--force" in sys.argv, verbose="-v" in sys.argv))
