// C-ABI entry points of the attention-forward library: argument validation,
// TMA tensor-map encoding, kernel selection and launch.  See include/ave_attn.h
// for the contract of every exported function.
#include "../../include/ave_attn.h"
#include "../../include/ave_gemm.h"
#include "../../include/ave_moe.h"

#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include "attn_fwd_ws.cuh"
#include "attn_fwd_1t.cuh"
#include "attn_fwd_pair.cuh"
#include "gemm_bf16.cuh"
#include "gemm_choice.cuh"
#include "moe_fp8.cuh"

// Scratch of ave_attn_fwd_splitkv_static: part of the device image, so every GPU that loads the
// library holds it until exit.  In host code this name is only a handle for
// cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_splitkv_static_scratch[AVE_SPLITKV_STATIC_SCRATCH_BYTES];

namespace {

thread_local int t_last_cuda_error = 0;
std::atomic<unsigned long long> g_launches{0};

constexpr int kVersion = 100;  // 0.1.0

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up through the runtime so the
// library does not link against libcuda.
EncodeTiledFn encode_fn() {
    static std::atomic<EncodeTiledFn> cached{nullptr};
    EncodeTiledFn f = cached.load(std::memory_order_acquire);
    if (f) return f;
    void *sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres);
    if (e != cudaSuccess || qres != cudaDriverEntryPointSuccess || !sym) {
        t_last_cuda_error = (e != cudaSuccess) ? int(e) : int(cudaErrorSymbolNotFound);
        return nullptr;
    }
    f = reinterpret_cast<EncodeTiledFn>(sym);
    cached.store(f, std::memory_order_release);
    return f;
}

std::atomic<int> g_inject_launch_failures{0};  // test hook: the next launches fail before reaching the GPU
std::atomic<int> g_inject_encode_failures{0};  // test hook: the next tensor-map encodes fail

bool take_injected(std::atomic<int> &counter) {
    int n = counter.load(std::memory_order_relaxed);
    while (n > 0)
        if (counter.compare_exchange_weak(n, n - 1, std::memory_order_relaxed)) return true;
    return false;
}

// Element strides of one tensor's batch, head and row dimensions (the D elements of a row are contiguous).
struct Strides {
    long long batch, head, row;
};
Strides contiguous_strides(int heads, int rows, int D) {
    return Strides{(long long)heads * rows * D, (long long)rows * D, (long long)D};
}

// bf16 tensor [batch, heads, rows, D] with the given strides as a 4-D map {D, rows, heads, batch} with a
// box of 64 columns x box_rows rows, 128-byte swizzle, zero fill outside the tensor.
struct MapKey {
    const void *base;
    int D, rows, heads, batch, box_rows;
    long long s_batch, s_head, s_row;
    bool operator==(const MapKey &o) const {
        return base == o.base && D == o.D && rows == o.rows && heads == o.heads && batch == o.batch &&
               box_rows == o.box_rows && s_batch == o.s_batch && s_head == o.s_head && s_row == o.s_row;
    }
};
// A tensor map is a pure function of its key (the encoder reads no device state), so repeated calls
// on the same buffers, the common case in a serving loop, reuse the encoded 128 bytes.  Per thread (no
// locks), 16 entries searched linearly and replaced in turn: the handful of maps of one call always fit.
struct MapCache {
    static constexpr int kEntries = 16;
    MapKey key[kEntries];
    CUtensorMap map[kEntries];
    bool valid[kEntries] = {};
    int next = 0;
    const CUtensorMap *find(const MapKey &k) const {
        for (int i = 0; i < kEntries; ++i)
            if (valid[i] && key[i] == k) return &map[i];
        return nullptr;
    }
    void insert(const MapKey &k, const CUtensorMap &m) {
        key[next] = k;
        map[next] = m;
        valid[next] = true;
        next = (next + 1) % kEntries;
    }
};
thread_local MapCache t_map_cache;
std::atomic<unsigned long long> g_map_encodes{0};  // encoder calls so far (a cache hit makes none)

bool encode_map(CUtensorMap *map, const void *base, int D, int rows, int heads, int batch, const Strides &st,
                int box_rows) {
    if (take_injected(g_inject_encode_failures)) {
        t_last_cuda_error = int(CUDA_ERROR_INVALID_VALUE);
        return false;
    }
    const MapKey key{base, D, rows, heads, batch, box_rows, st.batch, st.head, st.row};
    if (const CUtensorMap *hit = t_map_cache.find(key)) {
        *map = *hit;
        return true;
    }
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t gdim[4] = {cuuint64_t(D), cuuint64_t(rows), cuuint64_t(heads), cuuint64_t(batch)};
    cuuint64_t gstride[3] = {cuuint64_t(st.row) * 2, cuuint64_t(st.head) * 2, cuuint64_t(st.batch) * 2};
    cuuint32_t box[4] = {64, cuuint32_t(box_rows), 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), gdim, gstride, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    g_map_encodes.fetch_add(1, std::memory_order_relaxed);
    if (r != CUDA_SUCCESS) {
        t_last_cuda_error = int(r);
        return false;
    }
    t_map_cache.insert(key, *map);
    return true;
}

int validate(const void *q, const void *k, const void *v, const void *o, const void *lse, int B, int H, int Hkv,
             int Sq, int Sk, int D, float scale) {
    if (!q || !k || !v || !o || !lse) return AVE_ERR_NULL_POINTER;
    if (B <= 0 || H <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0 || D <= 0) return AVE_ERR_BAD_SHAPE;
    if (H % Hkv != 0) return AVE_ERR_BAD_SHAPE;
    if (Sq >= (1 << 30) || Sk >= (1 << 30)) return AVE_ERR_BAD_SHAPE;
    if ((long long)B * H >= (1ll << 31)) return AVE_ERR_BAD_SHAPE;
    if (D < 8 || D > 256 || D % 8 != 0) return AVE_ERR_UNSUPPORTED_D;
    const long long n_qblk = (Sq + ave::BM - 1) / ave::BM;
    if (n_qblk * B * H >= (1ll << 31)) return AVE_ERR_BAD_SHAPE;
    return -1;  // shape checks passed; pointer/scale checks follow
}

int validate_ptrs_and_scale(const void *q, const void *k, const void *v, const void *o, const void *lse,
                            float scale) {
    if ((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) |
         reinterpret_cast<uintptr_t>(o)) & 15u)
        return AVE_ERR_MISALIGNED;
    if (reinterpret_cast<uintptr_t>(lse) & 3u) return AVE_ERR_MISALIGNED;
    if (std::isnan(scale) || std::isinf(scale)) return AVE_ERR_BAD_SCALE;
    return AVE_OK;
}

int check_device() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    static std::atomic<int> ok_mask_lo{0};  // devices 0..30 already checked
    if (dev < 31 && (ok_mask_lo.load(std::memory_order_relaxed) >> dev) & 1) return AVE_OK;
    int major = 0;
    e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    if (major != 10) return AVE_ERR_UNSUPPORTED_DEVICE;
    if (dev < 31) ok_mask_lo.fetch_or(1 << dev, std::memory_order_relaxed);
    return AVE_OK;
}

// Per kernel instantiation: the devices (by ordinal) on which the kernel has been prepared.  The
// maximum dynamic shared-memory size is an attribute of a function ON ONE DEVICE, so a process that
// drives several GPUs has to set it once per device, not once per process.
struct PerDeviceOnce {
    std::atomic<unsigned long long> done{0};
    bool is_done(int dev) const { return dev >= 0 && dev < 64 && ((done.load(std::memory_order_acquire) >> dev) & 1ull); }
    void mark(int dev) {
        if (dev >= 0 && dev < 64) done.fetch_or(1ull << dev, std::memory_order_release);
    }
};

// The softmax warps raise their register count with setmaxnreg.inc, which can only draw on what
// the CTA was given at launch (threads x registers per thread as compiled).  A request beyond that
// never returns, so a kernel image compiled with fewer registers than the split assumes must not
// be launched at all.
bool register_split_fits(int regs_per_thread_at_launch) {
    using Cfg = ave::WsCfg<64>;  // (the largest sum of the instantiations)
    static_assert(Cfg::kRegsMoved == 0, "another instantiation has the largest sum");
    return 128 * Cfg::kRegsLight + 256 * Cfg::kRegsSoftmax <= Cfg::kThreads * regs_per_thread_at_launch;
}
bool register_split_fits_one_subtile(int regs_per_thread_at_launch) {
    using Cfg = ave::OneCfg<128>;
    return 128 * Cfg::kRegsLight + 128 * Cfg::kRegsSoftmax <= Cfg::kThreads * regs_per_thread_at_launch;
}

bool register_split_fits_moe_gemm(int regs_per_thread_at_launch) {
    using Cfg = ave::MoeGemmCfg<true>;
    return 128 * Cfg::kRegsLight + 256 * Cfg::kRegsEpilogue <= Cfg::kThreads * regs_per_thread_at_launch;
}

// Which attention kernel ordinary (not split-KV) launches use: 0 = chosen per problem, 1 = always the
// two-sub-tile kernel, 2 = always the single-sub-tile kernel (ave_attn_select_kernel).
std::atomic<int> g_kernel_choice{0};

// check_register_split: 0 = none, 1 = the two-sub-tile kernel's split, 2 = the single-sub-tile kernel's, 3 = the MoE GEMM's
template <class Kernel>
int prepare_kernel(Kernel kern, int smem_bytes, int check_register_split, PerDeviceOnce &once) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && once.is_done(dev)) return AVE_OK;
    if (e == cudaSuccess && check_register_split) {
        cudaFuncAttributes attr;
        e = cudaFuncGetAttributes(&attr, kern);
        if (e == cudaSuccess && !(check_register_split == 1   ? register_split_fits(attr.numRegs)
                                  : check_register_split == 2 ? register_split_fits_one_subtile(attr.numRegs)
                                                              : register_split_fits_moe_gemm(attr.numRegs)))
            return AVE_ERR_KERNEL_IMAGE;
    }
    // two CTAs of the single-sub-tile kernel share an SM: ask for the largest shared-memory carve-out
    if (e == cudaSuccess && check_register_split == 2)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    once.mark(dev);
    return AVE_OK;
}

// Launch a kernel that begins with grid_dependency_wait(): its blocks may be set up while the kernel before it in the
// stream still runs (programmatic dependent launch), which takes the launch latency out of a chain of kernels.  `cluster`:
// CTAs of a cluster.
template <class... Params, class... Args>
cudaError_t launch_dependent_clusters(void (*kern)(Params...), dim3 grid, dim3 block, int cluster, size_t smem, cudaStream_t s,
                                      Args... args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, Params(args)...);
}
template <class... Params, class... Args>
cudaError_t launch_dependent(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args) {
    return launch_dependent_clusters(kern, grid, block, 1, smem, s, args...);
}

template <int D, bool CAUSAL, bool SPLIT, bool VARLEN = false>
int launch_ws(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv, const CUtensorMap &to,
              const ave::FwdParams &p, cudaStream_t stream) {
    using Cfg = ave::WsCfg<D>;
    auto kern = ave::attn_fwd_ws_kernel<D, CAUSAL, SPLIT, VARLEN>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 1, once);
    if (st != AVE_OK) return st;
    if (take_injected(g_inject_launch_failures)) {
        t_last_cuda_error = int(cudaErrorLaunchFailure);
        return AVE_ERR_CUDA;
    }
    kern<<<dim3(p.total_blocks), dim3(Cfg::kThreads), Cfg::kSmemBytes, stream>>>(tq, tk, tv, to, p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}


template <int D, bool CAUSAL, bool SPLIT, bool VARLEN = false>
int launch_1t(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv, const ave::FwdParams &p,
              cudaStream_t stream) {
    using Cfg = ave::OneCfg<D>;
    auto kern = ave::attn_fwd_1t_kernel<D, CAUSAL, SPLIT, VARLEN>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 2, once);
    if (st != AVE_OK) return st;
    if (take_injected(g_inject_launch_failures)) {
        t_last_cuda_error = int(cudaErrorLaunchFailure);
        return AVE_ERR_CUDA;
    }
    cudaError_t e = launch_dependent(kern, dim3(p.total_blocks), dim3(Cfg::kThreads), Cfg::kSmemBytes, stream, tq, tk, tv, p);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

template <bool CAUSAL, bool VARLEN>
int launch_pair(const CUtensorMap &tq, const CUtensorMap &tk, const CUtensorMap &tv, const ave::FwdParams &p, cudaStream_t stream) {
    using Cfg = ave::PairCfg;
    auto kern = ave::attn_fwd_pair_kernel<CAUSAL, VARLEN>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 0, once);
    if (st != AVE_OK) return st;
    if (take_injected(g_inject_launch_failures)) {
        t_last_cuda_error = int(cudaErrorLaunchFailure);
        return AVE_ERR_CUDA;
    }
    const cudaError_t e = launch_dependent(kern, dim3(2u * unsigned(p.total_blocks)), dim3(Cfg::kThreads), Cfg::kSmemBytes, stream, tq,
                                           tk, tv, p);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

// Number of SMs of the current device (148, the part this library is written for, if it cannot be asked).
int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;
    return sms;
}

// Whether a launch of D <= 128 runs the single-sub-tile kernel (two CTAs per SM, 128-row tiles) instead of the two-sub-tile
// one.  total_q: query rows of all sequences of a variable-length launch, else 0.
bool use_one_subtile(int B, int H, int Hkv, int Sq, int Sk, int D, bool causal, bool split, int total_q) {
    const int choice = g_kernel_choice.load(std::memory_order_relaxed);
    if (choice == 1) return false;
    if (choice == 2) return true;
    // At most 128 query rows per problem (decode, one chunk of a chunked prefill; Sq counts the packed rows of a
    // head-packed split launch): the second sub-tile of a 256-row tile would be empty.  The single-sub-tile
    // kernel then keeps two independent K/V streams per SM in flight, which is what an HBM-bound pass needs
    // (measured on decode shapes: 0.63-0.66 -> 0.76-0.90 of the copy bandwidth).
    if (Sq <= ave::BM) return true;
    return !split && ave::one_subtile_is_faster(B, H, Hkv, Sq, Sk, D, causal, total_q, sm_count());
}

// Whether a launch of D > 128 runs on CTA pairs.
bool use_pairs(int B, int H, int Hkv, int Sq, int Sk, bool causal, int total_q) {
    const int choice = g_kernel_choice.load(std::memory_order_relaxed);
    // (a pair's grid, two CTAs a tile, must stay below 2^31)
    const long long blocks = ((long long)Sq + ave::BM - 1) / ave::BM * B * H;
    if (choice == 2 || blocks >= (1ll << 30)) return false;
    return choice == 1 || ave::pairs_are_faster(B, H, Hkv, Sq, Sk, causal, total_q, sm_count());
}

// Encode the tensor maps, fill the kernel parameters and launch.  In a `split` launch every work tile covers
// one range of keys_per_split keys and writes fp32 partials (with a single range and no partial buffers: the
// result itself).
// Variable-length launch: token-major tensors [rows, heads, D] and the sequences' row ranges.
struct VarlenArgs {
    const int *cu_q, *cu_k;  // device, B + 1 entries
    int total_q, total_k;
};

// `layout` (strides of q, k, v, o in this order) is NULL for contiguous [B, heads, rows, D] tensors; `varlen`
// is NULL unless the launch is a variable-length one (Sq and Sk are then the longest sequences).
int launch_attention(const void *q, const void *k, const void *v, void *o, float *lse, int B, int H, int Hkv, int Sq,
                     int Sk, int D, int causal, float scale, bool split, int n_splits, int keys_per_split,
                     float *o_partial, float *lse_partial, int rows_per_head, const Strides *layout,
                     const VarlenArgs *varlen, cudaStream_t s) {
    auto token_major = [&](int heads, int rows) { return Strides{(long long)rows * heads * D, (long long)D, (long long)heads * D}; };
    const int rows_q = varlen ? varlen->total_q : Sq, rows_k = varlen ? varlen->total_k : Sk, n_batch = varlen ? 1 : B;
    const Strides sq = layout ? layout[0] : varlen ? token_major(H, rows_q) : contiguous_strides(H, Sq, D);
    const Strides sk = layout ? layout[1] : varlen ? token_major(Hkv, rows_k) : contiguous_strides(Hkv, Sk, D);
    const Strides sv = layout ? layout[2] : varlen ? token_major(Hkv, rows_k) : contiguous_strides(Hkv, Sk, D);
    const Strides so = layout ? layout[3] : varlen ? token_major(H, rows_q) : contiguous_strides(H, Sq, D);
    // A head dimension above 128 leaves no TMEM for a second sub-tile in one CTA: CTA pairs, or the single-sub-tile kernel.
    const bool pair = D > 128 && use_pairs(B, H, Hkv, Sq, Sk, causal != 0, varlen ? varlen->total_q : 0);
    const bool one = D > 128 ? !pair : use_one_subtile(B, H, Hkv, Sq, Sk, D, causal != 0, split, varlen ? varlen->total_q : 0);
    CUtensorMap tq, tk, tv, to;
    if (!encode_map(&tq, q, D, rows_q, H, n_batch, sq, ave::BM)) return AVE_ERR_CUDA;
    // (the single-sub-tile kernel and the pairs store O without a map)
    if (!one && !pair && !encode_map(&to, o, D, rows_q, H, n_batch, so, ave::WsCfg<128>::kOutBoxRows)) return AVE_ERR_CUDA;
    if (!encode_map(&tk, k, D, rows_k, Hkv, n_batch, sk, pair ? ave::BN / 2 : ave::BN)) return AVE_ERR_CUDA;  // (a pair: half of the keys in each CTA)
    // (the single-sub-tile kernel takes V of head dimensions above 128 by halves of the keys, a pair by halves of the columns)
    if (!encode_map(&tv, v, D, rows_k, Hkv, n_batch, sv, D > 128 && one ? ave::BN / 2 : ave::BN)) return AVE_ERR_CUDA;

    ave::FwdParams p{};
    p.o = o;
    p.lse = lse;
    p.o_stride_b = so.batch;
    p.o_stride_h = so.head;
    p.o_stride_r = so.row;
    p.d_true = D;
    p.cu_q = varlen ? varlen->cu_q : nullptr;
    p.cu_k = varlen ? varlen->cu_k : nullptr;
    p.lse_stride_h = varlen ? varlen->total_q : 0;
    const int Dk = D <= 64 ? 64 : D <= 128 ? 128 : 256;  // the kernel's head dimension: TMA zero-fills the columns beyond D
    if (!ave::plan_work_tiles(p, B, H, Hkv, Sq, Sk, D, causal != 0, split, n_splits, keys_per_split, rows_per_head, one))
        return AVE_ERR_BAD_SHAPE;
    p.o_partial = o_partial;
    p.lse_partial = lse_partial;
    p.scale_log2 = scale * 1.4426950408889634f;

    if (pair) {
        if (varlen) return causal ? launch_pair<true, true>(tq, tk, tv, p, s) : launch_pair<false, true>(tq, tk, tv, p, s);
        return causal ? launch_pair<true, false>(tq, tk, tv, p, s) : launch_pair<false, false>(tq, tk, tv, p, s);
    }
    if (one && Dk == 256) {  // (the split-KV entry points take 64 or 128 only)
        if (varlen)
            return causal ? launch_1t<256, true, false, true>(tq, tk, tv, p, s) : launch_1t<256, false, false, true>(tq, tk, tv, p, s);
        return causal ? launch_1t<256, true, false>(tq, tk, tv, p, s) : launch_1t<256, false, false>(tq, tk, tv, p, s);
    }
    if (one) {
        if (split) {
            if (Dk == 128)
                return causal ? launch_1t<128, true, true>(tq, tk, tv, p, s) : launch_1t<128, false, true>(tq, tk, tv, p, s);
            return causal ? launch_1t<64, true, true>(tq, tk, tv, p, s) : launch_1t<64, false, true>(tq, tk, tv, p, s);
        }
        if (varlen) {
            if (Dk == 128)
                return causal ? launch_1t<128, true, false, true>(tq, tk, tv, p, s)
                              : launch_1t<128, false, false, true>(tq, tk, tv, p, s);
            return causal ? launch_1t<64, true, false, true>(tq, tk, tv, p, s)
                          : launch_1t<64, false, false, true>(tq, tk, tv, p, s);
        }
        if (Dk == 128)
            return causal ? launch_1t<128, true, false>(tq, tk, tv, p, s) : launch_1t<128, false, false>(tq, tk, tv, p, s);
        return causal ? launch_1t<64, true, false>(tq, tk, tv, p, s) : launch_1t<64, false, false>(tq, tk, tv, p, s);
    }
    if (split) {
        if (Dk == 128)
            return causal ? launch_ws<128, true, true>(tq, tk, tv, to, p, s) : launch_ws<128, false, true>(tq, tk, tv, to, p, s);
        return causal ? launch_ws<64, true, true>(tq, tk, tv, to, p, s) : launch_ws<64, false, true>(tq, tk, tv, to, p, s);
    }
    if (varlen) {
        if (Dk == 128)
            return causal ? launch_ws<128, true, false, true>(tq, tk, tv, to, p, s)
                          : launch_ws<128, false, false, true>(tq, tk, tv, to, p, s);
        return causal ? launch_ws<64, true, false, true>(tq, tk, tv, to, p, s)
                      : launch_ws<64, false, false, true>(tq, tk, tv, to, p, s);
    }
    if (Dk == 128)
        return causal ? launch_ws<128, true, false>(tq, tk, tv, to, p, s) : launch_ws<128, false, false>(tq, tk, tv, to, p, s);
    return causal ? launch_ws<64, true, false>(tq, tk, tv, to, p, s) : launch_ws<64, false, false>(tq, tk, tv, to, p, s);
}

__device__ __forceinline__ bool status_word_is_set() {
    return *reinterpret_cast<volatile unsigned int *>(&ave::g_device_status) != 0;
}

// Combine the partial results of the key ranges of every query row:
//   LSE = ln sum_s exp(LSE_s),  O = sum_s exp(LSE_s - LSE) * O_s.
// One or more warps per row (`warps_per_row`, a power of two up to 8), which share out the row's key ranges; a lane
// holds four neighbouring output columns (at D = 64 the half-warps take ranges in turn).  The bound is latency: a decode step has few rows and up to
// 64 ranges, and a thread that walks the ranges by itself waits for one load after the other (measured with 32 rows
// and 37 ranges: 23 us for a thread per 8 columns, 4 us with eight warps per row).  Many rows: splitkv_merge_rows_kernel.
constexpr int kMergeThreads = 256;
__global__ void __launch_bounds__(kMergeThreads)
splitkv_merge_kernel(const float *__restrict__ o_partial, const float *__restrict__ lse_partial,
                     __nv_bfloat16 *__restrict__ o, float *__restrict__ lse, long long rows, int D, int n_splits,
                     int warps_per_row) {
    __shared__ float4 part[kMergeThreads];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = warp & (warps_per_row - 1);  // which of the row's warps
    const long long row = (long long)blockIdx.x * (kMergeThreads / 32 / warps_per_row) + warp / warps_per_row;
    const bool live = row < rows;
    ave::grid_dependency_wait();
    const bool skip = status_word_is_set();  // (the partials were not written)
    const int lanes_per_range = D / 4, ranges_at_once = 32 / lanes_per_range;  // 32 and 1, or 16 and 2
    const int col4 = lane & (lanes_per_range - 1);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float m = -INFINITY, denom = 0.f;
    if (live) {
        // the ranges' weights: lane l holds those of ranges l and l + 32
        static_assert(AVE_SPLITKV_MAX_SPLITS <= 64, "two ranges per lane");
        const float l0 = lane < n_splits ? lse_partial[lane * rows + row] : -INFINITY;
        const float l1 = lane + 32 < n_splits ? lse_partial[(lane + 32) * rows + row] : -INFINITY;
        m = fmaxf(l0, l1);
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, x));
        const float w0 = m == -INFINITY ? 0.f : __expf(l0 - m);
        const float w1 = m == -INFINITY ? 0.f : __expf(l1 - m);
        denom = w0 + w1;
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) denom += __shfl_xor_sync(0xffffffffu, denom, x);
        const int stride = warps_per_row * ranges_at_once;
        const int n = m == -INFINITY ? 0 : n_splits;  // (a row that sees no key in any range: what the partials hold is not looked at)
#pragma unroll 4
        for (int s0 = sub * ranges_at_once; s0 < n; s0 += stride) {
            const int s = s0 + lane / lanes_per_range;
            const float w_lo = __shfl_sync(0xffffffffu, w0, s & 31), w_hi = __shfl_sync(0xffffffffu, w1, s & 31);
            const float ws = s < 32 ? w_lo : w_hi;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);  // (beyond the last range: nothing, not 0 x another range's infinity)
            if (s < n_splits) v = reinterpret_cast<const float4 *>(o_partial + (s * rows + row) * D)[col4];
            acc.x += ws * v.x; acc.y += ws * v.y; acc.z += ws * v.z; acc.w += ws * v.w;
        }
    }
    if (ranges_at_once == 2) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 16); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 16);
        acc.z += __shfl_xor_sync(0xffffffffu, acc.z, 16); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, 16);
    }
    if (warps_per_row > 1) {
        part[threadIdx.x] = acc;
        __syncthreads();
        if (sub != 0) return;
        for (int x = 1; x < warps_per_row; ++x) {
            const float4 v = part[threadIdx.x + x * 32];
            acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
        }
    }
    if (!live || skip) return;
    const float inv = denom > 0.f ? 1.f / denom : 0.f;
    if (lane < lanes_per_range) {
        uint2 out;
        out.x = ave::pack_bf16x2(acc.x * inv, acc.y * inv);
        out.y = ave::pack_bf16x2(acc.z * inv, acc.w * inv);
        reinterpret_cast<uint2 *>(o + row * D)[col4] = out;
    }
    if (lane == 0) lse[row] = (denom > 0.f) ? m + logf(denom) : -INFINITY;
}

// The same with a thread per row and 8 output columns that walks the ranges, for many rows, where the chip is full of loads
// anyway and a warp that shares out one row spends its time on shuffles and tails (measured, this / warps sharing rows:
// 524288 rows of 3 ranges, D = 64 98 / 229 us; 131072 rows of 4 ranges, D = 128 57 / 83 us).
__global__ void __launch_bounds__(kMergeThreads)
splitkv_merge_rows_kernel(const float *__restrict__ o_partial, const float *__restrict__ lse_partial,
                          __nv_bfloat16 *__restrict__ o, float *__restrict__ lse, long long rows, int D, int n_splits) {
    const int chunks = D / 8;
    const long long idx = (long long)blockIdx.x * kMergeThreads + threadIdx.x;
    ave::grid_dependency_wait();
    const bool skip = status_word_is_set();
    const long long row = idx / chunks;
    const int ch = int(idx - row * chunks);
    if (row >= rows) return;
    float m = -INFINITY;
#pragma unroll 4
    for (int s = 0; s < n_splits; ++s) m = fmaxf(m, lse_partial[s * rows + row]);
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float denom = 0.f;
    const int n = m == -INFINITY ? 0 : n_splits;  // (a row that sees no key in any range: what the partials hold is not looked at)
#pragma unroll 4
    for (int s = 0; s < n; ++s) {
        const float w = __expf(lse_partial[s * rows + row] - m);
        denom += w;
        const float4 *src = reinterpret_cast<const float4 *>(o_partial + (s * rows + row) * D + ch * 8);
        const float4 a = src[0], b = src[1];
        acc[0] += w * a.x; acc[1] += w * a.y; acc[2] += w * a.z; acc[3] += w * a.w;
        acc[4] += w * b.x; acc[5] += w * b.y; acc[6] += w * b.z; acc[7] += w * b.w;
    }
    if (skip) return;
    const float inv = denom > 0.f ? 1.f / denom : 0.f;
    uint4 out;
    out.x = ave::pack_bf16x2(acc[0] * inv, acc[1] * inv);
    out.y = ave::pack_bf16x2(acc[2] * inv, acc[3] * inv);
    out.z = ave::pack_bf16x2(acc[4] * inv, acc[5] * inv);
    out.w = ave::pack_bf16x2(acc[6] * inv, acc[7] * inv);
    reinterpret_cast<uint4 *>(o + row * D)[ch] = out;
    if (ch == 0) lse[row] = (denom > 0.f) ? m + logf(denom) : -INFINITY;
}

// One warp waits, with the library's bounded wait, on an mbarrier that nobody ever arrives on: the
// wait must give up after `limit_cycles`, record its code in the device status word and return.
__global__ void wait_timeout_selftest_kernel(long long limit_cycles) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        ave::mbar_init(ave::smem_u32(&bar), 1);
        ave::fence_mbar_init();
    }
    __syncthreads();
    ave::mbar_wait_bounded(ave::smem_u32(&bar), 0, &abort_flag, ave::STATUS_TIMEOUT_SELFTEST, limit_cycles);
}

int run_splitkv(const void *q, const void *k, const void *v, void *o, float *lse, int B, int H, int Hkv, int Sq,
                int Sk, int D, int causal, float scale, int n_splits, float *o_partial, float *lse_partial,
                cudaStream_t s) {
    const int kps = ave::splitkv_keys_per_split(Sk, n_splits);
    const int G = H / Hkv;
    const bool pack = ave::splitkv_packs_heads(H, Hkv, Sq);  // query heads of a KV head as rows of one problem
    // A single key range needs no merge: the attention kernel writes the result.  (It makes the O of a row without any visible
    // key by a product with 0, which infinite values turn into NaN, where the merge writes zeros.)
    const bool merge = n_splits > 1 || (causal && Sq > Sk);
    float *const op = merge ? o_partial : nullptr;
    float *const lp = merge ? lse_partial : nullptr;
    const int st = pack ? launch_attention(q, k, v, o, lse, B, Hkv, Hkv, G * Sq, Sk, D, causal, scale, true, n_splits, kps,
                                           op, lp, Sq, nullptr, nullptr, s)
                        : launch_attention(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, causal, scale, merge, n_splits,
                                           kps, op, lp, 0, nullptr, nullptr, s);
    if (st != AVE_OK || !merge) return st;
    const long long rows = (long long)B * H * Sq;
    __nv_bfloat16 *const out = static_cast<__nv_bfloat16 *>(o);
    cudaError_t e;
    // The row-wise merge takes some 1.7 us and 0.23 us a range until its loads fill the chip, the other one a time that goes
    // with rows x ranges (times at splitkv_merge_rows_kernel; at the line, 4096 rows, D = 64: 8 ranges 3.4 / 3.6 us, 16 ranges
    // 5.5 / 4.6; 8192 rows of 64 ranges 43 / 46; 32 rows of 32 ranges, D = 128 8.9 / 2.9)
    const long long threads = rows * (D / 8);
    if (threads >= 65536 || threads >= 3300ll * n_splits) {
        e = launch_dependent(splitkv_merge_rows_kernel, dim3(unsigned((threads + kMergeThreads - 1) / kMergeThreads)),
                             dim3(kMergeThreads), 0, s, o_partial, lse_partial, out, lse, rows, D, n_splits);
    } else {
        // enough warps to cover the chip a few times over, none with less than two ranges to add up
        constexpr int kWarps = kMergeThreads / 32;
        const long long enough = 16ll * sm_count();
        int wpr = 1;
        while (wpr < kWarps && rows * wpr < enough && 4 * wpr <= n_splits) wpr *= 2;
        e = launch_dependent(splitkv_merge_kernel, dim3(unsigned((rows * wpr + kWarps - 1) / kWarps)), dim3(kMergeThreads), 0, s,
                             o_partial, lse_partial, out, lse, rows, D, n_splits, wpr);
    }
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}


// C[M, N] = A[M, K] * B[N, K]^T (or * B[K, N]) in 128 x 128 tiles, one cluster of `splits` CTAs each.
template <bool B_NMAJOR>
int launch_gemm_tile(const void *a, const void *b, void *c, int M, int N, int K, int splits, cudaStream_t s) {
    using Cfg = ave::GemmCfg;
    CUtensorMap ta, tb, tc;
    const Strides sa{(long long)M * K, (long long)M * K, (long long)K};
    const Strides sb{(long long)N * K, (long long)N * K, (long long)(B_NMAJOR ? N : K)};
    const Strides sc{(long long)M * N, (long long)M * N, (long long)N};
    if (!encode_map(&ta, a, K, M, 1, 1, sa, Cfg::kTileM)) return AVE_ERR_CUDA;
    if (B_NMAJOR) {  // B [K, N]: rows of N elements, boxes of 64 columns x 64 rows of K
        if (!encode_map(&tb, b, N, K, 1, 1, sb, Cfg::kSliceK)) return AVE_ERR_CUDA;
    } else {         // B [N, K]: rows of K elements, boxes of 64 columns of K x the tile's rows
        if (!encode_map(&tb, b, K, N, 1, 1, sb, Cfg::kTileN)) return AVE_ERR_CUDA;
    }
    if (!encode_map(&tc, c, N, M, 1, 1, sc, Cfg::kOutBoxRows)) return AVE_ERR_CUDA;
    ave::GemmParams p{};
    p.M = M;
    p.N = N;
    p.K = K;
    p.tiles_m = (M + Cfg::kTileM - 1) / Cfg::kTileM;
    p.tiles_n = (N + Cfg::kTileN - 1) / Cfg::kTileN;
    p.group_m = 16;
    p.splits = splits;
    p.c = c;
    auto kern = ave::gemm_bf16_kernel<B_NMAJOR>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 0, once);
    if (st != AVE_OK) return st;
    cudaError_t e = launch_dependent_clusters(kern, dim3(unsigned(p.tiles_m) * p.tiles_n * splits), dim3(Cfg::kThreads), splits,
                                              Cfg::kSmemBytes, s, ta, tb, tc, p);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

// The same in 128 x 256 tiles of one CTA each.
template <bool B_NMAJOR>
int launch_gemm_wide(const void *a, const void *b, void *c, int M, int N, int K, int sms, cudaStream_t s) {
    using Cfg = ave::GemmWideCfg;
    CUtensorMap ta, tb, tc;
    const Strides sa{(long long)M * K, (long long)M * K, (long long)K};
    const Strides sb{(long long)N * K, (long long)N * K, (long long)(B_NMAJOR ? N : K)};
    const Strides sc{(long long)M * N, (long long)M * N, (long long)N};
    if (!encode_map(&ta, a, K, M, 1, 1, sa, Cfg::kTileM)) return AVE_ERR_CUDA;
    if (B_NMAJOR) {  // B [K, N]: rows of N elements, boxes of 64 columns x 64 rows of K
        if (!encode_map(&tb, b, N, K, 1, 1, sb, Cfg::kSliceK)) return AVE_ERR_CUDA;
    } else {         // B [N, K]: rows of K elements, boxes of 64 columns of K x the tile's columns
        if (!encode_map(&tb, b, K, N, 1, 1, sb, Cfg::kTileN)) return AVE_ERR_CUDA;
    }
    if (!encode_map(&tc, c, N, M, 1, 1, sc, Cfg::kOutBoxRows)) return AVE_ERR_CUDA;
    ave::GemmParams p{};
    p.M = M;
    p.N = N;
    p.K = K;
    p.tiles_m = (M + Cfg::kTileM - 1) / Cfg::kTileM;
    p.tiles_n = (N + Cfg::kTileN - 1) / Cfg::kTileN;
    p.group_m = 16;  // the ~148 tiles in flight cover 16 x 9.25 tiles, a near-square part of C
    auto kern = ave::gemm_bf16_wide_kernel<B_NMAJOR>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 0, once);
    if (st != AVE_OK) return st;
    const long long n_tiles = (long long)p.tiles_m * p.tiles_n;
    const dim3 grid(unsigned(n_tiles < sms ? n_tiles : sms));
    cudaError_t e;
    if (M <= 16 && K > 1024 && n_tiles > sms / 2 && n_tiles < sms) {
        // The early launch is slower here, and only here (75 to 147 CTAs, at most 16 rows, K of 2048 and 4096: 5 % on average, up
        // to 27 %; elsewhere it is 5-25 % faster): presumably because it puts the CTAs wherever the kernel before has left
        // room, some side by side on a pair of SMs and on others none, in a kernel that is bound by fetching B.
        kern<<<grid, dim3(Cfg::kThreads), Cfg::kSmemBytes, s>>>(ta, tb, tc, p);
        e = cudaGetLastError();
    } else {
        e = launch_dependent(kern, grid, dim3(Cfg::kThreads), Cfg::kSmemBytes, s, ta, tb, tc, p);
    }
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

// The same on CTA pairs, with tiles of 256 x tile_n.
template <bool B_NMAJOR>
int launch_gemm_pair(const void *a, const void *b, void *c, int M, int N, int K, int tile_n, int sms, cudaStream_t s) {
    using Cfg = ave::GemmPairCfg;
    CUtensorMap ta, tb, tc;
    const Strides sa{(long long)M * K, (long long)M * K, (long long)K};
    const Strides sb{(long long)N * K, (long long)N * K, (long long)(B_NMAJOR ? N : K)};
    const Strides sc{(long long)M * N, (long long)M * N, (long long)N};
    if (!encode_map(&ta, a, K, M, 1, 1, sa, 128)) return AVE_ERR_CUDA;
    if (B_NMAJOR) {  // B [K, N]: rows of N elements, boxes of 64 columns x 64 rows of K
        if (!encode_map(&tb, b, N, K, 1, 1, sb, Cfg::kSliceK)) return AVE_ERR_CUDA;
    } else {         // B [N, K]: rows of K elements, boxes of 64 columns of K x half of the tile's columns
        if (!encode_map(&tb, b, K, N, 1, 1, sb, tile_n / 2)) return AVE_ERR_CUDA;
    }
    if (!encode_map(&tc, c, N, M, 1, 1, sc, Cfg::kOutBoxRows)) return AVE_ERR_CUDA;
    ave::GemmParams p{};
    p.M = M;
    p.N = N;
    p.K = K;
    p.tiles_m = (M + Cfg::kTileM - 1) / Cfg::kTileM;
    p.tile_n = tile_n;
    p.tiles_n = (N + tile_n - 1) / tile_n;
    p.group_m = 8;  // the ~74 tiles in flight cover 8 x 9.25 tiles, a near-square part of C
    auto kern = ave::gemm_bf16_pair_kernel<B_NMAJOR>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 0, once);
    if (st != AVE_OK) return st;
    const long long n_tiles = (long long)p.tiles_m * p.tiles_n;
    const long long pairs = n_tiles < sms / 2 ? n_tiles : sms / 2;
    cudaError_t e = launch_dependent(kern, dim3(unsigned(2 * pairs)), dim3(Cfg::kThreads), Cfg::kSmemBytes, s, ta, tb, tc, p);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

template <bool B_NMAJOR>
int launch_gemm(const void *a, const void *b, void *c, int M, int N, int K, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || sms <= 0) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    const ave::GemmChoice g = ave::choose_gemm(B_NMAJOR, M, N, K, sms);
    if (g.splits > 0) return launch_gemm_tile<B_NMAJOR>(a, b, c, M, N, K, g.splits, s);
    if (g.tile_n > 0) return launch_gemm_pair<B_NMAJOR>(a, b, c, M, N, K, g.tile_n, sms, s);
    return launch_gemm_wide<B_NMAJOR>(a, b, c, M, N, K, sms, s);
}

// E4M3 codes [d2, rows, inner] (inner contiguous) as a 4-D map with boxes of 128 bytes x box_rows rows, 128-byte
// swizzle, zero fill outside.  (Not cached: two encodes per GEMM of a layer call.)
bool encode_map_u8(CUtensorMap *map, const void *base, long long inner, long long rows, long long d2, int box_rows) {
    if (take_injected(g_inject_encode_failures)) {
        t_last_cuda_error = int(CUDA_ERROR_INVALID_VALUE);
        return false;
    }
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t gdim[4] = {cuuint64_t(inner), cuuint64_t(rows), cuuint64_t(d2), 1};
    cuuint64_t gstride[3] = {cuuint64_t(inner), cuuint64_t(inner) * cuuint64_t(rows), cuuint64_t(inner) * cuuint64_t(rows) * cuuint64_t(d2)};
    cuuint32_t box[4] = {128, cuuint32_t(box_rows), 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void *>(base), gdim, gstride, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    g_map_encodes.fetch_add(1, std::memory_order_relaxed);
    if (r != CUDA_SUCCESS) {
        t_last_cuda_error = int(r);
        return false;
    }
    return true;
}

// fp32 matrix [rows, cols] as a 4-D map {cols, rows, 1, 1} with boxes of 32 columns x 32 rows, 128-byte swizzle.
bool encode_map_f32(CUtensorMap *map, const void *base, long long cols, long long rows) {
    if (take_injected(g_inject_encode_failures)) {
        t_last_cuda_error = int(CUDA_ERROR_INVALID_VALUE);
        return false;
    }
    EncodeTiledFn enc = encode_fn();
    if (!enc) return false;
    cuuint64_t gdim[4] = {cuuint64_t(cols), cuuint64_t(rows), 1, 1};
    cuuint64_t gstride[3] = {cuuint64_t(cols) * 4, cuuint64_t(cols) * cuuint64_t(rows) * 4, cuuint64_t(cols) * cuuint64_t(rows) * 4};
    cuuint32_t box[4] = {32, 32, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(base), gdim, gstride, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    g_map_encodes.fetch_add(1, std::memory_order_relaxed);
    if (r != CUDA_SUCCESS) {
        t_last_cuda_error = int(r);
        return false;
    }
    return true;
}

// Scratch of one fused-MoE call, carved out of the caller's workspace (every part 256-byte aligned).
struct MoeWorkspace {
    long long rows_cap;  // rows of the sorted order, padding included: a multiple of 128
    size_t xq_s, sx_s, o, aq, sa, row_of, w_s, counts, cursor, tiles, n_row_tiles, total;
};
bool moe_layout(MoeWorkspace &w, int T, int C, int F, int E, int K) {
    if (T <= 0 || C <= 0 || F <= 0 || E <= 0 || K <= 0 || C % 128 || F % 128 || E > 1024) return false;
    const long long pairs = (long long)T * K;
    if (pairs >= (1ll << 24)) return false;
    w.rows_cap = 128 * ((pairs + 127) / 128 + E);  // sum over experts of ceil(rows / 128) tiles is at most this many
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = (off + bytes + 255) & ~size_t(255);
        return at;
    };
    const size_t rows = size_t(w.rows_cap);
    w.xq_s = take(rows * C);
    w.sx_s = take(rows * (C / 128) * 4);
    w.o = take(rows * size_t(C) * 4);
    w.aq = take(rows * F);
    w.sa = take(rows * (F / 128) * 4);
    w.row_of = take(size_t(pairs) * 4);
    w.w_s = take(rows * 4);
    w.counts = take(size_t(E) * 4);
    w.cursor = take(size_t(E) * 4);
    w.tiles = take(rows / 128 * sizeof(ave::MoeRowTile));
    w.n_row_tiles = take(4);
    w.total = off;
    return true;
}

// One GEMM of the layer: A codes [rows_cap, K], B codes [E, N, K]; `out` (down projection): fp32 [rows_cap, N].
template <bool UP>
int launch_moe_gemm(const void *a, const void *b, int E, int N, int K, float *out, ave::MoeGemmParams p, int sms, cudaStream_t s) {
    using Cfg = ave::MoeGemmCfg<UP>;
    CUtensorMap ta, tb, tc{};
    if (!encode_map_u8(&ta, a, K, p.rows_cap, 1, Cfg::kBoxRows)) return AVE_ERR_CUDA;
    if (!encode_map_u8(&tb, b, K, N, E, 128)) return AVE_ERR_CUDA;
    if (!UP && !encode_map_f32(&tc, out, N, p.rows_cap)) return AVE_ERR_CUDA;
    p.nblk = N / 128;
    p.tiles_n = (p.nblk + 1) / 2;  // 256 columns per tile (up: 128 of the gate and 128 of the up half)
    p.kb = K / 128;
    auto kern = ave::moe_gemm_fp8_kernel<UP>;
    static PerDeviceOnce once;  // per instantiation
    const int st = prepare_kernel(kern, Cfg::kSmemBytes, 3, once);
    if (st != AVE_OK) return st;
    if (take_injected(g_inject_launch_failures)) {
        t_last_cuda_error = int(cudaErrorLaunchFailure);
        return AVE_ERR_CUDA;
    }
    const long long n_tiles = p.rows_cap / 128 * p.tiles_n;
    const unsigned grid = unsigned(n_tiles < sms ? n_tiles : sms);
    cudaError_t e = launch_dependent(kern, dim3(grid), dim3(Cfg::kThreads), Cfg::kSmemBytes, s, ta, tb, tc, p);
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

// One of the layer's small kernels has been launched with status e: count it or report the launch error.
int after_small_launch(cudaError_t e) {
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

}  // namespace

extern "C" {

size_t ave_moe_workspace_bytes(int T, int C, int F, int E, int K) {
    MoeWorkspace w;
    return moe_layout(w, T, C, F, E, K) ? w.total : 0;
}

int ave_moe_fused_fwd(const void *xq, const float *sx, const void *w13q, const float *s13, const void *w2q,
                      const float *s2, const int *ids, const float *wts, void *y, int T, int C, int F, int E, int K,
                      void *workspace, size_t workspace_bytes, void *stream) {
    if (!xq || !sx || !w13q || !s13 || !w2q || !s2 || !ids || !wts || !y) return AVE_ERR_NULL_POINTER;
    MoeWorkspace w;
    if (!moe_layout(w, T, C, F, E, K)) return AVE_ERR_BAD_SHAPE;
    if ((reinterpret_cast<uintptr_t>(xq) | reinterpret_cast<uintptr_t>(w13q) | reinterpret_cast<uintptr_t>(w2q) |
         reinterpret_cast<uintptr_t>(y)) & 15u)
        return AVE_ERR_MISALIGNED;
    if ((reinterpret_cast<uintptr_t>(sx) | reinterpret_cast<uintptr_t>(s13) | reinterpret_cast<uintptr_t>(s2) |
         reinterpret_cast<uintptr_t>(ids) | reinterpret_cast<uintptr_t>(wts)) & 3u)
        return AVE_ERR_MISALIGNED;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < w.total) return AVE_ERR_WORKSPACE;
    int st = check_device();
    if (st != AVE_OK) return st;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess || sms <= 0) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint8_t *base = static_cast<uint8_t *>(workspace);
    uint8_t *xq_s = base + w.xq_s;
    float *sx_s = reinterpret_cast<float *>(base + w.sx_s);
    float *o = reinterpret_cast<float *>(base + w.o);
    uint8_t *aq = base + w.aq;
    float *sa = reinterpret_cast<float *>(base + w.sa);
    int *row_of = reinterpret_cast<int *>(base + w.row_of);
    float *w_s = reinterpret_cast<float *>(base + w.w_s);
    int *counts = reinterpret_cast<int *>(base + w.counts);
    int *cursor = reinterpret_cast<int *>(base + w.cursor);
    ave::MoeRowTile *tiles = reinterpret_cast<ave::MoeRowTile *>(base + w.tiles);
    int *n_row_tiles = reinterpret_cast<int *>(base + w.n_row_tiles);
    const int pairs = T * K;

    // 1.-3. pairs per expert, rows and row tiles of every expert
    ave::moe_clear_kernel<<<1, 256, 0, s>>>(counts, E);
    if ((st = after_small_launch(cudaGetLastError())) != AVE_OK) return st;
    const int count_ctas = (pairs + 2047) / 2048 < 2 * sms ? (pairs + 2047) / 2048 : 2 * sms;
    st = after_small_launch(launch_dependent(ave::moe_count_kernel, dim3(count_ctas), dim3(512), size_t(E) * sizeof(int), s, ids,
                                             pairs, E, counts));
    if (st != AVE_OK) return st;
    st = after_small_launch(launch_dependent(ave::moe_plan_kernel, dim3(1), dim3(1024), 0, s, counts, E, cursor, tiles, n_row_tiles));
    if (st != AVE_OK) return st;
    // 4. the tokens' codes and scales in sorted order
    st = after_small_launch(launch_dependent(ave::moe_gather_kernel, dim3(T), dim3(ave::kMoeGatherThreads), 0, s,
                                             static_cast<const uint8_t *>(xq), sx, ids, wts, C, E, K, w.rows_cap, cursor, row_of, xq_s,
                                             sx_s, w_s));
    if (st != AVE_OK) return st;
    // 5. up projection, activation and requantisation
    ave::MoeGemmParams p{};
    p.tiles = tiles;
    p.n_row_tiles = n_row_tiles;
    p.rows_cap = w.rows_cap;
    p.a_scale = sx_s;
    p.b_scale = s13;
    p.q_out = aq;
    p.q_scale = sa;
    st = launch_moe_gemm<true>(xq_s, w13q, E, 2 * F, C, nullptr, p, sms, s);
    if (st != AVE_OK) return st;
    // 6. down projection, weighted: o = w * (a W2^T)
    p.a_scale = sa;
    p.b_scale = s2;
    p.row_weight = w_s;
    st = launch_moe_gemm<false>(aq, w2q, E, C, F, o, p, sms, s);
    if (st != AVE_OK) return st;
    // 7. every token's K rows summed
    const long long n = (long long)T * (C / 4);
    return after_small_launch(launch_dependent(ave::moe_combine_kernel, dim3(unsigned((n + 255) / 256)), dim3(256), 0, s, o, row_of, T,
                                               C, K, static_cast<__nv_bfloat16 *>(y)));
}

int ave_attn_fwd(const void *q, const void *k, const void *v, void *o, float *lse, int B, int H, int Hkv, int Sq,
                 int Sk, int D, int causal, float scale, void *stream) {
    int st = validate(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, scale);
    if (st >= 0) return st;
    st = validate_ptrs_and_scale(q, k, v, o, lse, scale);
    if (st != AVE_OK) return st;
    st = check_device();
    if (st != AVE_OK) return st;
    return launch_attention(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, causal, scale, false, 1, 0, nullptr, nullptr, 0, nullptr,
                            nullptr, static_cast<cudaStream_t>(stream));
}

int ave_attn_fwd_strided(const void *q, const void *k, const void *v, void *o, float *lse, int B, int H, int Hkv,
                         int Sq, int Sk, int D, const long long *q_strides, const long long *k_strides,
                         const long long *v_strides, const long long *o_strides, int causal, float scale,
                         void *stream) {
    if (!q_strides || !k_strides || !v_strides || !o_strides) return AVE_ERR_NULL_POINTER;
    int st = validate(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, scale);
    if (st >= 0) return st;
    Strides layout[4];
    const long long *in[4] = {q_strides, k_strides, v_strides, o_strides};
    for (int i = 0; i < 4; ++i) {
        layout[i] = Strides{in[i][0], in[i][1], in[i][2]};
        if (layout[i].batch <= 0 || layout[i].head <= 0 || layout[i].row < D) return AVE_ERR_BAD_SHAPE;
        if (layout[i].batch >= (1ll << 38) || layout[i].head >= (1ll << 38) || layout[i].row >= (1ll << 38))
            return AVE_ERR_BAD_SHAPE;  // the tensor map holds byte strides below 2^40
    }
    for (int i = 0; i < 4; ++i)
        if ((layout[i].batch | layout[i].head | layout[i].row) & 7) return AVE_ERR_MISALIGNED;  // 16-byte units
    st = validate_ptrs_and_scale(q, k, v, o, lse, scale);
    if (st != AVE_OK) return st;
    st = check_device();
    if (st != AVE_OK) return st;
    return launch_attention(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, causal, scale, false, 1, 0, nullptr, nullptr, 0, layout,
                            nullptr, static_cast<cudaStream_t>(stream));
}

int ave_attn_fwd_varlen(const void *q, const void *k, const void *v, void *o, float *lse, const int *cu_seqlens_q,
                        const int *cu_seqlens_k, int B, int H, int Hkv, int max_Sq, int max_Sk, int total_q,
                        int total_k, int D, int causal, float scale, void *stream) {
    if (!cu_seqlens_q || !cu_seqlens_k) return AVE_ERR_NULL_POINTER;
    int st = validate(q, k, v, o, lse, B, H, Hkv, max_Sq, max_Sk, D, scale);
    if (st >= 0) return st;
    if (total_q <= 0 || total_k <= 0 || total_q >= (1 << 30) || total_k >= (1 << 30)) return AVE_ERR_BAD_SHAPE;
    if (max_Sq > total_q || max_Sk > total_k) return AVE_ERR_BAD_SHAPE;
    st = validate_ptrs_and_scale(q, k, v, o, lse, scale);
    if (st != AVE_OK) return st;
    if ((reinterpret_cast<uintptr_t>(cu_seqlens_q) | reinterpret_cast<uintptr_t>(cu_seqlens_k)) & 3u)
        return AVE_ERR_MISALIGNED;
    st = check_device();
    if (st != AVE_OK) return st;
    const VarlenArgs vl{cu_seqlens_q, cu_seqlens_k, total_q, total_k};
    return launch_attention(q, k, v, o, lse, B, H, Hkv, max_Sq, max_Sk, D, causal, scale, false, 1, 0, nullptr, nullptr, 0,
                            nullptr, &vl, static_cast<cudaStream_t>(stream));
}

size_t ave_attn_host_workspace_bytes(int B, int H, int Hkv, int Sq, int Sk, int D) {
    if (validate(&B, &B, &B, &B, &B, B, H, Hkv, Sq, Sk, D, 1.f) >= 0) return 0;
    auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t qb = up(size_t(B) * H * Sq * D * 2);
    const size_t kb = up(size_t(B) * Hkv * Sk * D * 2);
    const size_t lb = up(size_t(B) * H * Sq * 4);
    return qb /*q*/ + 2 * kb /*k, v*/ + qb /*o*/ + lb /*lse*/;
}

int ave_attn_fwd_host(const void *q_host, const void *k_host, const void *v_host, void *o_host, float *lse_host,
                      int B, int H, int Hkv, int Sq, int Sk, int D, int causal, float scale, void *workspace,
                      size_t workspace_bytes, void *stream) {
    int st = validate(q_host, k_host, v_host, o_host, lse_host, B, H, Hkv, Sq, Sk, D, scale);
    if (st >= 0) return st;
    if (std::isnan(scale) || std::isinf(scale)) return AVE_ERR_BAD_SCALE;
    const size_t need = ave_attn_host_workspace_bytes(B, H, Hkv, Sq, Sk, D);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < need)
        return AVE_ERR_WORKSPACE;
    st = check_device();
    if (st != AVE_OK) return st;

    auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t q_bytes = size_t(B) * H * Sq * D * 2, kv_bytes = size_t(B) * Hkv * Sk * D * 2;
    const size_t lse_bytes = size_t(B) * H * Sq * 4;
    uint8_t *w = static_cast<uint8_t *>(workspace);
    void *dq = w;
    void *dk = w + up(q_bytes);
    void *dv = w + up(q_bytes) + up(kv_bytes);
    void *d_o = w + up(q_bytes) + 2 * up(kv_bytes);
    float *dl = reinterpret_cast<float *>(w + 2 * up(q_bytes) + 2 * up(kv_bytes));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    if ((e = cudaMemcpyAsync(dq, q_host, q_bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dk, k_host, kv_bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dv, v_host, kv_bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    st = ave_attn_fwd(dq, dk, dv, d_o, dl, B, H, Hkv, Sq, Sk, D, causal, scale, stream);
    if (st != AVE_OK) return st;
    if ((e = cudaMemcpyAsync(o_host, d_o, q_bytes, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(lse_host, dl, lse_bytes, cudaMemcpyDeviceToHost, s)) != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    return AVE_OK;
}

size_t ave_attn_splitkv_workspace_bytes(int B, int H, int Sq, int D, int n_splits) {
    if (B <= 0 || H <= 0 || Sq <= 0 || (D != 64 && D != 128) || n_splits < 1 || n_splits > AVE_SPLITKV_MAX_SPLITS)
        return 0;
    const size_t rows = size_t(B) * H * Sq;
    return size_t(n_splits) * rows * (size_t(D) + 1) * sizeof(float);
}

int ave_attn_splitkv_default_splits(int B, int H, int Hkv, int Sq, int Sk, int D) {
    if (B <= 0 || H <= 0 || Hkv <= 0 || Sq <= 0 || Sk <= 0 || H % Hkv != 0 || (D != 64 && D != 128)) return 0;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;  // no device to ask: the count of the part this library is written for
    return ave::splitkv_default_splits(B, H, Hkv, Sq, Sk, sms, AVE_SPLITKV_MAX_SPLITS);
}

int ave_attn_fwd_splitkv(const void *q, const void *k, const void *v, void *o, float *lse, int B, int H, int Hkv,
                         int Sq, int Sk, int D, int causal, float scale, int n_splits, void *workspace,
                         size_t workspace_bytes, void *stream) {
    int st = validate(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, scale);
    if (st >= 0) return st;
    if (D != 64 && D != 128) return AVE_ERR_UNSUPPORTED_D;
    if (n_splits < 1 || n_splits > AVE_SPLITKV_MAX_SPLITS) return AVE_ERR_BAD_SHAPE;
    st = validate_ptrs_and_scale(q, k, v, o, lse, scale);
    if (st != AVE_OK) return st;
    const size_t need = ave_attn_splitkv_workspace_bytes(B, H, Sq, D, n_splits);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) || workspace_bytes < need)
        return AVE_ERR_WORKSPACE;
    st = check_device();
    if (st != AVE_OK) return st;
    const size_t rows = size_t(B) * H * Sq;
    float *o_partial = static_cast<float *>(workspace);
    float *lse_partial = o_partial + size_t(n_splits) * rows * D;
    return run_splitkv(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, causal, scale, n_splits, o_partial, lse_partial,
                       static_cast<cudaStream_t>(stream));
}

int ave_attn_fwd_splitkv_static(const void *q, const void *k, const void *v, void *o, float *lse, int B, int H,
                                int Hkv, int Sq, int Sk, int D, int causal, float scale, int n_splits,
                                void *stream) {
    int st = validate(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, scale);
    if (st >= 0) return st;
    if (D != 64 && D != 128) return AVE_ERR_UNSUPPORTED_D;
    if (n_splits < 1 || n_splits > AVE_SPLITKV_MAX_SPLITS) return AVE_ERR_BAD_SHAPE;
    st = validate_ptrs_and_scale(q, k, v, o, lse, scale);
    if (st != AVE_OK) return st;
    const size_t need = ave_attn_splitkv_workspace_bytes(B, H, Sq, D, n_splits);
    if (need == 0 || need > size_t(AVE_SPLITKV_STATIC_SCRATCH_BYTES)) return AVE_ERR_STATIC_SCRATCH;
    st = check_device();
    if (st != AVE_OK) return st;

    // Device address of the built-in array, looked up once per device with that device current.
    constexpr int kMaxDevices = 64;
    static std::atomic<void *> scratch_of_device[kMaxDevices];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        t_last_cuda_error = int(e != cudaSuccess ? e : cudaErrorInvalidDevice);
        return AVE_ERR_CUDA;
    }
    void *scratch = scratch_of_device[dev].load(std::memory_order_acquire);
    if (!scratch) {
        e = cudaGetSymbolAddress(&scratch, g_splitkv_static_scratch);
        if (e != cudaSuccess || !scratch) {
            t_last_cuda_error = int(e);
            return AVE_ERR_CUDA;
        }
        scratch_of_device[dev].store(scratch, std::memory_order_release);
    }
    const size_t rows = size_t(B) * H * Sq;
    float *o_partial = static_cast<float *>(scratch);
    float *lse_partial = o_partial + size_t(n_splits) * rows * D;
    return run_splitkv(q, k, v, o, lse, B, H, Hkv, Sq, Sk, D, causal, scale, n_splits, o_partial, lse_partial,
                       static_cast<cudaStream_t>(stream));
}

int ave_attn_device_status(unsigned int *raw_word) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    unsigned int word = 0, zero = 0;
    e = cudaMemcpyFromSymbol(&word, ave::g_device_status, sizeof(word));
    if (e == cudaSuccess && word != 0) e = cudaMemcpyToSymbol(ave::g_device_status, &zero, sizeof(zero));
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    if (raw_word) *raw_word = word;
    return word ? AVE_ERR_DEVICE_TIMEOUT : AVE_OK;
}

unsigned long long ave_attn_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char *ave_attn_strerror(int status) {
    switch (status) {
        case AVE_OK: return "ok";
        case AVE_ERR_NULL_POINTER: return "a required pointer is NULL";
        case AVE_ERR_BAD_SHAPE: return "bad shape: sizes must be positive, H a multiple of Hkv, and within limits";
        case AVE_ERR_UNSUPPORTED_D: return "unsupported head dimension (a multiple of 8 up to 256; 64 or 128 for the split-KV calls)";
        case AVE_ERR_MISALIGNED: return "q, k, v, o must be 16-byte aligned and lse 4-byte aligned";
        case AVE_ERR_BAD_SCALE: return "scale is NaN or infinite";
        case AVE_ERR_UNSUPPORTED_DEVICE: return "the current CUDA device is not compute capability 10.x";
        case AVE_ERR_CUDA: return "a CUDA call failed (see ave_attn_last_cuda_error)";
        case AVE_ERR_DEVICE_TIMEOUT: return "a bounded wait inside a kernel gave up";
        case AVE_ERR_WORKSPACE: return "workspace is NULL, misaligned or too small";
        case AVE_ERR_STATIC_SCRATCH:
            return "the problem needs more scratch than the built-in array of ave_attn_fwd_splitkv_static holds";
        case AVE_ERR_KERNEL_IMAGE:
            return "the compiled kernel has fewer registers per thread than its warp roles' register split needs";
        default: return "unknown status";
    }
}

int ave_attn_version(void) { return kVersion; }

int ave_attn_select_kernel(int which) {
    if (which < 0 || which > 2) return AVE_ERR_BAD_SHAPE;
    g_kernel_choice.store(which, std::memory_order_relaxed);
    return AVE_OK;
}

unsigned long long ave_attn_tensor_map_encodes(void) { return g_map_encodes.load(std::memory_order_relaxed); }

int ave_attn_selftest_register_split(int regs_per_thread) {
    return register_split_fits(regs_per_thread) ? AVE_OK : AVE_ERR_KERNEL_IMAGE;
}

int ave_attn_selftest_inject_failures(int what, int count) {
    if (count < 0) return AVE_ERR_BAD_SHAPE;
    if (what == AVE_INJECT_LAUNCH_FAILURE) g_inject_launch_failures.store(count, std::memory_order_relaxed);
    else if (what == AVE_INJECT_ENCODE_FAILURE) g_inject_encode_failures.store(count, std::memory_order_relaxed);
    else return AVE_ERR_BAD_SHAPE;
    return AVE_OK;
}

int ave_attn_selftest_wait_timeout(int limit_cycles_log2, void *stream) {
    if (limit_cycles_log2 < 10 || limit_cycles_log2 > 26) return AVE_ERR_BAD_SHAPE;  // 1 us .. a few tens of ms
    int st = check_device();
    if (st != AVE_OK) return st;
    wait_timeout_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(1ll << limit_cycles_log2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        t_last_cuda_error = int(e);
        return AVE_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return AVE_OK;
}

#ifdef AVE_TRACE
// Trace builds only (not part of the public interface): copies the role
// timeline of the traced CTA, TRACE_ROLES x TRACE_ITERS x TRACE_SLOTS clocks.
int ave_attn_trace_read(long long *out) {
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(out, ave::g_trace, sizeof(ave::g_trace));
    return e == cudaSuccess ? AVE_OK : AVE_ERR_CUDA;
}
// The life span of the last launch's CTAs: n_ctas x {first ns, last ns, tiles processed}.
int ave_attn_trace_read_spans(unsigned long long *out, int n_ctas) {
    if (n_ctas > ave::TRACE_CTAS) n_ctas = ave::TRACE_CTAS;
    cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(out, ave::g_cta_span, size_t(n_ctas) * 3 * sizeof(unsigned long long));
    return e == cudaSuccess ? AVE_OK : AVE_ERR_CUDA;
}
int ave_attn_trace_clear_spans() {
    void *ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, ave::g_cta_span);
    if (e == cudaSuccess) e = cudaMemset(ptr, 0, sizeof(ave::g_cta_span));
    return e == cudaSuccess ? AVE_OK : AVE_ERR_CUDA;
}
#endif

static int gemm_validate(const void *a, const void *b, const void *c, int M, int N, int K) {
    if (!a || !b || !c) return AVE_ERR_NULL_POINTER;
    if (M <= 0 || N <= 0 || K <= 0) return AVE_ERR_BAD_SHAPE;
    const long long lim = 1ll << 39;  // elements: a tensor map holds byte strides below 2^40
    if ((long long)M * K >= lim || (long long)N * K >= lim || (long long)M * N >= lim) return AVE_ERR_BAD_SHAPE;
    if ((long long)((M + 127) / 128) * ((N + 127) / 128) >= (1ll << 31)) return AVE_ERR_BAD_SHAPE;
    if ((K & 7) || (N & 7)) return AVE_ERR_MISALIGNED;
    if ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & 15u)
        return AVE_ERR_MISALIGNED;
    return AVE_OK;
}

int ave_gemm_bf16_tn(const void *a, const void *b, void *c, int M, int N, int K, void *stream) {
    int st = gemm_validate(a, b, c, M, N, K);
    if (st != AVE_OK) return st;
    st = check_device();
    if (st != AVE_OK) return st;
    return launch_gemm<false>(a, b, c, M, N, K, static_cast<cudaStream_t>(stream));
}

int ave_gemm_bf16_nn(const void *a, const void *b, void *c, int M, int N, int K, void *stream) {
    int st = gemm_validate(a, b, c, M, N, K);
    if (st != AVE_OK) return st;
    st = check_device();
    if (st != AVE_OK) return st;
    return launch_gemm<true>(a, b, c, M, N, K, static_cast<cudaStream_t>(stream));
}

int ave_attn_last_cuda_error(void) { return t_last_cuda_error; }

}  // extern "C"
