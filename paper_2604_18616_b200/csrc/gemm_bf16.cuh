// Dense bf16 GEMM for sm_100a: C[M, N] = A[M, K] * B[N, K]^T (or A[M, K] * B[K, N]),
// fp32 accumulation in TMEM, bf16 result.  (The paper's first evaluated kernel family, Section 9:
// square bf16 matrices with normally distributed entries.)
//
// Three kernels.  Large products: CTA pairs with tiles of 256 x up to 256 (below).  Products of few tiles: one CTA, or a
// cluster that shares K, per 128 x 128 tile.  In between, above all with at most 128 rows, of which a pair would use half:
// one CTA per 128 x 256 tile.  In all of them the K dimension is streamed in slices of 64
// through a ring of shared-memory stages filled by TMA, and one thread issues the
// tcgen05 MMAs into TMEM; pairs and 128 x 256 tiles are persistent and have two accumulators, so that the
// epilogue of a tile (TMEM -> registers -> bf16 -> shared -> TMA store)
// overlaps the main loop of the next one.
//
//   warp 0      producer: TMA loads of the A and B slices
//   warp 1      MMA issuer
//   warp 2      TMEM allocation / release
//   warp 3      -
//   warps 4..7  epilogue (thread = accumulator row = TMEM lane)
//
// Rows and columns outside the matrices are zero-filled by the loads and
// clipped by the stores, so M, N and K need not be multiples of the tile.
#pragma once

#include <cuda_bf16.h>

#include "attn_common.cuh"
#include "gemm_choice.cuh"

namespace ave {

struct GemmCfg {
    static constexpr int kThreads = 256;
    static constexpr int kTileM = 128, kTileN = 128, kSliceK = 64;
    static constexpr int kStages = 5;
    static constexpr int kABytes = kTileM * kSliceK * 2;          // 16 KB
    static constexpr int kBBytes = kTileN * kSliceK * 2;          // 16 KB
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kOutBoxRows = 32;                        // each epilogue warp stores its own 32 rows
    static constexpr int kMaxSplits = kGemmMaxSplits;             // CTAs of a cluster that share a tile's K
    static constexpr int kRecvBytes = kTileM * kTileN * 4 / kMaxSplits * (kMaxSplits - 1);  // the others' partial sums
    static constexpr int kSmemBytes = kStages * kStageBytes + kRecvBytes + 1024;
    static constexpr uint32_t kTmemCols = kTileN;
};

struct GemmParams {
    int M, N, K;
    int tiles_m, tiles_n;  // output tiles along M and N
    int group_m;           // tiles along M walked together before moving along N (L2 reuse of the B tiles)
    int tile_n;            // (CTA pairs) columns of a tile: 64, 128, 192 or 256
    int splits;            // (one CTA per tile and share of K) CTAs of a cluster
    void *c;               // the result, for stores that do not go through its tensor map
};

// Output tile number `id` -> (block row, block column): groups of `group_m` block rows, column-major inside a
// group, so that CTAs working at the same time share a few A row blocks and neighbouring B column blocks.
__device__ __forceinline__ void gemm_tile_coords(int id, const GemmParams &p, int &bm, int &bn) {
    const int per_group = p.group_m * p.tiles_n;
    const int grp = id / per_group;
    const int rem = id - grp * per_group;
    const int m0 = grp * p.group_m;
    const int gm = min(p.group_m, p.tiles_m - m0);
    bn = rem / gm;
    bm = m0 + (rem - bn * gm);
}

// 64 columns of 32 accumulator rows (one per lane) as bf16 into a staging buffer of 32 rows x 128 bytes, in the
// 128-byte-swizzled layout that the TMA store expects.
__device__ __forceinline__ void gemm_stage_64_columns(uint32_t buf, int lane, const uint32_t (&v)[2][32]) {
#pragma unroll
    for (int e = 0; e < 64; e += 8) {
        const uint32_t *src = &v[e >> 5][e & 31];
        const uint32_t addr = buf + lane * 128 + (((e >> 3) ^ (lane & 7)) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr),
                     "r"(pack_bf16x2(__uint_as_float(src[0]), __uint_as_float(src[1]))),
                     "r"(pack_bf16x2(__uint_as_float(src[2]), __uint_as_float(src[3]))),
                     "r"(pack_bf16x2(__uint_as_float(src[4]), __uint_as_float(src[5]))),
                     "r"(pack_bf16x2(__uint_as_float(src[6]), __uint_as_float(src[7]))) : "memory");
    }
}

// B_NMAJOR = false: B is [N, K] with K contiguous (C = A * B^T).  B_NMAJOR = true: B is [K, N] with N
// contiguous (C = A * B); its slice then lands in shared memory as 64-column boxes of 64 K-rows each and is
// read through an MN-major descriptor, so neither form needs a transposition.
//
// A cluster of S = 1, 2, 4 or 8 CTAs computes one tile, each over its share of K; with S > 1 every CTA then sends the others
// their 128 / S columns of its fp32 sums through distributed shared memory and adds up, in the order of the shares, and
// stores its own columns.  A product of few tiles leaves most SMs idle, and a tile's time is its number of slices times the
// 32 KB a slice brings in.  200 x 512 x 8192 (8 tiles): 37.8 us with S = 1, 10.5 us with S = 8;
// 128 x 4096 x 4096 (32 tiles): 21.4 / 10.5 us with S = 4; 1939 x 440 x 2416 (64 tiles): 16.1 / 12.1 us with S = 2.
template <bool B_NMAJOR>
__global__ void __launch_bounds__(256, 1)
gemm_bf16_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                 const __grid_constant__ CUtensorMap tm_c, const GemmParams p) {
    using Cfg = GemmCfg;
    constexpr int NS = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[NS], bar_empty[NS], bar_acc_full, bar_drain;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, missing_sums;  // the second: another CTA of the cluster has no sums to send

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const uint32_t sRing = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sRecv = sRing + NS * Cfg::kStageBytes;

    if (tid == 0) {
        missing_sums = 0;
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        mbar_init(smem_u32(&bar_acc_full), 1);
        mbar_init(smem_u32(&bar_drain), 1);
        fence_mbar_init();
        tma_prefetch_desc(&tm_a);
        tma_prefetch_desc(&tm_b);
    }
    if (warp == 2) {
        tmem_alloc(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
        tmem_relinquish();
    }
    // what precedes overlaps the end of the kernel before this one in the stream
    grid_dependency_wait();
    grid_dependency_launch();
    if (tid == 0) abort_flag = (*reinterpret_cast<volatile unsigned int *>(&g_device_status) != 0) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    const bool poisoned = abort_flag != 0;

    const int S = p.splits;
    const int rank = S > 1 ? int(cluster_rank()) : 0;
    if (S > 1) cluster_arrive();  // waited for before anything is written to another CTA: it has started
    int bm, bn;
    gemm_tile_coords(blockIdx.x / S, p, bm, bn);
    const int all_slices = (p.K + Cfg::kSliceK - 1) / Cfg::kSliceK;
    const int slice0 = all_slices * rank / S, n_slices = all_slices * (rank + 1) / S - slice0;  // (S <= all_slices)

    if (poisoned) {
        // nothing
    } else if (warp == 0) {
        // =============================== producer ===============================
        if (elect_one()) {
            bool ok = true;
            int i = 0;  // slices loaded so far
            for (; i < n_slices; ++i) {
                const int slot = i % NS;
                if (i >= NS) ok = mbar_wait_bounded(smem_u32(&bar_empty[slot]), (i / NS - 1) & 1, &abort_flag, STATUS_TIMEOUT_SLOT);
                if (!ok) break;
                const int k = (slice0 + i) * Cfg::kSliceK;
                const uint32_t bar = smem_u32(&bar_full[slot]);
                const uint32_t dst = sRing + slot * Cfg::kStageBytes;
                mbar_arrive_expect_tx(bar, Cfg::kStageBytes);
                tma_load_4d(dst, &tm_a, bar, k, bm * Cfg::kTileM, 0, 0);
                if (!B_NMAJOR) {
                    tma_load_4d(dst + Cfg::kABytes, &tm_b, bar, k, bn * Cfg::kTileN, 0, 0);
                } else {
                    for (int x = 0; x < Cfg::kTileN / 64; ++x)  // boxes of 64 columns of B x 64 rows of K
                        tma_load_4d(dst + Cfg::kABytes + x * (Cfg::kSliceK * 128), &tm_b, bar, bn * Cfg::kTileN + x * 64, k, 0, 0);
                }
            }
            if (!ok) {
                // abandoned: give the loads still in flight a bounded chance to land
                for (int it = max(0, i - NS); it < i; ++it)
                    for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_full[it % NS]), (it / NS) & 1); ++w) {}
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // =============================== MMA issuer ===============================
        if (elect_one()) {
            constexpr uint32_t idesc = make_idesc_bf16(Cfg::kTileM, Cfg::kTileN, B_NMAJOR ? 1 : 0);
            constexpr uint64_t desc_kmajor = make_sdesc_sw128(16, 1024);
            constexpr uint32_t hi = uint32_t(desc_kmajor >> 32), lo = uint32_t(desc_kmajor);
            // N-contiguous B: 64-wide column groups are one box (64 K-rows x 128 B) apart, 8 K-rows 1024 B apart;
            // 16 K-rows further is 16 x 128 B
            constexpr uint64_t desc_nmajor = make_sdesc_sw128(Cfg::kSliceK * 128, 1024);
            constexpr uint32_t hi_b = B_NMAJOR ? uint32_t(desc_nmajor >> 32) : hi;
            constexpr uint32_t lo_b = B_NMAJOR ? uint32_t(desc_nmajor) : lo;
            constexpr uint32_t b_kstep = B_NMAJOR ? ((16 * 128) >> 4) : (32 >> 4);
            bool ok = true;
            for (int i = 0; i < n_slices; ++i) {
                const int slot = i % NS;
                ok = mbar_wait_bounded(smem_u32(&bar_full[slot]), (i / NS) & 1, &abort_flag, STATUS_TIMEOUT_LOAD);
                if (!ok) break;
                tc_fence_after();
                // (in a cluster the CTA's rank stands in the address bits above the window, where a descriptor has other fields)
                const uint32_t stage = (sRing + slot * Cfg::kStageBytes) & 0x3ffffu;
                const uint32_t a_lo = lo | (stage >> 4);
                const uint32_t b_lo = lo_b | ((stage + Cfg::kABytes) >> 4);
#pragma unroll
                for (int kk = 0; kk < Cfg::kSliceK / 16; ++kk)
                    umma_ss_words(tmem, a_lo + ((kk * 32) >> 4), hi, b_lo + kk * b_kstep, hi_b, idesc, (i > 0 || kk > 0));
                umma_commit(smem_u32(&bar_empty[slot]));
            }
            if (ok) {
                umma_commit(smem_u32(&bar_acc_full));
            } else {  // abandoned: let the MMAs already issued finish before TMEM is released
                umma_commit(smem_u32(&bar_drain));
                for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain), 0); ++w) {}
            }
        }
        __syncwarp();
    }
    if (warp < 4) {
        if (S > 1) {
            cluster_wait();
            cluster_sync();
        }
    } else {
        // =============================== epilogue ===============================
        const int wq = warp & 3;  // TMEM lane quadrant of this warp
        const int r = wq * 32 + lane;
        const uint32_t t_acc = tmem + (uint32_t(wq * 32) << 16);
        const int row0 = bm * Cfg::kTileM + wq * 32;
        bool ok = !poisoned;
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_acc_full), 0, &abort_flag, STATUS_TIMEOUT_MMA));
        tc_fence_after();
        if (S == 1) {
            const uint32_t sC = sRing + wq * (2 * Cfg::kOutBoxRows * 128);  // (the ring's slices have all been used)
            for (int c = 0; c < 2 && ok; ++c) {  // 64 columns at a time
                uint32_t v[2][32];
                tmem_ld_x32(t_acc + c * 64, v[0]);
                tmem_ld_x32(t_acc + c * 64 + 32, v[1]);
                tmem_wait_ld();
                tmem_pin_x32(v[0]);
                tmem_pin_x32(v[1]);
                const uint32_t buf = sC + c * (Cfg::kOutBoxRows * 128);
                gemm_stage_64_columns(buf, lane, v);
                fence_proxy_async_smem();
                __syncwarp();
                const int col0 = bn * Cfg::kTileN + c * 64;
                if (lane == 0 && row0 < p.M && col0 < p.N) {
                    tma_store_4d(&tm_c, buf, col0, row0, 0, 0);
                    tma_store_commit();
                }
            }
            if (lane == 0) tma_store_wait_all();
        } else {
            const int cols = Cfg::kTileN / S;  // 16, 32 or 64: the columns each CTA finishes
            cluster_wait();
            // Partial sums arrive as [sender][4 columns][row] float4s, so that a warp's 32 rows are 512 contiguous bytes.
            for (int q = 0; q < S && ok; ++q) {
                if (q == rank) continue;
                const uint32_t dst = map_to_cta(sRecv, q) + (((rank < q ? rank : rank - 1) * (cols / 4)) * 128 + r) * 16;
                for (int c = 0; c < cols; c += 16) {
                    uint32_t v[16];
                    tmem_ld_x16(t_acc + q * cols + c, v);
                    tmem_wait_ld();
                    tmem_pin_x16(v);
#pragma unroll
                    for (int e = 0; e < 16; e += 4)
                        st_cluster_v4(dst + ((c + e) / 4) * (128 * 16), v[e], v[e + 1], v[e + 2], v[e + 3]);
                }
            }
            // A CTA that found the status word set, or gave up a wait, has sent nothing: the others may have read the word before
            // it was set, and must not add up, and store, what was never written here.
            if (!ok && lane < S && lane != rank) st_cluster_s32(map_to_cta(smem_u32(&missing_sums), lane), 1);
            __syncwarp();
            cluster_sync();
            ok = ok && *reinterpret_cast<volatile int *>(&missing_sums) == 0;
            const int row = row0 + lane;
            for (int c = 0; c < cols && ok; c += 16) {
                uint32_t own[16];
                tmem_ld_x16(t_acc + rank * cols + c, own);
                tmem_wait_ld();
                tmem_pin_x16(own);
                float sum[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) sum[e] = 0.f;
                for (int q = 0; q < S; ++q) {  // in the order of K, whichever CTA adds up
                    if (q == rank) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[e] += __uint_as_float(own[e]);
                    } else {
                        const uint32_t src = sRecv + (((q < rank ? q : q - 1) * (cols / 4) + c / 4) * 128 + r) * 16;
#pragma unroll
                        for (int e = 0; e < 16; e += 4) {
                            float4 x;
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
                                         : "r"(src + (e / 4) * (128 * 16)) : "memory");
                            sum[e] += x.x; sum[e + 1] += x.y; sum[e + 2] += x.z; sum[e + 3] += x.w;
                        }
                    }
                }
                const int col = bn * Cfg::kTileN + rank * cols + c;
                __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(p.c) + size_t(row) * p.N + col;
#pragma unroll
                for (int e = 0; e < 16; e += 8) {
                    if (row < p.M && col + e < p.N)  // (N is a multiple of 8)
                        *reinterpret_cast<uint4 *>(out + e) = make_uint4(pack_bf16x2(sum[e], sum[e + 1]), pack_bf16x2(sum[e + 2], sum[e + 3]),
                                                                         pack_bf16x2(sum[e + 4], sum[e + 5]), pack_bf16x2(sum[e + 6], sum[e + 7]));
                }
            }
        }
    }

    // ---- common exit: every thread arrives, then TMEM is released
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, Cfg::kTmemCols);
}

// ------------------------------------------------------------------ 128 x 256 tiles, one CTA each
//
// What bounds it is the way from L2 into shared memory, 48 KB per slice against 512 clk of MMAs (see the CTA pairs); its
// place is where pairs would multiply rows that do not exist, or leave a last wave nearly empty (pairs / this kernel:
// 128 x 19000 x 2048 28.0 / 21.2 us, 128 x 28672 x 4096 60 / 48 us, 1 x 65536 x 512 25.9 / 17.1 us,
// 600 x 14336 x 4096 67.8 / 60.5 us).
struct GemmWideCfg {
    static constexpr int kThreads = 256;
    static constexpr int kTileM = 128, kTileN = 256, kSliceK = 64;
    static constexpr int kStages = 4;
    static constexpr int kABytes = kTileM * kSliceK * 2;          // 16 KB
    static constexpr int kBBytes = kTileN * kSliceK * 2;          // 32 KB
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kOutBoxRows = 32;
    static constexpr int kStageCBytes = 4 * kOutBoxRows * 128;    // 32 rows x 64 columns per epilogue warp
    static constexpr int kSmemBytes = kStages * kStageBytes + kStageCBytes + 1024;
    static constexpr uint32_t kTmemCols = 2 * kTileN;             // two accumulators
};

template <bool B_NMAJOR>
__global__ void __launch_bounds__(256, 1)
gemm_bf16_wide_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                      const __grid_constant__ CUtensorMap tm_c, const GemmParams p) {
    using Cfg = GemmWideCfg;
    constexpr int NS = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[NS], bar_empty[NS], bar_acc_full[2], bar_acc_empty[2], bar_drain;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const uint32_t sRing = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sStage = sRing + NS * Cfg::kStageBytes;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&bar_acc_full[a]), 1);
            mbar_init(smem_u32(&bar_acc_empty[a]), 4);  // one arrival per epilogue warp
        }
        mbar_init(smem_u32(&bar_drain), 1);
        fence_mbar_init();
        tma_prefetch_desc(&tm_a);
        tma_prefetch_desc(&tm_b);
    }
    if (warp == 2) {
        tmem_alloc(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
        tmem_relinquish();
    }
    // what precedes overlaps the end of the kernel before this one in the stream
    grid_dependency_wait();
    grid_dependency_launch();
    if (tid == 0) abort_flag = (*reinterpret_cast<volatile unsigned int *>(&g_device_status) != 0) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    const bool poisoned = abort_flag != 0;

    const int n_tiles = p.tiles_m * p.tiles_n;
    const int n_slices = (p.K + Cfg::kSliceK - 1) / Cfg::kSliceK;

    if (poisoned) {
        // nothing: fall through to the common exit
    } else if (warp == 0) {
        // =============================== producer ===============================
        if (elect_one()) {
            bool ok = true;
            int ring = 0;  // slices loaded so far
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
                int bm, bn;
                gemm_tile_coords(tile, p, bm, bn);
                for (int ks = 0; ks < n_slices; ++ks, ++ring) {
                    const int slot = ring % NS, round = ring / NS;
                    if (round > 0) ok = mbar_wait_bounded(smem_u32(&bar_empty[slot]), (round - 1) & 1, &abort_flag, STATUS_TIMEOUT_SLOT);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&bar_full[slot]);
                    const uint32_t dst = sRing + slot * Cfg::kStageBytes;
                    mbar_arrive_expect_tx(bar, Cfg::kStageBytes);
                    tma_load_4d(dst, &tm_a, bar, ks * Cfg::kSliceK, bm * Cfg::kTileM, 0, 0);
                    if (!B_NMAJOR) {
                        tma_load_4d(dst + Cfg::kABytes, &tm_b, bar, ks * Cfg::kSliceK, bn * Cfg::kTileN, 0, 0);
                    } else {
                        for (int x = 0; x < Cfg::kTileN / 64; ++x)  // boxes of 64 columns of B x 64 rows of K
                            tma_load_4d(dst + Cfg::kABytes + x * (Cfg::kSliceK * 128), &tm_b, bar, bn * Cfg::kTileN + x * 64,
                                        ks * Cfg::kSliceK, 0, 0);
                    }
                }
            }
            if (!ok) {
                // abandoned: give the loads still in flight a bounded chance to land
                for (int it = max(0, ring - NS); it < ring; ++it)
                    for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_full[it % NS]), (it / NS) & 1); ++w) {}
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // =============================== MMA issuer ===============================
        if (elect_one()) {
            constexpr uint32_t idesc = make_idesc_bf16(Cfg::kTileM, Cfg::kTileN, B_NMAJOR ? 1 : 0);
            constexpr uint64_t desc_kmajor = make_sdesc_sw128(16, 1024);
            constexpr uint32_t hi = uint32_t(desc_kmajor >> 32), lo = uint32_t(desc_kmajor);
            constexpr uint64_t desc_nmajor = make_sdesc_sw128(Cfg::kSliceK * 128, 1024);
            constexpr uint32_t hi_b = B_NMAJOR ? uint32_t(desc_nmajor >> 32) : hi;
            constexpr uint32_t lo_b = B_NMAJOR ? uint32_t(desc_nmajor) : lo;
            constexpr uint32_t b_kstep = B_NMAJOR ? ((16 * 128) >> 4) : (32 >> 4);
            bool ok = true;
            int ring = 0;
            int n_done = 0;  // tiles issued so far
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++n_done) {
                const int acc = n_done & 1;
                if (n_done >= 2) {  // the epilogue must have read this accumulator's previous tile out of TMEM
                    ok = mbar_wait_bounded(smem_u32(&bar_acc_empty[acc]), ((n_done >> 1) - 1) & 1, &abort_flag, STATUS_TIMEOUT_SOFTMAX);
                    if (!ok) break;
                    tc_fence_after();
                }
                const uint32_t d_tmem = tmem + acc * Cfg::kTileN;
                for (int ks = 0; ks < n_slices; ++ks, ++ring) {
                    const int slot = ring % NS;
                    ok = mbar_wait_bounded(smem_u32(&bar_full[slot]), (ring / NS) & 1, &abort_flag, STATUS_TIMEOUT_LOAD);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_lo = lo | ((sRing + slot * Cfg::kStageBytes) >> 4);
                    const uint32_t b_lo = lo_b | ((sRing + slot * Cfg::kStageBytes + Cfg::kABytes) >> 4);
#pragma unroll
                    for (int kk = 0; kk < Cfg::kSliceK / 16; ++kk)
                        umma_ss_words(d_tmem, a_lo + ((kk * 32) >> 4), hi, b_lo + kk * b_kstep, hi_b, idesc, (ks > 0 || kk > 0));
                    umma_commit(smem_u32(&bar_empty[slot]));
                    if (ks == n_slices - 1) umma_commit(smem_u32(&bar_acc_full[acc]));
                }
            }
            if (!ok) {  // abandoned: let the MMAs already issued finish before TMEM is released
                umma_commit(smem_u32(&bar_drain));
                for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain), 0); ++w) {}
            }
        }
        __syncwarp();
    } else if (warp >= 4) {
        // =============================== epilogue ===============================
        const int wq = warp & 3;  // TMEM lane quadrant of this warp
        const uint32_t lane_sel = uint32_t(wq * 32) << 16;
        const uint32_t sC = sStage + wq * (Cfg::kOutBoxRows * 128);  // this warp's 32 staging rows
        bool ok = true;
        bool store_pending = false;  // (lane 0) a TMA store may still be reading this warp's staging rows
        int n_done = 0;
        for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++n_done) {
            int bm, bn;
            gemm_tile_coords(tile, p, bm, bn);
            const int acc = n_done & 1;
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_acc_full[acc]), (n_done >> 1) & 1, &abort_flag, STATUS_TIMEOUT_MMA));
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_acc = tmem + acc * Cfg::kTileN + lane_sel;
            const int row0 = bm * Cfg::kTileM + wq * 32;
#pragma unroll 1
            for (int c = 0; c < Cfg::kTileN / 64; ++c) {  // 64 columns at a time
                uint32_t v[2][32];
                tmem_ld_x32(t_acc + c * 64, v[0]);
                tmem_ld_x32(t_acc + c * 64 + 32, v[1]);
                tmem_wait_ld();
                tmem_pin_x32(v[0]);
                tmem_pin_x32(v[1]);
                if (c == Cfg::kTileN / 64 - 1) {  // the accumulator is in registers: the MMAs may reuse it
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[acc]));
                }
                // this warp's previous TMA store must have finished reading the staging rows
                if (lane == 0 && store_pending) tma_store_wait_read();
                __syncwarp();
                gemm_stage_64_columns(sC, lane, v);
                fence_proxy_async_smem();
                __syncwarp();
                const int col0 = bn * Cfg::kTileN + c * 64;
                if (lane == 0 && row0 < p.M && col0 < p.N) {
                    tma_store_4d(&tm_c, sC, col0, row0, 0, 0);
                    tma_store_commit();
                    store_pending = true;
                }
            }
        }
        if (lane == 0 && store_pending) tma_store_wait_all();
    }

    // ---- common exit: every thread arrives, then TMEM is released
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, Cfg::kTmemCols);
}

// ------------------------------------------------------------------ CTA pairs
//
// The same product with two CTAs (the two SMs of a cluster) per output tile of 256 rows and up to 256 columns: each holds 128 of the
// tile's rows of A, half of its columns of B and the accumulators of its rows; the even CTA's thread issues
// M256 x N256 x K16 MMAs (cta_group::2) that read both CTAs' shared memory.  What bounds a one-CTA kernel here is the
// way from L2 into shared memory, about 54 B/clk per SM (measured with all SMs loading): a 128 x 256 tile
// takes 48 KB per slice of 64 for 512 clk of MMAs, 96 B/clk, a pair's CTA 32 KB.
struct GemmPairCfg {
    static constexpr int kThreads = 256;
    static constexpr int kTileM = 256, kMaxTileN = 256, kSliceK = 64;  // the launch chooses the tile's width
    static constexpr int kStages = 6;
    static constexpr int kABytes = kTileM / 2 * kSliceK * 2;      // 16 KB: this CTA's rows
    static constexpr int kBBytes = kMaxTileN / 2 * kSliceK * 2;   // up to 16 KB: this CTA's columns
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kOutBoxRows = 32;
    static constexpr int kStageCBytes = 4 * kOutBoxRows * 128;
    static constexpr int kSmemBytes = kStages * kStageBytes + kStageCBytes + 1024;
    static constexpr uint32_t kTmemCols = 2 * kMaxTileN;          // two accumulators
};

// Warp roles as above, in both CTAs, except that only the even CTA's MMA warp issues.  Barriers: "full" counts both
// CTAs' bytes on the even CTA's copy; "empty" and "accumulator full" are signalled in both CTAs by the MMAs' commits;
// "accumulator empty" collects both CTAs' epilogue warps on the even CTA's copy.
template <bool B_NMAJOR>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(256, 1)
gemm_bf16_pair_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                      const __grid_constant__ CUtensorMap tm_c, const GemmParams p) {
    using Cfg = GemmPairCfg;
    constexpr int NS = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[NS], bar_empty[NS], bar_acc_full[2], bar_acc_empty[2], bar_drain;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, poison_flag, drain_flag;  // the last: (odd CTA) the even one's MMA issuer gave up

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const uint32_t rank = cluster_rank();
    const uint32_t sRing = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sStage = sRing + NS * Cfg::kStageBytes;

    if (tid == 0) {
        abort_flag = drain_flag = 0;
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&bar_acc_full[a]), 1);
            mbar_init(smem_u32(&bar_acc_empty[a]), 8);  // one arrival per epilogue warp of both CTAs
        }
        mbar_init(smem_u32(&bar_drain), 1);
        fence_mbar_init();
        tma_prefetch_desc(&tm_a);
        tma_prefetch_desc(&tm_b);
    }
    if (warp == 2) {
        tmem_alloc_pair(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
        tmem_relinquish_pair();
    }
    grid_dependency_wait();
    grid_dependency_launch();
    if (tid == 0) poison_flag = (*reinterpret_cast<volatile unsigned int *>(&g_device_status) != 0) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    // both CTAs work or neither does
    const uint32_t pf = smem_u32(&poison_flag);
    const bool poisoned = (ld_cluster_s32(map_to_cta(pf, 0)) | ld_cluster_s32(map_to_cta(pf, 1))) != 0;

    const int n_tiles = p.tiles_m * p.tiles_n;
    const int n_slices = (p.K + Cfg::kSliceK - 1) / Cfg::kSliceK;
    const int half_n = p.tile_n / 2;                            // columns of B in each CTA
    const int b_bytes = (B_NMAJOR ? (half_n + 63) / 64 * 64 : half_n) * (Cfg::kSliceK * 2);
    const int first = blockIdx.x >> 1, stride = gridDim.x >> 1;  // this pair's tiles

    if (poisoned) {
        // nothing: fall through to the common exit
    } else if (warp == 0) {
        // =============================== producer ===============================
        if (elect_one()) {
            bool ok = true;
            int ring = 0;  // slices loaded so far
            for (int tile = first; tile < n_tiles && ok; tile += stride) {
                int bm, bn;
                gemm_tile_coords(tile, p, bm, bn);
                const int row = bm * Cfg::kTileM + int(rank) * 128, col = bn * p.tile_n + int(rank) * half_n;
                for (int ks = 0; ks < n_slices && ok; ++ks, ++ring) {
                    const int slot = ring % NS, round = ring / NS;
                    if (round > 0) {
                        ok = mbar_wait_bounded(smem_u32(&bar_empty[slot]), (round - 1) & 1, &abort_flag, STATUS_TIMEOUT_SLOT);
                        if (!ok) break;
                    }
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&bar_full[slot]), 2 * (Cfg::kABytes + b_bytes));
                    const uint32_t bar = map_to_cta(smem_u32(&bar_full[slot]), 0);
                    const uint32_t dst = sRing + slot * Cfg::kStageBytes;
                    tma_load_4d_pair(dst, &tm_a, bar, ks * Cfg::kSliceK, row, 0, 0);
                    if (!B_NMAJOR) {
                        tma_load_4d_pair(dst + Cfg::kABytes, &tm_b, bar, ks * Cfg::kSliceK, col, 0, 0);
                    } else {
                        for (int x = 0; x * 64 < half_n; ++x)  // boxes of 64 columns of B x 64 rows of K
                            tma_load_4d_pair(dst + Cfg::kABytes + x * (Cfg::kSliceK * 128), &tm_b, bar, col + x * 64,
                                             ks * Cfg::kSliceK, 0, 0);
                    }
                }
            }
            if (!ok) {
                // abandoned: the loads still in flight are counted on the even CTA's barriers only; give them time to land
                const long long t0 = clock64();
                while (clock64() - t0 < (1ll << 20)) __nanosleep(1000);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // =============================== MMA issuer ===============================
        if (rank == 0 && elect_one()) {
            const uint32_t idesc = make_idesc_bf16(Cfg::kTileM, p.tile_n, B_NMAJOR ? 1 : 0);
            constexpr uint64_t desc_kmajor = make_sdesc_sw128(16, 1024);
            constexpr uint32_t hi = uint32_t(desc_kmajor >> 32), lo = uint32_t(desc_kmajor);
            constexpr uint64_t desc_nmajor = make_sdesc_sw128(Cfg::kSliceK * 128, 1024);
            constexpr uint32_t hi_b = B_NMAJOR ? uint32_t(desc_nmajor >> 32) : hi;
            constexpr uint32_t lo_b = B_NMAJOR ? uint32_t(desc_nmajor) : lo;
            constexpr uint32_t b_kstep = B_NMAJOR ? ((16 * 128) >> 4) : (32 >> 4);
            bool ok = true;
            int ring = 0;
            int n_done = 0;  // tiles issued so far
            for (int tile = first; tile < n_tiles && ok; tile += stride, ++n_done) {
                const int acc = n_done & 1;
                if (n_done >= 2) {  // both epilogues must have read this accumulator's previous tile out of TMEM
                    ok = mbar_wait_bounded(smem_u32(&bar_acc_empty[acc]), ((n_done >> 1) - 1) & 1, &abort_flag, STATUS_TIMEOUT_SOFTMAX);
                    if (!ok) break;
                    tc_fence_after();
                }
                const uint32_t d_tmem = tmem + acc * Cfg::kMaxTileN;
                for (int ks = 0; ks < n_slices; ++ks, ++ring) {
                    const int slot = ring % NS;
                    ok = mbar_poll_bounded(smem_u32(&bar_full[slot]), (ring / NS) & 1, &abort_flag, STATUS_TIMEOUT_LOAD);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_lo = lo | ((sRing + slot * Cfg::kStageBytes) >> 4);
                    const uint32_t b_lo = lo_b | ((sRing + slot * Cfg::kStageBytes + Cfg::kABytes) >> 4);
#pragma unroll
                    for (int kk = 0; kk < Cfg::kSliceK / 16; ++kk)
                        umma_ss_pair_words(d_tmem, a_lo + ((kk * 32) >> 4), hi, b_lo + kk * b_kstep, hi_b, idesc, (ks > 0 || kk > 0));
                    umma_commit_pair(smem_u32(&bar_empty[slot]));
                    if (ks == n_slices - 1) umma_commit_pair(smem_u32(&bar_acc_full[acc]));
                }
            }
            if (!ok) {  // abandoned: let the MMAs already issued finish before TMEM is released
                umma_commit_pair(smem_u32(&bar_drain));
                st_cluster_s32(map_to_cta(smem_u32(&drain_flag), 1), 1);  // it arrives there too: the odd CTA has to stay for it
                for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain), 0); ++w) {}
            }
        }
        __syncwarp();
    } else if (warp >= 4) {
        // =============================== epilogue ===============================
        const int wq = warp & 3;  // TMEM lane quadrant of this warp
        const uint32_t lane_sel = uint32_t(wq * 32) << 16;
        const uint32_t sC = sStage + wq * (Cfg::kOutBoxRows * 128);  // this warp's 32 staging rows
        bool ok = true;
        bool store_pending = false;  // (lane 0) a TMA store may still be reading this warp's staging rows
        int n_done = 0;
        for (int tile = first; tile < n_tiles && ok; tile += stride, ++n_done) {
            int bm, bn;
            gemm_tile_coords(tile, p, bm, bn);
            const int acc = n_done & 1;
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&bar_acc_full[acc]), (n_done >> 1) & 1, &abort_flag, STATUS_TIMEOUT_MMA));
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_acc = tmem + acc * Cfg::kMaxTileN + lane_sel;
            const int row0 = bm * Cfg::kTileM + int(rank) * 128 + wq * 32;
#pragma unroll 1
            for (int c = 0; c < p.tile_n / 64; ++c) {  // 64 columns at a time
                uint32_t v[2][32];
                tmem_ld_x32(t_acc + c * 64, v[0]);
                tmem_ld_x32(t_acc + c * 64 + 32, v[1]);
                tmem_wait_ld();
                tmem_pin_x32(v[0]);
                tmem_pin_x32(v[1]);
                if (c == p.tile_n / 64 - 1) {  // the accumulator is in registers: the MMAs may reuse it
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster_relaxed(map_to_cta(smem_u32(&bar_acc_empty[acc]), 0));
                }
                // this warp's previous TMA store must have finished reading the staging rows
                if (lane == 0 && store_pending) tma_store_wait_read();
                __syncwarp();
                gemm_stage_64_columns(sC, lane, v);
                fence_proxy_async_smem();
                __syncwarp();
                const int col0 = bn * p.tile_n + c * 64;
                if (lane == 0 && row0 < p.M && col0 < p.N) {
                    tma_store_4d(&tm_c, sC, col0, row0, 0, 0);
                    tma_store_commit();
                    store_pending = true;
                }
            }
        }
        if (lane == 0 && store_pending) tma_store_wait_all();
    }

    // ---- common exit.  The commit of the last accumulator, which both epilogues wait for, follows all others; if the MMA issuer
    // gave up, its last commit is given a bounded time here, in the odd CTA as in the even one.
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == 2 && *reinterpret_cast<volatile int *>(&drain_flag) != 0)
        for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain), 0); ++w) {}
    if (warp == 2) tmem_dealloc_pair(tmem, Cfg::kTmemCols);
}

}  // namespace ave
