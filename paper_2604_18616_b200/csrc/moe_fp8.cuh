// Block-quantised FP8 fused mixture-of-experts layer for sm_100a (the paper's third kernel family, Section 9:
// DeepSeek-V3.2's block-quantised FP8 configuration; "quantize up-projection intermediates to FP8", "preserve
// blockwise quantization, route tokens through sorted expert maps, and group accesses for coalescing").
//
// Format: E4M3 codes; activations carry one fp32 scale per (token, 128 channels), weights one per 128 x 128
// block.  Steps of one call (all on the caller's stream, scratch in the caller's workspace):
//   1. moe_clear_kernel, 2. moe_count_kernel, 3. moe_plan_kernel: pairs per expert, every expert's first row in the
//      sorted order (a multiple of 128, so a 128-row tile belongs to one expert), the list of row tiles
//   4. moe_gather_kernel: every (token, k) pair gets a row of its expert; the token's codes and scales are copied there
//   5. moe_gemm_fp8_kernel<true>: a = silu(x Wg^T) * (x Wu^T), requantised to E4M3 per 128 columns (grouped by expert,
//      block-scaled, tensor cores)
//   6. moe_gemm_fp8_kernel<false>: o = w * (a W2^T), rows x C, fp32   (w: the pair's routing weight)
//   7. moe_combine_kernel: y[t] = sum over the token's K rows of o, rounded to bf16
// Kernels 2 to 7 are launched with programmatic stream serialisation; each waits for the one before it at its top.
//
// The GEMM: persistent CTAs over 128 x 256 output tiles; K is streamed in blocks of 128 (one scale block)
// through a TMA ring; each block is four M128 x N256 x K32 tcgen05 MMAs (kind::f8f6f4, 512 clk) into one of two TMEM
// accumulators, which the epilogue warps read out and add, multiplied by the block's scales, to fp32
// registers (the accumulation across scale blocks cannot stay in the tensor core: every block has its own
// factor).  Rows are TMEM lanes; two epilogue threads per row, 128 columns each.  Adding a block up takes 350 clk of
// the 512 (bound by the issue of its FMAs), so the read-out keeps up only if its loop does nothing else: a warp
// of its own fetches the scales, blocks ahead, and leaves each block's in shared memory; "accumulator full" then stands for
// the products and their scales.  (With every epilogue thread fetching its own scales a block took 1150-1400 clk.)
// In the up projection a tile is 128 gate columns and the same 128 up columns (one requantisation group); a thread
// holds 64 of each, so the activation needs no exchange but the group's maximum.
//
//   warp 0       producer: TMA loads of the A and B blocks
//   warps 1, 2   MMA issuers (even and odd K blocks); warp 2 also allocates and releases TMEM
//   warp 3       scales
//   warps 4..11  epilogue (thread = output row x half of the tile's columns)
#pragma once

#include <cuda_bf16.h>

#include "attn_common.cuh"

namespace ave {

constexpr int kMoeGroup = 128;  // channels per activation scale, rows and columns per weight scale block

template <bool UP>
struct MoeGemmCfg {
    static constexpr int kThreads = 384;
    static constexpr int kTile = 128;                          // rows of an output tile; K block; columns per epilogue thread
    static constexpr int kTileN = 256;                         // columns of an output tile (two weight scale blocks)
    static constexpr int kBoxRows = 32;                        // rows of A per TMA load: only 32-row groups with a token are loaded
    // The down projection's tiles have few K blocks and a large fp32 result: it trades a ring slot for a second
    // staging buffer per epilogue warp, so that a tile's stores do not wait for one another.
    static constexpr int kStages = UP ? 4 : 3;
    static constexpr int kStoreBufs = 2;
    static constexpr int kABytes = kTile * kMoeGroup;          // 16 KB of E4M3
    static constexpr int kBBytes = kTileN * kMoeGroup;         // 32 KB
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kStageCBytes = 8 * kStoreBufs * 32 * 128;  // result staging: buffers of 32 rows x 32 fp32 per epilogue warp
    static constexpr int kSmemBytes = kStages * kStageBytes + (UP ? 0 : kStageCBytes) + 1024;
    static constexpr int kAccs = 2;                            // TMEM accumulators of 256 columns
    static constexpr uint32_t kTmemCols = kAccs * kTileN;
    // The epilogue threads hold 128 fp32 sums plus a 32-column chunk in flight: they take registers from the
    // producer / MMA warpgroup (setmaxnreg moves them inside the CTA's allocation of kThreads x kRegsAtLaunch;
    // the build and the launch code check the compiled image against this split).
    static constexpr int kRegsLight = 56, kRegsEpilogue = 224, kRegsAtLaunch = 168;
    static_assert(128 * kRegsLight + 256 * kRegsEpilogue <= kThreads * kRegsAtLaunch, "register split exceeds the CTA's allocation");
};

// One 128-row tile of the sorted order.  Row tiles of an expert are visited in groups (of at most kMoeGroupTiles), all of a
// group's row tiles under one column tile before the next column tile, so that weights are read from HBM about once.
constexpr int kMoeGroupTiles = 8;
struct __align__(16) MoeRowTile {
    int expert;
    int group_first, group_tiles;  // the group this tile belongs to
    int rows;                      // rows of this tile that hold a token (the rest is padding: whatever is there is never used)
};

struct MoeGemmParams {
    const float *a_scale;       // [K/128, rows_cap]
    const float *b_scale;       // [E, N/128, K/128]
    const MoeRowTile *tiles;    // [tiles in use]
    const int *n_row_tiles;     // row tiles in use
    const float *row_weight;    // down projection: [rows_cap], factor applied to every output row
    uint8_t *q_out;             // up projection: codes [rows_cap, F] and scales [F/128, rows_cap]
    float *q_scale;
    long long rows_cap;
    int tiles_n;                // up: F / 128; down: ceil(N / 256)
    int nblk;                   // weight scale blocks along N: up 2F / 128, down N / 128
    int kb;                     // K / 128
};

// tcgen05 instruction descriptor, kind::f8f6f4: fp32 accumulator, E4M3 A and B, both K-major.
__host__ __device__ constexpr uint32_t make_idesc_e4m3(int m, int n) {
    return (1u << 4)                       // D format: f32
           | (0u << 7)                     // A format: E4M3
           | (0u << 10)                    // B format: E4M3
           | (uint32_t(n >> 3) << 17)      // N / 8
           | (uint32_t(m >> 4) << 24);     // M / 16
}

__device__ __forceinline__ void umma_f8_ss_words(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                                 uint32_t b_hi, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        ".reg .b64 da, db;\n"
        "setp.ne.b32 p, %6, 0;\n"
        "mov.b64 da, {%1, %2};\n"
        "mov.b64 db, {%3, %4};\n"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %5, p;\n"
        "}\n"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The n-th output tile of the launch: row tile, column tile, the row tile's record.
__device__ __forceinline__ MoeRowTile moe_tile(int id, const MoeGemmParams &p, int &bm, int &bn) {
    const int r = id / p.tiles_n;  // a group of row tiles owns the ids [group_first, group_first + group_tiles) * tiles_n
    const MoeRowTile g = p.tiles[r];
    const int rem = id - g.group_first * p.tiles_n;
    bn = rem / g.group_tiles;
    bm = g.group_first + (rem - bn * g.group_tiles);
    return p.tiles[bm];
}

// Two fp32 values -> two E4M3 codes (round to nearest even, saturating at +-448); `lo` lands in bits 0..7.
__device__ __forceinline__ uint32_t cvt_e4m3x2(float lo, float hi) {
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}

// x / d for two values, given r = 1 / d to within an ulp: one residual step, q + (x - q d) r with the residual exact in an
// FMA (Markstein, IBM J. Res. Dev. 34, 1990).  Nothing here may overflow or be subnormal: the callers see to it.
__device__ __forceinline__ float2 div2_residual(float2 x, float2 d, float2 r) {
    const float2 q = __fmul2_rn(x, r);
    const float2 e = __ffma2_rn(make_float2(-q.x, -q.y), d, x);
    return __ffma2_rn(e, r, q);
}
// silu(z) = z / (1 + exp(-z)) in fp32, for any z: from -88.8 down the exponential is infinite and the result -0.
__device__ __forceinline__ float silu(float z) { return __fdiv_rn(z, 1.f + expf(-z)); }
// The same for two values of at least kSiluFast, below which 1 / (1 + exp(-z)) is no longer a normal number.
constexpr float kSiluFast = -87.f;
__device__ __forceinline__ float2 silu2(float2 z) {
    const float2 d = make_float2(1.f + expf(-z.x), 1.f + expf(-z.y));
    float2 r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
    const float2 nd = make_float2(-d.x, -d.y);
    r = __ffma2_rn(__ffma2_rn(nd, r, make_float2(1.f, 1.f)), r, r);  // one Newton step
    return div2_residual(z, d, r);
}

// Keeps the additions to 16 pairs of sums ahead of what follows: the compiler otherwise loads further blocks of products
// first and, with 128 sums in registers, spills.
__device__ __forceinline__ void pin_sums(float2 *a) {
    asm volatile("" : "+f"(a[0].x), "+f"(a[0].y), "+f"(a[1].x), "+f"(a[1].y), "+f"(a[2].x), "+f"(a[2].y), "+f"(a[3].x), "+f"(a[3].y),
          "+f"(a[4].x), "+f"(a[4].y), "+f"(a[5].x), "+f"(a[5].y), "+f"(a[6].x), "+f"(a[6].y), "+f"(a[7].x), "+f"(a[7].y));
    asm volatile("" : "+f"(a[8].x), "+f"(a[8].y), "+f"(a[9].x), "+f"(a[9].y), "+f"(a[10].x), "+f"(a[10].y), "+f"(a[11].x), "+f"(a[11].y),
          "+f"(a[12].x), "+f"(a[12].y), "+f"(a[13].x), "+f"(a[13].y), "+f"(a[14].x), "+f"(a[14].y), "+f"(a[15].x), "+f"(a[15].y));
}

// UP: the up projection with activation and requantisation; else the down projection.
// tm_a: A codes [rows_cap, K] as {K, rows_cap, 1, 1}, boxes of 128 bytes x 32 rows; tm_b: B codes [E, N, K] as
// {K, N, E, 1}, boxes of 128 bytes x 128 rows (rows beyond N read as zero); tm_c: the down projection's fp32 result
// [rows_cap, N] as {N, rows_cap, 1, 1}, boxes of 32 columns x 32 rows (a thread-per-row store of fp32 rows would touch 32
// rows per instruction, one sector each: measured, that cost more than the tile's products).
template <bool UP>
__global__ void __launch_bounds__(384, 1)
moe_gemm_fp8_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                    const __grid_constant__ CUtensorMap tm_c, const MoeGemmParams p) {
    using Cfg = MoeGemmCfg<UP>;
    constexpr int NS = Cfg::kStages, NA = Cfg::kAccs;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[NS], bar_empty[NS], bar_acc_full[NA], bar_acc_empty[NA], bar_pair[4], bar_drain[NA];
    __shared__ float row_max[UP ? 2 : 1][2][UP ? Cfg::kTile : 1];  // [tile parity][half of the columns][row]
    __shared__ __align__(16) float row_scale[NA][Cfg::kTile];  // scales of the K block in each accumulator: the rows',
    __shared__ __align__(8) float2 col_scale[NA];              // and those of its two weight blocks
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const uint32_t sRing = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int a = 0; a < NA; ++a) {
            mbar_init(smem_u32(&bar_acc_full[a]), 2);   // the MMAs' commit and the scale warp
            mbar_init(smem_u32(&bar_acc_empty[a]), 8);  // one arrival per epilogue warp
        }
        for (int x = 0; x < 4; ++x) mbar_init(smem_u32(&bar_pair[x]), 2);  // the two warps of a row
        for (int a = 0; a < NA; ++a) mbar_init(smem_u32(&bar_drain[a]), 1);
        fence_mbar_init();
        tma_prefetch_desc(&tm_a);
        tma_prefetch_desc(&tm_b);
    }
    if (warp == 2) {
        tmem_alloc(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
        tmem_relinquish();
    }
    grid_dependency_wait();
    grid_dependency_launch();
    if (tid == 0) abort_flag = (*reinterpret_cast<volatile unsigned int *>(&g_device_status) != 0) ? 1 : 0;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_slot;
    const bool poisoned = abort_flag != 0;

    auto wait_bar = [&](uint64_t *bar, uint32_t parity, unsigned code) -> bool {
        const bool r = mbar_wait_bounded(smem_u32(bar), parity, &abort_flag, code);
        return __all_sync(0xffffffffu, r);
    };

    const int n_tiles = *p.n_row_tiles * p.tiles_n;

    if (poisoned) {
        // nothing: fall through to the common exit
    } else if (warp < 4) {
      setmaxnreg_dec<Cfg::kRegsLight>();
      if (warp == 0) {
        // =============================== producer ===============================
        const bool leader = elect_one();
        bool ok = true;
        int ring = 0;  // K blocks loaded so far
        for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
            int bm, bn;
            const MoeRowTile t = moe_tile(id, p, bm, bn);
            const int boxes = (t.rows + Cfg::kBoxRows - 1) / Cfg::kBoxRows;
            const int n0 = UP ? bn * 128 : bn * 256, n1 = UP ? (p.nblk / 2 + bn) * 128 : bn * 256 + 128;  // rows of B
            for (int kb = 0; kb < p.kb && ok; ++kb, ++ring) {
                const int slot = ring % NS, round = ring / NS;
                if (round > 0) {
                    ok = wait_bar(&bar_empty[slot], (round - 1) & 1, STATUS_TIMEOUT_SLOT);
                    if (!ok) break;
                }
                if (leader) {
                    const uint32_t bar = smem_u32(&bar_full[slot]);
                    const uint32_t dst = sRing + slot * Cfg::kStageBytes;
                    mbar_arrive_expect_tx(bar, boxes * (Cfg::kBoxRows * kMoeGroup) + Cfg::kBBytes);
                    tma_load_4d(dst + Cfg::kABytes, &tm_b, bar, kb * kMoeGroup, n0, t.expert, 0);
                    tma_load_4d(dst + Cfg::kABytes + Cfg::kBBytes / 2, &tm_b, bar, kb * kMoeGroup, n1, t.expert, 0);
                    for (int x = 0; x < boxes; ++x)
                        tma_load_4d(dst + x * (Cfg::kBoxRows * kMoeGroup), &tm_a, bar, kb * kMoeGroup,
                                    bm * Cfg::kTile + x * Cfg::kBoxRows, 0, 0);
                }
            }
        }
        if (!ok) {
            for (int it = max(0, ring - NS); it < ring; ++it)
                for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_full[it % NS]), (it / NS) & 1); ++w) {}
        }
      } else if (warp < 3) {
        // =============================== MMA issuers ===============================
        // Warp 1 issues the even K blocks (into accumulator 0), warp 2 the odd ones: issuing blocks the thread for about as
        // long as the MMAs take, so with one issuer the tensor pipe stood still while it went through the next
        // block's barriers (a ready wait costs some 100 clk; a block took 900 clk for 512 of work).
        static_assert(NA == 2, "one issuer per accumulator");
        if (elect_one()) {
            constexpr uint32_t idesc = make_idesc_e4m3(Cfg::kTile, Cfg::kTileN);
            constexpr uint64_t desc_kmajor = make_sdesc_sw128(16, 1024);  // rows of 128 bytes, 8-row atoms of 1024 bytes
            constexpr uint32_t hi = uint32_t(desc_kmajor >> 32), lo = uint32_t(desc_kmajor);
            const int acc = warp - 1;
            const uint32_t d_tmem = tmem + acc * Cfg::kTileN;
            int n_blocks = 0;  // K blocks of this CTA
            for (int id = blockIdx.x; id < n_tiles; id += gridDim.x) n_blocks += p.kb;
            bool ok = true;
            for (int ring = acc; ring < n_blocks; ring += NA) {
                const int slot = ring % NS;
                // Polled, not slept on: what passes from a barrier's completion to the first MMA is idle time of the tensor pipe.
                // The accumulator's wait (the epilogue must have read its previous block out of TMEM) comes last where
                // the ring allows it.  It does if this issuer sees every use of a slot: with an odd number of slots the
                // other issuer takes every second one, and "full" has only two phases to tell uses apart; there the
                // accumulator comes first, because by then the epilogue has gone past the other issuer's use.
                auto wait_full = [&]() { return mbar_poll_bounded(smem_u32(&bar_full[slot]), (ring / NS) & 1, &abort_flag, STATUS_TIMEOUT_LOAD); };
                if (NS % NA == 0) ok = wait_full();
                if (ok && ring >= NA)
                    ok = mbar_poll_bounded(smem_u32(&bar_acc_empty[acc]), ((ring / NA) - 1) & 1, &abort_flag, STATUS_TIMEOUT_SOFTMAX);
                if (ok && NS % NA != 0) ok = wait_full();
                if (!ok) break;
                tc_fence_after();
                const uint32_t a_lo = lo | ((sRing + slot * Cfg::kStageBytes) >> 4);
                const uint32_t b_lo = lo | ((sRing + slot * Cfg::kStageBytes + Cfg::kABytes) >> 4);
#pragma unroll
                for (int kk = 0; kk < kMoeGroup / 32; ++kk)  // K = 32 bytes per instruction
                    umma_f8_ss_words(d_tmem, a_lo + ((kk * 32) >> 4), hi, b_lo + ((kk * 32) >> 4), hi, idesc, kk > 0);
                umma_commit(smem_u32(&bar_empty[slot]));
                umma_commit(smem_u32(&bar_acc_full[acc]));
            }
            if (!ok) {  // abandoned: let the MMAs already issued finish before TMEM is released
                umma_commit(smem_u32(&bar_drain[acc]));
                for (uint32_t w = 0; w < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain[acc]), 0); ++w) {}
            }
        }
        __syncwarp();
      } else if (warp == 3) {
        // =============================== scales ===============================
        constexpr int kAhead = 4;  // K blocks fetched ahead
        bool ok = true;
        int ring = 0;
        for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
            int bm, bn;
            const MoeRowTile t = moe_tile(id, p, bm, bn);
            const float *sa = p.a_scale + bm * Cfg::kTile + lane * 4;
            // weight blocks of the tile's two halves (the last tile's second may lie beyond N: any value will do)
            const int nb0 = UP ? bn : bn * 2, nb1 = UP ? p.nblk / 2 + bn : min(bn * 2 + 1, p.nblk - 1);
            const float *sb = p.b_scale + (size_t(t.expert) * p.nblk + (lane == 0 ? nb0 : nb1)) * p.kb;
            float4 ra[kAhead];
            float rb[kAhead];
            auto fetch = [&](int kb, float4 &a, float &b) {
                kb = min(kb, p.kb - 1);
                a = *reinterpret_cast<const float4 *>(sa + kb * p.rows_cap);
                if (lane < 2) b = sb[kb];
            };
#pragma unroll
            for (int x = 0; x < kAhead; ++x) fetch(x, ra[x], rb[x]);
#pragma unroll 1
            for (int kb0 = 0; kb0 < p.kb && ok; kb0 += kAhead) {
#pragma unroll
                for (int x = 0; x < kAhead; ++x) {
                    if (kb0 + x >= p.kb) break;
                    const int acc = ring % NA;
                    if (ring >= NA) {
                        ok = wait_bar(&bar_acc_empty[acc], ((ring / NA) - 1) & 1, STATUS_TIMEOUT_SOFTMAX);
                        if (!ok) break;
                    }
                    ++ring;
                    *reinterpret_cast<float4 *>(&row_scale[acc][lane * 4]) = ra[x];
                    if (lane < 2) reinterpret_cast<float *>(&col_scale[acc])[lane] = rb[x];
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bar_acc_full[acc]));
                    fetch(kb0 + x + kAhead, ra[x], rb[x]);
                }
            }
        }
      }
    } else {
        // =============================== epilogue ===============================
        setmaxnreg_inc<Cfg::kRegsEpilogue>();
        const int wq = warp & 3;           // TMEM lane quadrant of this warp
        const int half = (warp - 4) >> 2;  // which half of the tile's columns
        const uint32_t lane_sel = uint32_t(wq * 32) << 16;
        const uint32_t sC = sRing + NS * Cfg::kStageBytes + (warp - 4) * (Cfg::kStoreBufs * 32 * 128);  // this warp's staging buffers
        bool ok = true;
        int ring = 0;
        uint32_t n_done = 0;         // tiles this warp has finished (up projection: phase of bar_pair)
        for (int id = blockIdx.x; id < n_tiles && ok; id += gridDim.x) {
            int bm, bn;
            const MoeRowTile t = moe_tile(id, p, bm, bn);
            const int nb = UP ? bn : bn * 2 + half;  // this thread's weight scale block along N (up: and F/128 further on)
            if (wq * 32 >= t.rows || nb >= p.nblk) {
                // no token among this warp's rows, or its half lies beyond N: only hand the accumulators back
                for (int kb = 0; kb < p.kb && ok; ++kb, ++ring) {
                    ok = wait_bar(&bar_acc_full[ring % NA], (ring / NA) & 1, STATUS_TIMEOUT_MMA);
                    if (ok && lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[ring % NA]));
                }
                continue;
            }
            const int row = bm * Cfg::kTile + wq * 32 + lane;
            float2 acc[Cfg::kTile / 2];  // up: 64 gate columns, then 64 up columns; down: 128 columns
#pragma unroll
            for (int c = 0; c < Cfg::kTile / 2; ++c) acc[c] = make_float2(0.f, 0.f);
#pragma unroll 1
            for (int kb = 0; kb < p.kb; ++kb) {
                const int a = ring % NA;
                ok = wait_bar(&bar_acc_full[a], (ring / NA) & 1, STATUS_TIMEOUT_MMA);
                if (!ok) break;
                ++ring;
                tc_fence_after();
                const float sr = row_scale[a][wq * 32 + lane];
                const float2 sc = col_scale[a];
                const float f0 = sr * ((UP || half == 0) ? sc.x : sc.y), f1 = UP ? sr * sc.y : f0;
                const uint32_t t_acc = tmem + a * Cfg::kTileN + lane_sel + half * (UP ? 64 : 128);
                // 32 columns at a time, in an order that has the last of them out of TMEM, and the accumulator handed back,
                // after half of the additions: the MMAs of the block after next wait for that
                uint32_t v[2][32];
                auto load = [&](int c) { tmem_ld_x32(t_acc + ((UP && c >= 2) ? 64 : 0) + c * 32, v[c & 1]); };
                auto add = [&](int c) {
                    const float s = c < 2 ? f0 : f1;
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        acc[c * 16 + e] = __ffma2_rn(make_float2(__uint_as_float(v[c & 1][2 * e]), __uint_as_float(v[c & 1][2 * e + 1])),
                                                     make_float2(s, s), acc[c * 16 + e]);
                    pin_sums(acc + c * 16);
                };
                load(0);
                load(1);
                tmem_wait_ld();
                tmem_pin_x32(v[0]);
                tmem_pin_x32(v[1]);
                add(0);
                load(2);
                add(1);
                load(3);
                tmem_wait_ld();
                tmem_pin_x32(v[0]);
                tmem_pin_x32(v[1]);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[a]));
                add(2);
                add(3);
            }
            if (!ok) break;
            if constexpr (UP) {
                // a = silu(gate) * up; the group's maximum with the thread that has the row's other 64 columns; codes
                float amax = 0.f, lowest = 0.f;
#pragma unroll
                for (int c = 0; c < 32; ++c) lowest = fminf(lowest, fminf(acc[c].x, acc[c].y));
                if (__any_sync(0xffffffffu, lowest < kSiluFast)) {
                    // (no model's gates.  A loop that turns the registers round, so that the code a tile usually jumps over is
                    // short: 64 divisions in line were 1 % of the layer in instruction fetches)
#pragma unroll 1
                    for (int x = 0; x < 32; ++x) {
                        const float2 gate = acc[0], up = acc[32];
#pragma unroll
                        for (int c = 0; c < 31; ++c) acc[c] = acc[c + 1], acc[c + 32] = acc[c + 33];
                        acc[31] = make_float2(silu(gate.x) * up.x, silu(gate.y) * up.y);
                        acc[63] = up;
                        amax = fmaxf(amax, fmaxf(fabsf(acc[31].x), fabsf(acc[31].y)));
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        acc[c] = __fmul2_rn(silu2(acc[c]), acc[c + 32]);
                        amax = fmaxf(amax, fmaxf(fabsf(acc[c].x), fabsf(acc[c].y)));
                    }
                }
                float *const buf = &row_max[n_done & 1][0][wq * 32 + lane];
                buf[half * Cfg::kTile] = amax;
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bar_pair[wq]));
                ok = wait_bar(&bar_pair[wq], n_done & 1, STATUS_TIMEOUT_SOFTMAX);
                if (!ok) break;
                amax = fmaxf(buf[0], buf[Cfg::kTile]);
                ++n_done;
                // (0 for a group of zeros, and where amax is so small, below 3.2e-43, that the quotient rounds to 0: with the
                // factor 1 all of either's codes are 0)
                float s = __fdiv_rn(amax, 448.f);
                if (s == 0.f) s = 1.f;
                if (half == 0) p.q_scale[(long long)bn * p.rows_cap + row] = s;
                float sd = s;
                if (s < 0x1p-60f) {  // a tiny group: scaled up exactly, so that 1 / s and the residuals stay normal
                    sd = s * 0x1p64f;
#pragma unroll
                    for (int c = 0; c < 32; ++c) acc[c] = __fmul2_rn(acc[c], make_float2(0x1p64f, 0x1p64f));
                }
                const float r = __frcp_rn(sd);
                uint4 *dst = reinterpret_cast<uint4 *>(p.q_out + (size_t(row) * (p.nblk / 2) + bn) * kMoeGroup + half * 64);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t w[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const float2 lo = div2_residual(acc[c * 8 + x * 2], make_float2(sd, sd), make_float2(r, r));
                        const float2 hi = div2_residual(acc[c * 8 + x * 2 + 1], make_float2(sd, sd), make_float2(r, r));
                        w[x] = cvt_e4m3x2(lo.x, lo.y) | (cvt_e4m3x2(hi.x, hi.y) << 16);
                    }
                    dst[c] = make_uint4(w[0], w[1], w[2], w[3]);
                }
            } else {
                const float w = p.row_weight[row];
                // 32 columns at a time through this warp's staging buffers (rows of 128 bytes, 128-byte swizzle) and out by
                // TMA; a buffer is written again once the store before the last has read it
#pragma unroll
                for (int c = 0; c < Cfg::kTile / 32; ++c) {
                    const uint32_t buf = sC + (c % Cfg::kStoreBufs) * (32 * 128);
                    if (lane == 0) tma_store_wait_read_but<Cfg::kStoreBufs - 1>();
                    __syncwarp();
#pragma unroll
                    for (int x = 0; x < 16; x += 2) {
                        const uint32_t addr = buf + lane * 128 + ((uint32_t(x >> 1) ^ uint32_t(lane & 7)) << 4);
                        const float2 lo = acc[c * 16 + x], hi = acc[c * 16 + x + 1];
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(__float_as_uint(lo.x * w)),
                                     "r"(__float_as_uint(lo.y * w)), "r"(__float_as_uint(hi.x * w)), "r"(__float_as_uint(hi.y * w))
                                     : "memory");
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_4d(&tm_c, buf, nb * Cfg::kTile + c * 32, bm * Cfg::kTile + wq * 32, 0, 0);
                        tma_store_commit();
                    }
                }
            }
        }
        if (!UP && lane == 0) tma_store_wait_all();
    }

    // ---- common exit: every thread arrives, then TMEM is released
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, Cfg::kTmemCols);
}

// ------------------------------------------------------------------ routing: sort (token, k) pairs by expert
__global__ void moe_clear_kernel(int *counts, int E) {
    for (int e = threadIdx.x; e < E; e += blockDim.x) counts[e] = 0;
}

// Pairs per expert: a histogram per CTA in shared memory, added to the global one.
__global__ void moe_count_kernel(const int *__restrict__ ids, int n_pairs, int E, int *counts) {
    extern __shared__ int hist[];  // E
    grid_dependency_wait();
    grid_dependency_launch();
    for (int e = threadIdx.x; e < E; e += blockDim.x) hist[e] = 0;
    __syncthreads();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_pairs; i += gridDim.x * blockDim.x) {
        const int e = ids[i];
        if (e >= 0 && e < E) atomicAdd(&hist[e], 1);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += blockDim.x)
        if (hist[e]) atomicAdd(&counts[e], hist[e]);
}

// One CTA of 1024 threads: every expert's first row (a multiple of 128; its cursor starts there) and the list of row tiles.
__global__ void __launch_bounds__(1024) moe_plan_kernel(const int *counts, int E, int *cursor, MoeRowTile *tiles, int *n_row_tiles) {
    __shared__ int first[1025], rows[1024], warp_sum[32];  // first row tile and rows of every expert
    const int e = threadIdx.x, lane = e & 31, warp = e >> 5;
    grid_dependency_wait();
    grid_dependency_launch();
    const int n = e < E ? counts[e] : 0;
    int x = (n + 127) / 128;
    const int mine = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = warp_sum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sum[lane] = w;
    }
    __syncthreads();
    const int before = x - mine + (warp > 0 ? warp_sum[warp - 1] : 0);
    first[e] = before;
    rows[e] = n;
    if (e < E) cursor[e] = before * 128;
    if (e == 1023) first[1024] = before + mine;
    __syncthreads();
    const int total = first[1024];
    if (e == 0) *n_row_tiles = total;
    for (int t = e; t < total; t += 1024) {
        int lo = 0, hi = E;  // the expert with first[lo] <= t < first[lo + 1]
        while (hi - lo > 1) {
            const int m = (lo + hi) / 2;
            if (first[m] <= t) lo = m;
            else hi = m;
        }
        const int k = t - first[lo], n_tiles = (rows[lo] + 127) / 128;
        MoeRowTile r;
        r.expert = lo;
        r.group_first = first[lo] + k / kMoeGroupTiles * kMoeGroupTiles;
        r.group_tiles = min(kMoeGroupTiles, first[lo] + n_tiles - r.group_first);
        r.rows = min(128, rows[lo] - k * 128);
        tiles[t] = r;
    }
}

// One CTA per token: every one of its K pairs takes the next row of its expert, and the token's codes, scales (into
// [channel group, row] order) and the pair's routing weight are copied there.  Rows that no pair takes stay as they are.
// (The order of an expert's rows depends on timing; no result does.)
constexpr int kMoeGatherThreads = 128;
__global__ void __launch_bounds__(kMoeGatherThreads)
moe_gather_kernel(const uint8_t *__restrict__ xq, const float *__restrict__ sx, const int *__restrict__ ids,
                  const float *__restrict__ wts, int C, int E, int K, long long rows_cap, int *cursor, int *row_of, uint8_t *xq_s,
                  float *sx_s, float *w_s) {
    __shared__ int row[kMoeGatherThreads];
    const long long t = blockIdx.x;
    const int CG = C / kMoeGroup;
    grid_dependency_wait();
    grid_dependency_launch();
    const uint4 *src = reinterpret_cast<const uint4 *>(xq + t * C);
    for (int k0 = 0; k0 < K; k0 += kMoeGatherThreads) {
        const int k = k0 + threadIdx.x;
        __syncthreads();
        if (k < K) {
            const int e = ids[t * K + k];
            const int r = (e >= 0 && e < E) ? atomicAdd(&cursor[e], 1) : -1;
            row[threadIdx.x] = r;
            row_of[t * K + k] = r;
            if (r >= 0) w_s[r] = wts[t * K + k];
        }
        __syncthreads();
        const int n = min(K - k0, kMoeGatherThreads);
        for (int i = threadIdx.x; i < C / 16; i += kMoeGatherThreads) {
            const uint4 v = src[i];
            for (int x = 0; x < n; ++x)
                if (row[x] >= 0) reinterpret_cast<uint4 *>(xq_s + (long long)row[x] * C)[i] = v;
        }
        for (int i = threadIdx.x; i < CG; i += kMoeGatherThreads) {
            const float v = sx[t * CG + i];
            for (int x = 0; x < n; ++x)
                if (row[x] >= 0) sx_s[i * rows_cap + row[x]] = v;
        }
    }
}

// y[t, :] = sum over the token's K sorted rows of o (already weighted), in the order k = 0..K-1, rounded to bf16.
__global__ void moe_combine_kernel(const float *__restrict__ o, const int *__restrict__ row_of, int T, int C, int K,
                                   __nv_bfloat16 *y) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int per_row = C / 4;
    grid_dependency_wait();
    if (idx >= (long long)T * per_row || *reinterpret_cast<volatile unsigned int *>(&g_device_status) != 0) return;
    const int t = int(idx / per_row), c4 = int(idx - (long long)t * per_row);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < K; ++k) {
        const int row = row_of[t * K + k];
        if (row < 0) continue;
        const float4 v = reinterpret_cast<const float4 *>(o + size_t(row) * C)[c4];
        acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    uint2 out;
    out.x = pack_bf16x2(acc.x, acc.y);
    out.y = pack_bf16x2(acc.z, acc.w);
    reinterpret_cast<uint2 *>(y + size_t(t) * C)[c4] = out;
}

}  // namespace ave
