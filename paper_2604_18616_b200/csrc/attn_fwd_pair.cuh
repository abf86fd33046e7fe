// Attention forward on CTA pairs (cta_group::2) for sm_100a: head dimensions 136 to 256.
//
// A work tile is that of the two-sub-tile kernel (256 query rows of a head, or 128 rows of two heads that share keys), but
// its two sub-tiles belong to the two CTAs of a cluster.  Each CTA has its 128 rows of Q, S, P and O and, in shared memory,
// half of every K and V tile (64 of the keys, half of the columns); the even CTA's thread issues M256 MMAs that read both
// halves.  With one CTA per tile (attn_fwd_1t.cuh) the products are bound by shared memory: a step of 128 keys reads
// 128 KB for Q K^T and 64 KB for P V while the loads write 128 KB, 2500 clk at its 128 B/clk for 2048 clk of MMAs.  Here a
// CTA reads 96 + 32 KB and loads 64 KB: 1500 clk.
// The single-sub-tile kernel / this one: 2 x 32 heads of 4096, causal, D = 256 549 / 460 us (at the power limit); D = 192, 32
// heads of 1602 56 / 46; 16 heads of 100 rows and 8000 keys 106.5 / 79.4.  What bounds it: the power limit, and where tiles are
// few the chain of a step's products and softmax.
//
//   warp 0       producer: TMA loads of Q and of this CTA's halves of K and V
//   warp 1       even CTA: MMA issuer
//   warp 2       TMEM allocation / release; even CTA: tile scheduler, odd CTA: tells it that a tile has been read here
//   warp 3       -
//   warps 4..7   softmax + epilogue (one thread per query row)
//
// TMEM columns (both CTAs): S0 [0,128) O [128,384) S1 [384,512).  Key steps are numbered through all tiles of a CTA; step g's
// scores are in buffer g & 1, and P (bf16 pairs) overwrites their first 64 columns.
#pragma once

#include <cstring>
#include <type_traits>

#include "attn_common.cuh"
#include "attn_fwd_ws.cuh"
#include "softmax_math.cuh"

namespace ave {

struct PairCfg {
    static constexpr int D = 256;
    static constexpr int kThreads = 256;
    static constexpr int kQBytes = BM * D * 2;           // 64 KB: this CTA's rows
    static constexpr int kQBoxBytes = BM * 128;          // 64 columns of them
    static constexpr int kKBoxBytes = (BN / 2) * 128;    // 64 columns of 64 keys
    static constexpr int kVBoxBytes = BN * 128;          // 64 columns of 128 keys
    static constexpr int kSlotBytes = BN * D;            // 32 KB: half a K tile, or half a V tile
    static constexpr int kStages = 5;                    // ring slots, in the order of use K_0, K_1, V_0, K_2, V_1, ...
    static constexpr int kSmemBytes = kQBytes + kStages * kSlotBytes + 1024;
    static constexpr uint32_t kTmemCols = 512;
    static constexpr uint32_t kColS = 0, kColO = 128, kColS1 = 384;
    static constexpr int kPFirst = 96;                   // keys of a step whose probabilities are handed over first
    // Columns of O rescaled at a time.  With scores that rise from key to key, 32 / 64 / 128: 6 x 16 heads of 1113 151 / 145 / 141 us
    // (single-sub-tile kernel 139), 16 heads of 100 rows and 8000 keys 107 / 101 / 98 (113); registers 200 to 208 either way.
    static constexpr int kRescaleCols = 128;
    static constexpr int kTileReaders = 7;               // even CTA: producer, MMA issuer, 4 softmax warps, and the odd CTA as one
    static constexpr int kTileReadersOdd = 5;            // odd CTA: producer, 4 softmax warps
};

// The bounded wait, with the other CTA's writes before its arrival made visible (tile records).
__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint32_t bar, uint32_t parity, volatile int *abort_flag, unsigned int code) {
    const long long t0 = clock64();
    for (;;) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if (*abort_flag != 0) return false;
        if (clock64() - t0 > WAIT_LIMIT_CYCLES) break;
    }
    *abort_flag = 1;
    atomicOr(&g_device_status, code);
    return false;
}

// Barriers: "full" (ring slots, Q) count both CTAs' bytes on the even CTA's copy; "s", "pv" and the "empty" ones are
// signalled in both CTAs by the MMAs' commits; "p" collects both CTAs' softmax warps on the even CTA's copy.  (A warp reads
// a tile's O out of TMEM before it hands over the next tile's first P, which is all that P V has to wait for.)
template <bool CAUSAL, bool VARLEN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(256, 1)
attn_fwd_pair_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v, const FwdParams p) {
    using Cfg = PairCfg;
    using Tile = TileOf<false, VARLEN>;
    constexpr int D = Cfg::D, NS = Cfg::kStages;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(16) unsigned long long clc_response[2][2];
    __shared__ __align__(8) uint64_t bar_q_full, bar_q_empty, bar_full[NS], bar_empty[NS];
    __shared__ __align__(8) uint64_t bar_s[2], bar_p[2][2], bar_pv[2];  // [score buffer]; p: [score buffer][part of the keys]
    __shared__ __align__(8) uint64_t bar_tile_full[2], bar_tile_ready[2], bar_tile_empty[2], bar_drain;
    __shared__ int tile_id[2];
    __shared__ __align__(4) Tile tile_info[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag, poison_flag, drain_flag;  // the last: (odd CTA) the even one's MMA issuer gave up

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int rank = int(cluster_rank());  // = sub-tile

    const uint32_t sQ = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sRing = sQ + Cfg::kQBytes;

    if (tid == 0) {
        abort_flag = drain_flag = 0;
        mbar_init(smem_u32(&bar_q_full), 1);
        mbar_init(smem_u32(&bar_q_empty), 1);
        for (int t = 0; t < 2; ++t) {
            mbar_init(smem_u32(&bar_s[t]), 1);
            mbar_init(smem_u32(&bar_p[t][0]), 8);  // one arrival per softmax warp of both CTAs
            mbar_init(smem_u32(&bar_p[t][1]), 8);
            mbar_init(smem_u32(&bar_pv[t]), 1);
            mbar_init(smem_u32(&bar_tile_full[t]), 1);
            mbar_init(smem_u32(&bar_tile_ready[t]), 1);
            mbar_init(smem_u32(&bar_tile_empty[t]), rank == 0 ? Cfg::kTileReaders : Cfg::kTileReadersOdd);
        }
        mbar_init(smem_u32(&bar_drain), 1);
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        fence_mbar_init();
    }
    if (warp == 2) {
        tmem_alloc_pair(smem_u32(&tmem_base_slot), Cfg::kTmemCols);
        tmem_relinquish_pair();
    }
    // what precedes overlaps the end of the kernel before this one in the stream
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

    // A full warp waits on an mbarrier phase; the verdict is made warp-uniform.
    auto wait_bar = [&](uint64_t *bar, uint32_t parity, unsigned code) -> bool {
        const bool r = mbar_wait_bounded(smem_u32(bar), parity, &abort_flag, code);
        return __all_sync(0xffffffffu, r);
    };
    // (the odd CTA's tile records are written by the even one)
    auto wait_tile = [&](int slot, uint32_t parity) -> bool {
        const uint32_t bar = smem_u32(&bar_tile_ready[slot]);
        const bool r = rank == 0 ? mbar_wait_bounded(bar, parity, &abort_flag, STATUS_TIMEOUT_SLOT)
                                 : mbar_wait_cluster_bounded(bar, parity, &abort_flag, STATUS_TIMEOUT_SLOT);
        return __all_sync(0xffffffffu, r);
    };
    // Every consumer warp of the tile sequence calls this to learn the tile after its n-th one (-1: none left).
    auto next_tile = [&](int n, bool &ok, Tile &w_out) -> int {
        const int slot = n & 1;
        ok = wait_tile(slot, (n >> 1) & 1);
        if (!ok) return -1;
        const int id = tile_id[slot];
        if (id >= 0) w_out = tile_info[slot];
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_tile_empty[slot]));
        return id;
    };
    const int first_id = blockIdx.x >> 1;

    if (poisoned) {
        // nothing: fall through to the common exit
    } else if (warp == 0) {
        // =============================== producer ===============================
        const bool leader = elect_one();
        if (leader) {
            tma_prefetch_desc(&tm_q);
            tma_prefetch_desc(&tm_k);
            tma_prefetch_desc(&tm_v);
        }
        const uint32_t even_q_full = map_to_cta(smem_u32(&bar_q_full), 0), even_full = map_to_cta(smem_u32(bar_full), 0);
        bool ok = true;
        int id = first_id, ring = 0, nt = 0;  // half tiles and Q tiles loaded so far
        Tile w = decode_tile<CAUSAL, false, VARLEN>(id, p);
        for (int n = 0; id >= 0 && ok; ++n) {
            if (w.n1 > 0) {
                if (nt > 0) ok = wait_bar(&bar_q_empty, (nt - 1) & 1, STATUS_TIMEOUT_SLOT);
                if (ok && leader) {
                    if (rank == 0) mbar_arrive_expect_tx(smem_u32(&bar_q_full), 2 * Cfg::kQBytes);
                    for (int x = 0; x < D / 64; ++x)  // the tensor maps are {D, rows, heads, batch}
                        tma_load_4d_pair(sQ + x * Cfg::kQBoxBytes, &tm_q, even_q_full, x * 64, q_base_of(w) + w.q0 + rank * w.dq,
                                         w.h + rank * w.dh, batch_coord(w));
                }
                ++nt;
                auto load = [&](bool is_v, int j) {
                    const int slot = ring % NS, round = ring / NS;
                    if (round > 0) ok = wait_bar(&bar_empty[slot], (round - 1) & 1, STATUS_TIMEOUT_SLOT);
                    if (!ok) return;
                    ++ring;
                    if (leader) {
                        const uint32_t bar = even_full + slot * 8, dst = sRing + slot * Cfg::kSlotBytes;
                        const int key = k_base_of(w) + j * BN;
                        if (rank == 0) mbar_arrive_expect_tx(smem_u32(&bar_full[slot]), 2 * Cfg::kSlotBytes);
                        if (is_v) {
                            for (int x = 0; x < D / 128; ++x)
                                tma_load_4d_pair(dst + x * Cfg::kVBoxBytes, &tm_v, bar, rank * (D / 2) + x * 64, key, w.g, batch_coord(w));
                        } else {
                            for (int x = 0; x < D / 64; ++x)
                                tma_load_4d_pair(dst + x * Cfg::kKBoxBytes, &tm_k, bar, x * 64, key + rank * (BN / 2), w.g, batch_coord(w));
                        }
                    }
                };
                for (int j = 0; j <= w.n1 && ok; ++j) {  // K_0, K_1, V_0, ..., K_{n-1}, V_{n-2}, V_{n-1}
                    if (j < w.n1) load(false, j);
                    if (ok && j > 0) load(true, j - 1);
                }
            }
            if (ok) id = next_tile(n, ok, w);
        }
        // The commits that release what was loaded last arrive in both CTAs, and nothing else waits for them: not before
        // they are here may this CTA's shared memory go to another one.
        for (int pos = first_unreleased(ring, NS); pos < ring && ok; ++pos)
            ok = wait_bar(&bar_empty[pos % NS], (pos / NS) & 1, STATUS_TIMEOUT_SLOT);
        if (nt > 0 && ok) ok = wait_bar(&bar_q_empty, (nt - 1) & 1, STATUS_TIMEOUT_SLOT);
        if (!ok) {
            // abandoned: the loads still in flight are counted on the even CTA's barriers only; give them time to land
            const long long t1 = clock64();
            while (clock64() - t1 < (1ll << 20)) __nanosleep(1000);
        }
    } else if (warp == 1 && rank == 0) {
        // =============================== MMA issuer ===============================
        const bool leader = elect_one();
        // (a negative scale: the tensor pipe negates A, see the two-sub-tile kernel)
        const uint32_t idesc_qk = make_idesc_bf16(2 * BM, BN, 0) | ((p.scale_log2 < 0.f) ? (1u << 13) : 0u);
        constexpr uint32_t idesc_pv = make_idesc_bf16(2 * BM, D, 1);
        constexpr uint64_t desc_k = make_sdesc_sw128(16, 1024), desc_v = make_sdesc_sw128(Cfg::kVBoxBytes, 1024);
        constexpr uint32_t hi_k = uint32_t(desc_k >> 32), lo_k = uint32_t(desc_k), hi_v = uint32_t(desc_v >> 32), lo_v = uint32_t(desc_v);
        const uint32_t q_lo = lo_k | (sQ >> 4);
        auto score_buf = [&](int g) { return tmem + ((g & 1) ? Cfg::kColS1 : Cfg::kColS); };
        bool ok = true;
        int ring = 0, nt = 0, g = 0;  // ring slots taken; tiles with steps; number of the step whose P V comes next
        auto take_slot = [&]() -> uint32_t {  // the next ring slot, once it is full
            ok = wait_bar(&bar_full[ring % NS], (ring / NS) & 1, STATUS_TIMEOUT_LOAD);
            tc_fence_after();
            return sRing + (ring % NS) * Cfg::kSlotBytes;
        };
        auto issue_qk = [&](int step, bool last) {
            const uint32_t k_lo = lo_k | (take_slot() >> 4);
            if (!ok) return;
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)
                    umma_ss_pair_words(score_buf(step), q_lo + (((kk / 4) * Cfg::kQBoxBytes + (kk % 4) * 32) >> 4), hi_k,
                                       k_lo + (((kk / 4) * Cfg::kKBoxBytes + (kk % 4) * 32) >> 4), hi_k, idesc_qk, kk > 0);
                umma_commit_pair(smem_u32(&bar_s[step & 1]));
                umma_commit_pair(smem_u32(&bar_empty[ring % NS]));
                if (last) umma_commit_pair(smem_u32(&bar_q_empty));
            }
            ++ring;
        };
        int id = first_id;
        Tile w = decode_tile<CAUSAL, false, VARLEN>(id, p);
        for (int n = 0; id >= 0 && ok; ++n) {
            if (w.n1 > 0) {
                ok = wait_bar(&bar_q_full, nt & 1, STATUS_TIMEOUT_LOAD);
                if (ok) issue_qk(g, w.n1 == 1);
                ++nt;
                for (int j = 0; j < w.n1 && ok; ++j, ++g) {
                    // the next scores while the softmax of this step runs; P V_{j-1} has read the other buffer's P
                    if (j + 1 < w.n1) issue_qk(g + 1, j + 2 == w.n1);
                    if (!ok) break;
                    const uint32_t v_lo = lo_v | (take_slot() >> 4);
                    if (!ok) break;
                    const uint32_t off0 = j >= w.n0 ? 0xffffffffu : 0u;  // a sub-tile 0 that has no such step keeps its O
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        ok = wait_bar(&bar_p[g & 1][part], (g >> 1) & 1, STATUS_TIMEOUT_SOFTMAX);
                        if (!ok) break;
                        tc_fence_after();
                        if (leader) {
#pragma unroll
                            for (int kk = part ? Cfg::kPFirst / 16 : 0; kk < (part ? BN : Cfg::kPFirst) / 16; ++kk)
                                umma_ts_pair_words(tmem + Cfg::kColO, score_buf(g) + kk * 8, v_lo + ((kk * 16 * 128) >> 4), hi_v, idesc_pv,
                                                   off0, j > 0 || kk > 0);
                        }
                    }
                    if (!ok) break;
                    if (leader) {
                        umma_commit_pair(smem_u32(&bar_pv[g & 1]));
                        umma_commit_pair(smem_u32(&bar_empty[ring % NS]));
                    }
                    ++ring;
                }
            }
            if (ok) id = next_tile(n, ok, w);
        }
        if (!ok) {  // abandoned: let the MMAs already issued finish before TMEM is released
            if (leader) {
                umma_commit_pair(smem_u32(&bar_drain));
                st_cluster_s32(map_to_cta(smem_u32(&drain_flag), 1), 1);  // it arrives there too: the odd CTA has to stay for it
            }
            for (uint32_t x = 0; x < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain), 0); ++x) {}
        }
    } else if (warp == 2 && rank == 0) {
        // =============================== tile scheduler ===============================
        // As in the two-sub-tile kernel (see there for how far ahead it asks), for the pair: what the even CTA's request takes
        // over is a whole cluster, and the decoded tile is written to both CTAs.
        const bool leader = elect_one();
        const uint32_t peer_id = map_to_cta(smem_u32(tile_id), 1), peer_info = map_to_cta(smem_u32(tile_info), 1);
        const uint32_t peer_ready = map_to_cta(smem_u32(bar_tile_ready), 1);
        bool ok = true;
        int last_id = first_id;
        unsigned requests = 0;
        auto all_read = [&](int slot, int use) {
            return __all_sync(0xffffffffu, mbar_wait_cluster_bounded(smem_u32(&bar_tile_empty[slot]), use & 1, &abort_flag, STATUS_TIMEOUT_SLOT));
        };
        for (int k = 0; ok; ++k) {
            const int slot = k & 1;
            if (k >= 2) ok = all_read(slot, (k >> 1) - 1);
            if (ok && k >= 1 && 2 * (p.total_blocks - last_id) <= kLastWaves * int(n_sm())) ok = all_read(slot ^ 1, (k - 1) >> 1);
            if (!ok) break;
            int id;
            for (;;) {
                if (leader) {
                    mbar_arrive_expect_tx(smem_u32(&bar_tile_full[slot]), 16);
                    clc_try_cancel(smem_u32(&clc_response[slot][0]), smem_u32(&bar_tile_full[slot]));
                }
                ok = wait_bar(&bar_tile_full[slot], (requests >> slot) & 1, STATUS_TIMEOUT_SLOT);
                if (!ok) break;
                requests ^= 1u << slot;
                id = clc_decode(clc_response[slot]);
                fence_proxy_async_smem();  // (every lane's read comes before the slot's next asynchronous write)
                __syncwarp();
                if (id < 0) break;
                id >>= 1;
                const Tile w = decode_tile<CAUSAL, false, VARLEN>(id, p);
                if constexpr (VARLEN)
                    if (w.q0 >= w.sq) continue;  // beyond its sequence's end
                if (lane == 0) {
                    tile_info[slot] = w;
                    int words[sizeof(Tile) / 4];
                    memcpy(words, &w, sizeof(Tile));
#pragma unroll
                    for (int x = 0; x < int(sizeof(Tile) / 4); ++x) st_cluster_s32(peer_info + slot * uint32_t(sizeof(Tile)) + x * 4, words[x]);
                }
                break;
            }
            if (!ok) break;
            if (lane == 0) {
                tile_id[slot] = id;
                st_cluster_s32(peer_id + slot * 4, id);
                mbar_arrive(smem_u32(&bar_tile_ready[slot]));
                mbar_arrive_cluster_release(peer_ready + slot * 8);
            }
            __syncwarp();
            if (id < 0) break;  // nothing left to take over: never ask again
            last_id = id;
        }
    } else if (warp == 2) {
        // =============================== odd CTA: tiles read ===============================
        // (an arrival that orders this CTA's reads before the even CTA's next write takes some 1100 clk: not of the softmax
        // warps' time)
        bool ok = true;
        for (int k = 0; ok; ++k) {
            const int slot = k & 1;
            ok = wait_tile(slot, (k >> 1) & 1);
            if (!ok) break;
            const int id = *reinterpret_cast<volatile int *>(&tile_id[slot]);
            ok = wait_bar(&bar_tile_empty[slot], (k >> 1) & 1, STATUS_TIMEOUT_SLOT);
            if (!ok) break;
            if (lane == 0) mbar_arrive_cluster_release(map_to_cta(smem_u32(&bar_tile_empty[slot]), 0));
            __syncwarp();
            if (id < 0) break;
        }
    } else if (warp >= 4) {
        // =============================== softmax warpgroup ===============================
        const int wq = warp & 3;                      // TMEM lane quadrant of this warp
        const int r = wq * 32 + lane;                 // row within the sub-tile = TMEM lane
        const uint32_t lane_sel = uint32_t(wq * 32) << 16;
        const uint32_t tO = tmem + Cfg::kColO + lane_sel;
        const uint32_t even_p = map_to_cta(smem_u32(bar_p), 0);
        // |scale|; a zero scale as 2^-100: see the two-sub-tile kernel
        const float sl2 = (p.scale_log2 == 0.f) ? 7.888609052210118e-31f : fabsf(p.scale_log2);
        bool ok = true;
        int g = 0;  // number of the next step

        int id = first_id;
        Tile w_tile = decode_tile<CAUSAL, false, VARLEN>(id, p);
        for (int n = 0; id >= 0 && ok; ++n) {
            Tile w = w_tile;
            w.h += rank * w.dh;                        // this CTA's query head (head-paired launches)
            w.bh += rank * w.dh;
            const int sq = seq_q(w, p);
            const int off = seq_k(w, p) - sq;
            const int i0 = w.q0 + rank * w.dq;
            const int i = i0 + r;                      // query row
            const int n_t = rank ? w.n1 : w.n0;
            float m_run = -INFINITY, l_run = 0.f;
            const int k_end = key_end(w, p);
            const int n_full = unmasked_steps<CAUSAL, false>(i0, n_t, 0, k_end, off, 0);
            auto step = [&](const int j, auto masked) -> bool {
                // `masked` is a run-time bool (causal kernels) or std::true_type / std::false_type
                constexpr bool kRuntimeFlag = std::is_same<decltype(masked), bool>::value;
                bool need_mask;
                if constexpr (kRuntimeFlag) need_mask = masked;
                else need_mask = decltype(masked)::value;
                const uint32_t buf = g & 1;
                const uint32_t tS = tmem + (buf ? Cfg::kColS1 : Cfg::kColS) + lane_sel;
                ok = wait_bar(&bar_s[buf], (g >> 1) & 1, STATUS_TIMEOUT_MMA);
                if (!ok) return false;
                ++g;
                tc_fence_after();
                uint32_t sraw[4][32];
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_ld_x32(tS + c * 32, sraw[c]);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 4; ++c) tmem_pin_x32(sraw[c]);
                const int mask_trips = kRuntimeFlag ? opaque(need_mask ? 1 : 0) : int(need_mask);
#pragma unroll 1
                for (int trip = 0; trip < mask_trips; ++trip) {
                    const int j0 = j * BN;  // first key of this step
                    int lim = k_end - 1 - j0;  // columns c <= lim of this tile are visible to row i
                    if (CAUSAL) lim = min(lim, i + off - j0);
                    // a masked score becomes -inf: it drops out of the maximum and its probability is exactly 0
#pragma unroll
                    for (int c = 0; c < 128; ++c)
                        sraw[c >> 5][c & 31] = (c <= lim) ? sraw[c >> 5][c & 31] : 0xff800000u;
                }
                // row maximum of the (masked) raw scores, as scale*log2(e)*s; -inf if nothing is visible
                float m_tile;
                {
                    float e0 = -INFINITY, e1 = -INFINITY, e2 = -INFINITY, e3 = -INFINITY;
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        e0 = max3(e0, __uint_as_float(sraw[0][c]), __uint_as_float(sraw[0][c + 1]));
                        e1 = max3(e1, __uint_as_float(sraw[1][c]), __uint_as_float(sraw[1][c + 1]));
                        e2 = max3(e2, __uint_as_float(sraw[2][c]), __uint_as_float(sraw[2][c + 1]));
                        e3 = max3(e3, __uint_as_float(sraw[3][c]), __uint_as_float(sraw[3][c + 1]));
                    }
                    const float ext = fmaxf(fmaxf(e0, e1), fmaxf(e2, e3));
                    m_tile = (ext == -INFINITY) ? -INFINITY : ext * sl2;
                }
                // running maximum, moved lazily (see kRescaleThreshold)
                float alpha = 1.f;
                if (j == 0) {
                    m_run = m_tile;
                } else if (m_tile - m_run > rescale_margin(l_run)) {
                    alpha = ex2_approx(m_run - m_tile);
                    m_run = m_tile;
                }
                // p = exp2(scale*log2e*s - m): P -> bf16 pairs into TMEM over the first 64 columns of S; the row sum is taken
                // from the fp32 probabilities, before the rounding
                const float neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
                float2 acc0 = make_float2(0.f, 0.f), acc1 = make_float2(0.f, 0.f);
                const float2 sc2 = make_float2(sl2, sl2), nm2 = make_float2(neg_m, neg_m);
#pragma unroll
                for (int cc = 0; cc < 4; ++cc) {
                    uint32_t pk[16];
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const float2 x = __ffma2_rn(
                            make_float2(__uint_as_float(sraw[cc][e]), __uint_as_float(sraw[cc][e + 1])), sc2, nm2);
                        float2 pr;
                        if ((kFmaPipeExpMask >> ((e >> 1) & 7)) & 1) {
                            pr = exp2_fma_pipe(x);
                        } else {
                            pr.x = ex2_approx(x.x);
                            pr.y = ex2_approx(x.y);
                        }
                        if (e & 2) acc1 = __fadd2_rn(acc1, pr);
                        else       acc0 = __fadd2_rn(acc0, pr);
                        pk[e >> 1] = pack_bf16x2(pr.x, pr.y);
                    }
                    tmem_st_x16(tS + cc * 16, pk);
                    if (cc != Cfg::kPFirst / 32 - 1 && cc != 3) continue;
                    // O <- alpha * O before P V_j, which is not issued before the first hand-over; P V_{j-1} has to have finished
                    if (cc < 3 && j > 0 && __any_sync(0xffffffffu, alpha != 1.f)) {
                        ok = wait_bar(&bar_pv[buf ^ 1], ((g - 2) >> 1) & 1, STATUS_TIMEOUT_MMA);
                        if (!ok) return false;
                        tc_fence_after();
                        scale_tmem_row<D, Cfg::kRescaleCols>(tO, alpha);
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster_relaxed(even_p + buf * 16 + (cc == 3 ? 8 : 0));
                }
                l_run = l_run * alpha + ((acc0.x + acc0.y) + (acc1.x + acc1.y));
                return true;
            };
            {
                int j = 0;
                if constexpr (CAUSAL) {
                    for (; j < n_t; ++j)
                        if (!step(j, j >= n_full)) break;
                } else {
                    for (; j < n_full; ++j)
                        if (!step(j, std::false_type{})) break;
                    for (; ok && j < n_t; ++j)
                        if (!step(j, std::true_type{})) break;
                }
                // steps that only the other sub-tile has: nothing of theirs reaches this one's O
                for (; ok && j < w.n1; ++j, ++g) {
                    ok = wait_bar(&bar_s[g & 1], (g >> 1) & 1, STATUS_TIMEOUT_MMA);
                    if (ok && lane == 0) {
                        mbar_arrive_cluster_relaxed(even_p + (g & 1) * 16);
                        mbar_arrive_cluster_relaxed(even_p + (g & 1) * 16 + 8);
                    }
                }
            }

            // ---- epilogue: O / l -> bf16 -> global (each thread its own row); LSE = ln2 * (m + log2 l)
            const int last = g - 1;
            if (ok && w.n1 > 0) ok = wait_bar(&bar_pv[last & 1], (last >> 1) & 1, STATUS_TIMEOUT_MMA);
            if (ok) {
                tc_fence_after();
                const float inv_l = (l_run > 0.f) ? 1.f / l_run : 0.f;
                if (i < sq) p.lse[lse_index(w, p, i)] = (l_run > 0.f) ? (m_run + log2f(l_run)) * 0.6931471805599453f : -INFINITY;
                __nv_bfloat16 *o_row = reinterpret_cast<__nv_bfloat16 *>(p.o) + batch_coord(w) * p.o_stride_b + w.h * p.o_stride_h +
                                       (q_base_of(w) + i) * p.o_stride_r;
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                    uint32_t oc[32];
                    if (n_t > 0) {
                        tmem_ld_x32(tO + c * 32, oc);
                        tmem_wait_ld();
                        tmem_pin_x32(oc);
                    } else {  // no key is visible to any row of this sub-tile
#pragma unroll
                        for (int e = 0; e < 32; ++e) oc[e] = 0;
                    }
                    if (i < sq) {
#pragma unroll
                        for (int e = 0; e < 32; e += 8) {
                            uint4 v4;
                            v4.x = pack_bf16x2(__uint_as_float(oc[e]) * inv_l, __uint_as_float(oc[e + 1]) * inv_l);
                            v4.y = pack_bf16x2(__uint_as_float(oc[e + 2]) * inv_l, __uint_as_float(oc[e + 3]) * inv_l);
                            v4.z = pack_bf16x2(__uint_as_float(oc[e + 4]) * inv_l, __uint_as_float(oc[e + 5]) * inv_l);
                            v4.w = pack_bf16x2(__uint_as_float(oc[e + 6]) * inv_l, __uint_as_float(oc[e + 7]) * inv_l);
                            if (c * 32 + e < p.d_true) *reinterpret_cast<uint4 *>(o_row + c * 32 + e) = v4;
                        }
                    }
                }
                tc_fence_before();
            }
            if (ok) id = next_tile(n, ok, w_tile);
        }
        // the commit of the step before the last one, in the other buffer, which only a rescale waits for (see the producer)
        if (g >= 2 && ok) ok = wait_bar(&bar_pv[g & 1], ((g - 2) >> 1) & 1, STATUS_TIMEOUT_MMA);
    }

    // ---- common exit.  All commits have arrived in both CTAs (every "s" and the last "pv" are waited for by the softmax, the
    // last "pv" of the other buffer and the last "empty" ones above) unless the MMA issuer gave up: then the last of them,
    // which follows all it issued, is given a bounded time here, in the odd CTA as in the even one.
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    if (warp == 2 && *reinterpret_cast<volatile int *>(&drain_flag) != 0)
        for (uint32_t x = 0; x < WAIT_LIMIT && !mbar_test_wait(smem_u32(&bar_drain), 0); ++x) {}
    if (warp == 2) tmem_dealloc_pair(tmem, Cfg::kTmemCols);
}

}  // namespace ave
