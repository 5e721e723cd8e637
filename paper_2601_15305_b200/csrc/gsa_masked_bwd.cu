// Backward of sparse gated attention on masked dense tiles (see gsa_masked.cuh): the same derivatives as
// gsa_attn_bwd.cu / gsa_attn_bwd_keys.cu, for index sets that hold more than a few per cent of the visible keys.
//
// With P = exp2(S - lse) on the set and 0 outside, dS = P (dP - delta), S = scale Q K^T, dP = do V'^T:
//   keys kernel (one CTA = 128 keys of a KV head, all rows that see them):    dV' = P^T do,   dK = scale dS^T Q
//   rows kernel (one CTA = 128 (query, head) rows of a KV head, all keys):    dQ = scale dS K
//   target kernel (one CTA = 128 rows x 256 keys at a time, all heads):       pbar = mean over the heads of P
// S and dP are computed in both of the first two: two products more than one fused kernel needs, but every sum stays in
// TMEM from the first tile to the last -- no fp32 array that the row tiles' dQ meet in, no atomics, results that do not
// depend on scheduling.  P and dS go back to TMEM as bf16 over the columns they came from and are the A operand of the
// next product; Q, do, K, V' tiles lie in shared memory once and are read along rows (K-major) for S and dP and along
// columns (MN-major) for the sums.
//
// Bound: the products and the elementwise work between them in turn.  Measured at L = 32K, 16 heads of 128 on 8 KV heads, mean
// budget 2080: 16.5 ms for a call with its target, 12.9 ms without (seven products, 1.20 PFLOP/s over the visible pairs; the keys
// kernel somewhat over 6, the rows kernel over 5), so 3.6 ms for the target (one product, and all the exponentials; 0.6 more while a
// thread alone searched a run's start in each set and every lane summed all heads); 8K 1.18 and 0.85 ms.  The gather kernels take 86
// and 19.0 ms for a call.  The sigmoids of dV and dg2 by rcp.approx or by a rounded division: the same errors against fp64 to six digits
// (1500 rows, 8 heads: 2.8377e-3 and 2.7844e-3), up to 2 % of the call for the division.
//
// Roles in all three: warps 0-15 the elementwise work (four warpgroups side by side, 32 columns of a tile each: with two of
// them the products waited for it), warp 16 copies, warp 17 MMA issue, 18 and 19 small loads.
#include <cooperative_groups.h>

#include "gsa_masked.cuh"

namespace gsa {

namespace {

constexpr int kBwdThreads = 640;
constexpr int kCopyWarp = 16, kMmaWarp = 17;
constexpr float kLog2e = 1.4426950408889634f;

template <int DH>
struct TileBytes {
    static constexpr int CHUNKS = DH / 64;
    static constexpr int CHUNK = 128 * 128;                        // 128 rows of 64 bf16
    static constexpr int TILE = CHUNKS * CHUNK;
};

struct MaskedBwdArgs {
    const uint4* mask;
    const float* lse;              // [B, Lq, n_h], natural logarithm
    const float* delta;            // [B, Lq, n_h]
    const __nv_bfloat16* V;
    const __nv_bfloat16* g2;
    const int32_t* idx;
    const int32_t* kt;
    IdxLayout il;
    __nv_bfloat16* dQ;
    __nv_bfloat16* dK;
    __nv_bfloat16* dV;
    __nv_bfloat16* dg2;
    float* pbar;
    int32_t* dev_status;
    const int32_t* general;
    int32_t q0, rows, row_pitch, key_tiles;
    int32_t B, Lq, Lk, n_h, n_kv, k_max;
    int32_t row_blocks;            // of 128 / G queries
    int32_t abreast_keys, abreast_rows;      // tile_order
    int32_t pairs_per_cta, runs;   // target kernel: runs of that many pairs of key tiles, one per CTA
    float scale, scale_log2;
    uint4* zero;                   // what the general path finds cleared (see launch_attn_bwd_keys_general)
    int64_t zero_vec;
    long long wait_cycles;
    int32_t withhold_first;        // fault injection: the first copy of a ring is left out (its barrier is never completed)
};

// 128-row K-major operand: k-step of 16 columns
__device__ __forceinline__ uint64_t kmajor_step(int k) { return (uint64_t)((k >> 2) * (TileBytes<128>::CHUNK >> 4) + 2 * (k & 3)); }

template <int DH>
__device__ __forceinline__ void mma_kmajor(uint32_t el, uint32_t d, uint32_t a_smem, uint32_t b_smem) {        // D = A B^T over DH columns
    const uint64_t ad = make_kmajor_desc<128>(a_smem), bd = make_kmajor_desc<128>(b_smem);
#pragma unroll
    for (int k = 0; k < DH / 16; ++k)
        warp_mma_ss(el, d, ad + kmajor_step(k), bd + kmajor_step(k), make_idesc_bf16(128, 128), k > 0);
}
// D += A B with A (128 x 128, bf16) in TMEM in four parts of 32 contraction elements, 32 columns apart, and B the rows of a tile
template <int DH>
__device__ __forceinline__ void mma_tmem_rows(uint32_t el, uint32_t d, uint32_t a_tmem, uint32_t b_smem, bool accumulate) {
    const uint64_t bd = make_mnmajor_desc(b_smem, TileBytes<DH>::CHUNK);
#pragma unroll
    for (int k = 0; k < 8; ++k)
        warp_mma_ts(el, d, a_tmem + (k >> 1) * 32 + (k & 1) * 8, bd + 128 * k, make_idesc_bf16(128, DH) | kIdescTransB,
                       accumulate || k > 0);
}

#define GSA_TILE_PROLOGUE(PLAN)                                                                                          \
    extern __shared__ unsigned char dyn_smem_raw[];                                                                     \
    const uint32_t raw_u32 = smem_u32(dyn_smem_raw);                                                                    \
    const uint32_t pad = (1024u - (raw_u32 & 1023u)) & 1023u;                                                           \
    unsigned char* const smem = dyn_smem_raw + pad;                                                                     \
    const uint32_t sbase = raw_u32 + pad;                                                                               \
    uint32_t* const s_tmem = reinterpret_cast<uint32_t*>(smem + PLAN::OFF_TMEM);                                        \
    volatile int* const s_abort = reinterpret_cast<volatile int*>(smem + PLAN::OFF_ABORT);                              \
    const uint32_t bar0 = sbase + PLAN::OFF_BAR;                                                                        \
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

__device__ __forceinline__ uint32_t tile_start(int timed_out, int warp, uint32_t tmem_slot, const uint32_t* s_tmem, volatile int* s_abort) {
    if (threadIdx.x == 0) {
        *s_abort = timed_out;                                      // (then every wait ends at once)
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tmem_slot) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    return *s_tmem;
}

// End of a kernel: on the give-up path what was issued completes first (each poll is bounded), then TMEM is released.
// drain_copies / drain_commits poll the barriers of the issuing threads' own copies / commits.
template <class FC, class FM>
__device__ __forceinline__ void tile_end(int warp, int lane, uint32_t tmem, volatile int* s_abort, uint32_t bar_drain,
                                         FC drain_copies, FM drain_commits) {
    tc_fence_before();
    __syncthreads();
    if (*s_abort) {
        if (warp == kCopyWarp && lane == 0) drain_copies();
        if (warp == kMmaWarp) {
            warp_commit(elect_lane(), bar_drain);
            mbar_drain(bar_drain, 0);
            drain_commits();
        }
        tc_fence_before();
        __syncthreads();
    }
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// ---- keys: dK, dV, dg2 -----------------------------------------------------------------------------------------
template <int DH, int G>
struct KeysSmem {
    using T = TileBytes<DH>;
    static constexpr int QT = 128 / G;
    static constexpr int STAGES = DH == 128 ? 2 : 4;               // (Q, do) tile pairs in flight
    static constexpr int OFF_K = 0, OFF_V = T::TILE, OFF_RING = 2 * T::TILE;
    static constexpr int OFF_STAT = OFF_RING + STAGES * 2 * T::TILE;
    static constexpr int STAT_BYTES = 128 * 8 + QT * 16;           // lse2 and delta per row, four mask words per query
    static constexpr int OFF_BAR = OFF_STAT + STAGES * STAT_BYTES;
    static constexpr int N_BARS = 5 * STAGES + 8;
    static constexpr int OFF_TMEM = OFF_BAR + N_BARS * 8;
    static constexpr int OFF_ABORT = OFF_TMEM + 8;
    static constexpr int ALLOC = OFF_ABORT + 8 + 1024;
};

struct KeysEndMaps { CUtensorMap v, g2, dk, dv, dg2; };            // V as given and the gate logits; the results

template <int DH, int G, int SPLIT>
__global__ void __launch_bounds__(kBwdThreads, 1)
gsa_masked_bwd_keys_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
                           const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                           const __grid_constant__ KeysEndMaps end, const MaskedBwdArgs a) {
    chain_wait();
    using P = KeysSmem<DH, G>;
    using T = TileBytes<DH>;
    constexpr int QT = P::QT, ST = P::STAGES;
    constexpr uint32_t kTmS = 0, kTmP = 128, kTmV = 256, kTmK = 384;
    int timed_out;
    if (!tiles_allowed(a.dev_status, &timed_out)) {                // (no one reads the masks, whose space this is, from here on)
        for (int64_t i = (int64_t)blockIdx.x * kBwdThreads + threadIdx.x; i < a.zero_vec; i += (int64_t)gridDim.x * kBwdThreads)
            a.zero[i] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    GSA_TILE_PROLOGUE(P)
    auto bar_q = [&](int s) { return bar0 + 8u * s; };                       // Q tile landed
    auto bar_d = [&](int s) { return bar0 + 8u * (ST + s); };                // do tile landed
    auto bar_free = [&](int s) { return bar0 + 8u * (2 * ST + s); };         // both consumed
    auto bar_stat = [&](int s) { return bar0 + 8u * (3 * ST + s); };         // row statistics and masks stored
    auto bar_statfree = [&](int s) { return bar0 + 8u * (4 * ST + s); };
    const uint32_t bar_kv = bar0 + 8u * (5 * ST), bar_s = bar_kv + 8, bar_dp = bar_kv + 16, bar_p = bar_kv + 24,
                   bar_ds = bar_kv + 32, bar_done = bar_kv + 40, bar_drain = bar_kv + 48;

    // (early key tiles are the long ones)  SPLIT = 2: a cluster of two CTAs shares a tile's
    // rows, every other row tile each, for calls whose key tiles leave half of the SMs without work; at the end each sends the
    // other one of its two sums through distributed shared memory, and the first finishes dK, the second dV and dg2.
    const int part_of = SPLIT > 1 ? (int)(blockIdx.x % SPLIT) : 0;
    const int item = (int)(blockIdx.x / SPLIT);
    int tile, bh;
    tile_order(item, a.key_tiles, (int)(gridDim.x / SPLIT) / a.key_tiles, a.abreast_keys, &tile, &bh);
    const int g = bh % a.n_kv, b = bh / a.n_kv;
    const int off = a.Lk - a.Lq;
    const int r_first = max(0, tile * kMaskTileKeys - off - a.q0);           // first row that sees a key of the tile
    const int i0 = r_first / QT + part_of;
    // (tiles that no row sees have no masks)
    auto row_tiles = [&](int from) { return r_first < a.rows && from < a.row_blocks ? (a.row_blocks - from + SPLIT - 1) / SPLIT : 0; };
    const int n = row_tiles(i0);
    const bool makes_k = part_of == 0, makes_v = part_of == SPLIT - 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(bar_q(s), 1); mbar_init(bar_d(s), 1); mbar_init(bar_free(s), 1);
            mbar_init(bar_stat(s), 64); mbar_init(bar_statfree(s), 16);
        }
        mbar_init(bar_kv, 1); mbar_init(bar_s, 1); mbar_init(bar_dp, 1); mbar_init(bar_p, 16); mbar_init(bar_ds, 16);
        mbar_init(bar_done, 1); mbar_init(bar_drain, 1);
    }
    const uint32_t tmem = tile_start(timed_out, warp, sbase + P::OFF_TMEM, s_tmem, s_abort);
    int copies = 0, kv_issued = 0, released = 0;
    bool done = false;

    if (warp == kCopyWarp) {
        if (lane == 0) {
            if (n > 0) {
                mbar_expect_tx(bar_kv, 2 * T::TILE);
                for (int c = 0; c < T::CHUNKS; ++c) {
                    tma_load_tile(sbase + P::OFF_K + c * T::CHUNK, &tm_k, c * 64, g, tile * kMaskTileKeys, b, bar_kv);
                    tma_load_tile(sbase + P::OFF_V + c * T::CHUNK, &tm_v, c * 64, g, tile * kMaskTileKeys, b, bar_kv);
                }
                kv_issued = 1;
            }
            bool ok = true;
            const int entries = n + (makes_v ? 1 : 0);             // the ring's last entry: V and the gate logits, for the end
            for (int i = 0; ok && i < entries; ++i) {
                const int s = i % ST;
                if (!mbar_wait(bar_free(s), ((i / ST) & 1) ^ 1, s_abort, a.wait_cycles)) { ok = false; break; }
                const uint32_t dst = sbase + P::OFF_RING + s * 2 * T::TILE;
                const bool rows = i < n;
                const int z = rows ? (i0 + i * SPLIT) * QT : tile * kMaskTileKeys, h = rows ? g * G : g;
                if (i > 0 || !a.withhold_first) {
                    mbar_expect_tx(bar_q(s), T::TILE);
                    for (int c = 0; c < T::CHUNKS; ++c) tma_load_tile(dst + c * T::CHUNK, rows ? &tm_q : &end.v, c * 64, h, z, b, bar_q(s));
                }
                mbar_expect_tx(bar_d(s), T::TILE);
                for (int c = 0; c < T::CHUNKS; ++c)
                    tma_load_tile(dst + T::TILE + c * T::CHUNK, rows ? &tm_do : &end.g2, c * 64, h, z, b, bar_d(s));
                copies = i + 1;
            }
            if (!ok) atomicCAS(a.dev_status, kDevOk, kDevTimeoutTma);
        }
    } else if (warp == kMmaWarp) {
        if (n > 0) {                                               // (converged warp)
            const uint32_t el = elect_lane();
            auto q_at = [&](int i) { return sbase + P::OFF_RING + (i % ST) * 2 * T::TILE; };
            auto d_at = [&](int i) { return q_at(i) + T::TILE; };
            auto wait = [&](uint32_t bar, uint32_t parity) { return warp_wait(bar, parity, s_abort, a.wait_cycles); };
            auto issue_s = [&](int i) {                            // S^T = K Q^T
                if (!wait(bar_q(i % ST), (i / ST) & 1)) return false;
                mma_kmajor<DH>(el, tmem + kTmS, sbase + P::OFF_K, q_at(i));
                warp_commit(el, bar_s);
                return true;
            };
            auto issue_dp = [&](int i) {                           // dP^T = V' do^T
                if (!wait(bar_d(i % ST), (i / ST) & 1)) return false;
                mma_kmajor<DH>(el, tmem + kTmP, sbase + P::OFF_V, d_at(i));
                warp_commit(el, bar_dp);
                return true;
            };
            bool ok = wait(bar_kv, 0) && issue_s(0) && issue_dp(0);
            for (int i = 0; ok && i < n; ++i) {
                // every product is issued behind the one that reads what it overwrites
                if (!(ok = wait(bar_p, i & 1))) break;
                mma_tmem_rows<DH>(el, tmem + kTmV, tmem + kTmS, d_at(i), i > 0);       // dV' += P^T do
                if (i + 1 < n && !(ok = issue_s(i + 1))) break;
                if (!(ok = wait(bar_ds, i & 1))) break;
                mma_tmem_rows<DH>(el, tmem + kTmK, tmem + kTmP, q_at(i), i > 0);       // dK += dS^T Q
                warp_commit(el, bar_free(i % ST));
                released = i + 1;
                if (i + 1 < n) ok = issue_dp(i + 1);
            }
            if (ok) warp_commit(el, bar_done);
            else if (lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutMma);
        }
    } else if (warp > kMmaWarp) {
        // row statistics and masks of the next tiles: thread = two rows
        const int j = threadIdx.x - (kMmaWarp + 1) * 32;
        bool ok = true;
        for (int i = 0; ok && i < n; ++i) {
            const int s = i % ST;
            float l2[2], dl[2];
            uint4 mk[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int m = j + 64 * u, r = (i0 + i * SPLIT) * QT + m / G;
                l2[u] = dl[u] = 0.f;
                if (r < a.rows) {
                    const size_t at = ((size_t)b * a.Lq + a.q0 + r) * a.n_h + g * G + m % G;
                    l2[u] = a.lse[at] * kLog2e;
                    dl[u] = a.delta[at];
                }
                const int rq = (i0 + i * SPLIT) * QT + m;                  // (this thread's query for the masks)
                mk[u] = make_uint4(0u, 0u, 0u, 0u);
                if (m < QT && rq < a.rows) mk[u] = a.mask[((int64_t)b * a.key_tiles + tile) * a.row_pitch + rq];
            }
            if (!(ok = warp_wait(bar_statfree(s), ((i / ST) & 1) ^ 1, s_abort, a.wait_cycles))) break;
            float* st = reinterpret_cast<float*>(smem + P::OFF_STAT + s * P::STAT_BYTES);
            uint32_t* sm = reinterpret_cast<uint32_t*>(st + 256);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int m = j + 64 * u;
                st[m] = l2[u];
                st[128 + m] = dl[u];
                if (m < QT) { sm[m] = mk[u].x; sm[QT + m] = mk[u].y; sm[2 * QT + m] = mk[u].z; sm[3 * QT + m] = mk[u].w; }
            }
            mbar_arrive(bar_stat(s));
        }
        if (!ok && lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutEpi);
    } else {
        // lane = key; this warpgroup's quarter of the 128 rows
        const int part = warp >> 2, quad = warp & 3;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t ts = lane_base + kTmS + 32 * part, tp = lane_base + kTmP + 32 * part;
        const uint32_t my_bit = 1u << lane;
        bool ok = true;
        for (int i = 0; i < n; ++i) {
            const int s = i % ST;
            const float* st = reinterpret_cast<const float*>(smem + P::OFF_STAT + s * P::STAT_BYTES) + 32 * part;
            const uint32_t* sm = reinterpret_cast<const uint32_t*>(smem + P::OFF_STAT + s * P::STAT_BYTES + 1024) +
                                 quad * QT + 32 / G * part;
            if (!(ok = warp_wait(bar_stat(s), (i / ST) & 1, s_abort, a.wait_cycles) &&
                       warp_wait(bar_s, i & 1, s_abort, a.wait_cycles))) break;
            uint32_t v[32], pk[16];
            tc_ld32(ts, v);
            tc_wait_ld32(v);
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                const float4 l2 = *reinterpret_cast<const float4*>(st + c);
                const float lv[4] = {l2.x, l2.y, l2.z, l2.w};
                float pv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x = ex2_approx(fmaf(__uint_as_float(v[c + e]), a.scale_log2, -lv[e]));
                    pv[e] = (sm[(c + e) / G] & my_bit) ? x : 0.f;
                    v[c + e] = __float_as_uint(pv[e]);
                }
                pk[c / 2] = pack_bf16(pv[0], pv[1]);
                pk[c / 2 + 1] = pack_bf16(pv[2], pv[3]);
            }
            tc_st16(ts, pk);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p);

            if (!(ok = warp_wait(bar_dp, i & 1, s_abort, a.wait_cycles))) break;
            uint32_t w[32];
            tc_ld32(tp, w);
            tc_wait_ld32(w);
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                const float4 dl = *reinterpret_cast<const float4*>(st + 128 + c);
                const float dv[4] = {dl.x, dl.y, dl.z, dl.w};
                float ds[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) ds[e] = __uint_as_float(v[c + e]) * (__uint_as_float(w[c + e]) - dv[e]);
                pk[c / 2] = pack_bf16(ds[0], ds[1]);
                pk[c / 2 + 1] = pack_bf16(ds[2], ds[3]);
            }
            tc_st16(tp, pk);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) { mbar_arrive(bar_ds); mbar_arrive(bar_statfree(s)); }
        }
        done = ok && (n == 0 || warp_wait(bar_done, 0, s_abort, a.wait_cycles)) &&
               (!makes_v || (warp_wait(bar_q(n % ST), (n / ST) & 1, s_abort, a.wait_cycles) &&
                             warp_wait(bar_d(n % ST), (n / ST) & 1, s_abort, a.wait_cycles)));
        if (!done && lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutEpi);
        tc_fence_after();
    }
    // ---- sums: dK and dV' of key (quad, lane), columns part * DH / 4 .. of the head ----
    const int part = (warp & 15) >> 2, quad = warp & 3, m = quad * 32 + lane;
    auto sum = [&](uint32_t tm, int c, uint32_t (&x)[16]) {        // 16 columns of one of the sums
        if (n > 0) {
            tc_ld16(tmem + ((uint32_t)(quad * 32) << 16) + tm + part * (DH / 4) + 16 * c, x);
            tc_wait_ld16(x);
        } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = 0u;
        }
    };
    // what the other CTA sends: one float per column and key, lanes side by side, in the ring's stage behind the last one used
    auto received = [&](int entries) {
        return reinterpret_cast<float*>(smem + P::OFF_RING + (entries + 1) % ST * 2 * T::TILE) + part * (DH / 4) * 128 + m;
    };
    if constexpr (SPLIT > 1) {
        namespace cg = cooperative_groups;
        static_assert(2 * T::TILE >= DH * 128 * 4, "a sum fits one stage of the ring");
        cg::this_cluster().sync();
        if (warp < 16 && done) {
            float* const to = cg::this_cluster().map_shared_rank(received(row_tiles(i0 + 1 - 2 * part_of)), 1 - part_of);
#pragma unroll
            for (int c = 0; c < DH / 64; ++c) {
                uint32_t x[16];
                sum(makes_k ? kTmV : kTmK, c, x);
#pragma unroll
                for (int e = 0; e < 16; ++e) to[(16 * c + e) * 128] = __uint_as_float(x[e]);
            }
        }
        cg::this_cluster().sync();
    }
    if (warp < 16) {
        // The results go where their tiles lie in shared memory (dK over K, dV over V, dg2 over the logits) and out as boxes; keys past
        // the last are clipped.
        unsigned char* const stage = smem + P::OFF_RING + n % ST * 2 * T::TILE;
        if (done) {
#pragma unroll
            for (int c = 0; c < DH / 64; ++c) {
                const int col = part * (DH / 4) + 16 * c;
                const uint32_t piece0 = (col >> 6) * T::CHUNK + m * 128;
                auto piece = [&](int q) { return piece0 + (((((col & 63) >> 3) + q) ^ (m & 7)) << 4); };
                auto whole_sum = [&](uint32_t tm, uint32_t (&x)[16]) {
                    sum(tm, c, x);
                    if constexpr (SPLIT > 1) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) x[e] = __float_as_uint(__uint_as_float(x[e]) + received(n)[(16 * c + e) * 128]);
                    }
                };
                if (makes_k) {
                    uint32_t dk[16];
                    whole_sum(kTmK, dk);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint32_t x[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            x[e] = pack_bf16(__uint_as_float(dk[8 * q + 2 * e]) * a.scale, __uint_as_float(dk[8 * q + 2 * e + 1]) * a.scale);
                        *reinterpret_cast<uint4*>(smem + P::OFF_K + piece(q)) = make_uint4(x[0], x[1], x[2], x[3]);
                    }
                }
                if (makes_v) {
                    uint32_t dv[16];
                    whole_sum(kTmV, dv);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        uint4* const at_v = reinterpret_cast<uint4*>(stage + piece(q));
                        uint4* const at_g = reinterpret_cast<uint4*>(stage + T::TILE + piece(q));
                        const uint4 vv = *at_v, gg = *at_g;
                        const __nv_bfloat162* vp = reinterpret_cast<const __nv_bfloat162*>(&vv);
                        const __nv_bfloat162* gp = reinterpret_cast<const __nv_bfloat162*>(&gg);
                        uint32_t ov[4], og[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 vf = __bfloat1622float2(vp[e]), gf = __bfloat1622float2(gp[e]);
                            const float s0 = fast_sigmoid(gf.x), s1 = fast_sigmoid(gf.y);
                            const float d0 = __uint_as_float(dv[8 * q + 2 * e]), d1 = __uint_as_float(dv[8 * q + 2 * e + 1]);
                            ov[e] = pack_bf16(d0 * s0, d1 * s1);
                            og[e] = pack_bf16(d0 * vf.x * s0 * (1.0f - s0), d1 * vf.y * s1 * (1.0f - s1));
                        }
                        *at_v = make_uint4(ov[0], ov[1], ov[2], ov[3]);
                        *at_g = make_uint4(og[0], og[1], og[2], og[3]);
                    }
                }
            }
        }
        if (tile_results_written(1, 512, done) && threadIdx.x == 0) {
            for (int c = 0; c < T::CHUNKS; ++c) {
                if (makes_k) tma_store_tile(&end.dk, c * 64, g, tile * kMaskTileKeys, b, sbase + P::OFF_K + c * T::CHUNK);
                if (makes_v) {
                    const uint32_t from = sbase + P::OFF_RING + n % ST * 2 * T::TILE + c * T::CHUNK;
                    tma_store_tile(&end.dv, c * 64, g, tile * kMaskTileKeys, b, from);
                    tma_store_tile(&end.dg2, c * 64, g, tile * kMaskTileKeys, b, from + T::TILE);
                }
            }
            tma_store_wait();
        }
    }
    tile_end(warp, lane, tmem, s_abort, bar_drain,
             [&] {
                 if (kv_issued) mbar_drain(bar_kv, 0);
                 for (int i = max(0, copies - ST); i < copies; ++i) {
                     if (i > 0 || !a.withhold_first) mbar_drain(bar_q(i % ST), (i / ST) & 1);
                     mbar_drain(bar_d(i % ST), (i / ST) & 1);
                 }
             },
             [&] { for (int i = max(0, released - ST); i < released; ++i) mbar_drain(bar_free(i % ST), (i / ST) & 1); });
}

// ---- rows: dQ --------------------------------------------------------------------------------------------------
template <int DH>
struct RowsSmem {
    using T = TileBytes<DH>;
    static constexpr int SLOTS = DH == 128 ? 5 : 8;                // K_0 V_0 K_1 V_1 ... in flight
    static constexpr int OFF_Q = 0, OFF_D = T::TILE, OFF_RING = 2 * T::TILE;
    static constexpr int OFF_BAR = OFF_RING + SLOTS * T::TILE;
    static constexpr int N_BARS = 2 * SLOTS + 8;
    static constexpr int OFF_TMEM = OFF_BAR + N_BARS * 8;
    static constexpr int OFF_ABORT = OFF_TMEM + 8;
    static constexpr int ALLOC = OFF_ABORT + 8 + 1024;
};

template <int DH, int G>
__global__ void __launch_bounds__(kBwdThreads, 1)
gsa_masked_bwd_rows_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
                           const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                           const MaskedBwdArgs a) {
    chain_wait();
    using P = RowsSmem<DH>;
    using T = TileBytes<DH>;
    constexpr int QT = 128 / G, SL = P::SLOTS;
    constexpr uint32_t kTmS = 0, kTmP = 256, kTmQ = 384;           // S at kTmS + 128 (i & 1)
    int timed_out;
    if (!tiles_allowed(a.dev_status, &timed_out)) return;
    GSA_TILE_PROLOGUE(P)
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (SL + s); };
    const uint32_t bar_qd = bar0 + 8u * (2 * SL), bar_s0 = bar_qd + 8, bar_dp = bar_qd + 24, bar_read = bar_qd + 32,
                   bar_ds = bar_qd + 40, bar_done = bar_qd + 48, bar_drain = bar_qd + 56;
    auto bar_s = [&](int i) { return bar_s0 + 8u * (i & 1); };     // (both buffers may be outstanding)

    int rank, bh;                                                  // (late rows are the long ones)
    tile_order(blockIdx.x, a.row_blocks, gridDim.x / a.row_blocks, a.abreast_rows, &rank, &bh);
    const int blk = a.row_blocks - 1 - rank;
    const int g = bh % a.n_kv, b = bh / a.n_kv;
    const int r0 = blk * QT, off = a.Lk - a.Lq;
    const int n = min((off + a.q0 + min(r0 + QT, a.rows) + kMaskTileKeys - 1) / kMaskTileKeys, a.key_tiles);

    if (threadIdx.x == 0) {
        for (int s = 0; s < SL; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        mbar_init(bar_qd, 1); mbar_init(bar_s(0), 1); mbar_init(bar_s(1), 1); mbar_init(bar_dp, 1); mbar_init(bar_read, 16);
        mbar_init(bar_ds, 16); mbar_init(bar_done, 1); mbar_init(bar_drain, 1);
    }
    const uint32_t tmem = tile_start(timed_out, warp, sbase + P::OFF_TMEM, s_tmem, s_abort);
    int copies = 0, qd_issued = 0, k_released = 0, v_released = 0;

    if (warp == kCopyWarp) {
        if (lane == 0) {
            mbar_expect_tx(bar_qd, 2 * T::TILE);
            for (int c = 0; c < T::CHUNKS; ++c) {
                tma_load_tile(sbase + P::OFF_Q + c * T::CHUNK, &tm_q, c * 64, g * G, r0, b, bar_qd);
                tma_load_tile(sbase + P::OFF_D + c * T::CHUNK, &tm_do, c * 64, g * G, r0, b, bar_qd);
            }
            qd_issued = 1;
            bool ok = true;
            for (int e = 0; ok && e < 2 * n; ++e) {
                const int s = e % SL;
                if (!mbar_wait(bar_empty(s), ((e / SL) & 1) ^ 1, s_abort, a.wait_cycles)) { ok = false; break; }
                copies = e + 1;
                if (e == 0 && a.withhold_first) continue;
                mbar_expect_tx(bar_full(s), T::TILE);
                for (int c = 0; c < T::CHUNKS; ++c)
                    tma_load_tile(sbase + P::OFF_RING + s * T::TILE + c * T::CHUNK, (e & 1) ? &tm_v : &tm_k, c * 64, g,
                                  (e >> 1) * kMaskTileKeys, b, bar_full(s));
            }
            if (!ok) atomicCAS(a.dev_status, kDevOk, kDevTimeoutTma);
        }
    } else if (warp == kMmaWarp) {
        {
            const uint32_t el = elect_lane();
            auto wait = [&](uint32_t bar, uint32_t parity) { return warp_wait(bar, parity, s_abort, a.wait_cycles); };
            auto slot = [&](int e) { return sbase + P::OFF_RING + (e % SL) * T::TILE; };
            auto landed = [&](int e) { return wait(bar_full(e % SL), (e / SL) & 1); };
            auto issue_s = [&](int i) {                            // S = Q K^T
                if (!landed(2 * i)) return false;
                mma_kmajor<DH>(el, tmem + kTmS + 128 * (i & 1), sbase + P::OFF_Q, slot(2 * i));
                warp_commit(el, bar_s(i));
                return true;
            };
            auto issue_dp = [&](int i) {                           // dP = do V'^T
                if (!landed(2 * i + 1)) return false;
                mma_kmajor<DH>(el, tmem + kTmP, sbase + P::OFF_D, slot(2 * i + 1));
                warp_commit(el, bar_dp);
                warp_commit(el, bar_empty((2 * i + 1) % SL));
                v_released = i + 1;
                return true;
            };
            bool ok = wait(bar_qd, 0) && issue_s(0) && issue_dp(0) && (n < 2 || issue_s(1));
            for (int i = 0; ok && i < n; ++i) {
                if (i + 1 < n) ok = wait(bar_read, i & 1) && issue_dp(i + 1);      // the columns of dP(i) have been read
                if (!ok || !(ok = wait(bar_ds, i & 1))) break;
                mma_tmem_rows<DH>(el, tmem + kTmQ, tmem + kTmS + 128 * (i & 1), slot(2 * i), i > 0);      // dQ += dS K
                warp_commit(el, bar_empty((2 * i) % SL));
                k_released = i + 1;
                if (i + 2 < n) ok = issue_s(i + 2);
            }
            if (ok) warp_commit(el, bar_done);
            else if (lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutMma);
        }
    } else if (warp < 16) {
        const int part = warp >> 2, quad = warp & 3;
        const int m = quad * 32 + lane, r = r0 + m / G, h = g * G + m % G;
        const bool live = r < a.rows;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t* __restrict__ mrow =
            reinterpret_cast<const uint32_t*>(a.mask + (int64_t)b * a.key_tiles * a.row_pitch + (live ? r : 0)) + part;
        float l2 = 0.f, dl = 0.f;
        if (live) {
            const size_t at = ((size_t)b * a.Lq + a.q0 + r) * a.n_h + h;
            l2 = a.lse[at] * kLog2e;
            dl = a.delta[at];
        }
        uint32_t mk_next = live ? __ldg(mrow) : 0u;
        bool ok = true;
        for (int i = 0; i < n; ++i) {
            const uint32_t mk = mk_next;
            if (live && i + 1 < n) mk_next = __ldg(mrow + (int64_t)(i + 1) * a.row_pitch * 4);
            const uint32_t ts = lane_base + kTmS + 128 * (i & 1) + 32 * part, tp = lane_base + kTmP + 32 * part;
            if (!(ok = warp_wait(bar_s(i), (i >> 1) & 1, s_abort, a.wait_cycles))) break;
            uint32_t v[32], w[32], pk[16];
            tc_ld32(ts, v);
            tc_wait_ld32(v);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const float x = ex2_approx(fmaf(__uint_as_float(v[j]), a.scale_log2, -l2));
                v[j] = __float_as_uint((mk >> j) & 1u ? x : 0.f);
            }
            if (!(ok = warp_wait(bar_dp, i & 1, s_abort, a.wait_cycles))) break;
            tc_ld32(tp, w);
            tc_wait_ld32(w);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_read);
#pragma unroll
            for (int j = 0; j < 32; j += 2)
                pk[j / 2] = pack_bf16(__uint_as_float(v[j]) * (__uint_as_float(w[j]) - dl),
                                      __uint_as_float(v[j + 1]) * (__uint_as_float(w[j + 1]) - dl));
            tc_st16(ts, pk);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_ds);
        }
        ok = ok && warp_wait(bar_done, 0, s_abort, a.wait_cycles);
        if (!ok) {
            if (lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutEpi);
        } else {
            tc_fence_after();
            __nv_bfloat16* dst = a.dQ + (((size_t)b * a.Lq + a.q0 + (live ? r : 0)) * a.n_h + h) * DH + part * (DH / 4);
#pragma unroll
            for (int c = 0; c < DH / 64; ++c) {
                uint32_t o[16];
                tc_ld16(lane_base + kTmQ + part * (DH / 4) + 16 * c, o);
                tc_wait_ld16(o);
                if (!live) continue;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    uint32_t x[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        x[e] = pack_bf16(__uint_as_float(o[8 * q + 2 * e]) * a.scale, __uint_as_float(o[8 * q + 2 * e + 1]) * a.scale);
                    *reinterpret_cast<uint4*>(dst + 16 * c + 8 * q) = make_uint4(x[0], x[1], x[2], x[3]);
                }
            }
        }
    }
    tile_end(warp, lane, tmem, s_abort, bar_drain,
             [&] {
                 if (qd_issued) mbar_drain(bar_qd, 0);
                 for (int e = max(a.withhold_first, copies - SL); e < copies; ++e) mbar_drain(bar_full(e % SL), (e / SL) & 1);
             },
             [&] {
                 // (commits arrive in order: the last one of either kind covers the others)
                 if (k_released) mbar_drain(bar_empty((2 * (k_released - 1)) % SL), ((2 * (k_released - 1)) / SL) & 1);
                 if (v_released) mbar_drain(bar_empty((2 * v_released - 1) % SL), ((2 * v_released - 1) / SL) & 1);
             });
}

// ---- target of the indexer's loss: pbar --------------------------------------------------------------------------
template <int DH>
struct TargetSmem {
    using T = TileBytes<DH>;
    static constexpr int STAGES = 2;                               // (Q tile, two K tiles) of a KV head
    static constexpr int STAGE = 3 * T::TILE;
    static constexpr int OFF_BAR = STAGES * STAGE;
    static constexpr int N_BARS = 2 * STAGES + 4 + 4 + 1;
    static constexpr int OFF_TMEM = OFF_BAR + N_BARS * 8;
    static constexpr int OFF_ABORT = OFF_TMEM + 8;
    static constexpr int OFF_RANK = OFF_ABORT + 8;                 // first position of the key run in every query's set
    static constexpr int ALLOC = OFF_RANK + 128 * 4 + 1024;
};

template <int DH, int G>
__global__ void __launch_bounds__(kBwdThreads, 1)
gsa_masked_target_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const MaskedBwdArgs a) {
    chain_wait();
    using P = TargetSmem<DH>;
    using T = TileBytes<DH>;
    constexpr int QT = 128 / G;
    int timed_out;
    if (!tiles_allowed(a.dev_status, &timed_out)) return;
    // (runs of keys innermost, then row blocks, then batch elements, all along x: y and z end at 65535)
    const int run = (int)blockIdx.x % a.runs, rest = (int)blockIdx.x / a.runs;
    const int blk = a.row_blocks - 1 - rest % a.row_blocks, b = rest / a.row_blocks;
    const int r0 = blk * QT, off = a.Lk - a.Lq;
    const int ntiles = min((off + a.q0 + min(r0 + QT, a.rows) + kMaskTileKeys - 1) / kMaskTileKeys, a.key_tiles);
    const int pair0 = run * a.pairs_per_cta, pair1 = min(pair0 + a.pairs_per_cta, (ntiles + 1) / 2);
    if (pair0 >= pair1) return;
    const int n = (pair1 - pair0) * a.n_kv;                        // steps: (key pair, KV head)
    GSA_TILE_PROLOGUE(P)
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (2 + s); };
    auto bar_s = [&](int s, int w) { return bar0 + 8u * (4 + 2 * s + w); };
    auto bar_sfree = [&](int s, int w) { return bar0 + 8u * (8 + 2 * s + w); };
    const uint32_t bar_drain = bar0 + 8u * 12;
    int* const s_rank = reinterpret_cast<int*>(smem + P::OFF_RANK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1);
            for (int w = 0; w < 2; ++w) { mbar_init(bar_s(s, w), 1); mbar_init(bar_sfree(s, w), 8); }
        }
        mbar_init(bar_drain, 1);
    }
    // where the CTA's run of keys starts in every query's set: eight lanes a query, nine ways a step (one thread and two ways took
    // twelve memory latencies in front of every CTA's work)
    for (int q0 = 0; q0 < QT; q0 += kBwdThreads / 8) {
        const int q = q0 + (int)(threadIdx.x >> 3), l8 = lane & 7, r = r0 + q, first = pair0 * 2 * kMaskTileKeys;
        const bool in = q < QT && r < a.rows;
        const int64_t irow = in ? a.il.row(b, a.q0 + r) : 0;
        const int32_t* __restrict__ set = a.idx + irow * a.k_max;
        int lo = 0, hi = in && first > 0 ? clamp_budget(a.kt[irow], a.k_max) : 0;
        while (__any_sync(0xFFFFFFFFu, lo < hi)) {
            const int len = hi - lo;
            const bool narrow = len > 8;
            const int at = narrow ? lo + len * (l8 + 1) / 9 : lo + l8;
            const uint32_t votes = __ballot_sync(0xFFFFFFFFu, at < hi && set[at] < first);
            const int below = __popc((votes >> (lane & 24)) & 0xFFu);          // (ascending sets: the first `below` probes)
            if (narrow) {
                if (below < 8) hi = lo + len * (below + 1) / 9;
                if (below > 0) lo += len * below / 9 + 1;
            } else {
                lo += below;
                hi = lo;
            }
        }
        if (q < QT && l8 == 0) s_rank[q] = lo;
    }
    const uint32_t tmem = tile_start(timed_out, warp, sbase + P::OFF_TMEM, s_tmem, s_abort);
    int copies = 0, released = 0;

    // 640 threads launched at 96 registers: 512 * 104 + 128 * 64 = 61440
    if (warp < 16) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
        const int w = warp >> 3, half = (warp >> 2) & 1, quad = warp & 3;      // half of a key tile of the pair
        const int m = quad * 32 + lane, q = m / G, r = r0 + q;
        const bool live = r < a.rows;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
        const float* __restrict__ lse = a.lse + ((size_t)b * a.Lq + a.q0 + (live ? r : 0)) * a.n_h + m % G;
        float* __restrict__ dst = a.pbar + a.il.row(b, a.q0 + (live ? r : 0)) * a.k_max;
        const float inv_heads = 1.0f / (float)a.n_h;
        const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2);
        int rank = s_rank[q];
        bool ok = true;
        int it = 0;
        for (int pair = pair0; ok && pair < pair1; ++pair) {
            uint64_t acc[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = 0ull;
            float l_next = live ? lse[0] : 0.f;
            for (int g = 0; g < a.n_kv; ++g, ++it) {
                const int s = it & 1;
                const float neg = -l_next * kLog2e;
                if (live && g + 1 < a.n_kv) l_next = lse[(g + 1) * G];
                const uint64_t neg2 = pack_f32x2(neg, neg);
                if (!(ok = warp_wait(bar_s(s, w), (it >> 1) & 1, s_abort, a.wait_cycles))) break;
                const uint32_t ts = lane_base + 256 * s + 128 * w + 64 * half;
                uint32_t v[16];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    tc_ld16(ts + 16 * c, v);
                    tc_wait_ld16(v);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1])), scale2, neg2), x0, x1);
                        acc[8 * c + j] = add_f32x2(acc[8 * c + j], pack_f32x2(ex2_approx(x0), ex2_approx(x1)));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_sfree(s, w));
            }
            if (!ok) break;
            // sum over the heads of the group (neighbouring lanes), then to the set's positions; the group's lanes share the
            // columns.  The ranks run through both tiles of the pair.
            uint4 mk0 = make_uint4(0u, 0u, 0u, 0u), mk1 = mk0;
            if (live) {
                mk0 = a.mask[((int64_t)b * a.key_tiles + 2 * pair) * a.row_pitch + r];
                if (2 * pair + 1 < ntiles) mk1 = a.mask[((int64_t)b * a.key_tiles + 2 * pair + 1) * a.row_pitch + r];
            }
            const int n0 = __popc(mk0.x) + __popc(mk0.y), n1 = n0 + __popc(mk0.z) + __popc(mk0.w),
                      n2 = n1 + __popc(mk1.x) + __popc(mk1.y);
            const int at = rank + (w ? (half ? n2 : n1) : (half ? n0 : 0));
            const uint4 mk = w ? mk1 : mk0;
            const uint32_t words[2] = {half ? mk.z : mk.x, half ? mk.w : mk.y};
            rank += n2 + __popc(mk1.z) + __popc(mk1.w);
            // at every step a lane keeps every other pair of columns and gives its neighbour the rest
            auto halve = [&](int n, int bit) {
                const bool odd = (lane >> bit) & 1;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (j < n) {
                        const uint64_t keep = odd ? acc[2 * j + 1] : acc[2 * j], give = odd ? acc[2 * j] : acc[2 * j + 1];
                        acc[j] = add_f32x2(keep, __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)give, 1 << bit));
                    }
            };
            if constexpr (G >= 2) halve(16, 0);
            if constexpr (G >= 4) halve(8, 1);
            if constexpr (G >= 8) halve(4, 2);
            // pair j now stands for columns 2 c, 2 c + 1 with c = j G + the lane's bits
            const int at1 = at + __popc(words[0]);
#pragma unroll
            for (int j = 0; j < 32 / G; ++j) {
                const int c = j * G + m % G;                       // (j < 16 / G: in the first word)
                const uint32_t word = words[j / (16 / G)];
                const int bit = 2 * c & 31, p0 = (j < 16 / G ? at : at1) + __popc(word & ((1u << bit) - 1u));
                float x0, x1;
                unpack_f32x2(acc[j], x0, x1);
                const uint32_t sel = word >> bit;
                if (sel & 1u) dst[p0] = x0 * inv_heads;
                if (sel & 2u) dst[p0 + (sel & 1u)] = x1 * inv_heads;
            }
        }
        if (!ok && lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutEpi);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
        if (warp == kCopyWarp) {
            if (lane == 0) {
                bool ok = true;
                for (int it = 0; ok && it < n; ++it) {
                    const int s = it & 1, g = it % a.n_kv, pair = pair0 + it / a.n_kv;
                    if (!mbar_wait(bar_empty(s), ((it >> 1) & 1) ^ 1, s_abort, a.wait_cycles)) { ok = false; break; }
                    copies = it + 1;
                    if (it == 0 && a.withhold_first) continue;
                    mbar_expect_tx(bar_full(s), P::STAGE);
                    const uint32_t dst = sbase + s * P::STAGE;
                    for (int c = 0; c < T::CHUNKS; ++c) {
                        tma_load_tile(dst + c * T::CHUNK, &tm_q, c * 64, g * G, r0, b, bar_full(s));
                        for (int w = 0; w < 2; ++w)
                            tma_load_tile(dst + (1 + w) * T::TILE + c * T::CHUNK, &tm_k, c * 64, g, (2 * pair + w) * kMaskTileKeys, b,
                                          bar_full(s));
                    }
                }
                if (!ok) atomicCAS(a.dev_status, kDevOk, kDevTimeoutTma);
            }
        } else if (warp == kMmaWarp) {
            const uint32_t el = elect_lane();                      // (converged warp)
            bool ok = true;
            for (int it = 0; ok && it < n; ++it) {
                const int s = it & 1;
                if (!(ok = warp_wait(bar_full(s), (it >> 1) & 1, s_abort, a.wait_cycles))) break;
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    if (!(ok = warp_wait(bar_sfree(s, w), ((it >> 1) & 1) ^ 1, s_abort, a.wait_cycles))) break;
                    mma_kmajor<DH>(el, tmem + 256 * s + 128 * w, sbase + s * P::STAGE, sbase + s * P::STAGE + (1 + w) * T::TILE);
                    warp_commit(el, bar_s(s, w));
                }
                if (!ok) break;
                warp_commit(el, bar_empty(s));
                released = it + 1;
            }
            if (!ok && lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutMma);
        }
    }
    tile_end(warp, lane, tmem, s_abort, bar_drain,
             [&] { for (int i = max(a.withhold_first, copies - 2); i < copies; ++i) mbar_drain(bar_full(i & 1), (i >> 1) & 1); },
             [&] { for (int i = max(0, released - 2); i < released; ++i) mbar_drain(bar_empty(i & 1), (i >> 1) & 1); });
}

template <int DH, int G>
cudaError_t launch_bwd_t(const MaskedBwdArgs& a, const gsa_params_t& p, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                         const __nv_bfloat16* Vg, const __nv_bfloat16* dOs, cudaStream_t st) {
    CUtensorMap tq, td, tk, tv;
    KeysEndMaps end;
    auto keys_map = [&](CUtensorMap* tm, const void* x) { return make_heads_tmap(tm, x, p.B, p.Lk, p.Lk, p.n_kv, DH, kMaskTileKeys, 1); };
    if (!keys_map(&end.v, a.V) || !keys_map(&end.g2, a.g2) || !keys_map(&end.dk, a.dK) || !keys_map(&end.dv, a.dV) ||
        !keys_map(&end.dg2, a.dg2)) return cudaErrorUnknown;
    if (!make_heads_tmap(&tq, Q + (size_t)a.q0 * p.n_h * DH, p.B, p.Lq, a.rows, p.n_h, DH, 128 / G, G)) return cudaErrorUnknown;
    if (!make_heads_tmap(&td, dOs + (size_t)a.q0 * p.n_h * DH, p.B, p.Lq, a.rows, p.n_h, DH, 128 / G, G)) return cudaErrorUnknown;
    if (!keys_map(&tk, K) || !keys_map(&tv, Vg)) return cudaErrorUnknown;
    auto set_smem = [](auto kern, int bytes) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); };
    constexpr int kSmemK = KeysSmem<DH, G>::ALLOC, kSmemR = RowsSmem<DH>::ALLOC, kSmemT = TargetSmem<DH>::ALLOC;
    static_assert(kSmemK <= 232448 && kSmemR <= 232448 && kSmemT <= 232448, "shared memory of one CTA");
    // one wave of key tiles at most: two CTAs per tile (2 x 2051 keys, two KV heads: 68 tiles, 103 -> 65 us)
    const int key_ctas = a.key_tiles * p.n_kv * p.B, split = key_ctas <= sm_count() && a.row_blocks > 1 ? 2 : 1;
    cudaError_t e = split == 2 ? set_smem(gsa_masked_bwd_keys_kernel<DH, G, 2>, kSmemK) : set_smem(gsa_masked_bwd_keys_kernel<DH, G, 1>, kSmemK);
    if (e == cudaSuccess) e = set_smem(gsa_masked_bwd_rows_kernel<DH, G>, kSmemR);
    if (e == cudaSuccess) e = set_smem(gsa_masked_target_kernel<DH, G>, kSmemT);
    if (e != cudaSuccess) return e;
    if (split == 2)
        launch_chained_cluster(2, gsa_masked_bwd_keys_kernel<DH, G, 2>, (unsigned)(key_ctas * 2), kBwdThreads, kSmemK, st, tq, td, tk, tv, end, a);
    else
        launch_chained(gsa_masked_bwd_keys_kernel<DH, G, 1>, (unsigned)key_ctas, kBwdThreads, kSmemK, st, tq, td, tk, tv, end, a);
    launch_chained(gsa_masked_bwd_rows_kernel<DH, G>, (unsigned)(a.row_blocks * p.n_kv * p.B), kBwdThreads, kSmemR, st, tq, td, tk, tv, a);
    g_launches += 2;
    if (a.pbar) {
        launch_chained(gsa_masked_target_kernel<DH, G>, (unsigned)a.runs * (unsigned)a.row_blocks * (unsigned)p.B, kBwdThreads, kSmemT, st, tq, tk, a);
        ++g_launches;
    }
    return cudaGetLastError();
}

}  // namespace

namespace {
size_t sets_bytes(const gsa_params_t& p, const RowRange& rr) {           // the masks, or the inverted sets of the general path
    const size_t masks = mask_plan(p, rr.q_begin, rr.R).bytes(p.B), inv = attn_bwd_keys_general_bytes(p, rr.R);
    return ((masks > inv ? masks : inv) + 255) / 256 * 256;
}
}  // namespace

// then the statistics, for calls that have not saved them
size_t masked_bwd_bytes(const gsa_params_t& p, const RowRange& rr) {
    return sets_bytes(p, rr) + ((size_t)p.B * p.Lq * p.n_h * 4 + 255) / 256 * 256;
}

// Two models in microseconds, as in the forward (masked_rows_end).  Tiles: 1.7 + 1.45 + 1.05 (d_h = 64: 1.3 + 1.1 + 0.9) per
// 128 x 128 tile in the keys, rows and target kernels, one CTA per SM, 40 for the launches around them (the target is charged
// whether it is asked for or not; measured before the order of the CTAs and the results by TMA, now a tenth less).  Gather: 0.115 ps per byte of the K, V', Q and do rows that a pair moves (1.41 ns at 16
// heads of 128 on 8 KV heads, measured at L = 32K), 20 for its launches.  Fewer row tiles than half of the SMs: the gather.
namespace {
struct BackwardCosts { double tiles_us, pair_us, selected; };
BackwardCosts backward_costs(const gsa_params_t& p, const RowRange& rr) {
    const int G = p.n_h / p.n_kv, block = 128 / G;
    const double ctas = (double)((rr.R + block - 1) / block) * p.n_kv * rr.nb, sms = sm_count();
    if (2.0 * ctas < sms) return {1e30, 0.0, 0.0};
    const RowsWork w = rows_work(p, rr.nb, rr.q_begin, rr.R, block);
    const double all = w.key_tiles * p.n_kv / sms, row_tiles = (double)((rr.R + block - 1) / block);
    const double key_ctas = (double)((p.Lk + kMaskTileKeys - 1) / kMaskTileKeys) * p.n_kv * rr.nb;
    const double keys_chain = key_ctas <= sms ? 0.5 * row_tiles : row_tiles;
    const bool wide = p.d_h == 128;
    const double tiles = (all > keys_chain ? all : keys_chain) * (wide ? 1.7 : 1.3) + (all > w.chain ? all : w.chain) * (wide ? 1.45 : 1.1) +
                         all * (wide ? 1.05 : 0.9) + 40.0;
    return {tiles, 4.0 * (p.n_kv + p.n_h) * p.d_h * 0.115e-6, w.selected};
}
}  // namespace

bool masked_bwd_preferred(const gsa_params_t& p, const RowRange& rr) {
    const BackwardCosts c = backward_costs(p, rr);
    return c.tiles_us < c.selected * c.pair_us + 20.0;
}

cudaError_t launch_masked_bwd(const gsa_params_t& p, const RowRange& rr, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                              const __nv_bfloat16* V, const __nv_bfloat16* Vg, const __nv_bfloat16* g1, const __nv_bfloat16* g2,
                              const __nv_bfloat16* out, const __nv_bfloat16* dout, const int32_t* idx, const int32_t* kt,
                              IdxLayout il, __nv_bfloat16* dQ, __nv_bfloat16* dK, __nv_bfloat16* dV, __nv_bfloat16* dg1,
                              __nv_bfloat16* dg2, __nv_bfloat16* dOs, float* lse_ws, float* delta, float* pbar,
                              const float* lse_in, void* ws, int32_t* dev_status, cudaStream_t st) {
    int32_t* general = dev_status + kStatusGeneralWord;
    // (outside the sets the tiles multiply dP - delta, Q, K and do by zero: all of them have to be finite.  They are watched where
    // they are read or written first; rows of dOs past the range read as zero)
    cudaError_t e = launch_bwd_prep(p, rr, g1, out, dout, Q, dOs, dg1, delta, general, st);
    const MaskPlan mp = mask_plan(p, rr.q_begin, rr.R);
    uint4* mask = (uint4*)ws;
    // sets so small that the gather, in the form that stands behind the tiles, takes less than seven tenths of their time
    const BackwardCosts costs = backward_costs(p, rr);
    const double few_pairs = (0.7 * costs.tiles_us - 20.0) / (1.15 * costs.pair_us);
    if (e == cudaSuccess) e = launch_build_masks(p, mp, masked_block_rows(p), idx, kt, il, mask, dev_status, few_pairs, st);
    if (e == cudaSuccess && !lse_in) {
        // the statistics were not saved: the forward's tiles once more (their output goes where dQ is written afterwards)
        float* const stats = (float*)((char*)ws + sets_bytes(p, rr));
        e = launch_masked_attn_fwd(p, mp, mask, Q, K, Vg, g1, dQ, stats, dev_status, st);
        if (e == cudaSuccess) e = launch_attn_direct(p, rr, Q, K, Vg, g1, idx, kt, il, dQ, stats, general, kRunAnyGeneral, st);
        lse_in = stats;
    }
    if (e != cudaSuccess) return e;
    MaskedBwdArgs a;
    a.mask = mask; a.lse = lse_in; a.delta = delta; a.V = V; a.g2 = g2; a.idx = idx; a.kt = kt; a.il = il;
    a.dQ = dQ; a.dK = dK; a.dV = dV; a.dg2 = dg2; a.pbar = pbar; a.dev_status = dev_status; a.general = general;
    a.q0 = mp.q0; a.rows = mp.rows; a.row_pitch = mp.row_pitch; a.key_tiles = mp.key_tiles;
    a.B = p.B; a.Lq = p.Lq; a.Lk = p.Lk; a.n_h = p.n_h; a.n_kv = p.n_kv; a.k_max = p.k_max;
    const int G = p.n_h / p.n_kv;
    a.row_blocks = (mp.rows + 128 / G - 1) / (128 / G);
    a.abreast_keys = pairs_abreast(p.n_kv * p.B, 4.0 * p.Lq * p.d_h * G);        // (Q and do of a pair's heads)
    a.abreast_rows = pairs_abreast(p.n_kv * p.B, 4.0 * p.Lk * p.d_h);            // (K and V')
    // target kernel: runs of key pairs long enough to pay for a CTA's start, short enough for four CTAs per SM (visible pairs
    // only: half of them in a square range)
    const int64_t pairs = (int64_t)((a.key_tiles + 1) / 2) * a.row_blocks * p.B;
    a.pairs_per_cta = (int)(pairs / 2 / (4 * sm_count()));
    a.pairs_per_cta = a.pairs_per_cta < 1 ? 1 : (a.pairs_per_cta > 8 ? 8 : a.pairs_per_cta);
    a.runs = ((a.key_tiles + 1) / 2 + a.pairs_per_cta - 1) / a.pairs_per_cta;
    a.scale = p.sm_scale > 0.f ? p.sm_scale : 1.0f / sqrtf((float)p.d_h);
    a.scale_log2 = a.scale * kLog2e;
    a.wait_cycles = wait_limit_cycles();
    a.withhold_first = withhold_first_copy() ? 1 : 0;
    a.zero = (uint4*)ws; a.zero_vec = (int64_t)(attn_bwd_keys_general_zero(p, rr.R) / 16);
    e = cudaErrorInvalidValue;
#define GSA_CASE(DH_, G_) if (p.d_h == DH_ && G == G_) e = launch_bwd_t<DH_, G_>(a, p, Q, K, Vg, dOs, st)
    GSA_CASE(128, 1); GSA_CASE(128, 2); GSA_CASE(128, 4); GSA_CASE(128, 8);
    GSA_CASE(64, 1); GSA_CASE(64, 2); GSA_CASE(64, 4); GSA_CASE(64, 8);
#undef GSA_CASE
    if (e == cudaSuccess) e = launch_attn_bwd_rows_general(p, rr, Q, K, Vg, dOs, idx, kt, il, dQ, lse_ws, delta, pbar, lse_in, general, st);
    if (e == cudaSuccess)
        e = launch_attn_bwd_keys_general(p, rr, Q, dOs, K, V, Vg, g2, lse_ws, delta, idx, kt, il, ws, dK, dV, dg2, general, st);
    return e;
}

}  // namespace gsa
