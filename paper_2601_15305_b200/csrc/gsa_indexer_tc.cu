// Gated lightning indexer (Eq. 7) on the 5th-generation tensor cores.
//
//   D[s, (t, j)] = k^I[s, :] . q^I[t, j, :]         tcgen05.mma, bf16 x bf16 -> fp32 in TMEM
//   I[t, s]      = sum_j w[t, j] * sigmoid(D[s, (t, j)] + b_j)      epilogue, in registers
//
// Orientation: keys are the M dimension (128 per tile = the 128 TMEM lanes), the N dimension is
// (query, indexer head) flattened, 256 columns = 256/H^I queries.  A thread of the epilogue owns
// one key: it reads that key's 256 accumulators, sums the H^I adjacent columns of each query
// after the sigmoid, and consecutive lanes write consecutive s of a score row (128-byte stores).
//
// One CTA per SM, each with the same number of (query group, key tile) pairs at or below the diagonal (tiles above it are never
// touched): the pairs are numbered group by group and a CTA takes a run of them, which crosses from one group into the next where
// it has to.  (CTAs of up to 64 tiles of one group, late groups first, left SMs idle at the end: 8K prefill 110 us.)
// Warp roles: warp 0 feeds shared memory by TMA (k^I tiles through a ring of stages, the q^I tile of every group of the run),
// warp 1 issues the MMAs and owns the TMEM allocation, warps 2..17 are the epilogue.  Two 256-column accumulators alternate, so the MMAs of tile i+1
// overlap the epilogue of tile i; the epilogue (exp2 + reciprocal per sigmoid on the
// special-function unit) is the longer of the two, which is why it gets sixteen warps (four per
// scheduler), each reading its 64 columns 16 at a time.
//
// Every mbarrier wait is bounded: when a wait runs out the CTA records it in the status word,
// stops issuing work, drains what it has in flight and exits with its TMEM released.
#include "gsa_common.cuh"
#include "gsa_tc.cuh"

namespace gsa {

namespace {

constexpr int kTileKeys = 128;
constexpr int kNCols = 256;            // N of one MMA = (queries x heads) of a group
constexpr int kStages = 6;
constexpr int kEpiWarps = 16;          // 4 per scheduler: keeps the special-function unit fed
constexpr int kThreads = 64 + kEpiWarps * 32;
constexpr int kColsPerWarp = kNCols / (kEpiWarps / 4);   // accumulator columns one epilogue warp handles
constexpr int kChunkCols = 16;         // columns per tcgen05.ld

struct TcArgs {
    const float* w;
    const float* bI;
    float* scores;
    int64_t row_stride;
    int32_t* dev_status;
    RowRange rr;
    int32_t Lq, Lk;
    int32_t groups_per_batch;
    int64_t tiles_per_batch;       // (query group, key tile) pairs of a batch element, and of the call
    int64_t tiles;
    long long wait_cycles;         // limit of every bounded wait
    int32_t withhold_q;            // fault injection: the q^I copy is left out, so its barrier is never completed
};

template <int DI>
struct SmemPlan {
    static constexpr int Q_BYTES = kNCols * DI * 2;
    static constexpr int K_BYTES = kTileKeys * DI * 2;
    static constexpr int OFF_Q = 0;
    static constexpr int OFF_K = OFF_Q + 2 * Q_BYTES;             // (two groups' q^I tiles in turn)
    static constexpr int OFF_W = OFF_K + kStages * K_BYTES;
    static constexpr int OFF_B = OFF_W + kEpiWarps * kColsPerWarp * 4;
    static constexpr int OFF_BAR = OFF_B + 64;                    // 8-byte aligned
    static constexpr int N_BARS = 2 * kStages + 4 + 4 + 1;
    static constexpr int OFF_TMEM = OFF_BAR + N_BARS * 8;
    static constexpr int OFF_ABORT = OFF_TMEM + 8;
    static constexpr int TOTAL = OFF_ABORT + 8;
    static constexpr int ALLOC = TOTAL + 1024;                    // slack to align the base to 1024
};

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// sum_j w_j * sigmoid(x_j + b_j) over HI heads, with one reciprocal per group of up to four heads:
//   w1/a1 + w2/a2 = (w1 a2 + w2 a1) / (a1 a2),   a_j = 1 + 2^(-(x_j + b_j) log2 e).
// The exponent is clamped at 28 (sigmoid < 4e-9 there), so a product of four a_j stays below
// 2^116 and cannot overflow.  nb[j] = -b_j log2 e.
// The epilogue is bound by instruction issue, so for four and eight heads the arithmetic runs on the
// packed fp32 instructions of sm_100 (two values per instruction).  Adjacent heads (2i, 2i+1) share a
// register pair; the tree combines head 2i with 2i+2 and 2i+1 with 2i+3 (elementwise on the pairs), then,
// for eight heads, those with their counterparts four heads on: the even and the odd heads end up as one
// quotient each (four factors per denominator), and one more step joins the two under a single reciprocal:
// the special-function unit, which bounds this kernel, then sees nine operations per eight sigmoids.  To keep
// a product of eight factors inside fp32, the a_j of eight heads are carried scaled by 2^-12 (the offset
// rides in the exponent's bias term and in the added constant; exponent clamped at 27: sigmoid < 8e-9), so
// each lies in [2^-12, 2^15], the product of eight in [2^-96, 2^120] and a head's numerator term within
// w_j 2^-96 .. 2^96: nothing overflows and only weights below 2^-30 could be flushed.  The 2^-12 left over
// per quotient is folded into the weights, which the caller passes pre-scaled (kWeightScale).
// 37 issue slots per eight sigmoids instead of 54.
// RELU: sum_j w_j * max(x_j + b_j, 0) (Eq. 3), nb[j] = b_j; no special-function work at all.
template <int HI> constexpr float kOne = HI == 8 ? 2.44140625e-04f : 1.0f;             // 2^-12 : 1
template <int HI> constexpr float kExpClamp = HI == 8 ? 15.0f : 28.0f;                 // 27 - 12 : 28
template <int HI> constexpr float kExpBias = HI == 8 ? -12.0f : 0.0f;                  // added to nb[j] by the caller
template <int HI> constexpr float kWeightScale = HI == 8 ? 2.44140625e-04f : 1.0f;     // applied to w[j] by the caller

template <int HI, bool RELU>
__device__ __forceinline__ float gated_head_sum(const uint32_t* x, const float* w, const float (&nb)[HI]) {
    if constexpr (RELU) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < HI; ++j) acc = fmaf(w[j], fmaxf(__uint_as_float(x[j]) + nb[j], 0.f), acc);
        return acc;
    }
    if constexpr (HI >= 4) {
        constexpr int NP = HI / 2;
        const float2 kScale = make_float2(-1.4426950408889634f, -1.4426950408889634f), kOne2 = make_float2(kOne<HI>, kOne<HI>);
        float2 a2[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 y = __ffma2_rn(make_float2(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])), kScale,
                                        make_float2(nb[2 * i], nb[2 * i + 1]));
            a2[i] = __fadd2_rn(make_float2(ex2_approx(fminf(y.x, kExpClamp<HI>)), ex2_approx(fminf(y.y, kExpClamp<HI>))), kOne2);
        }
        // heads (0,1) with (2,3) [and (4,5) with (6,7)]: numerators and denominators of the pairs (0,2), (1,3)
        float2 n2[NP / 2], d2[NP / 2];
#pragma unroll
        for (int q = 0; q < NP / 2; ++q) {
            const float2 wp = make_float2(w[4 * q], w[4 * q + 1]), wq = make_float2(w[4 * q + 2], w[4 * q + 3]);
            n2[q] = __ffma2_rn(wp, a2[2 * q + 1], __fmul2_rn(wq, a2[2 * q]));
            d2[q] = __fmul2_rn(a2[2 * q], a2[2 * q + 1]);
        }
        if constexpr (HI == 8) {
            const float2 nc = __ffma2_rn(n2[0], d2[1], __fmul2_rn(n2[1], d2[0]));     // even heads | odd heads
            const float2 dc = __fmul2_rn(d2[0], d2[1]);
            return fmaf(nc.x, dc.y, nc.y * dc.x) * rcp_approx(dc.x * dc.y);
        } else {
            return fmaf(n2[0].x, d2[0].y, n2[0].y * d2[0].x) * rcp_approx(d2[0].x * d2[0].y);
        }
    } else {
        float a[HI];
#pragma unroll
        for (int j = 0; j < HI; ++j)
            a[j] = 1.0f + ex2_approx(fminf(fmaf(__uint_as_float(x[j]), -1.4426950408889634f, nb[j]), 28.0f));
        if constexpr (HI == 2) return fmaf(w[0], a[1], w[1] * a[0]) * rcp_approx(a[0] * a[1]);
        else return w[0] * rcp_approx(a[0]);
    }
}

// Key tiles that the query groups of a batch element see.  A group of NQ rows has `off + its rows so far` visible keys at its last row.
struct TileCount {
    int32_t off, R, NQ;                    // keys in front of the first row; rows; rows of a group
    __host__ __device__ int of(int g) const {                                // group g's tiles
        const int rows = (g + 1) * NQ < R ? (g + 1) * NQ : R;
        return (off + rows + kTileKeys - 1) / kTileKeys;
    }
    // tiles of the groups before g: the sum of ceil((off + NQ j) / 128) over j = 1 .. g (none of these is cut off at R)
    __host__ __device__ int64_t before(int g) const {
        if (NQ >= kTileKeys) return (int64_t)g * ((off + kTileKeys - 1) / kTileKeys) + (int64_t)(NQ / kTileKeys) * g * (g + 1) / 2;
        // with off = 128 a + rest: ceil((rest + NQ j) / 128) = ceil((ceil(rest / NQ) + j) / r), r = 128 / NQ
        const int a = off / kTileKeys, beta = (off % kTileKeys + NQ - 1) / NQ, r = kTileKeys / NQ;
        auto u = [r](int64_t n) { const int64_t q = n / r; return r * q * (q + 1) / 2 + (n % r) * (q + 1); };   // sum of ceil(m / r), m <= n
        return (int64_t)g * a + u(beta + g) - u(beta);
    }
};

// instruction descriptor: D fp32, A = B = bf16, both K-major, M = 128, N = 256
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kNCols >> 3) << 17) |
                            ((uint32_t)(kTileKeys >> 4) << 24);

template <int DI, int HI, bool RELU>
__global__ void __launch_bounds__(kThreads, 1)
gsa_indexer_tc_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_q,
                      const TcArgs a) {
    chain_wait();
    using P = SmemPlan<DI>;
    constexpr int NQ = kNCols / HI;             // queries per group
    constexpr int KSTEPS = DI / 16;
    constexpr int ROW_BYTES = DI * 2;

    // ---- which work is mine: pairs first .. last - 1 ----------------------------------------------------
    const int off = a.Lk - a.Lq;
    const TileCount count{off + a.rr.q_begin, a.rr.R, NQ};
    const int64_t first = a.tiles * blockIdx.x / gridDim.x, last = a.tiles * (blockIdx.x + 1) / gridDim.x;
    const int64_t in_batch = first % a.tiles_per_batch;
    int g_first = 0;                                                  // the group of the first pair
    for (int lo = 0, hi = a.groups_per_batch - 1; lo <= hi;) {
        const int mid = (lo + hi) >> 1;
        if (count.before(mid) <= in_batch) { g_first = mid; lo = mid + 1; } else hi = mid - 1;
    }
    // the run, group by group: f(segment, batch element, first row of the group from q_begin, its rows, first key tile, key tiles)
    auto for_segments = [&](auto f) {
        int64_t left = last - first;
        int tile0 = (int)(in_batch - count.before(g_first)), g = g_first, bl = (int)(first / a.tiles_per_batch);
        for (int seg = 0; left > 0; ++seg) {
            const int n = (int)min((int64_t)(count.of(g) - tile0), left);
            if (!f(seg, bl, g * NQ, min(NQ, a.rr.R - g * NQ), tile0, n)) break;
            left -= n;
            tile0 = 0;
            if (++g == a.groups_per_batch) { g = 0; ++bl; }
        }
    };
    {   // an earlier CTA gave up: leave, all threads together (one thread reads the word)
        __shared__ int s_go;
        if (threadIdx.x == 0) s_go = *reinterpret_cast<volatile int32_t*>(a.dev_status) == kDevOk;
        __syncthreads();
        if (!s_go) return;
    }

    extern __shared__ unsigned char dyn_smem_raw[];
    const uint32_t raw_u32 = smem_u32(dyn_smem_raw);
    const uint32_t pad = (1024u - (raw_u32 & 1023u)) & 1023u;
    unsigned char* smem = dyn_smem_raw + pad;
    const uint32_t sbase = raw_u32 + pad;

    float* s_w0 = reinterpret_cast<float*>(smem + P::OFF_W);
    float* s_b = reinterpret_cast<float*>(smem + P::OFF_B);
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + P::OFF_TMEM);
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem + P::OFF_ABORT);
    const uint32_t bar0 = sbase + P::OFF_BAR;
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (kStages + s); };
    auto bar_q = [&](int i) { return bar0 + 8u * (2 * kStages + i); };
    auto bar_qempty = [&](int i) { return bar0 + 8u * (2 * kStages + 2 + i); };
    auto bar_tfull = [&](int i) { return bar0 + 8u * (2 * kStages + 4 + i); };
    auto bar_tempty = [&](int i) { return bar0 + 8u * (2 * kStages + 6 + i); };
    const uint32_t bar_drain = bar0 + 8u * (2 * kStages + 8);         // give-up path only

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(bar_q(i), 1); mbar_init(bar_qempty(i), 1); mbar_init(bar_tfull(i), 1); mbar_init(bar_tempty(i), kEpiWarps); }
        mbar_init(bar_drain, 1);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(sbase + P::OFF_TMEM)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x < 8) s_b[threadIdx.x] = (a.bI && threadIdx.x < HI) ? a.bI[threadIdx.x] : 0.f;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *s_tmem;
    // what this thread has put in flight (the copy producer's and the MMA issuer's own counts)
    int copies_issued = 0, mma_tiles_issued = 0, q_issued = 0, q_released = 0;

    if (warp == 0) {
        // ================= TMA producer =======================================================
        if (lane == 0) {
            bool ok = true;
            for_segments([&](int seg, int bl, int tr0, int, int tile0, int ntiles) {
                const int b = a.rr.b0 + bl;
                if (!(ok = mbar_wait(bar_qempty(seg & 1), ((seg >> 1) & 1) ^ 1, s_abort, a.wait_cycles))) return false;
                if (!a.withhold_q) {
                    mbar_expect_tx(bar_q(seg & 1), P::Q_BYTES);
                    tma_load_2d(sbase + P::OFF_Q + (seg & 1) * P::Q_BYTES, &tm_q, 0, (b * a.Lq + a.rr.q_begin + tr0) * HI, bar_q(seg & 1));
                    q_issued = seg + 1;
                }
                for (int i = 0; i < ntiles; ++i) {
                    const int s = copies_issued % kStages;
                    if (!(ok = !*s_abort && mbar_wait(bar_empty(s), ((copies_issued / kStages) & 1) ^ 1, s_abort, a.wait_cycles))) return false;
                    mbar_expect_tx(bar_full(s), P::K_BYTES);
                    tma_load_2d(sbase + P::OFF_K + s * P::K_BYTES, &tm_k, 0, b * a.Lk + (tile0 + i) * kTileKeys, bar_full(s));
                    ++copies_issued;
                }
                return true;
            });
            if (!ok) atomicCAS(a.dev_status, kDevOk, kDevTimeoutTma);
        }
    } else if (warp == 1) {
        // ================= MMA issuer =========================================================
        if (lane == 0) {
            bool ok = true;
            for_segments([&](int seg, int, int, int, int, int ntiles) {
                if (!(ok = mbar_wait(bar_q(seg & 1), (seg >> 1) & 1, s_abort, a.wait_cycles))) return false;
                const uint64_t bdesc = make_kmajor_desc<ROW_BYTES>(sbase + P::OFF_Q + (seg & 1) * P::Q_BYTES);
                for (int i = 0; i < ntiles; ++i) {
                    const int n = mma_tiles_issued, s = n % kStages, buf = n & 1;
                    if (!(ok = mbar_wait(bar_tempty(buf), ((n >> 1) & 1) ^ 1, s_abort, a.wait_cycles))) return false;
                    if (!(ok = mbar_wait(bar_full(s), (n / kStages) & 1, s_abort, a.wait_cycles))) return false;
                    tc_fence_after();
                    const uint64_t adesc = make_kmajor_desc<ROW_BYTES>(sbase + P::OFF_K + s * P::K_BYTES);
#pragma unroll
                    for (int k = 0; k < KSTEPS; ++k)       // 16 K-elements = 32 bytes = 2 descriptor units
                        tc_mma_bf16(tmem_base + buf * kNCols, adesc + 2 * k, bdesc + 2 * k, kIdesc, k > 0);
                    tc_commit(bar_empty(s));               // stage reusable once these MMAs have read it
                    tc_commit(bar_tfull(buf));             // accumulator ready for the epilogue
                    mma_tiles_issued = n + 1;
                }
                tc_commit(bar_qempty(seg & 1));
                q_released = seg + 1;
                return true;
            });
            if (!ok) atomicCAS(a.dev_status, kDevOk, kDevTimeoutMma);
        }
    } else {
        // ================= epilogue: sigmoid, head weights, head sum, store ===================
        const int ew = warp - 2;
        const int quad = warp & 3;                          // TMEM lanes this warp may touch: 32*quad ..
        const int part = ew >> 2;                           // which kColsPerWarp of the 256 columns
        constexpr int QPC = kChunkCols / HI;                // queries per 16-column chunk
        constexpr int NCHUNK = kColsPerWarp / kChunkCols;
        float bias[HI];
#pragma unroll
        for (int j = 0; j < HI; ++j) bias[j] = RELU ? s_b[j] : fmaf(s_b[j], -1.4426950408889634f, kExpBias<HI>);
        // this warp's columns of the group's weights; eight heads' are scaled by the power of two that the head sum leaves over
        float* const s_w = s_w0 + ew * kColsPerWarp;
        int it = 0;
        for_segments([&](int, int bl, int tr0, int nq, int tile0, int ntiles) {
            __syncwarp();
            for (int e = lane; e < kColsPerWarp; e += 32) {
                const int qi = (part * kColsPerWarp + e) / HI;
                s_w[e] = qi < nq ? a.w[((size_t)(a.rr.b0 + bl) * a.Lq + a.rr.q_begin + tr0 + qi) * HI + e % HI] * (RELU ? 1.0f : kWeightScale<HI>)
                                 : 0.f;
            }
            __syncwarp();
            for (int i = 0; i < ntiles; ++i, ++it) {
                const int buf = it & 1;
                if (!__all_sync(0xFFFFFFFFu, mbar_wait(bar_tfull(buf), (it >> 1) & 1, s_abort, a.wait_cycles))) {
                    if (lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutEpi);
                    return false;
                }
                tc_fence_after();
                const int s = (tile0 + i) * kTileKeys + quad * 32 + lane;
                const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + buf * kNCols + part * kColsPerWarp;
                // columns are read 16 at a time, the next chunk's load in flight behind the current
                // chunk's arithmetic
                float* const out_col = a.scores + ((int64_t)bl * a.rr.R + tr0) * a.row_stride + s;
                auto do_chunk = [&](const uint32_t (&r)[kChunkCols], int c) {
                    const int q_first = (part * kColsPerWarp + c * kChunkCols) / HI;
#pragma unroll
                    for (int qq = 0; qq < QPC; ++qq) {
                        const int qi = q_first + qq;
                        const float* const w = s_w + (c * QPC + qq) * HI;
                        float wv[HI];
                        if constexpr (HI >= 4) {
#pragma unroll
                            for (int j = 0; j < HI; j += 4) {
                                const float4 v = *reinterpret_cast<const float4*>(w + j);
                                wv[j] = v.x; wv[j + 1] = v.y; wv[j + 2] = v.z; wv[j + 3] = v.w;
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < HI; ++j) wv[j] = w[j];
                        }
                        const float acc = gated_head_sum<HI, RELU>(&r[qq * HI], wv, bias);
                        if (qi < nq && s <= off + a.rr.q_begin + tr0 + qi) out_col[(int64_t)qi * a.row_stride] = acc;
                    }
                };
                uint32_t ra[kChunkCols], rb[kChunkCols];
                tc_ld16(taddr, ra);
#pragma unroll
                for (int c = 0; c < NCHUNK; c += 2) {
                    tc_wait_ld16(ra);
                    tc_ld16(taddr + (c + 1) * kChunkCols, rb);
                    do_chunk(ra, c);
                    tc_wait_ld16(rb);
                    if (c + 2 < NCHUNK) tc_ld16(taddr + (c + 2) * kChunkCols, ra);
                    do_chunk(rb, c + 1);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_tempty(buf));
            }
            return true;
        });
    }

    tc_fence_before();
    __syncthreads();
    if (*s_abort) {
        // Give-up path.  Every role has left its loop, but what was issued before is still under way: copies
        // land in this CTA's stages, MMAs read them and write its TMEM, commits arrive on its barriers.  None
        // of that may outlive the CTA, whose TMEM and shared memory go to the next one.  All of it completes by
        // itself (nothing issued waits for anything that was not), so these polls end; each is bounded anyway.
        if (warp == 0 && lane == 0) {
            for (int i = max(0, q_issued - 2); i < q_issued; ++i) mbar_drain(bar_q(i & 1), (i >> 1) & 1);
            for (int i = max(0, copies_issued - kStages); i < copies_issued; ++i)
                mbar_drain(bar_full(i % kStages), (i / kStages) & 1);
        }
        if (warp == 1 && lane == 0) {
            tc_commit(bar_drain);                          // arrives once every MMA issued so far has completed
            mbar_drain(bar_drain, 0);
            for (int i = max(0, mma_tiles_issued - kStages); i < mma_tiles_issued; ++i)
                mbar_drain(bar_empty(i % kStages), (i / kStages) & 1);
            for (int i = max(0, mma_tiles_issued - 2); i < mma_tiles_issued; ++i)
                mbar_drain(bar_tfull(i & 1), (i >> 1) & 1);
            for (int i = max(0, q_released - 2); i < q_released; ++i) mbar_drain(bar_qempty(i & 1), (i >> 1) & 1);
        }
        tc_fence_before();
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
}

template <int DI, int HI, bool RELU>
cudaError_t launch_t(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* qI, const __nv_bfloat16* kI,
                     const float* w, const float* bI, float* scores, int64_t row_stride, int32_t* dev_status,
                     cudaStream_t st) {
    using P = SmemPlan<DI>;
    constexpr int NQ = kNCols / HI;
    CUtensorMap tm_k, tm_q;
    if (!make_rows_tmap(&tm_k, kI, (uint64_t)p.B * p.Lk, DI, kTileKeys)) return cudaErrorUnknown;
    if (!make_rows_tmap(&tm_q, qI, (uint64_t)p.B * p.Lq * HI, DI, kNCols)) return cudaErrorUnknown;

    TcArgs a;
    a.w = w; a.bI = bI; a.scores = scores; a.row_stride = row_stride; a.dev_status = dev_status;
    a.rr = rr; a.Lq = p.Lq; a.Lk = p.Lk;
    a.groups_per_batch = (rr.R + NQ - 1) / NQ;
    const TileCount count{p.Lk - p.Lq + rr.q_begin, rr.R, NQ};
    a.tiles_per_batch = count.before(a.groups_per_batch - 1) + count.of(a.groups_per_batch - 1);
    a.tiles = a.tiles_per_batch * rr.nb;
    a.wait_cycles = wait_limit_cycles();
    a.withhold_q = withhold_first_copy() ? 1 : 0;
    const unsigned grid = (unsigned)(a.tiles < sm_count() ? a.tiles : sm_count());

    // one CTA per SM: the kernel allocates all 512 TMEM columns, so a second resident CTA would
    // only sit in tcgen05.alloc until the first one leaves
    constexpr int kSmem = P::ALLOC > 120 * 1024 ? P::ALLOC : 120 * 1024;
    auto kern = gsa_indexer_tc_kernel<DI, HI, RELU>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    launch_chained(kern, grid, kThreads, kSmem, st, tm_k, tm_q, a);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace

bool indexer_tc_supported(const gsa_params_t& p) {
    if (!(p.dI == 64 || p.dI == 32)) return false;
    if (!(p.HI == 1 || p.HI == 2 || p.HI == 4 || p.HI == 8)) return false;
    if ((int64_t)p.B * p.Lq * p.HI >= (1ll << 31) || (int64_t)p.B * p.Lk >= (1ll << 31)) return false;
    return get_encode_fn() != nullptr;
}

cudaError_t launch_indexer_tc(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* qI,
                              const __nv_bfloat16* kI, const float* w, const float* bI, float* scores,
                              int64_t row_stride, int32_t* dev_status, cudaStream_t st) {
    if (rr.rows() <= 0) return cudaSuccess;
#define GSA_TC_CASE(DI_, HI_) \
    if (p.dI == DI_ && p.HI == HI_) \
        return p.act == 1 ? launch_t<DI_, HI_, true>(p, rr, qI, kI, w, bI, scores, row_stride, dev_status, st) \
                          : launch_t<DI_, HI_, false>(p, rr, qI, kI, w, bI, scores, row_stride, dev_status, st)
    GSA_TC_CASE(64, 8); GSA_TC_CASE(64, 4); GSA_TC_CASE(64, 2); GSA_TC_CASE(64, 1);
    GSA_TC_CASE(32, 8); GSA_TC_CASE(32, 4); GSA_TC_CASE(32, 2); GSA_TC_CASE(32, 1);
#undef GSA_TC_CASE
    return cudaErrorInvalidValue;
}

}  // namespace gsa
