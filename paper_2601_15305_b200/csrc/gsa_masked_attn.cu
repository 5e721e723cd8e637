// Sparse gated attention forward (Eq. 9, 11, 12, 10) on masked dense tiles (see gsa_masked.cuh): for index sets that
// hold more than a few per cent of the visible keys.
//
// One CTA = one KV head and 256 rows, a row being a (query, head of the group) pair: two M = 128 tiles whose chains
//     S = Q K^T (tcgen05, fp32 in TMEM) -> mask, softmax numerators P (registers) -> P as bf16 into the columns of S
//     -> O += P V' (tcgen05, A operand in TMEM, V' tile read as it lies: keys are the contraction, d runs along N)
// run against each other, by halves of 64 keys: while a half's numerators are made, the tensor cores take in the other halves' and
// score the same half of the next tile behind each product.  A K and a V' tile are fetched once for both.  Thread = row: no
// shuffles anywhere.
//
// Softmax reference: it moves only when the numerators' sum shows that a selected score may exceed it by more than 2^8, so the
// accumulator in TMEM is touched by the softmax warps on a row's first tiles only.  Masked scores are replaced by
// -inf before the exponentials; fp32 everywhere except P (bf16, as in the gather kernel).  The reference is
// set a little above the maximum it is taken from: that maximum may come from very few keys (a row of 50K keys has three selected
// ones in its first tile), and where scores are nearly flat half of the row's numerators would then lie just above 1, where bf16
// is half as fine as just below.  Error of the output against fp64, chunk of 2003 rows at 50021 keys: 2.78e-3 without the margin,
// 2.62e-3 with it, 2.64e-3 in the gather kernel; 50 prefill, chunk, dense and training shapes: 0.995 of the gather's on average.
//
// Bound: the tensor pipe and the hand-overs around it.  Per pair of tiles 3270-3390 cycles (a softmax warp: 1790 at the numerators, 490
// to hand them over, 750 waiting); the products count 2560 of them, for one of N = 64 out of shared memory takes 48 cycles a step of
// 16 (its A operand alone is 4 KB), not the 32 of its arithmetic.  Whole tiles, with the next scores only behind both halves' product,
// took 3600, 1500 of it in that wait.  A CTA costs 0.7 us of setup, 1.5 to its first scores and about 2 at its end (8.7 while gates
// and output went row by row).  Measured at 16 heads of 128 on 8 KV heads: 8K 247 us (319 before the order of tile_order and the halves,
// the gather kernel 4.6 ms), dense 2 x 3072 100 us (135), L = 32K 3.27 to 3.37 ms = 1.30 to 1.34 PFLOP/s over the visible pairs, at the power limit (3.41;
// the gather 19.6 ms).  Slower: four softmax warpgroups, a row's halves on two threads (8K 295 us); a share of the exponentials on
// the FMA pipe (every fourth pair 250 against 252 at 8K, 3.34 against 3.28 ms at 32K; every second 280).
//
// Warps 0-3 / 4-7: softmax and epilogue of tile 0 / 1; warp 8: TMA; warp 9: MMA issue and TMEM allocation; 10, 11
// only complete their warpgroup.
// TMEM: S0 | S1 (128 columns each, 64 of a half; a half's P overlays its first 32) | O0 | O1.
#include "gsa_masked.cuh"

namespace gsa {

namespace {

// ---- masks -----------------------------------------------------------------------------------------------
constexpr int kMaskWindowWords = 1024;                 // 32768 keys of every row at a time
constexpr int kPairsBits = 36;                         // (4 bytes an entry: 2^36 pairs would be 275 GB of sets)
constexpr int kMaskRowWords = kMaskWindowWords + 4;    // (padded: the rows' pieces of a key tile fall into different banks)

__global__ void __launch_bounds__(kMaskRowAlign * 32)
gsa_build_masks_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ kt, uint4* __restrict__ mask,
                       IdxLayout il, int q0, int rows, int row_pitch, int key_tiles, int block_rows, int k_max, int off,
                       int32_t* dev_status, unsigned long long few_pairs) {
    chain_wait();
    int32_t* const general = dev_status + kStatusGeneralWord;
    __shared__ __align__(16) uint32_t s_bits[kMaskRowAlign * kMaskRowWords];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row_ctas = row_pitch / kMaskRowAlign;      // (batch elements along x: y and z end at 65535)
    const int b = blockIdx.x / row_ctas, r0 = blockIdx.x % row_ctas * kMaskRowAlign, r = r0 + warp;
    const int blk_end = min((r0 / block_rows + 1) * block_rows, rows);
    const int tiles = min((off + q0 + blk_end + kMaskTileKeys - 1) / kMaskTileKeys, key_tiles);
    const int n_vis = off + q0 + r + 1;
    const int64_t irow = r < rows ? il.row(b, q0 + r) : 0;
    const int k = r < rows ? clamp_budget(kt[irow], k_max) : 0;
    const int32_t* __restrict__ row = idx + irow * k_max;
    const bool vec = (k_max & 3) == 0;                 // rows start on 16-byte boundaries
    uint32_t* const bits = s_bits + warp * kMaskRowWords;
    // The host chose the tiles by the budget that the sets centre on.  If they hold so few pairs that the gather is cheaper after
    // all (a normaliser of Eq. 8 far from the scores' variance), the last CTA to count says so, for this chunk of rows: one
    // atomic per CTA, CTAs in the upper bits and pairs in the lower, sent here and looked at behind the masks.
    unsigned long long pairs = 0, counted = 0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int j = 0; j < kMaskRowAlign; ++j)
            if (r0 + j < rows) pairs += clamp_budget(kt[il.row(b, q0 + r0 + j)], k_max);
        counted = atomicAdd(reinterpret_cast<unsigned long long*>(dev_status + kStatusPairsWord), (1ull << kPairsBits) + pairs);
    }
    int at = 0;                                        // entries below `at` have been placed
    bool regular = r >= rows || k == kt[irow];
    for (int w0 = 0; w0 < tiles * 4; w0 += kMaskWindowWords) {
        const int words = min(kMaskWindowWords, tiles * 4 - w0);
        for (int i = lane; i < words / 4; i += 32) reinterpret_cast<uint4*>(bits)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        const int lo = w0 * 32, hi = min((w0 + words) * 32, n_vis);
        int last = -1;                                 // entry in front of the batch (-1: compared already)
        // 256 entries a time, eight consecutive ones per lane: neighbours mostly share a word, which then takes
        // one shared-memory atomic.  The next 512 are on their way meanwhile.
        auto load = [&](int32_t (&e)[8], int from) {
            const int j0 = from + lane * 8;
            if (vec && (from & 3) == 0 && j0 + 8 <= k) {
                const int4 a = *reinterpret_cast<const int4*>(row + j0), c = *reinterpret_cast<const int4*>(row + j0 + 4);
                e[0] = a.x; e[1] = a.y; e[2] = a.z; e[3] = a.w; e[4] = c.x; e[5] = c.y; e[6] = c.z; e[7] = c.w;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) e[j] = j0 + j < k ? row[j0 + j] : 0x7FFFFFFF;
            }
        };
        int32_t e[8], ahead[2][8];
        load(e, at);
        load(ahead[0], at + 256);
        while (at < k) {
            load(ahead[1], at + 512);
            const int j0 = at + lane * 8;
            int before = __shfl_up_sync(0xFFFFFFFFu, e[7], 1);
            if (lane == 0) before = last;
            int taken = 0, word = -1;
            uint32_t acc = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (j0 + j < k && e[j] <= before) regular = false;       // not strictly ascending from 0 on
                before = e[j];
                if (e[j] < hi) {
                    ++taken;
                    if (e[j] >= lo) {
                        const int w = (e[j] - lo) >> 5;
                        if (w != word) {
                            if (acc) atomicOr(bits + word, acc);
                            word = w; acc = 0;
                        }
                        acc |= 1u << (e[j] & 31);
                    }
                }
            }
            if (acc) atomicOr(bits + word, acc);
            taken = __reduce_add_sync(0xFFFFFFFFu, taken);
            at += taken;
            if (taken < 256) break;
            last = __shfl_sync(0xFFFFFFFFu, e[7], 31);
#pragma unroll
            for (int j = 0; j < 8; ++j) { e[j] = ahead[0][j]; ahead[0][j] = ahead[1][j]; }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < words / 4 * kMaskRowAlign; i += kMaskRowAlign * 32) {
            const int tile = i / kMaskRowAlign, rr = i % kMaskRowAlign;
            mask[((int64_t)b * key_tiles + w0 / 4 + tile) * row_pitch + r0 + rr] =
                *reinterpret_cast<const uint4*>(&s_bits[rr * kMaskRowWords + tile * 4]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && (counted >> kPairsBits) == gridDim.x - 1) {
        *reinterpret_cast<unsigned long long*>(dev_status + kStatusPairsWord) = 0ull;        // (for the next chunk's masks)
        if ((counted & ((1ull << kPairsBits) - 1)) + pairs < few_pairs) atomicOr(general, kGeneralFew);
        else atomicAnd(general, ~kGeneralFew);
    }
    if (at < k || !regular) atomicOr(general, kGeneralSets);              // (at < k: an entry past what the row can see, or out of order)
}

// masks of sets that hold every visible key: nothing to read
__global__ void __launch_bounds__(256) gsa_visible_masks_kernel(uint4* __restrict__ mask, int64_t n, int row_pitch, int key_tiles,
                                                                int off, int q0, int rows) {
    chain_wait();
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const int r = (int)(i % row_pitch), tile = (int)(i / row_pitch % key_tiles);
    const int m = r < rows ? off + q0 + r + 1 - tile * kMaskTileKeys : 0;            // keys of the tile that the row sees
    auto word = [&](int lo) -> uint32_t { return m >= lo + 32 ? 0xFFFFFFFFu : (m > lo ? (1u << (m - lo)) - 1u : 0u); };
    mask[i] = make_uint4(word(0), word(32), word(64), word(96));
}

// ---- what the tiles cannot take -----------------------------------------------------------------------------
// A tile multiplies every value row of its 128 keys, by zero where the key is not in the set, and a bit mask holds a
// key once.  So a call whose gated values are not all finite and of sane size (untileable_bf16x8), or whose sets are not strictly
// ascending positions that the row can see, raises the `general` word; the tile kernels then leave at once and the gather kernels,
// enqueued behind them, do the work, at the speed that they have anyway.  Otherwise these cost a launch.
// raises `general` if a bf16 value is infinite, NaN or too large for the tiles
__global__ void __launch_bounds__(256) gsa_check_values_kernel(const uint4* __restrict__ x, int64_t n_vec, int32_t* general) {
    chain_wait();
    uint32_t bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_vec; i += (int64_t)gridDim.x * blockDim.x)
        bad |= untileable_bf16x8(__ldg(x + i));
    if (bad) atomicOr(general, kGeneralValues);
}

// ---- forward ---------------------------------------------------------------------------------------------
// Three warpgroups launched at 168 registers a thread; the two softmax groups take 216 (64 scores of a row and what is made of
// them live in registers), the copy / MMA group keeps 72: 2 * 216 + 72 = 504 of the 504 the block was launched with.
constexpr int kFwdThreads = 384;
// Margin of the reference, log2(256 / 245): the largest numerator is then a bf16 value, so that a row that one key dominates keeps
// its output exact (with 1/16, 2 % more error in dQ and dK, whose dominating terms cancel).  Over spreads of the scores from
// 0.003 to 3 the finest of 0, 0.02, 0.05, 1/16, 0.1, 0.2 and 0.4 on the whole.
constexpr float kRefMargin = 0.063362061f;
// Above this sum of 64 numerators the reference is taken anew.  The sum is at hand, where a maximum costs an instruction a score; a numerator
// above 2^8 makes it 2^8 (less what the roundings may hide), and so do 64 scores that average 2^2 above the reference.  (A line at
// 2^14, which some numerator above 2^8 has to cross, left a row that one key dominates with a numerator that is no bf16 value: error of
// its output against fp64, a key 2^9 to 2^13.5 above the others, 2.3e-3 against 1.65e-3, and no time saved.  Asking the
// maximum, behind the sum, whether a score lies 2^8 above costs 1.5 to 4 % where G = 1: 6000 rows 113.1 -> 117.5 us.)
constexpr float kRefSum = 255.f;

template <int DH>
struct FwdSmem {
    static constexpr int CHUNKS = DH / 64;
    static constexpr int CHUNK_BYTES = 128 * 128;                  // 128 rows of 64 bf16
    static constexpr int TILE_BYTES = CHUNKS * CHUNK_BYTES;
    static constexpr int SLOTS = DH == 128 ? 5 : 8;                // K / V' tiles in flight
    static constexpr int OFF_RING = 2 * TILE_BYTES;
    static constexpr int OFF_BAR = OFF_RING + SLOTS * TILE_BYTES;
    static constexpr int N_BARS = 2 * SLOTS + 2 + 4 + 4 + 2 + 1;       // ring full / empty, Q, S (halves), P (halves), g1, drain
    static constexpr int OFF_TMEM = OFF_BAR + N_BARS * 8;
    static constexpr int OFF_ABORT = OFF_TMEM + 8;
    static constexpr int ALLOC = OFF_ABORT + 8 + 1024;
};

struct MaskedFwdArgs {
    const uint4* mask;
    float* lse;                    // nullable
    int32_t* dev_status;
    const int32_t* general;
    int32_t q0, rows, row_pitch, key_tiles;      // MaskPlan
    int32_t Lq, Lk, n_h, n_kv, row_blocks;
    int32_t abreast;               // tile_order
    float scale_log2;
    long long wait_cycles;
    int32_t withhold_first;        // fault injection: the first copy into the ring is left out (its barrier is never completed)
};

template <int DH, int G>
__global__ void __launch_bounds__(kFwdThreads, 1)
gsa_masked_attn_fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                           const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_g,
                           const __grid_constant__ CUtensorMap tm_o, const MaskedFwdArgs a) {
    chain_wait();
    using P = FwdSmem<DH>;
    constexpr int QT = 128 / G;                                    // queries per M tile
    constexpr int CH = P::CHUNKS;
    constexpr uint32_t kTmS = 0, kTmO = 256;                       // TMEM columns: S / P at kTmS + 128 s, O at kTmO + 128 s
    constexpr int HALF = kMaskTileKeys / 2;
    constexpr uint32_t kIdescS = make_idesc_bf16(128, HALF);
    constexpr uint32_t kIdescO = make_idesc_bf16(128, DH) | kIdescTransB;

    extern __shared__ unsigned char dyn_smem_raw[];
    const uint32_t raw_u32 = smem_u32(dyn_smem_raw);
    const uint32_t pad = (1024u - (raw_u32 & 1023u)) & 1023u;
    unsigned char* smem = dyn_smem_raw + pad;
    const uint32_t sbase = raw_u32 + pad;
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + P::OFF_TMEM);
    volatile int* s_abort = reinterpret_cast<volatile int*>(smem + P::OFF_ABORT);
    const uint32_t bar0 = sbase + P::OFF_BAR;
    auto bar_full = [&](int s) { return bar0 + 8u * s; };
    auto bar_empty = [&](int s) { return bar0 + 8u * (P::SLOTS + s); };
    auto bar_q = [&](int s) { return bar0 + 8u * (2 * P::SLOTS + s); };
    auto bar_s = [&](int s, int p) { return bar0 + 8u * (2 * P::SLOTS + 2 + 2 * s + p); };      // (completion i: scores of tile i, and
                                                                                                // the product of tile i - 1's half)
    auto bar_p = [&](int s, int p) { return bar0 + 8u * (2 * P::SLOTS + 6 + 2 * s + p); };      // (one completion per tile each)
    auto bar_g = [&](int s) { return bar0 + 8u * (2 * P::SLOTS + 10 + s); };
    const uint32_t bar_drain = bar0 + 8u * (2 * P::SLOTS + 12);

    int timed_out;
    if (!tiles_allowed(a.dev_status, &timed_out)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int rank, bh;                                                  // (late rows are the long ones)
    tile_order(blockIdx.x, a.row_blocks, gridDim.x / a.row_blocks, a.abreast, &rank, &bh);
    const int blk = a.row_blocks - 1 - rank;
    const int g = bh % a.n_kv, b = bh / a.n_kv;
    const int r0 = blk * 2 * QT;                                   // first query row of the CTA (from q0)
    const int off = a.Lk - a.Lq;
    const int r_end = min(r0 + 2 * QT, a.rows);
    const int ntiles = min((off + a.q0 + r_end + kMaskTileKeys - 1) / kMaskTileKeys, a.key_tiles);

    if (threadIdx.x == 0) {
        for (int s = 0; s < P::SLOTS; ++s) { mbar_init(bar_full(s), 1); mbar_init(bar_empty(s), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(bar_q(s), 1); mbar_init(bar_g(s), 1); for (int p = 0; p < 2; ++p) { mbar_init(bar_s(s, p), 1); mbar_init(bar_p(s, p), 4); } }
        mbar_init(bar_drain, 1);
        *s_abort = timed_out;                                      // (then every wait ends at once)
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(sbase + P::OFF_TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    int copies_issued = 0, q_issued = 0, g_issued = 0;             // by the copy producer
    int slots_released = 0;                                        // by the MMA issuer

    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        // ================= softmax, then the epilogue: thread = row ==================================
        const int s = warp >> 2, quad = warp & 3;
        const int m = quad * 32 + lane;                            // row of the tile = TMEM lane
        const int r = r0 + s * QT + m / G;                         // query row from q0
        const bool live = r < a.rows;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
        const uint32_t ts = lane_base + kTmS + 128 * s, to = lane_base + kTmO + 128 * s;
        const uint4* __restrict__ mrow = a.mask + (int64_t)b * a.key_tiles * a.row_pitch + r;
        float m_ref = -INFINITY;
        uint64_t l2[2] = {0ull, 0ull};                             // (pairs of fp32 partial sums)
        uint4 mk_next = live ? __ldg(mrow) : make_uint4(0u, 0u, 0u, 0u);
        const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2);
        bool ok = true;
        for (int i = 0; i < ntiles; ++i) {
            const uint4 mk = mk_next;
            if (live && i + 1 < ntiles) mk_next = __ldg(mrow + (int64_t)(i + 1) * a.row_pitch);
            const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
            // Half a tile at a time: while one half's numerators are made, the tensor cores take in the other's and score the same
            // half of the next tile behind it.
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (!(ok = warp_wait(bar_s(s, p), i & 1, s_abort, a.wait_cycles))) break;
                // The reference of the tiles before nearly always still serves, so the numerators are taken against it at
                // once, 32 columns at a time with the next 32 on their way; only if their sum shows that a selected score may exceed
                // it by more than 2^8 (kRefSum; a row's first tiles) is the work done again from the scores, still in registers.
                uint32_t v[2][32];
                uint64_t sum[2] = {0ull, 0ull};
                const float neg0 = m_ref == -INFINITY ? 0.f : -m_ref;
                uint64_t neg2 = pack_f32x2(neg0, neg0);
                auto numerators = [&](int c) {
                    uint32_t pk[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const uint64_t x = fma_f32x2(pack_f32x2(__uint_as_float(v[c][2 * j]), __uint_as_float(v[c][2 * j + 1])), scale2, neg2);
                        float x0, x1;
                        unpack_f32x2(x, x0, x1);
                        x0 = ex2_approx(x0); x1 = ex2_approx(x1);
                        sum[j & 1] = add_f32x2(sum[j & 1], pack_f32x2(x0, x1));
                        pk[j] = pack_bf16(x0, x1);
                    }
                    tc_st16(ts + HALF * p + 16 * c, pk);
                };
                tc_ld32(ts + HALF * p, v[0]);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    tc_wait_ld32(v[c]);
                    if (c == 0) tc_ld32(ts + HALF * p + 32, v[1]);
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (!((mw[2 * p + c] >> j) & 1u)) v[c][j] = 0xFF800000u;             // -inf
                    // (the numerators of columns 32 n .. of the half go over its columns 16 n .., which have been read)
                    numerators(c);
                }
                float a0, a1, a2, a3;
                unpack_f32x2(sum[0], a0, a1); unpack_f32x2(sum[1], a2, a3);
                const bool first = m_ref == -INFINITY && (mw[2 * p] | mw[2 * p + 1]) != 0u;
                if (__any_sync(0xFFFFFFFFu, first || (a0 + a1) + (a2 + a3) > kRefSum)) {
                    float top = -INFINITY;
#pragma unroll
                    for (int j = 0; j < 64; ++j) top = fmaxf(top, __uint_as_float(v[j >> 5][j & 31]));
                    top *= a.scale_log2;
                    const float m_new = top > m_ref ? top + kRefMargin : m_ref;
                    const float alpha = m_ref == -INFINITY ? 0.f : ex2_approx(m_ref - m_new);
                    m_ref = m_new;
                    const float neg1 = m_ref == -INFINITY ? 0.f : -m_ref;
                    neg2 = pack_f32x2(neg1, neg1);
                    const uint64_t al2 = pack_f32x2(alpha, alpha);
                    l2[0] = mul_f32x2(l2[0], al2); l2[1] = mul_f32x2(l2[1], al2);
                    sum[0] = sum[1] = 0ull;
                    tc_wait_st();                                  // (the columns are written a second time)
                    numerators(0);
                    numerators(1);
                    if (i > 0 || p > 0) {
                        // once the last product handed over has completed, so has every product into O so far
                        if (!(ok = warp_wait(bar_s(s, p ^ 1), (i + p) & 1, s_abort, a.wait_cycles))) break;
                        uint32_t o[16];
#pragma unroll
                        for (int c = 0; c < DH / 16; ++c) {
                            tc_ld16(to + 16 * c, o);
                            tc_wait_ld16(o);
#pragma unroll
                            for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
                            tc_st16(to + 16 * c, o);
                        }
                    }
                }
                l2[0] = add_f32x2(l2[0], sum[0]); l2[1] = add_f32x2(l2[1], sum[1]);
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p(s, p));
            }
            if (!ok) break;
        }
        // (the last product, and this tile's g1)
        ok = ok && warp_wait(bar_s(s, 1), ntiles & 1, s_abort, a.wait_cycles) && warp_wait(bar_g(s), 0, s_abort, a.wait_cycles);
        if (!ok) {
            if (lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutEpi);
        } else {
            float la, lb, lc, ld;
            unpack_f32x2(l2[0], la, lb); unpack_f32x2(l2[1], lc, ld);
            const float l = (la + lb) + (lc + ld);
            const int h = g * G + m % G, t = a.q0 + r;
            const float inv = l != 0.f ? 1.0f / l : 0.f;           // (an empty set: a zero row; a NaN in a selected key shows)
            if (a.lse && live) a.lse[((size_t)b * a.Lq + t) * a.n_h + h] = (m_ref + log2f(l)) * 0.6931471805599453f;
            // g1 lies where Q was, in its layout; the output goes over it and out as one box (rows past the last are clipped).
            // Row by row from and to global memory this took 8.7 us of a CTA's time.
            unsigned char* const row = smem + s * P::TILE_BYTES + m * 128;
#pragma unroll
            for (int c = 0; c < DH / 32; ++c) {
                uint32_t o[32];
                tc_ld32(to + 32 * c, o);
                tc_wait_ld32(o);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint4* const at = reinterpret_cast<uint4*>(row + (c >> 1) * P::CHUNK_BYTES + (((4 * (c & 1) + q) ^ (m & 7)) << 4));
                    const uint4 gv = *at;
                    const __nv_bfloat162* gp = reinterpret_cast<const __nv_bfloat162*>(&gv);
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 gf = __bfloat1622float2(gp[e]);
                        const float o0 = l != 0.f ? __uint_as_float(o[q * 8 + 2 * e]) * inv : 0.f;
                        const float o1 = l != 0.f ? __uint_as_float(o[q * 8 + 2 * e + 1]) * inv : 0.f;
                        w[e] = pack_bf16(o0 * fast_sigmoid(gf.x), o1 * fast_sigmoid(gf.y));
                    }
                    *at = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
        }
        // (every thread of the tile comes here, whether its waits ended well or not)
        if (tile_results_written(1 + s, 128, ok) && (threadIdx.x & 127) == 0 && r0 + s * QT < a.rows) {
            for (int c = 0; c < CH; ++c) tma_store_tile(&tm_o, c * 64, g * G, r0 + s * QT, b, sbase + s * P::TILE_BYTES + c * P::CHUNK_BYTES);
            tma_store_wait();
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        if (warp == 8) {
            // ================= copies: Q tiles, then K_0 V_0 K_1 V_1 ... ================================
            if (lane == 0) {
                for (int s = 0; s < 2; ++s) {
                    mbar_expect_tx(bar_q(s), P::TILE_BYTES);
                    for (int c = 0; c < CH; ++c)
                        tma_load_tile(sbase + s * P::TILE_BYTES + c * P::CHUNK_BYTES, &tm_q, c * 64, g * G, r0 + s * QT, b, bar_q(s));
                    q_issued = s + 1;
                }
                bool ok = true;
                for (int n = 0; ok && n < 2 * ntiles; ++n) {
                    const int s = n % P::SLOTS;
                    if (!mbar_wait(bar_empty(s), ((n / P::SLOTS) & 1) ^ 1, s_abort, a.wait_cycles)) { ok = false; break; }
                    copies_issued = n + 1;
                    if (n == 0 && a.withhold_first) continue;
                    mbar_expect_tx(bar_full(s), P::TILE_BYTES);
                    for (int c = 0; c < CH; ++c)
                        tma_load_tile(sbase + P::OFF_RING + s * P::TILE_BYTES + c * P::CHUNK_BYTES, (n & 1) ? &tm_v : &tm_k,
                                      c * 64, g, (n >> 1) * kMaskTileKeys, b, bar_full(s));
                }
                // the output's gates take Q's place once the last scores have been made
                const int last = 2 * (ntiles - 1);
                ok = ok && mbar_wait(bar_empty(last % P::SLOTS), (last / P::SLOTS) & 1, s_abort, a.wait_cycles);
                for (int s = 0; ok && s < 2; ++s) {
                    mbar_expect_tx(bar_g(s), P::TILE_BYTES);
                    for (int c = 0; c < CH; ++c)
                        tma_load_tile(sbase + s * P::TILE_BYTES + c * P::CHUNK_BYTES, &tm_g, c * 64, g * G, r0 + s * QT, b, bar_g(s));
                    g_issued = s + 1;
                }
                if (!ok) atomicCAS(a.dev_status, kDevOk, kDevTimeoutTma);
            }
        } else if (warp == 9) {
            // ================= MMA issue (converged warp) ================================================
            const uint32_t el = elect_lane();
            bool ok = true;
            auto wait = [&](uint32_t bar, uint32_t parity) { return warp_wait(bar, parity, s_abort, a.wait_cycles); };
            auto wait_slot = [&](int n) { return wait(bar_full(n % P::SLOTS), (n / P::SLOTS) & 1); };      // ring entry n has landed
            auto slot_addr = [&](int n) { return sbase + P::OFF_RING + (n % P::SLOTS) * P::TILE_BYTES; };
            auto issue_s = [&](int s, int i, int p) {              // S_s = Q_s K_i^T, half p of the keys
                const uint64_t qd = make_kmajor_desc<128>(sbase + s * P::TILE_BYTES);
                const uint64_t kd = make_kmajor_desc<128>(slot_addr(2 * i) + p * HALF * 128);
#pragma unroll
                for (int k = 0; k < DH / 16; ++k) {
                    const uint64_t step = (uint64_t)((k >> 2) * (P::CHUNK_BYTES >> 4) + 2 * (k & 3));
                    warp_mma_ss(el, tmem + kTmS + 128 * s + HALF * p, qd + step, kd + step, kIdescS, k > 0);
                }
            };
            auto issue_o = [&](int s, int i, int p) {              // O_s += P_s V'_i, half p of the keys
                const uint64_t vd = make_mnmajor_desc(slot_addr(2 * i + 1), P::CHUNK_BYTES);
#pragma unroll
                for (int k = 0; k < 4; ++k)                        // 16 keys = 2048 bytes of the V' tile, 8 columns of P
                    warp_mma_ts(el, tmem + kTmO + 128 * s, tmem + kTmS + 128 * s + HALF * p + 8 * k, vd + 128 * (4 * p + k), kIdescO,
                                (i | p | k) != 0);
            };
            auto release = [&](int n) { warp_commit(el, bar_empty(n % P::SLOTS)); slots_released = n + 1; };
            ok = wait_slot(0) && wait(bar_q(0), 0) && wait(bar_q(1), 0);
#pragma unroll
            for (int h = 0; h < 4; ++h)
                if (ok) { issue_s(h & 1, 0, h >> 1); warp_commit(el, bar_s(h & 1, h >> 1)); }
            if (ok) release(0);
            for (int i = 0; ok && i < ntiles; ++i) {
                const bool more = i + 1 < ntiles;
                ok = wait_slot(2 * i + 1) && (!more || wait_slot(2 * i + 2));
                // the halves in the order in which the two groups of softmax warps hand them over
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int s = h & 1, p = h >> 1;
                    if (!ok || !(ok = wait(bar_p(s, p), i & 1))) break;
                    issue_o(s, i, p);
                    if (more) issue_s(s, i + 1, p);                // (in order behind the product that reads P from these columns)
                    warp_commit(el, bar_s(s, p));
                }
                if (!ok) break;
                release(2 * i + 1);
                if (more) release(2 * i + 2);
            }
            if (!ok && lane == 0) atomicCAS(a.dev_status, kDevOk, kDevTimeoutMma);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (*s_abort) {
        // give-up path: let what was issued complete (each poll is bounded) before shared memory and TMEM are released
        if (warp == 8 && lane == 0) {
            for (int s = 0; s < q_issued; ++s) mbar_drain(bar_q(s), 0);
            for (int s = 0; s < g_issued; ++s) mbar_drain(bar_g(s), 0);
            for (int n = max(a.withhold_first, copies_issued - P::SLOTS); n < copies_issued; ++n)
                mbar_drain(bar_full(n % P::SLOTS), (n / P::SLOTS) & 1);
        }
        if (warp == 9) {
            warp_commit(elect_lane(), bar_drain);
            mbar_drain(bar_drain, 0);
            for (int n = max(0, slots_released - P::SLOTS); n < slots_released; ++n)
                mbar_drain(bar_empty(n % P::SLOTS), (n / P::SLOTS) & 1);
        }
        tc_fence_before();
        __syncthreads();
    }
    if (warp == 9) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

template <int DH, int G>
cudaError_t launch_fwd_t(const MaskedFwdArgs& a, const gsa_params_t& p, const CUtensorMap& tq, const CUtensorMap& tk,
                         const CUtensorMap& tv, const CUtensorMap& tg, const CUtensorMap& to, cudaStream_t st) {
    constexpr int kSmem = FwdSmem<DH>::ALLOC;
    auto kern = gsa_masked_attn_fwd_kernel<DH, G>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    launch_chained(kern, (unsigned)(a.row_blocks * p.n_kv * p.B), kFwdThreads, kSmem, st, tq, tk, tv, tg, to, a);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_build_masks(const gsa_params_t& p, const MaskPlan& mp, int block_rows, const int32_t* idx,
                               const int32_t* kt, IdxLayout il, uint4* mask, int32_t* dev_status, double few_pairs, cudaStream_t st) {
    const unsigned grid = (unsigned)(mp.row_pitch / kMaskRowAlign) * (unsigned)p.B;
    launch_chained(gsa_build_masks_kernel, grid, kMaskRowAlign * 32, 0, st, idx, kt, mask, il, mp.q0, mp.rows, mp.row_pitch, mp.key_tiles,
                                                               block_rows, p.k_max, p.Lk - p.Lq, dev_status, (unsigned long long)(few_pairs > 0.0 ? few_pairs : 0.0));
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_visible_masks(const gsa_params_t& p, const MaskPlan& mp, uint4* mask, cudaStream_t st) {
    const int64_t n = (int64_t)p.B * mp.key_tiles * mp.row_pitch;
    launch_chained(gsa_visible_masks_kernel, (unsigned)((n + 255) / 256), 256, 0, st, mask, n, mp.row_pitch, mp.key_tiles,
                   p.Lk - p.Lq, mp.q0, mp.rows);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_check_values(const __nv_bfloat16* x, int64_t n_elems, int32_t* general, cudaStream_t st) {
    const int64_t n_vec = n_elems / 8;
    const int64_t want = (n_vec + 255) / 256, cap = (int64_t)sm_count() * 8;
    launch_chained(gsa_check_values_kernel, (unsigned)(want < cap ? want : cap), 256, 0, st, reinterpret_cast<const uint4*>(x), n_vec, general);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_masked_attn_fwd(const gsa_params_t& p, const MaskPlan& mp, const uint4* mask, const __nv_bfloat16* Q,
                                   const __nv_bfloat16* K, const __nv_bfloat16* Vg, const __nv_bfloat16* g1,
                                   __nv_bfloat16* out, float* lse, int32_t* dev_status, cudaStream_t st) {
    const int G = p.n_h / p.n_kv;
    CUtensorMap tq, tk, tv, tg, to;
    const size_t row0 = (size_t)mp.q0 * p.n_h * p.d_h;
    if (!make_heads_tmap(&tq, Q + row0, p.B, p.Lq, mp.rows, p.n_h, p.d_h, 128 / G, G)) return cudaErrorUnknown;
    if (!make_heads_tmap(&tg, g1 + row0, p.B, p.Lq, mp.rows, p.n_h, p.d_h, 128 / G, G)) return cudaErrorUnknown;
    if (!make_heads_tmap(&to, out + row0, p.B, p.Lq, mp.rows, p.n_h, p.d_h, 128 / G, G)) return cudaErrorUnknown;
    if (!make_heads_tmap(&tk, K, p.B, p.Lk, p.Lk, p.n_kv, p.d_h, kMaskTileKeys, 1)) return cudaErrorUnknown;
    if (!make_heads_tmap(&tv, Vg, p.B, p.Lk, p.Lk, p.n_kv, p.d_h, kMaskTileKeys, 1)) return cudaErrorUnknown;
    MaskedFwdArgs a;
    a.mask = mask; a.lse = lse; a.dev_status = dev_status; a.general = dev_status + kStatusGeneralWord;
    a.q0 = mp.q0; a.rows = mp.rows; a.row_pitch = mp.row_pitch; a.key_tiles = mp.key_tiles;
    a.Lq = p.Lq; a.Lk = p.Lk; a.n_h = p.n_h; a.n_kv = p.n_kv;
    a.row_blocks = (mp.rows + masked_block_rows(p) - 1) / masked_block_rows(p);
    a.abreast = pairs_abreast(p.n_kv * p.B, 4.0 * p.Lk * p.d_h);
    const float sc = p.sm_scale > 0.f ? p.sm_scale : 1.0f / sqrtf((float)p.d_h);
    a.scale_log2 = sc * 1.4426950408889634f;
    a.wait_cycles = wait_limit_cycles();
    a.withhold_first = withhold_first_copy() ? 1 : 0;
#define GSA_CASE(DH_, G_) if (p.d_h == DH_ && G == G_) return launch_fwd_t<DH_, G_>(a, p, tq, tk, tv, tg, to, st)
    GSA_CASE(128, 1); GSA_CASE(128, 2); GSA_CASE(128, 4); GSA_CASE(128, 8);
    GSA_CASE(64, 1); GSA_CASE(64, 2); GSA_CASE(64, 4); GSA_CASE(64, 8);
#undef GSA_CASE
    return cudaErrorInvalidValue;
}

}  // namespace gsa
