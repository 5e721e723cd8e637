// Sparse gated attention (Eq. 9, 11, 12, 10): the gather kernels, for sets that hold a small share of the visible keys
// (larger shares: masked tiles, gsa_masked_attn.cu; masked_rows_end below draws the line) and for decode.
//
// Work item = (query token, KV head, segment of the token's index set S_t); one warp per item,
// 16 warps per CTA, items dealt to warps round-robin so that the warps of a CTA work on the same
// two tokens.  A warp walks its segment 16 selected keys at a time:
//
//   K   the 16 keys' d_h-wide slices are read with 16-byte loads straight into the registers that
//       the tensor-core MMA takes as its A operand (keys are M).  The contraction index of Q.K is
//       d, and a sum does not care about the order of its terms, so each thread simply uses the 8
//       consecutive d it loaded as "its" k-indices and reads Q with the same permutation: no
//       shared memory, no shuffles.                          S^T[key, head] = K[key,:] . Q[head,:]
//   softmax  online, per head = per column of S^T: max/sum across the 8 lanes that hold a column.
//   P^T -> B operand: the bf16 pairs of S^T's fragment are an 8x8 matrix; one movmatrix
//       transposes it into the B-fragment layout.
//   V'  the 16 keys' slices arrive by 16-byte async copies in a private two-stage buffer in
//       shared memory and are read transposed (ldmatrix.trans) as the A operand of
//                                                          O^T[d, head] += V'^T[d, key] P^T[key, head]
//       With heads on the N side one MMA covers all G <= 8 query heads of the KV group, so the
//       whole tile costs d_h/16 + d_h/16 MMAs of m16n8k16.
//   The next tile's K loads, V' copies and indices are in flight while the current tile is
//   computed.  16 warps x (4 KB in registers + 4 KB in shared memory) per SM keep the L2 busy.
//
// The gather dominates: every selected (token, key) pair moves one K row and one V' row of all KV
// heads (4 KB at the 1.7B shape).  Random 2 KB rows come at ~8 TB/s out of HBM but at 11-13 TB/s
// out of the 126 MB L2, so for long contexts the key axis is cut into ranges whose K and V' rows
// fit in L2 and the kernel is launched once per range, over every query's sub-list in that range
// (index sets are ascending, so a sub-list is contiguous).  The online-softmax state (m, l, O) of a
// (token, head) is carried from range to range in fp32 in the workspace.  For decode-sized calls
// (few tokens) the same state slots hold the partial results of segments that run in parallel.
// A last small kernel merges the slots, normalises, applies G1 and rounds to bf16 once.
//
// G2 is either applied by a streaming pre-pass (V' = bf16(V * sigmoid(g2)), prefill) or on the gathered
// rows (decode, where gating the whole cache would cost more than the attention): the V and the g2 slices
// of a tile then arrive in two shared-memory tiles, both are read transposed into the same A-fragment
// layout, and the gate is applied to the fragments in registers right before the MMA.
#include "gsa_common.cuh"
#include "gsa_masked.cuh"

namespace gsa {

namespace {

constexpr int kTileKeys = 16;
constexpr int kWarpsPrefill = 16;          // warps per CTA, V' pre-gated
constexpr int kWarpsFused = 16;            // warps per CTA when V and g2 are gathered raw and gated in the fragments
constexpr float kRefSlack = 8.0f;          // a score may exceed the softmax reference by 2^8 before the reference moves
constexpr int kVStages = 2;                // shared-memory stages of a warp's V' tiles (one being read, the others in flight;
                                           // measured at L = 128K: 2 stages 90.2 ms, 3 stages 94.7 ms)
constexpr int kRangeKeysDefault = 16384;   // keys per L2 range: K + V' rows of 16K tokens = 64 MB at the 1.7B shape
constexpr int kMaxRanges = 48;
constexpr int kPartKeys = 32;              // decode: fewest keys worth a parallel segment (as exact as 128: 16 shapes x 3 inputs against fp64
                                           // 2.629e-3 and 2.635e-3, worst 2.75e-3 and 2.74e-3)

struct AttnArgs {
    const __nv_bfloat16* Q;
    const __nv_bfloat16* K;
    const __nv_bfloat16* V;
    const __nv_bfloat16* g2;
    const int32_t* idx;
    const int32_t* kt;
    const int32_t* cuts;      // range mode: [idx rows][n_cuts] positions in the index row where each range starts
    float* state;             // [slots][idx rows][n_kv][G*(d_h+2)] fp32
    RowRange rr;
    IdxLayout il;
    int64_t idx_rows;         // rows of the idx / kt / state tables
    int32_t Lq, Lk, n_h, n_kv, k_max;
    int32_t mode;             // 0: one key range per launch (range index `range`), 1: parallel parts
    int32_t max_parts;        // mode 1: segments (= state slots) per index set
    int32_t range, n_cuts;
    float scale_log2;         // sm_scale * log2(e)
    float* lse;               // optional output [B, Lq, n_h]: natural log of sum_j exp(sm_scale * q.k_j) over S_t
    const int32_t* only_if;   // see left_out
    int32_t run_if;
    const __nv_bfloat16* g1;  // DIRECT only
    __nv_bfloat16* out;
    int32_t* dev_status;      // where an out-of-range index or budget is reported (may be null)
};

struct RowId { int32_t b, t; int64_t irow; };

__device__ __forceinline__ RowId row_of(const RowRange& rr, const IdxLayout& il, int lr) {
    RowId r;
    r.b = rr.b0 + lr / rr.R;
    r.t = rr.q_begin + lr % rr.R;
    r.irow = il.row(r.b, r.t);
    return r;
}

__device__ __forceinline__ uint4 ldg_stream(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// 32 bytes per thread: a warp-wide load covers whole 128-byte lines of 8 rows
__device__ __forceinline__ void ldg_stream32(const void* p, uint4& lo, uint4& hi) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
                 : "l"(p));
}
__device__ __forceinline__ float ex2_fast(float x) {          // 2^x, one special-function instruction; 2^-inf = 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__host__ __device__ __forceinline__ int parts_of(int k_eff, int max_parts) {
    const int p = (k_eff + kPartKeys - 1) / kPartKeys;
    return p < 1 ? 1 : (p > max_parts ? max_parts : p);
}

// DIRECT: whole sets in one launch, in any order of their entries; rows are normalised, gated and written here instead of through
// the state (what the masked tiles leave to the gather).
template <int DH, int G, bool FUSE_G2, bool DIRECT = false>
__global__ void __launch_bounds__((FUSE_G2 ? kWarpsFused : kWarpsPrefill) * 32, 1)
gsa_sparse_attn_kernel(const AttnArgs a) {
    chain_wait();
    if (left_out(a.only_if, a.run_if)) return;
    constexpr int HEAD_BYTES = DH * 2;
    constexpr int NC = DH / 32;                         // 32-d chunks of a head row (one uint4 per thread each)
    constexpr int MT = DH / 16;                         // output m-tiles
    constexpr int VSTRIDE = HEAD_BYTES + 16;            // padded row of the staged V' tile
    constexpr int VTILE = kTileKeys * VSTRIDE;
    constexpr int VSTAGES = FUSE_G2 ? 2 : kVStages;     // fused G2: one tile of V and one of g2, each single-staged
    constexpr int CHUNKS = HEAD_BYTES / 16;             // 16-byte chunks per head row
    constexpr int KPI = 32 / CHUNKS;                    // keys one warp-wide 16-byte copy covers
    constexpr int ITS = kTileKeys / KPI;
    constexpr int STATE_F = G * (DH + 2);               // floats of one (row, KV head) state

    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gid = lane >> 2, tig = lane & 3;
    unsigned char* my_smem = smem + (size_t)warp * VSTAGES * VTILE;
    const uint32_t my_s32 = smem_u32(my_smem);
    const int n_kv = a.n_kv;
    const int vkey = lane / CHUNKS, vch = lane % CHUNKS;
    const bool real_head = gid < G;                     // this thread's column of Q^T is a real head
    const bool real_cols = 2 * tig < G;                 // this thread's output columns hold real heads

    const int rows = a.rr.rows();
    const int mode = DIRECT ? 0 : a.mode;
    const int64_t n_items = (int64_t)rows * n_kv * (mode == 1 ? a.max_parts : 1);
    const int warps = blockDim.x >> 5;                  // kWarpsPerCta, or fewer where few items are spread over the SMs
    const int64_t warps_total = (int64_t)gridDim.x * warps;

    for (int64_t item = (int64_t)blockIdx.x * warps + warp; item < n_items; item += warps_total) {
        const int g = (int)(item % n_kv);
        int64_t rest = item / n_kv;
        int part = 0;
        if (mode == 1) { part = (int)(rest % a.max_parts); rest /= a.max_parts; }
        const RowId r = row_of(a.rr, a.il, (int)rest);
        const int k_eff = checked_budget(a.kt[r.irow], a.k_max, a.dev_status);
        int lo, hi, slot = 0;
        if (mode == 0) {
            lo = 0;
            hi = k_eff;
            if (!DIRECT && a.n_cuts > 1) {
                const int32_t* c = a.cuts + r.irow * a.n_cuts + a.range;
                lo = c[0];
                if (a.range + 1 < a.n_cuts) hi = c[1];
            }
        } else {
            const int np = parts_of(k_eff, a.max_parts);
            if (part >= np) continue;
            const int per = ((k_eff + np - 1) / np + kTileKeys - 1) / kTileKeys * kTileKeys;
            lo = part * per;
            hi = min(k_eff, lo + per);
            slot = part;
        }
        const int count = hi - lo;
        if (count <= 0 && mode == 0 && !DIRECT) continue;
        const int32_t* __restrict__ idx_seg = a.idx + r.irow * a.k_max + lo;
        const int ntiles = (count + kTileKeys - 1) / kTileKeys;
        float* __restrict__ st = a.state + (((int64_t)slot * a.idx_rows + r.irow) * n_kv + g) * STATE_F;

        // ---- Q^T as the B operand, in the permuted-d order the K loads use ----------------------
        uint4 qb[NC];     // piece c = bytes [(c/2)*128 + tig*32 + (c%2)*16, +16) of the head row
        {
            const int h = g * G + (real_head ? gid : 0);
            const __nv_bfloat16* qp = a.Q + (((size_t)r.b * a.Lq + r.t) * a.n_h + h) * DH + tig * 16;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                qb[c] = real_head ? *reinterpret_cast<const uint4*>(qp + (c >> 1) * 64 + (c & 1) * 8)
                                  : make_uint4(0u, 0u, 0u, 0u);
        }

        // ---- state: O^T[d, head] fragments, running max and sum per head ----------------------
        float o[MT][4];
        float m_run[2], l_run[2];
        const bool carry_in = mode == 0 && !DIRECT && lo > 0;
        if (carry_in && real_cols) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int d = mt * 16 + hf * 8 + gid;
                    if (G >= 2) {
                        const float2 v = *reinterpret_cast<const float2*>(st + d * G + 2 * tig);
                        o[mt][hf * 2] = v.x; o[mt][hf * 2 + 1] = v.y;
                    } else {
                        o[mt][hf * 2] = st[d]; o[mt][hf * 2 + 1] = 0.f;
                    }
                }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool ok = 2 * tig + e < G;
                m_run[e] = ok ? st[G * DH + 2 * tig + e] : -INFINITY;
                // every lane of a column accumulates its own share of l; the carried sum goes to one of them
                l_run[e] = (ok && gid == 0) ? st[G * DH + G + 2 * tig + e] : 0.f;
            }
        } else {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) { o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f; }
            m_run[0] = m_run[1] = -INFINITY;
            l_run[0] = l_run[1] = 0.f;
        }

        // per-item address bases: a gathered row's address is base + position * row_bytes
        const uint32_t row_bytes = (uint32_t)n_kv * HEAD_BYTES;
        const size_t head0 = ((size_t)r.b * a.Lk * n_kv + g) * HEAD_BYTES;
        const unsigned char* kbase = reinterpret_cast<const unsigned char*>(a.K) + head0 + tig * 32;
        const unsigned char* vbase = reinterpret_cast<const unsigned char*>(a.V) + head0 + vch * 16;
        const unsigned char* gbase = reinterpret_cast<const unsigned char*>(a.g2) + head0 + vch * 16;
        const uint32_t vdst = my_s32 + vkey * VSTRIDE + vch * 16;
        const int32_t pad_pos = count > 0 ? idx_seg[0] : 0;          // tail keys re-read a valid row (P = 0 there)
        auto load_pos = [&](int tile) -> int32_t {
            const int j = tile * kTileKeys + (lane & 15);
            const int32_t p = j < count ? idx_seg[j] : pad_pos;
            return checked_pos(p, a.Lk, a.dev_status);               // a corrupt index must not leave the tensor
        };
        uint4 kb[2 * NC];                                            // K tile = A operand fragments
        auto issue_k = [&](int32_t pos16) {
            const uint32_t p0 = __shfl_sync(0xFFFFFFFFu, pos16, gid), p1 = __shfl_sync(0xFFFFFFFFu, pos16, gid + 8);
            const unsigned char* k0 = kbase + (uint64_t)p0 * row_bytes;
            const unsigned char* k1 = kbase + (uint64_t)p1 * row_bytes;
#pragma unroll
            for (int c = 0; c < NC; c += 2) {
                ldg_stream32(k0 + (c >> 1) * 128, kb[c], kb[c + 1]);
                ldg_stream32(k1 + (c >> 1) * 128, kb[NC + c], kb[NC + c + 1]);
            }
        };
        // (fused G2: `stage` is ignored; the V tile sits at stage 0 and the g2 tile at stage 1)
        auto issue_v = [&](int32_t pos16, int stage) {
#pragma unroll
            for (int i = 0; i < ITS; ++i) {
                const uint32_t p = __shfl_sync(0xFFFFFFFFu, pos16, i * KPI + vkey);
                const uint64_t goff = (uint64_t)p * row_bytes;
                if (FUSE_G2) {
                    cp_async16(vdst + i * KPI * VSTRIDE, vbase + goff);
                    cp_async16(vdst + VTILE + i * KPI * VSTRIDE, gbase + goff);
                } else {
                    cp_async16(vdst + stage * VTILE + i * KPI * VSTRIDE, vbase + goff);
                }
            }
        };

        // positions of the tile whose K loads are issued next (tile + 1) and of the tile whose V' copies are
        // issued next (tile + VSTAGES - 1)
        int32_t pos_nxt = load_pos(1), pos_vahead = load_pos(VSTAGES - 1);
        {
            const int32_t pos0 = load_pos(0);
            issue_v(pos0, 0);
            cp_async_commit();
            if (!FUSE_G2) {
#pragma unroll
                for (int t = 1; t < VSTAGES - 1; ++t) {
                    if (t < ntiles) issue_v(load_pos(t), t);
                    cp_async_commit();                                   // (possibly empty: one group per tile)
                }
            }
            issue_k(pos0);
        }

        for (int tile = 0, stage = 0; tile < ntiles; ++tile, stage = (FUSE_G2 || stage == VSTAGES - 1) ? 0 : stage + 1) {
            const bool more = tile + 1 < ntiles;
            const int32_t pos_v = pos_nxt;                            // fused G2: the next tile's V / g2 copies go out after this tile's product
            if (!FUSE_G2) {
                // the stage consumed by the previous tile takes the tile after the next one
                if (tile + VSTAGES - 1 < ntiles) issue_v(pos_vahead, stage == 0 ? VSTAGES - 1 : stage - 1);
                cp_async_commit();
            }

            // ---- S^T = K Q^T : rows = 16 keys, columns = heads --------------------------------
            // (two accumulators: half the length of the dependent MMA chain)
            float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                mma_bf16_16816(s, kb[c].x, kb[NC + c].x, kb[c].y, kb[NC + c].y, qb[c].x, qb[c].y);
                mma_bf16_16816(s2, kb[c].z, kb[NC + c].z, kb[c].w, kb[NC + c].w, qb[c].z, qb[c].w);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] += s2[e];
            if (more) issue_k(pos_nxt);
            pos_nxt = load_pos(tile + 2);
            pos_vahead = VSTAGES == 2 ? pos_nxt : load_pos(tile + VSTAGES);

            // ---- online softmax per head (column) ------------------------------------------------
            // The reference value m_run that the exponentials are taken against need not be the running
            // maximum itself: any value that no score exceeds by more than kRefSlack (in the log2 domain) keeps
            // 2^(s - m_run) <= 2^kRefSlack, harmless in fp32 and bf16, and the normalisation at the end divides
            // it out.  So the reduction over the tile's keys (shuffles across the lanes of a column) and the
            // rescaling run only when some score jumps above the reference: on a row's first tiles.
            const int j0 = tile * kTileKeys + gid;
            const bool v0 = j0 < count, v1 = j0 + 8 < count;
            float sc[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sc[e] = v0 ? s[e] * a.scale_log2 : -INFINITY;
                sc[2 + e] = v1 ? s[2 + e] * a.scale_log2 : -INFINITY;
            }
            const bool jump = fmaxf(sc[0], sc[2]) > m_run[0] + kRefSlack || fmaxf(sc[1], sc[3]) > m_run[1] + kRefSlack;
            if (__any_sync(0xFFFFFFFFu, jump)) {
                float alpha[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float mx = fmaxf(sc[e], sc[2 + e]);
                    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 4));
                    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 8));
                    mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, 16));
                    const float m_new = fmaxf(m_run[e], mx);          // finite: key 0 of every tile is valid
                    alpha[e] = ex2_fast(m_run[e] - m_new);
                    m_run[e] = m_new;
                    l_run[e] *= alpha[e];
                }
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    o[mt][0] *= alpha[0]; o[mt][1] *= alpha[1]; o[mt][2] *= alpha[0]; o[mt][3] *= alpha[1];
                }
            }
            float p[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                p[e] = ex2_fast(sc[e] - m_run[e]);
                p[2 + e] = ex2_fast(sc[2 + e] - m_run[e]);
                l_run[e] += p[e] + p[2 + e];
            }
            // P^T[key, head] as the B operand: transpose the two 8x8 bf16 blocks of the fragment
            const uint32_t pb0 = movmatrix_trans(pack_bf16(p[0], p[1]));     // keys 0..7
            const uint32_t pb1 = movmatrix_trans(pack_bf16(p[2], p[3]));     // keys 8..15

            // ---- O^T += V'^T P^T -------------------------------------------------------------------
            if (FUSE_G2) cp_async_wait<0>(); else cp_async_wait<kVStages - 1>();   // this tile's copies have landed
            __syncwarp();
            {
                const int mi = lane >> 3;
                const uint32_t vaddr = my_s32 + (FUSE_G2 ? 0 : stage) * VTILE + ((lane & 7) + (mi >> 1) * 8) * VSTRIDE + (mi & 1) * 16;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    uint32_t a0, a1, a2, a3;
                    ldmatrix_x4_trans(a0, a1, a2, a3, vaddr + mt * 32);
                    if constexpr (FUSE_G2) {
                        // Eq. 9 on the fragments: the g2 tile read the same way has the same layout
                        uint32_t g0, g1r, g2r, g3;
                        ldmatrix_x4_trans(g0, g1r, g2r, g3, vaddr + VTILE + mt * 32);
                        auto gate = [](uint32_t v, uint32_t g) -> uint32_t {
                            const float2 vf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v));
                            const float2 gf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&g));
                            return pack_bf16(vf.x * gate_sigmoid(gf.x), vf.y * gate_sigmoid(gf.y));
                        };
                        a0 = gate(a0, g0); a1 = gate(a1, g1r); a2 = gate(a2, g2r); a3 = gate(a3, g3);
                    }
                    mma_bf16_16816(o[mt], a0, a1, a2, a3, pb0, pb1);
                }
            }
            __syncwarp();                                             // the tiles are refilled from here on
            if (FUSE_G2) {
                if (more) issue_v(pos_v, 0);
                cp_async_commit();
            }
        }
        cp_async_wait<0>();

        // ---- write the state slot ---------------------------------------------------------------
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            l_run[e] += __shfl_xor_sync(0xFFFFFFFFu, l_run[e], 4);
            l_run[e] += __shfl_xor_sync(0xFFFFFFFFu, l_run[e], 8);
            l_run[e] += __shfl_xor_sync(0xFFFFFFFFu, l_run[e], 16);
        }
        if (DIRECT) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (2 * tig + e >= G) continue;
                const size_t head = ((size_t)r.b * a.Lq + r.t) * a.n_h + g * G + 2 * tig + e;
                const bool live = k_eff > 0 && l_run[e] != 0.f;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const size_t at = head * DH + mt * 16 + hf * 8 + gid;
                        a.out[at] = __float2bfloat16_rn(live ? o[mt][hf * 2 + e] / l_run[e] * fast_sigmoid(__bfloat162float(a.g1[at])) : 0.f);
                    }
                if (a.lse && gid == 0) a.lse[head] = (m_run[e] + log2f(l_run[e])) * 0.6931471805599453f;
            }
        } else if (real_cols) {
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const int d = mt * 16 + hf * 8 + gid;
                    if (G >= 2) *reinterpret_cast<float2*>(st + d * G + 2 * tig) = make_float2(o[mt][hf * 2], o[mt][hf * 2 + 1]);
                    else st[d] = o[mt][hf * 2];
                }
            if (gid == 0) {
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    if (2 * tig + e < G) { st[G * DH + 2 * tig + e] = m_run[e]; st[G * DH + G + 2 * tig + e] = l_run[e]; }
            }
        }
    }
}

// cuts[row][c] = number of selected positions of the row below c * range_keys (c = 0 .. n_cuts-1)
__global__ void __launch_bounds__(256) gsa_range_cuts_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ kt,
                                                             int32_t* __restrict__ cuts, RowRange rr, IdxLayout il,
                                                             int k_max, int n_cuts, int range_keys, const int32_t* only_if,
                                                             int32_t run_if) {
    chain_wait();
    if (left_out(only_if, run_if)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)rr.rows() * n_cuts) return;
    const int c = (int)(i % n_cuts);
    const RowId r = row_of(rr, il, (int)(i / n_cuts));
    const int32_t* __restrict__ row = idx + r.irow * k_max;
    const int k_eff = clamp_budget(kt[r.irow], k_max);
    const int bound = c * range_keys;
    int lo = 0, hi = k_eff;                      // first position with row[pos] >= bound
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (row[mid] < bound) lo = mid + 1; else hi = mid;
    }
    cuts[r.irow * n_cuts + c] = lo;
}

// merge the state slots of a (row, head): out = (sum_p 2^(m_p - M) O_p) / (sum_p 2^(m_p - M) l_p) * sigmoid(g1)
//  * a single slot per row (mode 0, prefill): a CTA takes kFinRows consecutive query rows; thread = (KV head, d), all G heads of the
//    group.  The loads of all rows are issued before any is used.
//  * many slots (decode): a CTA takes one row and KV head, thread = (one of kFinGroups shares of the slots, d): one or two memory
//    latencies, whatever the number of slots.  (In a kernel of its own ptxas gives this form 32 registers in place of 64 and its loads
//    go out a few at a time: G = 4, 64 slots 12.1 us instead of 10.6.)
//  * SERIAL, few slots: the same without shares, thread = d, one slot after another: a quarter of the threads and no barriers.  There
//    are few slots where there are many CTAs (finalize_serial has the line).
constexpr int kFinRows = 4;
constexpr int kFinGroups = 4;

// Attention stage in us, shares against serial form, d_h = 128 (64 where four or eight heads share a KV head): 300 rows x 8 KV heads (one
// slot), 16 keys 31.4 and 18.5, 256 keys 70.0 and 56.9; 64 x 8 (four), 128 keys 16.6 and 15.0, G = 8: 12.4 and 14.7; 56 x 8 (five),
// 128 keys 16.5 and 14.6, G = 4: 11.1 and 11.9; 40 x 8 (seven), 2048 keys 94.1 and 95.3; 24 x 8 (twelve), sets in one segment 9.6 and 9.1,
// G = 8: 8.7 and 9.8.
inline bool finalize_serial(int G, int slots, int slots_used) {
    return G <= 2 ? slots <= 6 || slots_used == 1 : slots <= 3;
}

template <int DH, int G, bool SERIAL>
__global__ void __launch_bounds__(SERIAL ? DH : 1024) gsa_attn_finalize_kernel(const float* __restrict__ state, const int32_t* __restrict__ kt,
                                                                const __nv_bfloat16* __restrict__ g1, __nv_bfloat16* __restrict__ out,
                                                                RowRange rr, IdxLayout il, int64_t idx_rows, int Lq, int n_h,
                                                                int n_kv, int k_max, int mode, int max_parts,
                                                                float* __restrict__ lse, const int32_t* only_if, int32_t run_if) {
    chain_wait();
    if (left_out(only_if, run_if)) return;
    constexpr int STATE_F = G * (DH + 2);
    if constexpr (SERIAL) {
        const RowId r = row_of(rr, il, (int)blockIdx.x);
        const int g = blockIdx.y;
        const float* __restrict__ st = state + ((int64_t)r.irow * n_kv + g) * STATE_F;
        const int64_t slot = idx_rows * n_kv * STATE_F;
        const int d = threadIdx.x;
        const int k_eff = clamp_budget(kt[r.irow], k_max), np = k_eff > 0 ? parts_of(k_eff, max_parts) : 0;
        float acc[G], mx[G], den[G];
#pragma unroll
        for (int e = 0; e < G; ++e) { acc[e] = 0.f; den[e] = 0.f; mx[e] = -INFINITY; }
        for (int p = 0; p < np; ++p)
#pragma unroll
            for (int e = 0; e < G; ++e) mx[e] = fmaxf(mx[e], st[p * slot + G * DH + e]);
        for (int p = 0; p < np; ++p)
#pragma unroll
            for (int e = 0; e < G; ++e) {
                const float m = st[p * slot + G * DH + e], sc = m == -INFINITY ? 0.f : exp2f(m - mx[e]);
                acc[e] = fmaf(sc, st[p * slot + d * G + e], acc[e]);
                den[e] = fmaf(sc, st[p * slot + G * DH + G + e], den[e]);
            }
#pragma unroll
        for (int e = 0; e < G; ++e) {
            const size_t at = (((size_t)r.b * Lq + r.t) * n_h + g * G + e) * DH + d;
            out[at] = __float2bfloat16_rn(den[e] != 0.f ? acc[e] / den[e] * fast_sigmoid(__bfloat162float(g1[at])) : 0.f);
            if (lse && d == 0) lse[((size_t)r.b * Lq + r.t) * n_h + g * G + e] = (mx[e] + log2f(den[e])) * 0.6931471805599453f;
        }
        return;
    }
    const int rows = rr.rows();
    if (mode == 0) {
        const int lr0 = blockIdx.x * kFinRows;
        // thread = (KV head, two consecutive d): 2 G consecutive floats of the state, bf16 pairs of g1 and out
        for (int i = threadIdx.x; i < n_kv * (DH / 2); i += blockDim.x) {
            const int d = (i % (DH / 2)) * 2;
            const int g = i / (DH / 2);
            float o[kFinRows][2 * G], l[kFinRows][G];
            __nv_bfloat162 gl[kFinRows][G];
            int keff[kFinRows];
            size_t at0[kFinRows];
#pragma unroll
            for (int q = 0; q < kFinRows; ++q) {
                const int lr = min(lr0 + q, rows - 1);
                const RowId r = row_of(rr, il, lr);
                const float* st = state + ((int64_t)r.irow * n_kv + g) * STATE_F;
                keff[q] = kt[r.irow];
                at0[q] = (((size_t)r.b * Lq + r.t) * n_h + g * G) * DH + d;
                if constexpr (G == 1) {
                    const float2 v = *reinterpret_cast<const float2*>(st + d);
                    o[q][0] = v.x; o[q][1] = v.y;
                } else {
#pragma unroll
                    for (int c = 0; c < 2 * G / 4; ++c) {
                        const float4 v = *reinterpret_cast<const float4*>(st + d * G + 4 * c);
                        o[q][4 * c] = v.x; o[q][4 * c + 1] = v.y; o[q][4 * c + 2] = v.z; o[q][4 * c + 3] = v.w;
                    }
                }
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    l[q][e] = st[G * DH + G + e];
                    gl[q][e] = *reinterpret_cast<const __nv_bfloat162*>(g1 + at0[q] + (size_t)e * DH);
                }
            }
#pragma unroll
            for (int q = 0; q < kFinRows; ++q) {
                if (lr0 + q >= rows) break;
#pragma unroll
                for (int e = 0; e < G; ++e) {
                    const bool live = keff[q] > 0 && l[q][e] != 0.f;      // (a NaN in a selected key shows)
                    const float2 gf = __bfloat1622float2(gl[q][e]);
                    const float v0 = live ? o[q][e] / l[q][e] * fast_sigmoid(gf.x) : 0.f;          // (d, head e)
                    const float v1 = live ? o[q][G + e] / l[q][e] * fast_sigmoid(gf.y) : 0.f;      // (d + 1, head e)
                    *reinterpret_cast<__nv_bfloat162*>(out + at0[q] + (size_t)e * DH) = __floats2bfloat162_rn(v0, v1);
                    if (lse && d == 0) {               // the running maximum sits in front of the sums (log2 domain)
                        const RowId r = row_of(rr, il, lr0 + q);
                        const float m = state[((int64_t)r.irow * n_kv + g) * STATE_F + G * DH + e];
                        lse[((size_t)r.b * Lq + r.t) * n_h + g * G + e] = (m + log2f(l[q][e])) * 0.6931471805599453f;
                    }
                }
            }
        }
        return;
    }
    __shared__ float s_m[kMaxParts * G], s_l[kMaxParts * G], s_top[G], s_den[G], s_acc[kFinGroups][G][DH];
    const int tid = threadIdx.x, d = tid % DH, grp = tid / DH, warp = tid >> 5, lane = tid & 31;
    const RowId r = row_of(rr, il, (int)blockIdx.x);
    const int g = blockIdx.y;
    const float* __restrict__ st = state + ((int64_t)r.irow * n_kv + g) * STATE_F;
    const int64_t slot = idx_rows * n_kv * STATE_F;
    // everything that does not depend on another load goes out at once: the budget, every slot's statistics and this thread's share of
    // the first slots' sums, also of slots that the row does not use (the workspace holds them; their weight stays out of the sums)
    constexpr int AHEAD = G <= 2 ? 4 : (G == 4 ? 2 : 1);
    float first[AHEAD][G];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u)
#pragma unroll
        for (int e = 0; e < G; ++e) first[u][e] = grp + u * kFinGroups < max_parts ? st[(grp + u * kFinGroups) * slot + d * G + e] : 0.f;
    const int k_eff = clamp_budget(kt[r.irow], k_max), np = k_eff > 0 ? parts_of(k_eff, max_parts) : 0;
    for (int i = tid; i < max_parts * G; i += kFinGroups * DH) {
        s_m[i] = st[(i / G) * slot + G * DH + i % G];
        s_l[i] = st[(i / G) * slot + G * DH + G + i % G];
    }
    __syncthreads();
    static_assert(kFinGroups * DH / 32 >= G, "a warp per head of the group");
    if (warp < G) {                                            // the slots' weights 2^(m_p - M)
        float top = -INFINITY, den = 0.f;
        for (int p = lane; p < np; p += 32) top = fmaxf(top, s_m[p * G + warp]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
        for (int p = lane; p < np; p += 32) {
            const float m = s_m[p * G + warp], sc = m == -INFINITY ? 0.f : exp2f(m - top);
            den = fmaf(sc, s_l[p * G + warp], den);
            s_m[p * G + warp] = sc;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xFFFFFFFFu, den, o);
        if (lane == 0) { s_top[warp] = top; s_den[warp] = den; }
    }
    __syncthreads();
    float acc[G];
#pragma unroll
    for (int e = 0; e < G; ++e) acc[e] = 0.f;
#pragma unroll
    for (int u = 0; u < AHEAD; ++u)
        if (grp + u * kFinGroups < np)
#pragma unroll
            for (int e = 0; e < G; ++e) acc[e] = fmaf(s_m[(grp + u * kFinGroups) * G + e], first[u][e], acc[e]);
#pragma unroll 4
    for (int p = grp + AHEAD * kFinGroups; p < np; p += kFinGroups)
#pragma unroll
        for (int e = 0; e < G; ++e) acc[e] = fmaf(s_m[p * G + e], st[p * slot + d * G + e], acc[e]);
#pragma unroll
    for (int e = 0; e < G; ++e) s_acc[grp][e][d] = acc[e];
    __syncthreads();
    for (int i = tid; i < G * DH; i += kFinGroups * DH) {
        const int e = i / DH, c = i % DH;
        float o = 0.f;
#pragma unroll
        for (int u = 0; u < kFinGroups; ++u) o += s_acc[u][e][c];
        const size_t at = (((size_t)r.b * Lq + r.t) * n_h + g * G + e) * DH + c;
        out[at] = __float2bfloat16_rn(s_den[e] != 0.f ? o / s_den[e] * fast_sigmoid(__bfloat162float(g1[at])) : 0.f);
        if (lse && c == 0) lse[((size_t)r.b * Lq + r.t) * n_h + g * G + e] = (s_top[e] + log2f(s_den[e])) * 0.6931471805599453f;
    }
}

// Eq. 9 as a streaming pre-pass: Vg = bf16(V * sigmoid(g2)), 8 elements per thread.
template <bool WATCH_K>
__global__ void __launch_bounds__(256) gsa_value_gate_kernel(const uint4* __restrict__ V,
                                                             const uint4* __restrict__ g2,
                                                             uint4* __restrict__ Vg, int64_t n_vec,
                                                             int32_t* untileable, const uint4* __restrict__ K) {
    chain_wait();
    uint32_t bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_vec;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint4 vv = __ldg(V + i);
        const uint4 gg = __ldg(g2 + i);
        __nv_bfloat162* v2 = reinterpret_cast<__nv_bfloat162*>(&vv);
        const __nv_bfloat162* g2v = reinterpret_cast<const __nv_bfloat162*>(&gg);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 vf = __bfloat1622float2(v2[e]), gf = __bfloat1622float2(g2v[e]);
            v2[e] = __floats2bfloat162_rn(vf.x * gate_sigmoid(gf.x), vf.y * gate_sigmoid(gf.y));
        }
        Vg[i] = vv;
        bad |= untileable_bf16x8(vv);
        if (WATCH_K) bad |= untileable_bf16x8(__ldg(K + i));
    }
    if (bad && untileable) atomicOr(untileable, kGeneralValues);
}

int g_range_keys = kRangeKeysDefault;

struct AttnPlan {
    int mode;            // 0 ranges, 1 parts
    int n_ranges;        // mode 0
    int slots;
    size_t state_bytes, cuts_bytes;
};

AttnPlan plan_attn(const gsa_params_t& p) {
    AttnPlan pl;
    const int64_t idx_rows = (int64_t)p.B * p.Lq;
    const int G = p.n_h / p.n_kv;
    const size_t row_state = (size_t)p.n_kv * G * (p.d_h + 2) * 4;
    // few rows: split every index set into parallel parts; otherwise one launch per L2-sized key range
    pl.mode = idx_rows * p.n_kv < 2 * (int64_t)sm_count() * kWarpsPrefill ? 1 : 0;
    int nr = (p.Lk + g_range_keys - 1) / g_range_keys;
    if (nr > kMaxRanges) nr = kMaxRanges;
    pl.n_ranges = pl.mode == 0 ? nr : 1;
    // as many segments per index set as fill the GPU's warp slots once: one wave of longer items beat two waves of
    // shorter ones at the decode workload (attention 0.115 against 0.119 ms)
    int mp = (int)(((int64_t)sm_count() * kWarpsPrefill) / (idx_rows * p.n_kv));
    mp = mp < 1 ? 1 : (mp > t_max_parts ? t_max_parts : mp);
    pl.slots = pl.mode == 1 ? mp : 1;
    pl.state_bytes = (size_t)pl.slots * idx_rows * row_state;
    pl.cuts_bytes = pl.mode == 0 && pl.n_ranges > 1 ? (size_t)idx_rows * pl.n_ranges * 4 : 0;
    return pl;
}

template <int DH, int G, bool FUSE_G2>
cudaError_t launch_attn_t(AttnArgs a, const gsa_params_t& p, const AttnPlan& pl, const __nv_bfloat16* g1,
                          __nv_bfloat16* out, int32_t* cuts, cudaStream_t st, AttnProgress* prog) {
    constexpr int VSTAGES = FUSE_G2 ? 2 : kVStages;
    constexpr int kWarpsPerCta = FUSE_G2 ? kWarpsFused : kWarpsPrefill;
    constexpr size_t smem = (size_t)kWarpsPerCta * VSTAGES * kTileKeys * (DH * 2 + 16);
    auto kern = gsa_sparse_attn_kernel<DH, G, FUSE_G2>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 1;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarpsPerCta * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int64_t cap = (int64_t)sm_count() * per_sm;
    const RowRange rr_all = a.rr;
    const int q_end = rr_all.q_begin + rr_all.R;
    const int off = p.Lk - p.Lq;

    if (pl.mode == 0 && pl.n_ranges > 1) {
        const int64_t n = (int64_t)rr_all.rows() * pl.n_ranges;
        launch_chained(gsa_range_cuts_kernel, (unsigned)((n + 255) / 256), 256, 0, st, a.idx, a.kt, cuts, rr_all, a.il, a.k_max,
                       pl.n_ranges, g_range_keys, a.only_if, a.run_if);
        ++g_launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (!a.only_if) timeline_mark(kStageRangeCuts, st);
    }
    a.cuts = cuts;
    a.n_cuts = pl.n_ranges;
    a.mode = pl.mode;
    a.max_parts = pl.slots;
    const int fin_threads = a.n_kv * (DH / 2) < 1024 ? a.n_kv * (DH / 2) : 1024;     // range mode: two d per thread
    // normalise + G1 + bf16 for rows t_lo <= t < t_hi of every batch element, then tell the caller
    auto finalize = [&](int t_lo, int t_hi) -> cudaError_t {
        if (t_hi <= t_lo) return cudaSuccess;
        RowRange fr = rr_all;
        fr.q_begin = t_lo; fr.R = t_hi - t_lo;
        const dim3 fin_grid = pl.mode == 0 ? dim3((unsigned)((fr.rows() + kFinRows - 1) / kFinRows), 1)
                                           : dim3((unsigned)fr.rows(), (unsigned)a.n_kv);
        const bool serial = pl.mode == 1 && finalize_serial(G, pl.slots, parts_of(p.k_max, pl.slots));
        launch_chained(serial ? gsa_attn_finalize_kernel<DH, G, true> : gsa_attn_finalize_kernel<DH, G, false>, fin_grid,
            pl.mode == 0 ? fin_threads : (serial ? DH : kFinGroups * DH), 0, st, a.state, a.kt, g1, out, fr, a.il, a.idx_rows, p.Lq,
            p.n_h, p.n_kv, p.k_max, pl.mode, pl.slots, a.lse, a.only_if, a.run_if);
        ++g_launches;
        cudaError_t fe = cudaGetLastError();
        if (!a.only_if) timeline_mark(kStageFinalize, st);
        if (fe == cudaSuccess && prog && prog->n < prog->cap && prog->n < 64) {
            fe = cudaEventRecord(prog->events[prog->n], st);
            prog->t_lo[prog->n] = t_lo; prog->t_hi[prog->n] = t_hi;
            ++prog->n;
        }
        return fe;
    };
    int finalized_to = rr_all.q_begin;                      // rows below this are final
    for (int rg = 0; rg < pl.n_ranges; ++rg) {
        AttnArgs ar = a;
        ar.range = rg;
        if (pl.mode == 0) {
            // queries that cannot see the range's first key have nothing in it
            const int t_min = rg * g_range_keys - off;
            if (t_min >= q_end) break;
            if (t_min > rr_all.q_begin) { ar.rr.q_begin = t_min; ar.rr.R = q_end - t_min; }
        }
        const int64_t items = (int64_t)ar.rr.rows() * a.n_kv * (pl.mode == 1 ? pl.slots : 1);
        // few items (a small decode step): one SM's share of them per CTA, so that no SM streams for sixteen warps while
        // others have nothing to do (one 32K-token stream, 128 items: 25 -> 5 us)
        const int64_t share = (items + sm_count() - 1) / sm_count();
        const int warps = share < kWarpsPerCta ? (int)share : kWarpsPerCta;
        const int64_t want = (items + warps - 1) / warps;
        const int ctas = (int)(want < cap ? want : cap);
        launch_chained(kern, ctas, warps * 32, smem / kWarpsPerCta * warps, st, ar);
        ++g_launches;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (!a.only_if) timeline_mark(kStageAttn, st);
        if (pl.mode == 0 && rg + 1 < pl.n_ranges) {
            // rows whose last visible key lies in this range are complete
            const int64_t t_done = (int64_t)(rg + 1) * g_range_keys - off;
            const int t_hi = (int)(t_done < finalized_to ? finalized_to : (t_done > q_end ? q_end : t_done));
            if ((e = finalize(finalized_to, t_hi)) != cudaSuccess) return e;
            finalized_to = t_hi;
        }
    }
    return finalize(finalized_to, q_end);
}

// First row from which the gather is the cheaper path (rr.q_begin: all of them; its end: none), from two models in
// microseconds.  Tiles: a CTA takes 2.1 (d_h = 64: 1.9) per key tile of its 256 (row, head) rows and the GPU one CTA per SM,
// plus 10 for the masks, the start and the gather's idle launch behind them (measured at L = 32K and 16K on the kernel of whole tiles; the
// present one takes 1.7, but a line moved by as much lost where it was tried: 128K, ~120K rows on tiles in place of 96896, 93.6 ms
// against 95.1).  Gather: 36 ps (24) per pair
// and KV head, 41 (27) out of several key ranges (measured at L = 16K and 128K for 1, 2, 4 and 8 query heads per KV head),
// and a warp's own chain of 16-key steps where a call has few rows.
struct ForwardCosts {
    double tile_us, pair_us;
    int block;
    double tiles(const gsa_params_t& p, int nb, int q0, int rows, int64_t rows_per_chunk) const {
        if (rows <= 0) return 0.0;
        const RowsWork w = rows_work(p, nb, q0, rows, block);
        const double chunks = (double)((rows + rows_per_chunk - 1) / rows_per_chunk);
        const double all = w.key_tiles * p.n_kv / sm_count(), longest = w.chain * chunks;
        return (all > longest ? all : longest) * tile_us + 10.0;
    }
    double gather(const gsa_params_t& p, const AttnPlan& pl, int nb, int q0, int rows) const {
        if (rows <= 0) return 0.0;
        const RowsWork w = rows_work(p, nb, q0, rows, block);
        const double all = w.selected * p.n_kv * pair_us;
        const double longest = w.selected / ((double)nb * rows) / kTileKeys / (pl.mode == 1 ? pl.slots : 1) * 0.45;
        return (all > longest ? all : longest) + 5.0 + 2.0 * pl.n_ranges;
    }
    // selected pairs of a chunk of rows below which the gather takes less than seven tenths of the tiles' time
    double few_pairs(const gsa_params_t& p, const AttnPlan& pl, int nb, int q0, int rows) const {
        const double us = 0.7 * tiles(p, nb, q0, rows, rows) - 5.0 - 2.0 * pl.n_ranges;
        const double all = us / (p.n_kv * pair_us), longest = us / 0.45 * kTileKeys * (pl.mode == 1 ? pl.slots : 1) * nb * rows;
        return all < longest ? all : longest;
    }
};

ForwardCosts forward_costs(const gsa_params_t& p, const AttnPlan& pl) {
    ForwardCosts c;
    c.block = masked_block_rows(p);
    c.tile_us = p.d_h == 128 ? 2.1 : 1.9;
    c.pair_us = (p.d_h == 128 ? 36e-6 : 24e-6) * (pl.n_ranges > 1 ? 41.0 / 36.0 : 1.0);
    return c;
}

int masked_rows_end(const gsa_params_t& p, const AttnPlan& pl, const RowRange& rr, size_t scratch_bytes) {
    const int q_end = rr.q_begin + rr.R;
    const ForwardCosts c = forward_costs(p, pl);
    const int64_t per = (int64_t)(scratch_bytes / (mask_plan(p, 0, kMaskRowAlign).bytes(p.B) / kMaskRowAlign)) / c.block * c.block;
    if (per < c.block) return rr.q_begin;                          // (no room for the masks of one block of rows)
    // the row that sees so many keys that its share of a block's tiles costs what gathering its set does
    const int64_t k = p.k_mode == 3 ? p.Lk : (p.k_base < p.k_min ? p.k_min : (p.k_base > p.k_max ? p.k_max : p.k_base));
    const double even = (double)k * c.pair_us * sm_count() * kMaskTileKeys * c.block / c.tile_us - (p.Lk - p.Lq);
    int cut = even >= q_end ? q_end : (even <= rr.q_begin ? rr.q_begin : rr.q_begin + ((int)even - rr.q_begin) / c.block * c.block);
    double best = c.gather(p, pl, rr.nb, rr.q_begin, rr.R);
    int t_end = rr.q_begin;
    for (const int t : {cut, q_end}) {
        const double us = c.tiles(p, rr.nb, rr.q_begin, t - rr.q_begin, per) + c.gather(p, pl, rr.nb, t, q_end - t);
        if (us < best) { best = us; t_end = t; }
    }
    return t_end;
}

template <int DH, bool FUSE_G2>
cudaError_t launch_attn_g(const AttnArgs& a, const gsa_params_t& p, const AttnPlan& pl, const __nv_bfloat16* g1,
                          __nv_bfloat16* out, int32_t* cuts, int G, cudaStream_t st, AttnProgress* prog) {
    switch (G) {
        case 1: return launch_attn_t<DH, 1, FUSE_G2>(a, p, pl, g1, out, cuts, st, prog);
        case 2: return launch_attn_t<DH, 2, FUSE_G2>(a, p, pl, g1, out, cuts, st, prog);
        case 4: return launch_attn_t<DH, 4, FUSE_G2>(a, p, pl, g1, out, cuts, st, prog);
        case 8: return launch_attn_t<DH, 8, FUSE_G2>(a, p, pl, g1, out, cuts, st, prog);
    }
    return cudaErrorInvalidValue;
}

// (the cuts lie behind the state)
template <bool FUSE_G2>
cudaError_t launch_attn_dh(const AttnArgs& a, const gsa_params_t& p, const AttnPlan& pl, const __nv_bfloat16* g1, __nv_bfloat16* out,
                           cudaStream_t st, AttnProgress* prog) {
    int32_t* cuts = reinterpret_cast<int32_t*>((char*)a.state + (pl.state_bytes + 255) / 256 * 256);
    const int G = p.n_h / p.n_kv;
    if (p.d_h == 128) return launch_attn_g<128, FUSE_G2>(a, p, pl, g1, out, cuts, G, st, prog);
    if (p.d_h == 64) return launch_attn_g<64, FUSE_G2>(a, p, pl, g1, out, cuts, G, st, prog);
    return cudaErrorInvalidValue;
}

AttnArgs attn_args(const gsa_params_t& p, const AttnPlan& pl, const RowRange& rr, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                   const __nv_bfloat16* V, const __nv_bfloat16* g2, const int32_t* idx, const int32_t* kt, IdxLayout il,
                   void* scratch, float* lse) {
    AttnArgs a;
    a.lse = lse;
    a.dev_status = t_dev_status;
    a.Q = Q; a.K = K; a.V = V; a.g2 = g2; a.idx = idx; a.kt = kt;
    a.state = reinterpret_cast<float*>(scratch);
    a.cuts = nullptr;
    a.rr = rr; a.il = il; a.idx_rows = (int64_t)p.B * p.Lq;
    a.Lq = p.Lq; a.Lk = p.Lk; a.n_h = p.n_h; a.n_kv = p.n_kv; a.k_max = p.k_max;
    a.mode = pl.mode; a.max_parts = pl.slots; a.range = 0; a.n_cuts = pl.n_ranges;
    const float sc = p.sm_scale > 0.f ? p.sm_scale : 1.0f / sqrtf((float)p.d_h);
    a.scale_log2 = sc * 1.4426950408889634f;
    a.only_if = nullptr; a.run_if = 0; a.g1 = nullptr; a.out = nullptr;
    return a;
}

template <int DH, int G>
cudaError_t launch_direct_t(const AttnArgs& a, cudaStream_t st) {
    constexpr int smem = kWarpsPrefill * kVStages * kTileKeys * (DH * 2 + 16);
    auto kern = gsa_sparse_attn_kernel<DH, G, false, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int64_t want = ((int64_t)a.rr.rows() * a.n_kv + kWarpsPrefill - 1) / kWarpsPrefill;
    launch_chained(kern, (unsigned)(want < sm_count() ? want : sm_count()), kWarpsPrefill * 32, smem, st, a);
    ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_masked_rows(const gsa_params_t& p, const AttnPlan& pl, const RowRange& rr, int t_end, const __nv_bfloat16* Q,
                               const __nv_bfloat16* K, const __nv_bfloat16* Vg, const __nv_bfloat16* g1, const int32_t* idx,
                               const int32_t* kt, IdxLayout il, __nv_bfloat16* out, void* scratch, size_t scratch_bytes,
                               cudaStream_t st, AttnProgress* prog, float* lse, bool all_visible) {
    const int block = masked_block_rows(p);
    const size_t row_bytes = mask_plan(p, 0, kMaskRowAlign).bytes(p.B) / kMaskRowAlign;
    int64_t per = (int64_t)(scratch_bytes / row_bytes) / block * block;
    if (per < block) return cudaErrorInvalidValue;
    int32_t* const general = t_dev_status + kStatusGeneralWord;
    const ForwardCosts costs = forward_costs(p, pl);
    for (int q = rr.q_begin; q < t_end; q += (int)per) {
        const MaskPlan mp = mask_plan(p, q, (int)(t_end - q < per ? t_end - q : per));
        cudaError_t e = all_visible ? launch_visible_masks(p, mp, (uint4*)scratch, st)
                                    : launch_build_masks(p, mp, block, idx, kt, il, (uint4*)scratch, t_dev_status,
                                                         costs.few_pairs(p, pl, rr.nb, q, mp.rows), st);
        if (e != cudaSuccess) return e;
        e = launch_masked_attn_fwd(p, mp, (const uint4*)scratch, Q, K, Vg, g1, out, lse, t_dev_status, st);
        if (e != cudaSuccess) return e;
        // What the tiles have left: the gather, key range by key range if the sets are in order, else whole sets at once.
        RowRange chunk = rr;
        chunk.q_begin = q; chunk.R = mp.rows;
        const bool ranges = pl.mode == 0 && pl.n_ranges > 1;
        e = launch_attn_direct(p, chunk, Q, K, Vg, g1, idx, kt, il, out, lse, general, ranges ? kRunGeneralSets : kRunAnyGeneral, st);
        if (e == cudaSuccess && ranges) {
            AttnArgs a = attn_args(p, pl, chunk, Q, K, Vg, nullptr, idx, kt, il, scratch, lse);
            a.only_if = general; a.run_if = kRunSetsInOrder;
            e = launch_attn_dh<false>(a, p, pl, g1, out, st, nullptr);
        }
        if (e != cudaSuccess) return e;
        timeline_mark(kStageTiles, st);
        if (prog && prog->n < prog->cap && prog->n < 64) {
            if ((e = cudaEventRecord(prog->events[prog->n], st)) != cudaSuccess) return e;
            prog->t_lo[prog->n] = q; prog->t_hi[prog->n] = q + mp.rows;
            ++prog->n;
        }
    }
    return cudaSuccess;
}

}  // namespace

thread_local int t_max_parts = kMaxParts;

size_t attn_scratch_bytes(const gsa_params_t& p) {
    const AttnPlan pl = plan_attn(p);
    return (pl.state_bytes + 255) / 256 * 256 + (pl.cuts_bytes + 255) / 256 * 256;
}

void set_attn_range_keys(int keys) { g_range_keys = keys >= 1024 ? keys : kRangeKeysDefault; }
int attn_range_keys() { return g_range_keys; }

cudaError_t launch_attn_direct(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                               const __nv_bfloat16* Vg, const __nv_bfloat16* g1, const int32_t* idx, const int32_t* kt, IdxLayout il,
                               __nv_bfloat16* out, float* lse, const int32_t* only_if, int32_t run_if, cudaStream_t st) {
    AttnArgs a = attn_args(p, plan_attn(p), rr, Q, K, Vg, nullptr, idx, kt, il, nullptr, lse);
    a.only_if = only_if; a.run_if = run_if; a.g1 = g1; a.out = out;
    const int G = p.n_h / p.n_kv;
#define GSA_CASE(DH_, G_) if (p.d_h == DH_ && G == G_) return launch_direct_t<DH_, G_>(a, st)
    GSA_CASE(128, 1); GSA_CASE(128, 2); GSA_CASE(128, 4); GSA_CASE(128, 8);
    GSA_CASE(64, 1); GSA_CASE(64, 2); GSA_CASE(64, 4); GSA_CASE(64, 8);
#undef GSA_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_value_gate(const __nv_bfloat16* V, const __nv_bfloat16* g2, __nv_bfloat16* Vg,
                              int64_t n_elems, cudaStream_t st, int32_t* untileable, const __nv_bfloat16* K) {
    const int64_t n_vec = n_elems / 8;
    if (n_vec <= 0) return cudaSuccess;
    const int blocks = (int)((n_vec + 255) / 256 < sm_count() * 16 ? (n_vec + 255) / 256 : sm_count() * 16);
    launch_chained(K ? gsa_value_gate_kernel<true> : gsa_value_gate_kernel<false>, blocks, 256, 0, st, reinterpret_cast<const uint4*>(V),
                                                  reinterpret_cast<const uint4*>(g2),
                                                  reinterpret_cast<uint4*>(Vg), n_vec, untileable,
                                                  reinterpret_cast<const uint4*>(K));
    ++g_launches;
    return cudaGetLastError();
}

int attn_tile_rows(const gsa_params_t& p, RowRange rr) {
    const AttnPlan pl = plan_attn(p);
    return masked_rows_end(p, pl, rr, (pl.state_bytes + 255) / 256 * 256 + pl.cuts_bytes) - rr.q_begin;
}

cudaError_t launch_sparse_attn(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* Q,
                               const __nv_bfloat16* K, const __nv_bfloat16* V,
                               const __nv_bfloat16* g1, const __nv_bfloat16* g2, const int32_t* idx,
                               const int32_t* kt, IdxLayout il, __nv_bfloat16* out, void* scratch,
                               cudaStream_t st, AttnProgress* progress, float* lse, bool values_scanned,
                               bool all_visible) {
    if (rr.rows() <= 0) return cudaSuccess;
    const AttnPlan pl = plan_attn(p);
    const size_t scratch_bytes = (pl.state_bytes + 255) / 256 * 256 + pl.cuts_bytes;
    if (!g2 && t_dev_status) {
        // rows whose sets hold a large enough share of what they see: masked tiles, in chunks whose masks fit the scratch
        const int t_end = masked_rows_end(p, pl, rr, scratch_bytes);
        if (t_end > rr.q_begin) {
            cudaError_t e = cudaSuccess;
            if (!values_scanned)
                e = launch_check_values(V, (int64_t)p.B * p.Lk * p.n_kv * p.d_h, t_dev_status + kStatusGeneralWord, st);
            if (e != cudaSuccess) return e;
            e = launch_masked_rows(p, pl, rr, t_end, Q, K, V, g1, idx, kt, il, out, scratch, scratch_bytes, st,
                                   progress, lse, all_visible);
            if (e != cudaSuccess || t_end >= rr.q_begin + rr.R) return e;
            rr.R = rr.q_begin + rr.R - t_end;
            rr.q_begin = t_end;
        }
    }
    const AttnArgs a = attn_args(p, pl, rr, Q, K, V, g2, idx, kt, il, scratch, lse);
    return g2 ? launch_attn_dh<true>(a, p, pl, g1, out, st, progress) : launch_attn_dh<false>(a, p, pl, g1, out, st, progress);
}

}  // namespace gsa
