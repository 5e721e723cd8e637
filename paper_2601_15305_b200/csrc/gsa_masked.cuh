// Masked tiles: the attention stage as dense 128-row x 128-key tiles on the 5th-generation tensor cores, with the
// index sets S_t as bit masks.  Shared by the forward (gsa_masked_attn.cu) and backward kernels.
//
// Why: the gather kernels move n_kv * d_h * 4 bytes per selected (query, key) pair through the L2 (0.30 ns per pair
// and forward at 16 heads of 128), a tile costs 4 * d_h flops per (query, key, head) whether selected or not.  Once
// more than a few per cent of the visible keys are selected the tensor cores win.
//
// Mask layout: one uint4 (128 bits, bit k of word w = key 32 w + k of the tile) per (batch element, key tile, query
// row): mask[(b * n_key_tiles + tile) * row_pitch + row], so that the threads of a tile (consecutive rows) read
// consecutive 16-byte pieces.
#pragma once

#include "gsa_common.cuh"
#include "gsa_tc.cuh"

namespace gsa {

constexpr int kMaskTileKeys = 128;
constexpr int kMaskRowAlign = 8;           // row_pitch is a multiple of this (rows a mask-building CTA handles)

struct MaskPlan {
    int32_t q0, rows;          // query rows q0 .. q0 + rows - 1 of every batch element
    int32_t row_pitch;         // rows rounded up to kMaskRowAlign
    int32_t key_tiles;         // ceil(Lk / 128)
    size_t bytes(int B) const { return (size_t)B * key_tiles * row_pitch * 16; }
};

inline MaskPlan mask_plan(const gsa_params_t& p, int q0, int rows) {
    MaskPlan m;
    m.q0 = q0; m.rows = rows;
    m.row_pitch = (rows + kMaskRowAlign - 1) / kMaskRowAlign * kMaskRowAlign;
    m.key_tiles = (p.Lk + kMaskTileKeys - 1) / kMaskTileKeys;
    return m;
}

// Builds the masks of rows mp.q0 .. of every batch element.  Row r gets the key tiles that the last row of its block
// of `block_rows` rows (counted from mp.q0) can see.  A set that a mask cannot stand for (not strictly ascending, an
// entry that the row cannot see, a budget out of range) raises a bit of the `general` word; so do sets of fewer than few_pairs
// entries in all (another bit, put down again by the next chunk's masks).
cudaError_t launch_build_masks(const gsa_params_t& p, const MaskPlan& mp, int block_rows, const int32_t* idx,
                               const int32_t* kt, IdxLayout il, uint4* mask, int32_t* dev_status, double few_pairs, cudaStream_t st);

// The same for sets known to hold every visible key (k_mode 3 inside gsa_forward): no set is read.
cudaError_t launch_visible_masks(const gsa_params_t& p, const MaskPlan& mp, uint4* mask, cudaStream_t st);

// Raises *general if one of n_elems (a multiple of 8) values is infinite, NaN or too large (untileable_bf16x8).
cudaError_t launch_check_values(const __nv_bfloat16* x, int64_t n_elems, int32_t* general, cudaStream_t st);

// What a range of rows sees and selects, per KV head: for the choice between the tiles and the gather.  The sets' sizes are on
// the device; the budget that they centre on stands for them.
struct RowsWork {
    double key_tiles;          // key tiles of the blocks of `block` rows, all batch elements
    double chain;              // ... of the last block
    double selected;           // selected (row, key) pairs, all batch elements
};
inline RowsWork rows_work(const gsa_params_t& p, int nb, int q0, int rows, int block) {
    const double first = (double)p.Lk - p.Lq + q0 + 1, last = first + rows - 1;        // keys the first and the last row see
    const int64_t k64 = p.k_mode == 3 ? p.Lk : (p.k_base < p.k_min ? p.k_min : (p.k_base > p.k_max ? p.k_max : p.k_base));
    const double k = (double)k64;
    RowsWork w;
    const double blocks = (double)((rows + block - 1) / block);
    w.chain = last / kMaskTileKeys + 1.0;
    w.key_tiles = nb * blocks * (0.5 * (first + last) / kMaskTileKeys + 0.5 * block / kMaskTileKeys + 0.5);
    if (w.key_tiles > nb * blocks * w.chain) w.key_tiles = nb * blocks * w.chain;
    const double short_rows = k <= first ? 0.0 : (k >= last ? rows : k - first);      // rows that see fewer keys than the budget
    w.selected = nb * (short_rows * (first + 0.5 * short_rows) + (rows - short_rows) * k);
    return w;
}

// query rows of a forward CTA (two M = 128 tiles of (query, head of the group) rows)
inline int masked_block_rows(const gsa_params_t& p) { return 256 / (p.n_h / p.n_kv); }

// Order of a tile kernel's CTAs: the longest blocks first, of as many (batch element, KV head) pairs abreast as have the tensors
// that their CTAs stream together in the L2.  One pair after another leaves the last wave to long blocks (8K prefill 319 us of
// tiles against 276 with all eight heads abreast, dense 2 x 3072 135 against 113); all pairs abreast at every length reads from
// HBM what the L2 would have had (128K prefill 93.4 ms in all against 94.7, training step of 32K 31.3 against 31.7).  The groups are
// of one size: a last group of one pair runs its long blocks alone (8K backward keys kernel, seven pairs and one, 552 us; all eight,
// whose Q and do are 67 MB, 426; forward at 16K, seven and one, 985, four and four 879).
inline int pairs_abreast(int pairs, double bytes_each) {
    const int fit = 80e6 > bytes_each ? (int)(80e6 / bytes_each) : 1;
    const int groups = (pairs + fit - 1) / fit;                   // (of one size, so that the last one is no straggler)
    return (pairs + groups - 1) / groups;
}
__device__ __forceinline__ void tile_order(int item, int blocks, int pairs, int abreast, int* block_rank, int* pair) {
    const int group = item / (abreast * blocks), rest = item - group * abreast * blocks, n = min(abreast, pairs - group * abreast);
    *block_rank = rest / n;
    *pair = group * abreast + rest % n;
}

// Attention of the rows of mp.  dev_status: the call's status head, whose `general` word says whether the tiles may be
// used (the masks and the scan of the values come first on the stream); if not, the launch leaves the rows to the gather.
cudaError_t launch_masked_attn_fwd(const gsa_params_t& p, const MaskPlan& mp, const uint4* mask, const __nv_bfloat16* Q,
                                   const __nv_bfloat16* K, const __nv_bfloat16* Vg, const __nv_bfloat16* g1,
                                   __nv_bfloat16* out, float* lse, int32_t* dev_status, cudaStream_t st);

// The gather over whole sets in one launch (gsa_attn.cu), run if the word at only_if is one that run_if names (left_out).
cudaError_t launch_attn_direct(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                               const __nv_bfloat16* Vg, const __nv_bfloat16* g1, const int32_t* idx, const int32_t* kt, IdxLayout il,
                               __nv_bfloat16* out, float* lse, const int32_t* only_if, int32_t run_if, cudaStream_t st);

// What the backward's tiles leave to the gather (gsa_attn_bwd.cu, gsa_attn_bwd_keys.cu), run if *general is raised: dQ (and pbar,
// lse2); then dK, dV, dg2 from the sets inverted inside ws (attn_bwd_keys_general_bytes), whose first attn_bwd_keys_general_zero
// bytes the tile kernels clear when they leave.
cudaError_t launch_attn_bwd_rows_general(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                                         const __nv_bfloat16* Vg, const __nv_bfloat16* dOs, const int32_t* idx, const int32_t* kt,
                                         IdxLayout il, __nv_bfloat16* dQ, float* lse2, const float* delta, float* pbar,
                                         const float* lse_in, const int32_t* general, cudaStream_t st);
size_t attn_bwd_keys_general_bytes(const gsa_params_t& p, int32_t rows_per_batch);
size_t attn_bwd_keys_general_zero(const gsa_params_t& p, int32_t rows_per_batch);
cudaError_t launch_attn_bwd_keys_general(const gsa_params_t& p, RowRange rr, const __nv_bfloat16* Q, const __nv_bfloat16* dOs,
                                         const __nv_bfloat16* K, const __nv_bfloat16* V, const __nv_bfloat16* Vg,
                                         const __nv_bfloat16* g2, const float* lse2, const float* delta, const int32_t* idx,
                                         const int32_t* kt, IdxLayout il, void* ws, __nv_bfloat16* dK, __nv_bfloat16* dV,
                                         __nv_bfloat16* dg2, const int32_t* general, cudaStream_t st);

// Backward (gsa_masked_bwd.cu): all gradients of the attention stage and the target of the indexer's loss (pbar, zeroed by
// the caller; may be null).  V: as given, Vg: gated; it and K have been watched (launch_value_gate).  ws: masked_bwd_bytes(p, rr) bytes.
bool masked_bwd_preferred(const gsa_params_t& p, const RowRange& rr);
size_t masked_bwd_bytes(const gsa_params_t& p, const RowRange& rr);
cudaError_t launch_masked_bwd(const gsa_params_t& p, const RowRange& rr, const __nv_bfloat16* Q, const __nv_bfloat16* K,
                              const __nv_bfloat16* V, const __nv_bfloat16* Vg, const __nv_bfloat16* g1, const __nv_bfloat16* g2,
                              const __nv_bfloat16* out, const __nv_bfloat16* dout, const int32_t* idx, const int32_t* kt,
                              IdxLayout il, __nv_bfloat16* dQ, __nv_bfloat16* dK, __nv_bfloat16* dV, __nv_bfloat16* dg1,
                              __nv_bfloat16* dg2, __nv_bfloat16* dOs, float* lse_ws, float* delta, float* pbar,
                              const float* lse_in /*nullable*/, void* ws, int32_t* dev_status, cudaStream_t st);

// ---- device helpers --------------------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_tile(uint32_t dst, const CUtensorMap* tm, int d, int head, int token, int b, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(tm), "r"(d), "r"(head), "r"(token), "r"(b), "r"(bar)
        : "memory");
}

// a box of a tile from shared memory to the tensor (what lies outside it is clipped); the issuing thread waits at the end
__device__ __forceinline__ void tma_store_tile(const CUtensorMap* tm, int d, int head, int token, int b, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
                 ::"l"(tm), "r"(d), "r"(head), "r"(token), "r"(b), "r"(src) : "memory");
}
__device__ __forceinline__ void tma_store_wait() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// behind a thread's stores of results into shared memory: meets the others of the named barrier; true if all of them are ok
__device__ __forceinline__ bool tile_results_written(int barrier, int threads, bool ok) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    uint32_t all;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(all) : "r"((uint32_t)ok), "r"(barrier), "r"(threads) : "memory");
    return all != 0;
}

// Start of a tile kernel: false if the call's inputs rule the tiles out (the gather does the work; the same for every
// thread).  *timed_out: an earlier CTA or launch of the call gave up on a wait (may differ between threads: use one's).
__device__ __forceinline__ bool tiles_allowed(const int32_t* dev_status, int* timed_out) {
    const int32_t st = *reinterpret_cast<const volatile int32_t*>(dev_status);
    *timed_out = st >= kDevTimeoutTma && st <= kDevTimeoutEpi;
    return *reinterpret_cast<const volatile int32_t*>(dev_status + kStatusGeneralWord) == 0;
}
// The MMA warp runs converged and one elected lane issues: descriptors then stay in uniform registers.  (A single lane in
// a branch of its own has to move every operand of every instruction there first, which cost more than
// a product of M = N = 128, K = 16 takes (64 cycles).  Backward at L = 32K: keys kernel 6.6 -> 6.1 ms, rows 5.7 -> 5.3 ms.)
__device__ __forceinline__ uint32_t elect_lane() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, long long limit) {
    const bool ok = __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag, limit));
    tc_fence_after();
    return ok;
}
__device__ __forceinline__ void warp_mma_ss(uint32_t elected, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(elected)
        : "memory");
}
// A operand in TMEM (bf16 pairs, one 32-bit column per two contraction elements), B in shared memory
__device__ __forceinline__ void warp_mma_ts(uint32_t elected, uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.ne.b32 e, %5, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(elected)
        : "memory");
}
__device__ __forceinline__ void warp_commit(uint32_t elected, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "setp.ne.b32 e, %1, 0;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        ::"r"(bar), "r"(elected)
        : "memory");
}

#define GSA_R32_OUT(r)                                                                                              \
    "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),    \
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),     \
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),    \
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
#define GSA_R32_TIE(r)                                                                                              \
    "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),    \
        "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),     \
        "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),    \
        "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])

// 32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
        "%29,%30,%31}, [%32];"
        : GSA_R32_OUT(r)
        : "r"(taddr)
        : "memory");
}
// waits for every tcgen05.ld of this thread; the registers of r may be used from here on
__device__ __forceinline__ void tc_wait_ld32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : GSA_R32_TIE(r) : : "memory");
}
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};"
        ::"r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
        "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// shared-memory descriptor of a [contraction rows][64-column chunks] operand tile whose 128-byte rows run along the
// M / N dimension ("MN-major", 128-byte swizzle): 8-row groups 1024 bytes apart, 64-column chunks chunk_bytes apart
__device__ __forceinline__ uint64_t make_mnmajor_desc(uint32_t smem_addr, uint32_t chunk_bytes) {
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(chunk_bytes >> 4) << 16;                           // leading byte offset: next 64 of M / N
    d |= (uint64_t)(1024u >> 4) << 32;                                 // stride byte offset: next 8 contraction rows
    d |= 1ull << 46;
    d |= 2ull << 61;                                                   // SWIZZLE_128B
    return d;
}
constexpr uint32_t kIdescTransA = 1u << 15, kIdescTransB = 1u << 16;   // operand is MN-major

__device__ __forceinline__ uint64_t pack_f32x2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(__float_as_uint(a)), "r"(__float_as_uint(b)));
    return r;
}
__device__ __forceinline__ void unpack_f32x2(uint64_t v, float& a, float& b) {
    uint32_t x, y;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(x), "=r"(y) : "l"(v));
    a = __uint_as_float(x); b = __uint_as_float(y);
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// batch x tokens x heads x d_h bf16 (row-major, batch_stride tokens from one batch element to the next); box = tokens_box x
// heads_box x 64 values (one 128-byte swizzle span).  Tokens past a batch element's last read as zero.
inline bool make_heads_tmap(CUtensorMap* tm, const void* base, uint64_t batch, uint64_t batch_stride, uint64_t tokens,
                            uint64_t heads, uint64_t d_h, uint32_t tokens_box, uint32_t heads_box) {
    auto fn = get_encode_fn();
    if (!fn) return false;
    cuuint64_t dims[4] = {(cuuint64_t)d_h, (cuuint64_t)heads, (cuuint64_t)tokens, (cuuint64_t)batch};
    cuuint64_t strides[3] = {(cuuint64_t)d_h * 2, (cuuint64_t)(heads * d_h) * 2, (cuuint64_t)(batch_stride * heads * d_h) * 2};
    cuuint32_t box[4] = {64u, heads_box, tokens_box, 1u};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace gsa
