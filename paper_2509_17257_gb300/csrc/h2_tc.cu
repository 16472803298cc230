// Tensor-core (tcgen05) kernels of the BF16 and FP32 products: the coupling phase
// (ŷ_t = Σ_{b∈C_t} S_b x̂_s, Sec. 3 Alg. "list_addeval" over the row-cluster
// lists of Alg. "prepare_addeval") and the leaf phase (Y|_t̂ += α(V_t ŷ_t +
// Σ_{b∈L-} G_b X|_ŝ + σ X|_t̂), Alg. "fast_addeval" inadmissible part + the
// backward transformation at the leaves), with the k×m coefficient blocks of
// Sec. 4.
//
// Formulation: every product is computed transposed, Dᵀ = Σ Aᵀ Bᵀ, so that the
// right-hand-side columns are the MMA rows (M) and the matrices (S_b, G_b, V_t)
// are the B operand in their natural row-major orientation:
//   D[r, n] = Σ_k act[r, k] · mat[n, k]
// act rows r = 2i + h hold column i of x̂ / X / ŷ split into a BF16 high part
// (h = 0) and the BF16 rounding remainder (h = 1); the two rows are added in
// the epilogue (adjacent TMEM lanes, one shuffle).  The matrices are stored in
// HBM once, in BF16, already in the tcgen05 "no swizzle, K-major" core-matrix
// order (8 rows × 16 bytes per core matrix, row groups outermost), so one bulk
// copy per tile lands it in shared memory ready for the MMA.
//
// The FP32 product (KIND 1) runs the same schedule on the TF32 units with
// split operands: the activation rows carry x and x - tf32(x), the matrix tiles
// are stored in FP32, and the splitter warps write each tile B together with
// its remainder B_lo = B - tf32(B) into TMEM, so A_hi·B + A_hi·B_lo + A_lo·B +
// A_lo·B_lo keeps FP32 accuracy ("3xTF32", the A_lo·B_lo term comes free with
// the row split).  Its MMA runs the other way round, D[n, r] = Σ_k [B; B_lo][n, k]
// · act[r, k] with M = 128 ([B; B_lo], the A operand in TMEM) and N = R: a
// tcgen05 MMA takes time in proportion to N and the same time for M = 64 as for
// M = 128, so B_lo rides along in M at no cost.
//
// Kernel roles (one persistent CTA per SM, or two with at most 32 columns; 7 warps
// for KIND 0, 12 for KIND 1):
//   warp 0, last    bulk-copy producers (cp.async.bulk + mbarrier complete_tx), one
//                   for the even stages and one for the odd
//   warp 1          TMEM owner and MMA issuer (tcgen05.mma kind::f16 or
//                   kind::tf32, FP32 accumulate): KIND 0 all terms, KIND 1 the
//                   even terms; the converged warp runs the loop and elect.sync
//                   issues, which keeps its operands warp-uniform
//   warps 2..5      epilogue (tcgen05.ld, hi+lo combine, stores)
//   warps 6..9      KIND 1 only: the splitter, [B; B_lo] into TMEM
//   warp 10         KIND 1 only: MMA issuer of the odd terms
// KIND 1: every term accumulates in its own TMEM buffer (round robin over the
// accumulators), so the epilogue's FP32 sum of earlier terms overlaps the MMAs
// of the next ones and keeps FP32 accuracy.  KIND 0 (BF16): all terms of an
// item accumulate in one buffer, read once per item.  Every wait is bounded; on a timeout the kernel raises an
// error flag, drains its own copies and MMAs, frees TMEM and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "h2_async.cuh"
#include "h2_internal.cuh"

namespace h2 {

namespace {

constexpr int kMaxStages = 16, kMaxStagesNarrow = 6;
constexpr int kSmemBudget = 225 * 1024;  // dynamic shared memory per CTA (one CTA per SM)
// NARROW instances (R <= 64 activation rows): two CTAs per SM.  Of an SM's 228 KiB
// each CTA's 1 KiB reserve and about 0.7 KiB of static shared memory come off.
constexpr int kSmemBudgetNarrow = 228 * 1024 / 2 - 1024 - 768;
constexpr int kSplitWarps = 4;  // KIND 1: warps 6..9 write [B; B_lo] into TMEM, one lane quadrant each
// warps: 0 and the last producers (even and odd stages), 1 and KIND 1's issuer2 MMA
// issuers (even and odd terms), 2..5 epilogue, KIND 1: 6..9 splitter
template <int KIND>
__host__ __device__ constexpr int tc_issuer2() { return KIND == 1 ? 6 + kSplitWarps : 6; }
template <int KIND>
__host__ __device__ constexpr int tc_producer2() { return KIND == 1 ? tc_issuer2<KIND>() + 1 : 6; }
template <int KIND>
__host__ __device__ constexpr int tc_threads() { return 32 * (tc_producer2<KIND>() + 1); }
constexpr int kAccCols = 64;                // output columns of one term (the matrix tile's rows)
constexpr int kAccBufs = 4;                 // accumulator buffers: MMAs of a term overlap the epilogue of the 3 before
// TF32 epilogue: remainder sums handed over, two items deep (64 rows of 64 columns, NARROW 32)
constexpr int xch_bytes(bool narrow) { return 2 * 64 * (narrow ? 32 : 64) * 4; }
constexpr int kTermBatch = 8;  // terms that a producer reads at once
constexpr int kNodeBytes = 64 * 16;        // MODE 2: the source cluster's nodes, in the stage after its activation tile
// MODE 2: evaluated tiles, two terms deep, rows of 68 floats (16-byte accesses of
// eight consecutive rows touch all 32 banks once)
constexpr int kEvalLd = 68, kEvalBytes = 2 * 64 * kEvalLd * 4;

// Shared-memory matrix descriptor, no swizzle, K-major: LBO = byte distance of
// core matrices adjacent along K, SBO = byte distance of adjacent 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
// Instruction descriptor: FP32 accumulate, A and B K-major, BF16 (KIND 0:
// format 1 of kind::f16) or TF32 (KIND 1: format 2 of kind::tf32).
template <int KIND>
__device__ __forceinline__ uint32_t idesc_for(int M, int N) {
    const uint32_t fmt = KIND == 0 ? 1u : 2u;
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// The MMAs of one term (D = A·Bᵀ, or D += A·Bᵀ when acc != 0) over nk <= 64 / K steps,
// then up to two commits, from a converged warp: one elect.sync hands them to the
// lowest active lane, so every MMA and commit of the warp comes from one thread, as
// tcgen05.commit requires.  One block of code: an elect.sync and fresh descriptors for
// every MMA cost 80 cycles each.  The descriptors move by 256 bytes a step (two core
// matrices along K, 16 in their 16-byte units).  bar2 = 0: one commit.
__device__ __forceinline__ void mma_term_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc, int nk,
                                              uint32_t bar1, uint32_t bar2) {
#define H2_STEP(K_)                                                                        \
    "add.s64 a, a, 16; add.s64 b, b, 16; setp.gt.and.s32 q, %5, " #K_ ", e;\n"             \
    "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
    asm volatile(
        "{ .reg .pred p, e, q, t; .reg .b64 a, b;\n"
        "elect.sync _|e, 0xffffffff;\n"
        "setp.ne.b32 p, %4, 0; setp.ge.s32 t, %5, 0; mov.b64 a, %1; mov.b64 b, %2;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n" H2_STEP(1) H2_STEP(2) H2_STEP(3)
        "setp.ne.and.b32 q, %7, 0, e;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%7]; }" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(nk), "r"(bar1), "r"(bar2)
        : "memory");
#undef H2_STEP
}
// The TF32 MMAs with their A operand (M = 128 rows, K = 8 columns a step) in TMEM at
// column address a, lanes 0..127, from zero; three commits.
__device__ __forceinline__ void mma_term_tf32(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, int nk, uint32_t bar1,
                                              uint32_t bar2, uint32_t bar3) {
#define H2_STEP(K_)                                                                        \
    "add.s32 a, a, 8; add.s64 b, b, 16; setp.gt.and.s32 q, %4, " #K_ ", e;\n"              \
    "@q tcgen05.mma.cta_group::1.kind::tf32 [%0], [a], b, %3, t;\n"
    asm volatile(
        "{ .reg .pred f, e, q, t; .reg .b64 b; .reg .b32 a;\n"
        "elect.sync _|e, 0xffffffff;\n"
        "setp.lt.s32 f, %4, 0; setp.ge.s32 t, %4, 0; mov.b32 a, %1; mov.b64 b, %2;\n"
        "@e tcgen05.mma.cta_group::1.kind::tf32 [%0], [a], b, %3, f;\n" H2_STEP(1) H2_STEP(2) H2_STEP(3) H2_STEP(4)
            H2_STEP(5) H2_STEP(6) H2_STEP(7)
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%5];\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%7]; }" ::"r"(d),
        "r"(a), "l"(b), "r"(idesc), "r"(nk), "r"(bar1), "r"(bar2), "r"(bar3)
        : "memory");
#undef H2_STEP
}
__device__ __forceinline__ void mma_commit_elect(uint64_t* bar) {
    asm volatile(
        "{ .reg .pred e; elect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0]; }" ::"r"(smem_u32(bar))
        : "memory");
}
// One stage from a converged warp (one elected lane): its metadata, the bytes that its
// barrier expects, and the two bulk copies.
__device__ __forceinline__ void stage_copy_elect(uint32_t meta, int m0, int m1, int m2, int m3, uint32_t bar, uint32_t dst_a,
                                                 const void* src_a, uint32_t bytes_a, uint64_t pol_a, uint32_t dst_b,
                                                 const void* src_b, uint32_t bytes_b, uint64_t pol_b) {
    asm volatile(
        "{ .reg .pred e; elect.sync _|e, 0xffffffff;\n"
        "@e st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n"
        "@e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%5], %6;\n"
        "@e cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%7], [%8], %9, [%5], %10;\n"
        "@e cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%11], [%12], %13, [%5], "
        "%14; }" ::"r"(meta),
        "r"(m0), "r"(m1), "r"(m2), "r"(m3), "r"(bar), "r"(bytes_a + bytes_b), "r"(dst_a), "l"(src_a), "r"(bytes_a),
        "l"(pol_a), "r"(dst_b), "l"(src_b), "r"(bytes_b), "l"(pol_b)
        : "memory");
}
// One of two halves of an item's result onto its cleared output: entries i < count at
// out[i·stride], of which those from `real` on are zero (the columns' padding; ROW: out and
// count are multiples of 4 floats, stride is 1).  An addition in memory counts FP32
// subnormals, its result too, as zero (a product whose results are of 1e-38 was off by 14 %
// instead of 6e-4), so it is for values from 2^-100 on: two of them, or one and a smaller
// normal one, differ by a multiple of 2^-124 or more, and a subnormal is less than half of
// the distance from one of them to its neighbours.  A thread with smaller values exchanges:
// the half that finds zero leaves its value, the other one stores the sum of both.  So the
// sum is the rounded one in any order of the halves.  µs, additions of 32 or 64 values one
// by one → this (rows by vectors; BF16, two lanes a column): FP32 n = 6000, q = 4, m = 1:
// 58.7 → 59.7, m = 32: 79.6 → 76.2, m = 64: 101.1 → 96.3; BF16 m = 1: 47.0 → 48.0, m = 32:
// 59.0 → 60.5; n = 4096, m = 32: 50.3 → 48.6.  All by exchange, a round trip for every 16
// values: BF16, n = 4096, m = 32: 63.
template <bool ROW, int N>
__device__ __forceinline__ void add_half(float* out, int64_t stride, const float (&v)[N], int count, int real) {
    constexpr uint32_t kAdd = 27u << 23;  // 2^-100
    uint32_t lo = ~0u, hi = 0u;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint32_t b = i < real ? __float_as_uint(v[i]) & 0x7FFFFFFFu : kAdd;
        lo = min(lo, b);
        if (i < real) hi = max(hi, b);
    }
    if (hi == 0u) return;
    if (lo >= kAdd) {
        if constexpr (ROW) {
#pragma unroll
            for (int i = 0; i < N; i += 4)
                if (i < count)
                    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(out + i), "f"(v[i]),
                                 "f"(v[i + 1]), "f"(v[i + 2]), "f"(v[i + 3])
                                 : "memory");
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (i < count) atomicAdd(out + i * stride, v[i]);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if (i >= real || v[i] == 0.f) continue;
        float* o = out + i * stride;
        const float other = atomicExch(o, v[i]);
        if (other != 0.f) asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(o), "f"(other + v[i]) : "memory");
    }
}
// Named barrier over `count` threads that also ORs a predicate across them.
__device__ __forceinline__ bool bar_red_or(int id, int count, bool pred) {
    uint32_t r;
    asm volatile(
        "{ .reg .pred pi, po; setp.ne.u32 pi, %1, 0; bar.red.or.pred po, %2, %3, pi; selp.u32 %0, 1, 0, po; }"
        : "=r"(r)
        : "r"((uint32_t)pred), "r"(id), "r"(count)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Ready flags of the transfer passes: the writer's generic stores are made
// visible to the bulk copies (async proxy) of other CTAs by a proxy fence and a
// release store; the reader acquires the flag and fences again before copying.
__device__ __forceinline__ int flag_acquire(const int* f) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
    return v;
}
__device__ __forceinline__ void flag_release(int* f, int v) {
    asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(f), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void fence_proxy_async_global() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// x - tf32(x) per component: what the TF32 MMA drops from an FP32 operand
// (it reads the top 19 bits).
__device__ __forceinline__ float4 tf32_lo(const float4 v) {
    float4 l;
    l.x = v.x - __uint_as_float(__float_as_uint(v.x) & 0xFFFFE000u);
    l.y = v.y - __uint_as_float(__float_as_uint(v.y) & 0xFFFFE000u);
    l.z = v.z - __uint_as_float(__float_as_uint(v.z) & 0xFFFFE000u);
    l.w = v.w - __uint_as_float(__float_as_uint(v.w) & 0xFFFFE000u);
    return l;
}

// 32 consecutive TMEM columns of this warp's 32 lanes, without waiting: the
// caller issues several and then one tcgen05.wait::ld.
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 consecutive TMEM columns of this warp's 32 lanes from registers; the
// caller waits with tmem_wait_st before signalling the MMA.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }


}  // namespace

// ---------------------------------------------------------------------------
// Packing kernels
// ---------------------------------------------------------------------------

// One tile per CTA: dst (np × kp core-matrix tile, BF16 if es = 2 else FP32)
// ← src (n × k row-major FP64, leading dimension ld), zero padding.  Tile
// offsets are given for BF16 and scaled by es/2.
__global__ void k_pack_tiles(const TcPackTile* __restrict__ tiles, int64_t count, const double* __restrict__ src,
                             uint8_t* __restrict__ dst, int es) {
    for (int64_t t = blockIdx.x; t < count; t += gridDim.x) {
        const TcPackTile d = tiles[t];
        uint8_t* base = dst + d.dst * (es / 2);
        for (int e = threadIdx.x; e < d.np * d.kp; e += blockDim.x) {
            const int r = e / d.kp, c = e % d.kp;
            double v = (r < d.n && c < d.k)
                           ? src[d.src + ((d.tr & 1) ? (int64_t)c * d.ld + r : (int64_t)r * d.ld + c)]
                           : 0.0;
            if (es == 2) {
                __nv_bfloat16 b = __double2bfloat16(v);
                if (d.tr & 2) b = __double2bfloat16(v - (double)__bfloat162float(b));
                *(__nv_bfloat16*)(base + cm_off(r, c, d.kp, 2)) = b;
            } else {
                *(float*)(base + cm_off(r, c, d.kp, 4)) = (float)v;
            }
        }
    }
}

// Activation tiles: for each id (cluster or leaf), rows r = 2i + h (i < mc)
// hold column i of the FP32 source split into a high part (h = 0) and the
// remainder (h = 1): BF16 (es = 2): bf16(x) and bf16(x - bf16(x)); TF32 (es = 4):
// x itself (the MMA reads tf32(x)) and x - tf32(x).  Columns κ < kdim(id) read
// src[(base(id) + κ) * ld + i]; zero padding to R rows and kp(id) columns;
// kp(id) = kp_fixed, or koff[id+1] - koff[id].  With idmap only the ids
// idmap[0..ids) are packed.
// Threads walk the tile in its memory order, 4 bytes each, so a warp writes one
// whole 128-byte core matrix (8 rows × 16 bytes).
__global__ void k_pack_act(const float* __restrict__ src, int64_t ld, int ids, const int32_t* __restrict__ idmap,
                           const int32_t* __restrict__ base, const int32_t* __restrict__ kdim, int kdim_fixed,
                           const int64_t* __restrict__ koff, int kp_fixed, int mc, int R, uint8_t* __restrict__ dst,
                           int es) {
    const int per = 16 / es;  // elements of one core-matrix row
    for (int j = blockIdx.x; j < ids; j += gridDim.x) {
        const int id = idmap ? idmap[j] : j;
        const int kp = koff ? (int)(koff[id + 1] - koff[id]) : kp_fixed;
        const int64_t tile = (koff ? koff[id] : (int64_t)id * kp_fixed) * (int64_t)R * es;
        const int kd = kdim ? kdim[id] : kdim_fixed;
        const int64_t b = base ? (int64_t)base[id] : (int64_t)id * kdim_fixed;
        const int cgroups = kp / per;
        const int words = R * kp * es / 4;  // 4-byte words of the tile
        uint32_t* out = (uint32_t*)(dst + tile);
        for (int w = threadIdx.x; w < words; w += blockDim.x) {
            const int cmi = w >> 5, within = (w & 31) * 4;  // core matrix, byte inside it
            const int r = (cmi / cgroups) * 8 + (within >> 4);
            const int c0 = (cmi % cgroups) * per + ((within & 15) / es);
            const int i = r >> 1;
            const bool lo = r & 1;
            if (es == 4) {
                float x = 0.f;
                if (i < mc && c0 < kd) x = src[(b + c0) * ld + i];
                const float v = lo ? x - __uint_as_float(__float_as_uint(x) & 0xFFFFE000u) : x;
                out[w] = __float_as_uint(v);
            } else {
                uint32_t pk = 0;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int c = c0 + u;
                    float x = 0.f;
                    if (i < mc && c < kd) x = src[(b + c) * ld + i];
                    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
                    const __nv_bfloat16 v = lo ? __float2bfloat16_rn(x - __bfloat162float(hi)) : hi;
                    pk |= (uint32_t)__bfloat16_as_ushort(v) << (16 * u);
                }
                out[w] = pk;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The tcgen05 segmented GEMM
// ---------------------------------------------------------------------------
// KIND 0: BF16 operands, one MMA (kind::f16) per 16-wide K step.
// KIND 1: FP32 data on the TF32 units with split operands ("3xTF32"): the
//   activation rows carry x and x - tf32(x); the matrix tile is read once as
//   tf32(S) (the MMA drops the low 13 mantissa bits) and once as the remainder
//   S - tf32(S): the splitter warps write both into TMEM as the MMA's A operand
//   [S; S - tf32(S)], so D = x·tf32(S) + x·(S - tf32(S)) with both parts of x
//   reaches FP32 accuracy.
// Stage layout: [A: R activation rows | B: 64 matrix rows], element size es = 2
// (KIND 0) or 4 (KIND 1), 64 contraction columns at most.
// MODE 0: coupling (outputs ŷ_t); MODE 1: leaf phase (outputs Z); MODE 2 (KIND 1
// only): coupling without the stored S_b, whose rows the splitter warps evaluate
// from the Chebyshev nodes (Eq. (h2_admissible)): only the activation tile is
// copied.  MODE 3 (KIND 1 only): a work list in dependency order whose items
// carry their role (item_role): transfer-pass items (Alg. "forward/backward",
// one per cluster) put their result, split, into the cluster's activation tile
// and release it with a ready flag; coupling items write split tiles; leaf items
// write rows of Z.  A term marked kTermWait waits (bounded) for the ready flag
// of the tile it reads before its copy.  MODE 4 (KIND 1 only): such a list for
// one system, whose role-0 items write rows of ŷ like MODE 0: the coupling
// launch that also computes the clusters above the upward pass's cut (their
// transfer items wait for their sons and release their own tiles).
// NARROW (R <= 64, at most 32 right-hand-side columns): two CTAs per SM, each with
// half of the SM's stages, accumulators and A slots.  A CTA's hand-offs (about
// 1300 cycles a term, of which copies and MMAs fill a part) are a serial chain, so
// two CTAs run two of them at once; 80 registers a thread (KIND 1) suffice because
// the epilogue sums 32 columns and moves TMEM 32 columns at a time.  One CTA → two
// (µs, n = 65536, q = 4, m = 32): hybrid coupling 167 → 140, leaf 86 → 73; BF16 130
// → 91 and 67 → 42; n = 262144, m = 16: 593 → 457 and 294 → 235.  More than 32
// columns need stages of 48 KiB and 128 accumulator columns: one CTA.
template <int MODE, int KIND, bool NARROW>
__global__ void __launch_bounds__(tc_threads<KIND>(), NARROW ? 2 : 1) k_tc_gemm(const TcGemmParams p) {
    constexpr bool MF = MODE == 2;
    constexpr bool FLOW = MODE == 3;
    constexpr bool LIST = MODE == 3 || MODE == 4;  // items carry roles, terms may wait for ready flags
    // the coupling writes its result as split tiles when the downward pass runs on
    // the tensor cores (p.out_act set)
    const bool COUP_SPLIT = (MODE == 0 || MODE == 2) && p.out_act != nullptr;
    constexpr int ES = KIND == 0 ? 2 : 4;
    constexpr int KSTEP = KIND == 0 ? 16 : 8;  // K of one MMA instruction
    constexpr int F_FIRST = 1, F_LAST = 2, F_END = 4, F_PARITY = 8;
    // TMEM: KIND 0 has kAccBufs accumulators of 64 columns.  KIND 1 has
    // accumulators of R columns (64 or 128: 4 or 2 of them, 256 columns) and
    // after them kASlots (4) slots of 64 columns for the MMA's A operand [B; B_lo].
    // NARROW halves both (KIND 1): accumulators of 32 or 64 columns in 128, two A slots.
    constexpr int TMEM_COLS = KIND == 1 ? (NARROW ? 256 : 512) : kAccBufs * kAccCols;
    constexpr int A_BASE = NARROW ? 128 : 256;
    constexpr int kASlots = NARROW ? 2 : 4;
    constexpr int kSums = KIND == 1 && NARROW ? 32 : kAccCols;  // right-hand-side columns (KIND 1), tile rows (KIND 0)
    constexpr int kSt = NARROW ? kMaxStagesNarrow : kMaxStages;
    extern __shared__ __align__(128) uint8_t smem_raw[];
    // 128 bytes: a core matrix, which is what bulk copies and descriptors without a swizzle need
    // (an offset, not a rounded pointer: through an integer the compiler loses the address
    // space, and every access to the stages becomes a generic load)
    uint8_t* smem = smem_raw + (-smem_u32(smem_raw) & 127u);
    __shared__ __align__(8) uint64_t full_bar[kSt], split_bar[kSt], empty_bar[kSt];
    __shared__ __align__(8) uint64_t accf_bar[kAccBufs], acce_bar[kAccBufs], drain_bar[2], aempty_bar[kASlots];
    __shared__ int s_total;  // terms of this CTA
    __shared__ uint32_t tmem_slot;
    // a stage's contraction length, flags | output width << 8 (-1: never used), activation
    // rows, target cluster (MODE 2)
    __shared__ __align__(16) int4 stage_meta[kSt];
    __shared__ __align__(16) int4 s_term[2][kTermBatch];  // the producers' current terms
    __shared__ int abort_shared;
    volatile int& abort_flag = abort_shared;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = p.R;
    const int M = R <= 64 ? 64 : 128;
    const int nst = p.nstages;
    const int a_bytes = p.a_stage_bytes, b_bytes = MF ? kNodeBytes : 64 * 64 * ES;
    const int stage_bytes = a_bytes + b_bytes;
    const int G = gridDim.x;
    // TMEM columns of one accumulator, and accumulator buffers
    const int acc_cols = KIND == 1 ? (NARROW ? (R <= 32 ? 32 : 64) : (R <= 64 ? 64 : 128)) : kAccCols;
    const int nacc = KIND == 1 ? A_BASE / acc_cols : kAccBufs;  // 2 or 4
    const int lacc = nacc >> 1;                                 // its logarithm

    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            mbar_init(&full_bar[s], 1);
            stage_meta[s] = make_int4(0, -1, 0, 0);
            mbar_init(&split_bar[s], kSplitWarps);
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < kAccBufs; ++b) {
            mbar_init(&accf_bar[b], 1);
            mbar_init(&acce_bar[b], 4);  // one arrival per epilogue warp
        }
        mbar_init(&drain_bar[0], 1);
        mbar_init(&drain_bar[1], 1);
        for (int a = 0; a < kASlots; ++a) mbar_init(&aempty_bar[a], 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        // the CTA's term count: the two issuers split the terms by parity and stop there
        int tot = 0;
        for (int w = blockIdx.x + lane * G; w < p.n_items; w += 32 * G) tot += p.items[w].e1 - p.items[w].e0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
        if (lane == 0) s_total = tot;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    // This CTA has its TMEM before a later launch can start (that one's CTAs may come to
    // this SM, take TMEM in their turn and wait for this grid).  The barriers, TMEM and
    // the item count (of static lists) are set up while the launch before still runs.
    chain_release();
    chain_wait();

    if (warp == 0 || warp == tc_producer2<KIND>()) {
        // ---------------- producers ----------------
        // Two warps issue the copies, each into its own stages (even and odd): a warp's
        // instructions a term bound the kernel where the copies do not (one producer with
        // six shuffles a term: 1070 cycles a term at KIND 0, 2100 at KIND 1, unchanged when
        // the copies were halved; one → two, µs at n = 65536, m = 32: coupling 140 → 139
        // with three stages a CTA, 133 before the stages were shared out, leaf 73 → 70,
        // BF16 88 → 80 and 42 → 31).  A batch of term descriptors (16 bytes each) is loaded
        // while the batch before is issued, and parked in shared memory: a term costs one
        // read of its descriptor, a wait for its stage, one store of the stage's metadata
        // (published to the other roles by the mbarrier arrive) and the copies, all from a
        // converged warp, which keeps the stage's addresses uniform.  Stages, not terms,
        // are shared out: a stage's producer then waits for every one of its uses in turn,
        // and a phase parity cannot be taken for that of the use two before (the two
        // issuers may finish terms out of order).
        const int me = warp == 0 ? 0 : 1;
        int stage = 0;  // of the next term, whichever warp's
        uint32_t phase = 0;
        bool dead = false;
        const uint64_t pol_keep = l2_policy_evict_last(), pol_stream = l2_policy_evict_first();
        // an item's system: its terms, buffers and sizes (PSYS reads a field of the
        // system table of a multi-system launch, else of the launch's own arguments)
#define PSYS(it_, f_) ((FLOW && p.sys) ? p.sys[item_sys(it_)].f_ : p.f_)
        const TcItem none{-1, 0, 0, 0};
        auto item_at = [&](int w) { return w < p.n_items ? p.items[w] : none; };
        // the lane's of the item's terms from base on
        auto term_at = [&](const TcItem& it, int base) {
            const int e = it.e0 + base + lane;
            return it.id >= 0 && lane < kTermBatch && e < it.e1 ? __ldg((const int4*)(PSYS(it, terms) + e))
                                                                : make_int4(0, 0, 0, 0);
        };
        TcItem cur = item_at(blockIdx.x), nxt = item_at(blockIdx.x + G);
        int4 tnext = term_at(cur, 0);
        for (int w = blockIdx.x; w < p.n_items && !dead; w += G) {
            if (__any_sync(0xffffffffu, abort_flag != 0)) break;
            const TcItem after = item_at(w + 2 * G);
            const int nterms = cur.e1 - cur.e0;
            const int Ri = PSYS(cur, R), npi = item_np(cur), row_bytes = Ri * ES;
            const uint8_t *a0 = PSYS(cur, act0), *a1 = PSYS(cur, act1), *a2 = PSYS(cur, act2), *bm = PSYS(cur, bmat);
            if (nterms <= 0) tnext = term_at(nxt, 0);
            for (int base = 0; base < nterms && !dead; base += kTermBatch) {
                const int4 t = tnext;
                tnext = base + kTermBatch < nterms ? term_at(cur, base + kTermBatch) : term_at(nxt, 0);
                const int cnt = min(kTermBatch, nterms - base);
                __syncwarp();
                if (lane < kTermBatch) s_term[me][lane] = t;
                // Terms that read a tile of this launch wait for its ready flag.  The
                // lanes poll the flags of the batch's terms together (one round trip
                // for all), and a term's copies are issued once its bit is set.
                uint32_t ready_mask = 0xffffffffu;
                const int* my_flag = nullptr;
                if (LIST) {
                    int sl = stage + lane;  // the lane's term's stage
                    while (sl >= nst) sl -= nst;
                    if (lane < cnt && (sl & 1) == me && ((t.w >> 16) & kTermWait)) my_flag = PSYS(cur, flag) + t.z / PSYS(cur, KP);
                    ready_mask = __ballot_sync(0xffffffffu, !my_flag || flag_acquire(my_flag) == p.epoch);
                }
                __syncwarp();
                int4 tj = s_term[me][0];
                for (int j = 0; j < cnt; ++j) {
                    if ((stage & 1) != me) {
                        if (j + 1 < cnt) tj = s_term[me][j + 1];
                        if (++stage == nst) { stage = 0; phase ^= 1; }
                        continue;
                    }
                    const int kpj = (int16_t)tj.w, asj = tj.w >> 16, akj = tj.z;
                    const int64_t bj = (int64_t)(((uint64_t)(uint32_t)tj.y << 32) | (uint32_t)tj.x);
                    if (j + 1 < cnt) tj = s_term[me][j + 1];
                    if (LIST && !((ready_mask >> j) & 1u)) {
                        // poll again (bounded: gives up after about one second)
                        const uint64_t t0 = global_ns();
                        while (true) {
                            __nanosleep(32);
                            ready_mask |= __ballot_sync(0xffffffffu, my_flag && flag_acquire(my_flag) == p.epoch);
                            __syncwarp();
                            if ((ready_mask >> j) & 1u) break;
                            if (__any_sync(0xffffffffu, abort_flag || global_ns() - t0 > 1000000000ull)) {
                                dead = true;  // warp-uniform: every lane leaves together
                                break;
                            }
                        }
                    }
                    // the flags acquired by the warp order the tiles' writes before this copy
                    if (LIST && (asj & kTermWait)) fence_proxy_async_global();
                    if (dead || !__any_sync(0xffffffffu, mbar_wait(&empty_bar[stage], phase ^ 1))) {
                        dead = true;
                        if (lane == 0) atomicExch(p.err, 1);
                        abort_flag = 1;
                        break;
                    }
                    const uint32_t ab = (uint32_t)(row_bytes * kpj);
                    const uint32_t sA = smem_u32(smem + stage * stage_bytes), bar = smem_u32(&full_bar[stage]);
                    const int term = base + j;
                    const int fl = (term == 0 ? F_FIRST : 0) | (term == nterms - 1 ? F_LAST : 0) | (phase ? F_PARITY : 0);
                    const int64_t aj = (int64_t)akj * row_bytes;
                    // the activation tiles are read by many terms, the matrix tiles once; MODE 2
                    // copies the source cluster's nodes (its rows and nodes start at s·KP)
                    const uint8_t* asrc = ((asj & 3) == 0 ? a0 : ((asj & 3) == 1 ? a1 : a2)) + aj;
                    const uint8_t* bsrc = MF ? (const uint8_t*)(p.nodes + akj) : bm + bj * (ES / 2);
                    const uint32_t bb = MF ? (uint32_t)(p.KP * 16) : (uint32_t)(npi * kpj * ES);
                    stage_copy_elect(smem_u32(&stage_meta[stage]), kpj, fl | (npi << 8), Ri, cur.id, bar, sA, asrc, ab,
                                     pol_keep, sA + a_bytes, bsrc, bb, MF ? pol_keep : pol_stream);
                    if (++stage == nst) { stage = 0; phase ^= 1; }
                }
            }
            cur = nxt;
            nxt = after;
        }
        __syncwarp();
        // the splitters' end marker, a stage without data, comes from the next stage's producer
        if (lane == 0 && !dead && (stage & 1) == me) {
            if (mbar_wait(&empty_bar[stage], phase ^ 1)) {
                stage_meta[stage] = make_int4(0, F_END | (phase ? F_PARITY : 0), 0, 0);
                mbar_arrive(&full_bar[stage]);
            } else {
                atomicExch(p.err, 1);
                abort_flag = 1;
            }
        }
#undef PSYS
    } else if (warp == 1 || (KIND == 1 && warp == tc_issuer2<KIND>())) {
        // ---------------- MMA issuers: driven by the stage metadata ----------------
        // Two warps take the terms by parity (term t uses stage t mod nst,
        // accumulator t mod nacc and A slot t mod kASlots), so one warp's waits
        // overlap the other's MMAs.  Each reuse of a stage, slot or accumulator
        // waits for the consumer of its previous use, so every barrier's
        // arrivals come in order whichever issuer commits them.  Each converged warp runs its loop (waits and descriptors are
        // warp-uniform); elect.sync hands each MMA and commit to one lane.
        const int j = warp == 1 ? 0 : 1;
        const int T = s_total;
        bool issued = false;
        if (KIND == 0 && j == 0) {
            // BF16: one issuer takes every term in order and accumulates all terms of
            // an item in one TMEM accumulator (an item's first term starts it from
            // zero); the epilogue reads each accumulator once per item.  The FP32
            // accumulation of the tensor cores is far finer than the BF16 operands.
            int item_idx = 0, acc = 0, stage = 0;
            uint32_t phase = 0;
            for (int it = 0; it < T; ++it) {
                if (!__any_sync(0xffffffffu, mbar_wait(&full_bar[stage], phase))) {
                    abort_flag = 1;
                    if (lane == 0) atomicExch(p.err, 4);
                    break;
                }
                const int4 mt = stage_meta[stage];
                const int fl = mt.y;
                if (fl & F_FIRST) {
                    acc = item_idx % kAccBufs;
                    if (!__any_sync(0xffffffffu, mbar_wait(&acce_bar[acc], ((item_idx / kAccBufs) & 1) ^ 1))) {
                        abort_flag = 1;
                        if (lane == 0) atomicExch(p.err, 3);
                        break;
                    }
                }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)(acc * acc_cols);
                const int kp = mt.x;
                const uint32_t sA = smem_u32(smem + stage * stage_bytes);
                const uint32_t sbo = (uint32_t)(kp * ES / 16) * 128;
                mma_term_bf16(d, smem_desc(sA, 128, sbo), smem_desc(sA + a_bytes, 128, sbo), idesc_for<KIND>(M, (fl >> 8) & 255),
                              (fl & F_FIRST) ? 0u : 1u, kp / KSTEP, smem_u32(&empty_bar[stage]),
                              (fl & F_LAST) ? smem_u32(&accf_bar[acc]) : 0u);
                issued = true;
                if (fl & F_LAST) ++item_idx;
                if (++stage == nst) { stage = 0; phase ^= 1; }
            }
            if (issued) {
                mma_commit_elect(&drain_bar[0]);
                if (!__any_sync(0xffffffffu, mbar_wait(&drain_bar[0], 0)) && lane == 0) atomicExch(p.err, 5);
                issued = false;  // drained
            }
        }
        int stage = j;
        uint32_t phase = 0;
        if (stage >= nst) { stage -= nst; phase ^= 1; }
        for (int it = j; it < T && KIND == 1; it += 2) {
            if (!__any_sync(0xffffffffu, mbar_wait(&split_bar[stage], phase))) {
                abort_flag = 1;
                if (lane == 0) atomicExch(p.err, 4);
                break;
            }
            // every term accumulates from zero in its own TMEM buffer; the epilogue
            // adds the terms of an item in FP32 registers (round to nearest), so
            // the tensor-core accumulator never sums more than one term's K steps
            const int acc = it & (nacc - 1);
            if (!__any_sync(0xffffffffu, mbar_wait(&acce_bar[acc], ((it >> lacc) & 1) ^ 1))) {
                abort_flag = 1;
                if (lane == 0) atomicExch(p.err, 3);
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(acc * acc_cols);
            const int4 mt = stage_meta[stage];
            const uint32_t sbo = (uint32_t)(mt.x * ES / 16) * 128;
            // D[n, r] = [mat; mat_lo] · actᵀ: M = 128, the tile (rows 0..63) and its TF32
            // remainder (rows 64..127), which the splitter warps have put into TMEM slot
            // `as`; N = R activation rows from shared memory.  The MMA time grows with N,
            // not with M up to 128, so the remainder costs no extra instructions.  Rows
            // np..63 of either part hold stale data whose TMEM lanes the epilogue ignores.
            const int as = it % kASlots;
            mma_term_tf32(d, tmem + (uint32_t)(A_BASE + 64 * as), smem_desc(smem_u32(smem + stage * stage_bytes), 128, sbo),
                          idesc_for<KIND>(128, mt.z), mt.x / KSTEP, smem_u32(&empty_bar[stage]), smem_u32(&aempty_bar[as]),
                          smem_u32(&accf_bar[acc]));
            issued = true;
            stage += 2;
            while (stage >= nst) { stage -= nst; phase ^= 1; }
        }
        if (issued) {
            mma_commit_elect(&drain_bar[j]);
            if (!__any_sync(0xffffffffu, mbar_wait(&drain_bar[j], 0)) && lane == 0) atomicExch(p.err, 5);
        }
    } else if (warp < 6 && KIND == 1) {
        // ---------------- epilogue, KIND 1 (warps 2..5, TMEM lane quadrant warp % 4) ----------------
        // TMEM lane 32q + lane holds row n = 32(q & 1) + lane of the tile (q = 0, 1)
        // or of its remainder (q = 2, 3); column r = 2i + h of that lane is the
        // product with the high (h = 0) or low (h = 1) part of right-hand-side
        // column i.  Each thread adds its two columns per i over the item's terms;
        // at the item's end the remainder warps hand their sums to the tile warps
        // through shared memory (double buffered by item parity, one barrier per
        // item), which add them and store row n.
        const int q = warp & 3;
        const int n = 32 * (q & 1) + lane;
        const bool lo_part = q >= 2;
        // [2][kSums i][64 n]
        float* xch = reinterpret_cast<float*>(smem + nst * stage_bytes + (MF ? kEvalBytes : 0));
        int it = 0, par = 0;
        // rows of Z: the leaf phase, and the leaf items of a transfer-pass launch
        auto leaf_rows = [&](const TcItem& t) { return MODE == 1 || (LIST && item_role(t) == kRoleLeaf); };
        TcItem cur = blockIdx.x < p.n_items ? p.items[blockIdx.x] : TcItem{-1, 0, 0, 0};
        // an item's system: its sizes and buffers (SYSF reads a field of the system
        // table of a multi-system launch, else of the launch's own arguments)
#define SYSF(it_, f_) ((FLOW && p.sys) ? p.sys[item_sys(it_)].f_ : p.f_)
        int cur_off = 0, cur_nt = 0;
        if (cur.id >= 0 && leaf_rows(cur)) {
            const int t = SYSF(cur, leaves)[cur.id];
            cur_off = SYSF(cur, cl_off)[t];
            cur_nt = SYSF(cur, cl_size)[t];
        }
        for (int w = blockIdx.x; w < p.n_items; w += G) {
            const TcItem nxt = w + G < p.n_items ? p.items[w + G] : TcItem{-1, 0, 0, 0};
            int nxt_off = 0, nxt_nt = 0;
            if (nxt.id >= 0 && leaf_rows(nxt)) {
                const int t = SYSF(nxt, leaves)[nxt.id];
                nxt_off = SYSF(nxt, cl_off)[t];
                nxt_nt = SYSF(nxt, cl_size)[t];
            }
            const int id = cur.id, np = item_np(cur), nterms = cur.e1 - cur.e0;
            const int Ri = SYSF(cur, R), mci = SYSF(cur, mc), ki = SYSF(cur, k), KPi = SYSF(cur, KP),
                      ldci = SYSF(cur, ldc);
            const bool wide = !NARROW && Ri > 64;
            const bool vec4 = (mci & 3) == 0 && (ldci & 3) == 0;
            const int role = LIST ? item_role(cur) : 0;
            // role 0 (MODE 4's coupling items): rows of ŷ, as in MODE 0
            const bool split_out = COUP_SPLIT || (LIST && role != kRoleLeaf && role != 0);
            float sum[kSums];
#pragma unroll
            for (int j = 0; j < kSums; ++j) sum[j] = 0.f;
            bool failed = false;
            uint32_t imask = 0;  // complex product: bit t of the batch of 32 terms applies i·act
            for (int term = 0; term < nterms; ++term, ++it) {
                if (!FLOW && p.cplx && (term & 31) == 0) {
                    const int tt = term + lane;
                    imask = __ballot_sync(0xffffffffu, tt < nterms && (p.terms[cur.e0 + tt].asrc & kTermImag));
                }
                const bool imag = (imask >> (term & 31)) & 1u;
                const int acc = it & (nacc - 1);
                if (!__any_sync(0xffffffffu, mbar_wait(&accf_bar[acc], (it >> lacc) & 1))) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * acc_cols);
                if constexpr (FLOW || NARROW) {
                    // 32 columns per read (16 right-hand-side columns; R > 64 takes four):
                    // one register buffer, which the multi-system bookkeeping and the two
                    // CTAs per SM need room for
                    uint32_t r0[32];
#pragma unroll
                    for (int h = 0; h < kSums / 16; ++h) {
                        if (NARROW ? 32 * h >= acc_cols : (h >= 2 && !wide)) break;
                        tmem_ld32_async(ta + 32 * h, r0);
                        tmem_wait_ld();
                        if (FLOW || !imag) {
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                sum[16 * h + j] += __uint_as_float(r0[2 * j]) + __uint_as_float(r0[2 * j + 1]);
                        } else {
                            // i·act: column 2j takes -(column 2j + 1), column 2j + 1 takes column 2j
#pragma unroll
                            for (int j = 0; j < 16; j += 2) {
                                sum[16 * h + j] -= __uint_as_float(r0[2 * j + 2]) + __uint_as_float(r0[2 * j + 3]);
                                sum[16 * h + j + 1] += __uint_as_float(r0[2 * j]) + __uint_as_float(r0[2 * j + 1]);
                            }
                        }
                    }
                } else {
                    // 64 columns per read (two loads in flight, one wait); R > 64 takes two
                    uint32_t r0[32], r1[32];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && !wide) break;
                        tmem_ld32_async(ta + 64 * h, r0);
                        tmem_ld32_async(ta + 64 * h + 32, r1);
                        tmem_wait_ld();
                        if (!imag) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                sum[32 * h + j] += __uint_as_float(r0[2 * j]) + __uint_as_float(r0[2 * j + 1]);
                                sum[32 * h + 16 + j] += __uint_as_float(r1[2 * j]) + __uint_as_float(r1[2 * j + 1]);
                            }
                        } else {
                            // i·act: column 2j takes -(column 2j + 1), column 2j + 1 takes column 2j
#pragma unroll
                            for (int j = 0; j < 16; j += 2) {
                                const float a0 = __uint_as_float(r0[2 * j]) + __uint_as_float(r0[2 * j + 1]);
                                const float a1 = __uint_as_float(r0[2 * j + 2]) + __uint_as_float(r0[2 * j + 3]);
                                const float b0 = __uint_as_float(r1[2 * j]) + __uint_as_float(r1[2 * j + 1]);
                                const float b1 = __uint_as_float(r1[2 * j + 2]) + __uint_as_float(r1[2 * j + 3]);
                                sum[32 * h + j] -= a1;
                                sum[32 * h + j + 1] += a0;
                                sum[32 * h + 16 + j] -= b1;
                                sum[32 * h + 16 + j + 1] += b0;
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce_bar[acc]);
            }
            float* xb = xch + par * (64 * kSums);
            if (lo_part && !failed) {
#pragma unroll
                for (int i = 0; i < kSums; ++i)
                    if (i < mci) xb[i * 64 + n] = sum[i];
            }
            // every epilogue warp reaches this barrier once per item, failed or not,
            // and all of them learn whether any failed
            if (bar_red_or(1, 128, failed)) {
                if (lane == 0) atomicExch(p.err, 6);
                abort_flag = 1;
                break;
            }
            if (!lo_part && split_out) {
#pragma unroll
                for (int i = 0; i < kSums; ++i)
                    if (i < mci) sum[i] += xb[i * 64 + n];
                // The result goes, split as the activations are (rows 2i: x; 2i + 1: x -
                // tf32(x); zero past the columns and past column k), into the cluster's
                // tile: staged in this item's exchange buffer (free once both tile warps
                // have read it) and stored by one bulk copy per SB rows.
                constexpr int SB = kSums;  // rows of KP <= 64 columns that the exchange buffer holds
                asm volatile("bar.sync 4, 64;" ::: "memory");
                uint8_t* gtile = (role == kRoleCoupling ? SYSF(cur, out_act2) : SYSF(cur, out_act)) + (int64_t)id * KPi * Ri * 4;
                const bool nv = n < ki;
#pragma unroll
                for (int hh = 0; hh < 2 * kSums / SB; ++hh) {
                    const int h0 = SB * hh;
                    if (h0 >= Ri) break;
                    const int rows = min(SB, Ri - h0);
                    if (h0 > 0) asm volatile("bar.sync 4, 64;" ::: "memory");  // the last store read the buffer
                    if (n < KPi) {
#pragma unroll
                        for (int i = 0; i < SB / 2; ++i) {
                            if (2 * i >= rows) break;
                            const int ii = SB / 2 * hh + i;
                            const float v = (nv && ii < mci) ? sum[ii] : 0.f;
                            const float lo = v - __uint_as_float(__float_as_uint(v) & 0xFFFFE000u);
                            *(float*)((uint8_t*)xb + cm_off(2 * i, n, KPi, 4)) = v;
                            *(float*)((uint8_t*)xb + cm_off(2 * i + 1, n, KPi, 4)) = lo;
                        }
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    asm volatile("bar.sync 4, 64;" ::: "memory");
                    if (q == 0 && lane == 0) {
                        const uint32_t bytes = (uint32_t)(rows * KPi * 4);
                        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(
                                         gtile + (int64_t)h0 * KPi * 4),
                                     "r"(smem_u32(xb)), "r"(bytes)
                                     : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                    }
                }
                // the tile is in global memory: release it to the CTAs that wait for it
                if (LIST && role == kRoleTransfer && q == 0 && lane == 0) {
                    fence_proxy_async_global();
                    flag_release(SYSF(cur, flag) + id, p.epoch);
                }
            } else if (!lo_part) {
#pragma unroll
                for (int i = 0; i < kSums; ++i)
                    if (i < mci) sum[i] += xb[i * 64 + n];
                float* out = nullptr;
                if (!leaf_rows(cur)) {
                    if (n < np && n < ki) out = p.yhat + ((int64_t)id * ki + n) * ldci;
                } else {
                    // Z in cluster order; the scatter into Y (with α, σX) is a separate
                    // coalesced pass, so the epilogue only stores
                    if (n < cur_nt) out = SYSF(cur, zp) + ((int64_t)cur_off + n) * ldci;
                }
                if (!LIST && (cur.np & kItemHalf)) {
                    if (out) add_half<true>(out, 1, sum, mci, p.mreal);
                } else if (out) {
                    if (vec4) {
#pragma unroll
                        for (int i = 0; i < kSums; i += 4)
                            if (i < mci)
                                *reinterpret_cast<float4*>(out + i) = make_float4(sum[i], sum[i + 1], sum[i + 2], sum[i + 3]);
                    } else {
#pragma unroll
                        for (int i = 0; i < kSums; ++i)
                            if (i < mci) out[i] = sum[i];
                    }
                }
            }
            par ^= 1;
            cur = nxt;
            cur_off = nxt_off;
            cur_nt = nxt_nt;
        }
#undef SYSF
    } else if (warp < 6) {
        // ---------------- epilogue, KIND 0 (warps 2..5, TMEM lane quadrant warp % 4) ----------------
        const int q = warp & 3;
        int row;
        if (M == 128) row = 32 * q + lane;
        else row = lane < 16 ? 16 * q + lane : -1;
        const int i = row >> 1;
        const bool writer = row >= 0 && !(row & 1) && i < p.mc;
        int it = 0;
        TcItem cur = blockIdx.x < p.n_items ? p.items[blockIdx.x] : TcItem{-1, 0, 0, 0};
        int cur_off = 0, cur_nt = 0;
        if (MODE == 1 && cur.id >= 0) {
            const int t = p.leaves[cur.id];
            cur_off = p.cl_off[t];
            cur_nt = p.cl_size[t];
        }
        for (int w = blockIdx.x; w < p.n_items; w += G) {
            // the next item's descriptor (and leaf extent) load while this one waits
            const TcItem nxt = w + G < p.n_items ? p.items[w + G] : TcItem{-1, 0, 0, 0};
            int nxt_off = 0, nxt_nt = 0;
            if (MODE == 1 && nxt.id >= 0) {
                const int t = p.leaves[nxt.id];
                nxt_off = p.cl_off[t];
                nxt_nt = p.cl_size[t];
            }
            const int id = cur.id, np = item_np(cur);
            float sum[kAccCols];
#pragma unroll
            for (int j = 0; j < kAccCols; ++j) sum[j] = 0.f;
            bool failed = false;
            {
                // the item's terms accumulate in one accumulator (`it` counts items)
                const int acc = it % kAccBufs;
                // warp-uniform wait: a completed phase stays completed, so any lane's
                // success is the warp's success
                const bool ok = __any_sync(0xffffffffu, mbar_wait(&accf_bar[acc], (it / kAccBufs) & 1));
                ++it;
                if (!ok) {
                    failed = true;
                }
            }
            // one of two halves of an item: the two lanes of a row pair take 32 rows of the
            // output each, which halves a thread's additions
            const bool half = !LIST && (cur.np & kItemHalf);
            if (!failed && half) {
                const int acc = (it - 1) % kAccBufs;
                tc_fence_after();
                const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * acc_cols);
                uint32_t r0[32], r1[32];
                tmem_ld32_async(ta, r0);
                tmem_ld32_async(ta + 32, r1);
                tmem_wait_ld();
                const bool odd = lane & 1;
                float v[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const uint32_t other = __shfl_xor_sync(0xffffffffu, odd ? r0[j] : r1[j], 1);
                    v[j] = __uint_as_float(odd ? r1[j] : r0[j]) + __uint_as_float(other);
                }
                const int j0 = odd ? 32 : 0, rows = (MODE == 1 ? cur_nt : min(np, p.k)) - j0;
                float* out = MODE == 1 ? p.zp + (int64_t)cur_off * p.ldc + i : p.yhat + (int64_t)id * p.k * p.ldc + i;
                if (row >= 0 && i < p.mc) add_half<false>(out + (int64_t)j0 * p.ldc, p.ldc, v, rows, rows);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce_bar[acc]);
            } else if (!failed) {
                const int acc = (it - 1) % kAccBufs;
                tc_fence_after();
                // both halves of the accumulator in flight, one wait; the row pair
                // (2i, 2i + 1) is adjacent lanes, added by one shuffle
                const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * acc_cols);
                uint32_t r0[32], r1[32];
                tmem_ld32_async(ta, r0);
                if (np > 32) tmem_ld32_async(ta + 32, r1);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float v = __uint_as_float(r0[j]);
                    sum[j] += v + __shfl_xor_sync(0xffffffffu, v, 1);
                }
                if (np > 32) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float v = __uint_as_float(r1[j]);
                        sum[32 + j] += v + __shfl_xor_sync(0xffffffffu, v, 1);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce_bar[acc]);
            }
            if (LIST && item_role(cur) == kRoleTransfer) {
                // A transfer item of the hybrid upward pass: x̂ of the cluster as a
                // split BF16 tile (row 2i: bf16(v), row 2i + 1: bf16(v - bf16(v)); zero
                // for columns i >= mc and past row k), stored by the even-row threads, ordered for the bulk copies of other
                // CTAs by a proxy fence, and released by the ready flag once all four
                // warps have stored.  Every epilogue warp meets the barrier once per
                // transfer item, failed or not, and all of them learn of a failure.
                if (bar_red_or(1, 128, failed)) {
                    if (lane == 0) atomicExch(p.err, 6);
                    abort_flag = 1;
                    break;
                }
                if (row >= 0 && !(row & 1) && i < R / 2) {
                    uint8_t* gt = p.out_act + (int64_t)id * p.KP * R * 2;
                    const bool live = i < p.mc;
#pragma unroll
                    for (int u = 0; u < kAccCols / 8; ++u) {
                        if (8 * u >= p.KP) break;
                        uint32_t hw[4], lw[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float v0 = live && 8 * u + 2 * e < p.k ? sum[8 * u + 2 * e] : 0.f;
                            const float v1 = live && 8 * u + 2 * e + 1 < p.k ? sum[8 * u + 2 * e + 1] : 0.f;
                            const __nv_bfloat16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
                            const __nv_bfloat16 l0 = __float2bfloat16_rn(v0 - __bfloat162float(h0));
                            const __nv_bfloat16 l1 = __float2bfloat16_rn(v1 - __bfloat162float(h1));
                            hw[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                            lw[e] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                        }
                        *(uint4*)(gt + cm_off(2 * i, 8 * u, p.KP, 2)) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                        *(uint4*)(gt + cm_off(2 * i + 1, 8 * u, p.KP, 2)) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                    }
                    fence_proxy_async_global();
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (warp == 2 && lane == 0) {
                    __threadfence();
                    flag_release(p.flag + id, p.epoch);
                }
            } else if (failed) {
                if (lane == 0) atomicExch(p.err, 6);
                abort_flag = 1;
                break;
            } else if (writer && !half) {
                if (MODE != 1) {
                    float* out = p.yhat + (int64_t)id * p.k * p.ldc;
#pragma unroll
                    for (int j = 0; j < kAccCols; ++j)
                        if (j < np && j < p.k) out[(int64_t)j * p.ldc + i] = sum[j];
                } else {
                    // Z in cluster order; the scatter into Y (with α, σX) is a separate
                    // coalesced pass, so the epilogue only stores
                    float* z = p.zp + (int64_t)cur_off * p.ldc + i;
#pragma unroll
                    for (int j = 0; j < kAccCols; ++j)
                        if (j < cur_nt) z[(int64_t)j * p.ldc] = sum[j];
                }
            }
            cur = nxt;
            cur_off = nxt_off;
            cur_nt = nxt_nt;
        }
    } else if (KIND == 1 && warp < 6 + kSplitWarps) {
        // ---------------- splitter (warps 6..9): [B; B_lo] into TMEM ----------------
        // Warp w owns TMEM lanes 32q..32q+31 (q = w mod 4): row n = 32(q & 1) + lane
        // of the tile B (q = 0, 1) or of its remainder B_lo = B - tf32(B) (q = 2, 3).
        // Each thread reads its row (kp values, 16 bytes per core matrix) from the
        // stage and writes it to TMEM slot `as` of the MMA's A operand.
        const int q = warp & 3;
        const int n = 32 * (q & 1) + lane;
        const bool lo_part = q >= 2;
        // The splitter is the one serial stage of the pipeline, so it tests the next
        // term's barriers while it works on the current one: a phase seen complete
        // then costs no wait at the top of the next iteration.
        int stage = 0, sit = 0;
        uint32_t phase = 0;
        bool pre = false;  // the next iteration's stage and A-slot phases were seen complete
        float4 xt = make_float4(0.f, 0.f, 0.f, 0.f);  // MODE 2: this row's target node, of cluster xt_of
        int xt_of = -1;
        while (true) {
            bool ok = pre || __any_sync(0xffffffffu, mbar_wait(&full_bar[stage], phase));
            const int4 mt = ok ? stage_meta[stage] : make_int4(0, 0, 0, 0);
            const int fl = mt.y;
            const bool end = ok && (fl & F_END);
            const int as = sit % kASlots;
            // the slot is free once the MMAs of term sit - kASlots have completed
            if (ok && !end && !pre) ok = __any_sync(0xffffffffu, mbar_wait(&aempty_bar[as], ((sit / kASlots) & 1) ^ 1));
            pre = false;
            if (ok && !end) tc_fence_after();
            const int kp = mt.x;
            // MODE 2: row n of the evaluated tile, two terms deep (a warp is past the
            // barrier of term t + 1 only when its partner has read term t's tile)
            float* xrow = (float*)(smem + nst * stage_bytes + (sit & 1) * (kEvalBytes / 2)) + n * kEvalLd;
            if (MF) {
                // row n of S_b: g(ξ_{t,n}, ξ_{s,μ}) = exp(-|ξ_{t,n} - ξ_{s,μ}| / length) for
                // n, μ < k, zero in the padding.  The tile warp (q < 2) and the remainder
                // warp (q + 2) of the same rows each evaluate half of the columns and
                // swap halves through shared memory.  The source nodes come with the stage
                // and are read by the whole warp at once (one broadcast per node); the
                // row's own node stays in a register over the item.  The nodes are scaled,
                // so a value is a hardware square root and a hardware 2^x: 8 instructions and
                // 16 cycles of the SFU per warp.  Their relative errors, 2^-23 and 2^-22 at
                // most, make a relative error of r ln 2 · 2^-23 + 2^-22 of the value 2^-r, which
                // grows with r; r 2^-r is 0.53 at most, so the absolute error stays below 3e-7
                // (besides the FP32 rounding of the nodes).  n = 65536, q = 4, m = 32: 786 µs with node loads from global memory, shuffles and one
                // CTA per SM, 670 with the nodes in the stage, 402 with two CTAs, about 190
                // with scaled nodes, a square root and 16-byte exchanges.
                if (ok && !end) {
                    const bool rv = n < p.k;
                    if (mt.w != xt_of) {
                        xt_of = mt.w;
                        xt = p.nodes[(int64_t)xt_of * p.KP + (rv ? n : 0)];
                    }
                    const int half = p.KP >> 1, mu0 = lo_part ? half : 0;
                    const float4* ys = (const float4*)(smem + stage * stage_bytes + a_bytes);
                    for (int j0 = mu0; j0 < mu0 + half; j0 += 8) {
                        float g[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const float4 y = ys[j0 + j];
                            const float d0 = xt.x - y.x, d1 = xt.y - y.y, d2 = xt.z - y.z;
                            const float r2 = fmaf(d2, d2, fmaf(d1, d1, d0 * d0));
                            float r;
                            asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(r2));
                            asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(g[j]) : "f"(-r));
                        }
                        if (p.k < p.KP) {
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                if (!rv || j0 + j >= p.k) g[j] = 0.f;
                        }
                        *(float4*)(xrow + j0) = make_float4(g[0], g[1], g[2], g[3]);
                        *(float4*)(xrow + j0 + 4) = make_float4(g[4], g[5], g[6], g[7]);
                    }
                }
                // the pair (quadrants q and q ^ 2, named barrier 2 or 3) meets once per
                // stage, end marker and failures included, and both learn whether to stop
                if (bar_red_or(2 + (q & 1), 64, !ok)) {
                    if (lane == 0) atomicExch(p.err, 8);
                    abort_flag = 1;
                    break;
                }
            } else if (!ok) {
                if (lane == 0) atomicExch(p.err, 7);
                abort_flag = 1;
                break;
            }
            if (!end) {
                const int nstage = stage + 1 == nst ? 0 : stage + 1;
                const uint32_t nphase = stage + 1 == nst ? phase ^ 1u : phase;
                const bool pf = mbar_test(&full_bar[nstage], nphase);
                const bool pa = mbar_test(&aempty_bar[(sit + 1) % kASlots], (((sit + 1) / kASlots) & 1) ^ 1);
                const uint8_t* row =
                    smem + stage * stage_bytes + a_bytes + (n >> 3) * (kp >> 2) * 128 + (n & 7) * 16;
                const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(A_BASE + 64 * as);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (32 * h >= kp) break;
                    uint32_t v[32];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (32 * h + 4 * c < kp)
                            x = *(const float4*)(MF ? (const uint8_t*)(xrow + 32 * h + 4 * c) : row + (8 * h + c) * 128);
                        if (lo_part) x = tf32_lo(x);
                        v[4 * c] = __float_as_uint(x.x);
                        v[4 * c + 1] = __float_as_uint(x.y);
                        v[4 * c + 2] = __float_as_uint(x.z);
                        v[4 * c + 3] = __float_as_uint(x.w);
                    }
                    tmem_st32(ta + 32 * h, v);
                }
                tmem_wait_st();
                tc_fence_before();
                ++sit;
                pre = __all_sync(0xffffffffu, pf && pa);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&split_bar[stage]);
            if (fl & F_END) break;
            if (++stage == nst) { stage = 0; phase ^= 1; }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // every copy lands before the CTA exits: the last use of each stage, whose parity
    // its metadata holds
    if (threadIdx.x < nst && stage_meta[threadIdx.x].y != -1)
        if (!mbar_wait(&full_bar[threadIdx.x], (stage_meta[threadIdx.x].y & F_PARITY) ? 1u : 0u)) atomicExch(p.err, 2);
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Zero ŷ of clusters whose coupling list is empty.
__global__ void k_zero_clusters(const int32_t* __restrict__ ids, int count, float* __restrict__ yhat, int k, int ldc,
                                int mc) {
    for (int c = blockIdx.x; c < count; c += gridDim.x) {
        float* y = yhat + (int64_t)ids[c] * k * ldc;
        for (int e = threadIdx.x; e < k * mc; e += blockDim.x) y[(int64_t)(e / mc) * ldc + e % mc] = 0.f;
    }
}

// Zero the activation tiles (bytes each, a multiple of 16) of the clusters ids[0..count).
__global__ void k_zero_tiles(const int32_t* __restrict__ ids, int count, uint8_t* __restrict__ buf, int64_t bytes) {
    for (int c = blockIdx.x; c < count; c += gridDim.x) {
        uint4* t = reinterpret_cast<uint4*>(buf + (int64_t)ids[c] * bytes);
        for (int64_t e = threadIdx.x; e < bytes / 16; e += blockDim.x) t[e] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// Stage geometry for R activation rows and element size es: A holds R rows (the
// BF16 MMA reads M = 64 or 128 of them), B 64 rows, both with up to 64
// contraction columns; MODE 2 has the source nodes in place of B.  After the
// stages come MODE 2's evaluated tiles and the TF32 kernel's epilogue exchange
// (its B_lo lives in TMEM).  NARROW instances split an SM's shared memory between
// two CTAs.
struct TcGeometry {
    int a_bytes, stage_bytes, nstages, after;
};
TcGeometry tc_geometry(int R, int mode, int kind, bool narrow) {
    TcGeometry g;
    const int es = kind == 0 ? 2 : 4;
    const int rows = kind == 1 && narrow ? R : (R <= 64 ? 64 : 128);
    g.a_bytes = rows * 64 * es;
    g.stage_bytes = g.a_bytes + (mode == 2 ? kNodeBytes : 64 * 64 * es);
    g.after = (mode == 2 ? kEvalBytes : 0) + (kind == 1 ? xch_bytes(narrow) : 0);
    const int budget = (narrow ? kSmemBudgetNarrow : kSmemBudget) - 128 - g.after;
    g.nstages = std::min(narrow ? kMaxStagesNarrow : kMaxStages, budget / g.stage_bytes);
    return g;
}

// CTAs of a NARROW instance that are resident on one SM with `smem` bytes of
// dynamic shared memory: two if shared memory, registers (four partitions of the
// register file, a warp's in units of 256) and TMEM (256 of 512 columns each)
// allow it.  The runtime's occupancy query answers one for every kernel with a
// tcgen05.alloc; on the device two start at once (304 CTAs of 352 threads, 256
// columns and 114816 bytes on 152 SMs: none started late).
struct NarrowFit {
    int regs = 0, static_smem = 0, sm_smem = 0, reserved = 0;
    int per_sm(int threads, int smem) const {
        const int warps = threads / 32, per_warp = (regs * 32 + 255) / 256 * 256;
        const bool fits = 2 * (smem + static_smem + reserved) <= sm_smem && (2 * warps + 3) / 4 * per_warp <= 65536 / 4;
        return fits ? 2 : 1;
    }
};
template <int MODE, int KIND>
NarrowFit& narrow_fit() {
    static NarrowFit f;
    return f;
}

template <int MODE, int KIND>
int launch_one(const TcGemmParams& p, bool narrow, int smem, bool overlap, cudaStream_t st) {
    // Every CTA has to be resident: those of modes 3 and 4 wait on each other's
    // ready flags (bounded).
    const int per_sm = narrow ? narrow_fit<MODE, KIND>().per_sm(tc_threads<KIND>(), smem) : 1;
    const int grid = std::min(p.n_items, per_sm * kTcGrid);
    return launch_chained(overlap, narrow ? k_tc_gemm<MODE, KIND, true> : k_tc_gemm<MODE, KIND, false>, grid,
                          tc_threads<KIND>(), smem, st, p);
}
template <int MODE, int KIND>
int prepare_one(int dev) {
    H2_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm<MODE, KIND, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget));
    H2_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm<MODE, KIND, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudgetNarrow));
    H2_CUDA_TRY(cudaFuncSetAttribute(k_tc_gemm<MODE, KIND, true>, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    cudaFuncAttributes at;
    H2_CUDA_TRY(cudaFuncGetAttributes(&at, k_tc_gemm<MODE, KIND, true>));
    NarrowFit f;
    f.regs = at.numRegs;
    f.static_smem = (int)at.sharedSizeBytes;
    H2_CUDA_TRY(cudaDeviceGetAttribute(&f.sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    H2_CUDA_TRY(cudaDeviceGetAttribute(&f.reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
    narrow_fit<MODE, KIND>() = f;
    return 0;
}

// Set the shared-memory attribute of every tensor-core kernel instance up
// front (needed before a product is captured into a CUDA graph).
namespace {
int g_tc_attr_device = -1;  // device whose kernel attributes are set
}

int tc_prepare() {
    int dev = 0;
    H2_CUDA_TRY(cudaGetDevice(&dev));
    if (dev == g_tc_attr_device) return 0;
    int rc = 0;
    if ((rc = prepare_one<0, 0>(dev)) || (rc = prepare_one<1, 0>(dev)) || (rc = prepare_one<4, 0>(dev)) ||
        (rc = prepare_one<0, 1>(dev)) || (rc = prepare_one<1, 1>(dev)) || (rc = prepare_one<2, 1>(dev)) ||
        (rc = prepare_one<3, 1>(dev)) || (rc = prepare_one<4, 1>(dev)))
        return rc;
    g_tc_attr_device = dev;
    return 0;
}

int tc_stages(int mc, int kind) {
    const int R = round16(2 * mc);
    return tc_geometry(R, 0, kind, R <= 64).nstages;
}

int launch_tc_gemm(int mode, int kind, TcGemmParams p, cudaStream_t st, int stages, bool overlap) {
    const bool narrow = p.R <= 64;
    TcGeometry g = tc_geometry(p.R, mode, kind, narrow);
    // a tuned stage count (h2_autotune) below the number that fits
    if (stages >= 2 && stages < g.nstages) g.nstages = stages;
    // A parity wait is exact only while its waiter cannot get two uses of a stage
    // ahead (the protocol model in tests/test_pipeline_protocol.py checks this).
    // The FP32 issuers wait on the in-order splitter, which keeps them in step;
    // the BF16 kernel has one issuer, which waits on every stage in order.
    if (g.nstages < 2) { set_error("tensor-core stage does not fit in shared memory"); return H2_E_UNSUPPORTED; }
    p.a_stage_bytes = g.a_bytes;
    p.nstages = g.nstages;
    int rc = tc_prepare();
    if (rc) return rc;
    const int smem = g.nstages * g.stage_bytes + g.after + 128;
    if (kind == 0) {
        if (mode == 0) return launch_one<0, 0>(p, narrow, smem, overlap, st);
        if (mode == 1) return launch_one<1, 0>(p, narrow, smem, overlap, st);
        if (mode == 4) return launch_one<4, 0>(p, narrow, smem, overlap, st);
        set_error(mode == 2 ? "matrix-free coupling runs on the TF32 path only"
                            : "the tensor-core transfer passes run on the TF32 path only");
        return H2_E_UNSUPPORTED;
    }
    if (mode == 2) return launch_one<2, 1>(p, narrow, smem, overlap, st);
    if (mode == 3) return launch_one<3, 1>(p, narrow, smem, overlap, st);
    if (mode == 4) return launch_one<4, 1>(p, narrow, smem, overlap, st);
    if (mode == 0) return launch_one<0, 1>(p, narrow, smem, overlap, st);
    return launch_one<1, 1>(p, narrow, smem, overlap, st);
}

int launch_pack_tiles(const TcPackTile* tiles, int64_t count, const double* src, uint8_t* dst, int es,
                      cudaStream_t st) {
    if (count <= 0) return 0;
    const unsigned g = (unsigned)std::min<int64_t>(count, 152 * 16);
    k_pack_tiles<<<g, 256, 0, st>>>(tiles, count, src, dst, es);
    H2_LAUNCH_CHECK();
    return 0;
}

int launch_pack_act(const float* src, int64_t ld, int ids, const int32_t* idmap, const int32_t* base,
                    const int32_t* kdim, int kdim_fixed, const int64_t* koff, int kp_fixed, int mc, int R,
                    uint8_t* dst, int es, cudaStream_t st) {
    if (ids <= 0) return 0;
    const unsigned g = (unsigned)std::min(ids, 152 * 8);
    k_pack_act<<<g, 256, 0, st>>>(src, ld, ids, idmap, base, kdim, kdim_fixed, koff, kp_fixed, mc, R, dst, es);
    H2_LAUNCH_CHECK();
    return 0;
}

int launch_zero_tiles(const int32_t* ids, int count, uint8_t* buf, int64_t tile_bytes, cudaStream_t st) {
    if (count <= 0) return 0;
    k_zero_tiles<<<(unsigned)std::min(count, 152 * 8), 256, 0, st>>>(ids, count, buf, tile_bytes);
    H2_LAUNCH_CHECK();
    return 0;
}

int launch_zero_clusters(const int32_t* ids, int count, float* yhat, int k, int ldc, int mc, cudaStream_t st) {
    if (count <= 0) return 0;
    k_zero_clusters<<<(unsigned)std::min(count, 152 * 8), 256, 0, st>>>(ids, count, yhat, k, ldc, mc);
    H2_LAUNCH_CHECK();
    return 0;
}

}  // namespace h2
