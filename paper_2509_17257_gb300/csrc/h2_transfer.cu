// The transfer passes of the FP32 and BF16 tensor-core products (the forward and
// backward transformations of Sec. 3 Alg. "forward/backward", with the k×m
// coefficient blocks of Sec. 4), for q = 2, 3 and 4.
//
// Level by level these passes are chains: depth times a hand-off, whatever the
// work.  But interpolation reproduces polynomials, so the product of the transfer
// matrices along a path from a cluster c up to an ancestor a is itself an
// interpolation matrix, E_{c←a}[μ, ν] = L_{a,ν}(ξ_{c,μ}), and a Kronecker product
// F_z ⊗ F_y ⊗ F_x of q×q matrices like every transfer matrix.  So
//   ŷ_c = ŷ_c(coupling) + Σ_{ancestors a of c} E_{c←a} ŷ_a(coupling)
//   x̂_a = Σ_{d} E_{d←a}ᵀ x̂_d over any set of descendants d that covers a,
// sums of independent terms.  A pass is cut at one or two levels and becomes two
// or three launches, each a list of pairs (cluster, source): upward the inner
// clusters below the first cut from their leaves, those between two cuts from the
// clusters at the lower one; downward the clusters at each cut from the path to
// the cut above, then the leaves.  About twice as many pairs as transfer matrices,
// but no pair waits for another of its launch.  What bounds a launch is the latency
// of three dependent loads and the pack of the result, four CTAs an SM.
//
// Against subtree passes (one CTA per subtree, three dependent steps a level), in
// µs: n = 65536, q = 4, m = 32: gather and upward pass below the cut 68 → 48,
// downward 57 → 37 (30 now); m = 16 with the whole climb: 86 → 55 and 44 → 29; n = 262144,
// m = 16: 164 → 104 and 99 → 80; n = 8192, m = 32 with the climb: 55 → 32, 22 → 19.
// The roundings of a path are now one product's: FP32 error at n = 262144, m = 16
// 3.1e-6 → 1.2e-6.
//
// A pair is worked on by as many lanes as there are columns (a power of two, at
// most 32), one column each: the k coefficients stay in registers through the
// three mode products (3·q·k multiply-adds), loads of a row are contiguous over the lanes,
// and nothing is exchanged until the list's partial sums meet in shared memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "h2_async.cuh"
#include "h2_internal.cuh"

namespace h2 {

namespace {

constexpr int kOutF32 = 1, kOutTile = 2;  // PairItem::flags: result kept in FP32, as a split tile

// ---- factors of the pairs: F_a[i][j] over the axes a, i the output's index on
// that axis (down: the cluster's node μ, up: the ancestor's polynomial ν) ----
__device__ __forceinline__ double lagrange_at(const double* nodes, int q, int nu, double x) {
    double v = 1.0;
    for (int j = 0; j < q; ++j)
        if (j != nu) v *= (x - nodes[j]) / (nodes[nu] - nodes[j]);
    return v;
}
__global__ void k_pair_factors(const int2* __restrict__ pair, int64_t np, const double* __restrict__ nodes, int q,
                               int up, float* __restrict__ F) {
    const int q2 = q * q, per = 3 * q2;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < np * per; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = e / per;
        const int r = (int)(e % per), a = r / q2, i = (r % q2) / q, j = r % q;
        const int mu = up ? j : i, nu = up ? i : j;
        const int c = pair[p].x, anc = pair[p].y;
        F[e] = (float)lagrange_at(nodes + ((size_t)anc * 3 + a) * q, q, nu, nodes[((size_t)c * 3 + a) * q + mu]);
    }
}

// Rows 2i, 2i + 1 (high and low parts of column i) of a split tile of kp
// contraction columns, for columns i0 <= i < i1: entry κ of column i is
// x[κ·ld + i - i0] for κ < rows and i - i0 < valid, zero elsewhere.  es = 4 (TF32): v and
// v - tf32(v), the MMA reading the top 19 bits of the first; es = 2 (BF16): bf16(v) and
// bf16(v - bf16(v)).  A thread has one column, so its rows' place (cm_off) is fixed and
// the entries advance by whole core matrices.
__device__ __forceinline__ void pack_cols(uint8_t* tile, int kp, int es, int i0, int i1, const float* x, int ld,
                                          int rows, int valid) {
    const int ni = i1 - i0, per = blockDim.x / ni, g0 = threadIdx.x / ni, i = threadIdx.x - g0 * ni;
    if (g0 >= per) return;
    const int r = 2 * (i0 + i);
    uint8_t* at = tile + (r >> 3) * (kp * es >> 4) * 128 + (r & 7) * 16;
    x += i;
    const bool live = i < valid;
#pragma unroll 2
    for (int g = g0; g < kp >> 2; g += per) {
        float v[4], lo[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = (live && 4 * g + u < rows) ? x[(4 * g + u) * ld] : 0.f;
        if (es == 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) lo[u] = v[u] - __uint_as_float(__float_as_uint(v[u]) & 0xFFFFE000u);
            *(float4*)(at + g * 128) = make_float4(v[0], v[1], v[2], v[3]);
            *(float4*)(at + g * 128 + 16) = make_float4(lo[0], lo[1], lo[2], lo[3]);
        } else {
            __nv_bfloat162 h[2], l[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                h[u] = __floats2bfloat162_rn(v[2 * u], v[2 * u + 1]);
                l[u] = __floats2bfloat162_rn(v[2 * u] - __low2float(h[u]), v[2 * u + 1] - __high2float(h[u]));
            }
            uint8_t* b = at + (g >> 1) * 128 + (g & 1) * 8;
            *(uint2*)b = make_uint2(*(uint32_t*)&h[0], *(uint32_t*)&h[1]);
            *(uint2*)(b + 16) = make_uint2(*(uint32_t*)&l[0], *(uint32_t*)&l[1]);
        }
    }
}

// ---- the leaves: x̂_t = V_tᵀ X|_t̂ ----
// One CTA per leaf, the largest first; thread (tx, ty) owns rows 4ty.. and columns
// 4tx.. of the k×m result (m a multiple of 4; the mreal columns of X, zeros after
// them).  It gathers the leaf's rows of X itself, writes X|_t̂ and x̂_t as the split
// tiles the tensor-core phases read, and x̂_t in FP32 for the pairs.  On the way the
// launch clears what later ones start from: the ready flags of the hybrid coupling
// launch, ŷ of the clusters without couplings or with a split list, and the leaf
// results if some are split.  Bound by its loads' latency (record, then indices and V,
// then rows of X) and by 1535 leaves being 1.1 waves of nine CTAs an SM: V comes into
// shared memory asynchronously beside the rows of X, whose indices are read before the
// wait for the launch before.  n = 65536, m = 32 (µs): through registers, one after the
// other 28.9 → 27.1, conversions to FP32 off the FP64 pipe 25.4.
struct LeafUp {
    const int4* rec;  // per leaf: cluster, first position, points, first column of its X tile
    const int32_t* perm;
    const float* V;
    const double* X;
    int64_t ldx;
    int mreal, m, k;
    float* xhat;
    uint8_t *act, *leafX;
    int KP, R, es;
    int* zflag;
    int nflag;
    const int32_t* zid;
    int nzid;
    float* yhat;
    float* z;  // the leaf results to clear, or null
};

// acc[r][c] += Σ_kk a[kk·lda + 4ty + r]·b[kk·ldb + 4tx + c]; rows and columns past
// the valid ones read neighbouring data and give outputs nobody stores.
__device__ __forceinline__ void contract44(float (&acc)[4][4], const float* a, int lda, const float* b, int ldb, int K,
                                           int tx, int ty) {
    const float* pa = a + 4 * ty;
    const float* pb = b + 4 * tx;
#pragma unroll 4
    for (int kk = 0; kk < K; ++kk) {
        const float4 x = *(const float4*)(pa + kk * lda), y = *(const float4*)(pb + kk * ldb);
        const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = fmaf(xv[r], yv[c], acc[r][c]);
    }
}

// (float)x, rounded to nearest even, by the bit patterns: a conversion instruction
// holds the FP64 pipe (two results a cycle and SM) as long as a multiply-add does.
// What does not round to a normal number takes the instruction.
__device__ __forceinline__ float narrow(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const uint32_t e = (hi >> 20) & 2047u;
    if (e - 897u < 253u) {  // 2^-126 <= |x| < 2^127
        // sign, exponent and 23 bits of the significand; the rest decides the rounding
        const uint32_t t = (hi & 0x80000000u) | (((hi & 0x7FFFFFFFu) - 0x38000000u) << 3) | (lo >> 29);
        const uint32_t rest = lo & 0x1FFFFFFFu;
        return __uint_as_float(t + (rest + (t & 1u) > 0x10000000u ? 1u : 0u));
    }
    return (float)x;
}

// FULL: k = 64 and m = 16·CN, so that every stride is a constant.
template <int CN, bool FULL>
__global__ void __launch_bounds__(CN == 4 ? 256 : 128) k_leaf_up(const LeafUp p) {
    constexpr int T = CN == 4 ? 256 : 128;
    constexpr int H = T / (64 * CN);  // 2 with at most 16 columns: each half contracts half of the points
    __shared__ __align__(16) float sv[64 * 64];       // V_t, then x̂_t
    __shared__ __align__(16) float sx[64 * 16 * CN];  // X|_t̂
    __shared__ __align__(16) float sh[H == 2 ? 64 * 16 : 4];  // the second half's sums
    chain_release();
    const int4 rec = p.rec[blockIdx.x];
    const int t = rec.x, off = rec.y, nt = rec.z;
    const int k = FULL ? 64 : p.k, m = FULL ? 16 * CN : p.m;
    // rows of X by the caller's order, a group of lanes along the columns: thread rows
    // sub, sub + step, ... (at most 16: 64 points, groups of at most 32 lanes)
    const int lg = m <= 4 ? 2 : (m <= 8 ? 3 : (m <= 16 ? 4 : 5));
    const int sub = threadIdx.x >> lg, col = threadIdx.x & ((1 << lg) - 1), step = T >> lg;
    constexpr int NR = 64 * 32 / T;
    int row[NR];
#pragma unroll
    for (int u = 0; u < NR; ++u) row[u] = sub + u * step < nt ? __ldg(p.perm + off + sub + u * step) : 0;
    const int ldv = (k + 3) & ~3;
    const float* V = p.V + (int64_t)off * k;
    if (ldv == k) {
        // straight into shared memory, in flight beside the rows of X
        for (int e = threadIdx.x; e < nt * k / 4; e += T)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(sv + 4 * e)), "l"(V + 4 * e) : "memory");
    } else {
#pragma unroll 4
        for (int e = threadIdx.x; e < nt * k; e += T) sv[(e / k) * ldv + e % k] = __ldg(V + e);
    }
    chain_wait();
    for (int c = col; c < m; c += 1 << lg) {
        const bool real = c < p.mreal;
        const double* X = p.X + c;
#pragma unroll
        for (int u0 = 0; u0 < NR; u0 += 8) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = real && sub + (u0 + u) * step < nt ? X[row[u0 + u] * p.ldx] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (sub + (u0 + u) * step < nt) sx[(sub + (u0 + u) * step) * m + c] = narrow(v[u]);
        }
    }
    {
        const int64_t i0 = blockIdx.x * (int64_t)T + threadIdx.x, n = (int64_t)gridDim.x * T;
        for (int64_t i = i0; i < p.nflag; i += n) p.zflag[i] = 0;
        const int64_t blk = (int64_t)k * m / 4;
        for (int64_t e = i0; e < p.nzid * blk; e += n)
            reinterpret_cast<float4*>(p.yhat)[p.zid[e / blk] * blk + e % blk] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p.z)
            for (int e = threadIdx.x; e < nt * m / 4; e += T)
                reinterpret_cast<float4*>(p.z + (int64_t)off * m)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // X|_t̂ first: its stores drain under the contraction
    pack_cols(p.leafX + (int64_t)rec.w * p.R * p.es, (nt + 15) & ~15, p.es, 0, p.R >> 1, sx, m, nt, m);
    const int h = threadIdx.x / (64 * CN), tt = threadIdx.x % (64 * CN);
    const int tx = tt % (4 * CN), ty = tt / (4 * CN);
    float acc[4][4] = {};
    const bool live = 4 * tx < m && 4 * ty < k;
    const int mid = H == 2 ? nt >> 1 : nt, k0 = h ? mid : 0;
    if (live) contract44(acc, sv + k0 * ldv, ldv, sx + k0 * m, m, h ? nt - mid : mid, tx, ty);
    if (H == 2 && h && live) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *(float4*)(sh + (4 * ty + r) * 16 + 4 * tx) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
    }
    __syncthreads();  // V_t has been read
    if (!h && live) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float4 v = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
            if (H == 2) {
                const float4 w = *(const float4*)(sh + (4 * ty + r) * 16 + 4 * tx);
                v.x += w.x;
                v.y += w.y;
                v.z += w.z;
                v.w += w.w;
            }
            *(float4*)(sv + (4 * ty + r) * m + 4 * tx) = v;
        }
    }
    __syncthreads();
    float4* out = reinterpret_cast<float4*>(p.xhat + (int64_t)t * k * m);
    for (int e = threadIdx.x; e < k * m / 4; e += T) out[e] = reinterpret_cast<const float4*>(sv)[e];
    pack_cols(p.act + (int64_t)t * p.KP * p.R * p.es, p.KP, p.es, 0, p.R >> 1, sv, m, k, m);
}

// ---- one launch of pairs ----
// CTA (item, tile of P columns): out_c = [own block of c +] Σ_p (F_z ⊗ F_y ⊗ F_x)_p in_{src[p]}.
// A group of P lanes takes every (groups)-th pair of the list, and adds its results
// in a block of shared memory of its own.  A pair's factors come in by the group's
// lanes together.  LOGP > 0: m = P = 2^LOGP, so that rows are at constant offsets
// (as many instructions went into addresses as into multiply-adds).  The first
// factors come in ahead of the wait for the launch before, the own block while slower
// groups finish: n = 65536, m = 32: up 19.8 → 18.2, down 12.3 + 24.7 → 9.8 + 20.5 µs.
struct Pairs {
    const PairItem* items;
    const int2* pair;  // (descendant, ancestor)
    const float* fac;
    const float* in;   // [cluster][k][m]
    float* out;        // [cluster][k][m]
    uint8_t* act;
    int m, P, logP, KP, R, es;
};
// The mode product along one axis: rows at stride S of each fiber, out_i = Σ_j F[i][j] v_j.
template <int Q, int S>
__device__ __forceinline__ void mode(float (&v)[Q * Q * Q], const float* F) {
    float f[Q * Q];
    if constexpr (Q == 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 w = reinterpret_cast<const float4*>(F)[i];
            f[4 * i] = w.x;
            f[4 * i + 1] = w.y;
            f[4 * i + 2] = w.z;
            f[4 * i + 3] = w.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q * Q; ++i) f[i] = F[i];
    }
#pragma unroll
    for (int b = 0; b < Q * Q; ++b) {
        const int at = (b / S) * S * Q + b % S;
        float o[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            o[i] = f[i * Q] * v[at];
#pragma unroll
            for (int j = 1; j < Q; ++j) o[i] = fmaf(f[i * Q + j], v[at + j * S], o[i]);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) v[at + i * S] = o[i];
    }
}
template <int Q, bool UP, int W, int LOGP>
__global__ void __launch_bounds__(32 * W, W == 4 ? 4 : 2) k_pairs(const Pairs p) {
    constexpr int K = Q * Q * Q, Q2 = Q * Q, FL = (3 * Q2 + 3) & ~3;
    extern __shared__ __align__(16) float red[];  // [groups][K][P], then the factors [groups][FL]
    const int logP = LOGP ? LOGP : p.logP, P = 1 << logP, m = LOGP ? P : p.m;
    const int col0 = LOGP ? 0 : P * blockIdx.y, mc = LOGP ? P : min(P, m - col0);
    const int grp = threadIdx.x >> logP, col = threadIdx.x & (P - 1), NG = 32 * W >> logP;
    chain_release();
    const PairItem it = p.items[blockIdx.x];
    const int np = it.p1 - it.p0;
    if (np == 0) chain_wait();
    float* mine = red + grp * K * P + col;
    float* fs = red + K * 32 * W + grp * FL;
    const bool live = LOGP || col < mc;
    for (int e0 = 0; e0 < np; e0 += NG) {
        const int e = e0 + grp;
        int src = 0;
        if (e < np) {
            if (e < kInlineSrc) {
                src = e == 0 ? it.src[0] : (e == 1 ? it.src[1] : (e == 2 ? it.src[2] : it.src[3]));
            } else {
                const int2 ca = p.pair[it.p0 + e];
                src = UP ? ca.x : ca.y;
            }
            const float* f = p.fac + (int64_t)(it.p0 + e) * 3 * Q2;
            for (int i = col; i < 3 * Q2; i += P) fs[i] = __ldg(f + i);
        }
        if (e0 == 0) chain_wait();  // the first factors do not
        __syncwarp();
        if (e < np) {
            const float* s = p.in + (int64_t)src * K * m + col0 + col;
            float v[K];
#pragma unroll
            for (int r = 0; r < K; ++r) v[r] = live ? __ldcg(s + r * m) : 0.f;
            mode<Q, 1>(v, fs);
            mode<Q, Q>(v, fs + Q2);
            mode<Q, Q2>(v, fs + 2 * Q2);
            if (e0 == 0) {
#pragma unroll
                for (int r = 0; r < K; ++r) mine[r * P] = v[r];
            } else {
#pragma unroll
                for (int r = 0; r < K; ++r) mine[r * P] += v[r];
            }
        }
        __syncwarp();
    }
    // the own block, in flight while the slower groups finish
    constexpr int NO = LOGP ? (K * (1 << LOGP) + 128 * W - 1) / (128 * W) : 1;
    float4 own[NO];
#pragma unroll
    for (int u = 0; u < NO; ++u) {
        const int e = 4 * (threadIdx.x + 32 * W * u);
        own[u] = LOGP && !UP && e < K * P ? __ldcg(reinterpret_cast<const float4*>(p.out + (int64_t)it.c * K * m + e))
                                          : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    // the own block, then the groups that had a pair, in their order; four columns a
    // thread (P is a multiple of 4, and so is m)
    const int used = min(np, NG);
    auto reduce4 = [&](int e, float4 v) {
        for (int i = 0; i < used; ++i) {
            const float4 w = *reinterpret_cast<const float4*>(red + i * K * P + e);
            v.x += w.x;
            v.y += w.y;
            v.z += w.z;
            v.w += w.w;
        }
        const int r = e >> logP, c = e & (P - 1);
        if ((it.flags & kOutF32) && c < mc)
            *reinterpret_cast<float4*>(p.out + ((int64_t)it.c * K + r) * m + col0 + c) = v;
        *reinterpret_cast<float4*>(red + e) = v;  // the first group's sums at e have been read, by this thread
    };
    if constexpr (LOGP > 0) {
#pragma unroll
        for (int u = 0; u < NO; ++u)
            if (4 * (threadIdx.x + 32 * W * u) < K * P) reduce4(4 * (threadIdx.x + 32 * W * u), own[u]);
    } else {
        for (int e = 4 * threadIdx.x; e < K * P; e += 128 * W) {
            const int c = e & (P - 1);
            reduce4(e, !UP && c < mc ? __ldcg(reinterpret_cast<const float4*>(p.out + ((int64_t)it.c * K + (e >> logP)) * m +
                                                                              col0 + c))
                                     : make_float4(0.f, 0.f, 0.f, 0.f));
        }
    }
    if (!(it.flags & kOutTile)) return;
    __syncthreads();
    const int half = p.R >> 1;
    pack_cols(p.act + (int64_t)it.c * p.KP * p.R * p.es, p.KP, p.es, col0,
              blockIdx.y + 1 == gridDim.y ? half : col0 + P, red, P, K, mc);
}

constexpr int kMaxPairSmem = 8 * 32 * (64 + 48 / 4) * 4;  // 8 warps, k = 64, 4 lanes a group

// The shallowest level that holds, with the leaves above it, at least `share` of
// the leaf count over 6 clusters: six leaves per cluster at the cut or fewer.
int cut_level(const Tree& T, int64_t n_leaves, int target, int usual) {
    for (int l = 0; l < T.depth; ++l) {
        int64_t count = 0;
        for (int64_t c = 0; c < T.n_clusters(); ++c)
            count += T.level[c] == l || (T.level[c] < l && T.is_leaf((int32_t)c));
        if (count * 6 * usual >= n_leaves * target) return l;
    }
    return T.depth;
}

template <int Q, bool UP, int W, int LOGP>
int launch_pairs_w(const Pairs& p, int n_items, bool overlap, cudaStream_t st) {
    constexpr int K = Q * Q * Q, FL = (3 * Q * Q + 3) & ~3;
    const dim3 grid((unsigned)n_items, (unsigned)((p.m + p.P - 1) / p.P));
    return launch_chained(overlap, k_pairs<Q, UP, W, LOGP>, grid, 32 * W,
                          (32 * W * K + (32 * W >> p.logP) * FL) * sizeof(float), st, p);
}
template <int Q, bool UP>
int launch_stage(const PairPass& ps, int s, Pairs p, bool overlap, cudaStream_t st) {
    const PairPass::Stage& g = ps.stages[s];
    if (g.i1 == g.i0) return 0;
    p.items = ps.items + g.i0;
    p.pair = ps.pair;
    p.fac = ps.fac;
    // As many lanes as columns, and four warps.  Where the launch leaves SMs idle and
    // that needs several rounds for the longest list, narrower column tiles (down to 8
    // columns, a sector) and then eight warps shorten it (15 lists of 16 pairs at m =
    // 32: 13 → 9 µs); with SMs busy both cost more than they give (1279 lists: 36 → 50).
    const int n = g.i1 - g.i0;
    p.logP = p.m <= 4 ? 2 : (p.m <= 8 ? 3 : (p.m <= 16 ? 4 : 5));
    auto few = [&](int lp) { return n * ((p.m + (1 << lp) - 1) >> lp) < 152; };
    while (p.logP > 3 && g.longest > (128 >> p.logP) && few(p.logP)) --p.logP;
    p.P = 1 << p.logP;
    if (g.longest > (128 >> p.logP) && few(p.logP)) return launch_pairs_w<Q, UP, 8, 0>(p, n, overlap, st);
    if (Q == 4 && p.m == p.P && p.logP == 5) return launch_pairs_w<Q, UP, 4, 5>(p, n, overlap, st);
    if (Q == 4 && p.m == p.P && p.logP == 4) return launch_pairs_w<Q, UP, 4, 4>(p, n, overlap, st);
    return launch_pairs_w<Q, UP, 4, 0>(p, n, overlap, st);
}

int g_pairs_device = -1;

int pairs_prepare() {
    int dev = 0;
    H2_CUDA_TRY(cudaGetDevice(&dev));
    if (dev == g_pairs_device) return 0;
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    H2_CUDA_TRY(cudaFuncSetAttribute(k_pairs<4, true, 8, 0>, smem, kMaxPairSmem));
    H2_CUDA_TRY(cudaFuncSetAttribute(k_pairs<4, false, 8, 0>, smem, kMaxPairSmem));
    g_pairs_device = dev;
    return 0;
}

int upload_pass(h2_matrix* A, PairPass& ps, std::vector<PairItem>& items, const std::vector<int2>& pair, bool up,
                cudaStream_t st) {
    int rc = 0;
    for (PairItem& it : items)
        for (int j = 0; j < std::min(kInlineSrc, it.p1 - it.p0); ++j)
            it.src[j] = up ? pair[it.p0 + j].x : pair[it.p0 + j].y;
    for (void* old : {(void*)ps.items, (void*)ps.pair, (void*)ps.fac}) release_allocation(A, old);
    ps.items = nullptr;
    ps.pair = nullptr;
    ps.fac = nullptr;
    const int per = 3 * A->q * A->q;
    const size_t np = std::max<size_t>(pair.size(), 1);
    if ((rc = device_alloc(A, (void**)&ps.items, items.size() * sizeof(PairItem)))) return rc;
    if ((rc = device_alloc(A, (void**)&ps.pair, np * sizeof(int2)))) return rc;
    if ((rc = device_alloc(A, (void**)&ps.fac, np * per * sizeof(float)))) return rc;
    H2_CUDA_TRY(cudaMemcpyAsync(ps.items, items.data(), items.size() * sizeof(PairItem), cudaMemcpyHostToDevice, st));
    if (!pair.empty()) {
        H2_CUDA_TRY(cudaMemcpyAsync(ps.pair, pair.data(), pair.size() * sizeof(int2), cudaMemcpyHostToDevice, st));
        k_pair_factors<<<1216, 256, 0, st>>>(ps.pair, (int64_t)pair.size(), A->d_nodes, A->q, up ? 1 : 0, ps.fac);
        H2_LAUNCH_CHECK();
    }
    return 0;
}

}  // namespace

// Lists of both passes for the cut targets A->up_target and A->down_target
// (replacing earlier ones once the stream has finished with them); sets A->up_cut.
int build_pairs(h2_matrix* A, cudaStream_t st) {
    ++A->pairs_gen;
    A->up_cut = 0;
    if (A->q < 2 || A->q > 4 || !A->use_kron) return 0;
    const Tree& T = A->T;
    const int64_t nc = A->nc, NL = (int64_t)A->leaves.size();
    // A tree that peels off a leaf a level has paths as long as it has leaves, and
    // lists that grow with their square; then the level-by-level passes serve.  (Its
    // depth is past 200, where the nested interpolation overflows in FP64 already; a
    // tree of depth 66 stays below a quarter of this.)
    const size_t most = (size_t)nc * 32 + 4096;
    A->pairs_built = false;
    if (A->up_pairs.items || A->down_pairs.items) H2_CUDA_TRY(cudaStreamSynchronize(st));
    int rc = pairs_prepare();
    if (rc) return rc;
    std::vector<int4> rec;
    std::vector<PairItem> up_items, down_items;
    std::vector<int2> up_list, down_list;
    // the copies from these vectors have finished before they go out of scope
    struct Drain {
        cudaStream_t st;
        ~Drain() { cudaStreamSynchronize(st); }
    } drain{st};
    std::vector<int64_t> end(nc);  // pre-order: the subtree of c is [c, end[c])
    for (int64_t c = nc - 1; c >= 0; --c) end[c] = T.is_leaf((int32_t)c) ? c + 1 : end[T.son1[c]];
    auto add_stage = [](PairPass& ps, const std::vector<PairItem>& items, int32_t from) {
        PairPass::Stage g{from, (int32_t)items.size(), 0};
        for (size_t i = from; i < items.size(); ++i) g.longest = std::max(g.longest, items[i].p1 - items[i].p0);
        ps.stages.push_back(g);
    };
    // longest lists first
    auto by_length = [](std::vector<PairItem>& items, int32_t from) {
        std::stable_sort(items.begin() + from, items.end(),
                         [](const PairItem& a, const PairItem& b) { return a.p1 - a.p0 > b.p1 - b.p0; });
    };
    if (!A->d_leaf_rec) {
        // the leaves by falling size; X tiles as in the leaf phase (columns rounded up to 16)
        rec.resize(NL);
        int32_t x0 = 0;
        for (int64_t lp = 0; lp < NL; ++lp) {
            const int32_t c = A->leaves[lp];
            rec[lp] = int4{c, (int32_t)T.off[c], (int32_t)T.size[c], x0};
            x0 += round16((int)T.size[c]);
        }
        std::stable_sort(rec.begin(), rec.end(), [](const int4& a, const int4& b) { return a.z > b.z; });
        if ((rc = device_alloc(A, (void**)&A->d_leaf_rec, NL * sizeof(int4)))) return rc;
        H2_CUDA_TRY(cudaMemcpyAsync(A->d_leaf_rec, rec.data(), NL * sizeof(int4), cudaMemcpyHostToDevice, st));
    }
    {
        // upward: inner clusters of the levels [cut, above) from the clusters at level
        // `above` and the leaves before it, cut after cut
        PairPass& ps = A->up_pairs;
        ps.stages.clear();
        std::vector<PairItem>& items = up_items;
        std::vector<int2>& pair = up_list;
        int above = T.depth + 1, cut = cut_level(T, NL, A->up_target, kUpTasks);
        A->up_cut = cut;
        while (above > 0) {
            const int32_t from = (int32_t)items.size();
            for (int64_t c = 0; c < nc; ++c) {
                if (T.is_leaf((int32_t)c) || T.level[c] < cut || T.level[c] >= above) continue;
                PairItem it{(int32_t)c, (int32_t)pair.size(), 0, kOutTile | (T.level[c] == cut ? kOutF32 : 0), {}};
                for (int64_t d = c + 1; d < end[c];) {
                    if (T.level[d] == above || T.is_leaf((int32_t)d)) {
                        pair.push_back(int2{(int32_t)d, (int32_t)c});
                        d = end[d];
                    } else {
                        ++d;
                    }
                }
                it.p1 = (int32_t)pair.size();
                items.push_back(it);
                if (pair.size() > most) return 0;
            }
            by_length(items, from);
            if ((int32_t)items.size() > from) add_stage(ps, items, from);
            above = cut;
            cut = cut > 5 ? (cut + 1) / 2 : 0;
        }
        ps.below_cut = A->up_cut == 0 ? (int)ps.stages.size() : (ps.stages.empty() ? 0 : 1);
        // a first cut at the depth leaves no inner cluster below it
        if (!ps.stages.empty() && A->up_cut > 0 && T.level[items[0].c] < A->up_cut) ps.below_cut = 0;
        if (items.empty()) items.push_back(PairItem{});
        if ((rc = upload_pass(A, ps, items, pair, true, st))) return rc;
    }
    {
        // downward: the inner clusters at each cut, then the leaves, from the path that
        // starts at the cut above (whose ŷ is final by then)
        PairPass& ps = A->down_pairs;
        ps.stages.clear();
        std::vector<PairItem>& items = down_items;
        std::vector<int2>& pair = down_list;
        const int cut = cut_level(T, NL, A->down_target, kDownTasks);
        std::vector<int> cuts;
        if (cut > 10) cuts.push_back((cut + 1) / 2);
        if (cut > 1) cuts.push_back(cut);
        auto path = [&](int64_t c, int32_t flags) {
            int top = 0;
            for (int b : cuts)
                if (b < T.level[c]) top = b;
            PairItem it{(int32_t)c, (int32_t)pair.size(), 0, flags, {}};
            for (int32_t a = T.parent[c]; a >= 0 && T.level[a] >= top; a = T.parent[a])
                pair.push_back(int2{(int32_t)c, a});
            it.p1 = (int32_t)pair.size();
            items.push_back(it);
        };
        for (int b : cuts) {
            const int32_t from = (int32_t)items.size();
            for (int64_t c = 0; c < nc; ++c)
                if (T.level[c] == b && !T.is_leaf((int32_t)c) && pair.size() <= most) path(c, kOutF32);
            if ((int32_t)items.size() > from) add_stage(ps, items, from);
        }
        const int32_t from = (int32_t)items.size();
        for (int32_t c : A->leaves) {
            path(c, kOutTile);
            if (pair.size() > most) return 0;
        }
        by_length(items, from);
        add_stage(ps, items, from);
        if ((rc = upload_pass(A, ps, items, pair, false, st))) return rc;
    }
    A->pairs_built = true;
    return 0;
}

// Forward transformation of m columns (mreal of X, m = mreal rounded up to a
// multiple of 4), with `below` only of the clusters at or below the cut.
int launch_forward(h2_matrix* A, const double* X, int64_t ldx, int mreal, int m, float* xhat, uint8_t* xcm,
                   uint8_t* Xcm, int R, int es, bool below, int* zflag, int nflag, const int32_t* zid, int nzid,
                   float* yhat, float* z, bool overlap, cudaStream_t st) {
    int rc = pairs_prepare();
    if (rc) return rc;
    const int NL = (int)A->leaves.size();
    LeafUp p{};
    p.rec = A->d_leaf_rec;
    p.perm = A->d_perm;
    p.V = (const float*)A->f32.V;
    p.X = X;
    p.ldx = ldx;
    p.mreal = mreal;
    p.m = m;
    p.k = A->k;
    p.xhat = xhat;
    p.act = xcm;
    p.leafX = Xcm;
    p.KP = A->tc.KP;
    p.R = R;
    p.es = es;
    p.zflag = zflag;
    p.nflag = nflag;
    p.zid = zid;
    p.nzid = nzid;
    p.yhat = yhat;
    p.z = z;
    const bool full = A->k == 64;
    auto leaves = [&](void (*kernel)(const LeafUp), int threads) {
        return launch_chained(overlap, kernel, NL, threads, 0, st, p);
    };
    if (m == 16 && full) rc = leaves(k_leaf_up<1, true>, 128);
    else if (m <= 16) rc = leaves(k_leaf_up<1, false>, 128);
    else if (m == 32 && full) rc = leaves(k_leaf_up<2, true>, 128);
    else if (m <= 32) rc = leaves(k_leaf_up<2, false>, 128);
    else if (m == 64 && full) rc = leaves(k_leaf_up<4, true>, 256);
    else rc = leaves(k_leaf_up<4, false>, 256);
    if (rc) return rc;
    const int stages = below ? A->up_pairs.below_cut : (int)A->up_pairs.stages.size();
    return launch_pairs(A, A->up_pairs, 0, stages, true, xhat, xhat, xcm, m, R, es, overlap, st);
}

// Backward transfer pass: ŷ of the leaves as split tiles, from ŷ after the coupling.
int launch_backward(h2_matrix* A, float* yhat, uint8_t* ycm, int m, int R, int es, bool overlap, cudaStream_t st) {
    return launch_pairs(A, A->down_pairs, 0, (int)A->down_pairs.stages.size(), false, yhat, yhat, ycm, m, R, es,
                        overlap, st);
}

int launch_pairs(h2_matrix* A, const PairPass& ps, int s0, int s1, bool up, const float* in, float* out, uint8_t* act,
                 int m, int R, int es, bool overlap, cudaStream_t st) {
    int rc = pairs_prepare();
    if (rc) return rc;
    Pairs p{};
    p.in = in;
    p.out = out;
    p.act = act;
    p.m = m;
    p.KP = A->tc.KP;
    p.R = R;
    p.es = es;
    for (int s = s0; s < s1 && !rc; ++s)
        if (A->q == 4) rc = up ? launch_stage<4, true>(ps, s, p, overlap, st) : launch_stage<4, false>(ps, s, p, overlap, st);
        else if (A->q == 3) rc = up ? launch_stage<3, true>(ps, s, p, overlap, st) : launch_stage<3, false>(ps, s, p, overlap, st);
        else rc = up ? launch_stage<2, true>(ps, s, p, overlap, st) : launch_stage<2, false>(ps, s, p, overlap, st);
    return rc;
}

}  // namespace h2
