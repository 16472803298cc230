// Block CG with m×m Gram matrices (variant H2_CG_GRAM): O'Leary's block CG
// written in the conjugacy form of Sec. 5.1, Alg. "CG", with the per-column
// scalars replaced by m×m matrices,
//
//   G = Pᵀ(AP),  W = PᵀR,  α = G⁻¹W,  X += Pα,  R -= (AP)α,
//   Γ = G⁻¹(AP)ᵀR,  P = R - PΓ.
//
// G⁻¹ is applied through the square-root-free Cholesky factors of G, computed with
// deflation: in index order, direction j is kept when its Schur pivot exceeds kDeflate times
// its diagonal (it is not A-dependent on the kept directions before it) and
// dropped for this step otherwise; a diagonal <p_j, A p_j> <= 0 on an active
// column is a breakdown.  Columns that reach the tolerance are frozen: their
// columns of α and Γ are zero and their direction is zero.
//
// Everything runs in FP64 on the device.  Per iteration, after the product:
//   k_gram_partial      per-CTA partial sums of [G | W] over row tiles
//   k_gram_reduce<0>    fixed-order sum of the partials: G, W
//   k_gram_solve<0>     deflating L·D·Lᵀ of G and α = G⁻¹W, 4 columns per CTA
//   k_gram_update       X += Pα, R -= (AP)α, partial sums of (AP)ᵀR and |r_j|²
//   k_gram_reduce<1>    fixed-order sum: (AP)ᵀR, |r_j|²
//   k_gram_solve<1>     active set and Γ = G⁻¹(AP)ᵀR, 4 columns per CTA
//   k_gram_dir          P = R - PΓ (zero on inactive columns)
// The row passes are FP64-FMA bound (2m² flops per row and Gram product).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "h2_internal.cuh"

namespace h2 {

namespace {

constexpr int kGramCtas = 152;   // one CTA per SM for the row passes
constexpr double kDeflate = 1e-10;
constexpr int kSolveLd = kGramMaxCols + 1;

__host__ __device__ __forceinline__ int pstride(int m) { return 2 * m * m + m; }

// Rows of a tile of the row passes: 256 elements, one a thread (m > 32: two).
template <int MP>
__host__ __device__ constexpr int tile_rows() { return MP == 64 ? 8 : 256 / MP; }

// One tile of an n×m array (ld m) in registers: elements t, t + 256 of the tile's
// rows × MP, zero outside.  The row passes load a tile's arrays while the one
// before is worked on, into two shared-memory buffers in turn, so that one barrier
// a tile is all that stands between its multiply-adds.
template <int MP>
struct TileRegs {
    static constexpr int E = tile_rows<MP>() * MP / 256;
    double v[E];
    __device__ __forceinline__ void load(const double* __restrict__ A, int64_t lda, int64_t r0, int64_t n, int m) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = threadIdx.x + 256 * e, c = o % MP;
            const int64_t row = r0 + o / MP;
            v[e] = row < n && c < m ? A[row * lda + c] : 0.0;
        }
    }
    __device__ __forceinline__ void store(double* s) const {
#pragma unroll
        for (int e = 0; e < E; ++e) s[threadIdx.x + 256 * e] = v[e];
    }
};

// part[cta][0:m²] = Uᵀ V0, part[cta][m²:2m²] = Uᵀ V1 over the CTA's row tiles
// (U, V0, V1: n×m, ld m).  MP is m rounded up to 16, 32 or 64; thread (tx, ty)
// owns entries (ty + 16a, tx + 16b).  NT = 2 (G = PᵀAP and PᵀR): of the symmetric
// G the factorisation reads the lower triangle, so the blocks above it are left
// out.  n = 8192, m = 32: 40 µs with 16-row tiles and exposed loads, 29 now (its
// multiply-adds: 23); NT = 1: 28 → 18 (13).
template <int MP, int NT>
__global__ void __launch_bounds__(256) k_gram_partial(const double* __restrict__ U, const double* __restrict__ V0,
                                                      const double* __restrict__ V1, int64_t n, int m,
                                                      double* __restrict__ part) {
    constexpr int T = MP / 16, TR = tile_rows<MP>();
    __shared__ double su[2][TR][MP], s0[2][TR][MP], s1[2][NT == 2 ? TR : 1][MP];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double a0[T][T], a1[T][T];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j) a0[i][j] = a1[i][j] = 0.0;
    const int64_t tiles = (n + TR - 1) / TR;
    TileRegs<MP> ru, r0, r1;
    auto fetch = [&](int64_t tile) {
        ru.load(U, m, tile * TR, n, m);
        r0.load(V0, m, tile * TR, n, m);
        if (NT == 2) r1.load(V1, m, tile * TR, n, m);
    };
    int b = 0;
    if (blockIdx.x < tiles) fetch(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, b ^= 1) {
        ru.store(&su[b][0][0]);
        r0.store(&s0[b][0][0]);
        if (NT == 2) r1.store(&s1[b][0][0]);
        __syncthreads();
        if (tile + gridDim.x < tiles) fetch(tile + gridDim.x);
#pragma unroll 4
        for (int r = 0; r < TR; ++r) {
            double u[T], v0[T], v1[T];
#pragma unroll
            for (int i = 0; i < T; ++i) {
                u[i] = su[b][r][ty + 16 * i];
                v0[i] = s0[b][r][tx + 16 * i];
                v1[i] = NT == 2 ? s1[b][r][tx + 16 * i] : 0.0;
            }
#pragma unroll
            for (int i = 0; i < T; ++i)
#pragma unroll
                for (int j = 0; j < T; ++j) {
                    if (NT == 1 || j <= i) a0[i][j] = fma(u[i], v0[j], a0[i][j]);
                    if (NT == 2) a1[i][j] = fma(u[i], v1[j], a1[i][j]);
                }
        }
    }
    double* out = part + (size_t)blockIdx.x * pstride(m);
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j) {
            const int r = ty + 16 * i, c = tx + 16 * j;
            if (r < m && c < m) {
                out[r * m + c] = a0[i][j];
                if (NT == 2) out[m * m + r * m + c] = a1[i][j];
            }
        }
}

// Fixed-order sum of the per-CTA partials: PHASE 0 gives G = Pᵀ(AP) (lower
// triangle by 16×16 blocks) and W = PᵀR, PHASE 1 gives C = (AP)ᵀR and |r_j|².
// Eight lanes an entry take a run of the partials each (four consecutive entries to
// a sector), so a thread has at most 19 loads one after the other instead of 152
// (26 → 10 µs at m = 32).
template <int PHASE>
__global__ void __launch_bounds__(256) k_gram_reduce(int nct, int m, GramDev g) {
    const int ps = pstride(m);
    const int nterm = PHASE == 0 ? 2 * m * m : m * m + m;
    const int lane = threadIdx.x & 31, sub = lane >> 2;
    const int e = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4 + (lane & 3);
    double s = 0.0;
    if (e < nterm) {
        const int run = (nct + 7) >> 3;
#pragma unroll 10
        for (int c = sub * run; c < min(nct, (sub + 1) * run); ++c) s += __ldcg(&g.part[(size_t)c * ps + e]);
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (e >= nterm || sub) return;
    if (e < m * m) (PHASE == 0 ? g.G : g.W)[e] = s;
    else if (PHASE == 0) g.W[e - m * m] = s;
    else g.rr[e - m * m] = s;
}

constexpr int kSolveCols = 4;     // right-hand-side columns of the m×m solve per CTA
constexpr int kSolveThreads = 256;

// The m×m step, kSolveCols columns per CTA, with G = L·D·Lᵀ on the kept
// directions: sA holds the columns of L·D (below the diagonal), rcp[j] = 1 / d_j,
// 0 for a dropped direction.
// PHASE 0: every CTA factors G (with deflation, identical in all CTAs) and solves
//   α[:, c] = G_KK⁻¹ W[K, c] for its active columns c; CTA 0 keeps the factors
//   (1 / d_j on the diagonal of L) and the kept set for PHASE 1.
// PHASE 1: each CTA updates the active set of its columns from |r_c| and solves
//   Γ[:, c] = G_KK⁻¹ C[K, c] for those still active.
// A step of the factorisation is one barrier: the thread that finishes the next
// pivot inverts it while the others update, and the right-hand sides are more
// columns of the matrix.  A substitution is one warp a column, which needs no
// barrier.  m = 32: 83 → 38 µs (PHASE 0), 45 → 17 µs (PHASE 1).
template <int PHASE>
__global__ void __launch_bounds__(kSolveThreads) k_gram_solve(int m, double tol, GramDev g, CgDev d) {
    __shared__ double sA[kGramMaxCols][kSolveLd];
    __shared__ double sB[kGramMaxCols][kSolveCols];
    __shared__ double sdg[kGramMaxCols], rcp[kGramMaxCols];
    __shared__ int sa[kGramMaxCols], sown[kSolveCols];
    __shared__ int sbrk;
    const int t = threadIdx.x;
    const int c0 = blockIdx.x * kSolveCols;
    const int nc = min(kSolveCols, m - c0);
    if (t == 0) sbrk = 0;
    for (int x = t; x < m * m; x += kSolveThreads) sA[x / m][x % m] = __ldcg(&(PHASE == 0 ? g.G : g.L)[x]);
    for (int x = t; x < m * nc; x += kSolveThreads) sB[x / nc][x % nc] = __ldcg(&g.W[(x / nc) * m + c0 + x % nc]);
    if (PHASE == 0) {
        for (int j = t; j < m; j += kSolveThreads) {
            sa[j] = d.active[j] != 0;
            sdg[j] = __ldcg(&g.G[j * m + j]);
        }
        __syncthreads();
        // 1 / d_j of a kept direction; thread 0 only
        auto pivot = [&](int j) {
            double r = 0.0;
            if (sa[j]) {
                const double gjj = sdg[j], dj = sA[j][j];
                if (!(gjj > 0.0) || !isfinite(gjj)) sbrk = 1;
                else if (dj > kDeflate * gjj) r = 1.0 / dj;
            }
            rcp[j] = r;
        };
        if (t == 0) pivot(0);
        const int tx = t & 15, ty = t >> 4;
        for (int j = 0; j < m; ++j) {
            __syncthreads();
            const double r = rcp[j];
            if (r != 0.0) {
                for (int i = j + 1 + ty; i < m; i += 16) {
                    const double f = sA[i][j] * r;
                    for (int k = j + 1 + tx; k <= i; k += 16) sA[i][k] = fma(-f, sA[k][j], sA[i][k]);
                    if (tx < nc) sB[i][tx] = fma(-f, sB[j][tx], sB[i][tx]);
                    // thread 0 finishes pivot j + 1 with its first element
                    if (t == 0 && i == j + 1) pivot(j + 1);
                }
            } else if (t == 0 && j + 1 < m) {
                pivot(j + 1);
            }
        }
        __syncthreads();
        for (int c = t; c < nc; c += kSolveThreads) sown[c] = sa[c0 + c];
        if (blockIdx.x == 0) {
            for (int x = t; x < m * m; x += kSolveThreads) {
                const int i = x / m, k = x % m;
                g.L[x] = i == k ? rcp[i] : sA[i][k];
            }
            for (int j = t; j < m; j += kSolveThreads) g.kept[j] = rcp[j] != 0.0;
        }
    } else {
        for (int j = t; j < m; j += kSolveThreads) rcp[j] = __ldcg(&g.L[j * m + j]);
        for (int c = t; c < nc; c += kSolveThreads) {
            const int col = c0 + c;
            int act = d.active[col] != 0;
            if (act) {
                const double rn = sqrt(__ldcg(&g.rr[col]));
                d.rnorm[col] = rn;
                d.conv_iter[col] += 1;  // iterations while active
                if (!isfinite(rn)) atomicOr(&d.summary[1], 1);
                if (rn / d.bnorm[col] <= tol) {
                    act = 0;
                    d.active[col] = 0;
                    atomicSub(&d.summary[0], 1);
                }
            }
            sown[c] = act;
        }
    }
    __syncthreads();
    // a warp's column: entries of rows lane and lane + 32
    const int c = t >> 5, lane = t & 31;
    double y0 = 0.0, y1 = 0.0;
    bool finite = true;
    if (c < nc) {
        y0 = lane < m ? sB[lane][c] : 0.0;
        y1 = lane + 32 < m ? sB[lane + 32][c] : 0.0;
        const double q0 = lane < m ? rcp[lane] : 0.0, q1 = lane + 32 < m ? rcp[lane + 32] : 0.0;
        if (PHASE == 1)  // L z = b
            for (int j = 0; j < m; ++j) {
                const double r = rcp[j];
                if (r == 0.0) continue;
                const double f = r * __shfl_sync(0xffffffffu, j < 32 ? y0 : y1, j & 31);
                if (lane > j && lane < m) y0 = fma(-sA[lane][j], f, y0);
                if (lane + 32 > j && lane + 32 < m) y1 = fma(-sA[lane + 32][j], f, y1);
            }
        // Lᵀ y = D⁻¹ z: entry i is final once the rows after it are; rows outside K are 0
        for (int j = m - 1; j >= 0; --j) {
            if (rcp[j] == 0.0) continue;
            const double f = __shfl_sync(0xffffffffu, j < 32 ? q0 * y0 : q1 * y1, j & 31);
            if (lane < j) y0 = fma(-sA[j][lane], f, y0);
            if (lane + 32 < j) y1 = fma(-sA[j][lane + 32], f, y1);
        }
        y0 = q0 != 0.0 ? q0 * y0 : 0.0;
        y1 = q1 != 0.0 ? q1 * y1 : 0.0;
        finite = isfinite(y0) && isfinite(y1);
        if (sown[c] && !finite) sbrk = 1;
    }
    __syncthreads();
    if (c < nc) {
        double* out = PHASE == 0 ? g.alpha : g.gamma;
        const bool ok = sown[c] && !(PHASE == 0 && sbrk);
        if (lane < m) out[lane * m + c0 + c] = ok && isfinite(y0) ? y0 : 0.0;
        if (lane + 32 < m) out[(lane + 32) * m + c0 + c] = ok && isfinite(y1) ? y1 : 0.0;
    }
    if (t == 0 && sbrk) atomicOr(&d.summary[1], 1);
}

// X += Pα, R -= Qα (Q = AP) over the CTA's row tiles, then the partial sums of
// QᵀR_new (WITH_C) and |r_j|² for k_gram_reduce<1>.  n = 8192, m = 32, without C:
// 45 → 35 µs (its multiply-adds: 27).
template <int MP, bool WITH_C>
__global__ void __launch_bounds__(256) k_gram_update(double* __restrict__ X, int64_t ldx, const double* __restrict__ P,
                                                     const double* __restrict__ Q, double* __restrict__ R, int64_t n,
                                                     int m, const double* __restrict__ alpha,
                                                     double* __restrict__ part) {
    constexpr int T = MP / 16, TR = tile_rows<MP>(), E = TileRegs<MP>::E;
    extern __shared__ __align__(16) double gsm[];
    double(*sal)[MP] = reinterpret_cast<double(*)[MP]>(gsm);             // [MP][MP]
    double(*sp)[MP] = sal + MP;                                          // [2·TR][MP]
    double(*sq)[MP] = sp + 2 * TR;                                       // [2·TR][MP]
    double(*sr)[MP] = sq + 2 * TR;                                       // [2·TR][MP], WITH_C only
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    for (int x = t; x < MP * MP; x += 256) {
        const int i = x / MP, j = x % MP;
        sal[i][j] = (i < m && j < m) ? alpha[i * m + j] : 0.0;
    }
    double acc[T][T];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < T; ++j) acc[i][j] = 0.0;
    double rr = 0.0;  // |r_j|² of this thread's rows, j = t mod MP
    const int64_t tiles = (n + TR - 1) / TR;
    TileRegs<MP> rp, rq, rres, rx;
    auto fetch = [&](int64_t tile) {
        rp.load(P, m, tile * TR, n, m);
        rq.load(Q, m, tile * TR, n, m);
        rres.load(R, m, tile * TR, n, m);
        rx.load(X, ldx, tile * TR, n, m);
    };
    int b = 0;
    if (blockIdx.x < tiles) fetch(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, b ^= 1) {
        const int64_t r0 = tile * TR;
        rp.store(&sp[b * TR][0]);
        rq.store(&sq[b * TR][0]);
        const TileRegs<MP> cr = rres, cx = rx;
        __syncthreads();
        if (tile + gridDim.x < tiles) fetch(tile + gridDim.x);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = t + 256 * e, r = b * TR + o / MP, j = o % MP;
            double xs = 0.0, rs = 0.0;
#pragma unroll 16
            for (int i = 0; i < MP; ++i) {
                xs = fma(sp[r][i], sal[i][j], xs);
                rs = fma(sq[r][i], sal[i][j], rs);
            }
            const int64_t row = r0 + o / MP;
            const double rn = cr.v[e] - rs;
            if (row < n && j < m) {
                X[row * ldx + j] = cx.v[e] + xs;
                R[row * m + j] = rn;
                rr = fma(rn, rn, rr);
            }
            if (WITH_C) sr[r][j] = row < n && j < m ? rn : 0.0;
        }
        if (WITH_C) {
            __syncthreads();
#pragma unroll
            for (int r = b * TR; r < b * TR + TR; ++r) {
                double u[T], v[T];
#pragma unroll
                for (int i = 0; i < T; ++i) {
                    u[i] = sq[r][ty + 16 * i];
                    v[i] = sr[r][tx + 16 * i];
                }
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int j = 0; j < T; ++j) acc[i][j] = fma(u[i], v[j], acc[i][j]);
            }
        }
    }
    double* out = part + (size_t)blockIdx.x * pstride(m);
    if (WITH_C)  // else k_gram_partial<MP, 1> fills them, from as many CTAs
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int j = 0; j < T; ++j) {
                const int r = ty + 16 * i, c = tx + 16 * j;
                if (r < m && c < m) out[r * m + c] = acc[i][j];
            }
    __syncthreads();  // sal has been read: its first row block takes the 256 / MP sums a column
    gsm[t] = rr;
    __syncthreads();
    if (t < m) {
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < 256 / MP; ++i) v += gsm[i * MP + t];
        out[m * m + t] = v;
    }
}
template <int MP>
constexpr int update_smem(bool with_c) { return (MP + (with_c ? 6 : 4) * tile_rows<MP>()) * MP * (int)sizeof(double); }

// P = R - PΓ on active columns, 0 on the others (in place, row tile by tile).
// n = 8192, m = 32: 27 → 20 µs (its multiply-adds: 13).
template <int MP>
__global__ void __launch_bounds__(256) k_gram_dir(double* __restrict__ P, const double* __restrict__ R, int64_t n,
                                                  int m, const double* __restrict__ gamma,
                                                  const int* __restrict__ active) {
    constexpr int TR = tile_rows<MP>(), E = TileRegs<MP>::E;
    __shared__ double sg[MP][MP];
    __shared__ double sp[2][TR][MP];
    const int t = threadIdx.x;
    for (int x = t; x < MP * MP; x += 256) {
        const int i = x / MP, j = x % MP;
        sg[i][j] = (i < m && j < m) ? gamma[i * m + j] : 0.0;
    }
    const int j = t % MP;  // the thread's column in every tile
    const bool act = j < m && active[j] != 0;
    const int64_t tiles = (n + TR - 1) / TR;
    TileRegs<MP> rp, rres;
    auto fetch = [&](int64_t tile) {
        rp.load(P, m, tile * TR, n, m);
        rres.load(R, m, tile * TR, n, m);
    };
    int b = 0;
    if (blockIdx.x < tiles) fetch(blockIdx.x);
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, b ^= 1) {
        rp.store(&sp[b][0][0]);
        const TileRegs<MP> cr = rres;
        __syncthreads();
        if (tile + gridDim.x < tiles) fetch(tile + gridDim.x);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int r = (t + 256 * e) / MP;
            const int64_t row = tile * TR + r;
            if (row >= n || j >= m) continue;
            double s = 0.0;
#pragma unroll 16
            for (int i = 0; i < MP; ++i) s = fma(sp[b][r][i], sg[i][j], s);
            P[row * m + j] = act ? cr.v[e] - s : 0.0;
        }
    }
}

__global__ void k_gram_mask(double* __restrict__ P, int64_t n, int m, const int* __restrict__ active) {
    const int64_t total = n * m;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x)
        if (!active[e % m]) P[e] = 0.0;
}

// CTAs of a row pass of n rows
template <int MP>
unsigned row_grid(int64_t n) {
    constexpr int rows = tile_rows<MP>();
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + rows - 1) / rows, kGramCtas));
}

template <int MP>
int launch_alpha(const double* P, const double* AP, const double* R, int64_t n, int m, const GramDev& g,
                 const CgDev& d, cudaStream_t st) {
    const unsigned gp = row_grid<MP>(n);
    k_gram_partial<MP, 2><<<gp, 256, 0, st>>>(P, AP, R, n, m, g.part);
    H2_LAUNCH_CHECK();
    const unsigned gr = (unsigned)((2 * m * m + 31) / 32);
    k_gram_reduce<0><<<gr, 256, 0, st>>>((int)gp, m, g);
    H2_LAUNCH_CHECK();
    k_gram_solve<0><<<(unsigned)((m + kSolveCols - 1) / kSolveCols), kSolveThreads, 0, st>>>(m, 0.0, g, d);
    H2_LAUNCH_CHECK();
    return 0;
}

template <int MP>
int launch_update(double* X, int64_t ldx, const double* P, const double* AP, double* R, int64_t n, int m,
                  bool with_c, const GramDev& g, cudaStream_t st) {
    const unsigned gu = row_grid<MP>(n);
    const int sm = update_smem<MP>(with_c);
    if (with_c) k_gram_update<MP, true><<<gu, 256, sm, st>>>(X, ldx, P, AP, R, n, m, g.alpha, g.part);
    else k_gram_update<MP, false><<<gu, 256, sm, st>>>(X, ldx, P, AP, R, n, m, g.alpha, g.part);
    H2_LAUNCH_CHECK();
    return 0;
}

template <int MP>
int launch_c_partial(const double* AP, const double* Z, int64_t n, int m, const GramDev& g, cudaStream_t st) {
    // as many CTAs as the update pass, which left the C slots of its partials to this one
    k_gram_partial<MP, 1><<<row_grid<MP>(n), 256, 0, st>>>(AP, Z, nullptr, n, m, g.part);
    H2_LAUNCH_CHECK();
    return 0;
}

template <int MP>
int launch_gamma_dir(double* P, const double* D, int64_t n, int m, double tol, const GramDev& g, const CgDev& d,
                     cudaStream_t st) {
    const unsigned gu = row_grid<MP>(n);
    const unsigned gr = (unsigned)((m * m + m + 31) / 32);
    k_gram_reduce<1><<<gr, 256, 0, st>>>((int)gu, m, g);
    H2_LAUNCH_CHECK();
    k_gram_solve<1><<<(unsigned)((m + kSolveCols - 1) / kSolveCols), kSolveThreads, 0, st>>>(m, tol, g, d);
    H2_LAUNCH_CHECK();
    k_gram_dir<MP><<<gu, 256, 0, st>>>(P, D, n, m, g.gamma, d.active);
    H2_LAUNCH_CHECK();
    return 0;
}

size_t carve_up(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

size_t gram_scratch_bytes(int m) {
    const size_t mm = (size_t)m * m * sizeof(double);
    return carve_up((size_t)kGramCtas * pstride(m) * sizeof(double)) + 5 * carve_up(mm) +
           carve_up(m * sizeof(double)) + carve_up(m * sizeof(int)) + carve_up(sizeof(unsigned));
}

void gram_carve(GramDev* g, void* base, int m) {
    char* p = (char*)base;
    const size_t mm = carve_up((size_t)m * m * sizeof(double));
    g->part = (double*)p;
    p += carve_up((size_t)kGramCtas * pstride(m) * sizeof(double));
    g->G = (double*)p;
    p += mm;
    g->W = (double*)p;
    p += mm;
    g->L = (double*)p;
    p += mm;
    g->alpha = (double*)p;
    p += mm;
    g->gamma = (double*)p;
    p += mm;
    g->rr = (double*)p;
    p += carve_up(m * sizeof(double));
    g->kept = (int*)p;
    p += carve_up(m * sizeof(int));
    g->ticket = (unsigned*)p;
}

namespace {
int g_gram_attr_device = -1;
}

int gram_prepare() {
    int dev = 0;
    H2_CUDA_TRY(cudaGetDevice(&dev));
    if (dev == g_gram_attr_device) return 0;
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    H2_CUDA_TRY(cudaFuncSetAttribute(k_gram_update<64, true>, smem, update_smem<64>(true)));
    H2_CUDA_TRY(cudaFuncSetAttribute(k_gram_update<64, false>, smem, update_smem<64>(false)));
    g_gram_attr_device = dev;
    return 0;
}

int gram_start(double* P, const double* R, int64_t n, int m, const GramDev& g, const CgDev& d, cudaStream_t st) {
    if (m < 1 || m > kGramMaxCols) { set_error("the Gram-matrix block CG takes 1 <= m <= 64 columns"); return H2_E_UNSUPPORTED; }
    H2_CUDA_TRY(cudaMemsetAsync(g.ticket, 0, sizeof(unsigned), st));
    H2_CUDA_TRY(cudaMemsetAsync(P, 0, (size_t)n * m * sizeof(double), st));
    H2_CUDA_TRY(cudaMemsetAsync(g.gamma, 0, (size_t)m * m * sizeof(double), st));
    if (m <= 16) k_gram_dir<16><<<row_grid<16>(n), 256, 0, st>>>(P, R, n, m, g.gamma, d.active);
    else if (m <= 32) k_gram_dir<32><<<row_grid<32>(n), 256, 0, st>>>(P, R, n, m, g.gamma, d.active);
    else k_gram_dir<64><<<row_grid<64>(n), 256, 0, st>>>(P, R, n, m, g.gamma, d.active);
    H2_LAUNCH_CHECK();
    return 0;
}

int gram_alpha(const double* P, const double* AP, const double* R, int64_t n, int m, const GramDev& g,
               const CgDev& d, cudaStream_t st) {
    if (m <= 16) return launch_alpha<16>(P, AP, R, n, m, g, d, st);
    if (m <= 32) return launch_alpha<32>(P, AP, R, n, m, g, d, st);
    return launch_alpha<64>(P, AP, R, n, m, g, d, st);
}

#define H2_GRAM_DISPATCH(call) (m <= 16 ? call<16> : m <= 32 ? call<32> : call<64>)

int gram_update_dir(double* X, int64_t ldx, double* P, const double* AP, double* R, int64_t n, int m, double tol,
                    const GramDev& g, const CgDev& d, cudaStream_t st) {
    int rc = H2_GRAM_DISPATCH(launch_update)(X, ldx, P, AP, R, n, m, true, g, st);
    if (rc) return rc;
    return H2_GRAM_DISPATCH(launch_gamma_dir)(P, R, n, m, tol, g, d, st);
}

int gram_update(double* X, int64_t ldx, const double* P, const double* AP, double* R, int64_t n, int m,
                const GramDev& g, cudaStream_t st) {
    return H2_GRAM_DISPATCH(launch_update)(X, ldx, P, AP, R, n, m, false, g, st);
}

int gram_gamma_dir_from(double* P, const double* AP, const double* Z, int64_t n, int m, double tol,
                        const GramDev& g, const CgDev& d, cudaStream_t st) {
    int rc = H2_GRAM_DISPATCH(launch_c_partial)(AP, Z, n, m, g, st);
    if (rc) return rc;
    return H2_GRAM_DISPATCH(launch_gamma_dir)(P, Z, n, m, tol, g, d, st);
}

int gram_mask(double* P, int64_t n, int m, const CgDev& d, cudaStream_t st) {
    const unsigned g = (unsigned)std::min<int64_t>((n * m + 255) / 256, 152 * 16);
    k_gram_mask<<<g, 256, 0, st>>>(P, n, m, d.active);
    H2_LAUNCH_CHECK();
    return 0;
}

}  // namespace h2
