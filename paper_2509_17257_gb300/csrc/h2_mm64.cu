// The FP64 phases of the H² product (Sec. 3 Alg. "H2_mvm" with the k×m
// coefficient blocks of Sec. 4).
//
// An SM of this GPU issues two FP64 multiply-adds per cycle, so a warp's DFMA
// holds the FP64 pipe for 16 cycles: the floor of every phase is its count of
// multiply-adds, and what has to be avoided is work on padding and SMs that
// stand idle while others finish.  So no operand is staged in shared memory for
// the contractions (a thread reads both operands through L1: two rows of S and
// one row of x̂ cost three loads per two DFMAs, 32 cycles of the pipe), the
// outputs of a cluster are numbered without padding (row pair major, column
// minor) and cut into chunks of 32 pairs, one CTA each, and CTAs are issued in
// order of falling list length.  64×16 shared-memory tiles, one CTA per cluster,
// spend 4.7 times the multiply-adds at k = 27, m = 8.  Every sum has a fixed
// order, so results repeat bit for bit.
//
// The transfer passes are chains: one level waits for the next.  One cluster's
// step (24.6k DFMAs at k = 64, m = 16) takes one SM 6 µs, so each pass is cut
// into slices of 1, 2 or 4 columns, which climb and descend independently.
#include <cuda_runtime.h>

#include <algorithm>

#include "h2_async.cuh"
#include "h2_internal.cuh"

namespace h2 {

namespace {

constexpr int kT = 128;       // threads of the transfer passes' CTAs
constexpr int kColTile = 32;  // columns of one contraction CTA at most

// acc0 += A[r0, 0:K]·B[0:K, c], acc1 likewise for r1, with the row of A at a0/a1
// (stride sa between contraction indices) and the column of B at b (stride ldb).  A is
// matrix data, which no kernel of the chain writes; B comes from earlier kernels.
template <bool UNIT>
__device__ __forceinline__ void dot2(double& acc0, double& acc1, const double* __restrict__ a0,
                                     const double* __restrict__ a1, int64_t sa, const double* b,
                                     int64_t ldb, int K) {
    constexpr int U = 8;
    double x[U], u[U], v[U];
    auto load = [&](int n) {
#pragma unroll
        for (int i = 0; i < U; ++i) {
            if (i < n) {
                x[i] = b[i * ldb];
                u[i] = __ldg(a0 + (UNIT ? i : i * sa));
                v[i] = __ldg(a1 + (UNIT ? i : i * sa));
            } else {
                x[i] = u[i] = v[i] = 0.0;
            }
        }
        a0 += UNIT ? U : U * sa;
        a1 += UNIT ? U : U * sa;
        b += U * ldb;
    };
    load(min(K, U));
    for (int kk = 0; kk < K; kk += U) {
        double xc[U], uc[U], vc[U];
#pragma unroll
        for (int i = 0; i < U; ++i) { xc[i] = x[i]; uc[i] = u[i]; vc[i] = v[i]; }
        if (kk + U < K) load(min(K - kk - U, U));
#pragma unroll
        for (int i = 0; i < U; ++i) {
            if (kk + i >= K) break;
            acc0 = fma(uc[i], xc[i], acc0);
            acc1 = fma(vc[i], xc[i], acc1);
        }
    }
}

// The output pair of this thread: rows r0 and r0 + half of `rows`, column c of
// the CTA's column tile.  The contractions' CTAs, numbered (position in the work
// order, chunk of 32 pairs) in x and by column tile in y, have one warp, or
// kSplitWarps64 warps with the same outputs that take the terms of the list in
// turn.  False: no output.
struct Pair {
    int r0, r1, c;
    bool second;  // r1 is a row of its own
};
__device__ __forceinline__ bool my_pair(int rows, int m, int chunk, Pair& p) {
    const int col0 = blockIdx.y * kColTile, cw = min(kColTile, m - col0), half = (rows + 1) >> 1;
    const int o = chunk * 32 + (threadIdx.x & 31);
    if (o >= half * cw) return false;
    p.r0 = o / cw;
    p.c = col0 + o - p.r0 * cw;
    p.second = p.r0 + half < rows;
    p.r1 = p.second ? p.r0 + half : p.r0;
    return true;
}

// Sums of the CTA's warps, added in the order of the warps; true in the warp that
// holds the total.
constexpr int kSplitWarps64 = 4;
__device__ __forceinline__ bool warp_total(double& a0, double& a1) {
    __shared__ double part[kSplitWarps64 - 1][2][32];
    const int w = threadIdx.x >> 5, W = blockDim.x >> 5, lane = threadIdx.x & 31;
    if (W == 1) return true;
    if (w > 0) {
        part[w - 1][0][lane] = a0;
        part[w - 1][1][lane] = a1;
    }
    __syncthreads();
    if (w > 0) return false;
    for (int i = 0; i < W - 1; ++i) {
        a0 += part[i][0][lane];
        a1 += part[i][1][lane];
    }
    return true;
}

// ---- multiplication phase, admissible part: ŷ_t = Σ_{b∈C_t} S_b x̂_s ----
// TRANS: the list is by column cluster and S_bᵀ is applied (product with Aᵀ).
// n = 32768, q = 4, m = 16: 2721 → 2100 µs (the shared-memory tiles against this),
// 97 % of what a DFMA probe reaches (1.204 TFLOP/s); n = 8192, m = 32: 2021 → 1103;
// n = 4096, q = 3, m = 8: 336 → 40.
template <bool TRANS>
__global__ void __launch_bounds__(32 * kSplitWarps64) k_coupling64(int chunks, const int32_t* __restrict__ order,
                                                   const int32_t* __restrict__ rowptr,
                                                   const int32_t* __restrict__ other,
                                                   const int32_t* __restrict__ blk, const double* __restrict__ S,
                                                   const double* xhat, double* yhat, int k, int m) {
    chain_release();
    chain_wait();
    const int pos = blockIdx.x / chunks;
    Pair p;
    const bool live = my_pair(k, m, blockIdx.x - pos * chunks, p);
    const int t = order[pos];
    const int64_t kk = (int64_t)k * k, km = (int64_t)k * m;
    double a0 = 0.0, a1 = 0.0;
    const int e1 = live ? rowptr[t + 1] : 0;
    for (int e = rowptr[t] + (threadIdx.x >> 5); e < e1; e += blockDim.x >> 5) {
        const int64_t j = TRANS ? blk[e] : e;
        const double* Sj = S + j * kk;
        const double* x = xhat + other[e] * km + p.c;
        if (TRANS) dot2<false>(a0, a1, Sj + p.r0, Sj + p.r1, k, x, m, k);
        else dot2<true>(a0, a1, Sj + (int64_t)p.r0 * k, Sj + (int64_t)p.r1 * k, 1, x, m, k);
    }
    if (!warp_total(a0, a1) || !live) return;
    double* y = yhat + t * km + p.c;
    y[(int64_t)p.r0 * m] = a0;
    if (p.second) y[(int64_t)p.r1 * m] = a1;
}

// ---- backward transformation at the leaves + inadmissible part + shift ----
// Y[perm[off_t + i], :] += α (V_t ŷ_t + Σ_b G_b Xp|_ŝ + σ Xp|_t̂)[i, :]
// n = 32768, q = 4, m = 16: 981 → 540 µs; n = 4096, q = 3, m = 8: 279 → 47.
template <bool TRANS>
__global__ void __launch_bounds__(32 * kSplitWarps64) k_leaf64(
    int chunks, const int32_t* __restrict__ order, const int32_t* __restrict__ leaves, const int32_t* __restrict__ cl_off,
    const int32_t* __restrict__ cl_size, const int32_t* __restrict__ perm, const double* __restrict__ V,
    const double* yhat, const int32_t* __restrict__ nptr, const int32_t* __restrict__ nother,
    const int32_t* __restrict__ nblk, const int64_t* __restrict__ near_off, const double* __restrict__ G,
    const double* Xp, double* Y, int64_t ldy, double alpha, double sigma, int k, int m, int overwrite) {
    chain_release();
    chain_wait();
    const int pos = blockIdx.x / chunks;
    const int lp = order[pos];
    const int t = leaves[lp];
    const int off = cl_off[t], nt = cl_size[t];
    Pair p;
    const bool live = my_pair(nt, m, blockIdx.x - pos * chunks, p);
    const int w = threadIdx.x >> 5, W = blockDim.x >> 5;
    double a0 = 0.0, a1 = 0.0;
    // the terms in turn: V_t ŷ_t, then the nearfield list
    if (live && w == 0)
        dot2<true>(a0, a1, V + (int64_t)(off + p.r0) * k, V + (int64_t)(off + p.r1) * k, 1,
                   yhat + (int64_t)t * k * m + p.c, m, k);
    const int e1 = live ? nptr[lp + 1] : 0;
    for (int e = nptr[lp] + (w == 0 ? W : w) - 1; e < e1; e += W) {
        const int s = nother[e];
        const int64_t j = TRANS ? nblk[e] : e;
        const int ns = cl_size[s];
        const double* Gj = G + near_off[j];
        const double* x = Xp + (int64_t)cl_off[s] * m + p.c;
        // G_j is |row leaf| × |column leaf| row-major; for Aᵀ the row leaf is s.
        if (TRANS) dot2<false>(a0, a1, Gj + p.r0, Gj + p.r1, nt, x, m, ns);
        else dot2<true>(a0, a1, Gj + (int64_t)p.r0 * ns, Gj + (int64_t)p.r1 * ns, 1, x, m, ns);
    }
    if (!warp_total(a0, a1) || !live) return;
    auto put = [&](int i, double a) {
        double* y = Y + (int64_t)perm[off + i] * ldy + p.c;
        const double z = a + sigma * Xp[(int64_t)(off + i) * m + p.c];
        if (overwrite) *y = alpha * z; else *y += alpha * z;
    };
    put(p.r0, a0);
    if (p.second) put(p.r1, a1);
}

// ---- forward transformation at the leaves: x̂_t = V_tᵀ Xp|_t̂ ----
__global__ void __launch_bounds__(32) k_leaf_fwd64(int chunks, const int32_t* __restrict__ leaves,
                                                   const int32_t* __restrict__ cl_off,
                                                   const int32_t* __restrict__ cl_size,
                                                   const double* __restrict__ V, const double* Xp, double* xhat, int k,
                                                   int m, int* flag, int64_t nflag, unsigned* claim, int nclaim) {
    chain_release();
    chain_wait();
    // the downward pass starts from cleared flags and claim tickets
    const int64_t cta = blockIdx.y * (int64_t)gridDim.x + blockIdx.x, ctas = (int64_t)gridDim.x * gridDim.y;
    for (int64_t e = cta * 32 + threadIdx.x; e < nflag; e += ctas * 32) flag[e] = 0;
    for (int64_t e = cta * 32 + threadIdx.x; e < nclaim; e += ctas * 32) claim[e] = 0u;
    const int lp = blockIdx.x / chunks;
    Pair p;
    if (!my_pair(k, m, blockIdx.x - lp * chunks, p)) return;
    const int t = leaves[lp];
    const int64_t off = cl_off[t];
    double a0 = 0.0, a1 = 0.0;
    dot2<false>(a0, a1, V + off * k + p.r0, V + off * k + p.r1, k, Xp + off * m + p.c, m, cl_size[t]);
    double* x = xhat + (int64_t)t * k * m + p.c;
    x[(int64_t)p.r0 * m] = a0;
    if (p.second) x[(int64_t)p.r1 * m] = a1;
}

// ---- transfer passes ----
// x (64 rows × CS columns, row stride CS) ← (F_z ⊗ F_y ⊗ F_x) x, or its
// transpose with TR: the x and y mode products, ping-pong between buf0 and buf1
// (blocks `nblk` deep: nblk independent blocks with their factors at F + 48·b);
// the z mode is left to the caller (kron_z).  The result of the y mode is in buf0.
template <bool TR>
__device__ __forceinline__ double kron_f(const double* F, int a, int mu, int nu) {
    return TR ? F[16 * a + 4 * nu + mu] : F[16 * a + 4 * mu + nu];
}
template <int CS, bool TR>
__device__ __forceinline__ void kron_xy(double* buf0, double* buf1, const double* F, int nblk) {
    const int total = nblk * 64 * CS;
    for (int e = threadIdx.x; e < total; e += kT) {
        const int b = e / (64 * CS), i = e - b * 64 * CS, r = i / CS, c = i - r * CS;
        const double* x = buf0 + b * 64 * CS + (r & ~3) * CS + c;
        double a = 0.0;
#pragma unroll
        for (int v = 0; v < 4; ++v) a = fma(kron_f<TR>(F + 48 * b, 0, r & 3, v), x[v * CS], a);
        buf1[e] = a;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < total; e += kT) {
        const int b = e / (64 * CS), i = e - b * 64 * CS, r = i / CS, c = i - r * CS;
        const double* x = buf1 + b * 64 * CS + ((r & 3) + 16 * (r >> 4)) * CS + c;
        double a = 0.0;
#pragma unroll
        for (int v = 0; v < 4; ++v) a = fma(kron_f<TR>(F + 48 * b, 1, (r >> 2) & 3, v), x[4 * v * CS], a);
        buf0[e] = a;
    }
    __syncthreads();
}
template <int CS, bool TR>
__device__ __forceinline__ double kron_z(const double* buf, const double* F, int r, int c) {
    const double* x = buf + (r & 15) * CS + c;
    double a = 0.0;
#pragma unroll
    for (int v = 0; v < 4; ++v) a = fma(kron_f<TR>(F, 2, r >> 4, v), x[16 * v * CS], a);
    return a;
}

// Partial chains of a dense k×k step: the contraction is cut into `parts` chains
// while the CTA has threads for them (a chain of 54 dependent DFMAs takes longer
// than the rest of a level's hand-off).
constexpr int kAhead = 16;  // contraction indices of one of four chains: k <= 32 there, two halves
__device__ __forceinline__ int dense_parts(int outputs) { return outputs * 4 <= kT ? 4 : (outputs * 2 <= kT ? 2 : 1); }

__device__ __forceinline__ unsigned acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void release_or(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.or.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned arrive_acq_rel(unsigned* p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// Upward pass in one launch: the second son to arrive computes the parent x̂_t =
// Σ_{t'} E_{t'}ᵀ x̂_{t'} and climbs on; the first one stops.  No CTA waits.  CTA
// (leaf, slice) owns CS columns; the arrivals of a cluster's slices are 2-bit
// fields of one counter per 64-column tile (at most 16 slices), reset by the
// second arrival.  Leaves and climb together: n = 4096, q = 3, m = 8: 162 → 45 µs;
// n = 32768, q = 4, m = 16: 307 → 173 (its multiply-adds alone take 115).
template <int CS>
__global__ void __launch_bounds__(kT) k_up64(const int32_t* __restrict__ leaves, int NL,
                                             const int32_t* __restrict__ parent, const int32_t* __restrict__ son0,
                                             const int32_t* __restrict__ son1, const double* __restrict__ E,
                                             const double* __restrict__ kron, double* xhat, unsigned* cnt, int k,
                                             int m) {
    chain_release();
    chain_wait();
    __shared__ double xs[2 * 64 * CS], ys[2 * 64 * CS], F[96];
    __shared__ int s_go;
    double fv = 0.0;
    const int tile = blockIdx.y, tiles = gridDim.y;
    const int slice = blockIdx.x / NL;
    int cl = leaves[blockIdx.x - slice * NL];
    const int c0 = tile * 64 + slice * CS, cs = min(CS, m - c0);
    if (cs <= 0) return;
    const int64_t kk = (int64_t)k * k, km = (int64_t)k * m;
    while (true) {
        const int par = parent[cl];
        if (par < 0) break;
        // the parent's factors, or this thread's entries of E, come in while the
        // arrival is on its way
        const int s0 = son0[par], s1 = son1[par];
        const int outs = k * CS, parts = kron ? 0 : dense_parts(outs);
        double ev[kAhead];
        if (kron) {
            if (threadIdx.x < 96)
                fv = __ldg(kron + (int64_t)(threadIdx.x < 48 ? s0 : s1) * 48 + threadIdx.x % 48);
        } else if (parts == 4 && threadIdx.x < outs * 4) {
            const int part = threadIdx.x / outs, i = threadIdx.x - part * outs, r = i % k;
            const int lo = (part & 1) * (k >> 1), len = (part & 1) ? k - (k >> 1) : k >> 1;
            const double* Eb = E + (part >> 1 ? s1 : s0) * kk + (int64_t)lo * k + r;
#pragma unroll
            for (int v = 0; v < kAhead; ++v) ev[v] = v < len ? __ldg(Eb + (int64_t)v * k) : 0.0;
        }
        __syncthreads();  // the CTA's stores precede thread 0's release
        if (threadIdx.x == 0) {
            unsigned* w = &cnt[(int64_t)par * tiles + tile];
            const unsigned old = (arrive_acq_rel(w, 1u << (2 * slice)) >> (2 * slice)) & 3u;
            s_go = old == 1u;
            if (old == 1u) atomicSub(w, 2u << (2 * slice));
        }
        __syncthreads();
        if (!s_go) break;
        cl = par;
        for (int e = threadIdx.x; e < 2 * k * CS; e += kT) {
            const int b = e / (k * CS), i = e - b * k * CS, r = i / CS, c = i - r * CS;
            xs[b * 64 * CS + i] = c < cs ? __ldcg(xhat + (b ? s1 : s0) * km + (int64_t)r * m + c0 + c) : 0.0;
        }
        if (kron && threadIdx.x < 96) F[threadIdx.x] = fv;
        __syncthreads();
        double* out = xhat + cl * km + c0;
        if (kron) {
            kron_xy<CS, true>(xs, ys, F, 2);
            for (int e = threadIdx.x; e < 64 * CS; e += kT) {
                const int r = e / CS, c = e - r * CS;
                const double a = kron_z<CS, true>(xs, F, r, c) + kron_z<CS, true>(xs + 64 * CS, F + 48, r, c);
                if (c < cs) out[(int64_t)r * m + c] = a;
            }
        } else {
            // chains (output, son, half of the contraction) where threads allow it
            if (parts == 4) {
                if (threadIdx.x < outs * 4) {
                    const int part = threadIdx.x / outs, i = threadIdx.x - part * outs, c = i / k;
                    const int lo = (part & 1) * (k >> 1), len = (part & 1) ? k - (k >> 1) : k >> 1;
                    const double* x = xs + (part >> 1) * 64 * CS + lo * CS + c;
                    double a = 0.0;
#pragma unroll
                    for (int v = 0; v < kAhead; ++v)
                        if (v < len) a = fma(ev[v], x[v * CS], a);
                    ys[threadIdx.x] = a;
                }
            } else for (int e = threadIdx.x; e < outs * parts; e += kT) {
                const int part = e / outs, i = e - part * outs, c = i / k, r = i - c * k;
                double a = 0.0;
                // one son each, or both in one chain
                for (int b = part; b < (parts == 2 ? part + 1 : 2); ++b) {
                    const double* Eb = E + (b ? s1 : s0) * kk + r;
                    const double* x = xs + b * 64 * CS + c;
#pragma unroll 8
                    for (int v = 0; v < k; ++v) a = fma(__ldg(Eb + (int64_t)v * k), x[v * CS], a);
                }
                if (parts > 1) ys[e] = a;
                else if (c < cs) out[(int64_t)r * m + c] = a;
            }
            if (parts > 1) {
                __syncthreads();
                for (int i = threadIdx.x; i < outs; i += kT) {
                    const int c = i / k, r = i - c * k;
                    double a = ys[i] + ys[outs + i];
                    if (parts == 4) a += ys[2 * outs + i] + ys[3 * outs + i];
                    if (c < cs) out[(int64_t)r * m + c] = a;
                }
            }
        }
    }
}

// Backward transfer pass ŷ_{t'} += E_{t'} ŷ_t in one launch.  Items are (non-root
// cluster in top-down level order, slice of CS columns).  A CTA claims the next
// item (atomic ticket), waits until its parent's ŷ is final (the parent's item
// has a smaller ticket, so a running CTA holds it; the wait is bounded and
// reports a timeout through err), adds E_{t'} ŷ_parent and sets its own bit of
// the cluster's ready flags (one word per 64-column tile, cleared by
// k_leaf_fwd64).  n = 4096, q = 3, m = 8: 99 → 34 µs; n = 32768, q = 4, m = 16: 121 → 71.
template <int CS>
__global__ void __launch_bounds__(kT) k_down64(const int32_t* __restrict__ order, int n_items, int slices,
                                               const int32_t* __restrict__ parent, const double* __restrict__ E,
                                               const double* __restrict__ kron, double* yhat,
                                               unsigned* claim, unsigned* flag, int* err, int k, int m,
                                               long long spin_limit) {
    chain_release();
    chain_wait();
    __shared__ double xs[64 * CS], ys[4 * 64 * CS], F[48];
    __shared__ int s_item, s_ok;
    const int tile = blockIdx.y, tiles = gridDim.y;
    const int64_t kk = (int64_t)k * k, km = (int64_t)k * m;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (int)atomicAdd(&claim[tile], 1u);
        __syncthreads();
        const int item = s_item;
        if (item >= n_items * slices) break;
        const int cl = order[item / slices], slice = item % slices;
        const int c0 = tile * 64 + slice * CS, cs = min(CS, m - c0);
        if (cs <= 0) continue;
        const int par = parent[cl];
        if (threadIdx.x == 0) {
            int ok = 1;
            if (parent[par] >= 0) {  // the root's ŷ is final after the coupling phase
                const unsigned* f = flag + (int64_t)par * tiles + tile;
                // spin_limit < 0: give up without looking at the flag (the timeout
                // path's test setting, h2_set_wait_limit)
                long long spins = 0;
                while (spin_limit < 0 || !((acquire_u32(f) >> slice) & 1u)) {
                    if (spin_limit < 0 || ++spins > spin_limit) { ok = 0; break; }
                    __nanosleep(32);
                }
            }
            s_ok = ok;
            if (!ok) atomicExch(err, 8);
        }
        if (kron && threadIdx.x < 48) F[threadIdx.x] = __ldg(kron + (int64_t)cl * 48 + threadIdx.x);
        // this thread's entries of E come in while thread 0 waits
        const int outs = k * CS, parts = kron ? 0 : dense_parts(outs);
        double ev[kAhead];
        if (parts == 4 && threadIdx.x < outs * 4) {
            const int part = threadIdx.x / outs, r = (threadIdx.x - part * outs) / CS;
            const int lo = k * part / 4, len = k * (part + 1) / 4 - lo;
            const double* Er = E + cl * kk + (int64_t)r * k + lo;
#pragma unroll
            for (int v = 0; v < kAhead; ++v) ev[v] = v < len ? __ldg(Er + v) : 0.0;
        }
        __syncthreads();
        if (!s_ok) break;
        for (int e = threadIdx.x; e < k * CS; e += kT) {
            const int r = e / CS, c = e - r * CS;
            xs[e] = c < cs ? __ldcg(yhat + par * km + (int64_t)r * m + c0 + c) : 0.0;
        }
        __syncthreads();
        double* out = yhat + cl * km + c0;
        if (kron) {
            kron_xy<CS, false>(xs, ys, F, 1);
            for (int e = threadIdx.x; e < 64 * CS; e += kT) {
                const int r = e / CS, c = e - r * CS;
                const double a = kron_z<CS, false>(xs, F, r, c);
                if (c < cs) out[(int64_t)r * m + c] += a;
            }
        } else {
            if (parts == 4) {
                if (threadIdx.x < outs * 4) {
                    const int part = threadIdx.x / outs, i = threadIdx.x - part * outs, c = i % CS;
                    const int lo = k * part / 4, len = k * (part + 1) / 4 - lo;
                    double a = 0.0;
#pragma unroll
                    for (int v = 0; v < kAhead; ++v)
                        if (v < len) a = fma(ev[v], xs[(lo + v) * CS + c], a);
                    ys[threadIdx.x] = a;
                }
            } else for (int e = threadIdx.x; e < outs * parts; e += kT) {
                const int part = e / outs, i = e - part * outs, r = i / CS, c = i - r * CS;
                const int lo = k * part / parts, hi = k * (part + 1) / parts;
                const double* Er = E + cl * kk + (int64_t)r * k;
                double a = 0.0;
#pragma unroll 8
                for (int v = lo; v < hi; ++v) a = fma(__ldg(Er + v), xs[v * CS + c], a);
                ys[e] = a;
            }
            __syncthreads();
            for (int i = threadIdx.x; i < outs; i += kT) {
                const int r = i / CS, c = i - r * CS;
                double a = ys[i];
                for (int p = 1; p < parts; ++p) a += ys[p * outs + i];
                if (c < cs) out[(int64_t)r * m + c] += a;
            }
        }
        __syncthreads();  // the CTA's stores precede thread 0's release
        if (threadIdx.x == 0) release_or(flag + (int64_t)cl * tiles + tile, 1u << slice);
    }
}

// Columns of one slice of the transfer passes: at most 16 slices share a
// bookkeeping word (m <= 16: 1 column each will do, m <= 32: 2, else 4 of a
// 64-column tile), and wider slices where there are many clusters anyway: above
// about 4096 (leaf, slice) pairs the claims cost more than shorter steps give
// (n = 32768, m = 16: the downward pass takes 120 µs with 16 slices, 71 with 4;
// n = 8192, m = 32: 54 with 16).
int slice_cols(int m, int64_t NL) {
    int cs = m <= 16 ? 1 : (m <= 32 ? 2 : 4);
    while (cs < 4 && NL * ((std::min(m, 64) + cs - 1) / cs) > 4096) cs *= 2;
    return cs;
}
// CTAs of a contraction: (clusters × chunks of 32 output pairs, column tiles)
dim3 chunk_grid(int64_t clusters, int chunks, int m) {
    return dim3((unsigned)(clusters * chunks), (unsigned)((m + kColTile - 1) / kColTile));
}
int chunks_of(int rows, int m) { return ((rows + 1) / 2 * std::min(kColTile, m) + 31) / 32; }
// Threads of a list contraction's CTA.  A warp alone issues a DFMA every 64
// cycles, so the longest list times its warp is a bound of its own: below 8 CTAs
// per SM four warps share a list (n = 4096, q = 3, m = 8, 5 CTAs per SM: coupling
// 90 → 40 µs, leaf phase 77 → 47 µs), above it the CTAs fill the pipe by
// themselves and one warp saves the exchange.
int list_threads(const dim3& g) { return (int64_t)g.x * g.y <= 152 * 8 ? 32 * kSplitWarps64 : 32; }

}  // namespace

int launch_up64(h2_matrix* A, const double* V, const double* E, const double* kron, const double* Xp, double* xhat,
                int m, const SyncBufs& sb, bool overlap, cudaStream_t st) {
    const int NL = (int)A->leaves.size(), CS = slice_cols(m, NL);
    const int tiles = (m + 63) / 64, slices = (std::min(m, 64) + CS - 1) / CS, chunks = chunks_of(A->k, m);
    int rc = launch_chained(overlap, k_leaf_fwd64, chunk_grid(NL, chunks, m), 32, 0, st, chunks, A->d_leaves,
                            A->d_cl_off, A->d_cl_size, V, Xp, xhat, A->k, m, sb.flag, A->nc * (int64_t)tiles, sb.claim,
                            tiles);
    if (rc || A->nc == 1) return rc;
    const dim3 g((unsigned)(NL * slices), (unsigned)tiles);
    return launch_chained(overlap, CS == 1 ? k_up64<1> : (CS == 2 ? k_up64<2> : k_up64<4>), g, kT, 0, st, A->d_leaves, NL,
                          A->d_parent, A->d_son0, A->d_son1, E, kron, xhat, sb.cnt, A->k, m);
}

int launch_down64(h2_matrix* A, const double* E, const double* kron, double* yhat, int m, const SyncBufs& sb,
                  bool overlap, cudaStream_t st) {
    const int n_items = (int)A->down_ptr[A->depth + 1], CS = slice_cols(m, (int64_t)A->leaves.size());
    if (n_items == 0) return 0;
    const int tiles = (m + 63) / 64, slices = (std::min(m, 64) + CS - 1) / CS;
    const dim3 g((unsigned)std::min<int64_t>((int64_t)n_items * slices, 152 * 12), (unsigned)tiles);
    return launch_chained(overlap, CS == 1 ? k_down64<1> : (CS == 2 ? k_down64<2> : k_down64<4>), g, kT, 0, st,
                          A->d_down_list, n_items, slices, A->d_parent, E, kron, yhat, sb.claim, (unsigned*)sb.flag,
                          sb.err, A->k, m, wait_limit());
}

int launch_coupling64(h2_matrix* A, const double* S, const double* xhat, double* yhat, int m, bool trans,
                      bool overlap, cudaStream_t st) {
    const int chunks = chunks_of(A->k, m);
    const dim3 g = chunk_grid(A->nc, chunks, m);
    return launch_chained(overlap, trans ? k_coupling64<true> : k_coupling64<false>, g, list_threads(g), 0, st, chunks,
                          trans ? A->d_admT_order : A->d_adm_order, trans ? A->d_admT_rowptr : A->d_adm_rowptr,
                          trans ? A->d_admT_row : A->d_adm_col, trans ? A->d_admT_blk : nullptr, S, xhat, yhat, A->k, m);
}

int launch_leaf64(h2_matrix* A, const double* V, const double* G, const double* yhat, const double* Xp, double* Y,
                  int64_t ldy, double alpha, int m, bool trans, bool overwrite, bool overlap, cudaStream_t st) {
    const int chunks = chunks_of((int)A->T.leaf_size, m);
    const dim3 g = chunk_grid((int64_t)A->leaves.size(), chunks, m);
    return launch_chained(overlap, trans ? k_leaf64<true> : k_leaf64<false>, g, list_threads(g), 0, st, chunks,
                          trans ? A->d_nearT_order : A->d_near_order, A->d_leaves, A->d_cl_off, A->d_cl_size, A->d_perm, V,
                          yhat, trans ? A->d_nearT_ptr : A->d_near_ptr, trans ? A->d_nearT_row : A->d_near_col,
                          trans ? A->d_nearT_blk : nullptr, A->d_near_off, G, Xp, Y, ldy, alpha, A->sigma, A->k, m,
                          overwrite ? 1 : 0);
}

}  // namespace h2
