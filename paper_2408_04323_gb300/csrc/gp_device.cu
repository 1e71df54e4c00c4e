// The per-round GP state (Section 4.3) built on the device: features of the
// observations, K + tau^2 I in fp64, its Cholesky factor, L^{-1} and
// alpha = (K + tau^2 I)^{-1} y, written into the same blob layout that the
// host preparation produces and the posterior and scoring kernels read.
//
// L^{-1} comes out of the factorisation itself: the elimination that turns
// K into L^T, applied to the identity, gives L^{-1}.  At step j, with pivot
// p_j = sqrt(A_jj) and l_ij = A_ij / p_j, every row i > j takes
//   A_ik -= l_ij l_kj   (j < k <= i)   and   W_ic -= l_ij W_jc / p_j   (c <= j),
// and row i of L^{-1} is W_i / p_i once the steps before i are done.  The
// rows of one step are independent, so a step is one barrier.  fp64 runs at
// a small fraction of the fp32 rate on this GPU; the n^3/3 multiply-adds of
// a factorisation are its cost.
#include <cmath>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "approx.cuh"
#include "internal.h"

namespace {

using namespace scoot_dev;

constexpr int kFeatThreads = 128;
constexpr int kKmatThreads = 128;
constexpr int kCholThreads = 1024;
constexpr int kRowBlockDev = 64;   // rows of L^{-1} per tile (the layout's)
constexpr int kColChunkDev = 32;   // columns of L^{-1} per tile
constexpr int kOneTriangleN = 160; // scratch of one packed triangle per objective up to this n, of two above

struct GpPrepArgs {
    int32_t n, d, M, kernel, n_ord, n_pat, n_rb, n_tiles;
    int64_t tri;                        // n (n + 1) / 2
    int32_t order[SCOOT_MAX_DIM];       // feature f -> source parameter
    int32_t kind[SCOOT_MAX_DIM];        // per source parameter
    int32_t n_choices[SCOOT_MAX_DIM];
    double lo[SCOOT_MAX_DIM], span[SCOOT_MAX_DIM];  // ordinal: (v - lo) / span; log: (ln v - lo) / span
    float fmap[SCOOT_MAX_DIM][4];       // the blob's feature map, computed on the host
    const uint32_t* obs;
    int64_t ld_obs;
    const float* y;                     // [M][n]
    const float* ls;                    // [M][d], source order
    const float* sf2;                   // [M]
    const float* tau2;                  // [M]
    const float* warp;                  // [M][d][2] or nullptr
    char* blob;
    int64_t off_fmap, off_xs, off_ils, off_alpha, off_linv, off_scal, off_cat, off_warp;
    double* U;                          // [M][n][d] scaled features, source order
    double* K;                          // [M][tri] packed lower triangle of K + tau^2 I (factorised in place when n is large)
    double* W;                          // [M][tri] elimination of the identity (NULL up to kOneTriangleN)
    uint32_t* err;
};

__device__ __forceinline__ int64_t tri_idx(int i, int k) { return (int64_t)i * (i + 1) / 2 + k; }

__device__ __forceinline__ double matern_dev(double r, int kernel) {
    if (kernel == SCOOT_MATERN32) {
        const double a = 1.7320508075688772 * r;  // sqrt(3) r
        return (1.0 + a) * exp(-a);
    }
    const double a = 2.23606797749979 * r;  // sqrt(5) r
    return (1.0 + a + a * a / 3.0) * exp(-a);
}

// One thread per (observation j, feature f) of objective m: the feature,
// warped and scaled (fp64 logarithms and powers are slow here, so they are
// spread over n d threads).
__global__ void __launch_bounds__(kFeatThreads) gp_feat_kernel(const __grid_constant__ GpPrepArgs a) {
    const int t = blockIdx.x * kFeatThreads + threadIdx.x, m = blockIdx.y;
    const int d = a.d, j = t / d, f = t - j * d;
    bool bad = false;
    if (j < a.n) {
        float* xs = reinterpret_cast<float*>(a.blob + a.off_xs) + ((int64_t)m * a.n + j) * d;
        double* U = a.U + ((int64_t)m * a.n + j) * d;
        const int c = a.order[f];
        const uint32_t w = a.obs[(int64_t)c * a.ld_obs + j];
        const double l = (double)a.ls[m * d + c];
        bad |= !(l > 0.0) || !isfinite(l);
        if (a.kind[c] == SCOOT_CATEGORICAL) {
            const double u = (double)(int32_t)w;
            U[c] = u;
            xs[f] = (float)u;
        } else {
            const double v = a.kind[c] == SCOOT_CONTINUOUS ? (double)__uint_as_float(w) : (double)(int32_t)w;
            bad |= !isfinite(v) || (a.kind[c] == SCOOT_INT_LOG && !(v > 0.0));
            double u;
            if (a.kind[c] == SCOOT_INT_LOG) u = (log(v) - a.lo[c]) / a.span[c];
            else u = a.span[c] > 0.0 ? (v - a.lo[c]) / a.span[c] : 0.0;
            if (a.warp) {
                const double wa = (double)a.warp[((int64_t)m * d + c) * 2];
                const double wb = (double)a.warp[((int64_t)m * d + c) * 2 + 1];
                bad |= !(wa > 0.0) || !isfinite(wa) || !(wb > 0.0) || !isfinite(wb);
                const double x = fmin(fmax(u, 0.0), 1.0);
                u = 1.0 - pow(1.0 - pow(x, wa), wb);
            }
            U[c] = u / l;
            xs[f] = (float)(u / l);
        }
        if (f == 0) bad |= !isfinite(a.y[(int64_t)m * a.n + j]);
    }
    if (t == 0) {  // per-objective scalars (thread 0 of the objective's first block)
        const float sf2 = a.sf2[m], tau2 = a.tau2[m];
        bad |= !(sf2 > 0.0f) || !isfinite(sf2) || !(tau2 >= 0.0f) || !isfinite(tau2);
        float* ils = reinterpret_cast<float*>(a.blob + a.off_ils) + m * d;
        float* wo = reinterpret_cast<float*>(a.blob + a.off_warp) + (int64_t)m * d * 2;
        for (int g = 0; g < d; ++g) {
            const int c = a.order[g];
            const double l = (double)a.ls[m * d + c];
            const bool cat = a.kind[c] == SCOOT_CATEGORICAL;
            ils[g] = cat ? (float)(1.0 / (l * l)) : (float)(1.0 / l);
            wo[2 * g] = (a.warp && !cat) ? a.warp[((int64_t)m * d + c) * 2] : 1.0f;
            wo[2 * g + 1] = (a.warp && !cat) ? a.warp[((int64_t)m * d + c) * 2 + 1] : 1.0f;
        }
        float* scal = reinterpret_cast<float*>(a.blob + a.off_scal) + m * 4;
        scal[0] = sf2;
        scal[1] = tau2;
        scal[3] = a.warp ? 1.0f : 0.0f;  // scal[2] (best observed y) is written by the factorisation
        if (m == 0) {
            float* fm = reinterpret_cast<float*>(a.blob + a.off_fmap);
            for (int g = 0; g < d; ++g)
                for (int q = 0; q < 4; ++q) fm[g * 4 + q] = a.fmap[g][q];
        }
    }
    if (bad) atomicOr(a.err, SCOOT_DEVERR_VALUE);
}

// Categorical part of r^2 for every (observation, category pattern).
__global__ void __launch_bounds__(kKmatThreads) gp_cat_kernel(const __grid_constant__ GpPrepArgs a) {
    const int64_t t = (int64_t)blockIdx.x * kKmatThreads + threadIdx.x;
    const int m = blockIdx.y;
    if (t >= (int64_t)a.n * a.n_pat) return;
    const int j = (int)(t / a.n_pat), pat = (int)(t - (int64_t)j * a.n_pat);
    double r2 = 0.0;
    int rest = pat;
    for (int f = a.n_ord; f < a.d; ++f) {
        const int c = a.order[f];
        const int v = rest % a.n_choices[c];
        rest /= a.n_choices[c];
        const double l = (double)a.ls[m * a.d + c];
        if (v != (int32_t)a.obs[(int64_t)c * a.ld_obs + j]) r2 += 1.0 / (l * l);
    }
    reinterpret_cast<float*>(a.blob + a.off_cat)[((int64_t)m * a.n + j) * a.n_pat + pat] = (float)r2;
}

// K + tau^2 I, one thread per entry of the lower triangle.
__global__ void __launch_bounds__(kKmatThreads) gp_kmat_kernel(const __grid_constant__ GpPrepArgs a) {
    const int64_t t = (int64_t)blockIdx.x * kKmatThreads + threadIdx.x;
    const int m = blockIdx.y;
    if (t >= a.tri) return;
    int i = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while ((int64_t)i * (i + 1) / 2 > t) --i;
    while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
    const int k = (int)(t - (int64_t)i * (i + 1) / 2);
    const double* ui = a.U + ((int64_t)m * a.n + i) * a.d;
    const double* uk = a.U + ((int64_t)m * a.n + k) * a.d;
    double r2 = 0.0;
    for (int c = 0; c < a.d; ++c) {
        const double diff = ui[c] - uk[c];
        if (a.kind[c] == SCOOT_CATEGORICAL) {
            const double l = (double)a.ls[m * a.d + c];
            r2 += diff != 0.0 ? 1.0 / (l * l) : 0.0;
        } else {
            r2 += diff * diff;
        }
    }
    double v = (double)a.sf2[m] * matern_dev(sqrt(r2), a.kernel);
    if (i == k) v += (double)a.tau2[m];
    a.K[(int64_t)m * a.tri + t] = v;
}

// The factorisation of the packed lower triangle A (n x n, K + tau^2 I on
// entry) with the elimination applied to the identity in W, by the whole
// block.  On return, row i of L^{-1} is W_i * rinv[i];
// rinv2[i] = rinv[i]^2; A holds the eliminated values.  col: [2][n] scratch.
// Returns false (in every thread) if a pivot is not positive and finite.
//
// Step j in a single multiply-add per entry: with g_i = A_ij / A_jj,
//   A_ik -= g_i A_kj (j < k <= i)   and   W_ic -= g_i W_jc (c <= j),
// one loop over t = 0 .. i per row (t <= j: W, t > j: A) so that the lanes
// of a warp stay busy.  Column j is read from a contiguous copy (col), which
// the threads that finish its entries in step j - 1 write (two buffers by
// step parity).
__device__ bool eliminate(double* A, double* W, double* col, double* rinv, double* rinv2, int n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    // s_bad_at: the first step whose pivot is not positive (n if none).  It is
    // written during step j - 1 with the value j, so a thread still reading it
    // for step j - 1 does not stop early; every thread stops at step j.  The
    // pivot's reciprocals are computed once, by the thread that finishes the
    // diagonal entry (fp64 square roots and divisions are slow here), and
    // read after the step's barrier.
    __shared__ int s_bad_at;
    __syncthreads();  // A is complete; s_bad_at of an earlier call is read by no one
    for (int i = warp; i < n; i += nwarps)
        for (int c = lane; c <= i; c += 32) W[tri_idx(i, c)] = c == i ? 1.0 : 0.0;
    for (int i = tid; i < n; i += (int)blockDim.x) col[i] = A[tri_idx(i, 0)];
    if (tid == 0) {
        const double s0 = A[0];
        const bool bad = !(s0 > 0.0) || !isfinite(s0);
        s_bad_at = bad ? 0 : n;
        rinv[0] = bad ? 0.0 : rsqrt_newton(s0);
        rinv2[0] = rinv[0] * rinv[0];
    }
    __syncthreads();
    for (int j = 0; j < n; ++j) {
        if (s_bad_at <= j) break;  // the same in every thread
        const double r2 = rinv2[j];
        const double* cj = col + (j & 1) * n;
        double* cn = col + ((j + 1) & 1) * n;
        const double* Wj = W + tri_idx(j, 0);
        for (int i = j + 1 + warp; i < n; i += nwarps) {
            double* Ai = A + tri_idx(i, 0);
            double* Wi = W + tri_idx(i, 0);
            const double g = cj[i] * r2;
            for (int t = lane; t <= i; t += 32) {
                double* dst = t <= j ? Wi + t : Ai + t;
                const double src = t <= j ? Wj[t] : cj[t];
                const double v = *dst - g * src;
                *dst = v;
                if (t == j + 1) {  // A[i][j+1] is final: column j + 1 of the next step
                    cn[i] = v;
                    if (i == j + 1) {
                        if (!(v > 0.0) || !isfinite(v)) {
                            s_bad_at = j + 1;
                        } else {
                            const double y = rsqrt_newton(v);
                            rinv[j + 1] = y;
                            rinv2[j + 1] = y * y;
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    const bool ok = s_bad_at >= n;  // read after the loop's last barrier: the same in every thread
    __syncthreads();                // before a later call rewrites s_bad_at
    return ok;
}

// (For more observations than gp_chol_cluster_kernel holds.)
// One block per objective: the factorisation with L^{-1} alongside, then
// alpha, the best observed y and the fp32 tiles of L^{-1}.
__global__ void __launch_bounds__(kCholThreads) gp_chol_kernel(const __grid_constant__ GpPrepArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, m = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kCholThreads / 32;
    double* rinv = reinterpret_cast<double*>(smem_raw);  // [n] 1 / pivot
    double* rinv2 = rinv + n;                            // [n] 1 / pivot^2
    double* z = rinv2 + n;                               // [n] L^{-1} y
    double* col = z + n;                                 // [2][n] column j of A
    double* A = a.K + (int64_t)m * a.tri;
    double* W = a.W + (int64_t)m * a.tri;
    if (!eliminate(A, W, col, rinv, rinv2, n)) {
        if (tid == 0) atomicOr(a.err, SCOOT_DEVERR_VALUE);
        return;
    }
    const float* y = a.y + (int64_t)m * n;
    // z = L^{-1} y, a warp per row
    for (int i = warp; i < n; i += nwarps) {
        const double* Wi = W + tri_idx(i, 0);
        double t = 0.0;
        for (int c = lane; c <= i; c += 32) t += Wi[c] * (double)y[c];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) z[i] = t * rinv[i];
    }
    __syncthreads();
    // alpha = L^{-T} z, a thread per column
    float* alpha = reinterpret_cast<float*>(a.blob + a.off_alpha) + (int64_t)m * n;
    for (int c = tid; c < n; c += kCholThreads) {
        double t = 0.0;
        for (int i = c; i < n; ++i) t += W[tri_idx(i, c)] * rinv[i] * z[i];
        alpha[c] = (float)t;
    }
    if (warp == 0) {
        float best = -INFINITY;
        for (int j = lane; j < n; j += 32) best = fmaxf(best, y[j]);
        for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (lane == 0) reinterpret_cast<float*>(a.blob + a.off_scal)[m * 4 + 2] = best;
    }
    // tiles: row block rb, column chunk cj; tile[jj][ii] = L^{-1}[64 rb + ii][32 cj + jj]
    float* tiles = reinterpret_cast<float*>(a.blob + a.off_linv) + (int64_t)m * a.n_tiles * kColChunkDev * kRowBlockDev;
    const int64_t total = (int64_t)a.n_tiles * kColChunkDev * kRowBlockDev;
    for (int64_t e = tid; e < total; e += kCholThreads) {
        const int t = (int)(e / (kColChunkDev * kRowBlockDev));
        const int jj = (int)(e / kRowBlockDev % kColChunkDev), ii = (int)(e % kRowBlockDev);
        int rb = 0;
        while ((rb + 1) * (rb + 2) <= t) ++rb;  // tiles of row blocks before rb: rb (rb + 1)
        const int cj = t - rb * (rb + 1);
        const int row = rb * kRowBlockDev + ii, c = cj * kColChunkDev + jj;
        float v = 0.0f;
        if (row < n && c <= row) v = (float)(W[tri_idx(row, c)] * rinv[row]);
        tiles[e] = v;
    }
}

constexpr int kClusterCTAs = 8;          // CTAs sharing one factorisation (portable cluster size)
constexpr int kClusterThreads = 256;
constexpr int kClusterB = kClusterCTAs;  // pivots per block: one row of a block per CTA

// Offset of local row li (global row rank + C li) in a CTA's packed rows:
// row i holds i + 1 entries.
__device__ __forceinline__ int64_t local_row_off(int li, int rank) {
    return (int64_t)li * (rank + 1) + (int64_t)kClusterCTAs * li * (li - 1) / 2;
}

// Entries of the CTA with the most, of rows 0 .. n over a cluster.
inline int64_t cluster_own(int n) {
    int64_t own = 0;
    for (int r = 0; r < kClusterCTAs; ++r) {
        const int64_t nl = (n + 1 - r + kClusterCTAs - 1) / kClusterCTAs;
        const int64_t e = nl * (r + 1) + (int64_t)kClusterCTAs * nl * (nl - 1) / 2;  // local_row_off(nl, r)
        if (e > own) own = e;
    }
    return own;
}

// What the eliminations of a block's pivots need of the pivot rows.
struct PanelPivots {
    double col[kClusterB][kClusterB];  // [p][c > p] entry (kb + c, kb + p) when pivot p is reached
    double rcp[kClusterB], piv[kClusterB];
};

// Eliminates pivots kb .. kb + be - 1 from the panel P ([n + 1][8], row j the
// entries of row or column j of the matrix in the block's columns) one after the
// other, by a block of kClusterThreads:
//   t = P_jp / A_pp,  P_jc -= t A_cp  for c > p,
// the operations of an unblocked elimination in its order, so no block is inverted
// (multiplying by the inverse of a block of repeated observations cost 1e3 to 1e7
// times the error).  The rows of the block are replaced by those that its columns of
// the identity end as.  gs[li][p] = t for the CTA's own rows j = rank + 8 li, the
// block's own row among them; rows before kb only if all_rows.  On return (after the
// caller's next __syncthreads) A_ij of two other rows loses gs[i] . P[j].
// Warp 0 runs the chain of pivots on the block's 8 rows and the identity's, in
// registers; the other warps follow it on their rows pivot by pivot (named barriers 1
// to 8), so that the panel costs little beyond that chain.
__device__ __forceinline__ void eliminate_panel(double* P, double* gs, PanelPivots& s, int* fail, int n, int kb, int be,
                                                int rank, bool all_rows) {
    constexpr int C = kClusterCTAs, B = kClusterB, kFirst = kClusterThreads - 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rows = n + 1 - be;  // rows outside the block
    double y[B], t[B];
#pragma unroll
    for (int p = 0; p < B; ++p) t[p] = 0.0;
    auto step = [&](int p, double rcp, const double* col) {
        t[p] = y[p] * rcp;
#pragma unroll
        for (int c = 0; c < B; ++c)
            if (c > p) y[c] = fma(-t[p], col[c], y[c]);
    };
    auto load = [&](int j) {
#pragma unroll
        for (int c = 0; c < B; ++c) y[c] = P[(size_t)j * B + c];
    };
    auto store = [&](int j) {
#pragma unroll
        for (int c = 0; c < B; ++c) P[(size_t)j * B + c] = y[c];
        if (j % C == rank && (all_rows || j >= kb)) {
#pragma unroll
            for (int c = 0; c < B; ++c) gs[(j / C) * B + c] = t[c];
        }
    };
    auto row_of = [&](int k) { return k < kb ? k : k + be; };
    if (warp == 0) {  // lanes 0 .. 7: the block's rows; 8 .. 15: the identity's
        const int r = lane % B;
#pragma unroll
        for (int c = 0; c < B; ++c) y[c] = lane < B ? (r < be ? P[(size_t)(kb + r) * B + c] : 0.0) : (r == c ? 1.0 : 0.0);
#pragma unroll
        for (int p = 0; p < B; ++p) {
            if (p >= be) break;
            const double v = __shfl_sync(0xffffffffu, y[p], p);
            double col[B];
#pragma unroll
            for (int c = 0; c < B; ++c) col[c] = c > p ? __shfl_sync(0xffffffffu, y[c], p) : 0.0;
            const bool ok = good_pivot(v);
            const double rcp = ok ? rcp_newton(v) : 0.0;
            if (lane == 0) {
                if (!ok) *fail = 1;
                s.piv[p] = v;
                s.rcp[p] = rcp;
#pragma unroll
                for (int c = 0; c < B; ++c)
                    if (c > p) s.col[p][c] = col[c];
            }
            __syncwarp();
            asm volatile("bar.arrive %0, %1;" ::"r"(p + 1), "n"(kClusterThreads) : "memory");
            step(p, rcp, col);
        }
        if (lane >= B && lane < B + be) store(kb + r);
    } else {  // (warp 4 shares warp 0's scheduler, so it comes last)
        const int k = (warp < 4 ? warp - 1 : warp == 4 ? 6 : warp - 2) * 32 + lane, j = row_of(k);
        if (k < rows) load(j);
#pragma unroll
        for (int p = 0; p < B; ++p) {
            if (p >= be) break;
            asm volatile("bar.sync %0, %1;" ::"r"(p + 1), "n"(kClusterThreads) : "memory");
            if (k < rows) step(p, s.rcp[p], s.col[p]);
        }
        if (k < rows) store(j);
    }
    for (int k = kFirst + tid; k < rows; k += kClusterThreads) {  // the rows that are left
        const int j = row_of(k);
        load(j);
#pragma unroll
        for (int p = 0; p < B; ++p) {
            if (p >= be) break;
            step(p, s.rcp[p], s.col[p]);
        }
        store(j);
    }
}

// Bytes of shared memory of gp_chol_cluster_kernel.
inline size_t chol_cluster_bytes(int n) {
    const size_t rows = (size_t)(n + 1 + kClusterCTAs - 1) / kClusterCTAs;
    return ((size_t)cluster_own(n) + 2 * (size_t)(n + 1) * kClusterB + rows * kClusterB) * sizeof(double);
}

// gp_chol_kernel's results by a cluster of eight CTAs per objective, in blocks of
// eight pivots.  CTA r owns rows i = r (mod 8) of K + tau^2 I, augmented by row n,
// which holds y^T.  The elimination is in place: entry t of row i holds A_it
// before pivot t and W_it, the elimination of the identity, after it.  A block of
// pivots kb .. kb + 7 finishes its rows of L^{-1} and takes from every later row i
//   A_ij -= g_i . P_j,   W_it -= g_i . P_t
// with the panel P and the multipliers g of eliminate_panel, so that row n ends as
// -alpha^T = -y^T (K + tau^2 I)^{-1}.  What a block needs of other CTAs' rows is
// that panel, eight values per row or column, which every CTA pushes its part
// of into all eight CTAs' shared memory: one cluster barrier per eight pivots
// (one per pivot and two triangles before).  Each CTA eliminates the panel for
// itself.
// Bound by the chain of pivots and the fp64 units (64 cycles a warp instruction
// and scheduler).  n = 200, three objectives, the whole state: 317 us, 602 with a
// barrier per pivot.
__global__ void __cluster_dims__(kClusterCTAs, 1, 1) __launch_bounds__(kClusterThreads)
gp_chol_cluster_kernel(const __grid_constant__ GpPrepArgs a, int64_t own) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int C = kClusterCTAs, B = kClusterB, nwarps = kClusterThreads / 32;
    const int n = a.n, rank = (int)cluster.block_rank(), m = blockIdx.x / C;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double* panel = reinterpret_cast<double*>(smem_raw);  // [2][n + 1][B]
    double* A = panel + 2 * (size_t)(n + 1) * B;          // owned rows, packed
    double* gs = A + own;                                 // [owned rows][B] the rows' g
    const int nl = (n + 1 - rank + C - 1) / C;            // rows owned, row n among them
    __shared__ PanelPivots pivots;
    __shared__ int s_fail;
    const double* K = a.K + (int64_t)m * a.tri;
    const float* y = a.y + (int64_t)m * n;
    if (tid == 0) s_fail = 0;
    for (int li = warp; li < nl; li += nwarps) {
        const int i = rank + C * li;
        double* Ai = A + local_row_off(li, rank);
        for (int t = lane; t <= i; t += 32) Ai[t] = i < n ? K[tri_idx(i, t)] : t < n ? (double)y[t] : 0.0;
    }
    // The panel of block kb: [j][c] = A_j,kb+c of the rows j >= kb + c (and its
    // mirror within the block), W_kb+c,j of the columns j < kb; 0 beyond pivot n - 1.
    auto push = [&](int kb) {
        const size_t off = (size_t)((kb / B) & 1) * (n + 1) * B;
        double* peer[C];  // every CTA's panel
#pragma unroll
        for (int r = 0; r < C; ++r) peer[r] = cluster.map_shared_rank(panel, r) + off;
        for (int e = tid; e < nl * B; e += kClusterThreads) {
            const int li = e / B, c = e - li * B, i = rank + C * li, kc = kb + c;
            if (kc < n && (i < kb || kc > i)) continue;
            const double v = kc < n ? A[local_row_off(li, rank) + kc] : 0.0;
#pragma unroll
            for (int r = 0; r < C; ++r) peer[r][i * B + c] = v;
        }
        const int row = kb + rank;
        if (row < n) {
            const double* Ar = A + local_row_off(row / C, rank);
            for (int j = tid; j < row; j += kClusterThreads) {
                const double v = Ar[j];
#pragma unroll
                for (int r = 0; r < C; ++r) peer[r][j * B + rank] = v;
            }
        }
    };
    cluster.sync();  // every CTA has started: its shared memory may be written
    push(0);
    cluster.sync();
    for (int kb = 0; kb < n; kb += B) {
        double* P0 = panel + (size_t)((kb / B) & 1) * (n + 1) * B;
        const int be = min(B, n - kb);
        eliminate_panel(P0, gs, pivots, &s_fail, n, kb, be, rank, false);
        __syncthreads();
        if (s_fail) break;  // the same in every CTA: each has eliminated the same panel
        for (int li = (kb / C) + warp; li < nl; li += nwarps) {
            const int i = rank + C * li, ii = i - kb;
            double* Ai = A + local_row_off(li, rank);
            if (ii < be) {  // the CTA's row of the block: L^{-1} of it
                const double q = rsqrt_newton(pivots.piv[ii]);
                for (int t = lane; t <= i; t += 32) Ai[t] = P0[(size_t)t * B + ii] * q;
                continue;
            }
            double gr[B];
#pragma unroll
            for (int c = 0; c < B; ++c) gr[c] = -gs[li * B + c];
            for (int j = lane; j <= i; j += 32) {
                const double* Pj = P0 + (size_t)j * B;
                double v = j >= kb && j < kb + be ? 0.0 : Ai[j];
#pragma unroll
                for (int c = 0; c < B; ++c) v = fma(gr[c], Pj[c], v);
                Ai[j] = v;
            }
        }
        __syncthreads();
        if (kb + B < n) {
            push(kb + B);
            cluster.sync();
        }
    }
    if (s_fail) {  // the same everywhere
        if (tid == 0 && rank == 0) atomicOr(a.err, SCOOT_DEVERR_VALUE);
    } else {
        if (n % C == rank) {  // row n: minus alpha
            const double* Ar = A + local_row_off(n / C, rank);
            float* alpha = reinterpret_cast<float*>(a.blob + a.off_alpha) + (int64_t)m * n;
            for (int c = tid; c < n; c += kClusterThreads) alpha[c] = (float)-Ar[c];
        }
        if (rank == 0 && warp == 0) {
            float best = -INFINITY;
            for (int j = lane; j < n; j += 32) best = fmaxf(best, y[j]);
            for (int sh = 16; sh > 0; sh >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, sh));
            if (lane == 0) reinterpret_cast<float*>(a.blob + a.off_scal)[m * 4 + 2] = best;
        }
        // tiles: the owner of a row writes its entries and zeros (CTA 0 the padding rows)
        float* tiles = reinterpret_cast<float*>(a.blob + a.off_linv) + (int64_t)m * a.n_tiles * kColChunkDev * kRowBlockDev;
        const int pad = a.n_rb * kRowBlockDev;
        for (int row = rank + C * warp; row < pad; row += C * nwarps) {
            const int rb = row / kRowBlockDev, ii = row % kRowBlockDev;
            const double* Ar = A + (row < n ? local_row_off(row / C, rank) : 0);
            for (int c = lane; c < (rb + 1) * kRowBlockDev; c += 32)
                tiles[((size_t)(rb * (rb + 1) + c / kColChunkDev) * kColChunkDev + c % kColChunkDev) * kRowBlockDev + ii] =
                    row < n && c <= row ? (float)Ar[c] : 0.0f;
        }
    }
    cluster.sync();  // no CTA leaves while another may still write to it
}

constexpr int kMleMaxP = SCOOT_MAX_DIM + 2;  // ln l_1 .. ln l_d, ln s_f^2, ln tau^2
constexpr int kMleNoScratchN = 128;           // no scratch up to this n: the matrices fit shared memory
constexpr int kMleThreads = 512;

struct MleArgs {
    int32_t n, d, M, P, kernel, S, steps;
    int64_t tri;
    uint32_t free_mask;                      // bit p: parameter p is fitted
    uint32_t cat_mask;                       // bit c: parameter c is categorical
    double lr;
    double lo[kMleMaxP], hi[kMleMaxP];
    const double* U;                         // [n][d] features (unscaled, unwarped)
    const float* y;                          // [M][n]
    const double* theta0;                    // [S][M][P]
    double* theta;                           // [S][M][P]
    double* lml;                             // [S][M]
    double* grad;                            // [S][M][P] or nullptr
    double* scratch;                         // [S M][2][tri] when n > kMleNoScratchN (else in shared memory)
};

// Features of the observations, once per call: one thread per (j, c).
__global__ void __launch_bounds__(kFeatThreads) mle_feat_kernel(const __grid_constant__ GpPrepArgs a) {
    const int t = blockIdx.x * kFeatThreads + threadIdx.x;
    const int j = t / a.d, c = t - j * a.d;
    if (j >= a.n) return;
    const uint32_t w = a.obs[(int64_t)c * a.ld_obs + j];
    double u;
    bool bad = false;
    if (a.kind[c] == SCOOT_CATEGORICAL) {
        u = (double)(int32_t)w;
    } else {
        const double v = a.kind[c] == SCOOT_CONTINUOUS ? (double)__uint_as_float(w) : (double)(int32_t)w;
        bad = !isfinite(v) || (a.kind[c] == SCOOT_INT_LOG && !(v > 0.0));
        if (a.kind[c] == SCOOT_INT_LOG) u = (log(v) - a.lo[c]) / a.span[c];
        else u = a.span[c] > 0.0 ? (v - a.lo[c]) / a.span[c] : 0.0;
    }
    a.U[(int64_t)j * a.d + c] = u;
    if (c == 0)
        for (int m = 0; m < a.M; ++m) bad |= !isfinite(a.y[(int64_t)m * a.n + j]);
    if (bad) atomicOr(a.err, SCOOT_DEVERR_VALUE);
}

// k(r) / s_f^2 and its derivative in r^2 for r^2 = r2.
__device__ __forceinline__ void matern_slope(double r2, int kernel, double* k, double* dk) {
    const double r = sqrt(r2);
    if (kernel == SCOOT_MATERN32) {
        const double a = 1.7320508075688772 * r, e = exp(-a);
        *k = (1.0 + a) * e;
        *dk = -1.5 * e;
    } else {
        const double a = 2.23606797749979 * r, e = exp(-a);
        *k = fma(a, fma(a, 1.0 / 3.0, 1.0), 1.0) * e;
        *dk = -(5.0 / 6.0) * (1.0 + a) * e;
    }
}

// (For more observations than gp_mle_cluster_kernel holds, and for many fits of few.)
// One block per (start s, objective m): `steps` projected Adam steps on the
// log marginal likelihood (beta1 0.9, beta2 0.999, eps 1e-8, step size
// lr (1 - t / steps)), then the likelihood and gradient at the result.  Each
// evaluation: K + tau^2 I from the features, the factorisation with L^{-1},
// alpha = K^{-1} y, K^{-1} = L^{-T} L^{-1} (into A), and
// d lml / d theta_p = sum_{i >= j} w_ij (alpha_i alpha_j - K^{-1}_ij) dK_ij / dtheta_p
// with w = 1 off the diagonal and 1/2 on it.
__global__ void __launch_bounds__(kMleThreads) gp_mle_kernel(const __grid_constant__ MleArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = a.n, d = a.d, P = a.P;
    const int sm = blockIdx.x, m = sm % a.M;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kMleThreads / 32;
    double* rinv = reinterpret_cast<double*>(smem_raw);  // [n]
    double* rinv2 = rinv + n;                            // [n]
    double* yv = rinv2 + n;                              // [n]
    double* z = yv + n;                                  // [n] L^{-1} y
    double* al = z + n;                                  // [n] alpha
    double* col = al + n;                                // [2][n]
    double* U = col + 2 * n;                             // [d][n]: feature c of observation j at c n + j
    double* A = a.scratch ? a.scratch + (size_t)sm * 2 * a.tri : U + (size_t)n * d;
    double* W = A + a.tri;
    __shared__ double th[kMleMaxP], m1[kMleMaxP], m2[kMleMaxP], g[kMleMaxP];
    __shared__ double il2[SCOOT_MAX_DIM];  // 1 / l_c^2
    __shared__ double s_sf2, s_tau2;
    __shared__ double red[kMleThreads / 32][kMleMaxP + 1];
    __shared__ double s_total;  // y^T alpha + log det K
    __shared__ int s_fail;
    for (int i = tid; i < n; i += kMleThreads) yv[i] = (double)a.y[(int64_t)m * n + i];
    for (int t = tid; t < n * d; t += kMleThreads) {  // transposed, so that lanes on consecutive
        const int j = t / d, c = t - j * d;           // observations read consecutive words
        U[c * n + j] = a.U[t];
    }
    if (tid < P) {
        th[tid] = a.theta0[(int64_t)sm * P + tid];
        m1[tid] = 0.0;
        m2[tid] = 0.0;
    }
    if (tid == 0) s_fail = 0;
    double lml = 0.0;
    for (int it = 0; it <= a.steps; ++it) {
        __syncthreads();
        if (tid < d) il2[tid] = exp(-2.0 * th[tid]);
        if (tid == 0) {
            s_sf2 = exp(th[d]);
            s_tau2 = exp(th[d + 1]);
        }
        __syncthreads();
        const double sf2 = s_sf2, tau2 = s_tau2;
        // K + tau^2 I
        for (int64_t t = tid; t < a.tri; t += kMleThreads) {
            int i = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
            while ((int64_t)i * (i + 1) / 2 > t) --i;
            while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
            const int k = (int)(t - (int64_t)i * (i + 1) / 2);
            double r2 = 0.0;
            for (int c = 0; c < d; ++c) {
                const double df = U[c * n + i] - U[c * n + k];
                r2 += ((a.cat_mask >> c) & 1u) ? (df != 0.0 ? il2[c] : 0.0) : df * df * il2[c];
            }
            double kv, dk;
            matern_slope(r2, a.kernel, &kv, &dk);
            A[t] = sf2 * kv + (i == k ? tau2 : 0.0);
        }
        if (!eliminate(A, W, col, rinv, rinv2, n)) {
            if (tid == 0) s_fail = 1;
            __syncthreads();
            break;
        }
        // z = L^{-1} y (a warp per row), then alpha = L^{-T} z (a thread per column)
        for (int i = warp; i < n; i += nwarps) {
            const double* Wi = W + tri_idx(i, 0);
            double t = 0.0;
            for (int c = lane; c <= i; c += 32) t += Wi[c] * yv[c];
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) z[i] = t * rinv[i];
        }
        __syncthreads();
        for (int c = tid; c < n; c += kMleThreads) {
            double t = 0.0;
            for (int i = c; i < n; ++i) t += W[tri_idx(i, c)] * rinv[i] * z[i];
            al[c] = t;
        }
        // K^{-1} into A: (i, j <= i) = sum_{k >= i} L^{-1}_ki L^{-1}_kj
        for (int64_t t = tid; t < a.tri; t += kMleThreads) {
            int i = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
            while ((int64_t)i * (i + 1) / 2 > t) --i;
            while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
            const int j = (int)(t - (int64_t)i * (i + 1) / 2);
            double v = 0.0;
            for (int k = i; k < n; ++k) v += W[tri_idx(k, i)] * W[tri_idx(k, j)] * rinv2[k];
            A[t] = v;
        }
        __syncthreads();
        // gradient terms and the likelihood's two sums, per thread
        double acc[kMleMaxP + 1];
#pragma unroll
        for (int p = 0; p <= kMleMaxP; ++p) acc[p] = 0.0;
        for (int64_t t = tid; t < a.tri; t += kMleThreads) {
            int i = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
            while ((int64_t)i * (i + 1) / 2 > t) --i;
            while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
            const int k = (int)(t - (int64_t)i * (i + 1) / 2);
            const double w = (al[i] * al[k] - A[t]) * (i == k ? 0.5 : 1.0);
            if (i == k) {
                acc[kMleMaxP - 1] += w * tau2;
                acc[kMleMaxP - 2] += w * sf2;  // k(0) = 1
                continue;
            }
            double r2 = 0.0;
            for (int c = 0; c < d; ++c) {
                const double df = U[c * n + i] - U[c * n + k];
                r2 += ((a.cat_mask >> c) & 1u) ? (df != 0.0 ? il2[c] : 0.0) : df * df * il2[c];
            }
            double kv, dk;
            matern_slope(r2, a.kernel, &kv, &dk);
            const double f = -2.0 * sf2 * dk * w;
#pragma unroll
            for (int c = 0; c < SCOOT_MAX_DIM; ++c) {  // the feature's term of r^2 again (unrolled:
                if (c < d) {                           // acc stays in registers)
                    const double df = U[c * n + i] - U[c * n + k];
                    acc[c] += f * (((a.cat_mask >> c) & 1u) ? (df != 0.0 ? il2[c] : 0.0) : df * df * il2[c]);
                }
            }
            acc[kMleMaxP - 2] += w * sf2 * kv;
        }
        for (int i = tid; i < n; i += kMleThreads) acc[kMleMaxP] += yv[i] * al[i] - 2.0 * log(rinv[i]);
        // acc: lengthscales in 0 .. d-1, s_f^2 and tau^2 at kMleMaxP - 2 and - 1, and
        // y^T alpha + log det K at kMleMaxP; block reduction of the sums
#pragma unroll
        for (int p = 0; p <= kMleMaxP; ++p) {
            double v = acc[p];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) red[warp][p] = v;
        }
        __syncthreads();
        if (tid <= kMleMaxP) {
            double v = 0.0;
            for (int w2 = 0; w2 < nwarps; ++w2) v += red[w2][tid];
            if (tid < d) g[tid] = v;
            else if (tid == kMleMaxP - 2) g[d] = v;
            else if (tid == kMleMaxP - 1) g[d + 1] = v;
            else if (tid == kMleMaxP) s_total = v;
        }
        __syncthreads();
        lml = -0.5 * s_total - 0.5 * n * 1.8378770664093453;  // log(2 pi)
        if (it == a.steps) break;
        if (tid == 0) {  // projected Adam step on the free parameters
            const double step = a.lr * (1.0 - (double)it / a.steps);
            const double c1 = 1.0 - pow(0.9, it + 1), c2 = 1.0 - pow(0.999, it + 1);
            for (int p = 0; p < P; ++p) {
                if (!((a.free_mask >> p) & 1u)) continue;
                const double gp = g[p];
                m1[p] = 0.9 * m1[p] + 0.1 * gp;
                m2[p] = 0.999 * m2[p] + 0.001 * gp * gp;
                const double upd = step * (m1[p] / c1) / (sqrt(m2[p] / c2) + 1e-8);
                th[p] = fmin(fmax(th[p] + upd, a.lo[p]), a.hi[p]);
            }
        }
    }
    if (tid < P) {
        a.theta[(int64_t)sm * P + tid] = th[tid];
        if (a.grad) a.grad[(int64_t)sm * P + tid] = s_fail ? 0.0 : g[tid];
    }
    if (tid == 0) a.lml[sm] = s_fail ? -INFINITY : lml;
}

// gp_mle_kernel's fit by a cluster of eight CTAs per (start, objective).
//
// One block per fit leaves most SMs idle at the tuning loop's 8 starts, and fp64
// runs at two lanes per clock per SM: an evaluation at n = 128 took 1.2 ms on one
// SM.  Here CTA r owns rows i = r (mod 8) of the symmetric matrix, and K^{-1},
// alpha and the determinant come from one elimination: the matrix is
// augmented by row n, which holds y^T and 0, and its first n pivots are swept in
// place: before pivot t entry (i, t) is A_it, after it W_it, the elimination of the
// identity, and after pivot i too what -K^{-1}_it has gathered, -sum_p W_pi W_pt / A_pp:
// with the panel P and the multipliers g of eliminate_panel every entry takes
//   A_ij -= g_i . P_j
// (from 0 where i or j is a pivot of the block), which leaves -K^{-1}, -alpha^T in
// row n and -y^T K^{-1} y at its end (n^3 / 2 multiply-adds, as many as a factor, its
// inverse and their product; the pivots are the Cholesky factor's squared).  Pivots
// go in blocks of eight,
// so that a block costs one exchange: every CTA pushes its part of the next
// block's columns into all eight CTAs' shared memory, and each eliminates the
// panel for itself.  The covariances and their slopes are kept for the
// gradient where two CTAs still fit an SM (a GPU has room for 15 clusters of one
// CTA per SM, a sixteenth would wait for them: the tuning loop has 8 starts of
// two objectives).  An fp64 instruction holds a scheduler's unit for 64 cycles, so
// what counts is their number: features are scaled once per evaluation,
// categories and pivots compared as integers.
// Measured (60 steps, 8 starts x 2 objectives, 4 or 8 parameters, gp_mle_kernel against
// this): n = 64 19.7 ms against 5.9, n = 128 72.8 against 16.5, n = 256 471 against 78;
// with one CTA per SM, n = 317 826 against 115 (covariances kept), n = 400 1608 against
// 232, n = 500 2977 against 404.  64 fits at n = 128 75.6 against 32.2, 128 fits 75.6
// against 63.4; 32 fits at n = 500 3051 against 606.  What does not fit (from 443
// observations of 16 parameters, 519 of 2) stays with gp_mle_kernel.  Keeping the squared
// differences as well cost the second CTA per SM and was slower (25 ms at n = 128).
// The gradient's error against 64 bits is that of gp_mle_kernel (1.1e-13 at n = 128; a
// sweep that multiplied by inverted blocks had 4.8e-13).
constexpr int kMleB = kClusterB;
constexpr int kMleClThreads = kClusterThreads;

constexpr size_t kMleClTwo = 108 * 1024;  // shared memory of which two CTAs fit an SM

struct MleClSizes {
    int64_t own;                  // entries of the CTA with the most
    size_t bytes, keep_bytes;     // without and of the kept covariances
};

inline MleClSizes mle_cl_sizes(int n, int d) {
    MleClSizes z;
    z.own = cluster_own(n);
    const size_t rows = (size_t)(n + 1 + kClusterCTAs - 1) / kClusterCTAs;
    z.bytes = ((size_t)2 * (n + 1) * kMleB + (size_t)n * d + (size_t)z.own + 2 * (size_t)(n + 1) + rows * kMleB) * sizeof(double);
    z.keep_bytes = 2 * (size_t)z.own * sizeof(double);
    return z;
}

__global__ void __cluster_dims__(kClusterCTAs, 1, 1) __launch_bounds__(kMleClThreads, 2)
gp_mle_cluster_kernel(const __grid_constant__ MleArgs a, int64_t own, int keep) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int C = kClusterCTAs, B = kMleB;
    const int n = a.n, d = a.d, P = a.P;
    const int rank = (int)cluster.block_rank(), sm = blockIdx.x / C, m = sm % a.M;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nwarps = kMleClThreads / 32;
    double* panel = reinterpret_cast<double*>(smem_raw);  // [2][n + 1][B] the pivot block's columns
    double* U = panel + 2 * (size_t)(n + 1) * B;          // [d][n] features, ordinal ones over their lengthscale
    double* A = U + (size_t)n * d;                        // owned rows, packed
    double* al = A + own;                                 // [n + 1] alpha, then y^T K^{-1} y
    double* piv = al + n + 1;                             // [n + 1]
    double* gs = piv + n + 1;                             // [owned rows][B] a row's multipliers in an elimination step
    double* kvs = gs + (size_t)((n + 1 + C - 1) / C) * B;  // if kept: k / s_f^2 of the owned rows
    double* dks = kvs + own;                              // and its slope in r^2
    __shared__ double th[kMleMaxP], g[kMleMaxP], am[2][kMleMaxP], il2[SCOOT_MAX_DIM], il[SCOOT_MAX_DIM];  // am: Adam's moments
    __shared__ double s_sf2, s_tau2, s_c1, s_c2, s_total;
    __shared__ double part[C][kMleMaxP + 1], red[nwarps][kMleMaxP + 1];
    __shared__ PanelPivots pivots;
    __shared__ int s_fail;
    const int nl = (n + 1 - rank + C - 1) / C;  // owned rows, row n among them
    if (tid < P) {
        th[tid] = a.theta0[(int64_t)sm * P + tid];
        am[0][tid] = am[1][tid] = 0.0;
    }
    if (tid == 0) s_fail = 0;
    // Term c of r^2 between rows i and k.
    auto term = [&](int c, int i, int k) {
        const double x = U[c * n + i], y = U[c * n + k];
        if ((a.cat_mask >> c) & 1u) return __double_as_longlong(x) != __double_as_longlong(y) ? il2[c] : 0.0;
        return (x - y) * (x - y);
    };
    auto distance2 = [&](int i, int k) {
        double r2 = 0.0;
        for (int c = 0; c < d; ++c) {
            const double x = U[c * n + i], y = U[c * n + k];
            if ((a.cat_mask >> c) & 1u) {
                if (__double_as_longlong(x) != __double_as_longlong(y)) r2 += il2[c];
            } else {
                r2 = fma(x - y, x - y, r2);
            }
        }
        return r2;
    };
    // The columns kb .. kb + 7 of the symmetric matrix into every CTA's panel,
    // [j][c] = A_j,kb+c (0 beyond the last pivot): an owned row j >= kb + c gives
    // its entries, the block's own rows those of the rows before them.
    auto push = [&](int kb) {
        const size_t off = (size_t)((kb / B) & 1) * (n + 1) * B;
        double* peer[C];  // every CTA's panel
#pragma unroll
        for (int r = 0; r < C; ++r) peer[r] = cluster.map_shared_rank(panel, r) + off;
        for (int e = tid; e < nl * B; e += kMleClThreads) {
            const int li = e / B, c = e - li * B, i = rank + C * li, kc = kb + c;
            if (kc < n && kc > i) continue;
            const double v = kc < n ? A[local_row_off(li, rank) + kc] : 0.0;
#pragma unroll
            for (int r = 0; r < C; ++r) peer[r][i * B + c] = v;
        }
        const int row = kb + rank;
        if (row < n) {
            const double* Ar = A + local_row_off(row / C, rank);
            for (int j = tid; j < row; j += kMleClThreads) {
                const double v = Ar[j];
#pragma unroll
                for (int r = 0; r < C; ++r) peer[r][j * B + rank] = v;
            }
        }
    };
    cluster.sync();  // every CTA has started: its shared memory may be written
    double lml = 0.0;
    for (int it = 0; it <= a.steps; ++it) {
        __syncthreads();
        if (tid < d) {
            il[tid] = exp(-th[tid]);
            il2[tid] = il[tid] * il[tid];
        } else if (tid == 32) s_sf2 = exp(th[d]);
        else if (tid == 64) s_tau2 = exp(th[d + 1]);
        else if (tid == 96) s_c1 = 1.0 - pow(0.9, it + 1);
        else if (tid == 128) s_c2 = 1.0 - pow(0.999, it + 1);
        __syncthreads();
        const double sf2 = s_sf2, tau2 = s_tau2;
        for (int t = tid; t < n * d; t += kMleClThreads) {
            const int c = t % d;
            const double u = a.U[t];
            U[c * n + t / d] = ((a.cat_mask >> c) & 1u) ? u : u * il[c];
        }
        __syncthreads();
        for (int li = warp; li < nl; li += nwarps) {
            const int i = rank + C * li;
            const int64_t o = local_row_off(li, rank);
            if (i == n) {
                for (int k = lane; k <= n; k += 32) A[o + k] = k < n ? (double)a.y[(int64_t)m * n + k] : 0.0;
                continue;
            }
            for (int k = lane; k <= i; k += 32) {
                double kv, dk;
                matern_slope(distance2(i, k), a.kernel, &kv, &dk);
                if (keep) {
                    kvs[o + k] = kv;
                    dks[o + k] = dk;
                }
                A[o + k] = sf2 * kv + (i == k ? tau2 : 0.0);
            }
        }
        __syncthreads();
        push(0);
        cluster.sync();
        for (int kb = 0; kb < n; kb += B) {
            double* P0 = panel + (size_t)((kb / B) & 1) * (n + 1) * B;
            const int be = min(B, n - kb);
            eliminate_panel(P0, gs, pivots, &s_fail, n, kb, be, rank, true);
            __syncthreads();
            if (s_fail) break;  // the same in every CTA: each has eliminated the same panel
            if (tid < be) piv[kb + tid] = pivots.piv[tid];
            for (int li = warp; li < nl; li += nwarps) {
                const int i = rank + C * li;
                const bool pivot = i >= kb && i < kb + be;
                double* Ai = A + local_row_off(li, rank);
                double gr[B];
#pragma unroll
                for (int c = 0; c < B; ++c) gr[c] = -gs[li * B + c];
                for (int j = lane; j <= i; j += 32) {
                    const double* Pj = P0 + (size_t)j * B;
                    double v = pivot || (j >= kb && j < kb + be) ? 0.0 : Ai[j];
#pragma unroll
                    for (int c = 0; c < B; ++c) v = fma(gr[c], Pj[c], v);
                    Ai[j] = v;
                }
            }
            __syncthreads();
            if (kb + B < n) {
                push(kb + B);
            } else if (n % C == rank) {  // row n: -alpha and -y^T alpha, everywhere
                const double* Ar = A + local_row_off(n / C, rank);
                for (int j = tid; j <= n; j += kMleClThreads)
                    for (int r = 0; r < C; ++r) cluster.map_shared_rank(al, r)[j] = -Ar[j];
            }
            cluster.sync();
        }
        if (s_fail) break;
        double acc[kMleMaxP + 1];
#pragma unroll
        for (int p = 0; p <= kMleMaxP; ++p) acc[p] = 0.0;
        for (int li = warp; li < nl; li += nwarps) {
            const int i = rank + C * li;
            if (i == n) continue;
            const int64_t o = local_row_off(li, rank);
            const double ai = al[i];
            for (int k = lane; k <= i; k += 32) {
                const double w = fma(ai, al[k], A[o + k]) * (i == k ? 0.5 : 1.0);  // A holds -K^{-1}
                if (i == k) {
                    acc[kMleMaxP - 1] += w * tau2;
                    acc[kMleMaxP - 2] += w * sf2;  // k(0) = 1
                    continue;
                }
                double kv, dk;
                if (keep) {
                    kv = kvs[o + k];
                    dk = dks[o + k];
                } else {
                    matern_slope(distance2(i, k), a.kernel, &kv, &dk);
                }
                const double f = -2.0 * sf2 * dk * w;
#pragma unroll
                for (int c = 0; c < SCOOT_MAX_DIM; ++c)
                    if (c < d) acc[c] = fma(f, term(c, i, k), acc[c]);
                acc[kMleMaxP - 2] = fma(w * sf2, kv, acc[kMleMaxP - 2]);
            }
        }
        if (it == a.steps && rank == 0)  // the likelihood, at the result alone
            for (int p = tid; p < n; p += kMleClThreads) acc[kMleMaxP] += log(piv[p]);
#pragma unroll
        for (int p = 0; p <= kMleMaxP; ++p) {
            if (p < d || p >= kMleMaxP - 2) {
                double v = acc[p];
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) red[warp][p] = v;
            }
        }
        __syncthreads();
        if (tid < d || (tid >= kMleMaxP - 2 && tid <= kMleMaxP)) {
            double v = 0.0;
            for (int w2 = 0; w2 < nwarps; ++w2) v += red[w2][tid];
            for (int r = 0; r < C; ++r) cluster.map_shared_rank(&part[0][0], r)[rank * (kMleMaxP + 1) + tid] = v;
        }
        cluster.sync();
        if (tid < d || (tid >= kMleMaxP - 2 && tid <= kMleMaxP)) {
            double v = 0.0;
            for (int r = 0; r < C; ++r) v += part[r][tid];
            if (tid < d) g[tid] = v;
            else if (tid == kMleMaxP) s_total = v;
            else g[tid - (kMleMaxP - 2) + d] = v;
        }
        __syncthreads();
        if (it == a.steps) {
            lml = -0.5 * (al[n] + s_total) - 0.5 * n * 1.8378770664093453;  // log(2 pi)
            break;
        }
        if (tid < P && ((a.free_mask >> tid) & 1u)) {  // projected Adam step on the free parameters
            const double step = a.lr * (1.0 - (double)it / a.steps), gp = g[tid];
            const double m1 = am[0][tid] = 0.9 * am[0][tid] + 0.1 * gp;
            const double m2 = am[1][tid] = 0.999 * am[1][tid] + 0.001 * gp * gp;
            const double upd = step * (m1 / s_c1) / (sqrt(m2 / s_c2) + 1e-8);
            th[tid] = fmin(fmax(th[tid] + upd, a.lo[tid]), a.hi[tid]);
        }
    }
    if (rank == 0) {
        if (tid < P) {
            a.theta[(int64_t)sm * P + tid] = th[tid];
            if (a.grad) a.grad[(int64_t)sm * P + tid] = s_fail ? 0.0 : g[tid];
        }
        if (tid == 0) a.lml[sm] = s_fail ? -INFINITY : lml;
    }
    cluster.sync();  // no CTA leaves while another may still write to it
}

}  // namespace

extern "C" {

scoot_status scoot_gp_device_work_bytes(const scoot_gp_layout* L, int64_t* bytes) {
    if (!L || !bytes || !scoot_gp_layout_valid(L)) return SCOOT_EINVAL;
    const int64_t n = L->n, tri = n * (n + 1) / 2;
    *bytes = 8 * (int64_t)L->n_obj * (n * L->d + tri * (n <= kOneTriangleN ? 1 : 2));
    return SCOOT_OK;
}

scoot_status scoot_gp_prepare_device(scoot_ctx* ctx, const scoot_param* h_space, const scoot_gp_layout* L,
                                     const uint32_t* obs, int64_t ld_obs, const float* y, const float* lengthscale,
                                     const float* signal_var, const float* noise_var, const float* warp, void* blob,
                                     void* work, int64_t work_bytes, void* stream) {
    scoot_status s = scoot_enter(ctx);
    if (s != SCOOT_OK) return s;
    if (!h_space || !L) return scoot_fail(ctx, SCOOT_EINVAL, "h_space or layout is NULL");
    scoot_gp_layout chk;
    if (scoot_gp_layout_init(h_space, L->n, L->d, L->n_obj, L->kernel, &chk) != SCOOT_OK ||
        std::memcmp(&chk, L, sizeof(chk)) != 0)
        return scoot_fail(ctx, SCOOT_EINVAL, "layout does not match h_space");
    if (!obs || !y || !lengthscale || !signal_var || !noise_var || !blob)
        return scoot_fail(ctx, SCOOT_EINVAL, "obs, y, lengthscale, signal_var, noise_var or blob is NULL");
    if (ld_obs < L->n) return scoot_fail(ctx, SCOOT_EINVAL, "ld_obs = %lld < n = %d", (long long)ld_obs, L->n);
    if (!scoot_aligned16(blob)) return scoot_fail(ctx, SCOOT_EINVAL, "blob is not 16-byte aligned");
    int64_t need = 0;
    scoot_gp_device_work_bytes(L, &need);
    if (!work || work_bytes < need || !scoot_aligned16(work))
        return scoot_fail(ctx, SCOOT_EINVAL, "work needs %lld bytes, 16-byte aligned", (long long)need);
    GpPrepArgs a;
    std::memset(&a, 0, sizeof(a));
    const int n = L->n, d = L->d, M = L->n_obj;
    a.n = n;
    a.d = d;
    a.M = M;
    a.kernel = L->kernel;
    a.n_ord = L->n_ord;
    a.n_pat = L->n_pat;
    a.n_rb = L->n_rb;
    a.n_tiles = L->n_tiles;
    a.tri = (int64_t)n * (n + 1) / 2;
    int f = 0;
    for (int pass = 0; pass < 2; ++pass)  // ordinal parameters first, then categorical ones
        for (int c = 0; c < d; ++c)
            if ((h_space[c].kind == SCOOT_CATEGORICAL) == (pass == 1)) a.order[f++] = c;
    int stride = 1;
    for (int g = 0; g < d; ++g) {
        const int c = a.order[g];
        const scoot_param& p = h_space[c];
        a.kind[c] = p.kind;
        a.n_choices[c] = p.n_choices;
        float fa = 0.f, fb = 0.f;
        if (p.kind == SCOOT_INT_LOG) {
            a.lo[c] = std::log((double)p.lo);
            a.span[c] = std::log((double)p.hi) - std::log((double)p.lo);
            fa = (float)a.lo[c];
            fb = (float)(1.0 / a.span[c]);
        } else if (p.kind != SCOOT_CATEGORICAL) {
            a.lo[c] = p.lo;
            a.span[c] = (double)p.hi - (double)p.lo;
            fa = p.lo;
            fb = p.hi > p.lo ? (float)(1.0 / ((double)p.hi - (double)p.lo)) : 0.0f;
        } else {
            fa = (float)p.n_choices;
            fb = (float)stride;
            stride *= p.n_choices;
        }
        a.fmap[g][0] = (float)p.kind;
        a.fmap[g][1] = fa;
        a.fmap[g][2] = fb;
        a.fmap[g][3] = (float)c;
    }
    a.obs = obs;
    a.ld_obs = ld_obs;
    a.y = y;
    a.ls = lengthscale;
    a.sf2 = signal_var;
    a.tau2 = noise_var;
    a.warp = warp;
    a.blob = static_cast<char*>(blob);
    a.off_fmap = L->off_fmap;
    a.off_xs = L->off_xs;
    a.off_ils = L->off_ils;
    a.off_alpha = L->off_alpha;
    a.off_linv = L->off_linv;
    a.off_scal = L->off_scal;
    a.off_cat = L->off_cat;
    a.off_warp = L->off_warp;
    const size_t u_bytes = (size_t)M * n * d * sizeof(double);
    const size_t k_bytes = (size_t)M * a.tri * sizeof(double);
    char* ws = static_cast<char*>(work);
    a.U = reinterpret_cast<double*>(ws);
    a.K = reinterpret_cast<double*>(ws + u_bytes);
    a.W = n <= kOneTriangleN ? nullptr : reinterpret_cast<double*>(ws + u_bytes + k_bytes);
    a.err = ctx->d_err;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    gp_feat_kernel<<<dim3((n * d + kFeatThreads - 1) / kFeatThreads, M), kFeatThreads, 0, st>>>(a);
    SCOOT_LAUNCHED(ctx);
    if (L->n_ord < d) {
        const int64_t cells = (int64_t)n * L->n_pat;
        gp_cat_kernel<<<dim3((unsigned)((cells + kKmatThreads - 1) / kKmatThreads), M), kKmatThreads, 0, st>>>(a);
        SCOOT_LAUNCHED(ctx);
    } else {
        // no categorical parameter: one pattern, zero distance
        SCOOT_CUDA(ctx, cudaMemsetAsync(static_cast<char*>(blob) + L->off_cat, 0, (size_t)M * n * sizeof(float), st));
    }
    gp_kmat_kernel<<<dim3((unsigned)((a.tri + kKmatThreads - 1) / kKmatThreads), M), kKmatThreads, 0, st>>>(a);
    SCOOT_LAUNCHED(ctx);
    int optin = 0;
    SCOOT_CUDA(ctx, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    const size_t csmem = chol_cluster_bytes(n);
    if (csmem + 4096 <= (size_t)optin) {
        SCOOT_CUDA(ctx, cudaFuncSetAttribute(gp_chol_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)csmem));
        gp_chol_cluster_kernel<<<M * kClusterCTAs, kClusterThreads, csmem, st>>>(a, cluster_own(n));
        SCOOT_LAUNCHED(ctx);
        return SCOOT_OK;
    }
    if (!a.W) return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "shared memory of %d bytes is too small", optin);
    const size_t smem = (size_t)5 * n * sizeof(double);
    SCOOT_CUDA(ctx, cudaFuncSetAttribute(gp_chol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    gp_chol_kernel<<<M, kCholThreads, smem, st>>>(a);
    SCOOT_LAUNCHED(ctx);
    return SCOOT_OK;
}

scoot_status scoot_gp_mle_work_bytes(int32_t n, int32_t d, int32_t n_obj, int32_t n_starts, int64_t* bytes) {
    if (!bytes || n < 1 || d < 1 || n_obj < 1 || n_starts < 1) return SCOOT_EINVAL;
    const int64_t tri = (int64_t)n * (n + 1) / 2;
    int64_t b = ((int64_t)n * d * 8 + 255) / 256 * 256;
    if (n > kMleNoScratchN) b += (int64_t)n_starts * n_obj * 2 * tri * 8;
    *bytes = b;
    return SCOOT_OK;
}

scoot_status scoot_gp_mle(scoot_ctx* ctx, const scoot_param* h_space, int32_t d, const uint32_t* obs, int64_t ld_obs,
                          int32_t n, const float* y, int32_t n_obj, int32_t kernel, const double* theta0,
                          int32_t n_starts, const double* h_lo, const double* h_hi, uint32_t free_mask, int32_t steps,
                          double lr, double* theta, double* lml, double* grad, void* work, int64_t work_bytes,
                          void* stream) {
    scoot_status s = scoot_enter(ctx);
    if (s != SCOOT_OK) return s;
    if (!h_space || !h_lo || !h_hi) return scoot_fail(ctx, SCOOT_EINVAL, "h_space, h_lo or h_hi is NULL");
    if (d < 1 || d > SCOOT_MAX_DIM) return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "d = %d outside 1..%d", d, SCOOT_MAX_DIM);
    if (n < 1 || n > SCOOT_MAX_OBS) return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "n = %d outside 1..%d", n, SCOOT_MAX_OBS);
    if (n_obj < 1 || n_obj > SCOOT_MAX_OBJ) return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "n_obj = %d", n_obj);
    if (kernel != SCOOT_MATERN52 && kernel != SCOOT_MATERN32) return scoot_fail(ctx, SCOOT_EINVAL, "kernel %d", kernel);
    if (n_starts < 1 || (int64_t)n_starts * n_obj > 65535)
        return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "n_starts = %d", n_starts);
    if (steps < 0 || !(lr >= 0.0) || !std::isfinite(lr)) return scoot_fail(ctx, SCOOT_EINVAL, "steps or lr");
    if (ld_obs < n) return scoot_fail(ctx, SCOOT_EINVAL, "ld_obs = %lld < n", (long long)ld_obs);
    if (!obs || !y || !theta0 || !theta || !lml) return scoot_fail(ctx, SCOOT_EINVAL, "a device array is NULL");
    const int P = d + 2;
    MleArgs a;
    std::memset(&a, 0, sizeof(a));
    for (int p = 0; p < P; ++p) {
        if (!std::isfinite(h_lo[p]) || !std::isfinite(h_hi[p]) || h_lo[p] > h_hi[p])
            return scoot_fail(ctx, SCOOT_EINVAL, "bounds of parameter %d", p);
        a.lo[p] = h_lo[p];
        a.hi[p] = h_hi[p];
    }
    GpPrepArgs f;
    std::memset(&f, 0, sizeof(f));
    for (int c = 0; c < d; ++c) {
        const scoot_param& p = h_space[c];
        f.kind[c] = p.kind;
        if (p.kind == SCOOT_CATEGORICAL) {
            if (p.n_choices < 1) return scoot_fail(ctx, SCOOT_EINVAL, "parameter %d: n_choices", c);
            a.cat_mask |= 1u << c;
        } else if (p.kind == SCOOT_INT_LOG) {
            if (!(p.lo > 0.0f) || !(p.hi > p.lo)) return scoot_fail(ctx, SCOOT_EINVAL, "parameter %d: log range", c);
            f.lo[c] = std::log((double)p.lo);
            f.span[c] = std::log((double)p.hi) - std::log((double)p.lo);
        } else if (p.kind == SCOOT_INT_UNIFORM || p.kind == SCOOT_CONTINUOUS) {
            f.lo[c] = p.lo;
            f.span[c] = (double)p.hi - (double)p.lo;
        } else {
            return scoot_fail(ctx, SCOOT_EINVAL, "parameter %d: kind %d", c, p.kind);
        }
    }
    int64_t need = 0;
    scoot_gp_mle_work_bytes(n, d, n_obj, n_starts, &need);
    if (!work || work_bytes < need || !scoot_aligned16(work))
        return scoot_fail(ctx, SCOOT_EINVAL, "work needs %lld bytes, 16-byte aligned", (long long)need);
    char* ws = static_cast<char*>(work);
    f.n = n;
    f.d = d;
    f.obs = obs;
    f.ld_obs = ld_obs;
    f.U = reinterpret_cast<double*>(ws);
    f.M = n_obj;
    f.y = y;
    f.err = ctx->d_err;
    a.n = n;
    a.d = d;
    a.M = n_obj;
    a.P = P;
    a.kernel = kernel;
    a.S = n_starts;
    a.steps = steps;
    a.tri = (int64_t)n * (n + 1) / 2;
    a.free_mask = free_mask & ((1u << P) - 1u);
    a.lr = lr;
    a.U = f.U;
    a.y = y;
    a.theta0 = theta0;
    a.theta = theta;
    a.lml = lml;
    a.grad = grad;
    a.scratch = n > kMleNoScratchN ? reinterpret_cast<double*>(ws + ((int64_t)n * d * 8 + 255) / 256 * 256) : nullptr;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    mle_feat_kernel<<<(n * d + kFeatThreads - 1) / kFeatThreads, kFeatThreads, 0, st>>>(f);
    SCOOT_LAUNCHED(ctx);
    int optin = 0;
    SCOOT_CUDA(ctx, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device));
    const MleClSizes cl = mle_cl_sizes(n, d);
    // Eight CTAs per fit share its pivot rows' work but each runs their chain, so where
    // the fits alone fill the SMs, a block each, a wave of blocks ends before the clusters
    // do: those get 80 + 0.6 n fits done in its time on 152 SMs.  (60 steps, n = 16: 64 fits
    // 3.7 ms against 4.2 by blocks, 128 7.2 against 4.2; n = 32: 128 fits 10.2 against 7.4; n =
    // 64: 64 fits 10.6 against 18.7, 128 20.9 against 18.7, 512 77.8 against 74.6; n = 128: 512
    // fits 229 against 278.)
    int sms = 0;
    SCOOT_CUDA(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
    const int fits = n_starts * n_obj, waves = (fits + sms - 1) / sms;
    const bool blocks = n <= kMleNoScratchN && fits * 152.0 > (double)waves * sms * (80.0 + 0.6 * n);
    if (!blocks && cl.bytes + 8192 <= (size_t)optin) {
        const int keep = cl.bytes + cl.keep_bytes <= kMleClTwo || (cl.bytes > kMleClTwo && cl.bytes + cl.keep_bytes + 8192 <= (size_t)optin);
        const size_t bytes = cl.bytes + (keep ? cl.keep_bytes : 0);
        SCOOT_CUDA(ctx, cudaFuncSetAttribute(gp_mle_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
        gp_mle_cluster_kernel<<<n_starts * n_obj * kClusterCTAs, kMleClThreads, bytes, st>>>(a, cl.own, keep);
        SCOOT_LAUNCHED(ctx);
        return SCOOT_OK;
    }
    const size_t smem = (size_t)(7 * n + (size_t)n * d) * sizeof(double) + (a.scratch ? 0 : (size_t)2 * a.tri * sizeof(double));
    SCOOT_CUDA(ctx, cudaFuncSetAttribute(gp_mle_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    gp_mle_kernel<<<n_starts * n_obj, kMleThreads, smem, st>>>(a);
    SCOOT_LAUNCHED(ctx);
    return SCOOT_OK;
}

static int64_t slot256(int64_t b) { return (b + 255) / 256 * 256; }

scoot_status scoot_gp_device_buffer_layout(const scoot_gp_layout* L, int32_t warped, int64_t* upload_bytes,
                                           int64_t* blob_off, int64_t* work_off, int64_t* total_bytes) {
    if (!L || !upload_bytes || !blob_off || !work_off || !total_bytes || !scoot_gp_layout_valid(L)) return SCOOT_EINVAL;
    const int64_t n = L->n, d = L->d, M = L->n_obj;
    int64_t off = slot256(4 * d * n) + slot256(4 * M * n) + slot256(4 * M * d) + 2 * slot256(4 * M);
    if (warped) off += slot256(8 * M * d);
    *upload_bytes = off;
    *blob_off = off;
    off += slot256(L->bytes);
    *work_off = off;
    int64_t wb = 0;
    scoot_gp_device_work_bytes(L, &wb);
    *total_bytes = off + slot256(wb);
    return SCOOT_OK;
}

scoot_status scoot_gp_prepare_device_from_host(scoot_ctx* ctx, const scoot_param* h_space, const scoot_gp_layout* L,
                                               const uint32_t* h_x_obs, int64_t ld_obs, const float* h_y,
                                               const float* h_lengthscale, const float* h_signal_var,
                                               const float* h_noise_var, const float* h_warp, void* h_stage,
                                               void* buf, int64_t buf_bytes, void* stream) {
    scoot_status s = scoot_enter(ctx);
    if (s != SCOOT_OK) return s;
    int64_t up = 0, blob_off = 0, work_off = 0, total = 0;
    if (scoot_gp_device_buffer_layout(L, h_warp != nullptr, &up, &blob_off, &work_off, &total) != SCOOT_OK)
        return scoot_fail(ctx, SCOOT_EINVAL, "invalid layout");
    if (!h_space || !h_x_obs || !h_y || !h_lengthscale || !h_signal_var || !h_noise_var || !h_stage || !buf)
        return scoot_fail(ctx, SCOOT_EINVAL, "a pointer is NULL");
    if (buf_bytes < total || !scoot_aligned16(buf))
        return scoot_fail(ctx, SCOOT_EINVAL, "buf needs %lld bytes, 16-byte aligned", (long long)total);
    if (ld_obs < L->n) return scoot_fail(ctx, SCOOT_EINVAL, "ld_obs < n");
    const int64_t n = L->n, d = L->d, M = L->n_obj;
    char* hs = static_cast<char*>(h_stage);
    int64_t off = 0, o_obs, o_y, o_ls, o_sf, o_tau, o_warp = -1;
    o_obs = off;
    for (int64_t c = 0; c < d; ++c) std::memcpy(hs + off + 4 * c * n, h_x_obs + c * ld_obs, 4 * n);
    off += slot256(4 * d * n);
    o_y = off;
    std::memcpy(hs + off, h_y, 4 * M * n);
    off += slot256(4 * M * n);
    o_ls = off;
    std::memcpy(hs + off, h_lengthscale, 4 * M * d);
    off += slot256(4 * M * d);
    o_sf = off;
    std::memcpy(hs + off, h_signal_var, 4 * M);
    off += slot256(4 * M);
    o_tau = off;
    std::memcpy(hs + off, h_noise_var, 4 * M);
    off += slot256(4 * M);
    if (h_warp) {
        o_warp = off;
        std::memcpy(hs + off, h_warp, 8 * M * d);
        off += slot256(8 * M * d);
    }
    char* db = static_cast<char*>(buf);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    SCOOT_CUDA(ctx, cudaMemcpyAsync(db, hs, (size_t)up, cudaMemcpyHostToDevice, st));
    return scoot_gp_prepare_device(ctx, h_space, L, reinterpret_cast<const uint32_t*>(db + o_obs), n,
                                   reinterpret_cast<const float*>(db + o_y), reinterpret_cast<const float*>(db + o_ls),
                                   reinterpret_cast<const float*>(db + o_sf), reinterpret_cast<const float*>(db + o_tau),
                                   o_warp >= 0 ? reinterpret_cast<const float*>(db + o_warp) : nullptr, db + blob_off,
                                   db + work_off, total - work_off, stream);
}

}  // extern "C"
