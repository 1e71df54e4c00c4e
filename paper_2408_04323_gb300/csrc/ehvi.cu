// Monte-Carlo EHVI (Eq. 7) of candidates whose posterior moments are already
// in memory by list position: the second half of scoot_score_ehvi where the
// first is the tensor-core posterior.
//
// Two kernels.  ehvi_dense sums every box for every sample (four threads per
// candidate, boxes read as broadcasts).  ehvi_walk (three objectives) visits
// only the boxes that a sample reaches: with the boxes of scoot_boxes_build
// the reached ones are, per strip of the first objective below the sample,
// a run of columns of the second that ends where the floor rises above the
// sample, so a sample looks up its strip and its column and walks down.  On
// fronts of 40 to 60 points (300 to 600 boxes) a sample reaches 8 boxes on
// average, three samples in four none at all.
#include <algorithm>
#include <cstring>

#include "device_common.cuh"
#include "internal.h"

namespace {

using namespace scoot_dev;

constexpr int kTC = 32;            // candidates per block of ehvi_dense
constexpr int kDenseThreads = 128;
constexpr int kQ = kDenseThreads / kTC;

constexpr int kPlanThreads = 512;
constexpr int kWalkThreads = 256;
constexpr int kWalkWarps = kWalkThreads / 32;
constexpr int kWalkBatch = 8;      // candidates per warp at a time (at most)
constexpr int kWalkIds = 1024;     // samples per warp at a time (at most)
constexpr int kLut = 256;          // cells of the lookup from a coordinate to its rank
constexpr int kWalkBoxMin = 96;    // fewer boxes: ehvi_dense
constexpr int kWalkBoxMax = 2048;
// Most strips, columns and strip-column pairs that a plan of B boxes may have
// (fronts of 23 to 76 points: B / 6 to B / 11 strips, 4.5 B to 7 B pairs);
// the shared memory of ehvi_walk is sized for them.
__host__ __device__ inline int walk_strips(int B) { return B / 3; }
__host__ __device__ inline int walk_cols(int B) { return B / 2; }
__host__ __device__ inline int walk_pairs(int B) { return 8 * B; }
constexpr int kRefetch = 8;        // idle lanes that make a warp hand out new samples
constexpr int kRun = 2;            // boxes a lane takes before the warp looks for finished strips

// The walk's tables, in the context workspace: this header, then
//   float2 box[n_boxes + n_strip]   (lo1, floor) per strip, each strip after a
//                                   sentinel of floor +inf (8 bytes a step: the
//                                   gathers from shared memory are the bound,
//                                   and a column's upper edge is the lower edge
//                                   of the one before it on the way down)
//   float axis0[n_strip + 1]        strips' lower edges, then +inf
//   float axis1[n_col + 1]          columns' lower edges, then +inf
//   uint16 lut[2][kLut]             a lower bound of the rank per cell
//   uint16 start[n_strip * n_col]   byte offset of strip i's box at column k
struct WalkPlan {
    int32_t ok, n_strip, n_col;
    uint32_t ticket;                // candidates handed out to the walk's warps
    float base[2], scale[2];
};

struct WalkSizes {
    size_t box, axis0, axis1, lut, start, bytes;
};

__host__ __device__ inline WalkSizes walk_sizes(int n_boxes, int n_strip, int n_col) {
    WalkSizes w;
    w.box = 64;
    w.axis0 = w.box + (size_t)(n_boxes + n_strip) * 8;
    w.axis1 = w.axis0 + (size_t)(n_strip + 1) * 4;
    w.lut = w.axis1 + (size_t)(n_col + 1) * 4;
    w.start = w.lut + (size_t)2 * kLut * 2;
    w.bytes = (w.start + (size_t)n_strip * n_col * 2 + 15) / 16 * 16;
    return w;
}

// Cell of coordinate y in a lookup table: monotone in y; NaN and values below
// the base fall into cell 0.
__device__ __forceinline__ int lut_cell(float y, float base, float scale) {
    return (int)fminf(fmaxf((y - base) * scale, 0.0f), (float)(kLut - 1));
}

// One block: whether the boxes are as scoot_boxes_build makes them for three
// objectives, and if so the walk's tables.  Checked: strips of equal (lo0,
// hi0), increasing and adjoining, the last one open; in each strip adjoining
// columns from one common lower edge to +inf, open on the last objective,
// with finite floors that never rise along the strip; and floors that never
// rise from a strip to the next at the same column.  Then the boxes with a
// lower corner below a sample are exactly those the walk visits.
__global__ void __launch_bounds__(kPlanThreads)
walk_plan(const float* __restrict__ lo, const float* __restrict__ hi, int B, char* out) {
    extern __shared__ __align__(16) float sm[];
    float* key = sm;                                              // [pow2 >= B] sorted second coordinates
    uint16_t* sid = reinterpret_cast<uint16_t*>(key + kWalkBoxMax);  // [B] strip of each box
    __shared__ int s_bad, s_tot, s_wt[kPlanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    WalkPlan* plan = reinterpret_cast<WalkPlan*>(out);
    // Exclusive prefix of a flag over the block, and the total.
    auto prefix = [&](bool f, int* tot) {
        const unsigned b = __ballot_sync(0xffffffffu, f);
        if (lane == 0) s_wt[warp] = __popc(b);
        __syncthreads();
        int off = 0, t = 0;
        for (int k = 0; k < kPlanThreads / 32; ++k) {
            off += k < warp ? s_wt[k] : 0;
            t += s_wt[k];
        }
        __syncthreads();
        *tot = t;
        return off + __popc(b & ((1u << lane) - 1u));
    };
    if (tid == 0) s_bad = 0;
    int P = 1;
    while (P < B) P *= 2;
    for (int b = tid; b < P; b += kPlanThreads) key[b] = b < B ? lo[3 * b + 1] : INFINITY;
    __syncthreads();
    // strips and the boxes' own conditions
    int ns = 0;
    for (int c0 = 0; c0 < B; c0 += kPlanThreads) {
        const int b = c0 + tid;
        bool first = false;
        if (b < B) {
            const float l0 = lo[3 * b], l1 = lo[3 * b + 1], l2 = lo[3 * b + 2];
            const float h0 = hi[3 * b], h1 = hi[3 * b + 1], h2 = hi[3 * b + 2];
            bool ok = isfinite(l0) && isfinite(l1) && isfinite(l2) && h0 > l0 && h1 > l1 && h2 == INFINITY;
            first = b == 0 || !(lo[3 * b - 3] == l0);
            if (b > 0) {
                const float p0 = lo[3 * b - 3], q0 = hi[3 * b - 3], q1 = hi[3 * b - 2], p2 = lo[3 * b - 1];
                if (first) ok &= q0 == l0 && p0 < l0 && q1 == INFINITY && l1 == lo[1];
                else ok &= q0 == h0 && q1 == l1 && l2 <= p2;
            }
            if (b == B - 1) ok &= h0 == INFINITY && h1 == INFINITY;
            if (!ok) s_bad = 1;
        }
        int tot;
        const int e = prefix(first, &tot);
        if (b < B) sid[b] = (uint16_t)(ns + e + (first ? 1 : 0) - 1);
        ns += tot;
    }
    __syncthreads();
    // columns: the distinct lower edges, sorted (bitonic, +inf padding)
    for (int k = 2; k <= P; k *= 2)
        for (int j = k / 2; j > 0; j /= 2) {
            for (int e = tid; e < P; e += kPlanThreads) {
                const int x = e ^ j;
                if (x > e) {
                    const float u = key[e], v = key[x];
                    if ((u > v) == ((e & k) == 0)) {
                        key[e] = v;
                        key[x] = u;
                    }
                }
            }
            __syncthreads();
        }
    int nc = 0;
    for (int c0 = 0; c0 < B; c0 += kPlanThreads) {  // a value moves only to a lower place
        const int e = c0 + tid;
        const float v = e < B ? key[e] : INFINITY;
        const bool f = e < B && (e == 0 || !(key[e - 1] == v));
        int tot;
        const int at = nc + prefix(f, &tot);
        if (f) key[at] = v;
        nc += tot;
        __syncthreads();
    }
    const bool fits = ns <= walk_strips(B) && nc <= walk_cols(B) && ns * nc <= walk_pairs(B);
    if (s_bad || !fits) {  // the same in every thread
        if (tid == 0) plan->ok = 0;
        return;
    }
    const WalkSizes w = walk_sizes(B, ns, nc);
    float2* box = reinterpret_cast<float2*>(out + w.box);
    float* axis0 = reinterpret_cast<float*>(out + w.axis0);
    float* axis1 = reinterpret_cast<float*>(out + w.axis1);
    uint16_t* lut = reinterpret_cast<uint16_t*>(out + w.lut);
    uint16_t* start = reinterpret_cast<uint16_t*>(out + w.start);
    auto rank1 = [&](float v) {  // columns whose lower edge is below v
        int a = 0, z = nc;
        while (a < z) {
            const int mid = (a + z) / 2;
            if (key[mid] < v) a = mid + 1;
            else z = mid;
        }
        return a;
    };
    for (int b = tid; b < B; b += kPlanThreads) {
        const int i = sid[b], at = b + i + 1;  // after the sentinels of strips 0 .. i
        box[at] = make_float2(lo[3 * b + 1], lo[3 * b + 2]);
        if (b == 0 || sid[b - 1] != i) {
            box[at - 1] = make_float2(0.0f, INFINITY);
            axis0[i] = lo[3 * b];
        }
        const int k1 = rank1(hi[3 * b + 1]);
        for (int k = rank1(lo[3 * b + 1]); k < k1; ++k) start[i * nc + k] = (uint16_t)(8 * at);
    }
    for (int k = tid; k <= nc; k += kPlanThreads) axis1[k] = k < nc ? key[k] : INFINITY;
    if (tid == 0) axis0[ns] = INFINITY;
    __threadfence_block();
    __syncthreads();
    for (int e = nc + tid; e < ns * nc; e += kPlanThreads)
        if (box[start[e] / 8].y > box[start[e - nc] / 8].y) s_bad = 1;
    // Lookup tables: entry c holds the number of edges in cells below c, less
    // one (every such edge is below any coordinate of cell c), at least 0.
    for (int e = tid; e < 2 * kLut; e += kPlanThreads) {
        const int ax = e / kLut, c = e - ax * kLut, G = ax ? nc : ns;
        auto edge = [&](int g) { return ax ? axis1[g] : axis0[g]; };
        const float base = edge(0), span = edge(G - 1) - base;
        const float scale = span > 0.0f ? (float)kLut / span : 0.0f;
        int a = 0, z = G;
        while (a < z) {
            const int mid = (a + z) / 2;
            if (lut_cell(edge(mid), base, scale) < c) a = mid + 1;
            else z = mid;
        }
        lut[e] = (uint16_t)max(a - 1, 0);
        if (c == 0) {
            plan->base[ax] = base;
            plan->scale[ax] = scale;
        }
    }
    __syncthreads();
    if (tid == 0) {
        plan->n_strip = ns;
        plan->n_col = nc;
        plan->ticket = 0u;
        plan->ok = !s_bad;
    }
}

struct EhviArgs {
    const float* mean;  // [M][ldm] by list position
    const float* var;
    int64_t n, ldm;
    const int32_t* list;
    const unsigned int* n_list;
    const float* box_lo;
    const float* box_hi;
    int32_t n_boxes;
    const float* eps;
    int32_t n_mc;
    char* plan;         // NULL: no walk was planned
    float* acq;
};

// Bytes of a plan of n_boxes boxes, and of ehvi_walk's shared memory.
size_t plan_bytes(int n_boxes) {
    const size_t start = walk_sizes(n_boxes, walk_strips(n_boxes), walk_cols(n_boxes)).start;
    return (start + (size_t)walk_pairs(n_boxes) * 2 + 15) / 16 * 16;
}

size_t walk_smem(int n_boxes, int n_mc) {
    return plan_bytes(n_boxes) + (size_t)n_mc * 16 +
           (size_t)kWalkWarps * (kWalkIds * 4 + kWalkBatch * 32);
}

// A warp takes up to eight candidates at a time.  First its lanes take their
// samples densely: coordinates, strip, column and whether the sample lies
// above the floor there; the others add nothing.  The samples above it queue
// (their numbers, in order), and the lanes walk them, one box per step.  A
// walk's length varies from 1 to several hundred boxes, so lanes that finish
// take the next sample from the queue once eight are idle (lanes that wait
// for the longest walk of 32 samples took four times the steps).  A sample's
// value takes its number's place in the queue, and a candidate's values are
// added in the order of its samples, so its sum depends on nothing else in the
// batch.
// Measured (408 000 candidates, 453 boxes, S = 128): 0.79 ms; the fused kernel
// that sums every box took 7.84 ms with the posterior, now 1.10 ms of its own.
// Bound by issue and the latency of the gathers (about 1100 instructions a
// candidate, half the lanes active in them); 8-byte boxes instead of 16-byte
// ones, two boxes per look for finished strips instead of one, and the dynamic
// hand-out of batches took it from 1.28 ms.
__global__ void __launch_bounds__(kWalkThreads, 4) ehvi_walk(const __grid_constant__ EhviArgs a) {
    WalkPlan* plan = reinterpret_cast<WalkPlan*>(a.plan);
    if (!plan->ok) return;  // ehvi_dense does the work
    extern __shared__ __align__(16) float sm[];
    const int ns = plan->n_strip, nc = plan->n_col, S = a.n_mc;
    const WalkSizes w = walk_sizes(a.n_boxes, ns, nc);
    char* tab = reinterpret_cast<char*>(sm);  // the plan from its boxes on
    float4* epsv = reinterpret_cast<float4*>(tab + (w.bytes - w.box));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* mom = reinterpret_cast<float*>(epsv + S) + warp * kWalkBatch * 8;  // [cand][8]: mu 0..2, sd 0..2
    uint32_t* queue = reinterpret_cast<uint32_t*>(epsv + S) + kWalkWarps * kWalkBatch * 8 + warp * kWalkIds;
    for (size_t e = tid; e < (w.bytes - w.box) / 16; e += kWalkThreads)
        reinterpret_cast<uint4*>(tab)[e] = reinterpret_cast<const uint4*>(a.plan + w.box)[e];
    for (int s = tid; s < S; s += kWalkThreads) epsv[s] = make_float4(a.eps[3 * s], a.eps[3 * s + 1], a.eps[3 * s + 2], 0.0f);
    __syncthreads();
    const float2* box = reinterpret_cast<const float2*>(tab);
    const float* axis0 = reinterpret_cast<const float*>(tab + (w.axis0 - w.box));
    const float* axis1 = reinterpret_cast<const float*>(tab + (w.axis1 - w.box));
    const uint16_t* lut = reinterpret_cast<const uint16_t*>(tab + (w.lut - w.box));
    const uint16_t* start = reinterpret_cast<const uint16_t*>(tab + (w.start - w.box));
    const float b0 = plan->base[0], s0 = plan->scale[0], b1 = plan->base[1], s1 = plan->scale[1];
    const int64_t n_work = a.list ? (int64_t)*a.n_list : a.n;
    // A few candidates for each warp of the grid before any warp takes eight.
    const int64_t share = (n_work + (int64_t)gridDim.x * kWalkWarps - 1) / ((int64_t)gridDim.x * kWalkWarps);
    const int batch = (int)max((int64_t)1, min(share, (int64_t)min(kWalkBatch, kWalkIds / S)));
    const float inv_mc = 1.0f / (float)S;
    // The sample's coordinates, strip and column; false if it lies on or below
    // the lower edge of the first strip or column (or is not a number).
    auto locate = [&](const float* mo, int s, float& y0, float& y1, float& y2, int& i, int& k) {
        const float4 e = epsv[s];
        y0 = fmaf(mo[3], e.x, mo[0]);
        y1 = fmaf(mo[4], e.y, mo[1]);
        y2 = fmaf(mo[5], e.z, mo[2]);
        i = lut[lut_cell(y0, b0, s0)];
        while (axis0[i + 1] < y0) ++i;
        k = lut[kLut + lut_cell(y1, b1, s1)];
        while (axis1[k + 1] < y1) ++k;
        return y0 > axis0[0] && y1 > axis1[0];
    };
    const char* boxb = reinterpret_cast<const char*>(box);
    const int sh = S > 1 ? 32 - __clz(S - 1) : 0;  // a sample's number in the queue: candidate << sh | sample
    while (true) {
        unsigned p0 = 0;
        if (lane == 0) p0 = atomicAdd(&plan->ticket, (unsigned)batch);
        const int64_t pos0 = __shfl_sync(0xffffffffu, p0, 0);
        if (pos0 >= n_work) break;
        const int cnt = (int)min((int64_t)batch, n_work - pos0);
        if (lane < cnt)
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                mom[lane * 8 + m] = __ldg(a.mean + m * a.ldm + pos0 + lane);
                mom[lane * 8 + 3 + m] = sqrtf(__ldg(a.var + m * a.ldm + pos0 + lane));
            }
        __syncwarp();
        int nq = 0, first = 0;  // first: where candidate `lane` starts in the queue
        for (int c = 0; c < cnt; ++c) {
            if (lane == c) first = nq;
            for (int s = lane; s - lane < S; s += 32) {
                bool above = false;
                if (s < S) {
                    float y0, y1, y2;
                    int i, k;
                    above = locate(mom + c * 8, s, y0, y1, y2, i, k) &&
                            y2 > reinterpret_cast<const float2*>(boxb + start[i * nc + k])->y;
                }
                const unsigned m = __ballot_sync(0xffffffffu, above);
                if (above) queue[nq + __popc(m & ((1u << lane) - 1u))] = (uint32_t)(c << sh | s);
                nq += __popc(m);
            }
        }
        __syncwarp();
        int head = 0, mine = 0, i = 0;  // mine: the lane's place in the queue
        int b = 0;  // byte offset of the box; 0, the first strip's sentinel, in an idle lane
        const uint16_t* col = start;  // the walk's column in strip i
        bool active = false;
        float y1 = 0.0f, y2 = 0.0f, up = 0.0f, lo0 = 0.0f, w0 = 0.0f, acc = 0.0f, tot = 0.0f;
        while (true) {
            const unsigned idle = __ballot_sync(0xffffffffu, !active);
            if (idle == 0xffffffffu && head >= nq) break;
            if (head < nq && __popc(idle) >= kRefetch) {
                const int at = head + __popc(idle & ((1u << lane) - 1u));
                if (!active && at < nq) {
                    const int id = (int)queue[at], c = id >> sh;
                    float y0;
                    int k;
                    locate(mom + c * 8, id - (c << sh), y0, y1, y2, i, k);
                    lo0 = axis0[i];
                    w0 = y0 - lo0;
                    col = start + i * nc + k;
                    b = *col;
                    up = y1;
                    acc = tot = 0.0f;
                    mine = at;
                    active = true;
                }
                head = min(nq, head + __popc(idle));
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float t;
#pragma unroll
                for (int u = 0; u < kRun; ++u) {  // down the strip's columns while their floor is below the sample
                    const float2 q = *reinterpret_cast<const float2*>(boxb + b);
                    t = y2 - q.y;
                    if (t > 0.0f) {
                        acc = fmaf(up - q.x, t, acc);
                        up = q.x;
                        b -= 8;
                    }
                }
                if (active && !(t > 0.0f)) {  // the strip is done
                    tot = fmaf(w0, acc, tot);
                    if (up == y1 || i == 0) {  // nothing in it, so nothing in those below; or it was the last
                        queue[mine] = __float_as_uint(tot);
                        active = false;
                        b = 0;
                    } else {
                        --i;
                        const float l = axis0[i];
                        w0 = lo0 - l;
                        lo0 = l;
                        col -= nc;
                        b = *col;
                        up = y1;
                        acc = 0.0f;
                    }
                }
            }
        }
        __syncwarp();
        for (int c = 0; c < cnt; ++c) {
            const int e0 = __shfl_sync(0xffffffffu, first, c);
            const int e1 = c + 1 < cnt ? __shfl_sync(0xffffffffu, first, c + 1) : nq;
            float v = 0.0f;
            for (int e = e0 + lane; e < e1; e += 32) v += __uint_as_float(queue[e]);
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) a.acq[a.list ? (int64_t)a.list[pos0 + c] : pos0 + c] = v * inv_mc;
        }
        __syncwarp();
    }
}

// Every box for every sample: 32 candidates per block of 128 threads, warp w
// taking the sample chunks w, w + 4, ...; boxes and samples in shared memory.
template <int M>
__global__ void __launch_bounds__(kDenseThreads) ehvi_dense(const __grid_constant__ EhviArgs a) {
    if (a.plan && reinterpret_cast<const WalkPlan*>(a.plan)->ok) return;
    extern __shared__ __align__(16) float sm[];
    float4* blo = reinterpret_cast<float4*>(sm);
    float4* bhi = blo + a.n_boxes;
    float4* epsv = bhi + a.n_boxes;
    __shared__ float part[kQ][kTC];
    stage_boxes(a.box_lo, a.box_hi, a.n_boxes, a.eps, a.n_mc, M, blo, bhi, epsv);
    __syncthreads();
    const bool fast = boxes_fast(blo, bhi, a.n_boxes, M);
    if (fast) {
        stage_boxes_sat(a.box_lo, a.box_hi, a.n_boxes, M, blo);
        __syncthreads();
    }
    const int slot = threadIdx.x & (kTC - 1), qtr = threadIdx.x / kTC;
    const int64_t n_work = a.list ? (int64_t)*a.n_list : a.n;
    for (int64_t p0 = (int64_t)blockIdx.x * kTC; p0 < n_work; p0 += (int64_t)gridDim.x * kTC) {
        const int64_t pos = p0 + slot;
        const bool live = pos < n_work;
        float mu[M], sd[M];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            mu[m] = live ? __ldg(a.mean + m * a.ldm + pos) : 0.0f;
            sd[m] = live ? sqrtf(__ldg(a.var + m * a.ldm + pos)) : 0.0f;
        }
        float v;
        if constexpr (M <= 3)
            v = fast ? ehvi_partial_sat<M>(mu, sd, blo, a.n_boxes, epsv, a.n_mc, qtr, kQ)
                     : ehvi_partial<M>(mu, sd, blo, bhi, a.n_boxes, epsv, a.n_mc, qtr, kQ);
        else
            v = ehvi_partial<M>(mu, sd, blo, bhi, a.n_boxes, epsv, a.n_mc, qtr, kQ);
        __syncthreads();  // part is free again
        part[qtr][slot] = v;
        __syncthreads();
        if (live && qtr == 0)
            a.acq[a.list ? (int64_t)a.list[pos] : pos] =
                ((part[0][slot] + part[1][slot]) + (part[2][slot] + part[3][slot])) * (1.0f / (float)a.n_mc);
    }
}

template <typename K>
scoot_status launch(scoot_ctx* ctx, K kern, int threads, size_t smem, int64_t want, const EhviArgs& a, cudaStream_t st) {
    SCOOT_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0, sms = 0;
    SCOOT_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
    SCOOT_CUDA(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
    if (per_sm < 1) return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "EHVI kernel needs %zu bytes of shared memory", smem);
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * per_sm));
    kern<<<(unsigned)blocks, threads, smem, st>>>(a);
    SCOOT_LAUNCHED(ctx);
    return SCOOT_OK;
}

}  // namespace

// The plan costs about 12 us, the walk's longest candidates 25, and its steps depend
// on how many boxes a sample reaches, so it takes work enough, boxes x samples x
// candidates: measured over three kinds of fronts (the workloads' with 65 to 296
// boxes, spread over a sphere that prior samples seldom and often lie beyond with 113
// to 362), S = 64 and 128, whole calls, dense against walk.  From 129 observations on:
// 8192 candidates x 304 x 64 103 to 104 us against 112 to 120, 16384 x 113 x 64 83 to
// 84 against 89 to 103; 4096 x 285 to 304 x 128 130 to 134 against 111 to 126 (2300 x 452 x
// 100 142 fused against 103), 16384 x
// 296 to 310 x 64 144 to 149 against 115 to 143, 2^18 x 296 x 128 2691 against 1090.
// Up to 128 observations the samples spread further: 16384 x 324 x 64 132 against 153
// to 161, 24576 x 324 x 64 194 against 224 to 228; 32768 x 324 x 128 366 against 306 to
// 334, 2^18 x 248 x 64 1209 against 658.
bool scoot_ehvi_walks(int M, int64_t n, int n_boxes, int n_mc, int n_rb) {
    return M == 3 && n * n_boxes >= 3 << 18 && n_boxes >= kWalkBoxMin && n_boxes <= kWalkBoxMax && n_mc <= kWalkIds &&
           (int64_t)n_boxes * n_mc * std::max<int64_t>(n, 8192) >= (n_rb <= 2 ? 520000000 : 230000000);
}

size_t scoot_ehvi_walk_bytes(int n_boxes) { return (plan_bytes(n_boxes) + 255) / 256 * 256; }

scoot_status scoot_ehvi_listed(scoot_ctx* ctx, int M, const float* mean, const float* var, int64_t n, int64_t ldm,
                               const int32_t* list, const unsigned int* n_list, const float* box_lo,
                               const float* box_hi, int32_t n_boxes, const float* eps, int32_t n_mc, void* work,
                               float* acq, cudaStream_t st) {
    EhviArgs a;
    std::memset(&a, 0, sizeof(a));
    a.mean = mean;
    a.var = var;
    a.n = n;
    a.ldm = ldm;
    a.list = list;
    a.n_list = n_list;
    a.box_lo = box_lo;
    a.box_hi = box_hi;
    a.n_boxes = n_boxes;
    a.eps = eps;
    a.n_mc = n_mc;
    a.acq = acq;
    if (work) {
        a.plan = static_cast<char*>(work);
        walk_plan<<<1, kPlanThreads, (size_t)kWalkBoxMax * 6, st>>>(box_lo, box_hi, n_boxes, static_cast<char*>(work));
        SCOOT_LAUNCHED(ctx);
        scoot_status s = launch(ctx, ehvi_walk, kWalkThreads, walk_smem(n_boxes, n_mc),
                                (n + kWalkWarps - 1) / kWalkWarps, a, st);
        if (s != SCOOT_OK) return s;
    }
    const size_t smem = (size_t)(2 * n_boxes + n_mc) * 16;
    const int64_t tiles = (n + kTC - 1) / kTC;
    switch (M) {
    case 2: return launch(ctx, ehvi_dense<2>, kDenseThreads, smem, tiles, a, st);
    case 3: return launch(ctx, ehvi_dense<3>, kDenseThreads, smem, tiles, a, st);
    case 4: return launch(ctx, ehvi_dense<4>, kDenseThreads, smem, tiles, a, st);
    default: return scoot_fail(ctx, SCOOT_EUNSUPPORTED, "M = %d", M);
    }
}
