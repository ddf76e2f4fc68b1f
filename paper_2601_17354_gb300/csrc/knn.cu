// K13 knn_grid and K14 features / PCA initializer (operator I of PocketGS, Sec. III-B).
//
// kNN: points are counting-sorted into a uniform grid whose cells lie row after row, so the cells of a
// box around a query are a few runs of consecutive points.  A warp takes one query (in cell order, so
// neighbouring warps read the same runs): its lanes take 32 candidates at a time and hold the K best
// (squared distance, index) pairs found so far, sorted, one per lane.  The box widens until the
// k-th distance is below its reach, which guarantees that no point outside can be closer: the result
// is the exact k nearest other points.  Squared distances use the fp32 sequence
// d2 = fma(dx, dx, fma(dy, dy, dz * dz)) with dx = p_j - p_i, ties broken by index, so the neighbour
// lists are reproducible bit for bit.  The bounding box and the grid stay on the device.
//
// Features and the paper's initializer are computed per point at about twice FP32's precision, in FP64 where that
// does not decide (k_features_init): Eq. 5 covariance of the K_n = 16 nearest neighbours about their centroid, its
// smallest-eigenvalue eigenvector as the normal (cyclic Jacobi, eigenvectors canonicalised so the
// largest-magnitude component is positive), Eq. 6 tangential scale from the K_s = 3 nearest neighbours, normal scale
// r_normal s_t, z axis rotated onto the normal, opacity logit(0.1); and the 16 features of the
// learned initializer from the 32 nearest neighbours.
#include <cuda_bf16.h>

#include <algorithm>

#include "df.cuh"
#include "pgs_internal.cuh"

namespace pgs {
namespace {

constexpr int kThreads = 256;

struct Grid {
    float lo[3];
    float h;
    int dim[3];
    int cells;
};

// Is this CTA the last of the grid to get here?  (Its earlier writes are visible to the last one; the
// last CTA resets the ticket.)  No CTA waits for another.
__device__ __forceinline__ bool last_cta(uint32_t* ticket) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (s_last) *ticket = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// Bounding box of the points and the grid over it (at most max_cells cells): per-CTA boxes into
// part [CTAs][6], combined by the last CTA.
constexpr int kBoxCtas = 152;
__global__ void __launch_bounds__(kThreads)
k_bbox(int64_t n, const float* __restrict__ P, float* __restrict__ part, uint32_t* ticket, int64_t max_cells,
       Grid* __restrict__ grid) {
    __shared__ float s_box[6][kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float lo[3] = {3.4e38f, 3.4e38f, 3.4e38f}, hi[3] = {-3.4e38f, -3.4e38f, -3.4e38f};
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kThreads)
        for (int d = 0; d < 3; ++d) {
            lo[d] = fminf(lo[d], P[d * n + i]);
            hi[d] = fmaxf(hi[d], P[d * n + i]);
        }
    auto reduce = [&] {  // over the CTA: thread 0 holds the box
        for (int d = 0; d < 3; ++d) {
            for (int o = 16; o > 0; o >>= 1) {
                lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
                hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
            }
            if (lane == 0) {
                s_box[d][warp] = lo[d];
                s_box[3 + d][warp] = hi[d];
            }
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int d = 0; d < 3; ++d)
                for (int w = 1; w < kThreads / 32; ++w) {
                    lo[d] = fminf(lo[d], s_box[d][w]);
                    hi[d] = fmaxf(hi[d], s_box[3 + d][w]);
                }
    };
    reduce();
    if (threadIdx.x == 0)
        for (int d = 0; d < 3; ++d) {
            part[6 * blockIdx.x + d] = lo[d];
            part[6 * blockIdx.x + 3 + d] = hi[d];
        }
    if (!last_cta(ticket)) return;
    for (int d = 0; d < 3; ++d) {
        lo[d] = 3.4e38f;
        hi[d] = -3.4e38f;
    }
    for (int c = threadIdx.x; c < (int)gridDim.x; c += kThreads)
        for (int d = 0; d < 3; ++d) {
            lo[d] = fminf(lo[d], __ldcg(&part[6 * c + d]));
            hi[d] = fmaxf(hi[d], __ldcg(&part[6 * c + 3 + d]));
        }
    reduce();
    if (threadIdx.x != 0) return;
    // cell edge from the bounding box volume per point (the box search keeps it exact whatever the
    // density): about 2.4 cells per point, so surface points fill few cells densely
    float e[3];
    for (int d = 0; d < 3; ++d) e[d] = fmaxf(hi[d] - lo[d], 1e-6f);
    float h = 0.75f * cbrtf(e[0] * e[1] * e[2] / (float)n);
    Grid g;
    for (int tries = 0;; ++tries) {
        int64_t cells = 1;
        for (int d = 0; d < 3; ++d) {
            g.lo[d] = lo[d];
            // (a box that is not finite, or no edge that fits, ends in one cell)
            g.dim[d] = tries < 256 && e[d] / h < 3.4e38f ? (int)fminf(1024.f, floorf(e[d] / h) + 1) : 1;
            cells *= g.dim[d];
        }
        g.h = h;
        g.cells = (int)cells;
        if (cells <= max_cells) break;
        h *= 1.25f;
    }
    *grid = g;
}

__device__ __forceinline__ int cell_coord(float x, float lo, float h, int dim) {
    return min(max((int)floorf((x - lo) / h), 0), dim - 1);
}

__global__ void k_cell_count(int64_t n, const float* __restrict__ P, const Grid* __restrict__ grid,
                             uint32_t* __restrict__ cell_of, uint32_t* __restrict__ counts) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const Grid g = *grid;
    const int cx = cell_coord(P[i], g.lo[0], g.h, g.dim[0]);
    const int cy = cell_coord(P[n + i], g.lo[1], g.h, g.dim[1]);
    const int cz = cell_coord(P[2 * n + i], g.lo[2], g.h, g.dim[2]);
    const uint32_t c = ((uint32_t)cz * g.dim[1] + cy) * g.dim[0] + cx;
    cell_of[i] = c;
    atomicAdd(&counts[c], 1u);
}

// Exclusive scan of the cells' counts into start [cells + 1] and, in place, into the scatter's cursors:
// runs of kScanRun cells per CTA, their totals first (the last CTA scans them), then the cells.  One CTA
// walking all cells took 0.42 ms of the 6.1 ms that 200k points took.
constexpr int kScanItems = 16;
constexpr int kScanRun = kThreads * kScanItems;

__device__ __forceinline__ uint32_t cta_exclusive(uint32_t v, uint32_t* s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    __syncthreads();
    return before + incl - v;
}

__global__ void __launch_bounds__(kThreads)
k_scan_totals(const Grid* __restrict__ grid, const uint32_t* __restrict__ counts, uint32_t* __restrict__ totals,
              uint32_t* ticket) {
    __shared__ uint32_t s_warp[kThreads / 32];
    __shared__ uint32_t s_carry;
    const int64_t cells = grid->cells, base = (int64_t)blockIdx.x * kScanRun;
    uint32_t sum = 0;
    for (int k = 0; k < kScanItems; ++k) {
        const int64_t c = base + k * kThreads + threadIdx.x;
        sum += c < cells ? counts[c] : 0u;
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < kThreads / 32; ++w) t += s_warp[w];
        totals[blockIdx.x] = t;
    }
    if (!last_cta(ticket)) return;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < (int)gridDim.x; b0 += kThreads) {
        const int b = b0 + threadIdx.x;
        const uint32_t v = b < (int)gridDim.x ? __ldcg(&totals[b]) : 0u;
        const uint32_t carry = s_carry, ex = carry + cta_exclusive(v, s_warp);
        if (b < (int)gridDim.x) totals[b] = ex;
        if (threadIdx.x == kThreads - 1) s_carry = ex + v;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kThreads)
k_scan_cells(int64_t n, const Grid* __restrict__ grid, uint32_t* __restrict__ counts, const uint32_t* __restrict__ totals,
             uint32_t* __restrict__ start) {
    __shared__ uint32_t s_warp[kThreads / 32];
    const int64_t cells = grid->cells, base = (int64_t)blockIdx.x * kScanRun + threadIdx.x * kScanItems;
    uint32_t v[kScanItems], sum = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < cells ? counts[base + k] : 0u;
        sum += v[k];
    }
    uint32_t run = totals[blockIdx.x] + cta_exclusive(sum, s_warp);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < cells) start[base + k] = counts[base + k] = run;
        run += v[k];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) start[cells] = (uint32_t)n;
}

// points in cell order: position and index bits in one 16-byte record
__global__ void k_cell_scatter(int64_t n, const float* __restrict__ P, const uint32_t* __restrict__ cell_of,
                               uint32_t* __restrict__ cursor, float4* __restrict__ Ps) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    const uint32_t s = atomicAdd(&cursor[cell_of[i]], 1u);
    Ps[s] = make_float4(P[i], P[n + i], P[2 * n + i], __int_as_float((int)i));
}

// One step of a bitonic network over the warp: the lane keeps the smaller of its key and lane ^ j's when
// `low`, else the larger.
__device__ __forceinline__ unsigned long long exchange(unsigned long long k, int j, bool low) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, k, j);
    return (o < k) == low ? o : k;
}

// The K nearest other points of each point, a warp per point.  Instruction-bound: 32 candidates cost
// about 40 instructions to fetch and rate, a batch with more than kFew candidates among the best so far
// one bitonic sort and merge (21 exchanges), fewer of them an insertion each (200k points on a plane: 408 us for
// the whole search at kFew = 4, 402 at 10, 436 at 20; on a sphere 324, 322, 333).  A thread per point
// with its list in registers paid a pass of 32 compare-and-swaps whenever any lane of its warp had
// a candidate and walked cells one by one: 200k surface points, K = 32, 2.35 ms.
constexpr int kQueryWarps = 4;
template <int K>
__global__ void __launch_bounds__(32 * kQueryWarps)
k_knn_query(int64_t n, const Grid* __restrict__ grid, const uint32_t* __restrict__ start, const float4* __restrict__ Ps,
            int32_t* __restrict__ nb) {
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kFew = 10;
    constexpr unsigned long long kNone = ~0ull;
    const int lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * kQueryWarps + (threadIdx.x >> 5);
    if (s >= n) return;  // the whole warp
    const Grid g = *grid;
    const float4 q = Ps[s];
    const int cx = cell_coord(q.x, g.lo[0], g.h, g.dim[0]);
    const int cy = cell_coord(q.y, g.lo[1], g.h, g.dim[1]);
    const int cz = cell_coord(q.z, g.lo[2], g.h, g.dim[2]);
    const int maxr = max(g.dim[0], max(g.dim[1], g.dim[2]));
    unsigned long long best = kNone;  // lane l: the l-th best key, distance bits << 32 | index
    int r0 = -1;                      // radius of the box scanned so far
    int R = 1;
    for (;;) {
        // the box of radius R less that of radius r0, as runs of cells along x: a row outside the inner
        // box is one run, a row through it two.  Only the grid's rows are numbered: on a plane or a line most of
        // the box lies outside (2,000 points on an axis, R up to 1,024 in a grid of one row: 97 ms with every row of
        // the box numbered, 0.07 ms so; 200k on an axis-aligned plane 0.82 -> 0.40 ms, on a sphere 0.32 both ways)
        const int ya = max(cy - R, 0), za = max(cz - R, 0);
        const int ny = min(cy + R, g.dim[1] - 1) - ya + 1, nz = min(cz + R, g.dim[2] - 1) - za + 1;
        const int halves = r0 < 0 ? 1 : 2, runs = ny * nz * halves;
        for (int base = 0; base < runs; base += 32) {
            const int run = base + lane, row = run / halves, half = run - row * halves;
            const int z = za + row / ny, y = ya + row % ny;
            int xa = cx - R, xb = cx + R;
            if (abs(y - cy) <= r0 && abs(z - cz) <= r0) {
                if (half == 0) xb = cx - r0 - 1;
                else xa = cx + r0 + 1;
            } else if (half) {
                xb = xa - 1;
            }
            xa = max(xa, 0);
            xb = min(xb, g.dim[0] - 1);
            uint32_t first = 0, cnt = 0;
            if (run < runs && xa <= xb) {
                const uint32_t c = ((uint32_t)z * g.dim[1] + y) * g.dim[0];
                first = start[c + xa];
                cnt = start[c + xb + 1] - first;
            }
            uint32_t incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kAll, incl, o);
                if (lane >= o) incl += t;
            }
            const uint32_t total = __shfl_sync(kAll, incl, 31);
            const uint32_t shift = first - (incl - cnt);  // candidate k of this run: point shift + k
            for (uint32_t k0 = 0; k0 < total; k0 += 32) {
                const uint32_t k = k0 + lane;
                int lo = 0, hi = 31;  // run of candidate k: the first lane whose inclusive count exceeds k
#pragma unroll
                for (int step = 0; step < 5; ++step) {
                    const int mid = (lo + hi) >> 1;
                    const uint32_t im = __shfl_sync(kAll, incl, mid);
                    if (lo < hi) {
                        if (im > k) hi = mid;
                        else lo = mid + 1;
                    }
                }
                const uint32_t at = __shfl_sync(kAll, shift, lo) + k;
                unsigned long long key = kNone;
                if (k < total && at != (uint32_t)s) {
                    const float4 c = Ps[at];
                    const float ex = c.x - q.x, ey = c.y - q.y, ez = c.z - q.z;
                    const float d2 = __fmaf_rn(ex, ex, __fmaf_rn(ey, ey, __fmul_rn(ez, ez)));
                    if (d2 <= 3.4e38f) key = (unsigned long long)__float_as_uint(d2) << 32 | __float_as_uint(c.w);
                }
                unsigned pass = __ballot_sync(kAll, key < __shfl_sync(kAll, best, K - 1));
                if (__popc(pass) <= kFew) {
                    for (; pass; pass &= pass - 1u) {
                        const unsigned long long in = __shfl_sync(kAll, key, __ffs(pass) - 1);
                        const unsigned long long up = __shfl_up_sync(kAll, best, 1);
                        if (in < best) best = lane > 0 && up > in ? up : in;
                    }
                } else {
                    // the batch sorted in descending order, the smaller of each lane's two keys, and the
                    // resulting bitonic sequence merged
#pragma unroll
                    for (int w = 2; w <= 32; w <<= 1)
#pragma unroll
                        for (int j = w >> 1; j > 0; j >>= 1)
                            key = exchange(key, j, ((lane & j) == 0) == ((lane & w) != 0 && w < 32));
                    best = key < best ? key : best;
#pragma unroll
                    for (int j = 16; j > 0; j >>= 1) best = exchange(best, j, (lane & j) == 0);
                }
            }
        }
        if (R >= maxr) break;  // the whole grid
        // every point within R h of the query lies in the scanned box
        const unsigned long long kth = __shfl_sync(kAll, best, K - 1);
        const float d2 = __uint_as_float((uint32_t)(kth >> 32)), reach = (float)R * g.h;
        if (kth != kNone && d2 < reach * reach * 0.9999f) break;
        r0 = R;
        // the radius the k-th distance asks for, or twice this one while there are fewer than K points
        R = kth != kNone ? (int)fminf(sqrtf(d2) / g.h * 1.0001f + 1.0f, 1024.f) : 2 * R;
        R = min(max(R, r0 + 1), maxr);
    }
    if (lane < K) nb[(int64_t)__float_as_int(q.w) * K + lane] = best == kNone ? -1 : (int32_t)(uint32_t)best;
}

// ---------------------------------------------------------------------------------------------
// features and the paper's initializer
// ---------------------------------------------------------------------------------------------

// Eigen-decomposition of the symmetric matrix (a[0] a[1] a[2]; a[1] a[3] a[4]; a[2] a[4] a[5]) by cyclic
// Jacobi: w ascending, V columns = eigenvectors with their largest-magnitude component positive.  A
// rotation's angle needs FP32 only (it leaves the element it clears at 1e-7 of itself, the next sweep
// at 1e-14); its cosine and sine are formed from that angle to full precision, so V stays orthonormal.
__device__ void jacobi3(const Df a[6], Df w[3], Df V[3][3]) {
    Df A[3][3] = {{a[0], a[1], a[2]}, {a[1], a[3], a[4]}, {a[2], a[4], a[5]}};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) V[i][j] = {i == j ? 1.0f : 0.0f, 0.0f};
    const float tiny = 1e-14f * (fabsf(a[0].h) + fabsf(a[3].h) + fabsf(a[5].h));
#pragma unroll 1
    for (int sweep = 0; sweep < 10; ++sweep) {
        if (!(fabsf(A[0][1].h) + fabsf(A[0][2].h) + fabsf(A[1][2].h) > tiny)) break;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int p = e < 2 ? 0 : 1, q = e == 0 ? 1 : 2, r = 3 - p - q;
            const Df x = A[p][p], y = A[q][q], z = A[p][q];
            if (z.h == 0.0f) continue;
            const float theta = df_sub(y, x).h / (2.0f * z.h);
            const float t = (theta >= 0.0f ? 1.0f : -1.0f) / (fabsf(theta) + sqrtf(fmaf(theta, theta, 1.0f)));
            // c = 1 / sqrt(1 + t^2) by one Newton step from the FP32 value, s = t c
            const float tt = __fmul_rn(t, t);
            const Df u = df_two(1.0f, tt);
            const float ul = __fadd_rn(u.l, __fmaf_rn(t, t, -tt));
            const float c0 = rsqrtf(u.h), cc0 = __fmul_rn(c0, c0);
            float err = __fmaf_rn(-u.h, cc0, 1.0f);
            err = __fmaf_rn(-ul, cc0, __fmaf_rn(-u.h, __fmaf_rn(c0, c0, -cc0), err));
            const Df c = df_fast(c0, __fmul_rn(0.5f * c0, err)), s = df_mul(c, {t, 0.0f});
            const Df c2 = df_mul(c, c), s2 = df_mul(s, s), cs = df_mul(c, s);
            const Df w2 = df_scale(df_mul(cs, z), 2.0f);
            A[p][p] = df_add(df_sub(df_mul(c2, x), w2), df_mul(s2, y));
            A[q][q] = df_add(df_add(df_mul(s2, x), w2), df_mul(c2, y));
            A[p][q] = A[q][p] = df_add(df_mul(cs, df_sub(x, y)), df_mul(df_sub(c2, s2), z));
            const Df f = A[r][p], g = A[r][q];
            A[r][p] = A[p][r] = df_sub(df_mul(c, f), df_mul(s, g));
            A[r][q] = A[q][r] = df_add(df_mul(s, f), df_mul(c, g));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Df vp = V[k][p], vq = V[k][q];
                V[k][p] = df_sub(df_mul(c, vp), df_mul(s, vq));
                V[k][q] = df_add(df_mul(s, vp), df_mul(c, vq));
            }
        }
    }
    auto less = [](Df u, Df v) { return u.h < v.h || (u.h == v.h && u.l < v.l); };
    // ascending eigenvalues (three-element sorting network over the columns)
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = A[k][k];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const int i = e == 1 ? 1 : 0, j = i + 1;
        if (less(w[j], w[i])) {
            const Df t = w[i];
            w[i] = w[j];
            w[j] = t;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const Df v = V[k][i];
                V[k][i] = V[k][j];
                V[k][j] = v;
            }
        }
    }
    auto mag = [](Df v) { return v.h < 0.0f ? df_neg(v) : v; };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Df big = V[0][k];
        if (less(mag(big), mag(V[1][k]))) big = V[1][k];
        if (less(mag(big), mag(V[2][k]))) big = V[2][k];
        if (big.h < 0.0f)
#pragma unroll
            for (int r = 0; r < 3; ++r) V[r][k] = df_neg(V[r][k]);
    }
}

// w (times scale^2) and V of the covariance of the first k neighbours [neighbour][axis][point] in FP64, for a
// point whose eigenvalues lie too close for two floats (see k_features_init).
struct Frame {
    Df w[3], V[3][3];
};
__device__ __noinline__ Frame frame64(const float (*nb)[3][33], int point, int k, double scale) {
    double c[3] = {0, 0, 0}, A[3][3] = {}, U[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
    for (int a = 0; a < k; ++a)
        for (int d = 0; d < 3; ++d) c[d] += (double)nb[a][d][point];
    for (int d = 0; d < 3; ++d) c[d] /= k;
    for (int a = 0; a < k; ++a) {
        double v[3];
        for (int d = 0; d < 3; ++d) v[d] = (double)nb[a][d][point] - c[d];
        for (int x = 0; x < 3; ++x)
            for (int y = 0; y < 3; ++y) A[x][y] += v[x] * v[y];
    }
    for (int x = 0; x < 3; ++x)
        for (int y = 0; y < 3; ++y) A[x][y] /= k;
    for (int sweep = 0; sweep < 64; ++sweep) {
        if (A[0][1] * A[0][1] + A[0][2] * A[0][2] + A[1][2] * A[1][2] < 1e-300) break;
        for (int p = 0; p < 2; ++p)
            for (int q = p + 1; q < 3; ++q) {
                if (A[p][q] == 0.0) continue;
                const double theta = (A[q][q] - A[p][p]) / (2.0 * A[p][q]);
                const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                const double co = 1.0 / sqrt(t * t + 1.0), si = t * co;
                auto turn = [&](double& f, double& g) {
                    const double h = co * f - si * g;
                    g = si * f + co * g;
                    f = h;
                };
                for (int r = 0; r < 3; ++r) turn(A[r][p], A[r][q]);
                for (int r = 0; r < 3; ++r) turn(A[p][r], A[q][r]);
                for (int r = 0; r < 3; ++r) turn(U[r][p], U[r][q]);
            }
    }
    int at[3] = {0, 1, 2};  // columns by ascending eigenvalue
    for (int e = 0; e < 3; ++e) {
        const int i = e == 1 ? 1 : 0;
        if (A[at[i + 1]][at[i + 1]] < A[at[i]][at[i]]) {
            const int t = at[i];
            at[i] = at[i + 1];
            at[i + 1] = t;
        }
    }
    Frame f;
    for (int j = 0; j < 3; ++j) {
        const int from = at[j];
        int big = 0;
        for (int r = 1; r < 3; ++r)
            if (fabs(U[r][from]) > fabs(U[big][from])) big = r;
        f.w[j] = df_from(A[from][from] * scale * scale);
        for (int r = 0; r < 3; ++r) f.V[r][j] = df_from(U[big][from] < 0 ? -U[r][from] : U[r][from]);
    }
    return f;
}

__device__ void mat_to_quat(const double R[3][3], double q[4]) {
    const double tr = R[0][0] + R[1][1] + R[2][2];
    if (tr > 0) {
        const double s = sqrt(tr + 1.0) * 2;
        q[0] = 0.25 * s;
        q[1] = (R[2][1] - R[1][2]) / s;
        q[2] = (R[0][2] - R[2][0]) / s;
        q[3] = (R[1][0] - R[0][1]) / s;
    } else if (R[0][0] > R[1][1] && R[0][0] > R[2][2]) {
        const double s = sqrt(1.0 + R[0][0] - R[1][1] - R[2][2]) * 2;
        q[0] = (R[2][1] - R[1][2]) / s;
        q[1] = 0.25 * s;
        q[2] = (R[0][1] + R[1][0]) / s;
        q[3] = (R[0][2] + R[2][0]) / s;
    } else if (R[1][1] > R[2][2]) {
        const double s = sqrt(1.0 + R[1][1] - R[0][0] - R[2][2]) * 2;
        q[0] = (R[0][2] - R[2][0]) / s;
        q[1] = (R[0][1] + R[1][0]) / s;
        q[2] = 0.25 * s;
        q[3] = (R[1][2] + R[2][1]) / s;
    } else {
        const double s = sqrt(1.0 + R[2][2] - R[0][0] - R[1][1]) * 2;
        q[0] = (R[1][0] - R[0][1]) / s;
        q[1] = (R[0][2] + R[2][0]) / s;
        q[2] = (R[1][2] + R[2][1]) / s;
        q[3] = 0.25 * s;
    }
}

// One thread per point: nb [n][32] ascending.  Writes features (fp32 [n][16] and bf16 [n][16]),
// the eigenframe quaternion frame_q [4][n], and the paper's initializer into init (log-scales,
// quaternions, opacity logits; means = the points; SH zero).  Each warp first gathers its 32 points'
// neighbours into shared memory, a point's 32 at a time (one coalesced read of its list), for the two
// passes over them.  Offsets from the point are exact in two floats and are scaled by a power of two to
// about 1.  In FP64 throughout, 200k points took 3.33 ms, all of it in the FP64 pipe; FP64 is left
// where a handful of values a point leave the kernel through a logarithm or a quaternion, and for neighbourhoods
// that two floats do not decide (of 200k points on a sphere or a plane none, on one line all: 568 us for 2,000
// points in FP64 throughout, 552 here).  0.36 to 0.38 ms now (on a plane the extra pass for the smallest eigenvalue
// is 0.01 of it), with one copy of the eigenvalue code for both neighbourhoods (expanded twice, the code
// outgrew the instruction cache: 0.46 ms) and one pass over the neighbours for both covariances.
constexpr int kFeatWarps = 2;
__global__ void __launch_bounds__(32 * kFeatWarps)
k_features_init(int64_t n, const float* __restrict__ P, const int32_t* __restrict__ nb, float r_normal,
                float* __restrict__ feats, __nv_bfloat16* __restrict__ feats_bf16, float* __restrict__ frame_q,
                pgs_gaussians init) {
    __shared__ float s_nb[kFeatWarps][32][3][33];  // [neighbour][axis][point], padded: gathered by neighbour, read by point
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = ((int64_t)blockIdx.x * kFeatWarps + warp) * 32, i = i0 + lane;
    for (int p = 0; p < 32 && i0 + p < n; ++p) {
        const int32_t j = nb[(i0 + p) * 32 + lane];
        const int64_t k = j >= 0 && j < n ? j : i0 + p;
        for (int d = 0; d < 3; ++d) s_nb[warp][lane][d][p] = P[d * n + k];
    }
    __syncwarp();
    if (i >= n) return;
    const float p0[3] = {P[i], P[n + i], P[2 * n + i]};
    // scale: the farthest neighbour's offset has its largest component in [1, 2); the coordinates are scaled
    // before the difference, which then neither overflows nor rounds
    float far = 0.f;
    for (int d = 0; d < 3; ++d) far = fmaxf(far, fabsf(0.5f * s_nb[warp][31][d][lane] - 0.5f * p0[d]));
    const int ex = far > 0.f && isfinite(far) ? min(max(ilogbf(far) + 1, -100), 127) : 0;
    const float scale = ldexpf(1.0f, -ex);
    const float q0[3] = {p0[0] * scale, p0[1] * scale, p0[2] * scale};
    auto offset = [&](int a, Df u[3]) {
#pragma unroll
        for (int d = 0; d < 3; ++d) u[d] = df_two(s_nb[warp][a][d][lane] * scale, -q0[d]);
    };
    // sums of the offsets (the first 16, all 32) and of the distances (the first 3, all 32)
    const Df zero = {0.f, 0.f};
    Df m16[3] = {zero, zero, zero}, m32[3] = {zero, zero, zero}, d3 = zero, d32 = zero;
#pragma unroll 1
    for (int a = 0; a < 32; ++a) {
        Df u[3];
        offset(a, u);
        if (a == 16)
            for (int d = 0; d < 3; ++d) m16[d] = m32[d];
        if (a == 3) d3 = d32;
#pragma unroll
        for (int d = 0; d < 3; ++d) df_acc(m32[d], u[d]);
        df_acc(d32, df_norm(u[0], u[1], u[2]));
    }
    auto settle = [](Df& v) { v = df_two(v.h, v.l); };
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        settle(m16[d]);
        settle(m32[d]);
    }
    settle(d3);
    settle(d32);
    // covariances (times 16 and 32), each about its own mean: the 16 nearest about theirs, moved to the mean of
    // all 32 by adding 16 e e^T, then the rest about that.  (Taken about one centre and corrected by a
    // subtraction, the covariance of 16 neighbours that lie close together drowns in the rounding of the other's.)
    Df c[3], e[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        c[d] = df_scale(m16[d], 0.0625f);
        m32[d] = df_scale(m32[d], 0.03125f);  // the means from here on
        e[d] = df_sub(c[d], m32[d]);
    }
    Df C16[6], C32[6] = {zero, zero, zero, zero, zero, zero};
#pragma unroll 1
    for (int a = 0; a < 32; ++a) {
        Df v[3];
        offset(a, v);
        if (a == 16) {
            int k = 0;
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                c[x] = m32[x];
#pragma unroll
                for (int y = x; y < 3; ++y, ++k) {
                    C16[k] = df_two(C32[k].h, C32[k].l);
                    C32[k] = df_add(C16[k], df_scale(df_mul(e[x], e[y]), 16.0f));
                }
            }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) v[d] = df_sub(v[d], c[d]);
        int k = 0;
#pragma unroll
        for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int y = x; y < 3; ++y) df_dot(C32[k++], v[x], v[y]);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        C16[k] = df_scale(C16[k], 0.0625f);
        C32[k] = df_scale(df_two(C32[k].h, C32[k].l), 0.03125f);
    }
    // both decompositions through one copy of the code: it and the loops above are several times the
    // instruction cache when expanded
    Df w[3], V[3][3], nrm[3];
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        Df C[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) C[k] = pass ? C32[k] : C16[k];
        jacobi3(C, w, V);
        // An eigenvector is known to 3e-14 of the trace over its distance from the next eigenvalue.  Below 4e-6 of
        // the trace that is no longer far under FP32's rounding; nor does it settle an eigenvector's sign when two
        // components of opposite sign are its largest to 3e-8, and nothing is known of points closer together than
        // 1e-10 of the farthest offset.  Such neighbourhoods (lines, lattices, coincident points) take FP64: about
        // 12 us to the launch where one warp in 200k points has one.
        const float trace = w[0].h + w[1].h + w[2].h, close = 4e-6f * trace;
        bool open = !(w[1].h - w[0].h > close) || (pass && !(w[2].h - w[1].h > close)) || !(trace > 1e-20f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {  // (the largest component is positive: the sign hangs on a negative one near it)
            const float big = fmaxf(V[0][k].h, fmaxf(V[1][k].h, V[2][k].h));
            open = open || ((k == 0 || pass) && !(big + fminf(V[0][k].h, fminf(V[1][k].h, V[2][k].h)) > 3e-8f));
        }
        if (open) {
            const Frame fr = frame64(s_nb[warp], lane, pass ? 32 : 16, scale);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                w[a] = fr.w[a];
#pragma unroll
                for (int b = 0; b < 3; ++b) V[a][b] = fr.V[a][b];
            }
        }
        if (pass == 0)  // the smallest eigenvector of the 16 neighbours: the normal
#pragma unroll
            for (int d = 0; d < 3; ++d) nrm[d] = V[d][0];
    }
    if (w[0].h < 4e-6f * w[2].h) {
        // A flat neighbourhood: the covariance knows its smallest eigenvalue to 1e-14 of the trace only.  The mean
        // square of the offsets along the normal, which cancels nothing, has it to FP32 however small.
        Df at = zero, sq = zero;
#pragma unroll
        for (int d = 0; d < 3; ++d) df_dot(at, V[d][0], m32[d]);
        at = df_two(at.h, at.l);
#pragma unroll 1
        for (int a = 0; a < 32; ++a) {
            Df u[3], t = zero;
            offset(a, u);
#pragma unroll
            for (int d = 0; d < 3; ++d) df_dot(t, V[d][0], u[d]);
            t = df_sub(df_two(t.h, t.l), at);
            df_dot(sq, t, t);
        }
        w[0] = df_scale(df_two(sq.h, sq.l), 0.03125f);
    }
    float f[16];
    const Df sum = df_add(df_add(w[0], w[1]), w[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) f[a] = sum.h > 0.f ? df_ratio(w[a], sum) : (float)(1.0 / 3.0);
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int d = 0; d < 3; ++d) f[3 + 3 * k + d] = V[d][k].h;
#pragma unroll
    for (int d = 0; d < 3; ++d) f[12 + d] = df_ratio(m32[d], df_scale(d32, 0.03125f));
    const double unit = ldexp(1.0, ex);
    f[15] = (float)(-3.0 * log(df_double(d32) * (0.03125 * unit)));
#pragma unroll
    for (int a = 0; a < 16; ++a) {
        feats[i * 16 + a] = f[a];
        feats_bf16[i * 16 + a] = __float2bfloat16_rn(f[a]);
    }
    double R[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        R[d][0] = df_double(V[d][2]);
        R[d][1] = df_double(V[d][1]);
        R[d][2] = df_double(V[d][0]);
    }
    const double det = R[0][0] * (R[1][1] * R[2][2] - R[1][2] * R[2][1]) -
                       R[0][1] * (R[1][0] * R[2][2] - R[1][2] * R[2][0]) +
                       R[0][2] * (R[1][0] * R[2][1] - R[1][1] * R[2][0]);
    if (det < 0)
#pragma unroll
        for (int d = 0; d < 3; ++d) R[d][0] = -R[d][0];
    double q[4];
    mat_to_quat(R, q);
#pragma unroll
    for (int a = 0; a < 4; ++a) frame_q[a * n + i] = (float)q[a];

    // the paper's initializer: normal from 16 neighbours (Eq. 5), scale from 3 (Eq. 6)
    const double nx = df_double(nrm[0]), ny = df_double(nrm[1]), nz = df_double(nrm[2]);
    const double st = df_double(d3) * unit / 3.0, ls = log(st);
    init.log_scales[i] = (float)ls;
    init.log_scales[n + i] = (float)ls;
    init.log_scales[2 * n + i] = (float)log((double)r_normal * st);
    double qw, qx, qy, qz;
    if (nz < -1.0 + 1e-12) {
        qw = 0; qx = 1; qy = 0; qz = 0;
    } else {
        qw = sqrt(0.5 * (1.0 + nz));
        const double s = 1.0 / (2.0 * qw);
        qx = -ny * s;
        qy = nx * s;
        qz = 0.0;
    }
    init.quats[i] = (float)qw;
    init.quats[n + i] = (float)qx;
    init.quats[2 * n + i] = (float)qy;
    init.quats[3 * n + i] = (float)qz;
    init.opacity_logits[i] = (float)log(0.1 / 0.9);
    for (int d = 0; d < 3; ++d) init.means[d * n + i] = p0[d];
    const int K = (init.sh_degree + 1) * (init.sh_degree + 1);
    for (int c = 0; c < 3 * K; ++c) init.sh[(int64_t)c * n + i] = 0.f;
}

// Hamilton product of (w, x, y, z) quaternions
__device__ __forceinline__ void qmul(const float a[4], const float b[4], float o[4]) {
    o[0] = a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3];
    o[1] = a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2];
    o[2] = a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1];
    o[3] = a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0];
}

// Learned parameters from MLP outputs y [n][8], as corrections of the paper's initializer `pca`
// of the same point: log-scales pca + y0..2, rotation normalise(pca q) (x) normalise(y3..6),
// logit pca + y7.  A point whose outputs are not finite (or whose quaternion is zero) keeps the
// paper's initializer and is counted in *fallbacks.
__global__ void k_apply_mlp(int64_t n, const float* __restrict__ y, pgs_gaussians pca, pgs_gaussians out,
                            uint32_t* fallbacks) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float* yi = y + i * 8;
    bool ok = true;
    for (int k = 0; k < 8; ++k) ok = ok && isfinite(yi[k]);
    const float qn = sqrtf(yi[3] * yi[3] + yi[4] * yi[4] + yi[5] * yi[5] + yi[6] * yi[6]);
    ok = ok && qn > 1e-12f;
    if (ok) {
        const float ql[4] = {yi[3] / qn, yi[4] / qn, yi[5] / qn, yi[6] / qn};
        float qb[4] = {pca.quats[i], pca.quats[n + i], pca.quats[2 * n + i], pca.quats[3 * n + i]};
        const float bn = sqrtf(qb[0] * qb[0] + qb[1] * qb[1] + qb[2] * qb[2] + qb[3] * qb[3]);
        for (int k = 0; k < 4; ++k) qb[k] /= bn;
        float q[4];
        qmul(qb, ql, q);
        for (int k = 0; k < 3; ++k) out.log_scales[k * n + i] = pca.log_scales[k * n + i] + yi[k];
        for (int k = 0; k < 4; ++k) out.quats[k * n + i] = q[k];
        out.opacity_logits[i] = pca.opacity_logits[i] + yi[7];
    } else {
        for (int k = 0; k < 3; ++k) out.log_scales[k * n + i] = pca.log_scales[k * n + i];
        for (int k = 0; k < 4; ++k) out.quats[k * n + i] = pca.quats[k * n + i];
        out.opacity_logits[i] = pca.opacity_logits[i];
        atomicAdd(fallbacks, 1u);
    }
}

// Training targets [n][8] of converged Gaussians relative to the paper's initializer `pca` of the
// same point: log-scale differences, conj(normalise(pca q)) (x) normalise(q), logit difference.
__global__ void k_make_targets(int64_t n, pgs_gaussians pca, pgs_gaussians conv, float* __restrict__ t) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    float q[4] = {conv.quats[i], conv.quats[n + i], conv.quats[2 * n + i], conv.quats[3 * n + i]};
    const float qn = sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    for (int k = 0; k < 4; ++k) q[k] /= qn;
    float qb[4] = {pca.quats[i], pca.quats[n + i], pca.quats[2 * n + i], pca.quats[3 * n + i]};
    const float bn = sqrtf(qb[0] * qb[0] + qb[1] * qb[1] + qb[2] * qb[2] + qb[3] * qb[3]);
    const float qc[4] = {qb[0] / bn, -qb[1] / bn, -qb[2] / bn, -qb[3] / bn};
    float ql[4];
    qmul(qc, q, ql);
    for (int k = 0; k < 3; ++k) t[i * 8 + k] = conv.log_scales[k * n + i] - pca.log_scales[k * n + i];
    for (int k = 0; k < 4; ++k) t[i * 8 + 3 + k] = ql[k];
    t[i * 8 + 7] = conv.opacity_logits[i] - pca.opacity_logits[i];
}

}  // namespace

int launch_apply_mlp(int64_t n, const float* y, const pgs_gaussians& pca, pgs_gaussians& out,
                     uint32_t* fallbacks, cudaStream_t s) {
    if (n <= 0) return 0;
    k_apply_mlp<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, y, pca, out, fallbacks);
    return 1;
}

int launch_make_targets(int64_t n, const pgs_gaussians& pca, const pgs_gaussians& conv, float* t,
                        cudaStream_t s) {
    if (n <= 0) return 0;
    k_make_targets<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, pca, conv, t);
    return 1;
}

// Scratch of the kNN for n points and at most `cells` cells: the cell-ordered points, the cell of each
// point, counts / cursors and starts of the cells, the scan's run totals, the CTAs' boxes, the grid.
namespace {
struct KnnScratch {
    float4* Ps;
    uint32_t *cell_of, *counts, *start, *totals;
    float* part;
    Grid* grid;
    size_t bytes;
};
KnnScratch knn_carve(char* base, int64_t n, int64_t cells) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base + off;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    KnnScratch k;
    k.Ps = reinterpret_cast<float4*>(take(16 * (size_t)n));
    k.cell_of = reinterpret_cast<uint32_t*>(take(4 * (size_t)n));
    k.counts = reinterpret_cast<uint32_t*>(take(4 * (size_t)cells));
    k.start = reinterpret_cast<uint32_t*>(take(4 * (size_t)(cells + 1)));
    k.totals = reinterpret_cast<uint32_t*>(take(4 * (size_t)((cells + kScanRun - 1) / kScanRun)));
    k.part = reinterpret_cast<float*>(take(4 * 6 * kBoxCtas));
    k.grid = reinterpret_cast<Grid*>(take(sizeof(Grid)));
    k.bytes = off;
    return k;
}
}  // namespace

int64_t knn_max_cells(int64_t n) { return std::min<int64_t>(4 * n + 1024, int64_t(1) << 30); }
size_t knn_scratch_bytes(int64_t n) { return knn_carve(nullptr, n, knn_max_cells(n)).bytes; }

// tickets: two zeroed words, zero again afterwards
int launch_knn(int64_t n, const float* P, int k, int32_t* nb, void* scratch, uint32_t* tickets, cudaStream_t s) {
    if (n <= 0) return 0;
    const int64_t cells = knn_max_cells(n);
    const KnnScratch w = knn_carve(static_cast<char*>(scratch), n, cells);
    cudaMemsetAsync(w.counts, 0, 4 * (size_t)cells, s);
    const unsigned blocks = (unsigned)((n + kThreads - 1) / kThreads);
    const unsigned scans = (unsigned)((cells + kScanRun - 1) / kScanRun);
    k_bbox<<<std::min(blocks, (unsigned)kBoxCtas), kThreads, 0, s>>>(n, P, w.part, tickets, cells, w.grid);
    k_cell_count<<<blocks, kThreads, 0, s>>>(n, P, w.grid, w.cell_of, w.counts);
    k_scan_totals<<<scans, kThreads, 0, s>>>(w.grid, w.counts, w.totals, tickets + 1);
    k_scan_cells<<<scans, kThreads, 0, s>>>(n, w.grid, w.counts, w.totals, w.start);
    k_cell_scatter<<<blocks, kThreads, 0, s>>>(n, P, w.cell_of, w.counts, w.Ps);
    const unsigned qb = (unsigned)((n + kQueryWarps - 1) / kQueryWarps);
    switch (k) {
        case 3: k_knn_query<3><<<qb, 32 * kQueryWarps, 0, s>>>(n, w.grid, w.start, w.Ps, nb); break;
        case 16: k_knn_query<16><<<qb, 32 * kQueryWarps, 0, s>>>(n, w.grid, w.start, w.Ps, nb); break;
        default: k_knn_query<32><<<qb, 32 * kQueryWarps, 0, s>>>(n, w.grid, w.start, w.Ps, nb); break;
    }
    return 6;
}

int launch_features_init(int64_t n, const float* P, const int32_t* nb, float r_normal, float* feats,
                         void* feats_bf16, float* frame_q, pgs_gaussians& init, cudaStream_t s) {
    if (n <= 0) return 0;
    k_features_init<<<(unsigned)((n + 32 * kFeatWarps - 1) / (32 * kFeatWarps)), 32 * kFeatWarps, 0, s>>>(
        n, P, nb, r_normal, feats, static_cast<__nv_bfloat16*>(feats_bf16), frame_q, init);
    return 1;
}

}  // namespace pgs
