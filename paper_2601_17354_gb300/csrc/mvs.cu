// Single-reference cost-volume MVS of the geometry prior (Sec. III-A): depth range from the
// projected sparse points ([0.5 q.05, 1.5 q.95]), reference keyframe by Eq. 4, census matching
// cost over a fronto-parallel plane sweep, SGM aggregation, confidence filter (0.4), fusion.
//
// Readings (the paper names the ingredients; the rest is fixed here):
//   luma Y = 0.299 R + 0.587 G + 0.114 B; census over a 7 x 7 window, 48 bits in raster order of
//   the neighbours (centre skipped), set when the neighbour is darker, outside neighbours clear;
//   D planes uniform in inverse depth, plane 0 the farthest; plane map H_k = K_r (R + t e3^T / d_k)
//   K_t^-1 built in FP64 in a fixed order, rounded to FP32, applied to pixel centres in FP32
//   (products and sums rounded separately, IEEE division: the reference pixel is an integer
//   decided in floating point, so the order is part of the definition); cost = Hamming distance,
//   24 when the point is behind the reference or outside it; SGM over 4 paths with P1 = 8,
//   P2 = 32 in integers; winner-take-all with S2 the best cost two or more planes away, kept when
//   the minimum is interior and 5 (S2 - S1) >= 2 S2 (confidence 1 - S1 / S2 >= 0.4); parabola
//   refinement in inverse depth; kept pixels back-projected in FP64.
//
// Layout: census codes [H][W] u64; cost C [H][W][D] u8, the four paths' L [4][H][W][D] u8 and the
// aggregated cost S [H][W][D] u16, the plane index innermost so a pixel's costs are one contiguous
// run for every path direction.
#include <cmath>

#include "pgs_internal.cuh"

namespace pgs {
namespace {

constexpr int kR = 3;                    // census radius
constexpr int kInvalid = 24;
constexpr int kP1 = 8, kP2 = 32;
constexpr int kCtx = 32, kCty = 8;       // census tile
constexpr int kRun = 32;                 // pixels per cost-volume CTA

__device__ __forceinline__ float luma(float r, float g, float b) {
    return __fadd_rn(__fadd_rn(__fmul_rn(0.299f, r), __fmul_rn(0.587f, g)), __fmul_rn(0.114f, b));
}

__device__ void census_tile(const float* __restrict__ rgb, int W, int H, uint64_t* __restrict__ code) {
    __shared__ float s[kCty + 2 * kR][kCtx + 2 * kR];
    const int x0 = blockIdx.x * kCtx, y0 = blockIdx.y * kCty;
    const size_t plane = (size_t)W * H;
    for (int k = threadIdx.y * kCtx + threadIdx.x; k < (kCty + 2 * kR) * (kCtx + 2 * kR); k += kCtx * kCty) {
        const int r = k / (kCtx + 2 * kR), c = k % (kCtx + 2 * kR);
        const int y = y0 - kR + r, x = x0 - kR + c;
        float v = __int_as_float(0x7f800000);  // outside: +inf, never darker
        if (x >= 0 && x < W && y >= 0 && y < H) {
            const size_t p = (size_t)y * W + x;
            v = luma(rgb[p], rgb[plane + p], rgb[2 * plane + p]);
        }
        s[r][c] = v;
    }
    __syncthreads();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    if (x >= W || y >= H) return;
    const float ctr = s[threadIdx.y + kR][threadIdx.x + kR];
    uint64_t out = 0;
    int bit = 0;
#pragma unroll
    for (int dy = -kR; dy <= kR; ++dy)
#pragma unroll
        for (int dx = -kR; dx <= kR; ++dx) {
            if (dy == 0 && dx == 0) continue;
            out |= (uint64_t)(s[threadIdx.y + kR + dy][threadIdx.x + kR + dx] < ctr) << bit;
            ++bit;
        }
    code[(size_t)y * W + x] = out;
}

struct CamF {
    float fx, fy, cx, cy;
    float v[12];
};

CamF camf(const pgs_camera& c) {
    CamF o;
    o.fx = c.fx;
    o.fy = c.fy;
    o.cx = c.cx;
    o.cy = c.cy;
    for (int i = 0; i < 12; ++i) o.v[i] = c.viewmat[i];
    return o;
}

__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dadd_rn(a, -b); }
__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double ddiv(double a, double b) { return __ddiv_rn(a, b); }

// plane map H_k (FP64 in the order of the definition, rounded to FP32)
__device__ void plane_map(const CamF& t, const CamF& r, double inv_far, double step, int k, float* __restrict__ maps) {
    double Rt[3][3], tt[3], Rr[3][3], tr[3];
    for (int i = 0; i < 3; ++i) {
        for (int j = 0; j < 3; ++j) {
            Rt[i][j] = t.v[4 * i + j];
            Rr[i][j] = r.v[4 * i + j];
        }
        tt[i] = t.v[4 * i + 3];
        tr[i] = r.v[4 * i + 3];
    }
    double R[3][3], tv[3];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            R[i][j] = dadd(dadd(dmul(Rr[i][0], Rt[j][0]), dmul(Rr[i][1], Rt[j][1])), dmul(Rr[i][2], Rt[j][2]));
    for (int i = 0; i < 3; ++i)
        tv[i] = dsub(tr[i], dadd(dadd(dmul(R[i][0], tt[0]), dmul(R[i][1], tt[1])), dmul(R[i][2], tt[2])));
    const double fxt = t.fx, fyt = t.fy, cxt = t.cx, cyt = t.cy;
    const double fxr = r.fx, fyr = r.fy, cxr = r.cx, cyr = r.cy;
    const double ax = ddiv(cxt, fxt), ay = ddiv(cyt, fyt);
    const double inv = dadd(inv_far, dmul((double)k, step));
    double g[3][3];
    for (int i = 0; i < 3; ++i) {
        const double m0 = R[i][0], m1 = R[i][1], m2 = dadd(R[i][2], dmul(tv[i], inv));
        g[i][0] = ddiv(m0, fxt);
        g[i][1] = ddiv(m1, fyt);
        g[i][2] = dsub(dsub(m2, dmul(m0, ax)), dmul(m1, ay));
    }
    float* h = maps + 9 * k;
    for (int j = 0; j < 3; ++j) {
        h[j] = __double2float_rn(dadd(dmul(fxr, g[0][j]), dmul(cxr, g[2][j])));
        h[3 + j] = __double2float_rn(dadd(dmul(fyr, g[1][j]), dmul(cyr, g[2][j])));
        h[6 + j] = __double2float_rn(g[2][j]);
    }
}

// Census codes of both images (blockIdx.z = 0 target, 1 reference) and, in the first CTA's row of a third
// layer, the plane maps, a thread per plane: they wait for nothing, so they take no launch of their own.
__global__ void __launch_bounds__(kCtx * kCty)
k_census(const float* __restrict__ rgb_t, const float* __restrict__ rgb_r, int W, int H, uint64_t* __restrict__ code_t,
         uint64_t* __restrict__ code_r, CamF t, CamF r, double inv_far, double step, int D, float* __restrict__ maps) {
    if (blockIdx.z == 2) {
        const int k = threadIdx.y * kCtx + threadIdx.x;
        if (blockIdx.x == 0 && blockIdx.y == 0 && k < D) plane_map(t, r, inv_far, step, k, maps);
        return;
    }
    census_tile(blockIdx.z ? rgb_r : rgb_t, W, H, blockIdx.z ? code_r : code_t);
}

// The integer nearest q - 1/2, which is floor(q) unless an integer lies within the margin (then `sure` turns
// false): rounding by adding 1.5 2^23, since conversions run at an eighth of the rate.
__device__ __forceinline__ int floor_fast(float q, bool& sure) {
    const float m = __fadd_rn(q, -0.5f), t = __fadd_rn(m, 12582912.0f);
    const float d = __fadd_rn(m, -__fadd_rn(t, -12582912.0f));
    // (the margin is used up from |q| = 499,998 on, and by NaN; below that the sums are exact to the rounding the
    // margin allows for, 1.5 2^23 holding integers to 2^22)
    sure = sure && fabsf(d) < __fmaf_rn(fabsf(q), -1e-6f, 0.499998f);
    return __float_as_int(t) - 0x4b400000;
}

// Cost volume: CTA = D threads (thread k = plane k, its map in registers) over a run of pixels.  Bound by
// instruction issue.  The reference pixel is the floor of a correctly rounded quotient; the
// quotient by the approximate reciprocal is within 4e-7 of itself of that, so only where an integer
// lies nearer do the divisions decide (a warp in thirty or so).  14.7 M pixels and planes: 43 us with both
// divisions always, 34 us now.
__global__ void k_cost(const uint64_t* __restrict__ cen_t, const uint64_t* __restrict__ cen_r, int W, int H,
                       int D, const float* __restrict__ maps, uint8_t* __restrict__ C) {
    const int k = threadIdx.x;
    const int y = blockIdx.y, xs = blockIdx.x * kRun, xe = min(xs + kRun, W);
    float h[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) h[q] = maps[9 * k + q];
    const float yc = (float)y + 0.5f;
    const float hy[3] = {__fmul_rn(h[1], yc), __fmul_rn(h[4], yc), __fmul_rn(h[7], yc)};
    const uint64_t* __restrict__ row = cen_t + (size_t)y * W;
    uint8_t* __restrict__ out = C + ((size_t)y * W + xs) * D + k;
    float xc = (float)xs + 0.5f;
#pragma unroll 2
    for (int x = xs; x < xe; ++x, xc += 1.0f, out += D) {
        const float a = __fadd_rn(__fadd_rn(__fmul_rn(h[0], xc), hy[0]), h[2]);
        const float b = __fadd_rn(__fadd_rn(__fmul_rn(h[3], xc), hy[1]), h[5]);
        const float c = __fadd_rn(__fadd_rn(__fmul_rn(h[6], xc), hy[2]), h[8]);
        int cost = kInvalid;
        if (c > 0.f) {
            float rc;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rc) : "f"(c));
            bool sure = c > 1e-30f && c < 1e30f;
            int iu = floor_fast(__fmul_rn(a, rc), sure), iv = floor_fast(__fmul_rn(b, rc), sure);
            if (!sure) {
                const float u = __fdiv_rn(a, c), v = __fdiv_rn(b, c);
                const bool in = u >= 0.f && u < (float)W && v >= 0.f && v < (float)H;
                iu = in ? (int)floorf(u) : -1;
                iv = in ? (int)floorf(v) : -1;
            }
            if ((unsigned)iu < (unsigned)W && (unsigned)iv < (unsigned)H)
                cost = __popcll(__ldg(row + x) ^ __ldg(cen_r + (iv * W + iu)));  // W H <= 2^28
        }
        *out = (uint8_t)cost;
    }
}

// A lane's KPL consecutive bytes of a pixel's D costs, as one word: one access when D is a multiple of
// KPL (then every lane's bytes are aligned to themselves, and lanes past D read nothing).
template <int KPL, bool kVec>
__device__ __forceinline__ uint32_t load_bytes(const uint8_t* __restrict__ p, int k0, int D) {
    if constexpr (kVec) {
        if (k0 >= D) return 0u;
        if constexpr (KPL == 1) return __ldg(p);
        if constexpr (KPL == 2) return __ldg(reinterpret_cast<const uint16_t*>(p));
        if constexpr (KPL == 4) return __ldg(reinterpret_cast<const uint32_t*>(p));
    }
    uint32_t v = 0;
#pragma unroll
    for (int j = 0; j < KPL; ++j)
        if (k0 + j < D) v |= (uint32_t)__ldg(p + j) << (8 * j);
    return v;
}
template <int KPL, bool kVec>
__device__ __forceinline__ void store_bytes(uint8_t* __restrict__ p, int k0, int D, uint32_t v) {
    if constexpr (kVec) {
        if (k0 >= D) return;
        if constexpr (KPL == 1) *p = (uint8_t)v;
        if constexpr (KPL == 2) *reinterpret_cast<uint16_t*>(p) = (uint16_t)v;
        if constexpr (KPL == 4) *reinterpret_cast<uint32_t*>(p) = v;
        return;
    }
#pragma unroll
    for (int j = 0; j < KPL; ++j)
        if (k0 + j < D) p[j] = (uint8_t)(v >> (8 * j));
}

// the four SGM paths in one launch (blockIdx.y = direction: 0 left to right, 1 right to left,
// 2 top down, 3 bottom up), warp per scanline, lane holding planes lane * KPL .. + KPL - 1; each
// path writes its own L (<= 48 + P2 = 80, a byte) so the directions run concurrently.  The walk along a
// line is serial: a step waits for the warp's minimum and two shuffles.  The costs of kBatch steps are loaded
// together while the batch before them is walked, and waited for once (loads issued step by step, 4 or 16
// ahead, share the few load counters, and the walk met the L2's latency at most steps: 182 and 158 us at
// 640 x 360 x 64, 73 us now).
constexpr int kSgmThreads = 64;
template <int KPL, bool kVec>
__global__ void __launch_bounds__(kSgmThreads)
k_sgm(const uint8_t* __restrict__ C, uint8_t* __restrict__ Lall, int W, int H, int D) {
    const int dir = blockIdx.y;
    const int line = (blockIdx.x * kSgmThreads + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const bool horiz = dir < 2;
    const int lines = horiz ? H : W, len = horiz ? W : H;
    if (line >= lines) return;
    constexpr int kBig = 1 << 20, kBatch = 16;
    const int k0 = lane * KPL;
    // offset of step s: first + s stride
    const int64_t along = horiz ? (int64_t)D : (int64_t)W * D, across = horiz ? (int64_t)W * D : (int64_t)D;
    const bool forward = dir == 0 || dir == 2;
    const int64_t stride = forward ? along : -along;
    const int64_t first = line * across + (forward ? 0 : (len - 1) * along) + k0;
    const uint8_t* pc = C + first;
    uint8_t* pl = Lall + (size_t)dir * W * H * D + first;
    uint32_t next[kBatch];
    auto fetch = [&](int s0) {  // the costs of steps s0 .. s0 + kBatch - 1
#pragma unroll
        for (int a = 0; a < kBatch; ++a) {
            next[a] = s0 + a < len ? load_bytes<KPL, kVec>(pc, k0, D) : 0u;
            pc += stride;
        }
    };
    fetch(0);
    int L[KPL];
    for (int s0 = 0; s0 < len; s0 += kBatch) {
        uint32_t cur[kBatch];
#pragma unroll
        for (int a = 0; a < kBatch; ++a) cur[a] = next[a];
        fetch(s0 + kBatch);
#pragma unroll
        for (int a = 0; a < kBatch; ++a) {
            const int s = s0 + a;
            if (s >= len) break;
            const uint32_t cw = cur[a];
            if (s == 0) {
#pragma unroll
                for (int j = 0; j < KPL; ++j) L[j] = k0 + j < D ? (int)((cw >> (8 * j)) & 255u) : kBig;
            } else {
                int mloc = L[0];
#pragma unroll
                for (int j = 1; j < KPL; ++j) mloc = min(mloc, L[j]);
                const int m = __reduce_min_sync(0xffffffffu, mloc);
                const int below = __shfl_up_sync(0xffffffffu, L[KPL - 1], 1);   // plane lane*KPL - 1
                const int above = __shfl_down_sync(0xffffffffu, L[0], 1);       // plane lane*KPL + KPL
                int nl[KPL];
#pragma unroll
                for (int j = 0; j < KPL; ++j) {
                    const int lm = j > 0 ? L[j - 1] : (lane > 0 ? below : kBig);
                    const int lp = j < KPL - 1 ? L[j + 1] : (lane < 31 ? above : kBig);
                    const int best = min(min(L[j], min(lm, lp) + kP1), m + kP2);
                    nl[j] = k0 + j < D ? (int)((cw >> (8 * j)) & 255u) + best - m : kBig;
                }
#pragma unroll
                for (int j = 0; j < KPL; ++j) L[j] = nl[j];
            }
            uint32_t out = 0;
#pragma unroll
            for (int j = 0; j < KPL; ++j) out |= (uint32_t)L[j] << (8 * j);
            store_bytes<KPL, kVec>(pl, k0, D, out);
            pl += stride;
        }
    }
}

// S = the sum of the four paths (written out), winner-take-all, confidence, parabola refinement;
// depth (NaN where not kept) and kept flags.  A warp takes 32 consecutive pixels, four at a time (their
// loads and warp reductions overlap): for each, lanes over the planes (as in the SGM walk: coalesced
// loads and stores) find the minimiser and its value in one reduction of value << 8 | plane, then S2 and
// the neighbours, and leave them with lane i for pixel i; then every lane refines its own pixel, so the
// FP64 refinement runs on full warps (GB300's FP64 pipe costs a warp instruction the same with one lane
// or thirty-two).  One pixel at a time, byte by byte, five reductions each: 66 us at 640 x 360 x 64, 39 us now.
constexpr int kSelectThreads = 256;

template <int KPL, bool kVec>
__global__ void __launch_bounds__(kSelectThreads)
k_select(const uint8_t* __restrict__ Lall, uint16_t* __restrict__ S, int W, int H, int D, double inv_far,
         double step, float* __restrict__ depth, uint8_t* __restrict__ kept, unsigned long long* __restrict__ count) {
    __shared__ int s_count;
    if (threadIdx.x == 0) s_count = 0;
    __syncthreads();
    constexpr int kPix = 4;
    constexpr uint32_t kBig = 1u << 30;
    const int lane = threadIdx.x & 31, k0 = lane * KPL;
    const int64_t n = (int64_t)W * H;
    const size_t plane = (size_t)n * D;
    const int64_t chunks = (n + 31) / 32, warps = (int64_t)gridDim.x * (kSelectThreads / 32);
    for (int64_t ch = (int64_t)blockIdx.x * (kSelectThreads / 32) + (threadIdx.x >> 5); ch < chunks; ch += warps) {
        int my_k1 = 0, my_s1 = 0, my_s2 = 0, my_sm = 0, my_sp = 0;
        for (int i0 = 0; i0 < 32 && ch * 32 + i0 < n; i0 += kPix) {  // warp-uniform
            uint32_t v[kPix][KPL];
#pragma unroll
            for (int u = 0; u < kPix; ++u) {
                const int64_t p = ch * 32 + i0 + u;
#pragma unroll
                for (int j = 0; j < KPL; ++j) v[u][j] = 0u;
                if (p < n) {
                    const size_t at = (size_t)p * D + k0;
#pragma unroll
                    for (int d = 0; d < 4; ++d) {
                        const uint32_t w = load_bytes<KPL, kVec>(Lall + d * plane + at, k0, D);
#pragma unroll
                        for (int j = 0; j < KPL; ++j) v[u][j] += (w >> (8 * j)) & 255u;
                    }
                    if constexpr (KPL == 2 && kVec) {
                        if (k0 < D) *reinterpret_cast<uint32_t*>(S + at) = v[u][0] | v[u][1] << 16;
                    } else {
#pragma unroll
                        for (int j = 0; j < KPL; ++j)
                            if (k0 + j < D) S[at + j] = (uint16_t)v[u][j];
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kPix; ++u) {
                uint32_t key = 0xffffffffu;
#pragma unroll
                for (int j = 0; j < KPL; ++j)
                    if (k0 + j < D) key = min(key, v[u][j] << 8 | (uint32_t)(k0 + j));
                key = __reduce_min_sync(0xffffffffu, key);  // the first minimiser and its value
                const int k1 = (int)(key & 255u);
                uint32_t far = kBig, below = 0, above = 0;  // values of planes k1 - 1 and k1 + 1, in their lanes
#pragma unroll
                for (int j = 0; j < KPL; ++j) {
                    const int k = k0 + j;
                    if (k < D && abs(k - k1) >= 2) far = min(far, v[u][j]);
                    if (j == ((k1 - 1) & 0xffff) % KPL) below = v[u][j];
                    if (j == (k1 + 1) % KPL) above = v[u][j];
                }
                const uint32_t s2 = __reduce_min_sync(0xffffffffu, far);
                const int sm = (int)__shfl_sync(0xffffffffu, below, max(k1 - 1, 0) / KPL);
                const int sp = (int)__shfl_sync(0xffffffffu, above, (k1 + 1) / KPL);
                if (lane == i0 + u) {
                    my_k1 = k1;
                    my_s1 = (int)(key >> 8);
                    my_s2 = s2 == kBig ? my_s1 : (int)s2;
                    my_sm = sm;  // (k1 on the first or last plane is not kept)
                    my_sp = sp;
                }
            }
        }
        const int64_t p = ch * 32 + lane;
        const bool live = p < n;
        const bool keep =
            live && my_k1 > 0 && my_k1 < D - 1 && my_s2 > 0 && 5 * (my_s2 - my_s1) >= 2 * my_s2;
        float out = __int_as_float(0x7fc00000);
        if (keep) {
            const int den = my_sm - 2 * my_s1 + my_sp;
            const float delta = den > 0 ? __fdiv_rn((float)(my_sm - my_sp), __fmul_rn(2.f, (float)den)) : 0.f;
            const double inv = dadd(inv_far, dmul(dadd((double)my_k1, (double)delta), step));
            out = __double2float_rn(ddiv(1.0, inv));
        }
        if (live) {
            depth[p] = out;
            kept[p] = keep ? 1 : 0;
        }
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0 && bal) atomicAdd(&s_count, __popc(bal));
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_count) atomicAdd(count, (unsigned long long)s_count);
}

// kept-pixel counts per CTA (pixel order) and, on the side, the FP64 ray slopes ((i + 0.5) - c) / f of every
// column and row (ray [W + H]); then an exclusive scan in one CTA, then the points.  The points are bound by the
// FP64 pipe: with the two divisions per pixel instead of per column and row they took 30 us at 640 x 360, 19 us now.
constexpr int kFuseThreads = 256;

__global__ void __launch_bounds__(kFuseThreads)
k_fuse_count(const float* __restrict__ depth, int W, int H, CamF cam, uint32_t* __restrict__ cta_count,
             double* __restrict__ ray) {
    const int64_t n = (int64_t)W * H, p = (int64_t)blockIdx.x * kFuseThreads + threadIdx.x;
    for (int64_t i = p; i < W + H; i += (int64_t)gridDim.x * kFuseThreads)
        ray[i] = i < W ? ddiv(dsub((double)i + 0.5, (double)cam.cx), (double)cam.fx)
                       : ddiv(dsub((double)(i - W) + 0.5, (double)cam.cy), (double)cam.fy);
    const bool keep = p < n && depth[p] == depth[p];
    const int c = __syncthreads_count(keep);
    if (threadIdx.x == 0) cta_count[blockIdx.x] = (uint32_t)c;
}

__global__ void __launch_bounds__(1024)
k_fuse_scan(uint32_t* __restrict__ cta_count, int ctas, int64_t* __restrict__ total) {
    __shared__ uint32_t s_warp[32];
    __shared__ uint64_t s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < ctas; base += 1024) {
        const int i = base + threadIdx.x;
        const uint32_t v = i < ctas ? cta_count[i] : 0u;
        uint32_t incl = v;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if ((threadIdx.x & 31) >= o) incl += u;
        }
        if ((threadIdx.x & 31) == 31) s_warp[threadIdx.x >> 5] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += s_warp[w];
        const uint64_t carry = s_carry;
        if (i < ctas) cta_count[i] = (uint32_t)(carry + before + incl - v);
        __syncthreads();
        if (threadIdx.x == 1023) s_carry = carry + before + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = (int64_t)s_carry;
}

__global__ void __launch_bounds__(kFuseThreads)
k_fuse_points(const float* __restrict__ depth, int W, int64_t n, CamF cam, const uint32_t* __restrict__ cta_off,
              const double* __restrict__ ray, int64_t capacity, float* __restrict__ points, int32_t* __restrict__ pix) {
    __shared__ uint32_t s_warp[kFuseThreads / 32];
    const int64_t p = (int64_t)blockIdx.x * kFuseThreads + threadIdx.x;
    const float d = p < n ? depth[p] : __int_as_float(0x7fc00000);
    const bool keep = d == d;
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_warp[warp] = __popc(bal);
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    if (!keep) return;
    const int64_t o = (int64_t)cta_off[blockIdx.x] + before + __popc(bal & ((1u << lane) - 1u));
    if (o >= capacity) return;
    const int y = (int)(p / W), x = (int)(p % W);
    const double dd = d;
    const double X0 = dsub(dmul(dd, ray[x]), (double)cam.v[3]);
    const double X1 = dsub(dmul(dd, ray[W + y]), (double)cam.v[7]);
    const double X2 = dsub(dd, (double)cam.v[11]);
    for (int j = 0; j < 3; ++j) {
        const double w =
            dadd(dadd(dmul((double)cam.v[j], X0), dmul((double)cam.v[4 + j], X1)), dmul((double)cam.v[8 + j], X2));
        points[3 * o + j] = __double2float_rn(w);
    }
    pix[o] = (int32_t)p;
}

// camera-z (FP64) of the sparse points in front of the target and inside its image, compacted
__global__ void k_sparse_depths(const float* __restrict__ P, int64_t n, CamF cam, int W, int H, double* __restrict__ z,
                                unsigned long long* __restrict__ count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double X = P[3 * i], Y = P[3 * i + 1], Z = P[3 * i + 2];
    double Xc[3];
    for (int r = 0; r < 3; ++r)
        Xc[r] = dadd(dadd(dadd(dmul((double)cam.v[4 * r], X), dmul((double)cam.v[4 * r + 1], Y)),
                          dmul((double)cam.v[4 * r + 2], Z)),
                     (double)cam.v[4 * r + 3]);
    const double zz = Xc[2];
    if (!(zz > 0.2)) return;
    const double u = dadd(dmul((double)cam.fx, ddiv(Xc[0], zz)), (double)cam.cx);
    const double v = dadd(dmul((double)cam.fy, ddiv(Xc[1], zz)), (double)cam.cy);
    if (!(u >= 0.0 && u < (double)W && v >= 0.0 && v < (double)H)) return;
    z[atomicAdd(count, 1ull)] = zz;
}

// One CTA: the order statistics of the quantiles 0.05, 0.5, 0.95 of z[0..m) by bucket selection on the FP64
// bit patterns (positive values order like their bits), all six ranks at once; out = (0.5 q.05, 1.5 q.95,
// q.5).  The interval from the values' own minimum to their maximum is counted in 2048 buckets; the few
// values of the ranks' buckets are listed and each rank's is the one with as many listed before it.
// Where a bucket holds many (equal or clustered values), its interval is cut into buckets again.  Eight
// 8-bit passes over the whole pattern put all values of a scene in a few bins: 162 us for 20k values
// even with a warp's equal bins counted together, 26 us now.
__global__ void __launch_bounds__(1024)
k_quantiles(const double* __restrict__ z, const unsigned long long* __restrict__ count, double* __restrict__ out,
            int* __restrict__ status) {
    constexpr int kQ = 6, kBits = 11, kBuckets = 1 << kBits, kList = 256;
    typedef unsigned long long u64;
    __shared__ unsigned s_hist[kBuckets];
    __shared__ u64 s_list[kList];
    __shared__ u64 s_lo[kQ], s_hi[kQ];  // rank q's value lies in [lo, hi]
    __shared__ int s_rank[kQ];          // and is that one of the interval's values, in order
    __shared__ int s_cut[kQ];           // round that last cut its interval
    __shared__ u64 s_min[32], s_max[32];
    __shared__ unsigned s_warp[32];
    __shared__ int s_listed;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long m = (long long)*count;
    if (m == 0) {
        if (threadIdx.x == 0) atomicOr(status, 1);
        return;
    }
    constexpr int kLoads = 8;  // values in flight per thread: a pass is a few memory latencies
    auto for_values = [&](auto&& f) {
        for (long long i0 = threadIdx.x; i0 < m; i0 += kLoads * 1024) {
            u64 b[kLoads];
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const long long i = i0 + u * 1024;
                b[u] = (u64)__double_as_longlong(z[i < m ? i : i0]);
            }
#pragma unroll
            for (int u = 0; u < kLoads; ++u)
                if (i0 + u * 1024 < m) f(b[u]);
        }
    };
    u64 lo = ~0ull, hi = 0ull;
    for_values([&](u64 b) {
        lo = min(lo, b);
        hi = max(hi, b);
    });
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
        s_min[warp] = lo;
        s_max[warp] = hi;
    }
    __syncthreads();
    const double ps[3] = {0.05, 0.5, 0.95};
    if (threadIdx.x < kQ) {
        for (int w = 0; w < 32; ++w) {
            lo = min(lo, s_min[w]);
            hi = max(hi, s_max[w]);
        }
        const double h = dmul((double)(m - 1), ps[threadIdx.x >> 1]);
        const long long r = (long long)floor(h);
        s_rank[threadIdx.x] = (int)((threadIdx.x & 1) ? (r + 1 < m ? r + 1 : m - 1) : r);
        s_lo[threadIdx.x] = lo;
        s_hi[threadIdx.x] = hi;
        s_cut[threadIdx.x] = 0;
    }
    __syncthreads();
    for (int round = 1;; ++round) {
        // list the values of the intervals that are not single values yet, unless they are too many
        if (round > 1 || m <= kList) {
            if (threadIdx.x == 0) s_listed = 0;
            __syncthreads();
            for_values([&](u64 b) {
                bool in = false;
#pragma unroll
                for (int e = 0; e < kQ; ++e) in = in || (b >= s_lo[e] && b <= s_hi[e] && s_lo[e] < s_hi[e]);
                if (in) {
                    const int at = atomicAdd(&s_listed, 1);
                    if (at < kList) s_list[at] = b;
                }
            });
            __syncthreads();
            if (s_listed <= kList) break;  // (0 when every rank's value is known)
        }
        // else cut each of these intervals into buckets and keep its ranks' (2^11 times narrower a round)
        for (int q = 0; q < kQ; ++q) {
            __syncthreads();
            const u64 l = s_lo[q], h = s_hi[q];
            const bool skip = l == h || s_cut[q] == round;  // the same for every thread
            __syncthreads();
            if (skip) continue;
            const int shift = max(0, 64 - __clzll((long long)(h - l)) - kBits);
            for (int e = threadIdx.x; e < kBuckets; e += 1024) s_hist[e] = 0u;
            __syncthreads();
            for_values([&](u64 b) {
                if (b >= l && b <= h) atomicAdd(&s_hist[(b - l) >> shift], 1u);
            });
            __syncthreads();
            // prefix of the counts, two buckets a thread
            const unsigned c0 = s_hist[2 * threadIdx.x], c1 = s_hist[2 * threadIdx.x + 1];
            unsigned incl = c0 + c1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) s_warp[warp] = incl;
            __syncthreads();
            unsigned first = incl - c0 - c1;
            for (int w = 0; w < warp; ++w) first += s_warp[w];
            unsigned mine = 0;  // the ranks of this interval that fall into the thread's buckets
            for (int e = q; e < kQ; ++e) {
                const unsigned r = (unsigned)s_rank[e];
                if (s_lo[e] == l && s_hi[e] == h && r >= first && r < first + c0 + c1) mine |= 1u << e;
            }
            __syncthreads();
            for (int e = q; e < kQ; ++e)
                if ((mine >> e) & 1u) {
                    const unsigned r = (unsigned)s_rank[e] - first, second = r >= c0 ? 1u : 0u;
                    const u64 start = l + ((u64)(2 * threadIdx.x + second) << shift);
                    s_rank[e] = (int)(r - (second ? c0 : 0u));
                    s_lo[e] = start;
                    s_hi[e] = min(h, start + ((1ull << shift) - 1));
                    s_cut[e] = round;
                }
        }
        __syncthreads();
    }
    __syncthreads();
    // the listed values: rank q's is the one with s_rank[q] of its interval's before it
    const int listed = min(s_listed, kList);
    if (threadIdx.x < listed) {
        const u64 x = s_list[threadIdx.x];
        for (int q = 0; q < kQ; ++q) {
            const u64 l = s_lo[q], h = s_hi[q];
            if (x < l || x > h || l == h) continue;
            int less = 0, same = 0;
            for (int k = 0; k < listed; ++k) {
                const u64 y = s_list[k];
                less += y >= l && y < x;
                same += y == x;
            }
            if (s_rank[q] >= less && s_rank[q] < less + same) s_min[q] = x;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double q[3];
        for (int j = 0; j < 3; ++j) {
            const double h = dmul((double)(m - 1), ps[j]);
            const double fl = floor(h);
            double v[2];
            for (int e = 0; e < 2; ++e) {
                const int k = 2 * j + e;
                v[e] = __longlong_as_double((long long)(s_lo[k] == s_hi[k] ? s_lo[k] : s_min[k]));
            }
            q[j] = dadd(v[0], dmul(dsub(h, fl), dsub(v[1], v[0])));
        }
        out[0] = dmul(0.5, q[0]);
        out[1] = dmul(1.5, q[2]);
        out[2] = q[1];
    }
}

// Eq. 4 score of every keyframe as the reference of `target`, and the best (ties: lowest index)
__global__ void __launch_bounds__(1024)
k_reference(const CamF* __restrict__ cams, int count, int target, double median, double* __restrict__ scores,
            int* __restrict__ best) {
    __shared__ double s_val[1024];
    __shared__ int s_idx[1024];
    const int j = threadIdx.x;
    auto centre = [&](const CamF& c, double o[3]) {
        for (int q = 0; q < 3; ++q)
            o[q] = -dadd(dadd(dmul((double)c.v[q], (double)c.v[3]), dmul((double)c.v[4 + q], (double)c.v[7])),
                         dmul((double)c.v[8 + q], (double)c.v[11]));
    };
    double sc = -INFINITY;
    if (j < count && j != target) {
        double ct[3], cj[3];
        centre(cams[target], ct);
        centre(cams[j], cj);
        const double dx = dsub(cj[0], ct[0]), dy = dsub(cj[1], ct[1]), dz = dsub(cj[2], ct[2]);
        const double b = sqrt(dadd(dadd(dmul(dx, dx), dmul(dy, dy)), dmul(dz, dz)));
        const CamF& A = cams[target];
        const CamF& B = cams[j];
        const double cosang = dadd(dadd(dmul((double)B.v[8], (double)A.v[8]), dmul((double)B.v[9], (double)A.v[9])),
                                   dmul((double)B.v[10], (double)A.v[10]));
        const double alpha = acos(fmax(-1.0, fmin(1.0, cosang)));
        const double bt = dmul(0.1, median), sb = dmul(0.5, bt);
        const double alpha_min = dmul(5.0, 0.017453292519943295);
        const double e = dsub(b, bt);
        sc = dmul(exp(ddiv(-dmul(e, e), dmul(dmul(2.0, sb), sb))), fmax(ddiv(alpha, alpha_min), 1.0));
    }
    if (j < count) scores[j] = sc;
    s_val[j] = sc;
    s_idx[j] = j;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if (j < w) {
            const double a = s_val[j], b2 = s_val[j + w];
            if (b2 > a || (b2 == a && s_idx[j + w] < s_idx[j])) {
                s_val[j] = b2;
                s_idx[j] = s_idx[j + w];
            }
        }
        __syncthreads();
    }
    if (j == 0) *best = s_idx[0];
}

unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

int launch_mvs_census(const pgs_camera& t, const pgs_camera& r, const float* rgb_t, const float* rgb_r, int W, int H, int D,
                      double inv_far, double step, uint64_t* code_t, uint64_t* code_r, float* maps, cudaStream_t s) {
    k_census<<<dim3(blocks(W, kCtx), blocks(H, kCty), 3), dim3(kCtx, kCty), 0, s>>>(rgb_t, rgb_r, W, H, code_t, code_r,
                                                                                   camf(t), camf(r), inv_far, step, D, maps);
    return 1;
}

int launch_mvs_cost(const uint64_t* cen_t, const uint64_t* cen_r, int W, int H, int D, const float* maps, uint8_t* C,
                    cudaStream_t s) {
    k_cost<<<dim3(blocks(W, kRun), H), D, 0, s>>>(cen_t, cen_r, W, H, D, maps, C);
    return 1;
}

// planes per lane for D planes: 1, 2, 3 or 4; one access for a lane's planes when they divide D
template <template <int, bool> class Launch, class... Args>
void by_planes(int D, Args... args) {
    if (D <= 32) Launch<1, true>::run(args...);
    else if (D <= 64) D % 2 == 0 ? Launch<2, true>::run(args...) : Launch<2, false>::run(args...);
    else if (D <= 96) Launch<3, false>::run(args...);
    else D % 4 == 0 ? Launch<4, true>::run(args...) : Launch<4, false>::run(args...);
}
template <int KPL, bool kVec>
struct SgmLaunch {
    static void run(const uint8_t* C, uint8_t* L, int W, int H, int D, cudaStream_t s) {
        const dim3 g(blocks((int64_t)(W > H ? W : H) * 32, kSgmThreads), 4);
        k_sgm<KPL, kVec><<<g, kSgmThreads, 0, s>>>(C, L, W, H, D);
    }
};
template <int KPL, bool kVec>
struct SelectLaunch {
    static void run(const uint8_t* L, uint16_t* S, int W, int H, int D, double inv_far, double step, float* depth,
                    uint8_t* kept, unsigned long long* count, cudaStream_t s) {
        const int64_t n = (int64_t)W * H;
        int64_t g = ((n + 31) / 32 + kSelectThreads / 32 - 1) / (kSelectThreads / 32);
        if (g > 152 * 8) g = 152 * 8;  // grid-stride: 8 resident CTAs an SM
        k_select<KPL, kVec><<<(unsigned)g, kSelectThreads, 0, s>>>(L, S, W, H, D, inv_far, step, depth, kept, count);
    }
};

int launch_mvs_sgm(const uint8_t* C, uint8_t* L, int W, int H, int D, cudaStream_t s) {
    by_planes<SgmLaunch>(D, C, L, W, H, D, s);
    return 1;
}

int launch_mvs_select(const uint8_t* L, uint16_t* S, int W, int H, int D, double inv_far, double step, float* depth,
                      uint8_t* kept, unsigned long long* count, cudaStream_t s) {
    cudaMemsetAsync(count, 0, sizeof(unsigned long long), s);
    by_planes<SelectLaunch>(D, L, S, W, H, D, inv_far, step, depth, kept, count, s);
    return 1;
}

int launch_mvs_fuse(const float* depth, int W, int H, const pgs_camera& cam, uint32_t* cta_scratch, double* ray,
                    int64_t* total, int64_t capacity, float* points, int32_t* pix, cudaStream_t s) {
    const int64_t n = (int64_t)W * H;
    const unsigned g = blocks(n, kFuseThreads);
    k_fuse_count<<<g, kFuseThreads, 0, s>>>(depth, W, H, camf(cam), cta_scratch, ray);
    k_fuse_scan<<<1, 1024, 0, s>>>(cta_scratch, (int)g, total);
    k_fuse_points<<<g, kFuseThreads, 0, s>>>(depth, W, n, camf(cam), cta_scratch, ray, capacity, points, pix);
    return 3;
}

int mvs_fuse_ctas(int W, int H) { return (int)blocks((int64_t)W * H, kFuseThreads); }

int launch_mvs_range(const float* P, int64_t n, const pgs_camera& cam, double* zbuf, unsigned long long* count,
                     double* out, int* status, cudaStream_t s) {
    cudaMemsetAsync(count, 0, sizeof(unsigned long long), s);
    if (n > 0)
        k_sparse_depths<<<blocks(n, 256), 256, 0, s>>>(P, n, camf(cam), cam.width, cam.height, zbuf, count);
    k_quantiles<<<1, 1024, 0, s>>>(zbuf, count, out, status);
    return n > 0 ? 2 : 1;
}

int launch_mvs_reference(const void* cams_f, int count, int target, double median, double* scores, int* best,
                         cudaStream_t s) {
    k_reference<<<1, 1024, 0, s>>>(static_cast<const CamF*>(cams_f), count, target, median, scores, best);
    return 1;
}

size_t mvs_camf_bytes() { return sizeof(CamF); }

void mvs_pack_cameras(const pgs_camera* cams, int count, void* host_out) {
    CamF* o = static_cast<CamF*>(host_out);
    for (int i = 0; i < count; ++i) o[i] = camf(cams[i]);
}

}  // namespace pgs
