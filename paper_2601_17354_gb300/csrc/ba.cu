// Bundle adjustment of the geometry prior (Sec. III-A): Levenberg-Marquardt on the robust
// reprojection objective of Eq. 2, each step solved through the reduced camera system of Eq. 3.
//
//   camera i: world-to-camera R_i (row-major 3 x 3), t_i; point P_j; pinhole (fx, fy, cx, cy);
//   r = pi(R_i P_j + t_i) - p_ij, whitened by sigma; Huber weight w = 1 (e <= delta) or delta / e
//   on the whitened norm e; camera update R <- exp([omega]x) R, t <- t + v; point update P <- P + d;
//   gauge: camera 0 fixed, and camera 1's translation component along the axis of its largest
//   initial baseline component (in its own frame) fixed.
//
// Observations are grouped by point with cameras increasing inside a group; every point carries a
// bit mask of the cameras that see it (the observation of camera a at point j is start[j] + the
// mask bits below a), and every camera a list of its observations in point order.  No kernel adds
// floating point with atomics except the scalar cost; every block of the normal equations has one
// owner:
//   linearize  8 lanes per point, a lane per observation: residual in two floats (pixel coordinates
//              ~1e3, residuals ~1), Jacobians (FP32), H_pp and b_p (two floats), H_tp of every
//              observation (6 x 3, FP32), robust cost;
//   camblocks  CTA per (camera, chunk of its observations): H_tt block (21) and b_t (6), Jacobians
//              recomputed from the state (cheaper than storing them);
//   points     thread per point, per trial: (H_pp + lam diag)^-1 in FP64, y = H_pp^-1 b_p (the
//              independent 3 x 3 inverses of Eq. 3);
//   schur      CTA per (camera a, chunk of its observations), a warp per second camera b >= a at a time:
//              sum over the points seen by both of H_tp,a H_pp^-1 H_tp,b^T (6 x 6) and, for a == b, of
//              H_tp,a y (the reduced rhs);
//   assemble   thread per entry: the damped reduced system from the chunk sums;
//   solve      one CTA: gauge and unobserved rows fixed, scaled to a unit diagonal (Jacobi; this takes its condition
//              number from ~1e8 to ~1e3 on ring-camera problems, so FP32 factorization keeps a
//              backward error ~1e-8 while GB300's FP64 rate is 1/64 of its FP32 rate), then
//              blocked Cholesky in shared memory (6C <= 224) or, for more cameras, symmetric
//              elimination of the packed upper triangle with the rhs carried along; candidate poses;
//   backsub    8 lanes per point: Delta_p = H_pp^-1 (b_p - sum H_tp^T Delta_t), the candidate point and
//              its share of the candidate's cost;
//   decide     one thread: takes the candidate when the robust cost drops (lam / 10) or keeps the
//              state and raises lam * 10 (the linearization is reused); the next linearize moves
//              the state.  A whole solve is enqueued without the host reading anything in between.
// With 32 cameras, 20k points and 124k observations an iteration took 0.45 ms: FP64 residuals on a
// thread per point (75 + 41 + 46 us), a 0.116 ms solve and a host decision between launches.  It takes
// 0.16 ms: linearize 15, camblocks 10, points 10, schur 34, assemble 9, solve 59, backsub 16, decide 3 us.
#include <cmath>

#include "df.cuh"
#include "pgs_internal.cuh"

namespace pgs {
namespace {

constexpr int kBaThreads = 256;
constexpr int kGroup = 8;  // lanes per point in linearize and backsub (a track holds 2-12 observations)
constexpr int kPointsPerCta = kBaThreads / kGroup;
constexpr int kSolveThreads = 1024;
constexpr int kBlockedThreads = 512;  // 128 registers a thread: the 32-float rows stay in registers
constexpr int kMaxN = 6 * 256;
constexpr int kMaxBlockedN = 224;
constexpr int kPanel = 16;  // columns per step of the blocked factorization
// shared memory of the blocked solve: NP rows and the rhs as one more, a row stride of NP + 4 (16-byte
// accesses of eight consecutive rows then fall in different banks), and the panel transposed
constexpr size_t blocked_smem(size_t NP) { return ((NP + 1) * (NP + 4) + kPanel * (NP + 4)) * sizeof(float); }
constexpr size_t kMaxPackedSmem = 200 * 1024;  // + 13 KB static: within the 227 KB a CTA may use
static_assert(blocked_smem(kMaxBlockedN) + 4 * 1024 <= 227 * 1024, "the largest blocked solve fits an SM");

struct Intr {
    float fx, fy, cx, cy;
};

// x = R_i P + t_i in double (the products of FP32 inputs are exact)
__device__ __forceinline__ void cam_point(const float* __restrict__ R, const float* __restrict__ t, int i,
                                          double px, double py, double pz, double X[3]) {
    const float* r = R + 9 * i;
    X[0] = fma((double)r[0], px, fma((double)r[1], py, fma((double)r[2], pz, (double)t[3 * i + 0])));
    X[1] = fma((double)r[3], px, fma((double)r[4], py, fma((double)r[5], pz, (double)t[3 * i + 1])));
    X[2] = fma((double)r[6], px, fma((double)r[7], py, fma((double)r[8], pz, (double)t[3 * i + 2])));
}

// noise and robust threshold in the forms the residual uses
struct Robust {
    Df inv_s2;  // 1 / sigma^2
    float inv_s2f, delta;
};

__device__ __forceinline__ Df df_mulf(Df a, float b) { return df_mul(a, {b, 0.0f}); }

// x = R_i P + t_i in two floats
__device__ __forceinline__ void cam_point_df(const float* __restrict__ R, const float* __restrict__ t, int i, float px,
                                             float py, float pz, Df X[3]) {
    const float* r = R + 9 * i;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Df v = {t[3 * i + a], 0.0f};
        df_dot(v, {r[3 * a], 0.0f}, {px, 0.0f});
        df_dot(v, {r[3 * a + 1], 0.0f}, {py, 0.0f});
        df_dot(v, {r[3 * a + 2], 0.0f}, {pz, 0.0f});
        X[a] = df_two(v.h, v.l);
    }
}

// residual, IRLS weight over sigma^2 and robust cost of one observation (two floats: the pixel
// coordinates are ~1e3 and the residuals ~1); false when behind the camera.  iz = 1 / z.
__device__ __forceinline__ bool residual(const Df X[3], Intr K, float u, float v, const Robust& rb, float r[2], float& iz,
                                         float& Wm, Df& rho) {
    if (!(X[2].h > 1e-6f)) return false;
    const Df z = df_recip(X[2]);
    const Df r0 = df_add(df_mulf(df_mul(X[0], z), K.fx), df_two(K.cx, -u));
    const Df r1 = df_add(df_mulf(df_mul(X[1], z), K.fy), df_two(K.cy, -v));
    const Df e2 = df_mul(df_add(df_mul(r0, r0), df_mul(r1, r1)), rb.inv_s2);
    r[0] = r0.h;
    r[1] = r1.h;
    iz = z.h;
    Wm = rb.inv_s2f;
    rho = e2;
    if (e2.h > rb.delta * rb.delta) {
        const Df e = df_sqrt(e2);
        Wm *= rb.delta / e.h;
        const float d2 = __fmul_rn(rb.delta, rb.delta);
        rho = df_sub(df_mulf(e, 2.0f * rb.delta), df_fast(d2, __fmaf_rn(rb.delta, rb.delta, -d2)));
    }
    return true;
}

// d pi / d(omega, v) and d pi / dP at camera-frame point X of camera i (FP32: their rounding is
// that of the stored H_tp)
__device__ __forceinline__ void jacobians(const float* __restrict__ R, const float* __restrict__ t, int i, const Df X[3],
                                          float iz, Intr K, float Jc[2][6], float Jp[2][3]) {
    const float x0 = X[0].h, x1 = X[1].h;
    // d pi / dx = [[a0, 0, a2], [0, b1, b2]]
    const float a0 = K.fx * iz, a2 = -K.fx * x0 * iz * iz;
    const float b1 = K.fy * iz, b2 = -K.fy * x1 * iz * iz;
    // q = R P = x - t; d x / d omega = -[q]x = [[0, q2, -q1], [-q2, 0, q0], [q1, -q0, 0]]
    const float q0 = df_add(X[0], {-t[3 * i], 0.f}).h, q1 = df_add(X[1], {-t[3 * i + 1], 0.f}).h,
                q2 = df_add(X[2], {-t[3 * i + 2], 0.f}).h;
    Jc[0][0] = a2 * q1;
    Jc[0][1] = a0 * q2 - a2 * q0;
    Jc[0][2] = -a0 * q1;
    Jc[0][3] = a0;
    Jc[0][4] = 0.f;
    Jc[0][5] = a2;
    Jc[1][0] = -b1 * q2 + b2 * q1;
    Jc[1][1] = -b2 * q0;
    Jc[1][2] = b1 * q0;
    Jc[1][3] = 0.f;
    Jc[1][4] = b1;
    Jc[1][5] = b2;
    const float* rr = R + 9 * i;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        Jp[0][c] = a0 * rr[c] + a2 * rr[6 + c];
        Jp[1][c] = b1 * rr[3 + c] + b2 * rr[6 + c];
    }
}

// over the kGroup lanes of a point (every lane ends with the sum); `lanes` = the warp's active mask
template <int kLanes>
__device__ __forceinline__ void df_lanes_sum(Df& s) {
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1) {
        const Df v = {__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.l, o)};
        df_acc(s, v);
    }
    s = df_two(s.h, s.l);
}
// the CTA's sum of every thread's s, added to *dst (every thread calls it)
__device__ __forceinline__ void cta_add(Df s, double* dst) {
    __shared__ double s_red[kBaThreads / 32];
    df_lanes_sum<32>(s);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = df_double(s);
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kBaThreads / 32; ++w) t += s_red[w];
        atomicAdd(dst, t);
    }
}

// sum of v over the CTA (kBaThreads) in FP32 (FP64 adds run at 1/64 of the FP32 rate here):
// returns the sum of element t in thread t < kN
template <int kN>
__device__ __forceinline__ float block_sum(float (&v)[kN], float (*s_red)[kN]) {
#pragma unroll
    for (int q = 0; q < kN; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int q = 0; q < kN; ++q) s_red[threadIdx.x >> 5][q] = v[q];
    __syncthreads();
    float t = 0.f;
    if (threadIdx.x < kN)
        for (int w = 0; w < kBaThreads / 32; ++w) t += s_red[w][threadIdx.x];
    return t;
}

// observation indices in range, grouped by point, cameras increasing inside a group; flag 1 otherwise
__global__ void k_ba_check(int64_t m, int64_t n, int C, const int32_t* __restrict__ cam,
                           const int32_t* __restrict__ pt, int* __restrict__ flag) {
    const int64_t o = (int64_t)blockIdx.x * kBaThreads + threadIdx.x;
    if (o >= m) return;
    const int32_t i = cam[o], j = pt[o];
    bool bad = i < 0 || i >= C || j < 0 || j >= n;
    if (o > 0) {
        const int32_t jp = pt[o - 1], ip = cam[o - 1];
        bad = bad || jp > j || (jp == j && ip >= i);
    }
    if (bad) atomicOr(flag, 1);
}

// the lower bound of point j in the point-ordered observations
__global__ void k_ba_offsets(int64_t n, int64_t m, const int32_t* __restrict__ pt, int64_t* __restrict__ start) {
    pdl_begin();
    const int64_t j = (int64_t)blockIdx.x * kBaThreads + threadIdx.x;
    if (j > n) return;
    int64_t lo = 0, hi = m;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (pt[mid] < j) lo = mid + 1;
        else hi = mid;
    }
    start[j] = lo;
}

__global__ void k_ba_masks(int64_t n, int W, const int64_t* __restrict__ start, const int32_t* __restrict__ cam,
                           uint32_t* __restrict__ mask) {
    pdl_begin();
    const int64_t j = (int64_t)blockIdx.x * kBaThreads + threadIdx.x;
    if (j >= n) return;
    uint32_t* mk = mask + (size_t)j * W;
    for (int w = 0; w < W; ++w) mk[w] = 0u;
    for (int64_t o = start[j]; o < start[j + 1]; ++o) mk[cam[o] >> 5] |= 1u << (cam[o] & 31);
}

// Each camera's observations in point order: a stable counting sort by camera.  Counts per block of
// kListBlock observations, their exclusive scan over the blocks (and over the cameras into cam_start),
// and the places: the block's first + the warps' before + the rank among the warp's equal cameras.
constexpr int kListBlock = 1024;

__global__ void __launch_bounds__(kListBlock)
k_ba_list_count(int64_t m, int C, const int32_t* __restrict__ cam, int64_t* __restrict__ count) {
    pdl_begin();
    __shared__ uint32_t s_count[256];
    for (int c = threadIdx.x; c < C; c += kListBlock) s_count[c] = 0u;
    __syncthreads();
    const int64_t o = (int64_t)blockIdx.x * kListBlock + threadIdx.x;
    if (o < m) atomicAdd(&s_count[cam[o]], 1u);
    __syncthreads();
    for (int c = threadIdx.x; c < C; c += kListBlock) count[(int64_t)blockIdx.x * C + c] = s_count[c];
}

__global__ void __launch_bounds__(256)
k_ba_list_scan(int64_t blocks, int C, int64_t* __restrict__ count, int64_t* __restrict__ cam_start) {
    pdl_begin();
    __shared__ int64_t s_total[256];
    const int c = threadIdx.x;
    int64_t run = 0;
    if (c < C) {
        int64_t b = 0;
        for (; b + 8 <= blocks; b += 8) {  // eight loads in flight
            int64_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = count[(b + k) * C + c];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                count[(b + k) * C + c] = run;
                run += v[k];
            }
        }
        for (; b < blocks; ++b) {
            const int64_t v = count[b * C + c];
            count[b * C + c] = run;
            run += v;
        }
        s_total[c] = run;
    }
    __syncthreads();
    if (c == 0) {
        int64_t at = 0;
        for (int k = 0; k < C; ++k) {
            cam_start[k] = at;
            at += s_total[k];
        }
        cam_start[C] = at;
    }
}

__global__ void __launch_bounds__(kListBlock)
k_ba_list_fill(int64_t m, int C, const int32_t* __restrict__ cam, const int64_t* __restrict__ count,
               const int64_t* __restrict__ cam_start, int64_t* __restrict__ cam_obs) {
    pdl_begin();
    __shared__ uint16_t s_warp[kListBlock / 32][256];
    for (int k = threadIdx.x; k < (kListBlock / 32) * 256; k += kListBlock) (&s_warp[0][0])[k] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t o = (int64_t)blockIdx.x * kListBlock + threadIdx.x;
    const int a = o < m ? cam[o] : 256;
    const unsigned same = __match_any_sync(0xffffffffu, a);
    const int rank = __popc(same & ((1u << lane) - 1u));
    if (a < 256 && rank == 0) s_warp[warp][a] = (uint16_t)__popc(same);
    __syncthreads();
    for (int c = threadIdx.x; c < C; c += kListBlock) {
        uint32_t run = 0;
        for (int w = 0; w < kListBlock / 32; ++w) {
            const uint32_t v = s_warp[w][c];
            s_warp[w][c] = (uint16_t)run;
            run += v;
        }
    }
    __syncthreads();
    if (a < 256) cam_obs[cam_start[a] + count[(int64_t)blockIdx.x * C + a] + s_warp[warp][a] + rank] = o;
}

// Sets the control words of a trial or a solve.
__global__ void k_ba_begin(double lam, BaCtl* __restrict__ ctl) {
    pdl_begin();
    ctl->lam = lam;
    ctl->cur = 0.0;
    ctl->accept = ctl->stop = ctl->accepted = ctl->it = 0;
}

// One thread: the solve's decision after a candidate's cost (cost[1], reset for the next one).  The first
// call (first = 1) only takes over the cost of the start (cost[0]).
__global__ void k_ba_decide(int first, BaCtl* __restrict__ ctl, double* __restrict__ cost, const int* __restrict__ status,
                            double* __restrict__ costs) {
    pdl_begin();
    if (ctl->stop) return;
    if (first) {
        costs[0] = ctl->cur = cost[0];
        return;
    }
    if (*status) {  // the reduced system was not positive definite
        ctl->stop = 1;
        return;
    }
    const double cand = cost[1];
    cost[1] = 0.0;
    if (cand < ctl->cur) {
        ctl->cur = cand;
        ctl->lam /= 10.0;
        ++ctl->accepted;
        ctl->accept = 1;
    } else {
        ctl->lam *= 10.0;
        ctl->accept = 0;
    }
    costs[++ctl->it] = ctl->cur;
}

// Linearization at (R, t, P).  move != nullptr (in a solve, after a decision): nothing to do unless the
// candidate (R, t, P are its buffers) was taken, which is then also copied into the state `move`.
__global__ void __launch_bounds__(kBaThreads)
k_ba_linearize(int64_t n, int C, const float* __restrict__ R, const float* __restrict__ t, const float* __restrict__ P,
               const int32_t* __restrict__ cam, const float* __restrict__ uv, const int64_t* __restrict__ start,
               Intr K, Robust rb, float4* __restrict__ Htp, float2* __restrict__ Hpp, float2* __restrict__ bp,
               double* __restrict__ cost, const BaCtl* __restrict__ ctl, BaState move, int copy_only) {
    pdl_begin();
    if (move.R) {
        if (ctl->stop || !ctl->accept) return;
        if (blockIdx.x == 0) {
            for (int k = threadIdx.x; k < 9 * C; k += kBaThreads) move.R[k] = R[k];
            for (int k = threadIdx.x; k < 3 * C; k += kBaThreads) move.t[k] = t[k];
        }
    }
    const int64_t j = (int64_t)blockIdx.x * kPointsPerCta + threadIdx.x / kGroup;
    const int l = threadIdx.x % kGroup;
    const Df zero = {0.f, 0.f};
    Df rho_sum = zero;
    Df hp[6] = {zero, zero, zero, zero, zero, zero}, gp[3] = {zero, zero, zero};
    if (j < n) {
        const float px = P[3 * j], py = P[3 * j + 1], pz = P[3 * j + 2];
        if (move.P && l < 3) move.P[3 * j + l] = l == 0 ? px : (l == 1 ? py : pz);
        const int64_t o1 = copy_only ? 0 : start[j + 1];
        for (int64_t o = start[j] + l; o < o1; o += kGroup) {
            const int i = cam[o];
            Df X[3], rho;
            float r[2], iz, w;
            cam_point_df(R, t, i, px, py, pz, X);
            float4* __restrict__ H = Htp + 5 * o;
            if (!residual(X, K, uv[2 * o], uv[2 * o + 1], rb, r, iz, w, rho)) {
                for (int k = 0; k < 5; ++k) H[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                continue;
            }
            df_acc(rho_sum, rho);
            float Jc[2][6], Jp[2][3], h[20];
            h[18] = h[19] = 0.f;
            jacobians(R, t, i, X, iz, K, Jc, Jp);
#pragma unroll
            for (int a = 0; a < 6; ++a)
#pragma unroll
                for (int c = 0; c < 3; ++c) h[3 * a + c] = w * (Jc[0][a] * Jp[0][c] + Jc[1][a] * Jp[1][c]);
#pragma unroll
            for (int k = 0; k < 5; ++k) H[k] = make_float4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
            // point block (upper: xx xy xz yy yz zz) and gradient
            int u = 0;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int c = a; c < 3; ++c) df_acc(hp[u++], w * (Jp[0][a] * Jp[0][c] + Jp[1][a] * Jp[1][c]));
#pragma unroll
            for (int a = 0; a < 3; ++a) df_acc(gp[a], -(w * (Jp[0][a] * r[0] + Jp[1][a] * r[1])));
        }
    }
    if (copy_only) return;
#pragma unroll
    for (int q = 0; q < 6; ++q) df_lanes_sum<kGroup>(hp[q]);
#pragma unroll
    for (int q = 0; q < 3; ++q) df_lanes_sum<kGroup>(gp[q]);
    if (j < n && l == 0) {
#pragma unroll
        for (int q = 0; q < 6; ++q) Hpp[6 * j + q] = make_float2(hp[q].h, hp[q].l);
#pragma unroll
        for (int q = 0; q < 3; ++q) bp[3 * j + q] = make_float2(gp[q].h, gp[q].l);
    }
    if (cost) cta_add(rho_sum, cost);
}

// items [q0, q1) of chunk c of `chunks` over `len` items
__device__ __forceinline__ void chunk_of(int64_t len, int c, int chunks, int64_t& q0, int64_t& q1) {
    q0 = len * c / chunks;
    q1 = len * (c + 1) / chunks;
}

// camera a's H_tt block (upper 21) and b_t (6) over one chunk of its observations
__global__ void __launch_bounds__(kBaThreads)
k_ba_camblocks(int C, const float* __restrict__ R, const float* __restrict__ t, const float* __restrict__ P,
               const int32_t* __restrict__ pt, const float* __restrict__ uv, const int64_t* __restrict__ cam_start,
               const int64_t* __restrict__ cam_obs, Intr K, Robust rb, float* __restrict__ camp,
               const BaCtl* __restrict__ ctl) {
    pdl_begin();
    if (ctl && (ctl->stop || !ctl->accept)) return;
    __shared__ float s_red[kBaThreads / 32][27];
    const int a = blockIdx.x, c = blockIdx.y;
    int64_t q0, q1;
    chunk_of(cam_start[a + 1] - cam_start[a], c, gridDim.y, q0, q1);
    const int64_t* __restrict__ list = cam_obs + cam_start[a];
    float acc[27];
#pragma unroll
    for (int q = 0; q < 27; ++q) acc[q] = 0.f;
    for (int64_t q = q0 + threadIdx.x; q < q1; q += kBaThreads) {
        const int64_t o = list[q], j = pt[o];
        Df X[3], rho;
        float r[2], iz, w;
        cam_point_df(R, t, a, P[3 * j], P[3 * j + 1], P[3 * j + 2], X);
        if (!residual(X, K, uv[2 * o], uv[2 * o + 1], rb, r, iz, w, rho)) continue;
        float Jc[2][6], Jp[2][3];
        jacobians(R, t, a, X, iz, K, Jc, Jp);
        int u = 0;
#pragma unroll
        for (int p = 0; p < 6; ++p)
#pragma unroll
            for (int s2 = p; s2 < 6; ++s2) acc[u++] += w * (Jc[0][p] * Jc[0][s2] + Jc[1][p] * Jc[1][s2]);
#pragma unroll
        for (int p = 0; p < 6; ++p) acc[21 + p] -= w * (Jc[0][p] * r[0] + Jc[1][p] * r[1]);
    }
    const float tot = block_sum<27>(acc, s_red);
    if (threadIdx.x < 27) camp[((size_t)c * C + a) * 27 + threadIdx.x] = tot;
}

// (H_pp + lam diag)^-1 in two floats and in FP32, y = H^-1 b_p
constexpr int kPointThreads = 128;  // FP64: spread over the SMs' pipes
__global__ void __launch_bounds__(kPointThreads)
k_ba_points(int64_t n, const float2* __restrict__ Hpp, const float2* __restrict__ bp, const BaCtl* __restrict__ ctl,
            float2* __restrict__ Hinv, float* __restrict__ M, float* __restrict__ y) {
    pdl_begin();
    if (ctl->stop) return;
    const int64_t j = (int64_t)blockIdx.x * kPointThreads + threadIdx.x;
    if (j >= n) return;
    const double lam = ctl->lam;
    double h[6], g[3];
#pragma unroll
    for (int q = 0; q < 6; ++q) h[q] = (double)Hpp[6 * j + q].x + (double)Hpp[6 * j + q].y;
#pragma unroll
    for (int q = 0; q < 3; ++q) g[q] = (double)bp[3 * j + q].x + (double)bp[3 * j + q].y;
    const double a = h[0] * (1 + lam), b = h[1], c = h[2], d = h[3] * (1 + lam), e = h[4], f = h[5] * (1 + lam);
    // symmetric [[a b c] [b d e] [c e f]]: inverse by cofactors
    const double A = d * f - e * e, B = c * e - b * f, Cc = b * e - c * d;
    const double det = a * A + b * B + c * Cc;
    double inv[6] = {0, 0, 0, 0, 0, 0};
    if (h[0] > 0.0 && det > 0.0) {  // a point no observation weighs keeps a zero step
        const double id = 1.0 / det;
        inv[0] = A * id;
        inv[1] = B * id;
        inv[2] = Cc * id;
        inv[3] = (a * f - c * c) * id;
        inv[4] = (b * c - a * e) * id;
        inv[5] = (a * d - b * b) * id;
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const Df v = df_from(inv[q]);
        Hinv[6 * j + q] = make_float2(v.h, v.l);
        M[6 * j + q] = v.h;
    }
    y[3 * j] = (float)(inv[0] * g[0] + inv[1] * g[1] + inv[2] * g[2]);
    y[3 * j + 1] = (float)(inv[1] * g[0] + inv[3] * g[1] + inv[4] * g[2]);
    y[3 * j + 2] = (float)(inv[2] * g[0] + inv[4] * g[1] + inv[5] * g[2]);
}

// H_tp of observation o: its 18 values in a record of 20, five 16-byte accesses (a warp's lanes read
// records apart, so each access of a lane is a cache line of its own: nine 8-byte ones held the Schur
// blocks to the L1's rate)
__device__ __forceinline__ void load_htp(const float4* __restrict__ Htp, int64_t o, float (&v)[20]) {
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const float4 u = __ldg(Htp + 5 * o + q);
        v[4 * q] = u.x;
        v[4 * q + 1] = u.y;
        v[4 * q + 2] = u.z;
        v[4 * q + 3] = u.w;
    }
}

// Over one chunk of camera a's observations, for every camera b >= a: sum over the points also seen
// by b of H_tp,a H_pp^-1 H_tp,b^T; for b == a also of H_tp,a y.  The chunk is taken kSchurObs observations
// at a time, staged once for all b; a warp owns the pairs b = a + warp, a + warp + 8, ...: it lists
// the staged observations whose point b sees and its lanes take them, so a pair's 36 sums are reduced
// once per kSchurObs observations.  A's side of the products is formed once, when it is staged.  Bound by
// the L1's rate over records read apart.  At 32 cameras, 20k points, 124k observations: a CTA per pair and
// walk of camera a's list 55 us (and 23 us for A's side), this 52 us with 72-byte records and A's side
// formed per pair, 34 us now.
// (kSchurObs: what fits the 48 KB of static shared memory; the solve of six iterations 1.14-1.16 ms with 320, 1.21 with
// 256 or 160.)
constexpr int kSchurObs = 320;
__global__ void __launch_bounds__(kBaThreads, 3)
k_ba_schur(int C, int W, const int32_t* __restrict__ pt, const int64_t* __restrict__ start,
           const uint32_t* __restrict__ mask, const int64_t* __restrict__ cam_start, const int64_t* __restrict__ cam_obs,
           const float4* __restrict__ Htp, const float* __restrict__ M, const float* __restrict__ y,
           float* __restrict__ schp, float* __restrict__ rhsp, const BaCtl* __restrict__ ctl) {
    pdl_begin();
    if (ctl->stop) return;
    __shared__ int64_t s_start[kSchurObs];
    __shared__ float s_E[18][kSchurObs];  // H_tp,a H_pp^-1 of the staged observations
    __shared__ int32_t s_pt[kSchurObs];
    __shared__ uint32_t s_mask[8][kSchurObs];
    __shared__ uint16_t s_list[kBaThreads / 32][kSchurObs];
    const int a = blockIdx.x, c = blockIdx.y, pairs = C * (C + 1) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t q0, q1;
    chunk_of(cam_start[a + 1] - cam_start[a], c, gridDim.y, q0, q1);
    const int64_t* __restrict__ list = cam_obs + cam_start[a];
    int64_t base = q0;
    do {  // at least once: an empty chunk writes zeros
        const int cnt = (int)min((int64_t)kSchurObs, q1 - base);
        __syncthreads();
        for (int e = threadIdx.x; e < cnt; e += kBaThreads) {
            const int64_t o = list[base + e];
            const int32_t j = pt[o];
            s_pt[e] = j;
            s_start[e] = start[j];
            for (int w = 0; w < W; ++w) s_mask[w][e] = mask[(size_t)j * W + w];
            float H[20], m[6];
            load_htp(Htp, o, H);
            const float2* m2 = reinterpret_cast<const float2*>(M + 6 * (int64_t)j);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float2 u = __ldg(m2 + q);
                m[2 * q] = u.x;
                m[2 * q + 1] = u.y;
            }
#pragma unroll
            for (int r = 0; r < 6; ++r) {
                const float h0 = H[3 * r], h1 = H[3 * r + 1], h2 = H[3 * r + 2];
                s_E[3 * r][e] = h0 * m[0] + h1 * m[1] + h2 * m[2];
                s_E[3 * r + 1][e] = h0 * m[1] + h1 * m[3] + h2 * m[4];
                s_E[3 * r + 2][e] = h0 * m[2] + h1 * m[4] + h2 * m[5];
            }
        }
        __syncthreads();
        for (int b = a + warp; b < C; b += kBaThreads / 32) {
            // the staged observations whose point b also sees
            int seen = 0;
            for (int e0 = 0; e0 < cnt; e0 += 32) {
                const int e = e0 + lane;
                const bool sees = e < cnt && ((s_mask[b >> 5][e] >> (b & 31)) & 1u);
                const unsigned bal = __ballot_sync(0xffffffffu, sees);
                if (sees) s_list[warp][seen + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)e;
                seen += __popc(bal);
            }
            __syncwarp();
            float acc[36], ry[6];
#pragma unroll
            for (int q = 0; q < 36; ++q) acc[q] = 0.f;
#pragma unroll
            for (int q = 0; q < 6; ++q) ry[q] = 0.f;
            const bool any = seen > 0;
            for (int k = lane; k < seen; k += 32) {
                const int e = s_list[warp][k];
                int64_t ob = s_start[e] + __popc(s_mask[b >> 5][e] & ((1u << (b & 31)) - 1u));
                for (int w = 0; w < (b >> 5); ++w) ob += __popc(s_mask[w][e]);
                float Hb[20];
                load_htp(Htp, ob, Hb);
#pragma unroll
                for (int r = 0; r < 6; ++r) {
                    const float e0r = s_E[3 * r][e], e1r = s_E[3 * r + 1][e], e2r = s_E[3 * r + 2][e];
#pragma unroll
                    for (int s2 = 0; s2 < 6; ++s2)
                        acc[6 * r + s2] = fmaf(e0r, Hb[3 * s2], fmaf(e1r, Hb[3 * s2 + 1], fmaf(e2r, Hb[3 * s2 + 2], acc[6 * r + s2])));
                }
                if (a == b) {
                    const int64_t j = s_pt[e];
                    const float y0 = y[3 * j], y1 = y[3 * j + 1], y2 = y[3 * j + 2];
#pragma unroll
                    for (int r = 0; r < 6; ++r) ry[r] = fmaf(Hb[3 * r], y0, fmaf(Hb[3 * r + 1], y1, fmaf(Hb[3 * r + 2], y2, ry[r])));
                }
            }
            __syncwarp();
            float* out = schp + ((size_t)c * pairs + (a * C - a * (a - 1) / 2 + (b - a))) * 36;
            float v0 = 0.f, v1 = 0.f, vy = 0.f;  // lane l: sums l, 32 + l (l < 4) and the rhs's l (l < 6)
            if (any) {
#pragma unroll
                for (int q = 0; q < 36; ++q) {
                    float x = acc[q];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                    if (lane == (q & 31)) (q < 32 ? v0 : v1) = x;
                }
                if (a == b)
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        float x = ry[q];
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                        if (lane == q) vy = x;
                    }
            }
            if (base == q0) {
                out[lane] = v0;
                if (lane < 4) out[32 + lane] = v1;
                if (a == b && lane < 6) rhsp[((size_t)c * C + a) * 6 + lane] = vy;
            } else if (any) {
                out[lane] += v0;
                if (lane < 4) out[32 + lane] += v1;
                if (a == b && lane < 6) rhsp[((size_t)c * C + a) * 6 + lane] += vy;
            }
        }
        base += kSchurObs;
    } while (base < q1);
}

__device__ __forceinline__ int64_t row_off(int i, int N) { return (int64_t)i * N - (int64_t)i * (i - 1) / 2; }

// The damped reduced matrix S [N][N] (both triangles) and rhs [N] from the chunk sums, summed in two
// floats and stored in FP32 (the scaled FP32 system is what gets factored).  Thread per entry of a camera
// pair's 6 x 6 block, in the order the chunks hold them, then per row of the rhs.
__global__ void __launch_bounds__(kBaThreads)
k_ba_assemble(int C, int chc, int chs, const float* __restrict__ camp, const float* __restrict__ schp,
              const float* __restrict__ rhsp, const BaCtl* __restrict__ ctl, float* __restrict__ S,
              float* __restrict__ rhs) {
    pdl_begin();
    if (ctl->stop) return;
    const int N = 6 * C, pairs = C * (C + 1) / 2, entries = 36 * pairs;
    const int e = blockIdx.x * kBaThreads + threadIdx.x;
    if (e >= entries + N) return;
    Df v = {0.f, 0.f};
    if (e >= entries) {
        const int i = e - entries, a = i / 6, r = i % 6;
#pragma unroll 8
        for (int k = 0; k < chc; ++k) df_acc(v, camp[((size_t)k * C + a) * 27 + 21 + r]);
#pragma unroll 8
        for (int k = 0; k < chs; ++k) df_acc(v, -rhsp[((size_t)k * C + a) * 6 + r]);
        rhs[i] = df_two(v.h, v.l).h;
        return;
    }
    const int p = e / 36, r = (e % 36) / 6, q = e % 6;
    // pair (a, b), a <= b, number p in row-major order of the upper triangle of C x C
    int a = (int)(((float)(2 * C + 1) - sqrtf((float)(2 * C + 1) * (float)(2 * C + 1) - 8.0f * (float)p)) * 0.5f);
    a = min(max(a, 0), C - 1);
    while (a > 0 && a * C - a * (a - 1) / 2 > p) --a;
    while ((a + 1) * C - (a + 1) * a / 2 <= p) ++a;
    const int b = a + p - (a * C - a * (a - 1) / 2);
    if (a == b && r > q) return;  // symmetric: the upper half writes both
#pragma unroll 8
    for (int k = 0; k < chs; ++k) df_acc(v, -schp[((size_t)k * pairs + p) * 36 + 6 * r + q]);
    if (a == b) {  // camera block, upper index of (r, q)
        const int u = r * 6 - r * (r - 1) / 2 + (q - r);
        Df h = {0.f, 0.f};
#pragma unroll 8
        for (int k = 0; k < chc; ++k) df_acc(h, camp[((size_t)k * C + a) * 27 + u]);
        h = df_two(h.h, h.l);
        df_acc(v, r == q ? df_mul(h, df_from(1.0 + ctl->lam)) : h);
    }
    const float x = df_two(v.h, v.l).h;
    const int i = 6 * a + r, j = 6 * b + q;
    S[(int64_t)i * N + j] = x;
    S[(int64_t)j * N + i] = x;
}

// fixed rows (gauge, unobserved) and the Jacobi scale: s_id[i] = 1 / sqrt(S_ii), 0 for a fixed row;
// s_rhs[i] = rhs_i / sqrt(S_ii) (FP32: the scaled system is what gets factored)
template <int kThreads>
__device__ __forceinline__ void scale_rows(int N, int NP, int fixed_axis, const float* __restrict__ S,
                                           const float* __restrict__ rhs, float* s_id, float* s_rhs) {
    for (int i = threadIdx.x; i < NP; i += kThreads) {
        if (i >= N) {
            s_id[i] = 0.f;
            s_rhs[i] = 0.f;
            continue;
        }
        const float dg = S[(int64_t)i * N + i];
        const bool fixed = i < 6 || i == 9 + fixed_axis || !(dg > 0.f);
        const float id = fixed ? 0.f : rsqrtf(dg);
        s_id[i] = id;
        s_rhs[i] = fixed ? 0.f : rhs[i] * id;
    }
}

__device__ __forceinline__ float scaled_entry(float v, int i, int j, const float* s_id) {
    if (i == j) return 1.f;
    const float a = s_id[i], b = s_id[j];
    return (a == 0.f || b == 0.f) ? 0.f : v * a * b;
}

// candidate pose of camera i: R <- exp([omega]x) R (Rodrigues, double), t <- t + v
__device__ void move_camera(int i, const double* __restrict__ dc, const float* __restrict__ R, const float* __restrict__ t,
                            float* __restrict__ Rn, float* __restrict__ tn, float* __restrict__ dcam) {
    const double w0 = dc[6 * i], w1 = dc[6 * i + 1], w2 = dc[6 * i + 2];
    const double x = w0 * w0 + w1 * w1 + w2 * w2;  // theta^2
    double s, c;  // sin(theta) / theta, (1 - cos(theta)) / theta^2
    if (x < 0.25) {  // their Taylor series: the ninth terms are below 1e-19
        s = c = 0.0;
#pragma unroll
        for (int k = 8; k >= 1; --k) {
            s = (1.0 - s) * x * (1.0 / (2.0 * k * (2.0 * k + 1.0)));
            c = (1.0 - c) * x * (1.0 / ((2.0 * k + 1.0) * (2.0 * k + 2.0)));
        }
        s = 1.0 - s;
        c = 0.5 * (1.0 - c);
    } else {
        const double th = sqrt(x);
        s = sin(th) / th;
        c = (1.0 - cos(th)) / x;
    }
    double Ex[3][3];
    const double Kx[3][3] = {{0, -w2, w1}, {w2, 0, -w0}, {-w1, w0, 0}};
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            double kk = 0.0;
#pragma unroll
            for (int q = 0; q < 3; ++q) kk += Kx[a][q] * Kx[q][b];
            Ex[a][b] = (a == b ? 1.0 : 0.0) + s * Kx[a][b] + c * kk;
        }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            double v = 0.0;
#pragma unroll
            for (int q = 0; q < 3; ++q) v += Ex[a][q] * (double)R[9 * i + 3 * q + b];
            Rn[9 * i + 3 * a + b] = (float)v;
        }
    for (int a = 0; a < 3; ++a) tn[3 * i + a] = (float)((double)t[3 * i + a] + dc[6 * i + 3 + a]);
    if (dcam)
        for (int a = 0; a < 6; ++a) dcam[6 * i + a] = (float)dc[6 * i + a];
}

// One CTA: the Jacobi-scaled reduced system in packed upper storage A (FP32; shared memory when it
// fits, else global scratch), eliminated with the rhs carried along, then back-substituted.
__global__ void __launch_bounds__(kSolveThreads)
k_ba_solve(int C, const float* __restrict__ S, const float* __restrict__ rhs, int fixed_axis,
           float* __restrict__ Aglob, double* __restrict__ dc, int* __restrict__ status, const BaCtl* __restrict__ ctl,
           const float* __restrict__ R, const float* __restrict__ t, float* __restrict__ Rn, float* __restrict__ tn,
           float* __restrict__ dcam) {
    pdl_begin();
    if (ctl->stop) return;
    extern __shared__ __align__(16) float s_dyn[];
    __shared__ float s_rhs[kMaxN];
    __shared__ float s_d[kMaxN];  // 1 / sqrt of the diagonal; 0 marks a fixed row
    const int N = 6 * C;
    float* A = Aglob ? Aglob : s_dyn;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = kSolveThreads / 32;
    scale_rows<kSolveThreads>(N, N, fixed_axis, S, rhs, s_d, s_rhs);
    __syncthreads();
    for (int i = warp; i < N; i += warps) {
        const int64_t oi = row_off(i, N);
        for (int j = i + lane; j < N; j += 32) A[oi + (j - i)] = scaled_entry(S[(int64_t)i * N + j], i, j, s_d);
    }
    __syncthreads();
    // symmetric elimination: row i -= (A_ki / A_kk) row k for i > k, upper part and rhs
    for (int k = 0; k < N - 1; ++k) {
        const int64_t ok = row_off(k, N);
        const float d = A[ok];
        const float inv = d > 0.f ? 1.0f / d : 0.f;
        if (threadIdx.x == 0 && !(d > 0.f)) atomicOr(status, 1);
        const float rk = s_rhs[k];
        for (int i = k + 1 + warp; i < N; i += warps) {
            const float f = A[ok + (i - k)] * inv;
            if (f == 0.f) continue;
            const int64_t oi = row_off(i, N);
            for (int j = i + lane; j < N; j += 32) A[oi + (j - i)] = fmaf(-f, A[ok + (j - k)], A[oi + (j - i)]);
            if (lane == 0) s_rhs[i] = fmaf(-f, rk, s_rhs[i]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && !(A[row_off(N - 1, N)] > 0.f)) atomicOr(status, 1);
    // back substitution by one warp, column-oriented: x_k = rhs_k / A_kk, rhs_i -= A_ik x_k (i < k)
    if (warp == 0) {
        for (int k = N - 1; k >= 0; --k) {
            const float dk = A[row_off(k, N)];
            const float x = dk > 0.f ? s_rhs[k] / dk : 0.f;
            for (int i = lane; i < k; i += 32) s_rhs[i] = fmaf(-A[row_off(i, N) + (k - i)], x, s_rhs[i]);
            if (lane == 0) dc[k] = (double)x * s_d[k];
            __syncwarp();
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < C; i += kSolveThreads) move_camera(i, dc, R, t, Rn, tn, dcam);
}

// ---- blocked solve (N padded to NP, a multiple of kPanel, NP <= 224): full lower triangle in shared
// memory with the rhs as row NP (so the factorization also solves L z = rhs), Cholesky right-looking
// by panels of kPanel columns: one warp factors the diagonal block in registers, a thread per row
// solves the rows below it and leaves them transposed in Pt, 4 x 4 register micro-tiles with 16-byte
// accesses update the trailing lower triangle.  Meanwhile another warp inverts the diagonal block into
// its own unused upper triangle, so that back substitution takes a product per panel instead of kPanel
// dependent steps, and the first warp factors the next diagonal block while the others update the rest.
// At 32 cameras 116 -> 59 us: the trailing updates and the row solves, each a third of it, are bound by
// one SM's shared memory and latency.

// warp: Cholesky of the kPanel x kPanel diagonal block at B (row stride ld), lane r < kPanel
// holding row r in registers; rdiag[k] = 1 / L_kk.  The pivot goes through the hardware
// reciprocal square root (2 ulp): the correctly rounded sqrt and division are multi-instruction
// sequences, and they sit on the dependent chain of every column.
__device__ __forceinline__ void factor_diag_block(float* B, int ld, int lane, float* rdiag, int* status) {
    float a[kPanel];
#pragma unroll
    for (int c = 0; c < kPanel; ++c) a[c] = (lane < kPanel && c <= lane) ? B[lane * ld + c] : 0.f;
    bool bad = false;
    float mine = 0.f;
    // no branch between the shuffles (a lane's entries right of its diagonal take part and are never
    // used): reconverging around each update cost 700 cycles a column
#pragma unroll
    for (int k = 0; k < kPanel; ++k) {
        const float p = __shfl_sync(0xffffffffu, a[k], k);
        bad = bad || !(p > 0.f);
        const float d = p > 0.f ? p : 1.f;
        const float rs = rsqrtf(d);
        mine = lane == k ? rs : mine;
        a[k] = (lane == k ? d : a[k]) * rs;
#pragma unroll
        for (int c = k + 1; c < kPanel; ++c) a[c] = fmaf(-a[k], __shfl_sync(0xffffffffu, a[k], c), a[c]);
    }
    if (bad && lane == 0) atomicOr(status, 1);
    if (lane < kPanel) {
        rdiag[lane] = mine;
#pragma unroll
        for (int c = 0; c < kPanel; ++c)
            if (c <= lane) B[lane * ld + c] = a[c];
    }
}

// warp: the strictly lower part of the inverse of the factored block at B, transposed into B's strictly
// upper part; lane j < kPanel solves L x = e_j
__device__ __forceinline__ void invert_diag_block(float* B, int ld, int lane, const float* rdiag) {
    if (lane >= kPanel) return;
    float x[kPanel];
#pragma unroll
    for (int i = 0; i < kPanel; ++i) {
        float v = i == lane ? 1.f : 0.f;
#pragma unroll
        for (int k = 0; k < i; ++k) v = fmaf(-B[i * ld + k], x[k], v);
        x[i] = v * rdiag[i];
        if (i > lane) B[lane * ld + i] = x[i];
    }
}

__global__ void __launch_bounds__(kBlockedThreads)
k_ba_solve_blocked(int C, const float* __restrict__ S, const float* __restrict__ rhs, int fixed_axis,
                   double* __restrict__ dc, int* __restrict__ status, const BaCtl* __restrict__ ctl,
                   const float* __restrict__ R, const float* __restrict__ t, float* __restrict__ Rn,
                   float* __restrict__ tn, float* __restrict__ dcam) {
    pdl_begin();
    if (ctl->stop) return;
    extern __shared__ __align__(16) float A[];
    __shared__ float s_rhs[kMaxBlockedN];
    __shared__ float s_id[kMaxBlockedN];  // 1 / sqrt of the diagonal; 0 marks a fixed (or padding) row
    __shared__ float s_rdiag[kMaxBlockedN];  // 1 / L_kk
    const int N = 6 * C, NP = (N + kPanel - 1) / kPanel * kPanel, ld = NP + 4;
    float* const Pt = A + (size_t)(NP + 1) * ld;  // [kPanel][ld]: the panel's rows, transposed
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = kBlockedThreads / 32;
    scale_rows<kBlockedThreads>(N, NP, fixed_axis, S, rhs, s_id, s_rhs);
    __syncthreads();
    // (whole rows, several loads in flight: above the diagonal nothing is read)
    for (int k0 = threadIdx.x; k0 < NP * (NP / 2); k0 += 4 * kBlockedThreads) {
        float2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u * kBlockedThreads, r = k / (NP / 2), c = 2 * (k % (NP / 2));  // N is even
            v[u] = r < N && c < N ? *reinterpret_cast<const float2*>(S + (int64_t)r * N + c) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + u * kBlockedThreads, r = k / (NP / 2), c = 2 * (k % (NP / 2));
            if (r < NP)
                *reinterpret_cast<float2*>(A + r * ld + c) =
                    make_float2(scaled_entry(v[u].x, r, c, s_id), scaled_entry(v[u].y, r, c + 1, s_id));
        }
    }
    for (int c = threadIdx.x; c < NP; c += kBlockedThreads) A[NP * ld + c] = s_rhs[c];
    __syncthreads();
    if (warp == 0) factor_diag_block(A, ld, lane, s_rdiag, status);
    __syncthreads();
    for (int c0 = 0; c0 < NP; c0 += kPanel) {
        // rows below the panel and the rhs, thread per row: x L_pp^T = a by forward substitution
        const int t0 = c0 + kPanel;
        if (warp == warps - 1) {
            invert_diag_block(A + c0 * ld + c0, ld, lane, s_rdiag + c0);
        } else {
            for (int r = t0 + threadIdx.x; r <= NP; r += kBlockedThreads - 32) {
                float4* const row = reinterpret_cast<float4*>(A + r * ld + c0);
                float x[kPanel];
#pragma unroll
                for (int q = 0; q < kPanel / 4; ++q) {
                    const float4 v = row[q];
                    x[4 * q] = v.x;
                    x[4 * q + 1] = v.y;
                    x[4 * q + 2] = v.z;
                    x[4 * q + 3] = v.w;
                }
#pragma unroll
                for (int k = 0; k < kPanel; ++k) {
                    x[k] *= s_rdiag[c0 + k];
#pragma unroll
                    for (int q = k + 1; q < kPanel; ++q) x[q] = fmaf(-A[(c0 + q) * ld + c0 + k], x[k], x[q]);
                }
#pragma unroll
                for (int q = 0; q < kPanel / 4; ++q) row[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
#pragma unroll
                for (int q = 0; q < kPanel; ++q) Pt[q * ld + r] = x[q];
            }
        }
        __syncthreads();
        // trailing lower triangle in 4 x 4 micro-tiles (row-major over the triangle), and the rhs:
        // A_rc -= sum_q L_rq L_cq over the panel
        const int mt = (NP - t0) >> 2, tiles = mt * (mt + 1) / 2;
        auto update = [&](int id) {
            int mi = (int)((sqrtf(8.0f * (float)id + 1.0f) - 1.0f) * 0.5f);
            while (mi * (mi + 1) / 2 > id) --mi;
            while ((mi + 1) * (mi + 2) / 2 <= id) ++mi;
            const int r = t0 + 4 * mi, c = t0 + 4 * (id - mi * (mi + 1) / 2);
            float acc[4][4] = {};
#pragma unroll
            for (int q = 0; q < kPanel; ++q) {
                const float4 lr = *reinterpret_cast<const float4*>(Pt + q * ld + r);
                const float4 lc = *reinterpret_cast<const float4*>(Pt + q * ld + c);
                const float vr[4] = {lr.x, lr.y, lr.z, lr.w}, vc[4] = {lc.x, lc.y, lc.z, lc.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(vr[u], vc[v], acc[u][v]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float4* const dst = reinterpret_cast<float4*>(A + (r + u) * ld + c);
                float4 o = *dst;  // (a diagonal tile's upper part holds nothing yet)
                o.x -= acc[u][0];
                o.y -= acc[u][1];
                o.z -= acc[u][2];
                o.w -= acc[u][3];
                *dst = o;
            }
        };
        // the first warp takes the next diagonal block's tiles (the first kAhead) and factors it while
        // the others work on the rest
        constexpr int kAhead = (kPanel / 4) * (kPanel / 4 + 1) / 2;
        if (warp == 0) {
            if (t0 < NP) {
                if (lane < kAhead) update(lane);
                __syncwarp();
                factor_diag_block(A + t0 * ld + t0, ld, lane, s_rdiag + t0, status);
            }
        } else {
            for (int id = kAhead + threadIdx.x - 32; id < tiles; id += kBlockedThreads - 32) update(id);
            for (int c = t0 + threadIdx.x - 32; c < NP; c += kBlockedThreads - 32) {
                float v = A[NP * ld + c];
#pragma unroll
                for (int q = 0; q < kPanel; ++q) v = fmaf(-Pt[q * ld + NP], Pt[q * ld + c], v);
                A[NP * ld + c] = v;
            }
        }
        __syncthreads();
    }
    // L^T x = z, panels from the last: x = L_pp^-T z of the panel, then the rows above
    float* const z = A + NP * ld;
    for (int c0 = NP - kPanel; c0 >= 0; c0 -= kPanel) {
        if (warp == 0) {
            float x = 0.f;
            if (lane < kPanel) {
                x = z[c0 + lane] * s_rdiag[c0 + lane];
#pragma unroll
                for (int k = 1; k < kPanel; ++k)
                    if (k > lane) x = fmaf(A[(c0 + lane) * ld + c0 + k], z[c0 + k], x);
            }
            __syncwarp();
            if (lane < kPanel) z[c0 + lane] = x;
        }
        __syncthreads();
        for (int r = threadIdx.x; r < c0; r += kBlockedThreads) {
            float v = z[r];
#pragma unroll
            for (int k = 0; k < kPanel; ++k) v = fmaf(-A[(c0 + k) * ld + r], z[c0 + k], v);
            z[r] = v;
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < N; i += kBlockedThreads) dc[i] = (double)z[i] * s_id[i];
    __syncthreads();
    for (int i = threadIdx.x; i < C; i += kBlockedThreads) move_camera(i, dc, R, t, Rn, tn, dcam);
}

// Delta_p = H^-1 (b_p - sum H_tp^T Delta_t), the candidate point, and its observations' robust cost at
// the candidate (behind a camera: 1e30)
__global__ void __launch_bounds__(kBaThreads)
k_ba_backsub(int64_t n, const int64_t* __restrict__ start, const int32_t* __restrict__ cam, const float* __restrict__ uv,
             Intr K, Robust rb, const float4* __restrict__ Htp, const float2* __restrict__ Hinv,
             const float2* __restrict__ bp, const double* __restrict__ dc, const float* __restrict__ P,
             const float* __restrict__ Rn, const float* __restrict__ tn, float* __restrict__ Pn, float* __restrict__ dP,
             double* __restrict__ cost, const BaCtl* __restrict__ ctl) {
    pdl_begin();
    if (ctl->stop) return;
    const int64_t j = (int64_t)blockIdx.x * kPointsPerCta + threadIdx.x / kGroup;
    const int l = threadIdx.x % kGroup;
    const Df zero = {0.f, 0.f};
    Df g[3] = {zero, zero, zero}, rho_sum = zero;
    const bool live = j < n;
    const int64_t o0 = live ? start[j] : 0, o1 = live ? start[j + 1] : 0;
    for (int64_t o = o0 + l; o < o1; o += kGroup) {
        const int i = cam[o];
        float H[20], dci[6];
        load_htp(Htp, o, H);
#pragma unroll
        for (int r = 0; r < 6; ++r) dci[r] = (float)dc[6 * i + r];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float v = 0.f;
#pragma unroll
            for (int r = 0; r < 6; ++r) v = fmaf(H[3 * r + c], dci[r], v);
            df_acc(g[c], -v);
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) df_lanes_sum<kGroup>(g[c]);
    if (live) {
        Df h[6], d[3];
        float pn[3];
#pragma unroll
        for (int q = 0; q < 6; ++q) h[q] = {Hinv[6 * j + q].x, Hinv[6 * j + q].y};
#pragma unroll
        for (int c = 0; c < 3; ++c) g[c] = df_add(g[c], {bp[3 * j + c].x, bp[3 * j + c].y});
        d[0] = df_add(df_add(df_mul(h[0], g[0]), df_mul(h[1], g[1])), df_mul(h[2], g[2]));
        d[1] = df_add(df_add(df_mul(h[1], g[0]), df_mul(h[3], g[1])), df_mul(h[4], g[2]));
        d[2] = df_add(df_add(df_mul(h[2], g[0]), df_mul(h[4], g[1])), df_mul(h[5], g[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            pn[c] = df_add(d[c], {P[3 * j + c], 0.f}).h;
            if (l == c) {
                Pn[3 * j + c] = pn[c];
                if (dP) dP[3 * j + c] = d[c].h;
            }
        }
        for (int64_t o = o0 + l; o < o1; o += kGroup) {
            Df X[3], rho;
            float r[2], iz, w;
            cam_point_df(Rn, tn, cam[o], pn[0], pn[1], pn[2], X);
            if (residual(X, K, uv[2 * o], uv[2 * o + 1], rb, r, iz, w, rho)) df_acc(rho_sum, rho);
            else df_acc(rho_sum, 1e30f);
        }
    }
    if (cost) cta_add(rho_sum, cost);
}

__global__ void k_ba_project(int64_t m, int64_t n, int C, const float* __restrict__ R, const float* __restrict__ t,
                             const float* __restrict__ P, const int32_t* __restrict__ cam,
                             const int32_t* __restrict__ pt, Intr K, float* __restrict__ uv, float* __restrict__ z) {
    const int64_t o = (int64_t)blockIdx.x * kBaThreads + threadIdx.x;
    if (o >= m) return;
    const int64_t j = pt[o];
    const int i = cam[o];
    if (i < 0 || i >= C || j < 0 || j >= n) {  // out of range: NaN, no access
        z[o] = uv[2 * o] = uv[2 * o + 1] = __int_as_float(0x7fc00000);
        return;
    }
    double X[3];
    cam_point(R, t, i, P[3 * j], P[3 * j + 1], P[3 * j + 2], X);
    z[o] = (float)X[2];
    const double iz = 1.0 / X[2];
    uv[2 * o] = (float)fma((double)K.fx * X[0], iz, (double)K.cx);
    uv[2 * o + 1] = (float)fma((double)K.fy * X[1], iz, (double)K.cy);
}

unsigned blocks_for(int64_t k) { return (unsigned)((k + kBaThreads - 1) / kBaThreads); }
unsigned points_blocks(int64_t k) { return (unsigned)((k + kPointsPerCta - 1) / kPointsPerCta); }

Intr intr(const float K[4]) { return Intr{K[0], K[1], K[2], K[3]}; }
Robust robust(float sigma, float delta) {
    const double inv = 1.0 / ((double)sigma * (double)sigma);
    const float h = (float)inv;
    return Robust{{h, (float)(inv - (double)h)}, h, delta};
}

}  // namespace

// ------------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------------
BaShape ba_shape(int C, int64_t n, int64_t m) {
    BaShape sh;
    sh.C = C;
    sh.n = n;
    sh.m = m;
    sh.W = (C + 31) / 32;
    sh.N = 6 * C;
    sh.pairs = C * (C + 1) / 2;
    // chunks of a camera's observation list: enough CTAs for four an SM, at least an item a thread
    const int64_t per_cam = C > 0 ? m / C : 0;
    const int64_t most = per_cam / kBaThreads > 1 ? per_cam / kBaThreads : 1, want = C > 0 ? (4 * 152 + C - 1) / C : 1;
    sh.chc = sh.chs = (int)(want < most ? want : most);
    const size_t NP = ((size_t)sh.N + kPanel - 1) / kPanel * kPanel;
    const size_t packed = (size_t)sh.N * (sh.N + 1) / 2 * sizeof(float);
    sh.blocked = NP <= (size_t)kMaxBlockedN;
    sh.solve_smem = sh.blocked ? blocked_smem(NP) : (packed <= kMaxPackedSmem ? packed : 0);
    sh.list_blocks = (m + kListBlock - 1) / kListBlock;
    return sh;
}

int ba_configure_solve() {
    // one bound for every problem size, so contexts of different sizes can coexist
    const bool ok =
        cudaFuncSetAttribute(k_ba_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxPackedSmem) == cudaSuccess &&
        cudaFuncSetAttribute(k_ba_solve_blocked, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)blocked_smem(kMaxBlockedN)) == cudaSuccess;
    return ok ? 0 : -1;
}

int launch_ba_check(int64_t m, int64_t n, int C, const int32_t* cam, const int32_t* pt, int* flag, cudaStream_t s) {
    cudaMemsetAsync(flag, 0, sizeof(int), s);
    if (m > 0) k_ba_check<<<blocks_for(m), kBaThreads, 0, s>>>(m, n, C, cam, pt, flag);
    return m > 0 ? 1 : 0;
}

int launch_ba_index(const BaShape& sh, const int32_t* pt, const int32_t* cam, int64_t* start, uint32_t* mask,
                    int64_t* cam_count, int64_t* cam_start, int64_t* cam_obs, cudaStream_t s) {
    launch_pdl(k_ba_offsets, dim3(blocks_for(sh.n + 1)), dim3(kBaThreads), 0, s, sh.n, sh.m, pt, start);
    if (sh.n > 0)
        launch_pdl(k_ba_masks, dim3(blocks_for(sh.n)), dim3(kBaThreads), 0, s, sh.n, sh.W, (const int64_t*)start, cam, mask);
    const unsigned lb = (unsigned)sh.list_blocks;
    if (lb) launch_pdl(k_ba_list_count, dim3(lb), dim3(kListBlock), 0, s, sh.m, sh.C, cam, cam_count);
    launch_pdl(k_ba_list_scan, dim3(1), dim3(256), 0, s, sh.list_blocks, sh.C, cam_count, cam_start);
    if (lb)
        launch_pdl(k_ba_list_fill, dim3(lb), dim3(kListBlock), 0, s, sh.m, sh.C, cam, (const int64_t*)cam_count,
                   (const int64_t*)cam_start, cam_obs);
    return 5;
}

int launch_ba_begin(double lam, BaCtl* ctl, double* cost, cudaStream_t s) {
    cudaMemsetAsync(cost, 0, 2 * sizeof(double), s);
    launch_pdl(k_ba_begin, dim3(1), dim3(1), 0, s, lam, ctl);
    return 1;
}

int launch_ba_decide(bool first, BaCtl* ctl, double* cost, const int* status, double* costs, cudaStream_t s) {
    launch_pdl(k_ba_decide, dim3(1), dim3(1), 0, s, first ? 1 : 0, ctl, cost, status, costs);
    return 1;
}

int launch_ba_linearize(const BaShape& sh, const float* R, const float* t, const float* P, const int32_t* cam,
                        const int32_t* pt, const float* uv, const int64_t* start, const int64_t* cam_start,
                        const int64_t* cam_obs, const float K[4], float sigma, float delta, float4* Htp, float2* Hpp,
                        float2* bp, float* camp, double* cost, const BaCtl* ctl, const BaState& move, bool copy_only,
                        cudaStream_t s, cudaEvent_t* ev) {
    const Robust rb = robust(sigma, delta);
    if (ev) cudaEventRecord(ev[0], s);
    const unsigned pb = sh.n > 0 ? points_blocks(sh.n) : 1;  // (the first CTA also moves the cameras)
    launch_pdl(k_ba_linearize, dim3(pb), dim3(kBaThreads), 0, s, sh.n, sh.C, R, t, P, cam, uv, start, intr(K), rb, Htp, Hpp,
               bp, cost, ctl, move, copy_only ? 1 : 0);
    if (copy_only) return 1;
    if (ev) cudaEventRecord(ev[1], s);
    launch_pdl(k_ba_camblocks, dim3(sh.C, sh.chc), dim3(kBaThreads), 0, s, sh.C, R, t, P, pt, uv, cam_start, cam_obs,
               intr(K), rb, camp, move.R ? ctl : (const BaCtl*)nullptr);
    if (ev) cudaEventRecord(ev[2], s);
    return 2;
}

int launch_ba_trial(const BaShape& sh, const int32_t* pt, const int64_t* start, const uint32_t* mask,
                    const int64_t* cam_start, const int64_t* cam_obs, const int32_t* cam, const float* uv,
                    const float K[4], float sigma, float delta, const float4* Htp, const float2* Hpp, const float2* bp,
                    const float* camp, const BaCtl* ctl, int fixed_axis, float2* Hinv, float* M, float* y, float* schp,
                    float* rhsp, float* Sfull, float* rhs, float* Aglob, double* dc, const float* R, const float* t,
                    const float* P, float* Rn, float* tn, float* Pn, float* dcam, float* dP, double* cost, int* status,
                    cudaStream_t s, cudaEvent_t* ev) {
    int launches = 3;
    if (sh.n > 0) {
        launch_pdl(k_ba_points, dim3((unsigned)((sh.n + kPointThreads - 1) / kPointThreads)), dim3(kPointThreads), 0, s, sh.n, Hpp, bp, ctl, Hinv, M, y);
        ++launches;
    }
    if (ev) cudaEventRecord(ev[0], s);
    launch_pdl(k_ba_schur, dim3(sh.C, sh.chs), dim3(kBaThreads), 0, s, sh.C, sh.W, pt, start, mask, cam_start, cam_obs, Htp,
               (const float*)M, (const float*)y, schp, rhsp, ctl);
    if (ev) cudaEventRecord(ev[1], s);
    launch_pdl(k_ba_assemble, dim3(blocks_for(36ll * sh.pairs + sh.N)), dim3(kBaThreads), 0, s,
               sh.C, sh.chc, sh.chs, camp, (const float*)schp, (const float*)rhsp, ctl, Sfull, rhs);
    if (sh.blocked)
        launch_pdl(k_ba_solve_blocked, dim3(1), dim3(kBlockedThreads), sh.solve_smem, s, sh.C, (const float*)Sfull,
                   (const float*)rhs, fixed_axis, dc, status, ctl, R, t, Rn, tn, dcam);
    else
        launch_pdl(k_ba_solve, dim3(1), dim3(kSolveThreads), sh.solve_smem, s, sh.C, (const float*)Sfull, (const float*)rhs,
                   fixed_axis, sh.solve_smem ? (float*)nullptr : Aglob, dc, status, ctl, R, t, Rn, tn, dcam);
    if (ev) cudaEventRecord(ev[2], s);
    if (sh.n > 0) {
        launch_pdl(k_ba_backsub, dim3(points_blocks(sh.n)), dim3(kBaThreads), 0, s, sh.n, start, cam, uv, intr(K),
                   robust(sigma, delta), Htp, (const float2*)Hinv, bp, (const double*)dc, P, (const float*)Rn,
                   (const float*)tn, Pn, dP, cost, ctl);
        ++launches;
    }
    if (ev) cudaEventRecord(ev[3], s);
    return launches;
}

int launch_ba_project(int64_t m, int64_t n, int C, const float* R, const float* t, const float* P, const int32_t* cam,
                      const int32_t* pt, const float K[4], float* uv, float* z, cudaStream_t s) {
    if (m <= 0) return 0;
    k_ba_project<<<blocks_for(m), kBaThreads, 0, s>>>(m, n, C, R, t, P, cam, pt, intr(K), uv, z);
    return 1;
}

}  // namespace pgs
