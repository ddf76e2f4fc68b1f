// L1 + D-SSIM loss of a rendered image against its target and the loss gradient (the paper
// reports SSIM, Sec. IV, and names no training loss; this is the 3DGS-style alternative to the
// plain L1 of K7).  Per colour plane, with G the 11 x 11 Gaussian window (sigma 1.5, taps
// normalised to sum 1) and zero padding:
//   mu_x = G*x, sigma_x^2 = G*x^2 - mu_x^2, sigma_xy = G*(xy) - mu_x mu_y,
//   SSIM = (2 mu_x mu_y + C1)(2 sigma_xy + C2) / ((mu_x^2 + mu_y^2 + C1)(sigma_x^2 + sigma_y^2 + C2)),
//   loss = (1 - lam) mean|x - y| + lam (1 - mean SSIM).
// Two tiled kernels, 32 x 22 output pixels of one plane per CTA with the 5-pixel halo staged in
// shared memory and the window applied separably (rows, then columns).  Shared-memory reads bound them, so a
// thread filters four neighbouring columns, then three rows, from one set of reads, and quantities that go
// together lie side by side (one read, and packed arithmetic); the swizzles keep every access free of bank
// conflicts.  22 rows and their halo are 32: a row's eight column groups fill the CTA's 256 threads.  At
// 1237 x 693 36 us forward, 35 us backward; one output at a time (32 x 32 tiles) took 52 each.
//   forward  the five filtered moments, SSIM, and per pixel the SSIM's derivatives with respect
//            to the three filtered moments of x (m1 = G*x, m2 = G*x^2, m12 = G*xy), written as
//            three planes; L1 and SSIM sums per CTA added in double;
//   backward filters the three derivative planes with the same window and combines them,
//            d(sum SSIM)/dx = G*ds/dm1 + 2 x G*ds/dm2 + y G*ds/dm12, with the L1 sign term.
#include "pgs_internal.cuh"

namespace pgs {
namespace {

constexpr int kR = 5;                 // window radius
constexpr int kTw = 32, kTh = 22;     // output tile
constexpr int kInW = kTw + 2 * kR, kInH = kTh + 2 * kR;  // staged, with the halo
constexpr int kCols = 4, kRows = 3;   // outputs of a thread in the row and in the column pass
constexpr int kThreads = 256;
static_assert(kInH * (kTw / kCols) == kThreads && kTw * 8 == kThreads && 8 * kRows >= kTh, "one task a thread and pass");
constexpr int kPairs = kInW + 2 * ((kInW + 3) / 4);  // row of float2: 16 bytes after every four columns
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

struct Taps {
    float w[2 * kR + 1];
};

__device__ __forceinline__ int pair_at(int c) { return c + 2 * (c >> 2); }
// column c of a row of float4 written four columns a thread and read one a thread
__device__ __forceinline__ int quad_at(int c) { return (c & ~3) | ((c & 3) ^ ((c >> 3) & 3)); }

// f(row, column, offset in the plane or -1 outside the image) for the tile and its halo
template <class F>
__device__ __forceinline__ void stage(int W, int H, int x0, int y0, F f) {
#pragma unroll
    for (int k = threadIdx.x; k < kInH * kInW; k += kThreads) {
        const int r = k / kInW, c = k % kInW, y = y0 - kR + r, x = x0 - kR + c;
        f(r, c, x >= 0 && x < W && y >= 0 && y < H ? (int64_t)y * W + x : (int64_t)-1);
    }
}

__global__ void __launch_bounds__(kThreads)
k_ssim_fwd(const float* __restrict__ img, const float* __restrict__ tgt, int W, int H, Taps taps,
           float* __restrict__ dm, double* __restrict__ sums) {
    __shared__ __align__(16) float2 sxy[kInH][kPairs];  // (x, y)
    __shared__ float4 hm[kInH][kTw];                    // row-filtered x, y, x^2, y^2
    __shared__ __align__(16) float hxy[kInH][kTw];      // and xy
    __shared__ double red[2][kThreads / 32];
    const int x0 = blockIdx.x * kTw, y0 = blockIdx.y * kTh, c = blockIdx.z;
    const size_t plane = (size_t)W * H;
    const float* __restrict__ X = img + c * plane;
    const float* __restrict__ Y = tgt + c * plane;
    stage(W, H, x0, y0, [&](int r, int col, int64_t o) {
        sxy[r][pair_at(col)] = o >= 0 ? make_float2(X[o], Y[o]) : make_float2(0.f, 0.f);
    });
    __syncthreads();
    {
        const int r = threadIdx.x >> 3, t = threadIdx.x & 7;
        constexpr int kN = kCols + 2 * kR;
        F2 m1[kCols], m2[kCols];
        float m12[kCols];
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
            m1[j] = m2[j] = f2(0.f);
            m12[j] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kN; i += 2) {
            const float4 two = *reinterpret_cast<const float4*>(&sxy[r][6 * t + pair_at(i)]);
            const float u[2] = {two.x, two.z}, v[2] = {two.y, two.w};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const F2 uv = f2(u[h], v[h]), sq = mul2(uv, uv);
                const float p = u[h] * v[h];
#pragma unroll
                for (int j = 0; j < kCols; ++j) {
                    const int k = i + h - j;  // tap
                    if (k < 0 || k > 2 * kR) continue;
                    const F2 w = f2(taps.w[k]);
                    m1[j] = fma2(w, uv, m1[j]);
                    m2[j] = fma2(w, sq, m2[j]);
                    m12[j] = fmaf(taps.w[k], p, m12[j]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
            const float2 a = un(m1[j]), b = un(m2[j]);
            hm[r][quad_at(kCols * t + j)] = make_float4(a.x, a.y, b.x, b.y);
        }
        *reinterpret_cast<float4*>(&hxy[r][kCols * t]) = make_float4(m12[0], m12[1], m12[2], m12[3]);
    }
    __syncthreads();
    float l1 = 0.f, ss = 0.f;  // a thread's at most 3 values; per CTA in double
    {
        const int col = threadIdx.x & 31, r0 = kRows * (threadIdx.x >> 5);
        const int q = quad_at(col);
        F2 m1[kRows], m2[kRows];
        float m12[kRows];
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
            m1[j] = m2[j] = f2(0.f);
            m12[j] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kRows + 2 * kR; ++i) {
            const int r = min(r0 + i, kInH - 1);  // the last rows of the last group are past the tile
            const float4 h = hm[r][q];
            const float p = hxy[r][col];
            const F2 a = f2(h.x, h.y), b = f2(h.z, h.w);
#pragma unroll
            for (int j = 0; j < kRows; ++j) {
                const int k = i - j;
                if (k < 0 || k > 2 * kR) continue;
                const F2 w = f2(taps.w[k]);
                m1[j] = fma2(w, a, m1[j]);
                m2[j] = fma2(w, b, m2[j]);
                m12[j] = fmaf(taps.w[k], p, m12[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
            const int r = r0 + j, x = x0 + col, y = y0 + r;
            if (r >= kTh || x >= W || y >= H) continue;
            const float2 mu = un(m1[j]), sq = un(m2[j]);
            const float mx = mu.x, my = mu.y;
            const float sxx = sq.x - mx * mx, syy = sq.y - my * my, sxyc = m12[j] - mx * my;
            // sxx + syy is a difference of filtered moments and may come out below zero on flat patches, by about 1e-7 of the
            // squared values: B2 stays positive, C2 = 9e-4, for images of values of order one
            const float A1 = 2.f * mx * my + kC1, A2 = 2.f * sxyc + kC2;
            const float B1 = mx * mx + my * my + kC1, B2 = sxx + syy + kC2;
            const float rb1 = __fdividef(1.0f, B1), rb2 = __fdividef(1.0f, B2);  // B1 >= C1; B2: see above
            const float inv = rb1 * rb2;
            const float s = A1 * A2 * inv;
            const float ds_dmu = 2.f * my * A2 * inv - s * 2.f * mx * rb1;  // sigmas held fixed
            const float ds_dsxx = -s * rb2;
            const float ds_dsxy = 2.f * A1 * inv;
            const size_t p = c * plane + (size_t)y * W + x;
            dm[p] = ds_dmu - 2.f * mx * ds_dsxx - my * ds_dsxy;  // d s / d m1
            dm[3 * plane + p] = ds_dsxx;                        // d s / d m2
            dm[6 * plane + p] = ds_dsxy;                        // d s / d m12
            ss += s;
            const float2 xy = sxy[r + kR][pair_at(col + kR)];
            l1 += fabsf(xy.x - xy.y);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        l1 += __shfl_xor_sync(0xffffffffu, l1, o);
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = (double)l1;
        red[1][threadIdx.x >> 5] = (double)ss;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) {
            a += red[0][w];
            b += red[1][w];
        }
        atomicAdd(&sums[0], a);
        atomicAdd(&sums[1], b);
    }
}

__global__ void __launch_bounds__(kThreads)
k_ssim_bwd(const float* __restrict__ img, const float* __restrict__ tgt, int W, int H, Taps taps, float lam,
           const float* __restrict__ dm, const double* __restrict__ sums, float* __restrict__ grad,
           float* __restrict__ loss_out) {
    __shared__ __align__(16) float2 s01[kInH][kPairs];      // d s / d (m1, m2)
    __shared__ __align__(16) float s2[kInH][kInW + 2];      // and m12
    __shared__ float4 hd[kInH][kTw];                        // row-filtered
    const int x0 = blockIdx.x * kTw, y0 = blockIdx.y * kTh, c = blockIdx.z;
    const size_t plane = (size_t)W * H;
    const double n = 3.0 * (double)plane;
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) {
        // the forward launch has finished: its sums are complete
        const double l1 = sums[0] / n, ssim = sums[1] / n;
        loss_out[0] = (float)((1.0 - lam) * l1 + lam * (1.0 - ssim));
        loss_out[1] = (float)ssim;
    }
    const float* __restrict__ D = dm + c * plane;
    stage(W, H, x0, y0, [&](int r, int col, int64_t o) {
        s01[r][pair_at(col)] = o >= 0 ? make_float2(D[o], D[3 * plane + o]) : make_float2(0.f, 0.f);
        s2[r][col] = o >= 0 ? D[6 * plane + o] : 0.f;
    });
    __syncthreads();
    {
        const int r = threadIdx.x >> 3, t = threadIdx.x & 7;
        F2 a[kCols];
        float b[kCols];
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
            a[j] = f2(0.f);
            b[j] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < kCols + 2 * kR; i += 2) {
            const float4 two = *reinterpret_cast<const float4*>(&s01[r][6 * t + pair_at(i)]);
            const float2 last = *reinterpret_cast<const float2*>(&s2[r][kCols * t + i]);
            const F2 d[2] = {f2(two.x, two.y), f2(two.z, two.w)};
            const float e[2] = {last.x, last.y};
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < kCols; ++j) {
                    const int k = i + h - j;
                    if (k < 0 || k > 2 * kR) continue;
                    a[j] = fma2(f2(taps.w[k]), d[h], a[j]);
                    b[j] = fmaf(taps.w[k], e[h], b[j]);
                }
        }
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
            const float2 v = un(a[j]);
            hd[r][quad_at(kCols * t + j)] = make_float4(v.x, v.y, b[j], 0.f);
        }
    }
    __syncthreads();
    const float inv_n = (float)(1.0 / n);
    const int col = threadIdx.x & 31, r0 = kRows * (threadIdx.x >> 5);
    const int q = quad_at(col);
    F2 a[kRows];
    float b[kRows];
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
        a[j] = f2(0.f);
        b[j] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < kRows + 2 * kR; ++i) {
        const float4 h = hd[min(r0 + i, kInH - 1)][q];
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
            const int k = i - j;
            if (k < 0 || k > 2 * kR) continue;
            a[j] = fma2(f2(taps.w[k]), f2(h.x, h.y), a[j]);
            b[j] = fmaf(taps.w[k], h.z, b[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
        const int r = r0 + j, x = x0 + col, y = y0 + r;
        if (r >= kTh || x >= W || y >= H) continue;
        const size_t p = c * plane + (size_t)y * W + x;
        const float xv = img[p], yv = tgt[p];
        const float2 g = un(a[j]);
        const float d_ssim = g.x + 2.f * xv * g.y + yv * b[j];
        const float d = xv - yv;
        const float sgn = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        grad[p] = ((1.f - lam) * sgn - lam * d_ssim) * inv_n;
    }
}

}  // namespace

int launch_loss_dssim(const float* image, const float* target, int W, int H, float lam, float* dm,
                      double* sums, float* grad, float* loss_out, cudaStream_t s) {
    Taps taps;
    double t[2 * kR + 1], tot = 0.0;
    for (int k = -kR; k <= kR; ++k) tot += t[k + kR] = exp(-(double)(k * k) / (2.0 * 1.5 * 1.5));
    for (int k = 0; k <= 2 * kR; ++k) taps.w[k] = (float)(t[k] / tot);
    const dim3 grid((unsigned)((W + kTw - 1) / kTw), (unsigned)((H + kTh - 1) / kTh), 3);
    cudaMemsetAsync(sums, 0, 2 * sizeof(double), s);
    k_ssim_fwd<<<grid, kThreads, 0, s>>>(image, target, W, H, taps, dm, sums);
    k_ssim_bwd<<<grid, kThreads, 0, s>>>(image, target, W, H, taps, lam, dm, sums, grad, loss_out);
    return 2;
}

}  // namespace pgs
