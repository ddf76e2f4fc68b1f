// K15: the learned initializer's MLP 16-64-64-8 (GELU), BF16 weights and activations, FP32
// accumulation on the tensor cores (mma.sync m16n8k16, bf16 x bf16 -> f32), operands staged in
// shared memory and loaded with ldmatrix (transposed where a product needs the transpose).
//
// At K = 16 / 64 and N = 8 / 64 each layer is a handful of 16x8x16 products per 16 points, and the 128 GELUs
// a point take the time.  Both kernels carry a warp's 16 points through the layers in registers;
// a training step reads the features and targets once and writes only the loss and the weight gradients.
//
// Training kernel, per CTA slice of 64 points (4 warps x 16):
//   forward  Z1 = X W1^T + b1, H1 = gelu(Z1), Z2 = H1 W2^T + b2, H2 = gelu(Z2), Y = H2 W3^T + b3
//   loss     |Y0..2 - t|^2 + (1 - <Y3..6/|Y3..6|, t_q>^2) + (Y7 - t)^2, mean over points
//   backward dH2 = dY W3, dZ2 = dH2 gelu'(Z2), dH1 = dZ2 W2, dZ1 = dH1 gelu'(Z1)
//   weights  dW3 = dY^T H2, dW2 = dZ2^T H1, dW1 = dZ1^T X (split across the warps, accumulated in
//            registers over the CTA's slices, added to the FP32 gradient once per CTA); bias
//            gradients are FP32 sums of the unrounded dY, dZ2, dZ1.
// BF16 rounding points: X, weights, H1, H2 and the gradients fed to products (dY, dZ2, dZ1).
#include <cuda_bf16.h>

#include "pgs_internal.cuh"

namespace pgs {
namespace {

constexpr int kIn = 16, kHid = 64, kOut = 8;
constexpr int kWarps = 4, kRows = 16 * kWarps;  // points per CTA slice
constexpr int LD16 = kIn + 8, LD64 = kHid + 8;  // padded bf16 row strides (16-byte multiples)
constexpr int kParams = kHid * kIn + kHid + kHid * kHid + kHid + kOut * kHid + kOut;  // 5768

// offsets of the flat FP32 parameter vector [W1 | b1 | W2 | b2 | W3 | b3]
constexpr int oW1 = 0, ob1 = oW1 + kHid * kIn, oW2 = ob1 + kHid, ob2 = oW2 + kHid * kHid,
              oW3 = ob2 + kHid, ob3 = oW3 + kOut * kHid;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm_x4(uint32_t r[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x2_t(uint32_t r[2], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(r[0]), "=r"(r[1]) : "r"(smem_addr(p)));
}
__device__ __forceinline__ void mma(float c[4], const uint32_t a[4], const uint32_t b[2]) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void mma_k8(float c[4], const uint32_t a[2], uint32_t b) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(b));
}

// A fragment of the transpose: A[m][k] = S[k][m], block rows (data) k0.., cols m0..
__device__ __forceinline__ void frag_a_t(uint32_t a[4], const __nv_bfloat16* S, int ld, int k0, int m0) {
    const int l = threadIdx.x & 31, i = l >> 3;
    ldsm_x4_t(a, S + (size_t)(k0 + (i >> 1) * 8 + (l & 7)) * ld + m0 + (i & 1) * 8);
}
// 1 + erf(x) by the rational approximation 7.1.26 of Abramowitz & Stegun (Handbook of
// Mathematical Functions, 1964): for x >= 0, erf(x) = 1 - (a1 s + a2 s^2 + ... + a5 s^5) e^{-x^2}
// with s = 1 / (1 + p x) and |error| <= 1.5e-7, far below the BF16 rounding of the activations.
// Evaluated as q = polynomial * e^{-x^2}, 1 + erf(x) = 2 - q for x >= 0 and q for x < 0 (the
// odd symmetry), so the left tail keeps its relative accuracy instead of cancelling.
//
// Two arguments at a time, in the halves: returns Phi of both, Phi(z) = (1 + erf(z / sqrt 2)) / 2 (the
// factor 1/2 is exact in the coefficients), and e = e^{-z^2 / 2}.
__device__ __forceinline__ F2 phi2(F2 z, F2& e) {
    const F2 x = mul2(z, f2(0.70710678118654752f));
    const float2 xv = un(x);
    // ex2 and rcp with flushed subnormals: the arguments of rcp are at least 1, and where e^{-x^2} is below 2^-126
    // (z < -13.2) the activation, itself below 2e-37, becomes zero.  Keeping those costs 471 -> 539 us at 6.4 M points.
    const float2 w = un(mul2(mul2(x, x), f2(-1.4426950408889634f)));
    F2 s;
    {
        float a, b;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(fmaf(0.3275911f, fabsf(xv.x), 1.0f)));
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(fmaf(0.3275911f, fabsf(xv.y), 1.0f)));
        s = f2(a, b);
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(w.x));
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(w.y));
        e = f2(a, b);
    }
    F2 poly = fma2(f2(0.5f * 1.061405429f), s, f2(0.5f * -1.453152027f));
    poly = fma2(poly, s, f2(0.5f * 1.421413741f));
    poly = fma2(poly, s, f2(0.5f * -0.284496736f));
    poly = fma2(poly, s, f2(0.5f * 0.254829592f));
    const F2 ps = mul2(poly, s);
    const float2 q = un(mul2(ps, e));
    return f2(xv.x >= 0.0f ? __fsub_rn(1.0f, q.x) : q.x, xv.y >= 0.0f ? __fsub_rn(1.0f, q.y) : q.y);
}
// GELU in the erf form, z Phi(z), and with its derivative d = Phi(z) + z phi(z)
__device__ __forceinline__ F2 gelu2(F2 z) {
    F2 e;
    return mul2(z, phi2(z, e));
}
__device__ __forceinline__ F2 gelu2(F2 z, F2& d) {
    F2 e;
    const F2 p = phi2(z, e);
    d = fma2(mul2(z, e), f2(0.3989422804014327f), p);
    return mul2(z, p);
}

__device__ __forceinline__ uint32_t pack_bf16(F2 v) {
    const float2 u = un(v);
    const __nv_bfloat162 p = __floats2bfloat162_rn(u.x, u.y);
    return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ F2 biased(const float* c, const float* bias) {
    const float2 b = *reinterpret_cast<const float2*>(bias);
    return add2(f2(c[0], c[1]), f2(b.x, b.y));
}
__device__ __forceinline__ void clear(float C[4]) { C[0] = C[1] = C[2] = C[3] = 0.f; }

struct WeightSmem {
    __nv_bfloat16 W1[kHid * LD16], W2[kHid * LD64], W3[kOut * LD64];
    float b1[kHid], b2[kHid], b3[kOut];
};

// By 32 * kWarps threads, all loads of a matrix in flight.
__device__ __forceinline__ void load_weights(WeightSmem& S, const __nv_bfloat16* __restrict__ W1,
                                             const __nv_bfloat16* __restrict__ W2, const __nv_bfloat16* __restrict__ W3,
                                             const float* __restrict__ b1, const float* __restrict__ b2,
                                             const float* __restrict__ b3) {
    constexpr int kStep = 32 * kWarps;
    __nv_bfloat16 r1[kHid * kIn / kStep], r2[kHid * kHid / kStep], r3[kOut * kHid / kStep];
#pragma unroll
    for (int i = 0; i < kHid * kHid / kStep; ++i) r2[i] = W2[i * kStep + threadIdx.x];
#pragma unroll
    for (int i = 0; i < kHid * kIn / kStep; ++i) r1[i] = W1[i * kStep + threadIdx.x];
#pragma unroll
    for (int i = 0; i < kOut * kHid / kStep; ++i) r3[i] = W3[i * kStep + threadIdx.x];
    if (threadIdx.x < kHid) {
        S.b1[threadIdx.x] = b1[threadIdx.x];
        S.b2[threadIdx.x] = b2[threadIdx.x];
    }
    if (threadIdx.x < kOut) S.b3[threadIdx.x] = b3[threadIdx.x];
    const int row = threadIdx.x / kHid, col = threadIdx.x % kHid;
#pragma unroll
    for (int i = 0; i < kHid * kHid / kStep; ++i) S.W2[(i * (kStep / kHid) + row) * LD64 + col] = r2[i];
#pragma unroll
    for (int i = 0; i < kOut * kHid / kStep; ++i) S.W3[(i * (kStep / kHid) + row) * LD64 + col] = r3[i];
#pragma unroll
    for (int i = 0; i < kHid * kIn / kStep; ++i)
        S.W1[(i * (kStep / kIn) + threadIdx.x / kIn) * LD16 + threadIdx.x % kIn] = r1[i];
}

// the words of lane (g, t) of the 16 x 16 A fragment of points sl * 16 ..
__device__ __forceinline__ void load_points(uint32_t a[4], const __nv_bfloat16* __restrict__ x, int64_t n, int64_t p0) {
    const int lane = threadIdx.x & 31, t = lane & 3;
    const uint32_t* __restrict__ xw = reinterpret_cast<const uint32_t*>(x);  // 8 words per point
    const int64_t pa = p0 + (lane >> 2), pb = pa + 8;
    a[0] = pa < n ? xw[pa * 8 + t] : 0u;
    a[1] = pb < n ? xw[pb * 8 + t] : 0u;
    a[2] = pa < n ? xw[pa * 8 + t + 4] : 0u;
    a[3] = pb < n ? xw[pb * 8 + t + 4] : 0u;
}

// Inference: activations never leave registers.  The f32 accumulator fragment of a 16 x 8
// product tile (rows g, g + 8; columns 2t, 2t + 1 of lane (g, t)) is, after bias, GELU and
// packing column pairs to bf16x2 exactly the A fragment of the next layer's 16 x 16 k-tile (the
// k-tile of columns 16 kk.. is made of n-tiles 2 kk and 2 kk + 1), so each warp carries its 16
// points through the three layers with no shared-memory round trip; only the weights are staged.
// The FP32 and special-function pipes bound it (56 % and 51 % busy, issue 59 %): 710 us for 6.4 M points with
// scalar arithmetic and a subnormal path around every special function (issue 83 %), 470 us with packed pairs.
// Four CTAs an SM: at six or more, with the registers that leaves, 520 us and up.

// bias and GELU of two neighbouring 16 x 8 accumulator tiles, packed into one A fragment of the next layer
__device__ __forceinline__ void activate(const float C[2][4], const float* bias, uint32_t A[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) A[e] = pack_bf16(gelu2(biased(C[e >> 1] + 2 * (e & 1), bias + 8 * (e >> 1))));
}

__global__ void __launch_bounds__(32 * kWarps, 4)
k_mlp_forward(const __nv_bfloat16* __restrict__ x, int64_t n, const __nv_bfloat16* __restrict__ W1,
              const __nv_bfloat16* __restrict__ W2, const __nv_bfloat16* __restrict__ W3,
              const float* __restrict__ b1, const float* __restrict__ b2, const float* __restrict__ b3,
              float* __restrict__ out) {
    __shared__ __align__(16) WeightSmem S;
    load_weights(S, W1, W2, W3, b1, b2, b3);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // four 8 x 8 weight tiles at a time: two products' B fragments, of output tiles j and j + 1 (first layer)
    // or of k-tiles kk and kk + 1
    const __nv_bfloat16* const w1 = S.W1 + (size_t)((lane & 7) + (lane >> 4) * 8) * LD16 + ((lane >> 3) & 1) * 8;
    const __nv_bfloat16* const w2 = S.W2 + (size_t)(lane & 7) * LD64 + (lane >> 3) * 8;
    const __nv_bfloat16* const w3 = S.W3 + (size_t)(lane & 7) * LD64 + (lane >> 3) * 8;
    const int64_t slices = (n + 15) / 16, step = (int64_t)gridDim.x * kWarps;
    int64_t sl = (int64_t)blockIdx.x * kWarps + warp;
    uint32_t a[4];
    load_points(a, x, n, sl * 16);
    for (; sl < slices; sl += step) {
        uint32_t A[4][4], b[4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float C[2][4];
            clear(C[0]);
            clear(C[1]);
            ldsm_x4(b, w1 + 16 * kk * LD16);
            mma(C[0], a, b);
            mma(C[1], a, b + 2);
            activate(C, S.b1 + 16 * kk + 2 * t, A[kk]);
        }
        load_points(a, x, n, (sl + step) * 16);  // the next points, while these are carried through
        float y[4];
        clear(y);
        uint32_t b3[4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float C[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                clear(C[j]);
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    ldsm_x4(b, w2 + 8 * (2 * kk + j) * LD64 + 16 * k);
                    mma(C[j], A[k], b);
                    mma(C[j], A[k + 1], b + 2);
                }
            }
            uint32_t H[4];
            activate(C, S.b2 + 16 * kk + 2 * t, H);
            if (kk % 2 == 0) ldsm_x4(b3, w3 + 16 * kk);
            mma(y, H, b3 + 2 * (kk % 2));
        }
        const int64_t pa = sl * 16 + g, pb = pa + 8;
        const int c = 2 * t;
        if (pa < n) *reinterpret_cast<float2*>(out + pa * kOut + c) = make_float2(y[0] + S.b3[c], y[1] + S.b3[c + 1]);
        if (pb < n) *reinterpret_cast<float2*>(out + pb * kOut + c) = make_float2(y[2] + S.b3[c], y[3] + S.b3[c + 1]);
    }
}

// What a slice's weight gradients contract over its 64 points, which the four warps exchange: BF16 rows of
// 4-byte words whose padding puts the fragments' stores and loads on different banks.
struct SliceSmem {
    __nv_bfloat16 H1[kRows * LD64], H2[kRows * LD64], dZ2[kRows * LD64], dZ1[kRows * LD64];
    __nv_bfloat16 X[kRows * LD16], dY[kRows * kOut];
};
struct TrainSmem {
    WeightSmem w;
    SliceSmem s[2];
};

__device__ __forceinline__ float quad_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// A slice's forward and backward chain stays in a warp's registers (accumulator fragments become the next
// product's A fragments, the GELU derivatives of the forward pass wait in FP32 registers); shared memory
// holds only what the weight gradients contract, in two buffers, so that a slice needs one barrier.  With
// every activation in shared memory, FP32 Z1 and Z2 among them, and the derivative's erf and exponential
// evaluated again, a pass over 65,536 points took 70 us; 35 us now, two CTAs an SM by registers, bound by latency
// (issue 22 %): 1,024 slices are 3.4 per CTA.
__global__ void __launch_bounds__(32 * kWarps, 2)
k_mlp_train(const __nv_bfloat16* __restrict__ x, const float* __restrict__ target, int64_t n,
            const __nv_bfloat16* __restrict__ W1, const __nv_bfloat16* __restrict__ W2,
            const __nv_bfloat16* __restrict__ W3, const float* __restrict__ b1, const float* __restrict__ b2,
            const float* __restrict__ b3, float* __restrict__ grad, double* __restrict__ loss_sum) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    TrainSmem& T = *reinterpret_cast<TrainSmem*>(s_raw);
    WeightSmem& W = T.w;
    load_weights(W, W1, W2, W3, b1, b2, b3);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int r0 = 16 * warp, row = r0 + g;
    const float inv_n = 1.0f / (float)n;
    // rows of four 8 x 8 tiles for ldmatrix: lanes 8 i .. 8 i + 7 give tile i's
    const int tr = lane & 7, ti = lane >> 3;
    const __nv_bfloat16* const w1 = W.W1 + (tr + (ti >> 1) * 8) * LD16 + (ti & 1) * 8;  // n-tiles j, j + 1
    const __nv_bfloat16* const w2 = W.W2 + tr * LD64 + ti * 8;                          // k-tiles k, k + 1
    const __nv_bfloat16* const w3 = W.W3 + tr * LD64 + ti * 8;
    const int back = (tr + (ti & 1) * 8) * LD64 + (ti >> 1) * 8;  // of a transposed pair of n-tiles, 16 rows
    float accW2[8][4], accW1[2][4], accW3[4];
    F2 db1[8], db2[8];  // columns 8 j + 2 t, + 1
    float db3[2] = {0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        clear(accW2[j]);
        db1[j] = db2[j] = f2(0.f);
    }
    clear(accW1[0]);
    clear(accW1[1]);
    clear(accW3);
    double lsum = 0.0;

    int buf = 0;
    uint32_t a[4];
    float tg[2][2];
    auto fetch = [&](int64_t p) {
        load_points(a, x, n, p + r0);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                tg[r][c] = p + row + 8 * r < n ? target[(p + row + 8 * r) * kOut + 2 * t + c] : 0.f;
    };
    const int64_t step = (int64_t)gridDim.x * kRows;
    fetch((int64_t)blockIdx.x * kRows);
    for (int64_t p0 = (int64_t)blockIdx.x * kRows; p0 < n; p0 += step, buf ^= 1) {
        SliceSmem& S = T.s[buf];
        uint32_t b[4], A[4][4];
        const bool in[2] = {p0 + row < n, p0 + row + 8 < n};
        // word e of an A fragment at columns c0..: rows row, row + 8, then the same 8 columns on
        auto put = [&](__nv_bfloat16* M, int ld, int c0, const uint32_t w[4]) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                *reinterpret_cast<uint32_t*>(M + (row + 8 * (e & 1)) * ld + c0 + 8 * (e >> 1) + 2 * t) = w[e];
        };
        put(S.X, LD16, 0, a);
        F2 g1[4][4], g2[4][4];  // gelu' at the pairs of the fragments' words
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float C[2][4];
            clear(C[0]);
            clear(C[1]);
            ldsm_x4(b, w1 + 16 * kk * LD16);
            mma(C[0], a, b);
            mma(C[1], a, b + 2);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                A[kk][e] = pack_bf16(
                    gelu2(biased(C[e >> 1] + 2 * (e & 1), W.b1 + 16 * kk + 8 * (e >> 1) + 2 * t), g1[kk][e]));
            put(S.H1, LD64, 16 * kk, A[kk]);
        }
        float y[4];
        clear(y);
        uint32_t bw[4];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float C[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                clear(C[j]);
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    ldsm_x4(b, w2 + 8 * (2 * kk + j) * LD64 + 16 * k);
                    mma(C[j], A[k], b);
                    mma(C[j], A[k + 1], b + 2);
                }
            }
            uint32_t H[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                H[e] = pack_bf16(
                    gelu2(biased(C[e >> 1] + 2 * (e & 1), W.b2 + 16 * kk + 8 * (e >> 1) + 2 * t), g2[kk][e]));
            put(S.H2, LD64, 16 * kk, H);
            if (kk % 2 == 0) ldsm_x4(bw, w3 + 16 * kk);
            mma(y, H, bw + 2 * (kk % 2));
        }
        // loss head: the four lanes of a row hold its outputs 2 t, 2 t + 1; 3..6 are the quaternion
        const bool qa = t >= 2, qb = t == 1 || t == 2;
        uint32_t dyw[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const float ya = y[2 * r] + W.b3[2 * t], yb = y[2 * r + 1] + W.b3[2 * t + 1];
            const float qn = sqrtf(quad_sum((qa ? ya * ya : 0.f) + (qb ? yb * yb : 0.f)));
            const float iq = qn > 0.f ? 1.0f / qn : 0.f;
            const float ua = ya * iq, ub = yb * iq;
            const float f = quad_sum((qa ? ua * tg[r][0] : 0.f) + (qb ? ub * tg[r][1] : 0.f));
            const float dqa = -2.f * f * tg[r][0], dqb = -2.f * f * tg[r][1];
            const float dot = quad_sum((qa ? dqa * ua : 0.f) + (qb ? dqb * ub : 0.f));
            const float da = ya - tg[r][0], db = yb - tg[r][1];
            float dya = qa ? (dqa - ua * dot) * iq * inv_n : 2.f * da * inv_n;
            float dyb = qb ? (dqb - ub * dot) * iq * inv_n : 2.f * db * inv_n;
            if (!in[r]) dya = dyb = 0.f;
            if (in[r]) lsum += (double)((qa ? 0.f : da * da) + (qb ? 0.f : db * db) + (t == 0 ? 1.f - f * f : 0.f));
            db3[0] += dya;
            db3[1] += dyb;
            dyw[r] = pack_bf16(f2(dya, dyb));
            *reinterpret_cast<uint32_t*>(S.dY + (row + 8 * r) * kOut + 2 * t) = dyw[r];
        }
        fetch(p0 + step);  // the next slice's, under the backward pass
        // dZ2 = (dY W3) gelu'(Z2)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            if (kk % 2 == 0) ldsm_x4_t(bw, w3 + 16 * kk);
            float C[2][4];
            clear(C[0]);
            clear(C[1]);
            mma_k8(C[0], dyw, bw[2 * (kk % 2)]);
            mma_k8(C[1], dyw, bw[2 * (kk % 2) + 1]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float* c = C[e >> 1] + 2 * (e & 1);
                const F2 dz = mul2(f2(c[0], c[1]), g2[kk][e]);
                db2[2 * kk + (e >> 1)] = add2(db2[2 * kk + (e >> 1)], dz);
                A[kk][e] = pack_bf16(dz);
            }
            put(S.dZ2, LD64, 16 * kk, A[kk]);
        }
        // dZ1 = (dZ2 W2) gelu'(Z1)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            float C[2][4];
            clear(C[0]);
            clear(C[1]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                ldsm_x4_t(b, W.W2 + back + 16 * k * LD64 + 16 * kk);
                mma(C[0], A[k], b);
                mma(C[1], A[k], b + 2);
            }
            uint32_t D[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float* c = C[e >> 1] + 2 * (e & 1);
                const F2 dz = mul2(f2(c[0], c[1]), g1[kk][e]);
                db1[2 * kk + (e >> 1)] = add2(db1[2 * kk + (e >> 1)], dz);
                D[e] = pack_bf16(dz);
            }
            put(S.dZ1, LD64, 16 * kk, D);
        }
        // The other buffer's readers are done: each warp came here after its products of the slice before.
        __syncthreads();
        // weight gradients over the slice's 64 points: this warp's 16 rows of dW2 and dW1, and columns of dW3
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            uint32_t at[4];
            frag_a_t(at, S.dZ2, LD64, 16 * kk, r0);
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                ldsm_x4_t(b, S.H1 + back + 16 * kk * LD64 + 8 * j);
                mma(accW2[j], at, b);
                mma(accW2[j + 1], at, b + 2);
            }
            frag_a_t(at, S.dZ1, LD64, 16 * kk, r0);
            ldsm_x4_t(b, S.X + (16 * kk + tr + (ti & 1) * 8) * LD16 + (ti >> 1) * 8);
            mma(accW1[0], at, b);
            mma(accW1[1], at, b + 2);
            frag_a_t(at, S.H2, LD64, 16 * kk, r0);  // transposed: rows are hidden units, columns outputs
            ldsm_x2_t(b, S.dY + (16 * kk + tr + (ti & 1) * 8) * kOut);
            mma(accW3, at, b);
        }
    }
    // flush: weight gradients (C fragment rows g / g + 8, cols 2t, 2t + 1)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int m = row + (e >> 1) * 8, c = 2 * t + (e & 1);
#pragma unroll
        for (int j = 0; j < 8; ++j) atomicAdd(&grad[oW2 + m * kHid + 8 * j + c], accW2[j][e]);
#pragma unroll
        for (int j = 0; j < 2; ++j) atomicAdd(&grad[oW1 + m * kIn + 8 * j + c], accW1[j][e]);
        atomicAdd(&grad[oW3 + c * kHid + m], accW3[e]);
    }
    // bias gradients: reduce over the lanes sharing t (rows)
    auto rows_sum = [&](float v) {
        for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float2 u = un(db1[j]), v = un(db2[j]);
        const float s[4] = {rows_sum(u.x), rows_sum(u.y), rows_sum(v.x), rows_sum(v.y)};
        if (g == 0)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                atomicAdd(&grad[ob1 + 8 * j + 2 * t + q], s[q]);
                atomicAdd(&grad[ob2 + 8 * j + 2 * t + q], s[2 + q]);
            }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float s = rows_sum(db3[q]);
        if (g == 0) atomicAdd(&grad[ob3 + 2 * t + q], s);
    }
    for (int o = 1; o < 32; o <<= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) atomicAdd(loss_sum, lsum);
}

// Adam on the FP32 master parameters; refreshes the BF16 weight copies and zeroes the gradient.
__global__ void k_mlp_adam(float* __restrict__ master, float* __restrict__ grad, float* __restrict__ m,
                           float* __restrict__ v, float lr, float b1, float b2, float eps, float bc1,
                           float bc2, __nv_bfloat16* __restrict__ W1, __nv_bfloat16* __restrict__ W2,
                           __nv_bfloat16* __restrict__ W3) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < kParams; k += gridDim.x * blockDim.x) {
        const float gk = grad[k];
        const float mm = b1 * m[k] + (1.f - b1) * gk;
        const float vv = b2 * v[k] + (1.f - b2) * gk * gk;
        m[k] = mm;
        v[k] = vv;
        const float p = master[k] - lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
        master[k] = p;
        grad[k] = 0.f;
        if (k < ob1) W1[k - oW1] = __float2bfloat16_rn(p);
        else if (k >= oW2 && k < ob2) W2[k - oW2] = __float2bfloat16_rn(p);
        else if (k >= oW3 && k < ob3) W3[k - oW3] = __float2bfloat16_rn(p);
    }
}

__global__ void k_mlp_pack(const float* __restrict__ master, __nv_bfloat16* __restrict__ W1,
                           __nv_bfloat16* __restrict__ W2, __nv_bfloat16* __restrict__ W3) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < kParams; k += gridDim.x * blockDim.x) {
        const float p = master[k];
        if (k < ob1) W1[k - oW1] = __float2bfloat16_rn(p);
        else if (k >= oW2 && k < ob2) W2[k - oW2] = __float2bfloat16_rn(p);
        else if (k >= oW3 && k < ob3) W3[k - oW3] = __float2bfloat16_rn(p);
    }
}

int grid_for(int64_t n) {
    static int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v;
    }();
    const int64_t slices = (n + kRows - 1) / kRows;
    return (int)std::max<int64_t>(1, std::min<int64_t>(slices, (int64_t)sms * 2));
}

void enable_smem() {
    static bool done = [] {
        cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
        return true;
    }();
    (void)done;
}

}  // namespace

int mlp_param_count() { return kParams; }

int launch_mlp_forward(const void* x, int64_t n, const float* master, const void* W1, const void* W2,
                       const void* W3, float* out, cudaStream_t s) {
    if (n <= 0) return 0;
    enable_smem();
    static int grid = [] {
        int dev = 0, sms = 0, per_sm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mlp_forward, 32 * kWarps, 0);
        return sms * (per_sm > 0 ? per_sm : 1);
    }();
    const int64_t slices = (n + 15) / 16;
    const int64_t blocks = std::min<int64_t>(grid, (slices + kWarps - 1) / kWarps);
    k_mlp_forward<<<(unsigned)blocks, 32 * kWarps, 0, s>>>(
        static_cast<const __nv_bfloat16*>(x), n, static_cast<const __nv_bfloat16*>(W1),
        static_cast<const __nv_bfloat16*>(W2), static_cast<const __nv_bfloat16*>(W3), master + ob1,
        master + ob2, master + ob3, out);
    return 1;
}

int launch_mlp_train(const void* x, const float* target, int64_t n, const float* master, const void* W1,
                     const void* W2, const void* W3, float* grad, double* loss_sum, cudaStream_t s) {
    if (n <= 0) return 0;
    enable_smem();
    k_mlp_train<<<grid_for(n), 32 * kWarps, sizeof(TrainSmem), s>>>(
        static_cast<const __nv_bfloat16*>(x), target, n, static_cast<const __nv_bfloat16*>(W1),
        static_cast<const __nv_bfloat16*>(W2), static_cast<const __nv_bfloat16*>(W3), master + ob1,
        master + ob2, master + ob3, grad, loss_sum);
    return 1;
}

int launch_mlp_adam(float* master, float* grad, float* m, float* v, float lr, float b1, float b2,
                    float eps, int64_t t, void* W1, void* W2, void* W3, cudaStream_t s) {
    const float bc1 = (float)(1.0 - pow((double)b1, (double)t));
    const float bc2 = (float)(1.0 - pow((double)b2, (double)t));
    k_mlp_adam<<<(kParams + 255) / 256, 256, 0, s>>>(master, grad, m, v, lr, b1, b2, eps, bc1, bc2,
                                                      static_cast<__nv_bfloat16*>(W1),
                                                      static_cast<__nv_bfloat16*>(W2),
                                                      static_cast<__nv_bfloat16*>(W3));
    return 1;
}

int launch_mlp_pack(const float* master, void* W1, void* W2, void* W3, cudaStream_t s) {
    k_mlp_pack<<<(kParams + 255) / 256, 256, 0, s>>>(master, static_cast<__nv_bfloat16*>(W1),
                                                      static_cast<__nv_bfloat16*>(W2),
                                                      static_cast<__nv_bfloat16*>(W3));
    return 1;
}

}  // namespace pgs
