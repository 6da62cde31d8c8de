// Register DFTs of the mixed-radix kernels (radices 2 .. 16) for one transform
// per thread (float2) or two side by side (C2), and the index helpers the
// kernels share.
#pragma once

#include "fft_common.cuh"
#include "fft_internal.h"

namespace gb300fft {
namespace mixed {

// cos and sin of 2 pi m / R, evaluated by the compiler: the angle is split
// in integers into a quadrant k (multiples of pi/2) and a remainder phi in
// [0, pi/2), whose sine and cosine are Taylor series summed in double (error
// below 1e-15; exactly 0 and +-1 on the axes), then rounded once to float.
constexpr double kPiD = 3.14159265358979323846264338327950288;
__host__ __device__ constexpr double taylor_sin(double x) {
    double term = x, sum = x;
    for (int k = 1; k < 30; ++k) {
        term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double taylor_cos(double x) {
    double term = 1.0, sum = 1.0;
    for (int k = 1; k < 30; ++k) {
        term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double cos_2pi(int m, int R) {
    const long long q = ((long long)(m % R) + R) % R, t = 4 * q, k = t / R, rem = t - k * R;
    const double phi = (kPiD / 2) * (double)rem / (double)R;
    return k == 0 ? taylor_cos(phi) : k == 1 ? -taylor_sin(phi) : k == 2 ? -taylor_cos(phi) : taylor_sin(phi);
}
__host__ __device__ constexpr double sin_2pi(int m, int R) {
    const long long q = ((long long)(m % R) + R) % R, t = 4 * q, k = t / R, rem = t - k * R;
    const double phi = (kPiD / 2) * (double)rem / (double)R;
    return k == 0 ? taylor_sin(phi) : k == 1 ? taylor_cos(phi) : k == 2 ? -taylor_sin(phi) : -taylor_cos(phi);
}

// cos and sin of 2 pi j / R for j = 1 .. (R-1)/2, rounded to float.  Built
// only in constant initialisers (a constexpr variable), so the double-precision
// series never reach device code.
template <int R>
struct OddRoots {
    float c[(R - 1) / 2], s[(R - 1) / 2];
};
template <int R>
__host__ __device__ constexpr OddRoots<R> odd_roots() {
    OddRoots<R> w{};
    for (int j = 1; j <= (R - 1) / 2; ++j) {
        w.c[j - 1] = (float)cos_2pi(j, R);
        w.s[j - 1] = (float)sin_2pi(j, R);
    }
    return w;
}

// Forward R-point DFT for odd prime R, legs paired as (k, R - k):
//   y_m     = a_0 + sum_k t_k cos(2 pi k m / R) - i sum_k d_k sin(2 pi k m / R)
//   y_{R-m} = a_0 + sum_k t_k cos(2 pi k m / R) + i sum_k d_k sin(2 pi k m / R)
// with t_k = a_k + a_{R-k}, d_k = a_k - a_{R-k}, k, m = 1 .. (R-1)/2.
// a + c b, for one transform (float2) or two (C2)
__device__ __forceinline__ float2 axpy(float c, float2 b, float2 a) {
    return make_float2(fmaf(c, b.x, a.x), fmaf(c, b.y, a.y));
}
__device__ __forceinline__ C2 axpy(float c, C2 b, C2 a) { return {fma2(both(c), b.re, a.re), fma2(both(c), b.im, a.im)}; }
__device__ __forceinline__ float2 scaled(float c, float2 b) { return make_float2(c * b.x, c * b.y); }
__device__ __forceinline__ C2 scaled(float c, C2 b) { return {mul2(both(c), b.re), mul2(both(c), b.im)}; }

template <int R, class V>
__device__ __forceinline__ void dft_odd(V *a) {
    constexpr int H = (R - 1) / 2;
    constexpr OddRoots<R> W = odd_roots<R>();
    V t[H], d[H];
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        t[k - 1] = cadd(a[k], a[R - k]);
        d[k - 1] = csub(a[k], a[R - k]);
    }
    V y0 = a[0];
#pragma unroll
    for (int k = 0; k < H; ++k) y0 = cadd(y0, t[k]);
    V y[R];
    y[0] = y0;
#pragma unroll
    for (int m = 1; m <= H; ++m) {
        V A = a[0], B;
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            const int q = (k * m) % R;  // angle index, folded into 1 .. H
            const int j = q <= H ? q : R - q;
            const float c = W.c[j - 1];
            const float sn = q <= H ? W.s[j - 1] : -W.s[j - 1];
            A = axpy(c, t[k - 1], A);
            B = k == 1 ? scaled(sn, d[k - 1]) : axpy(sn, d[k - 1], B);
        }
        y[m] = sub_i(A, B);  // A - i B
        y[R - m] = add_i(A, B);
    }
#pragma unroll
    for (int k = 0; k < R; ++k) a[k] = y[k];
}

// x * w_R^M with w_R = exp(-2 pi i / R); powers of -i are exact swaps
template <int M, int R>
__device__ __forceinline__ float2 mul_w(float2 x) {
    if constexpr ((4 * M) % R == 0) {
        constexpr int k = ((4 * M) / R) % 4;
        if constexpr (k == 0) return x;
        else if constexpr (k == 1) return make_float2(x.y, -x.x);
        else if constexpr (k == 2) return make_float2(-x.x, -x.y);
        else return make_float2(-x.y, x.x);
    } else {
        constexpr float wr = (float)cos_2pi(M, R), wi = (float)-sin_2pi(M, R);
        return make_float2(fmaf(x.x, wr, -x.y * wi), fmaf(x.x, wi, x.y * wr));
    }
}

template <int M, int R>
__device__ __forceinline__ C2 mul_w(C2 x) {
    if constexpr ((4 * M) % R == 0) {
        constexpr int k = ((4 * M) / R) % 4;
        const C2 zero = {both(0.f), both(0.f)};
        if constexpr (k == 0) return x;
        else if constexpr (k == 1) return sub_i(zero, x);
        else if constexpr (k == 2) return csub(zero, x);
        else return add_i(zero, x);
    } else {
        constexpr float wr = (float)cos_2pi(M, R), wi = (float)-sin_2pi(M, R);
        return {fma2(x.im, both(-wi), mul2(x.re, both(wr))), fma2(x.re, both(wi), mul2(x.im, both(wr)))};
    }
}

template <int R, class V>
__device__ __forceinline__ void dft_any(V *a);

// R = R1 R2 points in registers, natural order in and out: with input index
// i2 + R2 i1 and output index k1 + R1 k2, w_R^{ik} = w_R1^{i1 k1} w_R^{i2 k1}
// w_R2^{i2 k2}, so: R2 transforms of length R1 (over i1), the inner twiddles
// w_R^{i2 k1} (compile-time constants), R1 transforms of length R2 (over i2).
template <int R1, int R2, int I2, int K1, class V>
__device__ __forceinline__ void dft_2lvl_tw(const V *t, V *b) {
    if constexpr (K1 < R1) {
        b[I2 * R1 + K1] = mul_w<I2 * K1, R1 * R2>(t[K1]);
        dft_2lvl_tw<R1, R2, I2, K1 + 1>(t, b);
    }
}
template <int R1, int R2, int I2 = 0, class V>
__device__ __forceinline__ void dft_2lvl_cols(const V *a, V *b) {
    if constexpr (I2 < R2) {
        V t[R1];
#pragma unroll
        for (int i1 = 0; i1 < R1; ++i1) t[i1] = a[I2 + R2 * i1];
        dft_any<R1>(t);
        dft_2lvl_tw<R1, R2, I2, 0>(t, b);
        dft_2lvl_cols<R1, R2, I2 + 1>(a, b);
    }
}
template <int R1, int R2, class V>
__device__ __forceinline__ void dft_2lvl(V *a) {
    V b[R1 * R2];
    dft_2lvl_cols<R1, R2>(a, b);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
        V t[R2];
#pragma unroll
        for (int i2 = 0; i2 < R2; ++i2) t[i2] = b[i2 * R1 + k1];
        dft_any<R2>(t);
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) a[k1 + R1 * k2] = t[k2];
    }
}

template <int R, class V>
__device__ __forceinline__ void dft_any(V *a) {
    if constexpr ((R & (R - 1)) == 0) dft<R>(a);
    else if constexpr (R == 6) dft_2lvl<2, 3>(a);
    else if constexpr (R == 9) dft_2lvl<3, 3>(a);
    else if constexpr (R == 10) dft_2lvl<2, 5>(a);
    else if constexpr (R == 12) dft_2lvl<4, 3>(a);
    else if constexpr (R == 14) dft_2lvl<2, 7>(a);
    else if constexpr (R == 15) dft_2lvl<3, 5>(a);
    else dft_odd<R>(a);
}

// x / d for x * d < 2^32 by a multiply-high with m = ceil(2^32 / d) (d >= 2);
// d = 1 passes x through
__device__ __forceinline__ int fdiv(int x, int d, uint32_t m) {
    return d == 1 ? x : (int)__umulhi((uint32_t)x, m);
}

// Twiddle-table entries per butterfly of a radix-R stage: R - 1 rounded up
// to even, so each butterfly's twiddles are whole 16-byte pairs.
__host__ __device__ constexpr int mixed_tw_stride(int R) { return (R - 1 + 1) & ~1; }

// w_n^e from the two factor tables, w_n^e = hi[e >> L] lo[e & (2^L - 1)]
__device__ __forceinline__ float2 fs_root(const FourStepB &fs, int e) {
    return cmul(__ldg(fs.hi + (e >> fs.lshift)), __ldg(fs.lo + (e & fs.lmask)));
}

}  // namespace mixed
}  // namespace gb300fft
