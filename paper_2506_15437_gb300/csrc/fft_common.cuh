// Device building blocks shared by the gb300fft kernels (sm_103a).
//
// The transform is the radix-2^k Cooley-Tukey FFT of the paper's Section 2.2
// (Fig. 2, Listing 1) in its self-sorting (Stockham) arrangement: every
// butterfly stage reads its operands in the order that stage needs and writes
// its results straight into the order the NEXT stage needs.  That is the
// paper's "one reordering per step" idea (Section 4, Fig. 5) taken to its end
// point: the reordering is the address arithmetic of the stage's loads and
// stores, the intermediate orders live only in shared memory and registers,
// and no separate bit-reversal pass or HBM round trip exists.
//
// Twiddle tables: stage s >= 1 (radix R, span Ns) stores, for pair k < R/2
// and m < Ns, the float4 (w^{(2k+1) m}, w^{(2k+2) m}) with w = w_{Ns*R}, at
// float4 index k*Ns + m, so a warp's threads (consecutive m) load adjacent
// 16-byte words.
//
// Stage s of a length-N transform has radix R and span Ns = R_0 * ... * R_{s-1}.
// Butterfly j (0 <= j < N/R), with m = j mod Ns, reads a_r = d[j + r*N/R],
// multiplies a_r by w_{Ns*R}^{r*m} (w_K = exp(-2*pi*i/K)), takes the length-R
// DFT b_k = sum_r a_r w_R^{r*k}, and writes b_k to d'[(j - m)*R + m + k*Ns].
// The first stage (Ns = 1) needs no twiddles; the last one (Ns*R = N) writes
// natural order.  The inverse direction is computed as conj(F(conj(x))), so
// all tables and constants are for the forward sign only.
#pragma once

#include <type_traits>

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace gb300fft {

// Device status word codes (same values as the C ABI's FFT_ERR_*).
constexpr int kStatusOk = 0;
constexpr int kStatusTimeout = -6;

__host__ __device__ constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n >> 1); }
__host__ __device__ constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }

// ---------------------------------------------------------------------------
// Complex arithmetic on float2 (x = re, y = im).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// sin(2*pi*q/64) for 0 <= q <= 16, rounded to float (compile-time constants).
__host__ __device__ constexpr float qsin64(int q) {
    return q == 0    ? 0.0f
           : q == 1  ? 0.0980171403295606f
           : q == 2  ? 0.19509032201612825f
           : q == 3  ? 0.29028467725446233f
           : q == 4  ? 0.3826834323650898f
           : q == 5  ? 0.47139673682599764f
           : q == 6  ? 0.5555702330196022f
           : q == 7  ? 0.6343932841636455f
           : q == 8  ? 0.7071067811865475f
           : q == 9  ? 0.773010453362737f
           : q == 10 ? 0.8314696123025452f
           : q == 11 ? 0.8819212643483549f
           : q == 12 ? 0.9238795325112867f
           : q == 13 ? 0.9569403357322089f
           : q == 14 ? 0.9807852804032304f
           : q == 15 ? 0.9951847266721968f
                     : 1.0f;
}
// sin and cos of 2*pi*q/64 for any integer q, by quadrant symmetry.
__host__ __device__ constexpr float sin64(int q) {
    return (q & 63) < 16   ? qsin64(q & 63)
           : (q & 63) < 32 ? qsin64(32 - (q & 63))
           : (q & 63) < 48 ? -qsin64((q & 63) - 32)
                           : -qsin64(64 - (q & 63));
}
__host__ __device__ constexpr float cos64(int q) { return sin64(q + 16); }

// z * exp(-2*pi*i*q/64).  q is a compile-time constant after unrolling, so the
// branches fold: multiples of pi/2 become swaps and sign flips, odd multiples
// of pi/4 cost two adds and two multiplies, the rest a complex multiply by
// immediate constants.
__device__ __forceinline__ float2 mul_root64(float2 z, int q) {
    q &= 63;
    if (q == 0) return z;
    if (q == 16) return make_float2(z.y, -z.x);
    if (q == 32) return make_float2(-z.x, -z.y);
    if (q == 48) return make_float2(-z.y, z.x);
    if ((q & 15) == 8) {
        const float h = 0.7071067811865475f;
        if (q == 8) return make_float2((z.x + z.y) * h, (z.y - z.x) * h);
        if (q == 24) return make_float2((z.y - z.x) * h, (-z.x - z.y) * h);
        if (q == 40) return make_float2((-z.x - z.y) * h, (z.x - z.y) * h);
        return make_float2((z.x - z.y) * h, (z.x + z.y) * h);
    }
    const float c = cos64(q), s = sin64(q);
    return make_float2(fmaf(z.x, c, z.y * s), fmaf(z.y, c, -z.x * s));
}

__host__ __device__ constexpr int bitrev(int k, int bits) {
    return bits == 0 ? 0 : ((k & 1) << (bits - 1)) | bitrev(k >> 1, bits - 1);
}

// ---------------------------------------------------------------------------
// Two independent complex values side by side, one per lane of the packed
// float32 instructions (fma/add/mul .f32x2): re = (re_a, re_b), im = (im_a,
// im_b).  A packed instruction does two lanes in one issue slot at the same
// lane rate, so kernels bound by issue run the same butterflies over C2 --
// two transforms that share every twiddle -- in half the slots.  Keeping real
// and imaginary parts in separate registers (not (re, im) packed) leaves every
// complex operation lane-wise: no swaps, and each product is the same
// multiply-add as the scalar form's.
// ---------------------------------------------------------------------------
struct __align__(16) C2 {
    float2 re, im;
};

__device__ __forceinline__ unsigned long long f2_bits(float2 a) {
    unsigned long long u;
    asm("mov.b64 %0, {%1, %2};" : "=l"(u) : "f"(a.x), "f"(a.y));
    return u;
}
__device__ __forceinline__ float2 f2_from(unsigned long long u) {
    float2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(u));
    return a;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
    return f2_from(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(d);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(d);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(d);
}
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

__device__ __forceinline__ C2 cadd(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 csub(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// both lanes times one complex value
__device__ __forceinline__ C2 cmul(C2 a, float2 w) {
    const float2 wr = both(w.x);
    return {fma2(a.im, both(-w.y), mul2(a.re, wr)), fma2(a.im, wr, mul2(a.re, both(w.y)))};
}
// lane a times wa, lane b times wb
__device__ __forceinline__ C2 cmul(C2 a, float2 wa, float2 wb) {
    const float2 wr = make_float2(wa.x, wb.x);
    return {fma2(a.im, make_float2(-wa.y, -wb.y), mul2(a.re, wr)),
            fma2(a.im, wr, mul2(a.re, make_float2(wa.y, wb.y)))};
}
__device__ __forceinline__ float2 lane_a(C2 v) { return make_float2(v.re.x, v.im.x); }
__device__ __forceinline__ float2 lane_b(C2 v) { return make_float2(v.re.y, v.im.y); }
__device__ __forceinline__ C2 lanes(float2 a, float2 b) { return {make_float2(a.x, b.x), make_float2(a.y, b.y)}; }

// d * exp(-2*pi*i*q/64), 0 <= q < 48 a constant after unrolling, no multiple of 16
// but 0
__device__ __forceinline__ C2 mul_root64(C2 d, int q) {
    if (q == 0) return d;
    if ((q & 15) == 8) {
        const float h = 0.7071067811865475f;
        const float2 sum = add2(d.re, d.im), dif = sub2(d.im, d.re);
        return q == 8    ? C2{mul2(sum, both(h)), mul2(dif, both(h))}
               : q == 24 ? C2{mul2(dif, both(h)), mul2(sum, both(-h))}
                         : C2{mul2(sum, both(-h)), mul2(dif, both(-h))};
    }
    const float c = cos64(q), s = sin64(q);
    return {fma2(d.im, both(s), mul2(d.re, both(c))), fma2(d.re, both(-s), mul2(d.im, both(c)))};
}

// (u - v) * exp(-2*pi*i*q/64), 0 <= q < 32 a constant after unrolling
__device__ __forceinline__ float2 sub_root64(float2 u, float2 v, int q) { return mul_root64(csub(u, v), q); }
__device__ __forceinline__ C2 sub_root64(C2 u, C2 v, int q) {
    if (q == 16) return {sub2(u.im, v.im), sub2(v.re, u.re)};  // times -i: no negation left over
    return mul_root64(csub(u, v), q);
}

// a - i b and a + i b
__device__ __forceinline__ float2 sub_i(float2 a, float2 b) { return make_float2(a.x + b.y, a.y - b.x); }
__device__ __forceinline__ C2 sub_i(C2 a, C2 b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }
__device__ __forceinline__ float2 add_i(float2 a, float2 b) { return make_float2(a.x - b.y, a.y + b.x); }
__device__ __forceinline__ C2 add_i(C2 a, C2 b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }

// One radix-2 decimation-in-frequency level of span H over R registers:
// (u, v) -> (u + v, (u - v) * w_{2H}^k).  Levels recurse at compile time so
// every register index and twiddle is a constant.
template <int R, int H, class V>
__device__ __forceinline__ void dif_level(V *a) {
    if constexpr (H >= 1) {
#pragma unroll
        for (int blk = 0; blk < R; blk += 2 * H) {
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const V u = a[blk + k], v = a[blk + k + H];
                a[blk + k] = cadd(u, v);
                a[blk + k + H] = sub_root64(u, v, k * (64 / (2 * H)));
            }
        }
        dif_level<R, H / 2>(a);
    }
}

// Two such levels as one of radix 4 and span Q: the rotations between the two
// radix-2 levels fold into those behind the second, so a value is rotated (and
// rounded) at most once in two levels.  Results lie where the two radix-2 levels
// leave them.  The levels below follow, of radix 4 again; those of 8 points of
// radix 2 (the same rotations either way, and fewer registers: 512-point rows 110
// against 116).
template <int R, int Q, class V>
__device__ __forceinline__ void dif_level4(V *a) {
    static_assert(Q == 0 || Q == 1 || Q == 4 || Q == 8 || Q == 16, "16, 32 or 64 points");
    if constexpr (Q >= 1) {
        constexpr int U = 16 / Q;  // w_{4Q} = w_64^U
#pragma unroll
        for (int blk = 0; blk < R; blk += 4 * Q) {
#pragma unroll
            for (int k = 0; k < Q; ++k) {
                V *p = a + blk + k;
                const V s02 = cadd(p[0], p[2 * Q]), d02 = csub(p[0], p[2 * Q]);
                const V s13 = cadd(p[Q], p[3 * Q]), d13 = csub(p[Q], p[3 * Q]);
                p[0] = cadd(s02, s13);
                p[Q] = sub_root64(s02, s13, 2 * k * U);
                p[2 * Q] = mul_root64(sub_i(d02, d13), k * U);
                p[3 * Q] = mul_root64(add_i(d02, d13), 3 * k * U);
            }
        }
        if constexpr (Q == 8) dif_level<R, 4>(a);
        else dif_level4<R, Q / 4>(a);
    }
}

// a[K] = t[bitrev(K)] for K = 0..R-1, every index a constant expression.
template <int R, int K, class V>
__device__ __forceinline__ void bitrev_gather(V *a, const V *t) {
    if constexpr (K < R) {
        constexpr int src = bitrev(K, ilog2(R));
        a[K] = t[src];
        bitrev_gather<R, K + 1>(a, t);
    }
}

// In-register length-R DFT (forward sign), natural order in and out,
// R a power of two <= 64: DIF levels, then a compile-time bit-reversal of
// register names.  Levels of radix 4 from FOUR points on, of radix 2 below.
// Every rotation rounds: with radix-2 levels a pass in 32- and 64-point stages,
// which saves an exchange, came out further from the exact result than one in
// stages of 16 (relative L2 of Gaussian columns of 1024 points 1.182e-7 against
// 1.128e-7, 2048 points 1.256e-7 against 1.185e-7); with radix 4 it is the closer
// one (1.115e-7, 1.172e-7; 4096 points 1.330e-7 -> 1.229e-7).  Fewer operations
// too: 4 x 2^24 points 0.485 -> 0.470 ms, 8 x 2048^2 loss and gradient 0.414 ->
// 0.407.
template <int R, int FOUR = 32, class V>
__device__ __forceinline__ void dft(V *a) {
    if constexpr (R > 1) {
        if constexpr (R >= FOUR) dif_level4<R, R / 4>(a);
        else dif_level<R, R / 2>(a);
        V t[R];
#pragma unroll
        for (int k = 0; k < R; ++k) t[k] = a[k];
        bitrev_gather<R, 0>(a, t);
    }
}

// ---------------------------------------------------------------------------
// Stage schedule of a length-N transform with E elements held per thread:
// first stage radix R0 = N / E^(S-1) (absorbs the remainder), then S-1
// stages of radix E.  Requires E <= N, both powers of two.
// ---------------------------------------------------------------------------
template <int N, int E>
struct Sched {
    static_assert(E <= N, "E must not exceed N");
    static constexpr int L = ilog2(N);
    static constexpr int LE = ilog2(E);
    static constexpr int S = (L + LE - 1) / LE > 0 ? (L + LE - 1) / LE : 1;
    static constexpr int R0 = N >> (LE * (S - 1));
    // span Ns of stage s
    static constexpr int ns(int s) { return s == 0 ? 1 : R0 * ipow(E, s - 1); }
    // offset of stage s's twiddle table in float2 units (stage 1 starts at
    // 0); a stage of radix R and span Ns holds R/2 float4 pairs per m
    static constexpr int tw_off(int s) { return s <= 1 ? 0 : tw_off(s - 1) + E * ns(s - 1); }
    static constexpr int tw_size = tw_off(S);
};

// ---------------------------------------------------------------------------
// Payload policies.  The FFT moves float2 and runs DFTs; the reorder-map debug
// path moves integer tags through exactly the same addresses with identity
// butterflies, which exposes the permutation the data movement realises.
// ---------------------------------------------------------------------------
template <int FOUR>  // points from which a register DFT has radix-4 levels
struct FftLevels {
    using T = float2;
    static constexpr bool kUsesTwiddles = true;
    template <int R>
    __device__ __forceinline__ void butterfly(T *a) const { dft<R, FOUR>(a); }
    __device__ __forceinline__ T twiddle(T a, float2 w) const { return cmul(a, w); }
};
using FftPolicy = FftLevels<32>;
// two transforms per thread, one per lane of C2; radix-4 levels from 16 points:
// the half-length Bluestein's outer rotations cost what they save (16384 x 4093:
// 2.83e-7 with radix 2, 2.67e-7, and 0.553 -> 0.538 ms; the length-M form 2.78e-7;
// all with the filter's spectrum in FP32)
struct PairPolicy {
    using T = C2;
    static constexpr bool kUsesTwiddles = true;
    template <int R>
    __device__ __forceinline__ void butterfly(T *a) const { dft<R, 16>(a); }
    __device__ __forceinline__ T twiddle(T a, float2 w) const { return cmul(a, w); }
};
struct MovePolicy {
    using T = float2;  // integer tags carried bit-for-bit in the .x lane
    static constexpr bool kUsesTwiddles = false;
    template <int R>
    __device__ __forceinline__ void butterfly(T *) const {}
    __device__ __forceinline__ T twiddle(T a, float2) const { return a; }
};

struct SyncBlock {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct SyncWarp {
    __device__ __forceinline__ void operator()() const { __syncwarp(); }
};

// ---------------------------------------------------------------------------
// The Stockham engine.  A group of NT = W*N/E threads transforms W
// interleaved length-N vectors held in shared memory at element (i, c) ->
// padded flat index pad(i*W + c).  Thread t of the group owns column
// c = t % W and butterfly index tt = t / W.
//
// Caller contract: v[] holds the stage-0 inputs, v[b*R0 + r] = x[j + r*N/R0]
// for j = tt + b*(N/E).  `after_reads()` runs once every thread has issued its
// last shared-memory read (it must synchronise the group if it reuses the
// buffer); `store(i, c, value)` receives the natural-order outputs.
// SRC_IN_SMEM: stage-0 inputs were read from `sm` itself, so the first
// shared-memory write must wait for every thread's reads.
// ---------------------------------------------------------------------------
constexpr int kSwizzle = 31;  // Engine's PADSH: xor swizzle in place of padding

template <int N, int E, int W, int PADSH, int PADSH1 = PADSH>
struct Engine {
    using Sc = Sched<N, E>;
    static constexpr int T = N / E;   // threads per column
    static constexpr int NT = T * W;  // threads per group
    static constexpr int R0 = Sc::R0;
    static constexpr int S = Sc::S;
    static constexpr int RL = (S == 1) ? R0 : E;  // radix of the last stage
    // padded index of the exchange after stage s - 1: the first exchange may
    // use its own shift (PADSH1), since its write pattern follows radix R0
    __host__ __device__ static constexpr int pad(int f) { return f + (f >> PADSH); }
    __host__ __device__ static constexpr int pad_s(int f, int s) { return f + (f >> (s == 1 ? PADSH1 : PADSH)); }
    // PADSH = kSwizzle: no padding; the low three bits of the index are
    // xored with higher ones instead (16-byte elements, eight to a row of
    // banks): every write and read below is then conflict-free over the eight
    // lanes of a quarter-warp, and the buffer is exactly N*W elements
    static constexpr bool SWZ = PADSH == kSwizzle;
    __host__ __device__ static constexpr int swz(int f, int s) {
        return f ^ ((f >> (s == 1 && R0 < 16 ? 3 : 4)) & 7);
    }
    static constexpr int SMEM_ELEMS =
        (S == 1) ? 0
        : SWZ    ? N * W
                 : (pad_s(N * W - 1, 1) > pad(N * W - 1) ? pad_s(N * W - 1, 1) : pad(N * W - 1)) + 1;

    template <class Pol, bool SRC_IN_SMEM, class Sync, class AfterReads, class Store>
    __device__ static __forceinline__ void run(typename Pol::T (&v)[E], typename Pol::T *sm,
                                               const float2 *__restrict__ tw, int tt, int c,
                                               Sync sync, AfterReads after_reads, Store store) {
        // 512 = 16 * 32 is as exact with radix-2 levels as 2 * 16 * 16 (1.083e-7
        // both), and radix 4 costs its kernels registers (512^2 x 64: 92.6 us, with
        // radix 4 94.4; 2^22 points of rows 11.6 and 12.3)
        using P = std::conditional_t<N == 512 && std::is_same_v<Pol, FftPolicy>, FftLevels<64>, Pol>;
        run_with<P, SRC_IN_SMEM>(P{}, v, sm, tw, tt, c, sync, after_reads, store);
    }

    // Same, with a policy object (a stateful butterfly, e.g. the tensor-core one).
    template <class Pol, bool SRC_IN_SMEM, class Sync, class AfterReads, class Store>
    __device__ static __forceinline__ void run_with(const Pol &pol, typename Pol::T (&v)[E], typename Pol::T *sm,
                                                    const float2 *__restrict__ tw, int tt, int c, Sync sync,
                                                    AfterReads after_reads, Store store) {
        using V = typename Pol::T;
        // stage 0: butterflies in registers, no twiddles
#pragma unroll
        for (int b = 0; b < E / R0; ++b) pol.template butterfly<R0>(&v[b * R0]);
        if constexpr (S == 1) {
            after_reads();
        } else {
#pragma unroll
            for (int s = 1; s < S; ++s) {
                const int Rp = (s == 1) ? R0 : E;  // radix of stage s-1
                const int Nsp = Sc::ns(s - 1);     // span of stage s-1
                if (s > 1 || SRC_IN_SMEM) sync();
#pragma unroll
                for (int b = 0; b < E / Rp; ++b) {
                    const int j = tt + b * T;
                    const int m = j & (Nsp - 1);
#pragma unroll
                    for (int k = 0; k < Rp; ++k) {
                        // the swizzle is linear over xor, and k*Nsp (below:
                        // r*T) has no bit in common with the rest: its part
                        // of the index is a constant
                        if constexpr (SWZ)
                            sm[swz(((j - m) * Rp + m) * W + c, s) ^ swz(k * Nsp * W, s)] = v[b * Rp + k];
                        else
                            sm[pad_s(((j - m) * Rp + m + k * Nsp) * W + c, s)] = v[b * Rp + k];
                    }
                }
                sync();
                const int Ns = Sc::ns(s);
                const int m = tt & (Ns - 1);
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    if constexpr (SWZ) v[r] = sm[swz(tt * W + c, s) ^ swz(r * T * W, s)];
                    else v[r] = sm[pad_s((tt + r * T) * W + c, s)];
                }
                if (s == S - 1) after_reads();
                if constexpr (Pol::kUsesTwiddles) {
                    // twiddles r = 2k+1, 2k+2 of this butterfly in one 16-byte load
                    const float4 *tws = reinterpret_cast<const float4 *>(tw + Sc::tw_off(s)) + m;
#pragma unroll
                    for (int k = 0; k < E / 2; ++k) {
                        const float4 w2 = __ldg(tws + k * Ns);
                        v[2 * k + 1] = pol.twiddle(v[2 * k + 1], make_float2(w2.x, w2.y));
                        if (2 * k + 2 < E) v[2 * k + 2] = pol.twiddle(v[2 * k + 2], make_float2(w2.z, w2.w));
                    }
                }
                pol.template butterfly<E>(v);
            }
        }
        // natural-order outputs of the last stage: position j + k*N/RL
#pragma unroll
        for (int b = 0; b < E / RL; ++b) {
            const int j = tt + b * T;
#pragma unroll
            for (int k = 0; k < RL; ++k) store(j + k * (N / RL), c, v[b * RL + k]);
        }
    }
};

// Shared-memory padding shift used by every kernel for a given E: chosen so
// that the stage loads and stores of the common shapes hit each bank pair at
// most once per half-warp (checked by a bank model on the CPU).
template <int E>
struct PadShift {
    static constexpr int value = (E >= 64) ? 6 : (E >= 32) ? 5 : 4;
};
// First-exchange shift of the one-row engines (W = 1): with E = 32 the write
// after the radix-4/8 first stage puts 16 lanes 8 or 4 float2 apart, which
// a shift of 4 spreads over all banks (half-warp bank model; shift 5 leaves
// 2-way conflicts there).
template <int E>
struct RowPadShift1 {
    static constexpr int value = (E == 32) ? 4 : PadShift<E>::value;
};

// ---------------------------------------------------------------------------
// TMA / mbarrier helpers (inline PTX).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait on an mbarrier phase: gives up after ~`limit_ns` nanoseconds
// (or 2^26 polls) and returns false.  Never spins forever.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  uint64_t limit_ns = 2000000000ull) {
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t it = 0; it < (1u << 26); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255) == 255 && globaltimer_ns() - t0 > limit_ns) break;
    }
    return false;
}
// 2D tiled TMA load of one box into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
// 3D tiled TMA load (coordinates innermost first).
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                            uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int x, int y, int z) {
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z)
                 : "memory");
}
// 1D bulk copy global -> shared (16-byte aligned, size a multiple of 16),
// completing on `bar`.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
// 4D tiled TMA store of one box from shared memory (coordinates innermost
// first), tracked in the issuing thread's bulk async-group.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, const void *src, int x, int y, int z, int w) {
    asm volatile(
        "cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(src))
        : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until at most one of this thread's bulk groups still reads shared memory.
__device__ __forceinline__ void bulk_wait_read_1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
// Wait until every bulk group this thread issued has completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Prefetch of one box into L2 (no shared memory involved).
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap *map, int x, int y) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y)
                 : "memory");
}

// Bulk prefetch of a contiguous byte range into L2 (16-byte aligned address,
// size a multiple of 16).
__device__ __forceinline__ void bulk_prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(p)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void record_status(int *status, int code) {
    if (status) atomicCAS(status, kStatusOk, code);
}

}  // namespace gb300fft
