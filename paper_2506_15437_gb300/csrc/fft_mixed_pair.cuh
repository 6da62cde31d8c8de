// Mixed-radix transforms over pairs, in place in one shared-memory buffer.
//
// Each element of the buffer is a C2: two transforms (adjacent columns; rows c
// and c + W/2 of a group) in the two lanes of packed float32 instructions,
// sharing every index computation and twiddle load.
//
// n = R_0 ... R_{S-1}, decimation in frequency: index digits (i_0 .. i_{S-1}),
// i_0 most significant, are replaced one per stage by frequency digits k_s.
// Stage s transforms over digit s -- the R_s elements p R_s Q + r Q + q, with Q
// = R_{s+1} ... R_{S-1}, of one butterfly (p, q) -- multiplies result r by
// w_{R_s Q}^{r q} and puts it back where element r was.  So a butterfly owns
// what it reads and writes: one buffer serves every stage, a stage may run in
// as many rounds as it likes, and one barrier separates two stages.  (The
// autosorting form, which writes every stage to new places, needs two buffers
// or every leg held in registers across a barrier.)  The first stage reads
// global memory; the last takes its butterflies in output order, k_0 fastest,
// and stores result r of butterfly o to o + r n / R_{S-1}: natural order.
//
// In the buffer each block of one k_0 (Q_0 elements) is followed by `skew`
// unused ones, so that the last stage's lanes, one block apart, fall on
// different banks; the plan picks the skew with the fewest conflicts.
//
// Kernels are compiled per largest radix RMAX, since the widest butterfly sets
// every thread's registers and with them the threads an SM holds.  For launches
// too small to fill the GPU, for the passes of a four-step transform and for
// columns of an odd row length there is one transform per element instead (V =
// float2): twice the threads, half as long a chain of instructions each.
#pragma once

#include "fft_common.cuh"
#include "fft_internal.h"
#include "fft_mixed.cuh"

namespace gb300fft {

namespace {

using namespace mixed;

struct PairGeom {
    int W;        // elements per position (a power of two in the column layout and in four-step rows)
    int nv;       // valid transforms in this CTA (even for pairs of columns)
    int estride;  // element stride within a transform (1 for rows, nx for columns)
    int tstride;  // offset between the CTA's transforms (n for rows, 1 for columns)
    int cstride;  // rows: buffer elements from one transform (pair) to the next
    int wlog;     // log2 W, where it is a power of two
};

// One stage of radix R over the CTA's transforms.  Rows: butterfly index
// fastest within a transform (coalesced rows), buffer [c][position].  Columns,
// and the transposed store of a four-step row pass: transform fastest; columns'
// buffer [position][c].  `gin` and `gout` point at the CTA's first transform,
// so every offset within the group fits 32 bits.  Past the last valid transform
// a lane reads zeros and is not stored.
template <class V, int R, bool COLS, bool FIRST, bool LAST, bool FS>
__device__ __forceinline__ void pair_stage(const PairGeom &g, const MixedStages &st, int s, V *buf, const float2 *gin,
                                           float2 *gout, const float2 *__restrict__ tw, float si,
                                           const FourStepB &fs) {
    constexpr bool PAIR = sizeof(V) == sizeof(C2), CFAST = COLS || (LAST && FS), ADJ = PAIR && COLS;
    static_assert(!(PAIR && FS), "four-step passes run one transform per thread");
    const int nb = st.nb[s], Q = st.ns[s], skew = st.skew;
    const int total = (CFAST ? g.W : g.nv < g.W ? g.nv : g.W) * nb;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        int c, j;
        if (CFAST) {
            c = idx & (g.W - 1);
            j = idx >> g.wlog;
        } else {
            c = fdiv(idx, nb, st.mag_nb[s]);
            j = idx - c * nb;
        }
        const int t0 = ADJ ? 2 * c : c;                 // lane a's transform
        if (CFAST && t0 >= g.nv) continue;              // past the last column (row)
        const int tb = g.W * g.tstride;    // rows: lane b's, from lane a's
        const bool two = t0 + g.W < g.nv;  // rows: lane b holds a transform
        // butterfly (p, q) and its place in the buffer
        int q = j, pos = FIRST ? j : 0;
        if constexpr (FIRST) {
        } else if constexpr (LAST) {
            // j = k_0 + R_0 (k_1 + R_1 (...)), place k_0 Q_0 + ... : digits reversed
            int rest = j, k0 = 0;
            for (int t = 0; t < s; ++t) {
                const int d = fdiv(rest, st.radix[t], st.mag_r[t]), k = rest - d * st.radix[t];
                if (t == 0) k0 = k;
                pos = pos * st.radix[t] + k;
                rest = d;
            }
            pos = pos * R + k0 * skew;
        } else {
            const int p = fdiv(j, Q, st.mag_ns[s]);
            q = j - p * Q;
            pos = p * (R * Q) + q + (s == 1 ? p : fdiv(p, st.kdiv[s], st.mag_k[s])) * skew;
        }
        V *b = buf + (COLS ? pos * g.W + c : c * g.cstride + pos);
        const int bs = (FIRST ? Q + skew : Q) * (COLS ? g.W : 1);
        V v[R];
        if constexpr (FIRST) {
            const float2 *x = gin + t0 * g.tstride + j * g.estride;
            const int xs = nb * g.estride;
            if constexpr (!PAIR) {
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = x[r * xs];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r].y *= si;
            } else {
                if constexpr (COLS) {
                    // a pair is 16 bytes: nx and the first column are even
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float4 u = *reinterpret_cast<const float4 *>(x + r * xs);
                        v[r] = lanes(make_float2(u.x, u.y), make_float2(u.z, u.w));
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        v[r] = lanes(x[r * xs], two ? x[r * xs + tb] : make_float2(0.f, 0.f));
                }
#pragma unroll
                for (int r = 0; r < R; ++r) v[r].im = mul2(v[r].im, both(si));
            }
            if constexpr (FS) {
                // element i2 = j + r nb of row m = k1 + t0 times w_n^{i2 m} =
                // w_n^{j m} w_n^{r nb m}: one gather per thread, the second
                // factor a broadcast along the row
                const int m = fs.k1 + t0;
                const float2 wa = fs_root(fs, j * m);
                v[0] = cmul(v[0], wa);
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = cmul(v[r], cmul(wa, fs_root(fs, r * nb * m)));
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = b[r * bs];
        }
        dft_any<R>(v);
        if constexpr (!LAST) {
            // twiddles r, r + 1 of butterfly q as one 16-byte load
            const float4 *w = reinterpret_cast<const float4 *>(tw + st.tw_off[s]) + q;
#pragma unroll
            for (int r = 1; r < R; r += 2) {
                const float4 w2 = __ldg(w + ((r - 1) / 2) * Q);
                v[r] = cmul(v[r], make_float2(w2.x, w2.y));
                if (r + 1 < R) v[r + 1] = cmul(v[r + 1], make_float2(w2.z, w2.w));
            }
#pragma unroll
            for (int r = 0; r < R; ++r) b[r * bs] = v[r];
        } else {
            // four-step: output o of row k1 + t goes to k1 + t + n1 o (gout points at k1)
            const int ys = FS ? fs.n1 * nb : nb * g.estride;
            float2 *y = gout + (FS ? t0 + fs.n1 * j : t0 * g.tstride + j * g.estride);
            if constexpr (!PAIR) {
#pragma unroll
                for (int r = 0; r < R; ++r) y[r * ys] = make_float2(v[r].x, v[r].y * si);
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) v[r].im = mul2(v[r].im, both(si));
                if constexpr (COLS) {
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        *reinterpret_cast<float4 *>(y + r * ys) =
                            make_float4(v[r].re.x, v[r].im.x, v[r].re.y, v[r].im.y);
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) y[r * ys] = lane_a(v[r]);
                    if (two) {
#pragma unroll
                        for (int r = 0; r < R; ++r) y[r * ys + tb] = lane_b(v[r]);
                    }
                }
            }
        }
    }
}

template <class V, int RMAX, bool COLS, bool FIRST, bool LAST, bool FS>
__device__ __forceinline__ void pair_dispatch(const PairGeom &g, const MixedStages &st, int s, V *buf,
                                              const float2 *gin, float2 *gout, const float2 *tw, float si,
                                              const FourStepB &fs) {
#define GB300FFT_PAIR_CASE(r)                                                                              \
    case r:                                                                                                \
        if constexpr (r <= RMAX) pair_stage<V, r, COLS, FIRST, LAST, FS>(g, st, s, buf, gin, gout, tw, si, fs); \
        break;
    switch (st.radix[s]) {
        GB300FFT_PAIR_CASE(2)
        GB300FFT_PAIR_CASE(3)
        GB300FFT_PAIR_CASE(4)
        GB300FFT_PAIR_CASE(5)
        GB300FFT_PAIR_CASE(6)
        GB300FFT_PAIR_CASE(7)
        GB300FFT_PAIR_CASE(8)
        GB300FFT_PAIR_CASE(9)
        GB300FFT_PAIR_CASE(10)
        GB300FFT_PAIR_CASE(11)
        GB300FFT_PAIR_CASE(12)
        GB300FFT_PAIR_CASE(13)
        GB300FFT_PAIR_CASE(14)
        GB300FFT_PAIR_CASE(15)
        GB300FFT_PAIR_CASE(16)
    }
#undef GB300FFT_PAIR_CASE
}

template <class V, int RMAX, bool COLS, bool FS>
__global__ void __launch_bounds__(sizeof(V) == sizeof(C2) ? mixed_pair_threads(RMAX) : kMixedOneThreads, 1)
    k_mixed_pair(const float2 *in, float2 *out, const float2 *__restrict__ tw, const __grid_constant__ MixedStages st,
                 long long ntrans, int W, int nx, int conj, FourStepB fs) {
    extern __shared__ __align__(16) C2 pbuf[];
    V *buf = reinterpret_cast<V *>(pbuf);
    PairGeom g;
    g.W = W / (int)(sizeof(V) / sizeof(float2));
    g.wlog = st.wlog;
    g.cstride = st.buf_elems;
    long long base;
    long long t0 = (long long)blockIdx.x * W;  // rows: first transform of this CTA
    if (COLS) {
        // columns x0 .. of slice b; a slice's last group may be narrower
        const int gps = (nx + W - 1) / W;
        const long long b = blockIdx.x / gps;
        const int x0 = (int)(blockIdx.x - b * gps) * W;
        g.nv = nx - x0 < W ? nx - x0 : W;
        base = b * (long long)nx * st.n + x0;
        g.estride = nx;
        g.tstride = 1;
    } else {
        if (FS) {
            // rows k1 .. of transform b; its last group may be narrower
            const int gpt = (fs.n1 + W - 1) / W;
            const long long b = blockIdx.x / gpt;
            fs.k1 = (int)(blockIdx.x - b * gpt) * W;
            t0 = b * fs.n1 + fs.k1;
            g.nv = fs.n1 - fs.k1 < W ? fs.n1 - fs.k1 : W;
        } else {
            g.nv = (int)(ntrans - t0 < W ? ntrans - t0 : W);
        }
        base = t0 * st.n;
        g.estride = 1;
        g.tstride = st.n;
    }
    const float2 *gin = in + base;
    float2 *gout = FS ? out + (base - (long long)fs.k1 * st.n) + fs.k1 : out + base;
    if (!COLS) {
        if (threadIdx.x == 0) {
            // the group's rows are contiguous: ask L2 for all of it (the
            // 16-byte-aligned interior), so later rounds find it there
            const uintptr_t a0 = reinterpret_cast<uintptr_t>(gin);
            const uintptr_t a1 = a0 + (uintptr_t)g.nv * st.n * sizeof(float2);
            const uintptr_t p0 = (a0 + 15) & ~(uintptr_t)15, p1 = a1 & ~(uintptr_t)15;
            if (p1 > p0) bulk_prefetch_l2(reinterpret_cast<const void *>(p0), (uint32_t)(p1 - p0));
        }
    } else {
        for (int i = threadIdx.x; i < st.n; i += blockDim.x)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(gin + (long long)i * nx));
    }
    const float si = conj ? -1.f : 1.f;
    if (st.S == 1) {
        pair_dispatch<V, RMAX, COLS, true, true, FS>(g, st, 0, buf, gin, gout, tw, si, fs);
        return;
    }
    pair_dispatch<V, RMAX, COLS, true, false, FS>(g, st, 0, buf, gin, gout, tw, si, fs);
    __syncthreads();
    for (int s = 1; s < st.S - 1; ++s) {
        pair_dispatch<V, RMAX, COLS, false, false, FS>(g, st, s, buf, gin, gout, tw, si, fs);
        __syncthreads();
    }
    pair_dispatch<V, RMAX, COLS, false, true, FS>(g, st, st.S - 1, buf, gin, gout, tw, si, fs);
}

template <class V, int RMAX>
const void *pair_fn(bool cols) {
    return cols ? (const void *)k_mixed_pair<V, RMAX, true, false> : (const void *)k_mixed_pair<V, RMAX, false, false>;
}

}  // namespace

}  // namespace gb300fft
