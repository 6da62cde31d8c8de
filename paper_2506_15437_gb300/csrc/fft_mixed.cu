// Mixed-radix transforms for lengths of the form 2^a 3^b 5^c 7^d 11^e 13^f:
// schedules, tables and launches (the kernels are in fft_mixed_pair.cuh).
//
// The paper's kernels take powers of two only and name uneven sizes as
// further work (Sections 6 and 7).  Smooth lengths up to kMixedMaxN run as
// stages of radix 16, 15, 14, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3 or 2, chosen
// at plan time (15, 14, 12, 10, 9 and 6 are two-level DFTs in registers with
// compile-time inner twiddles; the odd primes 3 .. 13 one symmetric-pair DFT
// each): the fewest stages these radices allow, since each stage is one pass
// through shared memory and one barrier (mixed_factor has the count,
// pair_stages chooses the radices and their order).  One CTA owns whole transforms: the
// first stage reads global memory, the last writes it.
//
// Two layouts: rows (transforms along contiguous rows, W rows per CTA) and
// columns (the transforms of W adjacent columns of an [ny][nx] slice, element
// i of column x at i*nx + x), which serves the y axis of a 2D plan without a
// transpose.  Longer smooth lengths run as a four-step split n = n1 n2 over
// both layouts: columns of length n1 into a workspace, then rows of length n2
// whose first stage multiplies by the inter-pass twiddle and whose last stage,
// with its lanes taken transform first, stores the W rows' outputs transposed,
// W adjacent outputs per row of the result (FourStepB).
#include <math.h>
#include <stdlib.h>

#include <algorithm>

#include "fft_common.cuh"
#include "fft_internal.h"
#include "fft_mixed.cuh"

namespace gb300fft {

namespace {

using namespace mixed;

// stage s's table, as 16-byte pairs: pair p of butterfly k (k < Ns) at
// pair index p Ns + k holds w_{Ns R}^{k r} for r = 2p + 1 and 2p + 2 (the
// second zero when R - 1 is odd), from the FP64 root, rounded once
__global__ void k_mixed_twiddles(float2 *t, int Ns, int R) {
    const int M = mixed_tw_stride(R);
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= Ns * M) return;
    const int q = e >> 1, p = q / Ns, k = q - p * Ns, r = 2 * p + 1 + (e & 1);
    if (r >= R) {
        t[e] = make_float2(0.f, 0.f);
        return;
    }
    const int L = Ns * R;
    double sv, cv;
    sincospi(2.0 * (double)((k * r) % L) / (double)L, &sv, &cv);
    t[e] = make_float2((float)cv, (float)(-sv));
}

const void *mixed_fn(int rmax, bool cols, bool fs) {
    if (rmax == 0) return mixed_one_fn(cols, fs);
    if (fs) return nullptr;  // no four-step kernel over pairs
    return rmax <= 13 ? mixed_pair13_fn(cols) : mixed_pair16_fn(cols);
}
int mixed_threads(int rmax) { return rmax == 0 ? kMixedOneThreads : mixed_pair_threads(rmax); }

// A few kernels serve every mixed length, each plan with its own shared
// memory size, so the kernel's dynamic shared-memory limit is raised to the
// largest any plan may ask for, the same value from every plan: a
// plan-sized limit would let a plan created later (or concurrently, on
// another thread) lower it below what an earlier plan launches with.
bool smem_ok(const void *fn, size_t smem) {
    if (!fn || smem > kMixedMaxSmem) return false;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMixedMaxSmem) != cudaSuccess)
        return false;
    return true;
}

uint32_t magic(int d) { return d <= 1 ? 0u : (uint32_t)((((uint64_t)1 << 32) + (uint64_t)d - 1) / (uint64_t)d); }

constexpr int kMixedSms = 152;

// the compiled radices, largest first
constexpr int kMixedRadices[] = {16, 15, 14, 13, 12, 11, 10, 9, 8, 7, 6, 5, 4, 3, 2};

// rest as a product of exactly `left` compiled radices, none larger than
// `cap` (non-increasing, so each multiset is tried once), into out[]
bool factor_exact(int rest, int left, int cap, int *out) {
    if (left == 0) return rest == 1;
    long long reach = 1;
    for (int i = 0; i < left; ++i) reach *= cap;
    if (reach < rest) return false;
    for (int R : kMixedRadices) {
        if (R > cap || rest % R) continue;
        out[0] = R;
        if (factor_exact(rest / R, left - 1, R, out + 1)) return true;
    }
    return false;
}

}  // namespace

bool mixed_factor(int n, MixedStages *st) {
    if (n < 2 || n > kMixedMaxN) return false;
    MixedStages m;
    m.n = n;
    int rest = n, S = 0;
    auto push = [&](int R) {
        if (S >= kMixedMaxStages) return false;
        m.radix[S++] = R;
        rest /= R;
        return true;
    };
    // greedy: powers of two: 16s, then one 8, 4 or 2; odd part: 3 * 5 and 3 * 3
    // in one register stage each, then single 3, 5, 7, 11, 13 (a 25-point stage needs
    // twice the registers of a 16-point one and halves the CTAs per SM:
    // measured slower than two 5-point stages)
    int e3 = 0, e5 = 0;
    for (int t = rest; t % 3 == 0; t /= 3) ++e3;
    for (int t = rest; t % 5 == 0; t /= 5) ++e5;
    while (rest % 16 == 0)
        if (!push(16)) return false;
    for (int R : {8, 4, 2})
        if (rest % R == 0 && !push(R)) return false;
    for (; e5 >= 1 && e3 >= 1; --e5, --e3)
        if (!push(15)) return false;
    for (; e3 >= 2; e3 -= 2)
        if (!push(9)) return false;
    if (e3 == 1 && !push(3)) return false;
    for (; e5 >= 1; --e5)
        if (!push(5)) return false;
    for (int R : {7, 11, 13})
        while (rest % R == 0)
            if (!push(R)) return false;
    if (rest != 1) return false;
    // the greedy factorisation above is kept where none has fewer stages (e.g.
    // 3000 = 8 15 5 5); otherwise the first of the fewest, radices
    // non-increasing (1000 = 10 10 10 in place of 8 5 5 5, 1728 = 16 12 9 in
    // place of 16 4 9 3, 96 = 16 6 in place of 16 2 3).  The kernels run S
    // stages, of pair_stages' radices; these ones enter mixed_layout's rule for
    // small launches.
    for (int d = 1; d < S; ++d) {
        int r[kMixedMaxStages];
        if (factor_exact(n, d, 16, r)) {
            for (int i = 0; i < d; ++i) m.radix[i] = r[i];
            S = d;
            break;
        }
    }
    m.S = S;
    if (st) *st = m;
    return true;
}

cudaError_t build_mixed_twiddles(float2 *tw, const MixedStages &st, cudaStream_t s) {
    for (int i = 0; i < st.S; ++i) {
        const int R = st.radix[i], count = st.ns[i] * mixed_tw_stride(R);
        k_mixed_twiddles<<<(count + 255) / 256, 256, 0, s>>>(tw + st.tw_off[i], st.ns[i], R);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

namespace {

// rest as `left` radices up to `cap` (non-increasing, so each multiset once):
// the one with the fewest butterflies, sum of 1 / R, into out[]
void best_factors(int rest, int left, int cap, int *cur, int depth, double sum, double *best, int *out) {
    if (left == 0) {
        if (rest == 1 && sum < *best) {
            *best = sum;
            for (int i = 0; i < depth; ++i) out[i] = cur[i];
        }
        return;
    }
    long long reach = 1;
    for (int i = 0; i < left; ++i) reach *= cap;
    if (reach < rest) return;
    for (int R : kMixedRadices) {
        if (R > cap || rest % R) continue;
        cur[depth] = R;
        best_factors(rest / R, left - 1, R, cur, depth + 1, sum + 1.0 / R, best, out);
    }
}

// Shared-memory wavefronts of the first two warps of every stage, for the
// radices in this order, `words` elements per position and each skew 0 .. 7:
// eight lanes' 16-byte pairs cost as many wavefronts as the fullest of the eight
// bank groups holds.  Legs r differ by a constant, which moves every lane's bank
// alike, so one leg stands for all.  The one-transform kernels' 8-byte elements
// are counted as if they were pairs, which ranks orders and skews only
// approximately (exactly, sixteen lanes would share sixteen banks of 8 bytes).
void skew_costs(const int *radix, int S, int n, int words, bool cols, bool fs, long long cost[8]) {
    for (int k = 0; k < 8; ++k) cost[k] = 0;
    int Q = n, kdiv = 1;
    for (int s = 0; s < S; ++s) {
        const int R = radix[s], nb = n / R, total = words * nb;
        Q /= R;
        const bool last = s == S - 1, cfast = cols || (fs && last);
        const int weight = ((s > 0) + !last) * R;
        for (int w0 = 0; w0 < total && w0 < 64; w0 += 8) {
            uint32_t full[8] = {};  // per skew: eight 4-bit counters, one per bank group
            for (int l = 0; l < 8 && w0 + l < total; ++l) {
                const int idx = w0 + l;
                const int c = cfast ? idx % words : idx / nb, j = cfast ? idx / words : idx % nb;
                int pos = j, k0 = 0;
                if (s > 0 && last) {
                    int rest = j, p = 0;
                    for (int t = 0; t < s; ++t) {
                        const int k = rest % radix[t];
                        if (t == 0) k0 = k;
                        p = p * radix[t] + k;
                        rest /= radix[t];
                    }
                    pos = p * R;
                } else if (s > 0) {
                    const int p = j / Q;
                    pos = p * R * Q + j - p * Q;
                    k0 = p / kdiv;
                }
                for (int k = 0; k < 8; ++k) {
                    const int at = pos + k0 * k;
                    full[k] += 1u << (4 * ((cols ? at * words + c : at + c * (n + radix[0] * k)) & 7));
                }
            }
            for (int k = 0; k < 8; ++k) {
                int worst = 0;
                for (int g = 0; g < 8; ++g) {
                    const int f = (full[k] >> (4 * g)) & 15;
                    worst = f > worst ? f : worst;
                }
                cost[k] += (long long)weight * worst;
            }
        }
        if (s > 0) kdiv *= R;
    }
}

// The kernels' stages of a length in S stages: radices up to rmax, with the fewest butterflies, in the order
// and with the skew of the fewest bank conflicts.
MixedStages pair_stages(int n, int S, int words, bool cols, bool fs, int rmax) {
    MixedStages m;
    m.n = n;
    m.S = S;
    int cur[kMixedMaxStages], radix[kMixedMaxStages];
    double sum = 1e30;
    best_factors(n, S, rmax ? rmax : 16, cur, 0, 0.0, &sum, radix);
    std::sort(radix, radix + m.S);
    long long best = -1;
    int tried = 0;
    do {
        long long cost[8];
        skew_costs(radix, m.S, m.n, words, cols, fs, cost);
        for (int k = 0; k < 8; ++k) {
            if ((size_t)words * (m.n + radix[0] * k) * (rmax ? sizeof(C2) : sizeof(float2)) > kMixedMaxSmem) break;
            if (best < 0 || cost[k] < best) {
                best = cost[k];
                m.skew = k;
                for (int s = 0; s < m.S; ++s) m.radix[s] = radix[s];
            }
        }
    } while (++tried < 120 && std::next_permutation(radix, radix + m.S));
    m.wlog = ilog2(words);
    m.buf_elems = m.n + m.radix[0] * m.skew;
    int off = 0, Q = m.n;
    for (int s = 0; s < m.S; ++s) {
        const int R = m.radix[s];
        Q /= R;
        m.tw_off[s] = off;
        m.ns[s] = Q;
        m.nb[s] = m.n / R;
        off += Q * mixed_tw_stride(R);
        m.mag_nb[s] = magic(m.nb[s]);
        m.mag_ns[s] = magic(Q);
        m.mag_r[s] = magic(R);
        m.kdiv[s] = s < 2 ? 1 : m.kdiv[s - 1] * m.radix[s - 1];
        m.mag_k[s] = magic(m.kdiv[s]);
    }
    m.tw_size = off;
    return m;
}

// largest radix compiled into the kernels that take n in S stages
int mixed_class(int n, int S) {
    int cur[kMixedMaxStages], out[kMixedMaxStages];
    double sum = 1e30;
    best_factors(n, S, 13, cur, 0, 0.0, &sum, out);
    return sum < 1e29 ? 13 : 16;
}

// Transforms per CTA (even; a power of two in the column layout and in
// four-step rows), `count` transforms in all.
//
// Columns and four-step rows: 8 adjacent ones, 64 bytes of each global row
// (1080-point columns: 0.071 ms for 17.7 M points, 4 wide 0.080), while the
// buffer leaves room for a second CTA; 4 while it fits at all (2160 points: 8
// wide 0.091, 4 wide 0.094; 4095 points: 4 wide 0.111, 2 wide 0.154); more of
// very short ones, to have 1500 elements (128 x 120 four-step, 15360 points x
// 1024: 8 wide 0.119, 16 wide 0.109).  Rows: 4 up to 1024 points, then 2; of
// short ones as many as make 2048 elements, of very short ones 1280 (2^16 rows
// of 150 points: 8 to 12 rows 0.030 ms, 26 rows 0.034).  Fewer where that would
// leave SMs without two CTAs.
int mixed_group(int n, bool cols, int nx, int fs_n1, long long count) {
    const int wide = cols || fs_n1 ? 4 : 2;
    int W = 2;
    if (cols || fs_n1) {
        const int width = cols ? nx : fs_n1;
        while (W < 8 && W < width && (size_t)2 * W * n * sizeof(float2) <= (W == 4 ? 140 : 227) * 1024) W *= 2;
        while (W >= 8 && W < 32 && W < width && W * n < 1500) W *= 2;
    } else if (n <= 1024) {
        W = std::max(4, (n >= 128 ? 2048 : 1280) / n & ~1);
        if (W > 64) W = 64;
    }
    while (W > wide && count / W < kMixedSms * 2) W = cols || fs_n1 ? W / 2 : (W / 2 + 1) & ~1;
    return W;
}

// Threads per CTA: about 18 elements each (15 of short transforms), or two to
// three rounds of the average stage where low radices need more (2^19 rows of
// 20 points: 0.030 ms against 0.036), in steps that fill whole quarter-SM
// register files, and never so many that the CTAs the shared memory allows no
// longer fit (4095-point rows, three CTAs of 68 KB: 160 threads 0.067 ms, 256
// 0.077).
int mixed_block(const MixedStages &m, int words, int rmax, size_t smem) {
    int target = words * m.n / (m.n < 512 ? 15 : 18), sum = 0;
    for (int s = 0; s < m.S; ++s) sum += words * m.nb[s];
    if (sum * 5 / (13 * m.S) > target) target = sum * 5 / (13 * m.S);
    constexpr int steps[] = {32, 64, 96, 128, 160, 256, 320, 512};
    int i = 0;
    while (i < 7 && steps[i] < 256 && steps[i] * 20 < target * 19) ++i;
    while (i < 7 && steps[i] >= 256 && abs(steps[i + 1] - target) < abs(steps[i] - target)) ++i;
    const int ctas = (int)(228 * 1024 / (smem + 1024));
    if (ctas <= 5)
        while (i > 0 && steps[i] * (ctas > 1 ? ctas : 1) > mixed_threads(rmax)) --i;
    return steps[i];
}
}  // namespace

int mixed_layout(const MixedStages &st, bool cols, int nx, long long count, MixedLaunch *out, bool fourstep,
                 int fs_n1) {
    MixedLaunch L;
    L.cols = cols;
    L.nx = cols ? nx : 0;
    const bool fs = !cols && fs_n1 > 0;
    if (fs) L.fs.n1 = fs_n1;
    if (cols && nx <= 0) return -1;
    // lengths of one stage would read and write rows straight from registers,
    // lanes n elements apart; two stages read and write them coalesced
    // (2^20 rows of 15 points: 0.046 ms against 0.092)
    int S = st.S;
    if (S == 1 && st.n >= 8 && st.n != 11 && st.n != 13) S = 2;
    // One transform per thread or two?  Two halve the issue slots (3000-point
    // rows 0.081 ms against 0.095, 1000-point rows 0.048 / 0.055) but lengthen
    // each thread's chain and the smallest unit of work.  One where the
    // launch cannot fill the GPU (3 rows of 12000 points 11.6 us against 16.4,
    // 100 x 100 7.3 / 9.0), for both passes of a four-step transform (24000
    // points 0.068 / 0.078 ms, 120000 0.083 / 0.098), for lengths of which an
    // SM holds a single pair (10000-point rows 0.079 / 0.088), and for columns
    // that are not 16-byte pairs or hardly worth a group (1023 x 1080 0.216 /
    // 0.230, 1024 x 6 0.086 / 0.111).
    const bool one = fourstep || st.n > 7000 || (cols && (nx % 2 || st.n <= 16)) ||
                     count * (st.n / st.radix[0]) / 2 < kMixedSms * 400;
    L.rmax = one ? 0 : mixed_class(st.n, S);
    const int pair = L.rmax > 0 ? 2 : 1;
    L.W = mixed_group(st.n, cols, nx, fs ? fs_n1 : 0, count);
    if (pair == 1 && !cols && !fs) L.W /= 2;
    const int words = L.W / pair;
    L.m = pair_stages(st.n, S, words, cols, fs, L.rmax);
    L.smem = (size_t)words * L.m.buf_elems * pair * sizeof(float2);
    int most = 0;
    for (int s = 0; s < L.m.S; ++s) most = words * L.m.nb[s] > most ? words * L.m.nb[s] : most;
    L.T_most = (most + 31) & ~31;
    // (single-stage rows: 2^20 of 7 points 0.024 ms with 64 threads, 0.036 with
    // 32; 2^21 of 3 points 0.024 and 0.019)
    L.T = S == 1 ? (st.n < 5 ? 32 : 64) : std::min(mixed_block(L.m, words, L.rmax, L.smem), L.T_most);
    *out = L;
    return 0;
}

int mixed_prepare(const MixedStages &st, bool cols, int nx, long long count, MixedLaunch *out, bool fourstep,
                  int fs_n1) {
    if (mixed_layout(st, cols, nx, count, out, fourstep, fs_n1) != 0) return -1;
    return smem_ok(mixed_fn(out->rmax, cols, out->fs.n1 > 0), out->smem) ? 0 : -1;
}

bool mixed_split(int n, int *n1, int *n2) {
    int best = 0;
    double bd = 1e30;
    for (int d = 2; d <= kMixedMaxN && d < n; ++d) {
        if (n % d || n / d > kMixedMaxN || !mixed_factor(d, nullptr) || !mixed_factor(n / d, nullptr)) continue;
        const double dist = fabs(log((double)d) - 0.5 * log((double)n));
        if (dist < bd) {
            bd = dist;
            best = d;
        }
    }
    if (!best) return false;
    *n2 = best;
    *n1 = n / best;
    return true;
}

cudaError_t launch_mixed(const MixedLaunch &L, const float2 *tw, const float2 *in, float2 *out, long long count,
                         int conj, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    if (L.T <= 0) return cudaErrorInvalidValue;
    // rows: count transforms, in groups that stay within one transform of a
    // four-step pass; columns: count slices of nx columns
    const int span = L.cols ? L.nx : L.fs.n1;
    long long ntrans = L.cols ? count * L.nx : count;
    const long long grid = span > 0 ? ntrans / span * ((span + L.W - 1) / L.W) : (ntrans + L.W - 1) / L.W;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const void *fn = mixed_fn(L.rmax, L.cols, L.fs.n1 > 0);
    int W = L.W, nx = L.nx;
    FourStepB fs = L.fs;
    void *args[] = {(void *)&in, (void *)&out, (void *)&tw, (void *)&L.m, (void *)&ntrans, (void *)&W,
                    (void *)&nx, (void *)&conj, (void *)&fs};
    // a launch that leaves room on every SM takes more threads, up to every
    // stage in one round
    int T = L.T;
    const long long per_sm = (grid + kMixedSms - 1) / kMixedSms;
    if (per_sm * T < mixed_threads(L.rmax)) {
        const int room = mixed_threads(L.rmax) / (int)per_sm & ~31;
        T = std::max(T, std::min(room, L.T_most));
    }
    return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(T), args, L.smem, s);
}

}  // namespace gb300fft

// The launch a plan makes of one mixed-radix pass.
extern "C" int fft_debug_mixed_launch(int n, int nx, long long count, int fourstep, int n1, int *info) {
    if (!info || nx < 0 || count < 1 || n1 < 0 || (nx > 0 && n1 > 0)) return FFT_ERR_INVALID_ARG;
    gb300fft::MixedStages st;
    gb300fft::MixedLaunch L;
    if (!gb300fft::mixed_factor(n, &st)) return FFT_ERR_INVALID_SIZE;
    if (gb300fft::mixed_layout(st, nx > 0, nx, count, &L, fourstep != 0, n1) != 0) return FFT_ERR_UNSUPPORTED;
    info[0] = L.rmax > 0 ? 2 : 1;
    info[1] = L.W;
    info[2] = L.T;
    info[3] = (int)L.smem;
    info[4] = L.rmax > 0 ? L.rmax : 16;
    info[5] = L.m.skew;
    info[6] = L.m.buf_elems;
    info[7] = L.m.S;
    for (int k = 0; k < 16; ++k) info[8 + k] = k < L.m.S ? L.m.radix[k] : 0;
    return FFT_OK;
}

// The float constants the composite-radix DFTs multiply by, as the
// compiler evaluates them (host copy of the same constexpr functions).
extern "C" int fft_debug_root(int m, int r, float *c, float *s) {
    if (!c || !s || r < 1) return FFT_ERR_INVALID_ARG;
    *c = (float)gb300fft::mixed::cos_2pi(m, r);
    *s = (float)gb300fft::mixed::sin_2pi(m, r);
    return FFT_OK;
}
