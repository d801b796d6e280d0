// Two-stage register FFTs (FP32) of the lengths N = P x Q listed in fft2.h and the pass kernels built on them.
//
// A transform of length N is shared by max(P, Q) threads.  With k = t + Q j and n = n1 + P n2 (w_m = e^{DIR 2 pi i / m})
//   X[n1 + P n2] = sum_t w_Q^(t n2) [ w_N^(t n1) sum_j x[t + Q j] w_P^(j n1) ]:
// thread t < Q takes the P-point DFT over j of its points in registers and multiplies by the twiddles, one exchange
// through shared memory hands row n1 to thread n1 < P, which takes the Q-point DFT over t.  A staged Stockham pass of the
// same length goes through shared memory once per radix (three to five times); these passes are bound by shared-memory
// wavefronts and instruction issue, not by DRAM, so the single exchange is what they gain.  P and Q are as close as
// they can be, so that neither stage idles many threads.  The points of a thread and all DFT coefficients are
// compile-time indexed; twiddles come from a table laid out [n1][t], so that a warp reads consecutive entries.
// Measured on cubic grids, forward transform and the maps of 4 bins (2 above n = 320), us, staged passes (with passes written
// for one length at 256, 288 and 512) / these:
//   n            64       96      128      180      216      256      300      320      360      400      480      512
// (before k_inv_z and the columns lost their branches, which took another 2 and 20 % off)
//   forward   16/17    35/17    24/21   118/34   192/44    85/58  413/100  347/112  710/146  956/185 1567/327  715/395
//   maps      21/22    31/27    46/35   317/71  566/140  272/160 1295/349 579/398 1298/324 1764/417 2779/964  967/947
#pragma once
#include "fft.cuh"
#include "fft2.h"

namespace pb {
namespace f2 {

// ------------------------------------------------------------------------------------------------ roots of unity

// cos and sin of x in [0, pi/4] by their Taylor series (the next terms are below 1e-19), evaluated at compile time.
__host__ __device__ constexpr double taylor_cos(double x) {
    double term = 1.0, sum = 1.0;
    for (int i = 1; i <= 10; ++i) {
        term *= -x * x / ((2 * i - 1) * (2 * i));
        sum += term;
    }
    return sum;
}
__host__ __device__ constexpr double taylor_sin(double x) {
    double term = x, sum = x;
    for (int i = 1; i <= 10; ++i) {
        term *= -x * x / ((2 * i) * (2 * i + 1));
        sum += term;
    }
    return sum;
}
struct Root {
    double c, s;
};
// e^{2 pi i m / n}, reduced exactly to an octant first.
__host__ __device__ constexpr Root root(int m, int n) {
    m %= n;
    const int o = 8 * m / n;
    const double q = 0.78539816339744830962;                       // pi / 4
    double x = q * (double)(8 * m - o * n) / (double)n;            // angle within the octant
    const bool odd = (o & 1) != 0;
    if (odd) x = q * (double)((o + 1) * n - 8 * m) / (double)n;    // measured from the octant's end
    const double c = taylor_cos(x), s = taylor_sin(x);
    switch (o) {
        case 0: return Root{c, s};
        case 1: return Root{s, c};
        case 2: return Root{-s, c};
        case 3: return Root{-c, s};
        case 4: return Root{-c, -s};
        case 5: return Root{-s, -c};
        case 6: return Root{s, -c};
        default: return Root{c, -s};
    }
}
template <int D> struct RootTab {
    float c[D], s[D];
    __host__ __device__ constexpr RootTab() : c(), s() {
        for (int m = 0; m < D; ++m) {
            const Root r = root(m, D);
            c[m] = (float)r.c;
            s[m] = (float)r.s;
        }
    }
};
// Gain of the twiddles, in units of 10^-9 above 1.  The FP32 roots and DFT constants miss the unit circle by up to 2^-25, and
// their mean over the paths through a transform of n points is a factor common to all outputs, 4e-8 off 1 for the worst
// lengths: three transforms at 256 points made every power spectrum 1.6e-7 too small, six at 512 and 288 every bispectrum
// 6.7e-7, while the random errors of their sums are below 1e-7.  Twiddles longer by these amounts before they are
// rounded bring the mean within 6e-9 of 1 (the transform matrix with the rounded constants, worked out in FP64).
__host__ __device__ constexpr int gain(int n) {
    switch (n) {
        case 48: return 17;
        case 54: return 33;
        case 60: return -5;
        case 64: return 11;
        case 72: return 22;
        case 80: return -7;
        case 90: return -3;
        case 96: return 16;
        case 100: return -28;
        case 108: return 28;
        case 120: return -5;
        case 128: return 21;
        case 144: return 23;
        case 150: return -26;
        case 160: return 1;
        case 180: return 2;
        case 192: return 19;
        case 200: return -32;
        case 216: return 33;
        case 240: return 5;
        case 256: return 23;
        case 270: return 15;
        case 288: return 35;
        case 300: return -27;
        case 320: return 0;
        case 324: return 45;
        case 360: return 3;
        case 384: return 25;
        case 400: return -34;
        case 432: return 40;
        case 480: return 1;
        case 512: return 31;
        default: return 0;
    }
}
// w_N^(t n1) as [n1][t].
template <int P, int Q> struct TwTab {
    float2 w[P * Q];
    __host__ __device__ constexpr TwTab() : w() {
        constexpr double g = 1.0 + 1e-9 * gain(P * Q);
        for (int a = 0; a < P; ++a)
            for (int t = 0; t < Q; ++t) {
                const Root r = root(a * t, P * Q);
                w[a * Q + t].x = a * t ? (float)(r.c * g) : 1.f;
                w[a * Q + t].y = a * t ? (float)(r.s * g) : 0.f;
            }
    }
};
template <int P, int Q> __device__ const TwTab<P, Q> kTw = TwTab<P, Q>();

// ------------------------------------------------------------------------------------------------ codelets

// Factors of a composite codelet R = A x B (B taken last).
__host__ __device__ constexpr int codelet_b(int R) {
    return R == 16 || R == 32 ? 4 : (R % 3 == 0 ? 3 : (R % 5 == 0 ? 5 : 2));
}
// a e^{DIR 2 pi i m / D} for constants m, D (after unrolling).
template <int DIR, int D> __device__ __forceinline__ float2 rot(float2 a, int m) {
    constexpr RootTab<D> tab{};
    m %= D;
    if (m == 0) return a;
    if (4 * m == D) return muli<float>(a, DIR);
    if (2 * m == D) return make_float2(-a.x, -a.y);
    if (4 * m == 3 * D) return muli<float>(a, -DIR);
    const float c = tab.c[m], s = DIR * tab.s[m];
    return make_float2(a.x * c - a.y * s, a.x * s + a.y * c);
}
// X[n] = sum_j x[j] e^{DIR 2 pi i j n / R}, natural order in and out, in registers.
template <int DIR, int R> __device__ __forceinline__ void codelet(float2* x) {
    if constexpr (R == 1) {
    } else if constexpr (R == 2 || R == 3 || R == 4 || R == 5 || R == 8) {
        dft<float, DIR>(x, R);
    } else {
        constexpr int B = codelet_b(R), A = R / B;
        float2 y[B][A];
#pragma unroll
        for (int b = 0; b < B; ++b) {
#pragma unroll
            for (int a = 0; a < A; ++a) y[b][a] = x[B * a + b];
            codelet<DIR, A>(y[b]);
        }
#pragma unroll
        for (int c = 0; c < A; ++c) {
            float2 z[B];
#pragma unroll
            for (int b = 0; b < B; ++b) z[b] = rot<DIR, R>(y[b][c], b * c);
            codelet<DIR, B>(z);
#pragma unroll
            for (int d = 0; d < B; ++d) x[c + A * d] = z[d];
        }
    }
}

// Stage 1 of thread t: v[j] = x[t + Q j] -> the twiddled rows v[n1].
template <int DIR, int P, int Q> __device__ __forceinline__ void stage1(float2* v, int t) {
    codelet<DIR, P>(v);
#pragma unroll
    for (int n1 = 1; n1 < P; ++n1) {
        const float2 w = kTw<P, Q>.w[n1 * Q + t];
        v[n1] = DIR > 0 ? mul<float>(v[n1], w) : mulc<float>(v[n1], w);
    }
}

// ------------------------------------------------------------------------------------------------ columns

// CTAs per SM asked of the compiler: registers for about 2.5 max(P, Q) complex values a thread (17 and 18 points: 72, so that
// three column CTAs of 288 threads fit an SM; with 80, two did, and the maps of 30 bins on 288^3 took 1.50 ms instead of 1.41).
__host__ __device__ constexpr int min_ctas(int threads, int pts) {
    const int regs = pts <= 12 ? 56 : (pts <= 16 ? 64 : (pts <= 18 ? 72 : (pts <= 20 ? 80 : 128)));
    const int n = 65536 / (threads * regs);
    return n < 1 ? 1 : n;
}

// Shared-memory wavefronts of the line exchanges of a CTA with TG threads a transform (8-byte accesses, half a warp at a
// time): rows of stride `row`, transforms gs apart; the writes of `act_w` threads at consecutive places and the reads of
// `act_r` threads one row apart.
__host__ __device__ constexpr int exchange_cost(int threads, int TG, int gs, int row, int act_w, int act_r) {
    int cost = 0;
    for (int h = 0; h < threads; h += 16) {
        int w[16] = {}, r[16] = {}, wm = 0, rm = 0;
        for (int i = h; i < h + 16 && i < threads; ++i) {
            const int g = i / TG, t = i % TG;
            if (t < act_w) {
                const int n = ++w[(g * gs + t) % 16];
                wm = n > wm ? n : wm;
            }
            if (t < act_r) {
                const int n = ++r[(g * gs + t * row) % 16];
                rm = n > rm ? n : rm;
            }
        }
        cost += wm + rm;
    }
    return cost;
}
// The same for the 4-byte stores of the real lines, transforms os numbers apart.
__host__ __device__ constexpr int store_cost(int threads, int TG, int os, int act) {
    int cost = 0;
    for (int h = 0; h < threads; h += 32) {
        int w[32] = {}, wm = 0;
        for (int i = h; i < h + 32 && i < threads; ++i)
            if (i % TG < act) {
                const int n = ++w[((i / TG) * os + i % TG) % 32];
                wm = n > wm ? n : wm;
            }
        cost += wm;
    }
    return cost;
}

template <int N> struct Geo {
    static constexpr int P = stage_p(N), Q = N / P, TG = P > Q ? P : Q;
    // columns: TC consecutive columns a CTA (128 or 64 bytes a row); with 64 bytes two rows share a half-warp, which an odd
    // row count keeps apart.  64 bytes where the buffer of 16 columns would leave an SM too few CTAs (forward / maps at 360
    // points 152 / 347 us with 16 columns, 146 / 324 with 8; at 400 193 / 451 and 185 / 417; at 324 no difference).
    static constexpr int TC = TG > 20 || N >= 360 ? 8 : 16, kColThreads = TG * TC;
    static constexpr int kColRow = TC == 8 ? (Q | 1) : Q;
    static constexpr int kColSmem = P * kColRow * TC * (int)sizeof(float2);
    // lines: G transforms a CTA
    static constexpr int G = 256 / TG, kLineThreads = G * TG;
    // odd row strides of the exchange buffers (P rows of Q, and Q rows of P for the masked pass) and the distance of the
    // transforms: the one of sixteen with the fewest bank conflicts
    static constexpr int QP = Q | 1, PP = P | 1;
    static constexpr int kBuf0 = P * QP > Q * PP ? P * QP : Q * PP, kBuf = kBuf0 > N ? kBuf0 : N;
    __host__ __device__ static constexpr int best_gs() {
        int best = kBuf, bc = 1 << 30;
        for (int gs = kBuf; gs < kBuf + 16; ++gs) {
            const int c = exchange_cost(kLineThreads, TG, gs, QP, Q, P) * 2 + exchange_cost(kLineThreads, TG, gs, PP, P, Q);
            if (c < bc) { bc = c; best = gs; }
        }
        return best;
    }
    static constexpr int GS = best_gs();
    // real lines on their way out: V numbers a global store, transforms OS numbers apart
    static constexpr int V = N % 4 == 0 ? 4 : 2;
    __host__ __device__ static constexpr int best_os() {
        int best = 2 * N, bc = 1 << 30;
        for (int os = 2 * N; os < 2 * N + 32; os += V) {
            const int c = store_cost(kLineThreads, TG, os, P);
            if (c < bc) { bc = c; best = os; }
        }
        return best;
    }
    static constexpr int OS = best_os();
    static constexpr int kLineSmem0 = G * GS * (int)sizeof(float2), kLineSmem1 = G * OS * (int)sizeof(float);
    static constexpr int kLineSmem = kLineSmem0 > kLineSmem1 ? kLineSmem0 : kLineSmem1;
};

// Wave number of point k = t + step j of N (j of cnt steps): k below N / 2, k - N from there on.  The half is known at compile
// time but for the middle j of an odd count.
template <int N> __device__ __forceinline__ int wave(int k, int j, int cnt) {
    return (2 * j + 1 == cnt ? 2 * k >= N : 2 * j >= cnt) ? k - N : k;
}

// One column (thread (t, c) of the CTA: column c of TC): load(k, f) gives point k, store(n, f, X) takes the results; f is
// the point's wave number.
template <int DIR, int N, class L, class S>
__device__ __forceinline__ void col_fft(float2* buf, int t, int c, L load, S store) {
    using E = Geo<N>;
    constexpr int P = E::P, Q = E::Q, TC = E::TC, QR = E::kColRow;
    if (t < Q) {
        float2 v[P];
#pragma unroll
        for (int j = 0; j < P; ++j) v[j] = load(t + Q * j, wave<N>(t + Q * j, j, P));
        stage1<DIR, P, Q>(v, t);
#pragma unroll
        for (int n1 = 0; n1 < P; ++n1) buf[(n1 * QR + t) * TC + c] = v[n1];
    }
    __syncthreads();
    if (t < P) {
        float2 v[Q];
#pragma unroll
        for (int u = 0; u < Q; ++u) v[u] = buf[(t * QR + u) * TC + c];
        codelet<DIR, Q>(v);
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) store(t + P * n2, wave<N>(t + P * n2, n2, Q), v[n2]);
    }
}

// Strided column pass, the same items and results as k_col.
template <int DIR, int N>
__global__ void __launch_bounds__(Geo<N>::kColThreads, min_ctas(Geo<N>::kColThreads, Geo<N>::TG)) k_col(ColBatch batch) {
    extern __shared__ __align__(16) float2 f2_smem[];
    constexpr int TC = Geo<N>::TC;
    const ColItem& item = batch.it[blockIdx.z];
    const int c0 = blockIdx.x * TC, o = blockIdx.y;
    if (c0 >= item.ncols || o >= item.nouter) return;   // uniform over the CTA
    const int t = threadIdx.x / TC, c = threadIdx.x - t * TC;
    const bool act = c0 + c < item.ncols;
    const float2* __restrict__ in = static_cast<const float2*>(item.in) + (long)o * item.in_os + c0 + c;
    float2* __restrict__ out = static_cast<float2*>(item.out) + (long)o * item.out_os + c0 + c;
    // 32-bit offsets (an outer index spans fewer than 2^31 elements); inactive columns keep nothing
    const int lo = item.rng.lo;
    const unsigned cnt = act ? item.rng.cnt : 0, in_es = (unsigned)item.in_es, out_es = (unsigned)item.out_es;
    col_fft<DIR, N>(
        f2_smem, t, c,
        [&](int k, int f) {
            if (DIR < 0) return act ? in[(unsigned)k * in_es] : make_float2(0.f, 0.f);
            const unsigned i = (unsigned)(f - lo);    // zero outside the kept range
            return i < cnt ? in[i * in_es] : make_float2(0.f, 0.f);
        },
        [&](int n, int f, float2 v) {
            if (DIR > 0) {
                if (act) out[(unsigned)n * out_es] = v;
            } else {
                const unsigned i = (unsigned)(f - lo);
                if (i < cnt) out[i * out_es] = v;
            }
        });
}

// First inverse pass with the shell filter, the same items and results as k_inv_x_filter.
template <int N>
__global__ void __launch_bounds__(Geo<N>::kColThreads, min_ctas(Geo<N>::kColThreads, Geo<N>::TG))
    k_xfilter(XInvBatch batch, const float2* __restrict__ spec, AxisRange gx, AxisRange gy, AxisRange gz, float scale) {
    extern __shared__ __align__(16) float2 f2_smem[];
    constexpr int TC = Geo<N>::TC;
    const XInvItem& item = batch.it[blockIdx.y];
    const int ncols = item.ry.cnt * item.rz.cnt;
    const int c0 = blockIdx.x * TC;
    if (c0 >= ncols) return;                          // uniform over the CTA
    const int t = threadIdx.x / TC, c = threadIdx.x - t * TC;
    const int cc = c0 + c;
    const bool act = cc < ncols;
    const int fy = act ? item.ry.lo + cc / item.rz.cnt : 0;
    const int fz = act ? item.rz.lo + cc % item.rz.cnt : 0;
    float2* __restrict__ out = static_cast<float2*>(item.out) + cc;
    const int rlo = item.rx.lo;
    const unsigned rcnt = act ? item.rx.cnt : 0;
    col_fft<+1, N>(
        f2_smem, t, c,
        [&](int, int fx) {
            float2 v = make_float2(0.f, 0.f);          // stays zero outside the bin
            if ((unsigned)(fx - rlo) < rcnt) x_filter_value<float>(item, spec, gx, gy, gz, scale, fx, fy, fz, v);
            return v;
        },
        [&](int n, int, float2 v) {
            if (act) out[(unsigned)(n * ncols)] = v;
        });
}

// First inverse pass of a triplet's Q-derivative spectrum, combined from the pair spectra on load.
template <int N>
__global__ void __launch_bounds__(Geo<N>::kColThreads, min_ctas(Geo<N>::kColThreads, Geo<N>::TG))
    k_xq(XqBatch batch, const float2* __restrict__ pairs, AxisRange gx, AxisRange gy, AxisRange gz) {
    extern __shared__ __align__(16) float2 f2_smem[];
    constexpr int TC = Geo<N>::TC;
    const XqItem& item = batch.it[blockIdx.y];
    const int ncols = item.ry.cnt * item.rz.cnt;
    const int c0 = blockIdx.x * TC;
    if (c0 >= ncols) return;                          // uniform over the CTA
    const int t = threadIdx.x / TC, c = threadIdx.x - t * TC;
    const int cc = c0 + c;
    const bool act = cc < ncols;
    const int fy = act ? item.ry.lo + cc / item.rz.cnt : 0;
    const int fz = act ? item.rz.lo + cc % item.rz.cnt : 0;
    const int syz = fy * fy + fz * fz;
    const float2* __restrict__ p = pairs + (fy - gy.lo) * gz.cnt + (fz - gz.lo);
    const int xs = gy.cnt * gz.cnt;
    float2* __restrict__ out = item.out + cc;
    const int rlo = item.rx.lo;
    const unsigned rcnt = act ? item.rx.cnt : 0;
    col_fft<+1, N>(
        f2_smem, t, c,
        [&](int, int fx) {
            float2 v = make_float2(0.f, 0.f);
            if ((unsigned)(fx - rlo) < rcnt) {
                const int s = fx * fx + syz;
                const long o = (long)(fx - gx.lo) * xs;
                if (s >= item.clo && s <= item.chi) v = add<float>(v, p[item.pab + o]);
                if (s >= item.alo && s <= item.ahi) v = add<float>(v, p[item.pbc + o]);
                if (s >= item.blo && s <= item.bhi) v = add<float>(v, p[item.pac + o]);
                v.x *= item.fac;
                v.y *= item.fac;
            }
            return v;
        },
        [&](int n, int, float2 v) {
            if (act) out[(unsigned)(n * ncols)] = v;
        });
}

// ------------------------------------------------------------------------------------------------ lines

// Stage-1 input of thread t of an inverse transform: points k = t + Q j of the packed Hermitian pair Z = X1 + i X2
// (kz < kin, zero above; imaginary parts of the kz = 0 and N/2 coefficients ignored).  Which half of the spectrum a point
// lies in is known at compile time (but for the middle j of an odd P), so the loads need one comparison each and are issued
// together.
template <int N>
__device__ __forceinline__ void load_hermitian(float2* v, const float2* __restrict__ in1, const float2* __restrict__ in2,
                                               bool has2, int kin, int t) {
    constexpr int P = Geo<N>::P, Q = Geo<N>::Q;
    float2 a[P], b[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int k = t + Q * j;
        const bool up = 2 * j + 1 == P ? 2 * k >= N : 2 * j >= P;   // k >= N / 2
        const int i = up ? N - k : k;
        const bool in = i < kin;
        a[j] = in ? in1[i] : make_float2(0.f, 0.f);
        b[j] = in && has2 ? in2[i] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < P; ++j) {
        const int k = t + Q * j;
        const bool up = 2 * j + 1 == P ? 2 * k >= N : 2 * j >= P;
        float ay = up ? -a[j].y : a[j].y, by = up ? -b[j].y : b[j].y;
        if ((j == 0 || 2 * j == P || 2 * j + 1 == P) && (k == 0 || 2 * k == N)) ay = by = 0.f;
        v[j] = make_float2(a[j].x - by, ay + b[j].x);
    }
}

// The transform's kz < kout coefficients of the two real lines from the packed result Z (in buf): thread t of TG.
template <int N>
__device__ __forceinline__ void split_lines(const float2* buf, float2* __restrict__ o1, float2* __restrict__ o2, bool has2,
                                            int kout, int t) {
    for (int k = t; k < kout; k += Geo<N>::TG) {
        const float2 zk = buf[k], zm = buf[k ? N - k : 0];
        // X1 = (Z[k] + conj Z[N-k]) / 2 ;  X2 = (Z[k] - conj Z[N-k]) / (2i)
        o1[k] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
        if (has2) o2[k] = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
    }
}

// Second half of a forward line transform: exchange and second stage, the packed result in buf.
template <int N>
__device__ __forceinline__ void fwd_rest(float2* v, float2* buf, int t, bool act, int kout) {
    constexpr int P = Geo<N>::P, Q = Geo<N>::Q, QP = Geo<N>::QP;
    __syncthreads();
    if (t < P && act) {
#pragma unroll
        for (int u = 0; u < Q; ++u) v[u] = buf[t * QP + u];
        codelet<-1, Q>(v);
    }
    __syncthreads();
    if (t < P && act) {
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            const int n = t + P * n2;
            if (n < kout || N - n < kout) buf[n] = v[n2];
        }
    }
    __syncthreads();
}

// z-pass, forward (R2C), the same results as k_fwd_z: lines 2p and 2p + 1 packed as one complex line, multiplied on
// load, kz < kout stored.  An item with sub holds differences of two products, in m1 - sub sub_m (m2 unused).
template <int N>
__global__ void __launch_bounds__(Geo<N>::kLineThreads, min_ctas(Geo<N>::kLineThreads, Geo<N>::TG))
    k_fwd_z(ZFwdBatch batch, long nlines, int kout) {
    extern __shared__ __align__(16) float2 f2_smem[];
    using E = Geo<N>;
    constexpr int P = E::P, Q = E::Q, QP = E::QP;
    const ZFwdItem& item = batch.it[blockIdx.y];
    const int g = threadIdx.x / E::TG, t = threadIdx.x - g * E::TG;
    float2* buf = f2_smem + g * E::GS;
    const long l1 = 2 * ((long)blockIdx.x * E::G + g);
    const bool act = l1 < nlines, has2 = l1 + 1 < nlines;
    float2 v[E::TG];
    if (t < Q && act) {
        const long i0 = l1 * N + t;
        const float* __restrict__ in = item.in + i0;
        const int d2 = has2 ? N : 0;                  // without a second line the first stands in for it, zeroed
#pragma unroll
        for (int j = 0; j < P; ++j) v[j] = make_float2(in[Q * j], in[Q * j + d2]);
        if (item.m1) {
            const float* __restrict__ m = item.m1 + i0;
#pragma unroll
            for (int j = 0; j < P; ++j) {
                v[j].x *= m[Q * j];
                v[j].y *= m[Q * j + d2];
            }
        }
        if (item.sub) {
            const float* __restrict__ a = item.sub + i0;
            const float* __restrict__ b = item.sub_m + i0;
#pragma unroll
            for (int j = 0; j < P; ++j) {
                v[j].x -= a[Q * j] * b[Q * j];
                v[j].y -= a[Q * j + d2] * b[Q * j + d2];
            }
        } else if (item.m2) {
            const float* __restrict__ m = item.m2 + i0;
#pragma unroll
            for (int j = 0; j < P; ++j) {
                v[j].x *= m[Q * j];
                v[j].y *= m[Q * j + d2];
            }
        }
        if (!has2) {
#pragma unroll
            for (int j = 0; j < P; ++j) v[j].y = 0.f;
        }
        stage1<-1, P, Q>(v, t);
#pragma unroll
        for (int n1 = 0; n1 < P; ++n1) buf[n1 * QP + t] = v[n1];
    }
    fwd_rest<N>(v, buf, t, act, kout);
    if (act) split_lines<N>(buf, item.out + l1 * kout, item.out + (l1 + 1) * kout, has2, kout, t);
}

// The same for harmonic-weighted fields.  Along a line Ybar_l,m and Ybar_l,-m differ by a constant, Re or Im of
// e^{i |m| phi}, so an item is one |m|: the field times the part that depends on the polar angle is transformed once and
// leaves multiplied by either constant.  With u = cos^2, s2 = sin^2 and sc = sin cos of the polar angle (one reciprocal a
// cell, no root), that part is s2^(|m| / 2) (times sc for odd |m|) times a polynomial in u.  The items of a line block are
// consecutive blocks, so that those that read the same lines run together (the field and its weight come from DRAM once
// for all of them).  Bound by instruction issue.  The numerator with ell = 2 and 4 on 256^3 took 1295 us with a transform and
// a root and a division a cell for every harmonic (950 in this kernel) and takes 855.
template <int N>
__global__ void __launch_bounds__(Geo<N>::kLineThreads, min_ctas(Geo<N>::kLineThreads, Geo<N>::TG))
    k_fwd_z_ylm(YlmBatch batch, int nitem, long nlines, int kout) {
    extern __shared__ __align__(16) float2 f2_smem[];
    using E = Geo<N>;
    constexpr int P = E::P, Q = E::Q, QP = E::QP;
    const unsigned lb = blockIdx.x / (unsigned)nitem;
    const YlmItem& item = batch.it[blockIdx.x - lb * (unsigned)nitem];
    const int g = threadIdx.x / E::TG, t = threadIdx.x - g * E::TG;
    float2* buf = f2_smem + g * E::GS;
    const long l1 = 2 * ((long)lb * E::G + g);
    const bool act = l1 < nlines, has2 = l1 + 1 < nlines;
    // offset of line l from the observer in the plane
    auto plane = [&](long l, float& px, float& py) {
        const int ix = (int)((unsigned)l / (unsigned)batch.n1), iy = (int)l - ix * batch.n1;
        px = ((float)(ix - batch.cell[0]) - batch.frac[0]) * batch.h[0];
        py = ((float)(iy - batch.cell[1]) - batch.frac[1]) * batch.h[1];
    };
    float2 v[E::TG];
    if (t < Q && act) {
        const float c0 = item.am < 2 ? 1.f : 0.f, c1 = (item.am >> 1) == 1 ? 1.f : 0.f, c2 = item.am == 4 ? 1.f : 0.f;
        const float tz = (float)(t - batch.cell[2]);
        const float o0 = item.am & 1 ? 0.f : 1.f, o1 = 1.f - o0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long l = l1 + (has2 ? h : 0);
            const float* __restrict__ in = batch.in + l * N + t;
            float px, py;
            plane(l, px, py);
            const float rho2 = px * px + py * py, rho = sqrtf(rho2);
#pragma unroll
            for (int j = 0; j < P; ++j) {
                const float pz = (tz + (float)(Q * j) - batch.frac[2]) * batch.h[2];
                const float r2 = rho2 + pz * pz;
                const bool at = r2 > 0.f;             // the z axis where the centre coincides with the observer
                const float q = __frcp_rn(at ? r2 : 1.f);
                const float zq = pz * q, u = at ? pz * zq : 1.f, s2 = rho2 * q, sc = rho * zq;
                const float y = ((item.d4 * u + item.d2) * u + item.d0) * (c0 + s2 * (c1 + s2 * c2)) * (o0 + o1 * sc);
                float f = in[Q * j];
                if (batch.w) f *= batch.w[l * N + t + Q * j];
                f *= y;
                if (h == 0) v[j].x = f;
                else v[j].y = has2 ? f : 0.f;
            }
        }
        stage1<-1, P, Q>(v, t);
#pragma unroll
        for (int n1 = 0; n1 < P; ++n1) buf[n1 * QP + t] = v[n1];
    }
    fwd_rest<N>(v, buf, t, act, kout);
    if (!act) return;
    float re[2], im[2];                               // e^{i |m| phi} of the two lines (1 on the axis)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float px, py;
        plane(l1 + h, px, py);
        const float rho2 = px * px + py * py;
        const float inv = rho2 > 0.f ? 1.f / sqrtf(rho2) : 0.f;
        const float cx = rho2 > 0.f ? px * inv : 1.f, cy = py * inv;
        float a = 1.f, b = 0.f;
        for (int q = 0; q < item.am; ++q) {
            const float a2 = a * cx - b * cy;
            b = a * cy + b * cx;
            a = a2;
        }
        re[h] = a;
        im[h] = b;
    }
    for (int k = t; k < kout; k += E::TG) {
        const float2 zk = buf[k], zm = buf[k ? N - k : 0];
        const float2 x1 = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
        const float2 x2 = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
        const long o = l1 * kout + k;
        if (item.re) {
            item.re[o] = make_float2(x1.x * re[0], x1.y * re[0]);
            if (has2) item.re[o + kout] = make_float2(x2.x * re[1], x2.y * re[1]);
        }
        if (item.im) {
            item.im[o] = make_float2(x1.x * im[0], x1.y * im[0]);
            if (has2) item.im[o + kout] = make_float2(x2.x * im[1], x2.y * im[1]);
        }
    }
}

// z-pass, inverse (C2R), the same results as k_inv_z.  The real lines go through shared memory so that the CTA's 2G lines,
// one contiguous block, are written in 16-byte pieces (4-byte stores of P consecutive numbers straight from the registers
// took 1.54 ms for 30 maps of 288^3 cells).  With absmax, absmax[item] takes the largest magnitude written (bit pattern),
// which the triplet contraction scales by.  Bound by instruction issue and by the latency of its loads: 30 maps of 288^3
// cells took 1.25 ms while the branches of the Hermitian input kept its loads apart, and take 0.93 ms (0.57 ms at the copy
// rate).
template <int N>
__global__ void __launch_bounds__(Geo<N>::kLineThreads, min_ctas(Geo<N>::kLineThreads, Geo<N>::TG))
    k_inv_z(ZInvBatch batch, long nlines, float scale, const float* __restrict__ mulout, uint32_t* __restrict__ absmax) {
    extern __shared__ __align__(16) float2 f2_smem[];
    using E = Geo<N>;
    constexpr int P = E::P, Q = E::Q, QP = E::QP;
    const ZInvItem& item = batch.it[blockIdx.y];
    const int kin = item.kin;
    const int g = threadIdx.x / E::TG, t = threadIdx.x - g * E::TG;
    float2* buf = f2_smem + g * E::GS;
    const long l0 = 2 * (long)blockIdx.x * E::G, l1 = l0 + 2 * g;
    const bool act = l1 < nlines, has2 = l1 + 1 < nlines;
    const float2* __restrict__ in = static_cast<const float2*>(item.in) + l1 * kin;
    float2 v[E::TG];
    if (t < Q && act) {
        load_hermitian<N>(v, in, in + kin, has2, kin, t);
        stage1<+1, P, Q>(v, t);
#pragma unroll
        for (int n1 = 0; n1 < P; ++n1) buf[n1 * QP + t] = v[n1];
    }
    __syncthreads();
    if (t < P && act) {
#pragma unroll
        for (int u = 0; u < Q; ++u) v[u] = buf[t * QP + u];
        codelet<+1, Q>(v);
    }
    __syncthreads();
    if (t < P && act) {
        float* re = reinterpret_cast<float*>(f2_smem) + g * E::OS + t;
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            re[P * n2] = v[n2].x * scale;
            re[P * n2 + N] = v[n2].y * scale;
        }
    }
    __syncthreads();
    // lines l0 .. of the CTA, V numbers a store
    constexpr int V = E::V, NV = N / V, T = E::kLineThreads, STEPS = (2 * E::G * NV + T - 1) / T;
    using VT = typename std::conditional<V == 4, float4, float2>::type;
    const int nl = (int)min((long)2 * E::G, nlines - l0);
    VT* __restrict__ out = reinterpret_cast<VT*>(static_cast<float*>(item.out) + l0 * N);
    float top = 0.f;
    int l = (int)threadIdx.x / NV, e = (int)threadIdx.x - l * NV;
#pragma unroll
    for (int i = 0; i < STEPS; ++i) {
        if (l >= nl) break;
        VT a = *reinterpret_cast<const VT*>(reinterpret_cast<const float*>(f2_smem) + (l >> 1) * E::OS + (l & 1) * N + V * e);
        float* p = reinterpret_cast<float*>(&a);
        if (mulout) {
#pragma unroll
            for (int c = 0; c < V; ++c) p[c] *= mulout[(l0 + l) * N + V * e + c];
        }
#pragma unroll
        for (int c = 0; c < V; ++c) top = fmaxf(top, fabsf(p[c]));
        out[l * NV + e] = a;
        l += T / NV;
        e += T % NV;
        if (e >= NV) { e -= NV; ++l; }
    }
    if (absmax) {
        const int lanes = E::kLineThreads - (int)(threadIdx.x & ~31u);     // of this warp (the last one may be partial)
        const uint32_t most = __reduce_max_sync(lanes >= 32 ? 0xffffffffu : (1u << lanes) - 1u, __float_as_uint(top));
        // (a look first: of the hundreds of thousands of warps few still raise the maximum)
        if ((threadIdx.x & 31) == 0 && most > __ldcg(absmax + blockIdx.y)) atomicMax(absmax + blockIdx.y, most);
    }
}

// C2R z-pass, product with the real map s (same grid, lines l1, l1 + 1) and R2C z-pass in one kernel: the real lines
// never leave the registers.  The inverse transform leaves n = n1 + P n2 in thread n1, which is what the forward one with
// P and Q exchanged starts from.
template <int N>
__global__ void __launch_bounds__(Geo<N>::kLineThreads, min_ctas(Geo<N>::kLineThreads, Geo<N>::TG))
    k_mask_z(ZMaskBatch batch, long nlines, const float* __restrict__ s, int kout) {
    extern __shared__ __align__(16) float2 f2_smem[];
    using E = Geo<N>;
    constexpr int P = E::P, Q = E::Q, QP = E::QP, PP = E::PP;
    const ZMaskItem& item = batch.it[blockIdx.y];
    const int kin = item.kin;
    const int g = threadIdx.x / E::TG, t = threadIdx.x - g * E::TG;
    float2* buf = f2_smem + g * E::GS;
    const long l1 = 2 * ((long)blockIdx.x * E::G + g);
    const bool act = l1 < nlines, has2 = l1 + 1 < nlines;
    const float2* __restrict__ in = item.in + l1 * kin;
    float2 v[E::TG];
    if (t < Q && act) {
        load_hermitian<N>(v, in, in + kin, has2, kin, t);
        stage1<+1, P, Q>(v, t);
#pragma unroll
        for (int n1 = 0; n1 < P; ++n1) buf[n1 * QP + t] = v[n1];
    }
    __syncthreads();
    if (t < P && act) {
#pragma unroll
        for (int u = 0; u < Q; ++u) v[u] = buf[t * QP + u];
        codelet<+1, Q>(v);
        const float* __restrict__ sm = s + l1 * N + t;
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            v[n2].x *= sm[P * n2];
            v[n2].y = has2 ? v[n2].y * sm[P * n2 + N] : 0.f;
        }
        stage1<-1, Q, P>(v, t);
    }
    __syncthreads();                                  // every row of the first exchange has been read
    if (t < P && act) {
#pragma unroll
        for (int n1 = 0; n1 < Q; ++n1) buf[n1 * PP + t] = v[n1];
    }
    __syncthreads();
    if (t < Q && act) {
#pragma unroll
        for (int u = 0; u < P; ++u) v[u] = buf[t * PP + u];
        codelet<-1, P>(v);
    }
    __syncthreads();
    if (t < Q && act) {
#pragma unroll
        for (int n2 = 0; n2 < P; ++n2) {
            const int n = t + Q * n2;
            if (n < kout || N - n < kout) buf[n] = v[n2];
        }
    }
    __syncthreads();
    if (act) split_lines<N>(buf, item.out + l1 * kout, item.out + (l1 + 1) * kout, has2, kout, t);
}

}  // namespace f2
}  // namespace pb
