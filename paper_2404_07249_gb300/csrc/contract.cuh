// Triplet contraction M[(j<=k)][i] = sum_x g_j(x) g_k(x) h_i(x) over all grid cells x
// (the real-space sum of the separable bispectrum, Sec. 4.3.1 eq. beta-def; with h = g it gives
// S_abc for every a <= b and every c).  SIMT version: each CTA owns a range of cells and a group of
// pair rows; per chunk of CH cells it stages the maps in shared memory, forms the pair products once,
// and every thread accumulates a TM x TN register tile of outputs.
//
// Few rows leave most of a CTA without a tile (36 pairs x 8 singles are nine tiles of 4 x 8), so the tiles are
// replicated kg times over the threads, replica q taking the cells q, q + kg, .. of every chunk; the replicas are added
// in order at the end.  The next chunk's maps are loaded into registers while the current one is worked on, and
// products and singles are written as 16-byte pieces with row strides of an odd number of pieces (no bank conflicts, no
// division by run-time sizes per element).
//
// FP32 sums are register pairs (fma.rn.f32x2), and the places of a row's maps are looked up once a CTA, not once a product.
// Measured at 13 bins (55 rows x 13 singles) on 100^3 cells: 845 us before the replicas, 359 us with them, 270 us now;
// instruction issue bounds it.
//
// Precision: products and sums of kFlush chunks in the maps' precision, added to FP64 totals (FP32: the sums are short enough
// for 24 bits; FP64: no sum is longer than 512 terms however many cells a CTA takes); per-CTA FP64 partials are reduced
// across CTAs in a fixed order (deterministic).
#pragma once
#include <algorithm>

#include "common.cuh"

namespace pb {

constexpr int kCH = 32;       // cells per chunk (one a lane when products are formed)
constexpr int kTM = 4;        // pair rows per thread
constexpr int kTN = 8;        // singles per thread
constexpr int kFlush = 16;    // chunks per partial sum (512 cells)
constexpr int kGS = kCH + 1;  // row stride of the staged maps

struct ContractGeom {
    int nb, nh, npairs;
    int rt, ct;        // thread tile grid (rt * ct <= 256)
    int kg;            // replicas of the tile grid over the cells of a chunk (rt * ct * kg <= 256)
    int rows_cta;      // pair rows per CTA (multiple of kTM)
    int rps;           // row stride of the product array (elements; an odd multiple of 4, >= rows_cta)
    int nhp;           // row stride of the singles array (an odd multiple of 4, >= ct * kTN)
    int ngroups;       // row groups
    int ncb;           // cell blocks
    long cells_cta;    // cells per CTA (multiple of kCH)
};

// Geometry of npairs rows against nh singles out of nb staged maps over ncell cells.
inline ContractGeom contract_geom_rows(int nb, int npairs, int nh, long ncell) {
    ContractGeom G;
    G.nb = nb; G.nh = nh; G.npairs = npairs;
    G.ct = (nh + kTN - 1) / kTN;
    const int need = (npairs + kTM - 1) / kTM * kTM;
    G.rows_cta = std::min(256 / G.ct * kTM, need);
    G.rt = G.rows_cta / kTM;
    G.kg = std::min(256 / (G.rt * G.ct), kCH);
    G.rps = G.rows_cta / 4 % 2 ? G.rows_cta : G.rows_cta + 4;
    G.nhp = G.ct * kTN + 4;
    G.ngroups = (npairs + G.rows_cta - 1) / G.rows_cta;
    const long nchunks = (ncell + kCH - 1) / kCH;
    long ncb = std::max(1L, std::min(nchunks, (long)(4 * 152 / G.ngroups)));
    G.cells_cta = ((ncell + ncb - 1) / ncb + kCH - 1) / kCH * kCH;
    G.ncb = (int)((ncell + G.cells_cta - 1) / G.cells_cta);
    return G;
}

// Dynamic shared memory: products [kCH][rps], singles [kCH][nhp], maps [nb][kGS]; at the end the tiles' sums of one
// replica (FP64; only with replicas, then at most 128 tiles) in the place of the products.
constexpr size_t kMaxSmem = 227 * 1024;
template <typename T> __host__ __device__ inline size_t contract_work(const ContractGeom& G) {
    return ((size_t)kCH * G.rps + (size_t)kCH * G.nhp + (size_t)G.nb * kGS) * sizeof(T);
}
// Behind them a row of zeros and the places of the rows' maps, where shared memory has room for these (it has but for
// about 800 FP64 rows and more; the pairs are then looked up a product).
template <typename T> __host__ __device__ inline size_t contract_table(const ContractGeom& G) {
    const size_t n = kGS * sizeof(T) + (size_t)G.rows_cta * sizeof(int2) + 16;
    return contract_work<T>(G) + n + 16 <= kMaxSmem ? n : 0;
}
template <typename T> inline size_t contract_smem(const ContractGeom& G) {
    const size_t sums = G.kg > 1 ? (size_t)G.rt * G.ct * kTM * kTN * sizeof(double) : 0;
    return std::max(contract_work<T>(G) + contract_table<T>(G), sums) + 16;
}

template <typename T> struct Vec4;
template <> struct Vec4<float> {
    __device__ __forceinline__ static void load(const float* p, float* v) {
        float4 a = *reinterpret_cast<const float4*>(p);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    }
    __device__ __forceinline__ static void store(float* p, const float* v) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <> struct Vec4<double> {
    __device__ __forceinline__ static void load(const double* p, double* v) {
        double2 a = *reinterpret_cast<const double2*>(p);
        double2 b = *reinterpret_cast<const double2*>(p + 2);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
    __device__ __forceinline__ static void store(double* p, const double* v) {
        *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
    }
};

__device__ __forceinline__ uint64_t pair_bits(float a, float b) {
    return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}

// Singles: rows hsub .. hsub + nh - 1 of g when h is null, else the maps h.
template <typename T>
__global__ void __launch_bounds__(256, 2) k_contract(const T* __restrict__ g, const T* __restrict__ h, int hsub, long ncell,
                                                  const short2* __restrict__ pairs, ContractGeom G,
                                                  double* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int RPS = G.rps, NHP = G.nhp;
    T* sP = reinterpret_cast<T*>(smem_raw);          // [kCH][RPS]
    T* sH = sP + (size_t)kCH * RPS;                   // [kCH][NHP]
    T* sG = sH + (size_t)kCH * NHP;                   // [nb][kGS], and with a table a row of zeros
    // table: places of the rows' maps in sG (the zeros beyond the last pair)
    const bool table = contract_table<T>(G) != 0;
    int2* sO = reinterpret_cast<int2*>((reinterpret_cast<uintptr_t>(sG + (G.nb + 1) * kGS) + 15) & ~(uintptr_t)15);
    const int r0 = blockIdx.x * G.rows_cta;
    if (table) {
        for (int i = tid; i < G.rows_cta; i += 256) {
            const bool in = r0 + i < G.npairs;
            const short2 jk = in ? pairs[r0 + i] : make_short2(0, 0);
            sO[i] = in ? make_int2(jk.x * kGS, jk.y * kGS) : make_int2(G.nb * kGS, G.nb * kGS);
        }
        if (tid < kGS) sG[G.nb * kGS + tid] = T(0);
    }
    const long cbeg = (long)blockIdx.y * G.cells_cta;
    const long cend = min(ncell, cbeg + G.cells_cta);
    // tile (rt, ct) of replica kq; threads beyond the last replica only stage
    const int ntile = G.rt * G.ct;
    const int kq = tid / ntile, tt = tid - kq * ntile;
    const int ct = tt / G.rt, rt = tt - ct * G.rt;
    const bool active = kq < G.kg;

    // FP32 sums two a register pair: one f32x2 instruction is two fused multiply-adds
    uint64_t acc[kTM][kTN / 2];
    double acc64[kTM][kTN];                           // totals; FP64: the sums
#pragma unroll
    for (int u = 0; u < kTM; ++u)
#pragma unroll
        for (int v = 0; v < kTN; ++v) { acc[u][v / 2] = 0; acc64[u][v] = 0.0; }
    // FP64 totals lie in local memory, touched every 512 cells: with both in registers an SM holds one CTA, and the bispectrum
    // of 8 bins on 64^3 cells took 462 us instead of 337 (334 with one running sum)
    volatile double total[sizeof(T) == 8 ? kTM * kTN : 1];
    bool have_total = false;
    auto flush = [&]() {
#pragma unroll
        for (int u = 0; u < kTM; ++u)
#pragma unroll
            for (int v = 0; v < kTN; v += 2) {
                if constexpr (sizeof(T) == 8) {
                    for (int q = v; q < v + 2; ++q) {
                        total[u * kTN + q] = have_total ? total[u * kTN + q] + acc64[u][q] : acc64[u][q];
                        acc64[u][q] = 0.0;
                    }
                } else {
                    acc64[u][v] += (double)__uint_as_float((unsigned)acc[u][v / 2]);
                    acc64[u][v + 1] += (double)__uint_as_float((unsigned)(acc[u][v / 2] >> 32));
                    acc[u][v / 2] = 0;
                }
            }
        have_total = true;
    };

    // warp w stages maps w, w + 8, .. (at most 8 of g, 8 of h), lane = cell
    T pre[8], preh[8];
    auto fetch = [&](long c0) {
        const long cell = c0 + lane;
        const bool in = cell < cend;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int b = warp + 8 * i;
            pre[i] = in && b < G.nb ? g[(long)b * ncell + cell] : T(0);
        }
        if (h) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int b = warp + 8 * i;
                preh[i] = in && b < G.nh ? h[(long)b * ncell + cell] : T(0);
            }
        }
    };
    int chunk = 0;
    fetch(cbeg);
    for (long c0 = cbeg; c0 < cend; c0 += kCH, ++chunk) {
        __syncthreads();                              // the previous chunk's products and singles have been read
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (warp + 8 * i < G.nb) sG[(warp + 8 * i) * kGS + lane] = pre[i];
        if (h) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (warp + 8 * i < G.nh) sH[lane * NHP + warp + 8 * i] = preh[i];
        }
        __syncthreads();
        if (c0 + kCH < cend) fetch(c0 + kCH);
        if (table) {
            for (int q = warp; q < G.rows_cta / 4; q += 8) {
                const int4 o = *reinterpret_cast<const int4*>(sO + 4 * q), p = *reinterpret_cast<const int4*>(sO + 4 * q + 2);
                const T v[4] = {sG[o.x + lane] * sG[o.y + lane], sG[o.z + lane] * sG[o.w + lane],
                                sG[p.x + lane] * sG[p.y + lane], sG[p.z + lane] * sG[p.w + lane]};
                Vec4<T>::store(sP + lane * RPS + 4 * q, v);
            }
        } else {
            for (int q = warp; q < G.rows_cta / 4; q += 8) {
                T v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int gp = r0 + 4 * q + u;
                    const short2 jk = gp < G.npairs ? pairs[gp] : make_short2(0, 0);
                    v[u] = gp < G.npairs ? sG[jk.x * kGS + lane] * sG[jk.y * kGS + lane] : T(0);
                }
                Vec4<T>::store(sP + lane * RPS + 4 * q, v);
            }
        }
        if (!h) {
            for (int q = warp; q < G.ct * (kTN / 4); q += 8) {
                T v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = 4 * q + u < G.nh ? sG[(hsub + 4 * q + u) * kGS + lane] : T(0);
                Vec4<T>::store(sH + lane * NHP + 4 * q, v);
            }
        }
        __syncthreads();
        if (active) {
#pragma unroll 2
            for (int x = kq; x < kCH; x += G.kg) {
                T a[kTM], b[kTN];
                Vec4<T>::load(sP + x * RPS + rt * kTM, a);
                Vec4<T>::load(sH + x * NHP + ct * kTN, b);
                Vec4<T>::load(sH + x * NHP + ct * kTN + 4, b + 4);
#pragma unroll
                for (int u = 0; u < kTM; ++u)
#pragma unroll
                    for (int v = 0; v < kTN; v += 2) {
                        if constexpr (sizeof(T) == 8) {
                            acc64[u][v] = fma(a[u], b[v], acc64[u][v]);
                            acc64[u][v + 1] = fma(a[u], b[v + 1], acc64[u][v + 1]);
                        } else {
                            asm("fma.rn.f32x2 %0, %1, %2, %0;"
                                : "+l"(acc[u][v / 2])
                                : "l"(pair_bits(a[u], a[u])), "l"(pair_bits(b[v], b[v + 1])));
                        }
                    }
            }
            if ((chunk + 1) % kFlush == 0) flush();
        }
    }
    if constexpr (sizeof(T) == 4) {
        flush();
    } else if (have_total) {
#pragma unroll
        for (int u = 0; u < kTM; ++u)
#pragma unroll
            for (int v = 0; v < kTN; ++v) acc64[u][v] += total[u * kTN + v];
    }
    // replicas 1, 2, .. are added to replica 0 in order
    double* red = reinterpret_cast<double*>(smem_raw);   // [kTM * kTN][ntile]
    for (int q = 1; q < G.kg; ++q) {
        __syncthreads();
        if (kq == q) {
#pragma unroll
            for (int u = 0; u < kTM; ++u)
#pragma unroll
                for (int v = 0; v < kTN; ++v) red[(u * kTN + v) * ntile + tt] = acc64[u][v];
        }
        __syncthreads();
        if (kq == 0) {
#pragma unroll
            for (int u = 0; u < kTM; ++u)
#pragma unroll
                for (int v = 0; v < kTN; ++v) acc64[u][v] += red[(u * kTN + v) * ntile + tt];
        }
    }
    if (kq != 0) return;
    double* out = partial + (size_t)blockIdx.y * G.npairs * G.nh;
#pragma unroll
    for (int u = 0; u < kTM; ++u) {
        const int gp = r0 + rt * kTM + u;
        if (gp >= G.npairs) continue;
#pragma unroll
        for (int v = 0; v < kTN; ++v) {
            const int i = ct * kTN + v;
            if (i < G.nh) out[(size_t)gp * G.nh + i] = acc64[u][v];
        }
    }
}

// Sum per-cell-block partials in a fixed order: out[o] = sum_cb partial[cb][o].  32 outputs x 16 slices of the blocks a
// CTA (blockDim (32, 16)): slice q sums blocks q, q + 16, .. with coalesced loads that do not wait for one another, the
// slices are then added in order.  Bound by load latency: one thread an output took 94 us for 559 blocks.
constexpr int kRedSlices = 16;
static __global__ void __launch_bounds__(32 * kRedSlices) k_reduce_partials(const double* __restrict__ partial, int ncb,
                                                                            long nout, double* __restrict__ out) {
    __shared__ double red[kRedSlices][33];
    const long o = (long)blockIdx.x * 32 + threadIdx.x;
    double s = 0.0;
    if (o < nout) {
#pragma unroll 8
        for (int cb = threadIdx.y; cb < ncb; cb += kRedSlices) s += partial[(size_t)cb * nout + o];
    }
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y || o >= nout) return;
    for (int q = 1; q < kRedSlices; ++q) s += red[q][threadIdx.x];
    out[o] = s;
}
inline unsigned reduce_blocks(long nout) { return (unsigned)((nout + 31) / 32); }

// ------------------------------------------------------------------------------------------------
// The double of a float.  A conversion instruction takes a slot of the FP64 pipe, which has two lanes a clock an SM on this
// part; for normal numbers the bits are moved by integer instructions instead.
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), m = u & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
    return (double)f;                                 // zeros, subnormal numbers, infinities, NaN
}
__device__ __forceinline__ double widen(double f) { return f; }

// Binned products over the half spectrum (Sec. 3.4.1, eq. pk-limit; Sec. 3.3.2, eq. fish-from-Q):
//   partial[z][b][seg][ell] = sum_{modes of segment seg of bin b} coef_ell Re(conj X_z A),
// coef_ell = w_k L_ell(mu) (w_k = 1 on the kz = 0 and Nyquist planes, 2 elsewhere) precomputed per mode in FP64; with
// X = A it gives the sums of L_ell |D|^2 over the full k-grid.  X_z = X + z x_stride.  One CTA per (bin, segment of that
// bin's mode list, NZ of the nx spectra); FP64 sums in a fixed order.  Bound by the FP64 pipe (two lanes a clock an SM):
// two operations a mode and spectrum for the product and one for each ell, after the conversions have left it (four of nine
// operations) and with one warp a sum at the end instead of a tree over all threads.  plan_pk cuts the lists into about four
// segments an SM, at most 8192 a bin: with 8192 modes a segment, 20 to 40 CTAs took 70 us for 64^3 and for 256^3 alike.
// Measured, before and after these two: 64^3 FP64 14.0 -> 6.7 us, 24 x 3 spectra on 256^3 (24 bins, three ells) 814 -> 575 us,
// 512^3 with 30 bins 58 -> 44 us (a segment of at most 1024 modes keeps enough warps in flight there: 87 us with 3072).
constexpr int kXbThreads = 128;
template <typename T, int NZ>
__global__ void __launch_bounds__(kXbThreads) k_cross_bin(const C<T>* __restrict__ X, const C<T>* __restrict__ A, long x_stride,
                                                          int nx, const int* __restrict__ offs,
                                                          const double* __restrict__ coef, long nmodes_total,
                                                          const int* __restrict__ bin_start, int nell, int seg_len,
                                                          double* __restrict__ partial) {
    __shared__ double red[NZ * 3][kXbThreads];
    const int b = blockIdx.x, seg = blockIdx.y, z0 = blockIdx.z * NZ, nz = min(NZ, nx - z0), tid = threadIdx.x;
    const long beg = bin_start[b] + (long)seg * seg_len;
    const long end = min((long)bin_start[b + 1], beg + seg_len);
    const C<T>* __restrict__ Xz = X + (long)z0 * x_stride;
    auto out = [&](int z) { return partial + (((long)(z0 + z) * gridDim.x + b) * gridDim.y + seg) * nell; };
    if (beg >= end) {
        if (tid < nell)
            for (int z = 0; z < nz; ++z) out(z)[tid] = 0.0;
        return;
    }
    double s[NZ][3] = {};
#pragma unroll NZ == 1 ? 4 : 2
    for (long m = beg + tid; m < end; m += kXbThreads) {
        const int o = offs[m];
        const C<T> a = A[o];
        C<T> x[NZ];
#pragma unroll
        for (int z = 0; z < NZ; ++z) x[z] = Xz[(long)(z < nz ? z : 0) * x_stride + o];
        double c[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) c[l] = l < nell ? coef[(long)l * nmodes_total + m] : 0.0;
        const double ax = widen(a.x), ay = widen(a.y);
#pragma unroll
        for (int z = 0; z < NZ; ++z) {
            if (z >= nz) break;
            const double p = widen(x[z].x) * ax + widen(x[z].y) * ay;
#pragma unroll
            for (int l = 0; l < 3; ++l)
                if (l < nell) s[z][l] += c[l] * p;
        }
    }
#pragma unroll
    for (int z = 0; z < NZ; ++z)
#pragma unroll
        for (int l = 0; l < 3; ++l) red[z * 3 + l][tid] = s[z][l];
    __syncthreads();
    const int lane = tid & 31;
    for (int v = tid >> 5; v < nz * 3; v += kXbThreads / 32) {
        const int z = v / 3, l = v - z * 3;
        if (l >= nell) continue;
        double t = red[v][lane];
#pragma unroll
        for (int w = 32; w < kXbThreads; w += 32) t += red[v][lane + w];
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) t += __shfl_down_sync(0xffffffffu, t, w);
        if (lane == 0) out(z)[l] = t;
    }
}

// out[z][l][b] = sum_seg partial[z][b][seg][l] (one warp per (b, l, z); fixed order).  With counts: the normalised
// P_ell, (4 l + 1) scale sum / counts[b], NaN for an empty bin.
static __global__ void __launch_bounds__(32) k_bin_sum(const double* __restrict__ partial, int nseg, int nell,
                                                       const double* __restrict__ counts, double scale,
                                                       double* __restrict__ out) {
    const int nb = gridDim.x, b = blockIdx.x, l = blockIdx.y, z = blockIdx.z;
    const double* p = partial + ((long)z * nb + b) * nseg * nell + l;
    double s = 0.0;
#pragma unroll 4
    for (int q = threadIdx.x; q < nseg; q += 32) s += p[(long)q * nell];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) s += __shfl_down_sync(0xffffffffu, s, w);
    if (threadIdx.x) return;
    if (counts) s = counts[b] > 0 ? (4 * l + 1) * scale * s / counts[b] : __longlong_as_double(0x7ff8000000000000LL);
    out[((long)z * nell + l) * nb + b] = s;
}

}  // namespace pb
