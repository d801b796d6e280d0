// Host interface of the two-stage FFT passes (fft2.cuh): the lengths, the batch items and the launchers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace pb {
struct ColBatch;
struct XInvBatch;
struct ZInvBatch;
namespace f2 {

// Stage-1 points P of a length N = P x Q (0: not a two-stage length).
__host__ __device__ constexpr int stage_p(int n) {
    switch (n) {
        case 48: return 6;
        case 54: return 6;
        case 60: return 6;
        case 64: return 8;
        case 72: return 8;
        case 80: return 8;
        case 90: return 9;
        case 96: return 8;
        case 100: return 10;
        case 108: return 9;
        case 120: return 10;
        case 128: return 8;
        case 144: return 12;
        case 150: return 10;
        case 160: return 10;
        case 180: return 12;
        case 192: return 12;
        case 200: return 10;
        case 216: return 12;
        case 240: return 15;
        case 256: return 16;
        case 270: return 15;
        case 288: return 16;
        case 300: return 15;
        case 320: return 16;
        case 324: return 18;
        case 360: return 18;
        case 384: return 16;
        case 400: return 20;
        case 432: return 18;
        case 480: return 20;
        case 512: return 16;
        default: return 0;
    }
}
inline bool has(int n) { return stage_p(n) != 0; }

constexpr int kBatch = 64;   // items of one launch (kMaxItems)

struct ZFwdItem {
    const float *in, *m1, *m2;   // product on load (m1, m2 may be null)
    const float *sub, *sub_m;    // subtracted product (then m2 is not used)
    float2* out;                 // [nlines][kout]
};
struct ZFwdBatch {
    ZFwdItem it[kBatch];
};
// Forward z-pass of harmonic-weighted fields: field x (w) x Ybar_l,m and Ybar_l,-m of each cell's direction from the
// observer, m = am >= 0, l even.
struct YlmItem {
    float2 *re, *im;             // [nlines][kout] of m = am and of m = -am (either may be null)
    // Ybar_lm = (Re or Im of (x + i y)^am) z^(am odd) (d4 z^4 + d2 z^2 + d0) for the unit vector (x, y, z)
    int am;
    float d4, d2, d0;
};
struct YlmBatch {
    YlmItem it[16];
    const float *in, *w;         // w may be null
    int n1;                      // lines: (i, j) = (l / n1, l % n1)
    // cell centre from the observer (i - cell - frac) h, in units of the box side: exact to FP32's last bit near the observer
    float h[3], frac[3];
    int cell[3];
};
struct ZMaskItem {
    const float2* in;            // [nlines][kin]
    float2* out;                 // [nlines][kout]
    int kin;
};
struct ZMaskBatch {
    ZMaskItem it[kBatch];
};
// Q-derivative spectrum of a triplet (a, b, c) from pair spectra P (box layout): fac [Theta_c P_ab + Theta_a P_bc +
// Theta_b P_ac], each Theta the bin's range of integer |n|^2.
struct XqItem {
    float2* out;                 // [N][ry.cnt * rz.cnt]
    AxisRange rx, ry, rz;        // box of the modes of the three bins
    long pab, pbc, pac;          // offsets of the pair spectra
    int alo, ahi, blo, bhi, clo, chi;
    float fac;
};
struct XqBatch {
    XqItem it[kBatch];
};

// Launchers over nitem items; false when n is not a two-stage length (nothing is launched).
bool col(int n, int dir, const ColBatch& b, int nitem, int max_cols, int max_outer, cudaStream_t st);
bool xfilter(int n, const XInvBatch& b, int nitem, int max_cols, const float2* spec, AxisRange gx, AxisRange gy,
             AxisRange gz, float scale, cudaStream_t st);
bool fwd_z(int n, const ZFwdBatch& b, int nitem, long nlines, int kout, cudaStream_t st);
bool fwd_z_ylm(int n, const YlmBatch& b, int nitem, long nlines, int kout, cudaStream_t st);
bool inv_z(int n, const ZInvBatch& b, int nitem, long nlines, float scale, const float* mulout, uint32_t* absmax,
           cudaStream_t st);
bool mask_z(int n, const ZMaskBatch& b, int nitem, long nlines, const float* s, int kout, cudaStream_t st);

// First inverse pass of the Q-derivative spectra of nitem triplets.
bool xq(int n, const XqBatch& b, int nitem, int max_cols, const float2* pairs, AxisRange gx, AxisRange gy, AxisRange gz,
        cudaStream_t st);

}  // namespace f2
}  // namespace pb
