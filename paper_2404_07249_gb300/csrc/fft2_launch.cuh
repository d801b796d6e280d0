// Launchers of the two-stage FFT passes for one group of lengths.  Each group is a translation unit of its own
// (fft2_a.cu .. fft2_d.cu), compiled in parallel.
#pragma once
#include "fft2.cuh"

namespace pb {
namespace f2 {

template <typename K> static void allow_smem(K* k, int bytes) {
    if (bytes > 48 * 1024) cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <int N> struct Run {
    using E = Geo<N>;
    static void col(int dir, const ColBatch& b, int nitem, int max_cols, int max_outer, cudaStream_t st) {
        const dim3 grid((max_cols + E::TC - 1) / E::TC, max_outer, nitem);
        if (dir > 0) {
            allow_smem(k_col<1, N>, E::kColSmem);
            k_col<1, N><<<grid, E::kColThreads, E::kColSmem, st>>>(b);
        } else {
            allow_smem(k_col<-1, N>, E::kColSmem);
            k_col<-1, N><<<grid, E::kColThreads, E::kColSmem, st>>>(b);
        }
    }
    static void xfilter(const XInvBatch& b, int nitem, int max_cols, const float2* spec, AxisRange gx, AxisRange gy,
                        AxisRange gz, float scale, cudaStream_t st) {
        allow_smem(k_xfilter<N>, E::kColSmem);
        k_xfilter<N><<<dim3((max_cols + E::TC - 1) / E::TC, nitem), E::kColThreads, E::kColSmem, st>>>(b, spec, gx, gy, gz,
                                                                                                     scale);
    }
    static void xq(const XqBatch& b, int nitem, int max_cols, const float2* pairs, AxisRange gx, AxisRange gy, AxisRange gz,
                   cudaStream_t st) {
        allow_smem(k_xq<N>, E::kColSmem);
        k_xq<N><<<dim3((max_cols + E::TC - 1) / E::TC, nitem), E::kColThreads, E::kColSmem, st>>>(b, pairs, gx, gy, gz);
    }
    static dim3 line_grid(long nlines, int nitem) {
        return dim3((unsigned)(((nlines + 1) / 2 + E::G - 1) / E::G), nitem);
    }
    static void fwd_z(const ZFwdBatch& b, int nitem, long nlines, int kout, cudaStream_t st) {
        k_fwd_z<N><<<line_grid(nlines, nitem), E::kLineThreads, E::kLineSmem, st>>>(b, nlines, kout);
    }
    static void fwd_z_ylm(const YlmBatch& b, int nitem, long nlines, int kout, cudaStream_t st) {
        // one dimension: 1024 x 1024 lines of 512 points are 65536 line blocks, more than a grid's y takes
        k_fwd_z_ylm<N><<<line_grid(nlines, 1).x * nitem, E::kLineThreads, E::kLineSmem, st>>>(b, nitem, nlines, kout);
    }
    static void inv_z(const ZInvBatch& b, int nitem, long nlines, float scale, const float* mulout, uint32_t* absmax,
                      cudaStream_t st) {
        k_inv_z<N><<<line_grid(nlines, nitem), E::kLineThreads, E::kLineSmem, st>>>(b, nlines, scale, mulout, absmax);
    }
    static void mask_z(const ZMaskBatch& b, int nitem, long nlines, const float* s, int kout, cudaStream_t st) {
        k_mask_z<N><<<line_grid(nlines, nitem), E::kLineThreads, E::kLineSmem, st>>>(b, nlines, s, kout);
    }
    static_assert(E::kLineSmem <= 48 * 1024, "line passes use at most 48 KB");
};

}  // namespace f2
}  // namespace pb

// Defines the group's launchers NAME##_##G over the lengths of LENGTHS(X).
#define PB_F2_CASE_(N, CALL) case N: Run<N>::CALL; return true;
#define PB_F2_GROUP(G, LENGTHS)                                                                                        \
    namespace pb {                                                                                                     \
    namespace f2 {                                                                                                     \
    bool col_##G(int n, int dir, const ColBatch& b, int nitem, int mc, int mo, cudaStream_t st) {                      \
        switch (n) { LENGTHS(col(dir, b, nitem, mc, mo, st)) }                                                         \
        return false;                                                                                                  \
    }                                                                                                                  \
    bool xfilter_##G(int n, const XInvBatch& b, int nitem, int mc, const float2* spec, AxisRange gx, AxisRange gy,     \
                     AxisRange gz, float scale, cudaStream_t st) {                                                     \
        switch (n) { LENGTHS(xfilter(b, nitem, mc, spec, gx, gy, gz, scale, st)) }                                     \
        return false;                                                                                                  \
    }                                                                                                                  \
    bool xq_##G(int n, const XqBatch& b, int nitem, int mc, const float2* pairs, AxisRange gx, AxisRange gy,           \
                AxisRange gz, cudaStream_t st) {                                                                       \
        switch (n) { LENGTHS(xq(b, nitem, mc, pairs, gx, gy, gz, st)) }                                                \
        return false;                                                                                                  \
    }                                                                                                                  \
    bool fwd_z_##G(int n, const ZFwdBatch& b, int nitem, long nl, int kout, cudaStream_t st) {                         \
        switch (n) { LENGTHS(fwd_z(b, nitem, nl, kout, st)) }                                                          \
        return false;                                                                                                  \
    }                                                                                                                  \
    bool fwd_z_ylm_##G(int n, const YlmBatch& b, int nitem, long nl, int kout, cudaStream_t st) {                      \
        switch (n) { LENGTHS(fwd_z_ylm(b, nitem, nl, kout, st)) }                                                      \
        return false;                                                                                                  \
    }                                                                                                                  \
    bool inv_z_##G(int n, const ZInvBatch& b, int nitem, long nl, float scale, const float* mulout, uint32_t* absmax,  \
                   cudaStream_t st) {                                                                                  \
        switch (n) { LENGTHS(inv_z(b, nitem, nl, scale, mulout, absmax, st)) }                                         \
        return false;                                                                                                  \
    }                                                                                                                  \
    bool mask_z_##G(int n, const ZMaskBatch& b, int nitem, long nl, const float* s, int kout, cudaStream_t st) {       \
        switch (n) { LENGTHS(mask_z(b, nitem, nl, s, kout, st)) }                                                      \
        return false;                                                                                                  \
    }                                                                                                                  \
    }                                                                                                                  \
    }
