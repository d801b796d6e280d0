// Dispatch of the two-stage FFT passes over the groups of lengths (fft2_a.cu .. fft2_d.cu).
#include "fft.cuh"
#include "fft2.h"

namespace pb {
namespace f2 {

#define PB_F2_DECL(G)                                                                                                  \
    bool col_##G(int, int, const ColBatch&, int, int, int, cudaStream_t);                                              \
    bool xfilter_##G(int, const XInvBatch&, int, int, const float2*, AxisRange, AxisRange, AxisRange, float,           \
                     cudaStream_t);                                                                                    \
    bool xq_##G(int, const XqBatch&, int, int, const float2*, AxisRange, AxisRange, AxisRange, cudaStream_t);          \
    bool fwd_z_##G(int, const ZFwdBatch&, int, long, int, cudaStream_t);                                               \
    bool fwd_z_ylm_##G(int, const YlmBatch&, int, long, int, cudaStream_t);                                            \
    bool inv_z_##G(int, const ZInvBatch&, int, long, float, const float*, uint32_t*, cudaStream_t);                    \
    bool mask_z_##G(int, const ZMaskBatch&, int, long, const float*, int, cudaStream_t);
PB_F2_DECL(a)
PB_F2_DECL(b)
PB_F2_DECL(c)
PB_F2_DECL(d)

static_assert(kBatch == kMaxItems, "one batch size for every pass");

bool col(int n, int dir, const ColBatch& b, int nitem, int mc, int mo, cudaStream_t st) {
    return col_a(n, dir, b, nitem, mc, mo, st) || col_b(n, dir, b, nitem, mc, mo, st) ||
           col_c(n, dir, b, nitem, mc, mo, st) || col_d(n, dir, b, nitem, mc, mo, st);
}
bool xfilter(int n, const XInvBatch& b, int nitem, int mc, const float2* spec, AxisRange gx, AxisRange gy, AxisRange gz,
             float scale, cudaStream_t st) {
    return xfilter_a(n, b, nitem, mc, spec, gx, gy, gz, scale, st) || xfilter_b(n, b, nitem, mc, spec, gx, gy, gz, scale, st) ||
           xfilter_c(n, b, nitem, mc, spec, gx, gy, gz, scale, st) || xfilter_d(n, b, nitem, mc, spec, gx, gy, gz, scale, st);
}
bool xq(int n, const XqBatch& b, int nitem, int mc, const float2* pairs, AxisRange gx, AxisRange gy, AxisRange gz,
        cudaStream_t st) {
    return xq_a(n, b, nitem, mc, pairs, gx, gy, gz, st) || xq_b(n, b, nitem, mc, pairs, gx, gy, gz, st) ||
           xq_c(n, b, nitem, mc, pairs, gx, gy, gz, st) || xq_d(n, b, nitem, mc, pairs, gx, gy, gz, st);
}
bool fwd_z(int n, const ZFwdBatch& b, int nitem, long nl, int kout, cudaStream_t st) {
    return fwd_z_a(n, b, nitem, nl, kout, st) || fwd_z_b(n, b, nitem, nl, kout, st) || fwd_z_c(n, b, nitem, nl, kout, st) ||
           fwd_z_d(n, b, nitem, nl, kout, st);
}
bool fwd_z_ylm(int n, const YlmBatch& b, int nitem, long nl, int kout, cudaStream_t st) {
    return fwd_z_ylm_a(n, b, nitem, nl, kout, st) || fwd_z_ylm_b(n, b, nitem, nl, kout, st) ||
           fwd_z_ylm_c(n, b, nitem, nl, kout, st) || fwd_z_ylm_d(n, b, nitem, nl, kout, st);
}
bool inv_z(int n, const ZInvBatch& b, int nitem, long nl, float scale, const float* mulout, uint32_t* absmax,
           cudaStream_t st) {
    return inv_z_a(n, b, nitem, nl, scale, mulout, absmax, st) || inv_z_b(n, b, nitem, nl, scale, mulout, absmax, st) ||
           inv_z_c(n, b, nitem, nl, scale, mulout, absmax, st) || inv_z_d(n, b, nitem, nl, scale, mulout, absmax, st);
}
bool mask_z(int n, const ZMaskBatch& b, int nitem, long nl, const float* s, int kout, cudaStream_t st) {
    return mask_z_a(n, b, nitem, nl, s, kout, st) || mask_z_b(n, b, nitem, nl, s, kout, st) ||
           mask_z_c(n, b, nitem, nl, s, kout, st) || mask_z_d(n, b, nitem, nl, s, kout, st);
}

}  // namespace f2
}  // namespace pb
