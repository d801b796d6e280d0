// Masked operator of the Fisher matrices (Sec. 3.3.2, eq. fish-from-Q; Sec. 4.3.4, eq. bk-fish-def): spectra on the box
// |n_i| <= m of the binned modes are taken to real space, multiplied by s = S^-1 P = w n and taken back to the box.
//
// Product grid.  With inputs and outputs on |n_i| <= m only the modes |n_i| <= 2m of s take part, and on a grid of L_i
// points an axis the products (|n_i| <= 3m) alias onto the box only if L_i <= 4m.  So with s low-passed to 2m the result on
// any grid of more than 4m points is that of the data grid, up to rounding: 144^3 instead of 256^3 (5.6 times fewer cells)
// for 16 bispectrum bins up to 33 k_F, 192^3 for 24 power spectrum bins up to 48 k_F.
//
// Memory.  The transforms of s run in the caller's scratch; what stays is s and one batch's intermediates.  Where these do not
// fit, the operator runs on the data grid with the maps n and w (mask_direct), which takes no memory of its own.
//
// Batches.  The FP32 passes run over a chunk of bins or triplets a launch (as many as keep the intermediates near the
// L2's size), the first one filters or combines on load, and the z passes around the product are one kernel (f2::mask_z),
// so the real maps are never stored.
// A draw on 256^3 (with the batched pair spectra and the parallel binned sums): bispectrum, 16 bins and 564 triplets, 110.7 ms
// before, 10.7 ms; power spectrum, 24 bins and 3 multipoles, 16.4 ms before, 2.84 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "fft.cuh"
#include "fft2.h"
#include "polybin_internal.h"

namespace pb {

struct MaskOp {
    InvGrid pg;
    Box3 keep{};                  // wave numbers of s that are kept
    void* tw[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    bool reduced = false;         // the product grid is smaller than the data grid
    bool fast = false;
    bool direct = false;          // no map of s: the data grid, multiplied by w and n
    void* smap = nullptr;         // s N / N' on the product grid
    // batches of `chunk` items: x passes [N0][By][Bz], y passes [N0][N1][Bz] before and after the product, boxes
    int chunk = 0;
    float2 *bx = nullptr, *by = nullptr, *bz = nullptr, *boxes = nullptr;
};

static MaskOp* op_of(const polybin_ctx* ctx) { return static_cast<MaskOp*>(ctx->maskop); }
const InvGrid& mask_grid(const polybin_ctx* ctx) { return op_of(ctx)->pg; }
const void* mask_map(const polybin_ctx* ctx) { return op_of(ctx)->smap; }
bool mask_direct(const polybin_ctx* ctx) { return op_of(ctx)->direct; }
bool mask_fast(const polybin_ctx* ctx) { return op_of(ctx)->fast && !op_of(ctx)->direct; }
int mask_chunk(const polybin_ctx* ctx) { return op_of(ctx)->chunk; }

// (their places are null afterwards: they may be allocated again)
static void free_maps(MaskOp* o) {
    void** ptrs[] = {&o->smap, (void**)&o->bx, (void**)&o->by, (void**)&o->bz, (void**)&o->boxes};
    for (void** p : ptrs) {
        if (*p) cudaFree(*p);
        *p = nullptr;
    }
}

bool mask_release(polybin_ctx* ctx) {
    MaskOp* o = op_of(ctx);
    if (!o || !o->smap) return false;
    free_maps(o);
    o->direct = true;
    return true;
}

void destroy_maskop(polybin_ctx* ctx) {
    MaskOp* o = op_of(ctx);
    if (!o) return;
    free_maps(o);
    for (void* p : o->tw)
        if (p) cudaFree(p);
    delete o;
    ctx->maskop = nullptr;
}

// out = n w (the product grid is the data grid).
template <typename T>
__global__ void k_weight(const float* __restrict__ n, const float* __restrict__ w, long count, T* __restrict__ out) {
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long)gridDim.x * blockDim.x)
        out[i] = T(w[i]) * T(n[i]);
}

static unsigned map_blocks(long n) { return (unsigned)std::min<long>((n + 255) / 256, 152L * 16); }

static int checked(polybin_ctx* ctx, const char* what) {
    ctx->launches++;
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? POLYBIN_OK : fail_cuda(ctx, e, what, __FILE__, __LINE__);
}

// The grid, and on first use (or after a call that found no room) the maps.
template <typename T>
static int mask_plan(polybin_ctx* ctx) {
    MaskOp* o = op_of(ctx);
    int rc;
    if (!o) {
        o = new (std::nothrow) MaskOp();
        if (!o) return fail(ctx, POLYBIN_ENOMEM, "masked operator: out of host memory");
        ctx->maskop = o;
        if ((rc = plan_product_grid(ctx, o->pg, o->keep, o->tw))) {
            destroy_maskop(ctx);
            return rc;
        }
        o->reduced = o->pg.ncell < ctx->ncell;
        o->fast = sizeof(T) == 4 && f2::has(o->pg.N[0]) && f2::has(o->pg.N[1]) && f2::has(o->pg.N[2]);
    }
    o->direct = !o->reduced && !o->fast;
    if (o->direct || o->smap) return POLYBIN_OK;
    const long By = ctx->gy.cnt, Bz = ctx->gz.cnt, nbox = (long)ctx->gx.cnt * By * Bz;
    const long P0 = o->pg.N[0], P1 = o->pg.N[1];
    PB_CUDA_OK(cudaMalloc(&o->smap, sizeof(T) * o->pg.ncell));
    if (o->fast) {
        // intermediates of a chunk near the L2's 129 MB
        const long item = (long)sizeof(float2) * (P0 * By * Bz + 2 * P0 * P1 * Bz + nbox);
        o->chunk = (int)std::min<long>(f2::kBatch, std::max<long>(1, (112L << 20) / item));
        PB_CUDA_OK(cudaMalloc(&o->bx, sizeof(float2) * o->chunk * P0 * By * Bz));
        PB_CUDA_OK(cudaMalloc(&o->by, sizeof(float2) * o->chunk * P0 * P1 * Bz));
        PB_CUDA_OK(cudaMalloc(&o->bz, sizeof(float2) * o->chunk * P0 * P1 * Bz));
        PB_CUDA_OK(cudaMalloc(&o->boxes, sizeof(float2) * o->chunk * nbox));
    }
    return POLYBIN_OK;
}

// s = w n low-passed to the product grid.  The steps lie in `scratch`, two regions that they use in turn.
template <typename T>
static int mask_lowpass(polybin_ctx* ctx, const float* n, const float* w, void* scratch, size_t bytes) {
    MaskOp* o = op_of(ctx);
    const long sx = o->keep.x.cnt, sy = o->keep.y.cnt, sz = o->keep.z.cnt, P0 = o->pg.N[0], P1 = o->pg.N[1];
    // t1 [N0][N1][sz], then box [sx][sy][sz], then v2 [P0][P1][sz]; t2 [N0][sy][sz], then v1 [P0][sy][sz]
    const size_t one = sizeof(C<T>) * std::max({(long)ctx->N[0] * ctx->N[1] * sz, sx * sy * sz, P0 * P1 * sz});
    const size_t two = sizeof(C<T>) * std::max(ctx->N[0] * sy * sz, P0 * sy * sz);
    void* own = nullptr;
    if (one + two > bytes) {
        PB_CUDA_OK(cudaMalloc(&own, one + two));
        scratch = own;
    }
    C<T>* const r1 = (C<T>*)scratch;
    C<T>* const r2 = (C<T>*)((char*)scratch + one);
    int rc = run_forward_box<T, float, float>(ctx, n, w, (const float*)nullptr, r1, r2, r1, ctx->fg, o->keep);
    // 1/N' instead of 1/N: the sums over the product grid's cells then have the data grid's normalisation
    if (!rc)
        rc = run_inverse_from<T>(ctx, r1, r2, r1, (T*)o->smap, (const T*)nullptr, o->pg, o->keep, 1.0 / (double)o->pg.ncell);
    if (own) cudaFree(own);                           // (waits for the steps)
    return rc;
}

template <typename T>
int mask_setup(polybin_ctx* ctx, const float* n, const float* w, void* scratch, size_t bytes) {
    int rc = mask_plan<T>(ctx);
    MaskOp* o = op_of(ctx);
    if (!rc && !o->direct) {
        if (o->reduced) {
            rc = mask_lowpass<T>(ctx, n, w, scratch, bytes);
        } else {
            k_weight<T><<<map_blocks(ctx->ncell), 256, 0, ctx->stream>>>(n, w, ctx->ncell, (T*)o->smap);
            rc = checked(ctx, "k_weight");
        }
    }
    if (rc == POLYBIN_ENOMEM && o) {
        cudaGetLastError();                           // no room: the data grid
        free_maps(o);
        o->direct = true;
        rc = POLYBIN_OK;
    }
    return rc;
}
template int mask_setup<float>(polybin_ctx*, const float*, const float*, void*, size_t);
template int mask_setup<double>(polybin_ctx*, const float*, const float*, void*, size_t);

// The passes after the first: item i (its box ry, rz) from bx to boxes.
static int finish(polybin_ctx* ctx, int cnt, const AxisRange* ry, const AxisRange* rz) {
    MaskOp* o = op_of(ctx);
    const long By = ctx->gy.cnt, Bz = ctx->gz.cnt, nbox = (long)ctx->gx.cnt * By * Bz;
    const int P0 = o->pg.N[0], P1 = o->pg.N[1], P2 = o->pg.N[2];
    const long nlines = (long)P0 * P1;
    cudaStream_t st = ctx->stream;
    int rc, maxz = 1;
    ColBatch b;
    f2::ZMaskBatch z;
    for (int i = 0; i < cnt; ++i) {
        ColItem& it = b.it[i];
        it.in = o->bx + (size_t)i * P0 * By * Bz;
        it.out = o->by + (size_t)i * nlines * Bz;
        it.in_os = (long)ry[i].cnt * rz[i].cnt; it.in_es = rz[i].cnt;
        it.out_os = (long)P1 * rz[i].cnt; it.out_es = rz[i].cnt;
        it.ncols = rz[i].cnt; it.nouter = P0; it.rng = ry[i];
        maxz = std::max(maxz, rz[i].cnt);
        z.it[i] = {o->by + (size_t)i * nlines * Bz, o->bz + (size_t)i * nlines * Bz, rz[i].cnt};
    }
    f2::col(P1, +1, b, cnt, maxz, P0, st);
    if ((rc = checked(ctx, "f2::col"))) return rc;
    f2::mask_z(P2, z, cnt, nlines, (const float*)o->smap, (int)Bz, st);
    if ((rc = checked(ctx, "f2::mask_z"))) return rc;
    for (int i = 0; i < cnt; ++i) {
        ColItem& it = b.it[i];
        it.in = o->bz + (size_t)i * nlines * Bz;
        it.out = o->bx + (size_t)i * P0 * By * Bz;
        it.in_os = (long)P1 * Bz; it.in_es = Bz; it.out_os = By * Bz; it.out_es = Bz;
        it.ncols = (int)Bz; it.nouter = P0; it.rng = ctx->gy;
    }
    f2::col(P1, -1, b, cnt, (int)Bz, P0, st);
    if ((rc = checked(ctx, "f2::col"))) return rc;
    for (int i = 0; i < cnt; ++i) {
        ColItem& it = b.it[i];
        it.in = o->bx + (size_t)i * P0 * By * Bz;
        it.out = o->boxes + (size_t)i * nbox;
        it.in_os = 0; it.in_es = By * Bz; it.out_os = 0; it.out_es = By * Bz;
        it.ncols = (int)(By * Bz); it.nouter = 1; it.rng = ctx->gx;
    }
    f2::col(P0, -1, b, cnt, (int)(By * Bz), 1, st);
    return checked(ctx, "f2::col");
}

int mask_shells(polybin_ctx* ctx, const float2* spec, int ell, int b0, int cnt, float2** boxes) {
    MaskOp* o = op_of(ctx);
    const long xs = (long)o->pg.N[0] * ctx->gy.cnt * ctx->gz.cnt;
    XInvBatch b;
    AxisRange ry[f2::kBatch], rz[f2::kBatch];
    int maxcols = 1, rc;
    for (int i = 0; i < cnt; ++i) {
        const BinBox& bb = o->pg.bbox[b0 + i];
        XInvItem& it = b.it[i];
        it.out = o->bx + (size_t)i * xs;
        it.rx = bb.rx; it.ry = bb.ry; it.rz = bb.rz;
        it.bin = b0 + i;
        it.slo = ctx->bin_slo[b0 + i];
        it.shi = ctx->bin_shi[b0 + i];
        it.ell = ell;
        it.m = kLegendreM;
        ry[i] = bb.ry;
        rz[i] = bb.rz;
        maxcols = std::max(maxcols, bb.ry.cnt * bb.rz.cnt);
    }
    f2::xfilter(o->pg.N[0], b, cnt, maxcols, spec, ctx->gx, ctx->gy, ctx->gz, (float)(1.0 / (double)ctx->ncell), ctx->stream);
    if ((rc = checked(ctx, "f2::xfilter"))) return rc;
    *boxes = o->boxes;
    return finish(ctx, cnt, ry, rz);
}

int mask_triplets(polybin_ctx* ctx, const float2* pairs, int t0, int cnt, float2** boxes) {
    MaskOp* o = op_of(ctx);
    const long xs = (long)o->pg.N[0] * ctx->gy.cnt * ctx->gz.cnt;
    const long nbox = (long)ctx->gx.cnt * ctx->gy.cnt * ctx->gz.cnt;
    const int nb = ctx->nb;
    f2::XqBatch q;
    AxisRange ry[f2::kBatch], rz[f2::kBatch];
    int maxcols = 1, rc;
    for (int i = 0; i < cnt; ++i) {
        const int a = ctx->trip[3 * (t0 + i)], b = ctx->trip[3 * (t0 + i) + 1], c = ctx->trip[3 * (t0 + i) + 2];
        const double dl = (a == b && b == c) ? 6.0 : ((a == b || b == c) ? 2.0 : 1.0);
        const BinBox& bb = o->pg.bbox[c];             // c is the triplet's largest bin
        f2::XqItem& it = q.it[i];
        it.out = o->bx + (size_t)i * xs;
        it.rx = bb.rx; it.ry = bb.ry; it.rz = bb.rz;
        it.pab = (long)pair_index(nb, a, b) * nbox;
        it.pbc = (long)pair_index(nb, b, c) * nbox;
        it.pac = (long)pair_index(nb, a, c) * nbox;
        it.alo = ctx->bin_slo[a]; it.ahi = ctx->bin_shi[a];
        it.blo = ctx->bin_slo[b]; it.bhi = ctx->bin_shi[b];
        it.clo = ctx->bin_slo[c]; it.chi = ctx->bin_shi[c];
        it.fac = (float)(2.0 / dl * ctx->cg_ratio / (double)ctx->ncell);
        ry[i] = bb.ry;
        rz[i] = bb.rz;
        maxcols = std::max(maxcols, bb.ry.cnt * bb.rz.cnt);
    }
    f2::xq(o->pg.N[0], q, cnt, maxcols, pairs, ctx->gx, ctx->gy, ctx->gz, ctx->stream);
    if ((rc = checked(ctx, "f2::xq"))) return rc;
    *boxes = o->boxes;
    return finish(ctx, cnt, ry, rz);
}

}  // namespace pb
