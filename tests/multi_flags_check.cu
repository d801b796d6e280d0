// A wait that gives up in any field of a batched call is reported.  This program defines run_bk_normalise, which the library
// calls after the contraction of every field: the one here (taking precedence over the library's, which it calls) also
// sets the context's error flag on the stream, as a wait of that field's contraction would, for one chosen field.
#include <cuda_runtime.h>
#include <dlfcn.h>

#include <cstdio>
#include <vector>

#include "polybin.h"
#include "polybin_internal.h"

static int g_next = 0, g_flagged = -1;

namespace pb {
int run_bk_normalise(polybin_ctx* ctx, const double* d_S, double* d_B, double fac) {
    using Fn = int (*)(polybin_ctx*, const double*, double*, double);
    static Fn real = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "_ZN2pb16run_bk_normaliseEP11polybin_ctxPKdPdd"));
    if (!real) return POLYBIN_ECUDA;
    if (g_next++ == g_flagged && cudaMemsetAsync(ctx->d_err + kErrPipeline, 1, sizeof(int), ctx->stream) != cudaSuccess)
        return POLYBIN_ECUDA;
    return real(ctx, d_S, d_B, fac);
}
}  // namespace pb

int main() {
    const int grid[3] = {32, 32, 32}, nf = 5, n = 32 * 32 * 32;
    const double box[3] = {800.0, 800.0, 800.0};
    double edges[5];
    for (int i = 0; i < 5; ++i) edges[i] = 2.0 * M_PI / 800.0 * (1.0 + 2.0 * i);
    polybin_ctx* ctx[2] = {nullptr, nullptr};
    for (polybin_ctx*& c : ctx)
        if (polybin_init(&c, grid, box, edges, 4, 0, POLYBIN_SPLIT_TF32X3, nullptr)) return std::printf("init failed\n"), 1;
    // contexts in turn (a branch of the graph each); fields at new places a call, so that each makes its own graph
    polybin_ctx* ctxs[nf];
    for (int i = 0; i < nf; ++i) ctxs[i] = ctx[i % 2];
    float* mem = nullptr;
    if (cudaMalloc(&mem, sizeof(float) * n * (nf + 8)) != cudaSuccess) return 1;
    std::vector<float> h((size_t)n * (nf + 8));
    for (size_t i = 0; i < h.size(); ++i) h[i] = (float)((i * 2654435761u) % 1000) / 1000.f - 0.5f;
    cudaMemcpy(mem, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice);
    std::vector<double> out((size_t)nf * 4096);
    int bad = 0;
    for (int flagged = -1; flagged <= nf; ++flagged) {
        const float* fields[nf];
        double* outs[nf];
        for (int i = 0; i < nf; ++i) {
            fields[i] = mem + (size_t)n * (i + flagged + 1);
            outs[i] = out.data() + (size_t)i * 4096;
        }
        g_next = 0;
        g_flagged = flagged;
        for (int rep = 0; rep < 2; ++rep) {           // as captured, and replayed
            const int rc = polybin_bk_ideal_multi(ctxs, fields, nf, outs), want = flagged >= 0 && flagged < nf ? POLYBIN_ETIMEOUT : POLYBIN_OK;
            if (rc != want) {
                ++bad;
                std::printf("flag in field %d of %d, call %d: code %d, expected %d\n", flagged, nf, rep, rc, want);
            }
        }
        if (g_next != nf) { ++bad; std::printf("%d fields seen, expected %d\n", g_next, nf); }
    }
    for (polybin_ctx* c : ctx) polybin_destroy(c);
    std::printf("%d failures\n", bad);
    return bad ? 1 : 0;
}
