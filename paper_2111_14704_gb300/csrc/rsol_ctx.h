// Context object behind the opaque rsol_ctx handle of rsol.h, and the
// argument-checking helpers shared by the C-ABI translation units.
#pragma once

#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>

#include <cuda_runtime.h>

#include "../../include/rsol.h"
#include "rsol_internal.h"

struct rsol_ctx {
    rsol_params p;
    int device;
    int sm_count;
    int bin;
    int nbx, nby, nbz;
    int64_t nbins;
    int key_bits;
    char err[512];
    int *d_status;            // device status word
    double *d_totals;         // 16 doubles + partials
    double *d_partials;
    // sort scratch (grown on demand)
    void *sort_mem;
    size_t sort_bytes;
    rsol::SortScratch sort;
    const uint32_t *sorted_cell; // identity of the set the last sort wrote
    int64_t sorted_n;
    // counting-sort scratch (allocated on first use)
    void *count_mem;
    size_t count_bytes;
    rsol::CountScratch count;
    // deterministic-mode fixed-point grid
    long long *fx;
    size_t fx_bytes;
    double fx_scale;
    // field-source scratch
    void *field_mem;
    size_t field_bytes;
    int64_t launches;         // kernels launched through this context
    // differentiable run (rsol_gradient): checkpoints, segment states, adjoints
    void *grad_mem;
    size_t grad_bytes;
    // sub-cycled push: per-packet levels, level-major order, level counts
    void *sub_mem;
    size_t sub_bytes;
};


namespace rsol_api {


constexpr int TOTALS_BLOCKS = 1024;

inline rsol_status fail(rsol_ctx *ctx, rsol_status st, const char *fmt, ...)
{
    if (ctx) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(ctx->err, sizeof(ctx->err), fmt, ap);
        va_end(ap);
    }
    return st;
}

inline rsol_status cuda_fail(rsol_ctx *ctx, cudaError_t e, const char *what)
{
    return fail(ctx, RSOL_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Expected us of a FP32 push of n packets on the context's 8^3 bins, from one GB300
// (p packets per bin): by the order-free kernel
//   max(12.5, 5 + 0.31e-3 n) TSC, max(5.2, 4 + 0.08e-3 n) CIC
// and by the binned one, per wave of CTAs,
//   10 + 0.07 p / slices TSC, 6.2 + 0.018 p / slices CIC in sparse bins (160, 384
//   packets a slice); 11 + 9.5e-3 p TSC, 10.5 + 3e-3 p CIC in tiles
// (binned / order-free, TSC: 16^3 nodes x 4096 packets 11.4 / 10.9, 40^3 x 16000 20.5 / 13.8,
// 48^3 x 55296 26.8 / 23.4, 48^3 x 110592 32.2 / 41.4, 64^3 x 65536 71.5 / 24.2, x 262144
// 63.3 / 80.5; CIC: 16^3 x 4096 6.2 / 4.9, 64^3 x 262144 47.2 / 24.8).
struct PushEstimate {
    double order_free, binned;
};
inline PushEstimate push_estimate(const rsol_ctx *ctx, int64_t n)
{
    const bool cic = ctx->p.shape == 1;
    const double p = double(n) / double(ctx->nbins);
    const int slices = rsol::bin_slices(ctx->sm_count, ctx->nbins);
    const double waves = double((ctx->nbins + ctx->sm_count - 1) / ctx->sm_count);
    const bool sparse = p <= double((cic ? 384 : 160) * slices);
    const double wave = sparse ? (cic ? 6.2 + 0.018 * p / slices : 10.0 + 0.07 * p / slices)
                               : (cic ? 10.5 + 3e-3 * p : 11.0 + 9.5e-3 * p);
    return {cic ? std::fmax(5.2, 4.0 + 0.08e-3 * n) : std::fmax(12.5, 5.0 + 0.31e-3 * n), waves * wave};
}

// Whether a sorted FP32 set is sparse enough, on bins enough to fill the GPU, for its sparse
// bins to go to a kernel of their own (push_sparse_bins_kernel; the bins' kernel then runs
// over the dense ones, an empty pass of 2 us and 1 us a wave where there are none): at
// most 640 packets per 8^3 nodes, so that few bins of an even set are dense.  Deterministic
// sums round alike only in one path.  us per push with one CTA a bin / split:
//   TSC 40^3 x 16000 20.5 / 14.8, 64^3 x 32768 57.4 / 21.0, x 81920 64.0 / 36.8, x 131072 52.8 / 54.9
//   CIC 40^3 x 32000 11.1 / 8.0, 64^3 x 65536 28.6 / 14.2, x 262144 47.2 / 28.6
inline bool split_faster(const rsol_ctx *ctx, int64_t n)
{
    if (ctx->p.precision != 32 || ctx->p.deterministic || ctx->bin != 8 ||
        rsol::bin_slices(ctx->sm_count, ctx->nbins) > 1)
        return false;
    const double nodes = double(ctx->p.nx) * ctx->p.ny * ctx->p.nz;
    const double waves = double((ctx->nbins + ctx->sm_count - 1) / ctx->sm_count);
    const PushEstimate e = push_estimate(ctx, n);
    return 512.0 * double(n) <= 640.0 * nodes && e.order_free + 2.0 + waves < e.binned;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline int elem_bytes(const rsol_ctx *ctx) { return ctx->p.precision == 32 ? 4 : 8; }

inline rsol_status check_particles(rsol_ctx *ctx, const rsol_particles *P, const char *name)
{
    if (!P)
        return fail(ctx, RSOL_ERR_INVALID_ARG, "%s: particle set is NULL", name);
    if (P->n < 0 || P->n > int64_t(0xFFFFFFFFll) - 1)
        return fail(ctx, RSOL_ERR_INVALID_ARG, "%s: n = %lld out of range", name, (long long)P->n);
    if (P->n == 0)
        return RSOL_OK;
    const void *ptrs[8] = {P->cell, P->off[0], P->off[1], P->off[2], P->u[0], P->u[1], P->u[2], P->w};
    for (int i = 0; i < 8; ++i) {
        if (!ptrs[i])
            return fail(ctx, RSOL_ERR_INVALID_ARG, "%s: particle array %d is NULL", name, i);
        if (!aligned16(ptrs[i]))
            return fail(ctx, RSOL_ERR_INVALID_ARG, "%s: particle array %d not 16-byte aligned", name, i);
    }
    return RSOL_OK;
}

inline int64_t n_nodes(const rsol_ctx *ctx) { return int64_t(ctx->p.nx) * ctx->p.ny * ctx->p.nz; }

} // namespace rsol_api

namespace rsol_api {

// Grow-only device buffer owned by the context.
inline rsol_status ensure_buffer(rsol_ctx *ctx, void **mem, size_t *bytes, size_t need, const char *what)
{
    if (*bytes >= need && *mem)
        return RSOL_OK;
    if (*mem)
        cudaFree(*mem);
    *mem = nullptr;
    *bytes = 0;
    if (cudaMalloc(mem, need) != cudaSuccess)
        return fail(ctx, RSOL_ERR_OOM, "%s: cudaMalloc(%zu) failed", what, need);
    *bytes = need;
    return RSOL_OK;
}

} // namespace rsol_api
