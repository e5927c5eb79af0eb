// Binned push kernel: one CTA per sort bin of B^3 anchor nodes.
//
// The packets of a bin are contiguous after rsol_sort (keyed on the anchor
// node of their stencil: the cell for CIC, the nearest node for TSC), so the
// CTA stages the E, B tile of its bin plus a two-node halo in shared memory,
// and deposits into a shared-memory tile that is added to the global grid
// once at the end.  FP32 (octet_cta): packets are pushed in memory order, their
// densities staged and deposited by stencil origin.  FP64 (binned_cta), per warp
// and batch of 32 packets:
//   phase 1, one packet per lane: weights, gather from the tile, Boris,
//            feedback densities, drift; the packet's stencil weights and its
//            eight densities are staged per warp.
//   phase 2, one stencil offset per lane (TSC: 27 lanes x 8 quantities;
//            CIC: 8 offsets x 4 pairs of quantities): walk the runs of equal
//            stencil origin along the lanes (equal anchors are adjacent after
//            the sort), accumulate W * Q in registers and add the run's sum
//            to the tile once per run.
// Packets whose stencil leaves the tile (they drifted more than a node since
// the sort) take the order-free path: gather from global memory and deposit
// with global atomics.  Results equal the order-free kernel's up to the order
// of floating-point additions (bitwise run to run in deterministic mode).
#pragma once

#include <type_traits>

#include "octets.cuh"
#include "push.cuh"
#include "tma.cuh"

namespace rsol {

// Bins with at most this many packets skip the shared-memory tiles: staging
// and flushing a (B + 4)^3 tile then costs more than the packets' own global
// gathers and atomics.  Measured with 8^3 bins (sort and four steps): the batch of 512
// boxes 24.3 ms at 768, 23.6 at 512, 23.8 at 384, 24.9 at 256; a 61 x 45 x 97 grid
// with 1 M packets, CIC, 0.478 ms at 768 and 0.451 at 512, 384 and 256.
// Deterministic FP32: 64-bit global atomics cost more, the crossover lies lower.
template <typename T, int B, bool DET>
__host__ __device__ constexpr uint32_t sparse_bin_limit()
{
    return sizeof(T) == 4 && DET ? 160u : B == 8 ? 512u : 256u;
}

// The same for the state moments and the adjoint step.
template <int B>
__host__ __device__ constexpr uint32_t sparse_sum_limit()
{
    return B == 8 ? 768u : 256u;
}

// The same for one box's CTAs (octet_cta), where a sparse bin holds a whole CTA
// through its packets' global atomics: 512 TSC packets of an 8^3 bin take 37 us
// that way and 16 us through the tiles (CIC 13 and 12).  A batch's sparse bins share
// SMs, one warp each, so its limit lies higher.  Deterministic sums round per
// packet in one path and per run in the other: one limit, so that a batch equals
// its boxes bit for bit.
template <int SHAPE, int B, bool DET>
__host__ __device__ constexpr uint32_t sparse_cta_limit()
{
    return DET ? sparse_bin_limit<float, B, DET>() : B == 8 ? (SHAPE == 1 ? 384u : 160u) : 128u;
}

// Where a box has fewer bins than half the SMs, a sparse bin is dealt to `slices` CTAs
// (bin_slices), which raises the crossover to `slices` times the limit: a CTA then waits
// for 1 / slices of the bin's atomics (TSC, 512 packets a bin: 8 bins 16.6 -> 11.4 us per
// push, 27 bins 16.8 -> 15.6).  At most 768 packets of an 8^3 bin (256 of a 4^3 one), 1.5
// (4) a node on average, go through global FP32 sums, however idle the GPU is: those
// round once per packet and node, a tile's integers once per run of packets.
template <int SHAPE, int B, bool DET>
__host__ __device__ constexpr uint32_t sliced_cta_limit(uint32_t slices)
{
    const uint32_t limit = sparse_cta_limit<SHAPE, B, DET>(), most = B == 8 ? kGlobalBinMost : 256u;
    return DET ? limit : limit * slices < most ? limit * slices : most;
}

struct BinGeom {
    const uint32_t *bin_start;
    int nbx, nby, nbz;
    uint32_t skip = 0;  // push: bins of at most this many packets are another kernel's
};

template <typename T, int SHAPE, int B, int NW, bool DET>
struct BinnedCfg {
    static constexpr int NP = SHAPE == 1 ? 2 : 3;   // stencil nodes per axis
    static constexpr int NS = NP * NP * NP;         // stencil nodes
    static constexpr int TE = B + 4;                // tile edge in nodes, origin at bin origin - 2
    static constexpr int RS = TE;                   // row stride
    static constexpr int PS = TE * RS;              // plane stride
    static constexpr int TN = TE * PS;              // tile slots
    // deposit-tile element: 64-bit fixed point (deterministic mode), or T
    using Acc = typename std::conditional<DET, long long, T>::type;
    static constexpr size_t fields_bytes = size_t(TN) * 8 * sizeof(T);  // [slot][8]: E, B, 2 unused
    static constexpr size_t dep_bytes = size_t(TN) * 8 * sizeof(Acc);   // [q][slot]
    // per warp: stencil weights W[32][WS] and densities QO[32][12]
    static constexpr int WS = NS == 27 ? 28 : NS;   // weight rows padded to 16-byte stores
    static constexpr int QO = 12;                   // rows apart: fewer conflicts of the 16-byte stores
    static constexpr size_t stage_words = 32 * (WS + QO);
    static constexpr size_t stage_bytes = size_t(NW) * stage_words * sizeof(T);
    static constexpr size_t smem_bytes = fields_bytes + dep_bytes + stage_bytes;
};

__device__ __forceinline__ int wrap_mod(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// v periodic in [0, n) for v in [-n, 2n)
__device__ __forceinline__ int wrap_once(int v, int n)
{
    v += v < 0 ? n : 0;
    return v - (v >= n ? n : 0);
}

// First stencil node relative to the cell (axis_weights without the weights).
template <int SHAPE, typename T>
__device__ __forceinline__ int first_node(T f)
{
    return SHAPE == 1 || f >= T(0.5) ? 0 : -1;
}

// Anchor node and stencil data of one axis: returns the anchor (periodic) and
// the first stencil node offset relative to the anchor; w[] are the weights of
// the stencil nodes first, first+1, first+2 (relative to the anchor).
template <int SHAPE, typename T>
__device__ __forceinline__ int anchor_axis(int i, T f, int n, T w[3], int &first_rel)
{
    const int first = axis_weights<SHAPE>(f, w);  // relative to the cell
    if (SHAPE == 1) {
        first_rel = 0;
        return i;
    }
    // TSC: anchor = cell + (first + 1); stencil starts one node below it
    first_rel = -1;
    int j = i + first + 1;
    j -= (j >= n) ? n : 0;
    return j;
}

// Tile-local stencil-origin slot of a packet (cell c, offsets f0..f2) for the
// tile whose first node is (ox, oy, oz): lz * PS + ly * RS + lx, or TN when the
// packet is off the grid or its stencil leaves the tile.
template <int SHAPE, int TE, int RS, int PS, int TN, typename T>
__device__ __forceinline__ int origin_slot(uint32_t c, T f0, T f1, T f2, int ox, int oy, int oz,
                                           int nx, int ny, int nz)
{
    constexpr int NP = SHAPE == 1 ? 2 : 3;
    const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
    if (ix >= nx || iy >= ny || iz >= nz)
        return TN;
    T w3[3];
    int rx, ry, rz;
    const int jx = anchor_axis<SHAPE>(ix, f0, nx, w3, rx);
    const int jy = anchor_axis<SHAPE>(iy, f1, ny, w3, ry);
    const int jz = anchor_axis<SHAPE>(iz, f2, nz, w3, rz);
    const int lx = wrap_once(jx + rx - ox, nx), ly = wrap_once(jy + ry - oy, ny),
              lz = wrap_once(jz + rz - oz, nz);
    return lx + NP <= TE && ly + NP <= TE && lz + NP <= TE ? lz * PS + ly * RS + lx : TN;
}

__device__ __forceinline__ void lds_node(const float *p, float F[6])
{
    const float4 a = *reinterpret_cast<const float4 *>(p);
    const float2 b = *reinterpret_cast<const float2 *>(p + 4);
    F[0] = a.x; F[1] = a.y; F[2] = a.z; F[3] = a.w; F[4] = b.x; F[5] = b.y;
}
__device__ __forceinline__ void lds_node(const double *p, double F[6])
{
    const double2 a = *reinterpret_cast<const double2 *>(p);
    const double2 b = *reinterpret_cast<const double2 *>(p + 2);
    const double2 c = *reinterpret_cast<const double2 *>(p + 4);
    F[0] = a.x; F[1] = a.y; F[2] = b.x; F[3] = b.y; F[4] = c.x; F[5] = c.y;
}

// E, B of one node into a tile slot of 8 elements (16-byte stores)
__device__ __forceinline__ void sts_node(float *p, const float F[6])
{
    reinterpret_cast<float4 *>(p)[0] = make_float4(F[0], F[1], F[2], F[3]);
    reinterpret_cast<float2 *>(p)[2] = make_float2(F[4], F[5]);
}
__device__ __forceinline__ void sts_node(double *p, const double F[6])
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(F[0], F[1]);
    reinterpret_cast<double2 *>(p)[1] = make_double2(F[2], F[3]);
    reinterpret_cast<double2 *>(p)[2] = make_double2(F[4], F[5]);
}

__device__ __forceinline__ void store_q8(double *p, const double Q[8])
{
#pragma unroll
    for (int q = 0; q < 8; q += 2)
        reinterpret_cast<double2 *>(p)[q / 2] = make_double2(Q[q], Q[q + 1]);
}
// one packet's stencil weights into its padded staging row (16-byte stores)
template <int WS, int NS>
__device__ __forceinline__ void store_wrow(double *p, const double (&W)[NS])
{
#pragma unroll
    for (int k = 0; k < WS; k += 2)
        reinterpret_cast<double2 *>(p)[k / 2] = make_double2(W[k], k + 1 < NS ? W[k + 1] : 0.0);
}

// the N densities of a phase-2 lane role, starting at p (N = 8: all; N = 2: a pair)
template <int N>
__device__ __forceinline__ void load_qpart(const double *p, double Q[N])
{
#pragma unroll
    for (int q = 0; q < N; q += 2) {
        const double2 v = reinterpret_cast<const double2 *>(p)[q / 2];
        Q[q] = v.x;
        Q[q + 1] = v.y;
    }
}

// L2 prefetch of elements [lo, hi) of p: one 128-byte line per thread and pass;
// every address issued is that of an element of the range.
template <typename E>
__device__ __forceinline__ void prefetch_l2(const E *p, uint32_t lo, uint32_t hi)
{
    if (lo >= hi)
        return;
    const uintptr_t s = reinterpret_cast<uintptr_t>(p + lo), e = reinterpret_cast<uintptr_t>(p + hi);
    for (uintptr_t l = (s & ~uintptr_t(127)) + uintptr_t(threadIdx.x) * 128; l < e;
         l += uintptr_t(blockDim.x) * 128) {
        const uintptr_t addr = l < s ? s : l;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(addr));
    }
}

// Exclusive prefix sum of the origin histogram hist[0..TN) of a CTA of NW warps
// into cursor[] (each origin's first position in origin order); *s_out = the
// packets counted, i.e. the first position after them.  Ends synchronised.
template <int NW, int TN>
__device__ __forceinline__ void origin_cursors(const int *hist, int *cursor, int *s_out)
{
    __shared__ int s_wsum[NW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int CH = (TN + NW * 32 - 1) / (NW * 32);
    const int t0 = int(threadIdx.x) * CH;
    int vals[CH];
    int tsum = 0;
#pragma unroll
    for (int u = 0; u < CH; ++u) {
        vals[u] = t0 + u < TN ? hist[t0 + u] : 0;
        tsum += vals[u];
    }
    int incl = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        incl += lane >= o ? v : 0;
    }
    if (lane == 31)
        s_wsum[warp] = incl;
    __syncthreads();
    int wbase = 0;
    for (int w = 0; w < warp; ++w)
        wbase += s_wsum[w];
    if (threadIdx.x == blockDim.x - 1)
        *s_out = wbase + incl;
    int run = wbase + incl - tsum;
#pragma unroll
    for (int u = 0; u < CH; ++u) {
        if (t0 + u < TN)
            cursor[t0 + u] = run;
        run += vals[u];
    }
    __syncthreads();
}

// Largest total weight any node of a tile can receive from the packets counted
// in hist(slot) (packets per tile-local stencil origin, slot z PS + y RS + x): the
// sum over the stencil origins around the node of (packets at the origin) x
// (largest axis weights for that offset: CIC 1, 1; TSC 1/2, 3/4, 1/2 per
// axis).  The weights are per-axis products, so the sum is three 3-tap passes
// along x, y and z, one tile row per thread and pass; exact in float (the terms
// are small integers times products of 1/2 and 3/4).  One pass per call, 0 to 2, all
// threads, with a barrier between the calls; scratch holds 2 TE^3 floats.  Pass 2 raises
// gmax to this thread's largest node value (reduce over the CTA).
template <int SHAPE, int TE, int RS, int PS, typename Hist>
__device__ __forceinline__ void weight_bound_pass(int pass, Hist hist, float *scratch, float &gmax)
{
    constexpr int NP = SHAPE == 1 ? 2 : 3;
    constexpr int TT = TE * TE * TE;
    float *g1 = scratch, *g2 = scratch + TT;  // [z][y][x], TE each
    auto tap = [](int c) { return SHAPE == 1 ? 1.f : (c == 1 ? 0.75f : 0.5f); };
    // the rows go to the last threads (the first warps may have other work)
    for (int r = int(blockDim.x) - 1 - int(threadIdx.x); r < TE * TE; r += blockDim.x) {
        const int u = r % TE, z = r / TE;  // pass 0: row (z, y = u); 1: (z, x = u); 2: (y = z, x = u)
        float h[TE];
#pragma unroll
        for (int i = 0; i < TE; ++i)
            h[i] = pass == 0 ? float(hist(z * PS + u * RS + i)) : pass == 1 ? g1[(z * TE + i) * TE + u]
                                                                          : g2[(i * TE + z) * TE + u];
#pragma unroll
        for (int i = 0; i < TE; ++i) {
            float v = 0.f;
#pragma unroll
            for (int c = 0; c < NP; ++c)
                v += i >= c ? tap(c) * h[i - c] : 0.f;
            if (pass == 0)
                g1[(z * TE + u) * TE + i] = v;
            else if (pass == 1)
                g2[(z * TE + i) * TE + u] = v;
            else
                gmax = fmaxf(gmax, v);
        }
    }
}
// Few packets: staging and flushing the tiles would cost more than the
// packets' own global-memory gathers and atomics.
template <typename T, int SHAPE, bool DET>
__device__ __forceinline__ void sparse_cta(const PushArgs<T> &a, uint32_t lo, uint32_t hi)
{
    int sflag = 0;
    auto gather_global = [&](int64_t node, T F[6]) { load_node(a.fields + node * 8, F); };
    auto deposit_global = [&](int64_t node, T W, const T Q[8]) {
        if constexpr (DET)
            red_node_fixed(a.fx + node * 8, W, Q, a.fx_scale);
        else
            red_node(a.fb + node * 8, W, Q);
    };
    for (uint32_t j = lo + threadIdx.x; j < hi; j += blockDim.x)
        push_one<T, SHAPE, true>(a, int64_t(j), gather_global, deposit_global, &sflag);
    if (sflag)
        atomicOr(a.status, sflag);
}

// Grid offsets of the rows along each axis (periodic) of the tile of TE^3 nodes
// from node (ox, oy, oz): the grid node of tile point (lx, ly, lz) is
// axis[lx] + axis[TE + ly] + axis[2 TE + lz].
template <int TE>
__device__ __forceinline__ void tile_axes(int *axis, int ox, int oy, int oz, int nx, int ny, int nz)
{
    if (threadIdx.x < 3 * TE) {
        const int ax = threadIdx.x / TE, l = threadIdx.x % TE;
        const int o = ax == 0 ? ox : (ax == 1 ? oy : oz);
        const int n = ax == 0 ? nx : (ax == 1 ? ny : nz);
        const int stride = ax == 0 ? 1 : (ax == 1 ? nx : nx * ny);
        axis[threadIdx.x] = wrap_mod(o + l, n) * stride;
    }
}

// The work of one CTA on one bin (FP64): packets [lo, hi) of the bin whose anchors
// were in bin (bx, by, bz) of the box described by a at the last sort.
template <int SHAPE, int B, int NW, bool DET>
__device__ __forceinline__ void binned_cta(const PushArgs<double> &a, uint32_t lo, uint32_t hi,
                                           int bx, int by, int bz)
{
    using T = double;
    using Cfg = BinnedCfg<T, SHAPE, B, NW, DET>;
    using Acc = typename Cfg::Acc;
    constexpr int TE = Cfg::TE, RS = Cfg::RS, PS = Cfg::PS, TN = Cfg::TN;
    constexpr int NP = Cfg::NP, NS = Cfg::NS, WS = Cfg::WS, QO = Cfg::QO;
    extern __shared__ __align__(16) unsigned char smem[];
    T *sf = reinterpret_cast<T *>(smem);
    Acc *sd = reinterpret_cast<Acc *>(smem + Cfg::fields_bytes);
    T *stage = reinterpret_cast<T *>(smem + Cfg::fields_bytes + Cfg::dep_bytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T *sW = stage + warp * Cfg::stage_words;  // [32][WS]
    T *sQ = sW + 32 * WS;                     // [32][QO]: Q[0..7]

    if (lo >= hi)
        return;
    if (hi - lo <= sparse_bin_limit<T, B, DET>()) {
        sparse_cta<T, SHAPE, DET>(a, lo, hi);
        return;
    }
    const int ox = bx * B - 2, oy = by * B - 2, oz = bz * B - 2;
    constexpr int TT = TE * TE * TE;
    // grid offsets of the tile's rows along each axis (periodic): node of tile
    // point (lx, ly, lz) = s_axis[lx] + s_axis[TE + ly] + s_axis[2 TE + lz]
    __shared__ int s_axis[3 * TE];
    tile_axes<TE>(s_axis, ox, oy, oz, a.nx, a.ny, a.nz);
    __syncthreads();

    // stage the field tile (periodic) and clear the deposit tile
    constexpr int UF = 4;  // nodes per thread per pass: all loads issued first
    for (int t0 = threadIdx.x; t0 < TT; t0 += UF * blockDim.x) {
        T F[UF][6];
#pragma unroll
        for (int u = 0; u < UF; ++u) {
            const int t = t0 + u * int(blockDim.x);
            if (t < TT) {
                const int lx = t % TE, ly = (t / TE) % TE, lz = t / (TE * TE);
                const int node = s_axis[lx] + s_axis[TE + ly] + s_axis[2 * TE + lz];
                load_node(a.fields + int64_t(node) * 8, F[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < UF; ++u) {
            const int t = t0 + u * int(blockDim.x);
            if (t < TT) {
                const int lx = t % TE, ly = (t / TE) % TE, lz = t / (TE * TE);
                const int slot = lz * PS + ly * RS + lx;
                sts_node(sf + slot * 8, F[u]);
            }
        }
    }
    for (int t = threadIdx.x; t < 8 * TN; t += blockDim.x)
        sd[t] = Acc(0);
    __syncthreads();

    // phase-2 lane role: stencil offset and quantity range [q0, q0 + 2 or 8)
    const int off_id = SHAPE == 1 ? (lane & 7) : (lane < 27 ? lane : 0);
    const bool p2_active = SHAPE == 1 ? true : lane < 27;
    const int pax = off_id % NP, pay = (off_id / NP) % NP, paz = off_id / (NP * NP);
    const int q0 = SHAPE == 1 ? 2 * (lane >> 3) : 0;
    const int lane_off = paz * PS + pay * RS + pax;

    int flag = 0;
    // each warp walks a contiguous slice of the bin, so a run of equal stencil
    // origin that straddles two batches is carried over instead of flushed twice
    const uint32_t n_bin = hi - lo;
    const uint32_t per_warp = ((n_bin + NW - 1) / NW + 31) & ~31u;
    const uint32_t w_lo = lo + per_warp * uint32_t(warp);
    const uint32_t w_hi = w_lo + per_warp < hi ? w_lo + per_warp : hi;
    int carry_origin = -1;
    constexpr int NQ_ = SHAPE == 1 ? 2 : 8;
    T acc[NQ_];
#pragma unroll
    for (int q = 0; q < NQ_; ++q)
        acc[q] = T(0);
    auto flush_acc = [&](int origin) {
        if (p2_active && origin >= 0) {
            const int t = origin + lane_off;
#pragma unroll
            for (int q = 0; q < NQ_; ++q) {
                if (DET)
                    atomicAdd(reinterpret_cast<unsigned long long *>(&sd[(q0 + q) * TN + t]),
                              static_cast<unsigned long long>(to_fixed(acc[q] * a.fx_scale)));
                else
                    atomicAdd(reinterpret_cast<T *>(&sd[(q0 + q) * TN + t]), acc[q]);
            }
        }
    };
    // software pipeline: the packet fields of batch k+1 are loaded into
    // registers while batch k is pushed and deposited
    uint32_t n_c = 0;
    T n_o[3] = {T(0), T(0), T(0)}, n_u[3] = {T(0), T(0), T(0)}, n_w = T(0);
    auto prefetch = [&](uint32_t jj) {
        if (jj < w_hi) {
            n_c = a.cell[jj];
            n_o[0] = a.off0[jj];
            n_o[1] = a.off1[jj];
            n_o[2] = a.off2[jj];
            n_u[0] = a.u0[jj];
            n_u[1] = a.u1[jj];
            n_u[2] = a.u2[jj];
            n_w = a.w[jj];
        }
    };
    prefetch(w_lo + uint32_t(lane));
    for (uint32_t base = w_lo; base < w_hi; base += 32) {
        const uint32_t j = base + uint32_t(lane);
        const uint32_t c = n_c;
        T fx = n_o[0], fy = n_o[1], fz = n_o[2];
        const T u0[3] = {n_u[0], n_u[1], n_u[2]};
        const T wj = n_w;
        prefetch(j + 32);
        int staged = -1;
        if (j < w_hi) {
            const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
            if (ix >= a.nx || iy >= a.ny || iz >= a.nz) {
                flag |= ST_BADCELL;
            } else {
                T wx[3], wy[3], wz[3];
                int rx, ry, rz;
                const int jx = anchor_axis<SHAPE>(ix, fx, a.nx, wx, rx);
                const int jy = anchor_axis<SHAPE>(iy, fy, a.ny, wy, ry);
                const int jz = anchor_axis<SHAPE>(iz, fz, a.nz, wz, rz);
                // tile-local stencil origin
                int lx = jx + rx - ox, ly = jy + ry - oy, lz = jz + rz - oz;
                lx += lx < 0 ? a.nx : 0;
                ly += ly < 0 ? a.ny : 0;
                lz += lz < 0 ? a.nz : 0;
                lx -= lx >= a.nx ? a.nx : 0;
                ly -= ly >= a.ny ? a.ny : 0;
                lz -= lz >= a.nz ? a.nz : 0;
                const bool in_tile = lx >= 0 && ly >= 0 && lz >= 0 && lx + NP <= TE &&
                                     ly + NP <= TE && lz + NP <= TE;
                T E[3] = {T(0), T(0), T(0)}, Bf[3] = {T(0), T(0), T(0)};
                T Wk[NS];
#pragma unroll
                for (int cz = 0; cz < NP; ++cz)
#pragma unroll
                    for (int cy = 0; cy < NP; ++cy) {
                        const T wyz = wy[cy] * wz[cz];
#pragma unroll
                        for (int cx = 0; cx < NP; ++cx)
                            Wk[(cz * NP + cy) * NP + cx] = wx[cx] * wyz;
                    }
                int kx[3], ky[3], kz[3];
                if (in_tile) {
                    const int s0 = lz * PS + ly * RS + lx;
#pragma unroll
                    for (int cz = 0; cz < NP; ++cz)
#pragma unroll
                        for (int cy = 0; cy < NP; ++cy)
#pragma unroll
                            for (int cx = 0; cx < NP; ++cx) {
                                const T W = Wk[(cz * NP + cy) * NP + cx];
                                T F[6];
                                lds_node(sf + (s0 + cz * PS + cy * RS + cx) * 8, F);
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    E[q] += W * F[q];
                                    Bf[q] += W * F[3 + q];
                                }
                            }
                    staged = s0;
                } else {
                    axis_nodes(jx, rx, a.nx, kx);
                    axis_nodes(jy, ry, a.ny, ky);
                    axis_nodes(jz, rz, a.nz, kz);
#pragma unroll
                    for (int cz = 0; cz < NP; ++cz)
#pragma unroll
                        for (int cy = 0; cy < NP; ++cy) {
                            const int64_t row = (int64_t(kz[cz]) * a.ny + ky[cy]) * a.nx;
#pragma unroll
                            for (int cx = 0; cx < NP; ++cx) {
                                const T W = Wk[(cz * NP + cy) * NP + cx];
                                T F[6];
                                load_node(a.fields + (row + kx[cx]) * 8, F);
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    E[q] += W * F[q];
                                    Bf[q] += W * F[3 + q];
                                }
                            }
                        }
                }
                const BorisOut<T> b = boris(a.k.h, E, Bf, u0);
                const T g0 = Math<T>::sqrt(T(1) + dot3(u0, u0));
                T Q[8];
                feedback(a.k, wj, E, Bf, b, g0, Q);
                if (in_tile) {
                    store_wrow<WS>(sW + lane * WS, Wk);
                    store_q8(sQ + lane * QO, Q);
                } else {
#pragma unroll
                    for (int cz = 0; cz < NP; ++cz)
#pragma unroll
                        for (int cy = 0; cy < NP; ++cy) {
                            const int64_t row = (int64_t(kz[cz]) * a.ny + ky[cy]) * a.nx;
#pragma unroll
                            for (int cx = 0; cx < NP; ++cx) {
                                const T W = Wk[(cz * NP + cy) * NP + cx];
                                if (DET)
                                    red_node_fixed(a.fx + (row + kx[cx]) * 8, W, Q, a.fx_scale);
                                else
                                    red_node(a.fb + (row + kx[cx]) * 8, W, Q);
                            }
                        }
                }
                if (Math<T>::finite(b.u1[0]) && Math<T>::finite(b.u1[1]) &&
                    Math<T>::finite(b.u1[2])) {
                    const T s = a.k.adv * b.inv_g1;
                    const int nx_ = drift_axis(ix, fx, s * b.u1[0], a.nx, &flag);
                    const int ny_ = drift_axis(iy, fy, s * b.u1[1], a.ny, &flag);
                    const int nz_ = drift_axis(iz, fz, s * b.u1[2], a.nz, &flag);
                    a.cell[j] = pack_cell(nx_, ny_, nz_);
                    a.off0[j] = fx;
                    a.off1[j] = fy;
                    a.off2[j] = fz;
                    a.u0[j] = b.u1[0];
                    a.u1[j] = b.u1[1];
                    a.u2[j] = b.u1[2];
                } else {
                    flag |= ST_NONFINITE;
                }
            }
        }
        // runs of equal stencil origin along the lanes (the sorted order; equal
        // origin = same stencil nodes); a lane with no staged packet (-1: out of
        // the tile, or past the slice) starts a run that phase 2 skips
        const int left = __shfl_up_sync(0xffffffffu, staged, 1);
        const uint32_t starts = __ballot_sync(0xffffffffu, lane == 0 || staged != left);
        __syncwarp();

        // phase 2: stencil-offset lanes sum each run in registers (two packets per
        // pass) and add the sum to the tile when the origin changes (runs continue
        // across batches); all control below is warp-uniform
        uint32_t st = starts;
        while (st) {
            const int L = __ffs(st) - 1;
            st &= st - 1;
            const int R = st ? __ffs(st) - 1 : 32;
            const int origin = __shfl_sync(0xffffffffu, staged, L);
            if (origin < 0) {
                flush_acc(carry_origin);
                carry_origin = origin;
                continue;
            }
            const T *wrow = sW + L * WS + off_id;
            const T *qrow = sQ + L * QO + q0;
            int p = L;
            if (origin != carry_origin) {  // a new run: its first packet starts the sums
                flush_acc(carry_origin);
                carry_origin = origin;
                const T W = wrow[0];
                T Qp[NQ_];
                load_qpart<NQ_>(qrow, Qp);
#pragma unroll
                for (int q = 0; q < NQ_; ++q)
                    acc[q] = W * Qp[q];
                ++p;
                wrow += WS;
                qrow += QO;
            }
            for (; p + 1 < R; p += 2, wrow += 2 * WS, qrow += 2 * QO) {
                const T W = wrow[0], W2 = wrow[WS];
                T Qp[NQ_], Qp2[NQ_];
                load_qpart<NQ_>(qrow, Qp);
                load_qpart<NQ_>(qrow + QO, Qp2);
#pragma unroll
                for (int q = 0; q < NQ_; ++q) {
                    acc[q] += W * Qp[q];
                    acc[q] += W2 * Qp2[q];
                }
            }
            if (p < R) {
                const T W = wrow[0];
                T Qp[NQ_];
                load_qpart<NQ_>(qrow, Qp);
#pragma unroll
                for (int q = 0; q < NQ_; ++q)
                    acc[q] += W * Qp[q];
            }
        }
        __syncwarp();
    }
    flush_acc(carry_origin);
    __syncthreads();

    // add the deposit tile to the global grid (skip untouched nodes)
    for (int t = threadIdx.x; t < TE * TE * TE; t += blockDim.x) {
        const int lx = t % TE, ly = (t / TE) % TE, lz = t / (TE * TE);
        const int slot = lz * PS + ly * RS + lx;
        const int64_t node = s_axis[lx] + s_axis[TE + ly] + s_axis[2 * TE + lz];
        if (DET) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const long long v = sd[q * TN + slot];
                if (v != 0)
                    atomicAdd(reinterpret_cast<unsigned long long *>(a.fx + node * 8 + q),
                              static_cast<unsigned long long>(v));
            }
        } else {
            T v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q)
                v[q] = T(sd[q * TN + slot]);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (v[q] != T(0))
                    atomicAdd(a.fb + node * 8 + q, v[q]);
        }
    }
    if (flag)
        atomicOr(a.status, flag);
}


// ---------------------------------------------------------------------------
// FP32: packets pushed in memory order, deposited in octet order (octets.cuh).
// ---------------------------------------------------------------------------
template <int SHAPE, int B, int NW, bool DET>
struct OctPushCfg {
    // the deterministic deposit tile is twice as large, which leaves less to stage
    using O = OctetCfg<SHAPE, B + 4, DET ? (B == 8 ? 1480 : 1024) : 2680, DET ? 16 : 32>;
    static constexpr int TE = B + 4, TT = O::TT;
    // deposit planes: 2 DTN = 8 mod 32 puts the four value pairs of a run on
    // banks eight apart
    static constexpr int DTN = TT + 4;
    static_assert((2 * DTN) % 32 == 8, "deposit planes eight banks apart");
    // Field tile as two planes, {Ex, Ey, Ez, Bx} and {By, Bz} per node, z planes two
    // nodes apart: 16-byte loads of nearby nodes then spread over all banks.  (The
    // lanes of a warp hold packets of four neighbouring cells when fresh, of
    // about twenty after three steps of drift; with 32-byte nodes a gather load
    // then took 10 wavefronts, here 5, and 3 when fresh.)
    static constexpr int FZ = TE * TE + 2, FN = TE * FZ;
    static constexpr size_t fields_bytes = size_t(FN) * 6 * sizeof(float);
    // the bulk copy of the field tile (32-byte nodes) lands in the deposit tile
    // (deterministic: 64-bit sums, low words in planes 0..7, high words in 8..15)
    static constexpr size_t dep_bytes = size_t(DTN) * (DET ? 16 : 8) * sizeof(int);
    static constexpr size_t raw_bytes = size_t(TT) * 8 * sizeof(float);
    static_assert(raw_bytes <= dep_bytes && fields_bytes % 16 == 0, "field tile");
    static constexpr size_t align_pad = 128;  // of the bulk copy's destination
    static constexpr size_t smem_bytes = align_pad + dep_bytes + fields_bytes + O::stage_bytes + O::keep_bytes;
};

// One packet through global memory.  Not inlined: rare, and its unrolled gather
// and deposit would take registers from the CTA body.
template <int SHAPE, bool DET>
__device__ __noinline__ int push_global(const PushArgs<float> &a, uint32_t j)
{
    int flag = 0;
    auto gather_global = [&](int64_t node, float F[6]) { load_node(a.fields + node * 8, F); };
    auto deposit_global = [&](int64_t node, float W, const float Q[8]) {
        if constexpr (DET)
            red_node_fixed(a.fx + node * 8, W, Q, a.fx_scale);
        else
            red_node(a.fb + node * 8, W, Q);
    };
    push_one<float, SHAPE, true>(a, int64_t(j), gather_global, deposit_global, &flag);
    return flag;
}

// Add a 64-bit integer to the shared sum whose low word is *p and whose high word
// lies HI words further, with native 32-bit atomics: the carry out of the low
// word follows from the value the atomic returns.  (A 64-bit shared atomic is a
// compare-and-swap loop.)  The order of the additions does not matter.
template <int HI>
__device__ __forceinline__ void add_fixed64(int *p, long long v)
{
    const uint32_t lo = uint32_t(v);
    const uint32_t old = atomicAdd(reinterpret_cast<uint32_t *>(p), lo);
    const int hi = int(v >> 32) + (old + lo < lo ? 1 : 0);
    if (hi != 0)
        atomicAdd(p + HI, hi);
}

// Parts of a bin of n packets: two chunks each.
template <typename O>
__device__ __forceinline__ uint32_t octet_parts(uint32_t n)
{
    return ((n + O::CHUNK - 1) / O::CHUNK + 1) / 2;
}

// Parts [part, part + n_parts) of the bin's packets [lo, hi).
template <int SHAPE, int B, int NW, bool DET>
__device__ __forceinline__ void octet_cta(const PushArgs<float> &a, uint32_t lo, uint32_t hi, int bx,
                                          int by, int bz, uint32_t part, uint32_t n_parts,
                                          const CUtensorMap *tmap = nullptr)
{
    using Cfg = OctPushCfg<SHAPE, B, NW, DET>;
    using O = typename Cfg::O;
    constexpr int TE = Cfg::TE, TT = Cfg::TT, DTN = Cfg::DTN, NP = O::NP, NS = O::NS, NT = NW * 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((Cfg::align_pad - (smem_addr(smem_raw) & (Cfg::align_pad - 1))) &
                                      (Cfg::align_pad - 1));
    int *sd = reinterpret_cast<int *>(smem);  // first: 128-byte aligned
    float4 *sf4 = reinterpret_cast<float4 *>(smem + Cfg::dep_bytes);
    f32x2 *sf2 = reinterpret_cast<f32x2 *>(sf4 + Cfg::FN);
    unsigned char *stage = smem + Cfg::dep_bytes + Cfg::fields_bytes;
    const OctetMem<O> m(stage + O::stage_bytes, stage);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (lo >= hi)
        return;
    int flag = 0;
    if (hi - lo <= sparse_cta_limit<SHAPE, B, DET>()) {
        for (uint32_t j = lo + threadIdx.x; j < hi; j += NT)
            flag |= push_global<SHAPE, DET>(a, j);
        if (flag)
            atomicOr(a.status, flag);
        return;
    }
    const int ox = bx * B - 2, oy = by * B - 2, oz = bz * B - 2;
    // A tile that does not wrap around the periodic grid on any axis is one box
    // of the field grid: one bulk tensor copy (TMA) issued by thread 0 lands it
    // while the threads count the origins below.
    const bool tma = tmap != nullptr && ox >= 0 && oy >= 0 && oz >= 0 && ox + TE <= a.nx &&
                     oy + TE <= a.ny && oz + TE <= a.nz;
    __shared__ uint64_t s_tma_bar;
    if (tma && threadIdx.x == 0)
        mbar_init(&s_tma_bar, 1);
    __shared__ int s_axis[3 * TE];
    tile_axes<TE>(s_axis, ox, oy, oz, a.nx, a.ny, a.nz);
    octet_clear<O, NW>(m);
    __syncthreads();
    if (tma && threadIdx.x == 0) {
        mbar_arrive_expect_tx(&s_tma_bar, uint32_t(Cfg::raw_bytes));
        tma_load_4d(sd, tmap, 0, ox, oy, oz, &s_tma_bar);
    }
    // a node of the tile into its planes; the fixed-point scale needs the largest
    // |E| and, per axis a, the largest |B| across a (B with its a component removed)
    float e2max = 0.f, bp2max[3] = {0.f, 0.f, 0.f};
    auto set_node = [&](int t, const float F[6]) {
        const int k = t + (t / (TE * TE)) * (Cfg::FZ - TE * TE);
        sf4[k] = make_float4(F[0], F[1], F[2], F[3]);
        sf2[k] = f2_pack(F[4], F[5]);
        e2max = fmaxf(e2max, F[0] * F[0] + F[1] * F[1] + F[2] * F[2]);
        const float bx2 = F[3] * F[3], by2 = F[4] * F[4], bz2 = F[5] * F[5];
        bp2max[0] = fmaxf(bp2max[0], by2 + bz2);
        bp2max[1] = fmaxf(bp2max[1], bx2 + bz2);
        bp2max[2] = fmaxf(bp2max[2], bx2 + by2);
    };
    if (!tma) {
        constexpr int UF = 4;  // nodes per thread per pass: all loads issued first
        for (int t0 = threadIdx.x; t0 < TT; t0 += UF * NT) {
            float F[UF][6];
#pragma unroll
            for (int u = 0; u < UF; ++u) {
                const int t = t0 + u * NT;
                if (t < TT) {
                    const int node = s_axis[t % TE] + s_axis[TE + (t / TE) % TE] + s_axis[2 * TE + t / (TE * TE)];
                    load_node(a.fields + int64_t(node) * 8, F[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < UF; ++u) {
                const int t = t0 + u * NT;
                if (t < TT)
                    set_node(t, F[u]);
            }
        }
    }
    for (int t = threadIdx.x + (tma ? 2 * TT : 0); t < int(Cfg::dep_bytes / 16); t += NT)
        reinterpret_cast<int4 *>(sd)[t] = make_int4(0, 0, 0, 0);

    // Origin counts of packets [lo_, hi_), chunk 1 from packet split_ on, and each
    // packet's origin and rank within it and its chunk; returns the largest |w|.
    auto count_origins = [&](uint32_t lo_, uint32_t split_, uint32_t hi_) {
        float wmax = 0.f;
        constexpr int U = 4;  // packets per thread per pass: all loads issued first
        for (uint32_t j0 = lo_ + threadIdx.x; j0 < hi_; j0 += U * NT) {
            uint32_t cc[U];
            float f0[U], f1[U], f2[U], ww[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + uint32_t(u) * NT;
                const bool ok = j < hi_;
                cc[u] = ok ? a.cell[j] : 0xFFFFFFFFu;
                f0[u] = ok ? a.off0[j] : 0.f;
                f1[u] = ok ? a.off1[j] : 0.f;
                f2[u] = ok ? a.off2[j] : 0.f;
                ww[u] = ok ? a.w[j] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + uint32_t(u) * NT;
                wmax = fmaxf(wmax, fabsf(ww[u]));
                // tile slot of the stencil's first node; out of the tile or off the grid: TT
                const int ix = cell_x(cc[u]), iy = cell_y(cc[u]), iz = cell_z(cc[u]);
                const int lx = wrap_once(ix + first_node<SHAPE>(f0[u]) - ox, a.nx),
                          ly = wrap_once(iy + first_node<SHAPE>(f1[u]) - oy, a.ny),
                          lz = wrap_once(iz + first_node<SHAPE>(f2[u]) - oz, a.nz);
                const bool in = ix < a.nx && iy < a.ny && iz < a.nz && max(max(lx, ly), lz) <= TE - NP;
                const int key = in ? (lz * TE + ly) * TE + lx : TT;
                int *h = m.hist + (j >= split_ ? TT : 0) + key;
                if (key < TT)
                    m.rank[j - lo_] = uint16_t(atomicAdd(h, 1));
                if (j < hi_)
                    m.key[j - lo_] = uint16_t(key);
            }
        }
        return wmax;
    };
    const int pair = lane & 3;
    auto flush = [&](int slot, f32x2 (&acc)[NS]) {
        int *p = sd + 2 * pair * DTN + slot;
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const int off = (k / (NP * NP)) * TE * TE + ((k / NP) % NP) * TE + k % NP;
            float x, y;
            f2_unpack(acc[k], x, y);
            if constexpr (DET) {
                add_fixed64<8 * DTN>(p + off, to_fixed(x * a.fx_scale));
                add_fixed64<8 * DTN>(p + DTN + off, to_fixed(y * a.fx_scale));
            } else {  // values staged pre-scaled
                atomicAdd(p + off, __float2int_rn(x));
                atomicAdd(p + DTN + off, __float2int_rn(y));
            }
        }
    };
    // The bin in chunks of nearly equal size (all but the last a multiple of the widest
    // CTA where that leaves room in the last), ordered two at a time.  Each two chunks
    // have their own scale, from the packets in them, and their own tile.  The cut does
    // not depend on this CTA's width: deterministic sums round per run, and the runs
    // end with their chunk.
    constexpr uint32_t STEP = 512;
    const uint32_t n_bin = hi - lo, n_chunks = (n_bin + O::CHUNK - 1) / O::CHUNK;
    uint32_t chunk = (n_bin + n_chunks - 1) / n_chunks;
    if (chunk >= STEP && n_bin - chunk / STEP * STEP * (n_chunks - 1) <= O::CHUNK)
        chunk = chunk / STEP * STEP;
    const uint32_t c_first = 2 * part;
    const uint32_t c_end = n_parts < octet_parts<O>(n_bin) - part ? 2 * (part + n_parts) : n_chunks;
    __shared__ float s_scale[8], s_iscale[8];
#pragma unroll 1
    for (uint32_t c = c_first; c < c_end; c += 2) {
        const uint32_t p_lo = lo + c * chunk;
        const uint32_t split = c + 1 < n_chunks ? p_lo + chunk : hi;
        const uint32_t p_hi = c + 2 < n_chunks ? split + chunk : hi;
        if (c > c_first) {
            __syncthreads();  // the previous part's tile has been added and cleared
            octet_clear<O, NW>(m);
            __syncthreads();
        }
        const float wmax = count_origins(p_lo, split, p_hi);
        __syncthreads();
        if constexpr (DET)
            octet_stable_ranks<O, NW>(m, int(split - p_lo), int(p_hi - p_lo));
        // the weight bound's three passes run between the order's barriers
        float gmax = 0.f;
        auto bound_pass = [&](int pass) {
            if (!DET)
                weight_bound_pass<SHAPE, TE, TE, TE * TE>(
                    pass, [&](int t) { return m.hist[t] + m.hist[TT + t]; }, m.scratch, gmax);
        };
        int noct[2];
        octet_order<O, NW>(m, int(split - p_lo), int(p_hi - p_lo), noct, bound_pass);
        if (tma && c == c_first) {
            // the bulk copy: wait for it (bounded), then the planes from the copied tile,
            // which is cleared for the deposit
            const bool arrived = mbar_wait_bounded(&s_tma_bar, 0, kTmaWaitCycles);
            if (!__syncthreads_and(arrived)) {
                // report it, give the copy one more bounded wait, skip the bin
                if (threadIdx.x == 0) {
                    atomicOr(a.status, ST_TIMEOUT);
                    mbar_wait_bounded(&s_tma_bar, 0, kTmaWaitCycles);
                }
                __syncthreads();
                return;
            }
            for (int t = threadIdx.x; t < TT; t += NT) {
                float F[6];
                lds_node(reinterpret_cast<const float *>(sd) + t * 8, F);
                set_node(t, F);
                reinterpret_cast<int4 *>(sd)[2 * t] = make_int4(0, 0, 0, 0);
                reinterpret_cast<int4 *>(sd)[2 * t + 1] = make_int4(0, 0, 0, 0);
            }
        }
        // 32-bit fixed point: scale_q = 2^e with (largest weight a node can receive) *
        // bound_q below 2^31 / 1.002 (the margin covers the rounding of the bound and
        // of the sums added), bound_q a bound on one packet's |Q_q| (|beta_bar| < 1):
        //   rho: w q / dx^3;  J: rho c;  S_a: rho (|E| + |B across a|), since
        //   |(beta_bar x B)_a| <= |beta_bar| |B with its a component removed|;
        //   H: rho c |E| (1 + h |E|)
        // (deterministic: the context's scale, in 64 bits)
        if constexpr (!DET) {
            __shared__ float s_red[6][NW];
            float red[6] = {e2max, wmax, bp2max[0], bp2max[1], bp2max[2], gmax};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    red[k] = fmaxf(red[k], __shfl_xor_sync(0xffffffffu, red[k], o));
            if (lane == 0)
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    s_red[k][warp] = red[k];
            __syncthreads();
            if (threadIdx.x < 8) {
                const int q = threadIdx.x;
                const int bp = q >= 4 && q < 7 ? 2 + (q - 4) : 2;  // S_q: |B| across axis q - 4
                float em = 0.f, bm = 0.f, wm = 0.f, gm = 0.f;
                for (int w = 0; w < NW; ++w) {
                    em = fmaxf(em, s_red[0][w]);
                    wm = fmaxf(wm, s_red[1][w]);
                    bm = fmaxf(bm, s_red[bp][w]);
                    gm = fmaxf(gm, s_red[5][w]);
                }
                em = sqrtf(em);
                bm = sqrtf(bm);
                const float rho = wm * fabsf(a.k.qv);
                float bound = q == 0 ? rho
                            : q < 4  ? rho * a.k.c
                            : q < 7  ? rho * (em + bm)
                                     : rho * a.k.c * em * (1.f + fabsf(a.k.h) * em);
                bound *= gm > 1.f ? gm : 1.f;
                bound *= 1.002f;
                int e = 30;
                if (bound > 0.f && isfinite(bound))
                    e = 31 - int(ceilf(log2f(bound)));
                e = e > 60 ? 60 : (e < -60 ? -60 : e);
                s_scale[q] = ldexpf(1.0f, e);
                s_iscale[q] = ldexpf(1.0f, -e);
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int ch = 0; ch < 2; ++ch) {
            const uint32_t c_lo = ch ? split : p_lo, c_hi = ch ? p_hi : split;
            if (c_lo >= c_hi)
                break;
            // software pipeline: a thread's next packet is loaded into registers while
            // this one is pushed
            uint32_t n_c = 0;
            int n_place = 0;
            float n_o[3] = {0.f, 0.f, 0.f}, n_u[3] = {0.f, 0.f, 0.f}, n_w = 0.f;
            auto prefetch = [&](uint32_t j) {
                if (j < c_hi) {
                    n_place = m.place[j - p_lo];
                    n_c = a.cell[j];
                    n_o[0] = a.off0[j];
                    n_o[1] = a.off1[j];
                    n_o[2] = a.off2[j];
                    n_u[0] = a.u0[j];
                    n_u[1] = a.u1[j];
                    n_u[2] = a.u2[j];
                    n_w = a.w[j];
                }
            };
            prefetch(c_lo + threadIdx.x);
            for (uint32_t j = c_lo + threadIdx.x; j < c_hi; j += NT) {
                const uint32_t c = n_c;
                const int place = n_place;
                float fx = n_o[0], fy = n_o[1], fz = n_o[2];
                const float u0[3] = {n_u[0], n_u[1], n_u[2]};
                const float wj = n_w;
                prefetch(j + NT);
                const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
                if (place == kOctNone) {  // off the grid, or drifted out of the tile since the sort
                    flag |= push_global<SHAPE, DET>(a, j);
                    continue;
                }
                float wx[3], wy[3], wz[3];
                // tile slot of the stencil's first node (place is set: it lies in the tile)
                const int slot = wrap_once(iz + axis_weights<SHAPE>(fz, wz) - oz, a.nz) * Cfg::FZ +
                                 wrap_once(iy + axis_weights<SHAPE>(fy, wy) - oy, a.ny) * TE +
                                 wrap_once(ix + axis_weights<SHAPE>(fx, wx) - ox, a.nx);
                // pairs {Ex, Ey}, {Ez, Bx}, {By, Bz}: a node is one 16-byte and one
                // 8-byte load, one paired product (its weight in both halves) and
                // three paired multiply-adds; same bits as the order-free kernel
                f32x2 g01 = 0, g23 = 0, g45 = 0;  // +0.0f in both halves
                f32x2 wx2[NP];
#pragma unroll
                for (int cx = 0; cx < NP; ++cx)
                    wx2[cx] = f2_pack(wx[cx], wx[cx]);
                const float4 *p4 = sf4 + slot;
                const f32x2 *p2 = sf2 + slot;
#pragma unroll
                for (int k = 0; k < NP * NP; ++k) {
                    const float wyz = wy[k % NP] * wz[k / NP];
                    const f32x2 wk = f2_pack(wyz, wyz);
#pragma unroll
                    for (int cx = 0; cx < NP; ++cx) {
                        const f32x2 W2 = f2_mul(wx2[cx], wk);
                        const int off = (k / NP) * Cfg::FZ + (k % NP) * TE + cx;
                        const ulonglong2 a2 = *reinterpret_cast<const ulonglong2 *>(p4 + off);
                        const f32x2 b2 = p2[off];
                        g01 = f2_fma(W2, a2.x, g01);
                        g23 = f2_fma(W2, a2.y, g23);
                        g45 = f2_fma(W2, b2, g45);
                    }
                }
                float E[3], Bf[3];
                f2_unpack(g01, E[0], E[1]);
                f2_unpack(g23, E[2], Bf[0]);
                f2_unpack(g45, Bf[1], Bf[2]);
                const BorisOut<float> b = boris(a.k.h, E, Bf, u0);
                const float g0 = Math<float>::sqrt(1.f + dot3(u0, u0));
                float Q[8];
                feedback(a.k, wj, E, Bf, b, g0, Q);
                if constexpr (!DET) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)  // the tile's fixed-point scale (a power of two: exact)
                        Q[q] *= s_scale[q];
                }
                octet_stage<O>(m, place, octet_offset<SHAPE>(fx), octet_offset<SHAPE>(fy),
                                       octet_offset<SHAPE>(fz), Q);
                if (Math<float>::finite(b.u1[0]) && Math<float>::finite(b.u1[1]) &&
                    Math<float>::finite(b.u1[2])) {
                    const float s = a.k.adv * b.inv_g1;
                    const int nx_ = drift_axis(ix, fx, s * b.u1[0], a.nx, &flag);
                    const int ny_ = drift_axis(iy, fy, s * b.u1[1], a.ny, &flag);
                    const int nz_ = drift_axis(iz, fz, s * b.u1[2], a.nz, &flag);
                    a.cell[j] = pack_cell(nx_, ny_, nz_);
                    a.off0[j] = fx;
                    a.off1[j] = fy;
                    a.off2[j] = fz;
                    a.u0[j] = b.u1[0];
                    a.u1[j] = b.u1[1];
                    a.u2[j] = b.u1[2];
                } else {
                    flag |= ST_NONFINITE;
                }
            }
            __syncthreads();
            octet_deposit<O, NW, !DET>(m, ch, noct[ch], flush);
            __syncthreads();  // the next chunk reuses the stage
        }
        // add the deposit tile to the global grid (skip untouched nodes); exact 64-bit
        // sums wait for the last part
        if (DET && c + 2 < c_end)
            continue;
        for (int t = threadIdx.x; t < TT; t += NT) {
            const int64_t node = s_axis[t % TE] + s_axis[TE + (t / TE) % TE] + s_axis[2 * TE + t / (TE * TE)];
            if constexpr (DET) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const unsigned long long v = uint32_t(sd[q * DTN + t]) |
                                                 (unsigned long long)(uint32_t(sd[(8 + q) * DTN + t])) << 32;
                    if (v != 0)
                        atomicAdd(reinterpret_cast<unsigned long long *>(a.fx + node * 8 + q), v);
                }
            } else {
                float v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    v[q] = float(sd[q * DTN + t]) * s_iscale[q];
                    sd[q * DTN + t] = 0;
                }
                float *p = a.fb + node * 8;
                if (v[0] != 0.f || v[1] != 0.f || v[2] != 0.f || v[3] != 0.f)
                    atomicAdd(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
                if (v[4] != 0.f || v[5] != 0.f || v[6] != 0.f || v[7] != 0.f)
                    atomicAdd(reinterpret_cast<float4 *>(p + 4), make_float4(v[4], v[5], v[6], v[7]));
            }
        }
    }
    if (flag)
        atomicOr(a.status, flag);
    if (tma && threadIdx.x == 0)  // every thread waited on it before the chunks
        mbar_inval(&s_tma_bar);
}

// The CTA body and its shared memory: octet order for FP32, one run per pass for FP64
// (whose accumulators, a double per node and value, would not fit the registers).
template <typename T>
constexpr bool kUsesOctets = sizeof(T) == 4;
template <typename T, int SHAPE, int B, int NW, bool DET>
constexpr size_t tile_smem_bytes()
{
    if constexpr (kUsesOctets<T>)
        return OctPushCfg<SHAPE, B, NW, DET>::smem_bytes;
    else
        return BinnedCfg<T, SHAPE, B, NW, DET>::smem_bytes;
}
template <typename T, int SHAPE, int B, int NW, bool DET>
__device__ __forceinline__ void tile_cta(const PushArgs<T> &a, uint32_t lo, uint32_t hi, int bx, int by,
                                         int bz, uint32_t part = 0, uint32_t n_parts = 0xFFFFFFFFu,
                                         const CUtensorMap *tmap = nullptr)
{
    if constexpr (kUsesOctets<T>)
        octet_cta<SHAPE, B, NW, DET>(a, lo, hi, bx, by, bz, part, n_parts, tmap);
    else
        binned_cta<SHAPE, B, NW, DET>(a, lo, hi, bx, by, bz);
}

template <typename T, int SHAPE, int B, int NW, bool DET>
__global__ void __launch_bounds__(NW * 32)
    push_binned_kernel(const __grid_constant__ PushArgs<T> a, const __grid_constant__ BinGeom g,
                       int ahead, const __grid_constant__ CUtensorMap tmap, int use_tma)
{
    const int bin = blockIdx.x;
    const int bx = bin % g.nbx, by = (bin / g.nbx) % g.nby, bz = bin / (g.nbx * g.nby);
    // the bin that starts about one wave of CTAs later: its packets into L2 now
    if (bin + ahead < int(gridDim.x)) {
        const uint32_t plo = g.bin_start[bin + ahead], phi = g.bin_start[bin + ahead + 1];
        prefetch_l2(a.cell, plo, phi);
        prefetch_l2(a.off0, plo, phi);
        prefetch_l2(a.off1, plo, phi);
        prefetch_l2(a.off2, plo, phi);
        prefetch_l2(a.u0, plo, phi);
        prefetch_l2(a.u1, plo, phi);
        prefetch_l2(a.u2, plo, phi);
        prefetch_l2(a.w, plo, phi);
    }
    const uint32_t lo = g.bin_start[bin];
    uint32_t hi = g.bin_start[bin + 1];
    if constexpr (kUsesOctets<T>) {
        hi = hi - lo <= g.skip ? lo : hi;  // (an early return here cost CIC bins 4 %)
        if (gridDim.y > 1) {  // a sparse bin in slices; a dense one is the first slice's
            const uint32_t n = hi - lo, slice = blockIdx.y;
            if (n <= sliced_cta_limit<SHAPE, B, DET>(gridDim.y)) {
                const uint32_t share = (n + gridDim.y - 1) / gridDim.y;
                const uint32_t s_hi = min((slice + 1) * share, n);
                int flag = 0;
                for (uint32_t i = slice * share + threadIdx.x; i < s_hi; i += NW * 32)
                    flag |= push_global<SHAPE, DET>(a, lo + i);
                if (flag)
                    atomicOr(a.status, flag);
                return;
            }
            if (slice > 0)
                return;
        }
    }
    tile_cta<T, SHAPE, B, NW, DET>(a, lo, hi, bx, by, bz, 0, 0xFFFFFFFFu, use_tma ? &tmap : nullptr);
}

// The bins of at most kGlobalBinMost packets of one box, a CTA per kSplitShare packets: for
// sets sparse on many bins, where a CTA with tiles per bin leaves each SM one bin's few
// packets to wait for.  A denser bin is left to push_binned_kernel, launched after it, so
// that crowded packets keep their tile's accuracy.
constexpr int kSplitShare = 128;
template <int SHAPE>
__global__ void __launch_bounds__(kSplitShare) push_sparse_bins_kernel(const __grid_constant__ PushArgs<float> a,
                                                                       const uint32_t *__restrict__ bin_start)
{
    const uint32_t lo = bin_start[blockIdx.x], n = bin_start[blockIdx.x + 1] - lo;
    const uint32_t i = blockIdx.y * kSplitShare + threadIdx.x;
    if (n > kGlobalBinMost || i >= n)
        return;
    int flag = 0;
    auto gather_global = [&](int64_t node, float F[6]) { load_node(a.fields + node * 8, F); };
    auto deposit_global = [&](int64_t node, float W, const float Q[8]) { red_node(a.fb + node * 8, W, Q); };
    push_one<float, SHAPE, true>(a, int64_t(lo) + i, gather_global, deposit_global, &flag);
    if (flag)
        atomicOr(a.status, flag);
}

// One box of a batch: grid, node offset into the concatenated grids, first
// global bin, and its step constants (c~ and dt differ between boxes).
template <typename T>
struct BatchBox {
    int nx, ny, nz, nbx, nby, nbz;
    int64_t node_off;
    uint32_t bin_base;
    StepConst<T> k;
};

// Box of global bin gb: the last box whose first bin is <= gb.
template <typename T>
__device__ __forceinline__ int batch_box_of(const BatchBox<T> *__restrict__ boxes, int n_boxes,
                                            uint32_t gb)
{
    int lo_b = 0, hi_b = n_boxes - 1;
    while (lo_b < hi_b) {
        const int mid = (lo_b + hi_b + 1) >> 1;
        if (boxes[mid].bin_base <= gb)
            lo_b = mid;
        else
            hi_b = mid - 1;
    }
    return lo_b;
}

// The batch's push arguments narrowed to one box: its geometry, constants and
// slices of the concatenated grids.
template <typename T>
__device__ __forceinline__ PushArgs<T> batch_box_args(const PushArgs<T> &base, const BatchBox<T> &bx_)
{
    PushArgs<T> a = base;
    a.nx = bx_.nx;
    a.ny = bx_.ny;
    a.nz = bx_.nz;
    a.k = bx_.k;
    a.fields = base.fields + bx_.node_off * 8;
    a.fb = base.fb ? base.fb + bx_.node_off * 8 : nullptr;
    a.fx = base.fx ? base.fx + bx_.node_off * 8 : nullptr;
    return a;
}

// Work area of a batch push (device, batch_work_words): claim counters,
// zeroed before each push, and the list of the dense bins of this push.
constexpr int kClaimSparse = 0;  // next bin a warp of the sparse kernel claims
constexpr int kDenseCount = 1;   // parts of dense bins listed by the sparse kernel
constexpr int kClaimDense = 2;   // next list entry a CTA of the tiled kernel claims
constexpr int kDenseList = 3;    // the list itself, a bin and a part each

// The sparse bins of a batch (at most sparse_bin_limit packets): one warp per
// bin, each lane one packet at a time, gathering from global memory and
// depositing with global vector atomics.  Independent warps in small CTAs
// keep more gathers and atomics in flight than the tiled kernel's CTAs, which
// would stall a whole CTA on each sparse bin.  Warps claim the bins in order
// from a counter (a bin's cost follows its packet count, so a fixed share per
// warp would leave some warps with several large bins); a dense bin is only
// listed for the tiled kernel, an entry per part.  Each bin is claimed once and a
// bin of n packets has at most 1 + n / (2 chunk) parts, chunk >= 776, so the list
// holds at most one entry per bin and one per 1024 packets.
constexpr int kSparseWarps = 4;
template <typename T, int SHAPE, int B, bool DET>
__global__ void __launch_bounds__(kSparseWarps * 32) push_batch_sparse_kernel(
    PushArgs<T> base, const BatchBox<T> *__restrict__ boxes, int n_boxes,
    const uint32_t *__restrict__ bin_start, uint32_t total_bins, uint32_t *work)
{
    const int lane = threadIdx.x & 31;
    int sflag = 0;
    uint32_t next = 0;
    if (lane == 0)
        next = atomicAdd(&work[kClaimSparse], 1u);
    uint32_t gb = __shfl_sync(0xffffffffu, next, 0);
    while (gb < total_bins) {
        if (lane == 0)  // the next claim is in flight while this bin is pushed
            next = atomicAdd(&work[kClaimSparse], 1u);
        const uint32_t lo = bin_start[gb], hi = bin_start[gb + 1];
        if (hi - lo > sparse_bin_limit<T, B, DET>()) {
            if (lane == 0) {
                // one entry per part of the bin, so that a very dense bin is shared out
                uint32_t parts = 1;
                if constexpr (kUsesOctets<T>)
                    parts = octet_parts<typename OctPushCfg<SHAPE, B, 16, DET>::O>(hi - lo);
                const uint32_t at = atomicAdd(&work[kDenseCount], parts);
                for (uint32_t p = 0; p < parts; ++p) {
                    work[kDenseList + 2 * (at + p)] = gb;
                    work[kDenseList + 2 * (at + p) + 1] = p;
                }
            }
        } else if (lo < hi) {
            const PushArgs<T> a = batch_box_args(base, boxes[batch_box_of(boxes, n_boxes, gb)]);
            auto gather_global = [&](int64_t node, T F[6]) { load_node(a.fields + node * 8, F); };
            auto deposit_global = [&](int64_t node, T W, const T Q[8]) {
                if (DET)
                    red_node_fixed(a.fx + node * 8, W, Q, a.fx_scale);
                else
                    red_node(a.fb + node * 8, W, Q);
            };
            for (uint32_t j = lo + uint32_t(lane); j < hi; j += 32)
                push_one<T, SHAPE, true>(a, int64_t(j), gather_global, deposit_global, &sflag);
        }
        gb = __shfl_sync(0xffffffffu, next, 0);
    }
    if (sflag)
        atomicOr(base.status, sflag);
}

// Persistent kernel over the dense bins the sparse kernel listed: CTAs claim
// list entries from a counter (dynamic balance: an entry holds from just over
// sparse_bin_limit to 4352 packets); each is processed by the same CTA body as the single-box kernel, with its box's geometry, grids and
// constants.
template <typename T, int SHAPE, int B, int NW, bool DET>
__global__ void __launch_bounds__(NW * 32) push_batch_kernel(PushArgs<T> base,
                                                             const BatchBox<T> *__restrict__ boxes,
                                                             int n_boxes,
                                                             const uint32_t *__restrict__ bin_start,
                                                             uint32_t *work)
{
    __shared__ uint32_t s_gb, s_part;
    const uint32_t n_dense = work[kDenseCount];  // complete: the sparse kernel ran before
    for (;;) {
        if (threadIdx.x == 0) {
            const uint32_t i = atomicAdd(&work[kClaimDense], 1u);
            s_gb = i < n_dense ? work[kDenseList + 2 * i] : 0xFFFFFFFFu;
            s_part = i < n_dense ? work[kDenseList + 2 * i + 1] : 0u;
        }
        __syncthreads();
        const uint32_t gb = s_gb;
        if (gb == 0xFFFFFFFFu)
            break;  // block-uniform
        const int ib = batch_box_of(boxes, n_boxes, gb);
        const BatchBox<T> bx_ = boxes[ib];
        PushArgs<T> a = batch_box_args(base, bx_);
        const int lb = int(gb - bx_.bin_base);
        const int bx = lb % bx_.nbx, by = (lb / bx_.nbx) % bx_.nby, bz = lb / (bx_.nbx * bx_.nby);
        tile_cta<T, SHAPE, B, NW, DET>(a, bin_start[gb], bin_start[gb + 1], bx, by, bz, s_part, 1);
        __syncthreads();  // the next bin reuses the shared tiles and s_gb
    }
}

// Warps per CTA: as many as the shared-memory budget allows (at most 16, a
// multiple of 4); 0 when even four warps do not fit (the order-free kernel runs).
template <typename T, int SHAPE, int B, bool DET>
constexpr int binned_warps()
{
    if constexpr (kUsesOctets<T>)
        return 16;
    using C0 = BinnedCfg<T, SHAPE, B, 0, DET>;
    constexpr size_t budget = 232448 - 1024;  // leave room for static shared memory
    constexpr size_t fixed = C0::fields_bytes + C0::dep_bytes;
    constexpr size_t per_warp = C0::stage_words * sizeof(T);
    constexpr size_t fit = fixed >= budget ? 0 : (budget - fixed) / per_warp;
    constexpr int cap = DET ? 8 : 16;  // deterministic kernels need more registers
    constexpr int nw = int(fit > size_t(cap) ? size_t(cap) : fit) & ~3;
    return nw;
}

// Tensor map of a node-major FP32 field grid (eight components per node)
// whose box is one bin's tile of te^3 nodes; false (no bulk copies: the tiles
// are staged with ordinary loads) when the driver does not provide the encoder,
// the grid is smaller than a tile or the grid is not 16-byte aligned.
inline bool encode_field_tile_map(CUtensorMap *map, const void *fields, int nx, int ny, int nz, int te)
{
    using Encode = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Encode encode = []() -> Encode {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault,
                                             &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<Encode>(f);
    }();
    if (!encode || (reinterpret_cast<uintptr_t>(fields) & 15u) || nx < te || ny < te || nz < te)
        return false;
    const cuuint64_t dims[4] = {8, cuuint64_t(nx), cuuint64_t(ny), cuuint64_t(nz)};
    const cuuint64_t strides[3] = {32, 32ull * uint64_t(nx), 32ull * uint64_t(nx) * uint64_t(ny)};
    const cuuint32_t box[4] = {8, cuuint32_t(te), cuuint32_t(te), cuuint32_t(te)};
    const cuuint32_t elem[4] = {1, 1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<void *>(fields), dims, strides,
                  box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename T, int SHAPE, int B, bool DET, int NW>
cudaError_t launch_binned_nw(const PushArgs<T> &a, const BinGeom &g, int nbins, int sm_count,
                             cudaStream_t s)
{
    constexpr size_t smem = tile_smem_bytes<T, SHAPE, B, NW, DET>();
    static_assert(smem <= 232448, "binned tile exceeds shared memory");
    auto kern = push_binned_kernel<T, SHAPE, B, NW, DET>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(smem));
    if (e != cudaSuccess)
        return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NW * 32, smem);
    if (e != cudaSuccess)
        return e;
    const int wave = sm_count * (per_sm > 0 ? per_sm : 1);  // CTAs resident at a time
    // FP32 tiles: interior bins take their fields with one bulk tensor copy
    CUtensorMap map{};
    const int use_tma = sizeof(T) == 4 && encode_field_tile_map(&map, a.fields, a.nx, a.ny, a.nz, B + 4);
    const int slices = kUsesOctets<T> ? bin_slices(sm_count, nbins) : 1;
    kern<<<dim3(unsigned(nbins), unsigned(slices)), NW * 32, smem, s>>>(a, g, wave, map, use_tma);
    return cudaGetLastError();
}

// The binned kernel with the requested CTA width: 8 warps, or (0, 16) the
// widest that fits shared memory; the order-free kernel if not even 4 fit.
template <typename T, int SHAPE, int B, bool DET>
cudaError_t launch_binned(const PushArgs<T> &a, const BinGeom &g, int nbins, int sm_count, int warps,
                          cudaStream_t s)
{
    constexpr int NW = binned_warps<T, SHAPE, B, DET>();
    if constexpr (NW < 4) {
        return launch_unbinned<T, SHAPE, true, DET>(a, sm_count, s);
    } else if constexpr (NW > 8) {
        if (warps == 8)
            return launch_binned_nw<T, SHAPE, B, DET, 8>(a, g, nbins, sm_count, s);
        return launch_binned_nw<T, SHAPE, B, DET, NW>(a, g, nbins, sm_count, s);
    } else {
        return launch_binned_nw<T, SHAPE, B, DET, NW>(a, g, nbins, sm_count, s);
    }
}

template <typename T>
cudaError_t push_binned_dispatch(const PushDesc &d, cudaStream_t s)
{
    const PushArgs<T> a = make_push_args<T>(d);
    BinGeom g{d.bin_start, d.nbx, d.nby, d.nbz};
    const int nbins = d.nbx * d.nby * d.nbz;
    const bool det = d.det != 0;
    if constexpr (kUsesOctets<T>) {
        if (d.split) {
            const dim3 grid{unsigned(nbins), unsigned((kGlobalBinMost + kSplitShare - 1) / kSplitShare)};
            auto kern = d.shape == 1 ? push_sparse_bins_kernel<1> : push_sparse_bins_kernel<2>;
            kern<<<grid, kSplitShare, 0, s>>>(a, d.bin_start);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess)
                return e;
            g.skip = kGlobalBinMost;
        }
    }
#define RSOL_BINNED(SH, BB)                                                                  \
    return det ? launch_binned<T, SH, BB, true>(a, g, nbins, d.sm_count, d.warps, s)        \
               : launch_binned<T, SH, BB, false>(a, g, nbins, d.sm_count, d.warps, s)
    if (d.shape == 1) {
        if (d.bin == 4) { RSOL_BINNED(1, 4); }
        RSOL_BINNED(1, 8);
    }
    if (d.bin == 4) { RSOL_BINNED(2, 4); }
    RSOL_BINNED(2, 8);
#undef RSOL_BINNED
}

template <typename T, int SHAPE, int B, bool DET, int NWREQ>
cudaError_t launch_batch(const PushArgs<T> &a, const BatchBox<T> *boxes, int n_boxes,
                         const uint32_t *bin_start, uint32_t total_bins, uint32_t *work,
                         int sm_count, cudaStream_t s)
{
    constexpr int NWMAX = binned_warps<T, SHAPE, B, DET>();
    constexpr int NW = NWREQ < NWMAX ? NWREQ : NWMAX;
    if constexpr (NW < 4) {
        return cudaErrorInvalidConfiguration;
    } else {
        constexpr size_t smem = tile_smem_bytes<T, SHAPE, B, NW, DET>();
        auto kern = push_batch_kernel<T, SHAPE, B, NW, DET>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(smem));
        if (e != cudaSuccess)
            return e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NW * 32, smem);
        if (e != cudaSuccess)
            return e;
        uint32_t grid = uint32_t(sm_count) * uint32_t(per_sm > 0 ? per_sm : 1);
        // the sparse bins first (one warp per bin; the dense ones listed), then the
        // dense ones
        e = cudaMemsetAsync(work, 0, kDenseList * sizeof(uint32_t), s);
        if (e != cudaSuccess)
            return e;
        auto sk = push_batch_sparse_kernel<T, SHAPE, B, DET>;
        int sp_per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&sp_per_sm, sk, kSparseWarps * 32, 0);
        if (e != cudaSuccess)
            return e;
        uint64_t sgrid = uint64_t(sm_count) * uint64_t(sp_per_sm > 0 ? sp_per_sm : 1);
        const uint64_t sgrid_max = (uint64_t(total_bins) + kSparseWarps - 1) / kSparseWarps;
        if (sgrid > sgrid_max)
            sgrid = sgrid_max > 0 ? sgrid_max : 1;
        sk<<<unsigned(sgrid), kSparseWarps * 32, 0, s>>>(a, boxes, n_boxes, bin_start, total_bins, work);
        kern<<<grid, NW * 32, smem, s>>>(a, boxes, n_boxes, bin_start, work);
        return cudaGetLastError();
    }
}

template <typename T>
cudaError_t push_batch_dispatch(const PushDesc &d, const void *boxes, int n_boxes,
                                uint32_t total_bins, int warps, uint32_t *work, cudaStream_t s)
{
    const PushArgs<T> a = make_push_args<T>(d);
    const BatchBox<T> *bx = static_cast<const BatchBox<T> *>(boxes);
    const bool det = d.det != 0;
    const bool w8 = warps == 8;
#define RSOL_BATCH(SH, BB)                                                                 \
    if (det)                                                                              \
        return w8 ? launch_batch<T, SH, BB, true, 8>(a, bx, n_boxes, d.bin_start, total_bins, work, d.sm_count, s) \
                  : launch_batch<T, SH, BB, true, 16>(a, bx, n_boxes, d.bin_start, total_bins, work, d.sm_count, s); \
    return w8 ? launch_batch<T, SH, BB, false, 8>(a, bx, n_boxes, d.bin_start, total_bins, work, d.sm_count, s) \
              : launch_batch<T, SH, BB, false, 16>(a, bx, n_boxes, d.bin_start, total_bins, work, d.sm_count, s)
    if (d.shape == 1) {
        if (d.bin == 4) { RSOL_BATCH(1, 4); }
        RSOL_BATCH(1, 8);
    }
    if (d.bin == 4) { RSOL_BATCH(2, 4); }
    RSOL_BATCH(2, 8);
#undef RSOL_BATCH
}

inline size_t batch_box_bytes(int precision)
{
    return precision == 32 ? sizeof(BatchBox<float>) : sizeof(BatchBox<double>);
}

template <typename T>
void fill_batch_box(void *dst, int nx, int ny, int nz, int nbx, int nby, int nbz, int64_t node_off,
                    uint32_t bin_base, double h, double adv, double qv, double c)
{
    BatchBox<T> b;
    b.nx = nx; b.ny = ny; b.nz = nz; b.nbx = nbx; b.nby = nby; b.nbz = nbz;
    b.node_off = node_off;
    b.bin_base = bin_base;
    b.k.h = T(h); b.k.adv = T(adv); b.k.qv = T(qv); b.k.c = T(c);
    *static_cast<BatchBox<T> *>(dst) = b;
}

} // namespace rsol
