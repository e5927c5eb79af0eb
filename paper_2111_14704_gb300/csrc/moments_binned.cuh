// State moments (Sec. 2 packet totals per unit volume: n, N m c u,
// N gamma m c^2, N q c beta) deposited with W at the current positions, for a
// packet set in the order rsol_sort wrote: one CTA per sort bin sums its
// packets into a shared-memory tile (bin + 2-node halo) and adds the tile to
// the grid once.  No field gather: the tile holds only the eight moments.
// FP32 (moments_octet_kernel): packets are read in memory order, their moments
// staged and deposited by stencil origin, as in the push (octets.cuh), into 32-bit
// fixed point with a scale from a bound on the packets (largest weight, largest
// |u|^2; |beta| < 1 bounds the current); the three momentum-density components,
// whose sums over isotropic packets cancel, also keep each addition's rounding
// remainder in three more planes.  FP64 (moments_binned_kernel): within a warp, runs
// of packets of equal stencil origin along the lanes are summed in registers by
// stencil-offset lanes before each shared-memory add.
#pragma once

#include <type_traits>

#include "push_binned.cuh"

namespace rsol {

template <int SHAPE, int B, int NW>
struct MomCfg {
    using T = double;
    static constexpr int NP = SHAPE == 1 ? 2 : 3;
    static constexpr int NS = NP * NP * NP;
    static constexpr int TE = B + 4;
    static constexpr int RS = TE + 1, PS = TE * RS + 1;  // strides that spread rows and planes
    static constexpr int TN = TE * PS;
    static constexpr int WS = NS == 27 ? 28 : NS;  // weight rows padded to 16-byte stores
    static constexpr int QO = 12;
    static constexpr size_t tile_bytes = size_t(TN) * 8 * sizeof(T);
    static constexpr size_t stage_words = 32 * (WS + QO);
    // origin keys and local visiting order of the bin's first KEYCAP packets
    static constexpr int KEYCAP = 4096;
    static constexpr size_t stage_bytes = size_t(NW) * stage_words * sizeof(T);
    static constexpr size_t smem_bytes = tile_bytes + stage_bytes + 2 * size_t(KEYCAP) * sizeof(uint16_t);
};

// The eight state moments of one packet (weight w, momentum u).
template <typename T>
__device__ __forceinline__ void state_moments(const MomArgs<T> &a, T w, const T u[3], T Q[8])
{
    const T g = Math<T>::sqrt(T(1) + dot3(u, u));
    const T N = w * a.inv_vol;
    Q[0] = N;
#pragma unroll
    for (int q = 0; q < 3; ++q)
        Q[1 + q] = N * a.mc * u[q];
    Q[4] = N * g * a.mc2;
    const T ig = Math<T>::div(T(1), g);
#pragma unroll
    for (int q = 0; q < 3; ++q)
        Q[5 + q] = N * a.qc * (u[q] * ig);
}

template <int SHAPE, int B, int NW>
__global__ void __launch_bounds__(NW * 32) moments_binned_kernel(MomArgs<double> a, BinGeom g)
{
    using T = double;
    using Cfg = MomCfg<SHAPE, B, NW>;
    constexpr int TE = Cfg::TE, RS = Cfg::RS, PS = Cfg::PS, TN = Cfg::TN;
    constexpr int NP = Cfg::NP, NS = Cfg::NS, WS = Cfg::WS, QO = Cfg::QO;
    extern __shared__ __align__(16) unsigned char smem[];
    T *sd = reinterpret_cast<T *>(smem);  // [q][slot]
    T *stage = reinterpret_cast<T *>(smem + Cfg::tile_bytes);
    uint16_t *s_key = reinterpret_cast<uint16_t *>(smem + Cfg::tile_bytes + Cfg::stage_bytes);
    uint16_t *s_perm = s_key + Cfg::KEYCAP;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T *sW = stage + warp * Cfg::stage_words;  // [32][WS]
    T *sQ = sW + 32 * WS;                     // [32][QO]

    const int bin = blockIdx.x;
    const int bx = bin % g.nbx, by = (bin / g.nbx) % g.nby, bz = bin / (g.nbx * g.nby);
    const uint32_t lo = g.bin_start[bin], hi = g.bin_start[bin + 1];
    if (lo >= hi)
        return;

    // the packet's own nodes in the global grid
    auto deposit_global = [&](int ix, int iy, int iz, const T wx[3], const T wy[3], const T wz[3],
                              int rx, int ry, int rz, const T Q[8]) {
        int kx[3], ky[3], kz[3];
        axis_nodes(ix, rx, a.nx, kx);
        axis_nodes(iy, ry, a.ny, ky);
        axis_nodes(iz, rz, a.nz, kz);
#pragma unroll
        for (int cz = 0; cz < NP; ++cz)
#pragma unroll
            for (int cy = 0; cy < NP; ++cy) {
                const T wyz = wy[cy] * wz[cz];
                const int64_t row = (int64_t(kz[cz]) * a.ny + ky[cy]) * a.nx;
#pragma unroll
                for (int cx = 0; cx < NP; ++cx)
                    red_node(a.grid + (row + kx[cx]) * 8, wx[cx] * wyz, Q);
            }
    };

    if (hi - lo <= sparse_sum_limit<B>()) {  // few packets: the tile would cost more than their atomics
        for (uint32_t j = lo + threadIdx.x; j < hi; j += blockDim.x) {
            const uint32_t c = a.cell[j];
            const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
            if (ix >= a.nx || iy >= a.ny || iz >= a.nz)
                continue;
            const T u[3] = {a.u0[j], a.u1[j], a.u2[j]};
            T Q[8], wx[3], wy[3], wz[3];
            state_moments(a, a.w[j], u, Q);
            const int rx = axis_weights<SHAPE>(a.off0[j], wx);
            const int ry = axis_weights<SHAPE>(a.off1[j], wy);
            const int rz = axis_weights<SHAPE>(a.off2[j], wz);
            deposit_global(ix, iy, iz, wx, wy, wz, rx, ry, rz, Q);
        }
        return;
    }
    const int ox = bx * B - 2, oy = by * B - 2, oz = bz * B - 2;
    for (int t = threadIdx.x; t < 8 * TN; t += blockDim.x)
        sd[t] = T(0);
    __shared__ int s_desc, s_sorted, s_out;
    if (threadIdx.x == 0) {
        s_desc = 0;
        s_sorted = 0;
    }
    __syncthreads();

    // packets drifted since the last global sort break the origin order; once
    // more than one in 32 does, a counting sort by stencil origin (local to the
    // CTA, as in the binned push) gives the order the runs below are taken in
    const uint32_t n_bin = hi - lo;
    const bool keep = n_bin <= uint32_t(Cfg::KEYCAP);  // origin keys kept for a local sort
    if (keep) {
        // origin histogram (packets per stencil origin) and order breaks
        int *hist = reinterpret_cast<int *>(sd);  // plane 0 of the zeroed tile
        int desc = 0;
        for (uint32_t rb = 0; rb < n_bin; rb += blockDim.x) {  // warp-uniform trip count
            const uint32_t r = rb + threadIdx.x;
            int key = TN;  // out of the tile or off the grid: last
            if (r < n_bin) {
                const uint32_t j = lo + r;
                key = origin_slot<SHAPE, TE, RS, PS, TN>(a.cell[j], a.off0[j], a.off1[j], a.off2[j], ox,
                                                         oy, oz, a.nx, a.ny, a.nz);
                if (key < TN)
                    atomicAdd(&hist[key], 1);
                s_key[r] = uint16_t(key);
            }
            const int prev = __shfl_up_sync(0xffffffffu, key, 1);
            desc += (lane > 0 && r < n_bin && key < prev) ? 1 : 0;
        }
        desc = __reduce_add_sync(0xffffffffu, desc);
        if (lane == 0 && desc)
            atomicAdd(&s_desc, desc);
        __syncthreads();
        if (s_desc * 32 > int(n_bin)) {
            int *cursor = reinterpret_cast<int *>(stage);  // free until the batches
            origin_cursors<NW, TN>(hist, cursor, &s_out);
            for (uint32_t r = threadIdx.x; r < n_bin; r += blockDim.x) {
                const int key = s_key[r];
                const int pos = key < TN ? atomicAdd(&cursor[key], 1) : atomicAdd(&s_out, 1);
                s_perm[pos] = uint16_t(r);
            }
            if (threadIdx.x == 0)
                s_sorted = 1;
        }
        __syncthreads();
        for (int t = threadIdx.x; t < TN; t += blockDim.x)
            hist[t] = 0;
        __syncthreads();
    }
    const bool use_perm = s_sorted != 0;

    // phase-2 lane role: stencil offset and quantity range [q0, q0 + 2 or 8)
    const int off_id = SHAPE == 1 ? (lane & 7) : (lane < 27 ? lane : 0);
    const bool p2_active = SHAPE == 1 ? true : lane < 27;
    const int pax = off_id % NP, pay = (off_id / NP) % NP, paz = off_id / (NP * NP);
    const int q0 = SHAPE == 1 ? 2 * (lane >> 3) : 0;
    const int lane_off = paz * PS + pay * RS + pax;
    constexpr int NQ_ = SHAPE == 1 ? 2 : 8;
    T acc[NQ_];
#pragma unroll
    for (int q = 0; q < NQ_; ++q)
        acc[q] = T(0);
    int carry_origin = -1;
    auto flush_acc = [&](int origin) {
        if (p2_active && origin >= 0) {
#pragma unroll
            for (int q = 0; q < NQ_; ++q) {
                atomicAdd(&sd[(q0 + q) * TN + origin + lane_off], acc[q]);
            }
        }
    };

    // each warp walks a contiguous slice of the bin (runs carry across batches)
    const uint32_t per_warp = ((n_bin + NW - 1) / NW + 31) & ~31u;
    const uint32_t w_lo = lo + per_warp * uint32_t(warp);
    const uint32_t w_hi = w_lo + per_warp < hi ? w_lo + per_warp : hi;
    // software pipeline: the packet of visiting position pos (base + lane) of
    // the next batch is loaded into registers while this batch is deposited
    uint32_t n_c = 0xFFFFFFFFu;
    T n_o[3] = {T(0), T(0), T(0)}, n_u[3] = {T(0), T(0), T(0)}, n_w = T(0);
    auto prefetch = [&](uint32_t pos) {
        n_c = 0xFFFFFFFFu;  // off the grid: nothing to deposit
        if (pos < w_hi) {
            const uint32_t j = use_perm ? lo + s_perm[pos - lo] : pos;
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
    prefetch(w_lo + uint32_t(lane));
    for (uint32_t base = w_lo; base < w_hi; base += 32) {
        const uint32_t c = n_c;
        const T f[3] = {n_o[0], n_o[1], n_o[2]};
        const T u[3] = {n_u[0], n_u[1], n_u[2]};
        const T wj = n_w;
        prefetch(base + 32 + uint32_t(lane));
        int staged = -1;
        {
            const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
            if (ix < a.nx && iy < a.ny && iz < a.nz) {
                T Q[8], wx[3], wy[3], wz[3];
                state_moments(a, wj, u, Q);
                int rx, ry, rz;
                const int jx = anchor_axis<SHAPE>(ix, f[0], a.nx, wx, rx);
                const int jy = anchor_axis<SHAPE>(iy, f[1], a.ny, wy, ry);
                const int jz = anchor_axis<SHAPE>(iz, f[2], a.nz, wz, rz);
                int lx = jx + rx - ox, ly = jy + ry - oy, lz = jz + rz - oz;
                lx += lx < 0 ? a.nx : 0;
                ly += ly < 0 ? a.ny : 0;
                lz += lz < 0 ? a.nz : 0;
                lx -= lx >= a.nx ? a.nx : 0;
                ly -= ly >= a.ny ? a.ny : 0;
                lz -= lz >= a.nz ? a.nz : 0;
                const bool in_tile = lx >= 0 && ly >= 0 && lz >= 0 && lx + NP <= TE &&
                                     ly + NP <= TE && lz + NP <= TE;
                if (in_tile) {
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
                    store_wrow<WS>(sW + lane * WS, Wk);
                    store_q8(sQ + lane * QO, Q);
                    staged = lz * PS + ly * RS + lx;
                } else {
                    deposit_global(jx, jy, jz, wx, wy, wz, rx, ry, rz, Q);
                }
            }
        }
        // runs of equal stencil origin along the lanes; a lane with no staged
        // packet (-1) starts a run that is skipped
        const int left = __shfl_up_sync(0xffffffffu, staged, 1);
        uint32_t st = __ballot_sync(0xffffffffu, lane == 0 || staged != left);
        __syncwarp();
        while (st) {  // warp-uniform: one run per pass, summed in registers
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

    // add the tile to the global grid (untouched nodes skipped)
    for (int t = threadIdx.x; t < TE * TE * TE; t += blockDim.x) {
        const int lx = t % TE, ly = (t / TE) % TE, lz = t / (TE * TE);
        const int slot = lz * PS + ly * RS + lx;
        const int64_t node =
            (int64_t(wrap_mod(oz + lz, a.nz)) * a.ny + wrap_mod(oy + ly, a.ny)) * a.nx +
            wrap_mod(ox + lx, a.nx);
        T v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            v[q] = sd[q * TN + slot];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (v[q] != T(0))
                atomicAdd(a.grid + node * 8 + q, v[q]);
    }
}

// FP32: the push's staged deposit (octets.cuh) without the push.
template <int SHAPE, int B>
struct MomOctCfg {
    using O = OctetCfg<SHAPE, B + 4, 2640, 32>;
    static constexpr int NW = 16, TE = B + 4, TT = O::TT;
    static constexpr int DTN = TT + 4;  // 2 DTN = 8 mod 32: value pairs on banks eight apart
    // Order of the moments: momentum and one current component as the first of each
    // pair, with planes 8..11 for their remainders, so that every lane of a flush
    // does the same work.
    static constexpr size_t tile_bytes = size_t(DTN) * 12 * sizeof(int);
    __host__ __device__ static constexpr int moment(int s) { return s % 2 ? (s == 1 ? 0 : (s == 3 ? 4 : (s + 7) / 2)) : (s == 6 ? 5 : s / 2 + 1); }
    static constexpr size_t smem_bytes = tile_bytes + O::stage_bytes + O::keep_bytes;
    static_assert(tile_bytes % 16 == 0, "16-byte accesses of the stage");
};

// One packet's moments into the global grid (sparse bins, packets that left the tile).
template <int SHAPE>
__device__ __noinline__ void moments_global(const MomArgs<float> &a, uint32_t j)
{
    constexpr int NP = SHAPE == 1 ? 2 : 3;
    const uint32_t c = a.cell[j];
    const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
    if (ix >= a.nx || iy >= a.ny || iz >= a.nz)
        return;
    const float u[3] = {a.u0[j], a.u1[j], a.u2[j]};
    float Q[8], wx[3], wy[3], wz[3];
    state_moments(a, a.w[j], u, Q);
    int kx[3], ky[3], kz[3];
    axis_nodes(ix, axis_weights<SHAPE>(a.off0[j], wx), a.nx, kx);
    axis_nodes(iy, axis_weights<SHAPE>(a.off1[j], wy), a.ny, ky);
    axis_nodes(iz, axis_weights<SHAPE>(a.off2[j], wz), a.nz, kz);
#pragma unroll
    for (int cz = 0; cz < NP; ++cz)
#pragma unroll
        for (int cy = 0; cy < NP; ++cy) {
            const float wyz = wy[cy] * wz[cz];
            const int64_t row = (int64_t(kz[cz]) * a.ny + ky[cy]) * a.nx;
#pragma unroll
            for (int cx = 0; cx < NP; ++cx)
                red_node(a.grid + (row + kx[cx]) * 8, wx[cx] * wyz, Q);
        }
}

// Bound like the push by the shared-memory pipe and by issue; 2^24 packets two steps
// after a sort, TSC: 1.42 -> 0.93 ms
// against the run walk it replaced (2^18 packets, 64^3: 70 -> 53 us).
template <int SHAPE, int B>
__global__ void __launch_bounds__(512) moments_octet_kernel(const __grid_constant__ MomArgs<float> a,
                                                            const __grid_constant__ BinGeom g)
{
    using Cfg = MomOctCfg<SHAPE, B>;
    using O = typename Cfg::O;
    constexpr int TE = Cfg::TE, TT = Cfg::TT, DTN = Cfg::DTN, NP = O::NP, NS = O::NS;
    constexpr int NW = Cfg::NW, NT = NW * 32;
    extern __shared__ __align__(16) unsigned char smem[];
    int *sd = reinterpret_cast<int *>(smem);
    unsigned char *stage = smem + Cfg::tile_bytes;
    const OctetMem<O> m(stage + O::stage_bytes, stage);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int bin = blockIdx.x;
    const int bx = bin % g.nbx, by = (bin / g.nbx) % g.nby, bz = bin / (g.nbx * g.nby);
    const uint32_t lo = g.bin_start[bin], hi = g.bin_start[bin + 1];
    if (lo >= hi)
        return;
    if (hi - lo <= sparse_cta_limit<SHAPE, B, false>()) {
        for (uint32_t j = lo + threadIdx.x; j < hi; j += NT)
            moments_global<SHAPE>(a, j);
        return;
    }
    const int ox = bx * B - 2, oy = by * B - 2, oz = bz * B - 2;
    __shared__ int s_axis[3 * TE];
    tile_axes<TE>(s_axis, ox, oy, oz, a.nx, a.ny, a.nz);
    octet_clear<O, NW>(m);
    for (int t = threadIdx.x; t < int(Cfg::tile_bytes / 16); t += NT)
        reinterpret_cast<int4 *>(sd)[t] = make_int4(0, 0, 0, 0);
    __syncthreads();

    __shared__ float s_scale[8], s_iscale[8], s_lo, s_ilo;  // s_lo: 2^bits kept of a remainder
    const int pair = lane & 3;
    // Rounding to an integer by adding 1.5 2^23 (|x| <= 2^22): conversions run at a
    // quarter of the rate of additions.
    constexpr float kRound = 12582912.f;
    auto flush = [&](int slot, f32x2 (&acc)[NS]) {
        int *p = sd + 2 * pair * DTN + slot, *rest = sd + (8 + pair) * DTN + slot;
        const float lo_scale = s_lo;
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const int off = (k / (NP * NP)) * TE * TE + ((k / NP) % NP) * TE + k % NP;
            float x, y;
            f2_unpack(acc[k], x, y);
            const float t = __fadd_rn(x, kRound);
            const float r = __fsub_rn(x, __fsub_rn(t, kRound));  // exact, |r| <= 1/2
            atomicAdd(p + off, __float_as_int(t) - __float_as_int(kRound));
            atomicAdd(rest + off, __float_as_int(__fmaf_rn(r, lo_scale, kRound)) - __float_as_int(kRound));
            atomicAdd(p + DTN + off, __float2int_rn(y));
        }
    };
    const uint32_t n_bin = hi - lo, n_chunks = (n_bin + O::CHUNK - 1) / O::CHUNK;
    uint32_t chunk = (n_bin + n_chunks - 1) / n_chunks;
    if (chunk >= uint32_t(NT) && n_bin - chunk / NT * NT * (n_chunks - 1) <= O::CHUNK)
        chunk = chunk / NT * NT;
#pragma unroll 1
    for (uint32_t c = 0; c < n_chunks; c += 2) {
        const uint32_t p_lo = lo + c * chunk;
        const uint32_t split = c + 1 < n_chunks ? p_lo + chunk : hi;
        const uint32_t p_hi = c + 2 < n_chunks ? split + chunk : hi;
        if (c > 0) {
            __syncthreads();  // the previous part's tile has been added and cleared
            octet_clear<O, NW>(m);
            __syncthreads();
        }
        // origin counts, origins and ranks; the largest weight and |u|^2; a sum that is 0
        // unless some packet's weight, |u|^2 or offset is not finite
        float wmax = 0.f, u2max = 0.f, nonfinite = 0.f;
        constexpr int U = 4;  // packets per thread per pass: all loads issued first
        for (uint32_t j0 = p_lo + threadIdx.x; j0 < p_hi; j0 += U * NT) {
            uint32_t cc[U];
            float f0[U], f1[U], f2[U], v0[U], v1[U], v2[U], ww[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + uint32_t(u) * NT;
                const bool ok = j < p_hi;
                cc[u] = ok ? a.cell[j] : 0xFFFFFFFFu;
                f0[u] = ok ? a.off0[j] : 0.f;
                f1[u] = ok ? a.off1[j] : 0.f;
                f2[u] = ok ? a.off2[j] : 0.f;
                v0[u] = ok ? a.u0[j] : 0.f;
                v1[u] = ok ? a.u1[j] : 0.f;
                v2[u] = ok ? a.u2[j] : 0.f;
                ww[u] = ok ? a.w[j] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = j0 + uint32_t(u) * NT;
                const float uu[3] = {v0[u], v1[u], v2[u]};
                const float uu2 = dot3(uu, uu);
                wmax = fmaxf(wmax, fabsf(ww[u]));
                u2max = fmaxf(u2max, uu2);
                nonfinite = __fmaf_rn(0.f, ((f0[u] + f1[u]) + f2[u]) + (fabsf(ww[u]) + uu2), nonfinite);
                const int ix = cell_x(cc[u]), iy = cell_y(cc[u]), iz = cell_z(cc[u]);
                const int lx = wrap_once(ix + first_node<SHAPE>(f0[u]) - ox, a.nx),
                          ly = wrap_once(iy + first_node<SHAPE>(f1[u]) - oy, a.ny),
                          lz = wrap_once(iz + first_node<SHAPE>(f2[u]) - oz, a.nz);
                const bool in = ix < a.nx && iy < a.ny && iz < a.nz && max(max(lx, ly), lz) <= TE - NP;
                const int key = in ? (lz * TE + ly) * TE + lx : TT;
                if (key < TT)
                    m.rank[j - p_lo] = uint16_t(atomicAdd(m.hist + (j >= split ? TT : 0) + key, 1));
                if (j < p_hi)
                    m.key[j - p_lo] = uint16_t(key);
            }
        }
        __syncthreads();
        float gmax = 0.f;
        auto bound_pass = [&](int pass) {
            weight_bound_pass<SHAPE, TE, TE, TE * TE>(
                pass, [&](int t) { return m.hist[t] + m.hist[TT + t]; }, m.scratch, gmax);
        };
        int noct[2];
        octet_order<O, NW>(m, int(split - p_lo), int(p_hi - p_lo), noct, bound_pass);
        // fixed-point scale 2^e per moment: (largest total weight of a node) x
        // (bound on one packet's moment) below 2^31 / 1.002, or 2^22 / 1.002 with a
        // plane for the remainders; bounds per packet:
        // n: w/dx^3;  momentum: n m c |u|_max;  energy: n m c^2 gamma_max;
        // current: n |q| c
        __shared__ float s_red[3][NW];
        float red[3] = {gmax, wmax, u2max};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                red[k] = fmaxf(red[k], __shfl_xor_sync(0xffffffffu, red[k], o));
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                s_red[k][warp] = red[k];
        __syncthreads();
        if (threadIdx.x < 8) {
            float gm = 0.f, wm = 0.f, um = 0.f;
            for (int w = 0; w < NW; ++w) {
                gm = fmaxf(gm, s_red[0][w]);
                wm = fmaxf(wm, s_red[1][w]);
                um = fmaxf(um, s_red[2][w]);
            }
            const int q = Cfg::moment(threadIdx.x), top = threadIdx.x % 2 ? 31 : 22;
            const float n1 = wm * fabsf(a.inv_vol);
            float bound = q == 0 ? n1
                        : q < 4  ? n1 * fabsf(a.mc) * sqrtf(um)
                        : q == 4 ? n1 * fabsf(a.mc2) * sqrtf(1.f + um)
                                 : n1 * fabsf(a.qc);
            bound *= gm > 1.f ? gm : 1.f;
            bound *= 1.002f;
            // a finite bound is at most 2^128, so e >= 22 - 128 and the values stay within
            // what the rounding by addition holds; 2^120 leaves both scales normal numbers
            int e = top - 1;
            if (bound > 0.f && isfinite(bound))
                e = top - int(ceilf(log2f(bound)));
            e = e > 120 ? 120 : e;
            if (!isfinite(bound))
                nonfinite = bound;
            s_scale[threadIdx.x] = ldexpf(1.0f, e);
            s_iscale[threadIdx.x] = ldexpf(1.0f, -e);
            if (threadIdx.x == 0) {
                // a remainder is at most 2^(k-1) units; a node receives at most one
                // per run, i.e. at most n of them: n 2^(k-1) < 2^30
                int k = 31 - int(ceilf(log2f(float(p_hi - p_lo) + 1.f)));
                k = k > 22 ? 22 : (k < 0 ? 0 : k);
                s_lo = ldexpf(1.0f, k);
                s_ilo = ldexpf(1.0f, -k);
            }
        }
        if (__syncthreads_or(nonfinite != 0.f)) {
            // no bound for the integers (a value that is not finite, or sums that may
            // leave the FP32 range): each packet to its own nodes, as in a sparse bin
            for (uint32_t j = p_lo + threadIdx.x; j < p_hi; j += NT)
                moments_global<SHAPE>(a, j);
            continue;
        }
#pragma unroll 1
        for (int ch = 0; ch < 2; ++ch) {
            const uint32_t c_lo = ch ? split : p_lo, c_hi = ch ? p_hi : split;
            if (c_lo >= c_hi)
                break;
            constexpr int V = 2;
            for (uint32_t j0 = c_lo + threadIdx.x; j0 < c_hi; j0 += V * NT) {
                float f[V][3], u[V][3], w[V];
                int place[V];
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    const uint32_t j = j0 + uint32_t(k) * NT;
                    place[k] = -1;
                    if (j < c_hi) {
                        place[k] = m.place[j - p_lo];
                        f[k][0] = a.off0[j];
                        f[k][1] = a.off1[j];
                        f[k][2] = a.off2[j];
                        u[k][0] = a.u0[j];
                        u[k][1] = a.u1[j];
                        u[k][2] = a.u2[j];
                        w[k] = a.w[j];
                    }
                }
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    if (place[k] == kOctNone) {
                        moments_global<SHAPE>(a, j0 + uint32_t(k) * NT);
                    } else if (place[k] >= 0) {
                        float M[8], Q[8];
                        state_moments(a, w[k], u[k], M);
#pragma unroll
                        for (int q = 0; q < 8; ++q)  // powers of two: exact
                            Q[q] = M[Cfg::moment(q)] * s_scale[q];
                        octet_stage<O>(m, place[k], octet_offset<SHAPE>(f[k][0]), octet_offset<SHAPE>(f[k][1]),
                                       octet_offset<SHAPE>(f[k][2]), Q);
                    }
                }
            }
            __syncthreads();
            octet_deposit<O, NW, true>(m, ch, noct[ch], flush);
            __syncthreads();  // the next chunk reuses the stage
        }
        // add the tile to the global grid (untouched nodes skipped)
        for (int t = threadIdx.x; t < TT; t += NT) {
            const int64_t node = s_axis[t % TE] + s_axis[TE + (t / TE) % TE] + s_axis[2 * TE + t / (TE * TE)];
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float x = float(sd[q * DTN + t]);
                sd[q * DTN + t] = 0;
                if (q % 2 == 0) {
                    x += float(sd[(8 + q / 2) * DTN + t]) * s_ilo;
                    sd[(8 + q / 2) * DTN + t] = 0;
                }
                v[Cfg::moment(q)] = x * s_iscale[q];
            }
            float *p = a.grid + node * 8;
            if (v[0] != 0.f || v[1] != 0.f || v[2] != 0.f || v[3] != 0.f)
                atomicAdd(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
            if (v[4] != 0.f || v[5] != 0.f || v[6] != 0.f || v[7] != 0.f)
                atomicAdd(reinterpret_cast<float4 *>(p + 4), make_float4(v[4], v[5], v[6], v[7]));
        }
    }
}

template <typename T, int SHAPE, int B>
cudaError_t launch_moments_binned(const MomArgs<T> &a, const BinGeom &g, int64_t nbins, cudaStream_t s)
{
    if constexpr (sizeof(T) == 4) {
        using Cfg = MomOctCfg<SHAPE, B>;
        static_assert(Cfg::smem_bytes <= 232448 - 1024, "moments tiles exceed shared memory");
        auto kern = moments_octet_kernel<SHAPE, B>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(Cfg::smem_bytes));
        if (e != cudaSuccess)
            return e;
        kern<<<unsigned(nbins), Cfg::NW * 32, Cfg::smem_bytes, s>>>(a, g);
        return cudaGetLastError();
    } else {
        constexpr int NW = B == 8 ? 8 : 16;  // 8^3 tiles: fewer warps fit
        using Cfg = MomCfg<SHAPE, B, NW>;
        static_assert(Cfg::smem_bytes <= 232448 - 1024, "moments tiles exceed shared memory");
        auto kern = moments_binned_kernel<SHAPE, B, NW>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(Cfg::smem_bytes));
        if (e != cudaSuccess)
            return e;
        kern<<<unsigned(nbins), NW * 32, Cfg::smem_bytes, s>>>(a, g);
        return cudaGetLastError();
    }
}

} // namespace rsol

namespace rsol {

template <typename T>
cudaError_t moments_binned_dispatch(const MomentsDesc &d, cudaStream_t s)
{
    MomArgs<T> a;
    a.n = d.n;
    a.cell = d.cell;
    a.off0 = static_cast<const T *>(d.off[0]);
    a.off1 = static_cast<const T *>(d.off[1]);
    a.off2 = static_cast<const T *>(d.off[2]);
    a.u0 = static_cast<const T *>(d.u[0]);
    a.u1 = static_cast<const T *>(d.u[1]);
    a.u2 = static_cast<const T *>(d.u[2]);
    a.w = static_cast<const T *>(d.w);
    a.grid = static_cast<T *>(d.grid);
    a.fx = nullptr;
    a.nx = d.nx;
    a.ny = d.ny;
    a.nz = d.nz;
    a.inv_vol = T(d.inv_vol);
    a.mc = T(d.mc);
    a.mc2 = T(d.mc2);
    a.qc = T(d.qc);
    a.fx_scale = T(0);
    BinGeom g;
    g.bin_start = d.bin_start;
    g.nbx = d.nbx;
    g.nby = d.nby;
    g.nbz = d.nbz;
    const int64_t nbins = int64_t(d.nbx) * d.nby * d.nbz;
    if (d.shape == 1)
        return d.bin == 4 ? launch_moments_binned<T, 1, 4>(a, g, nbins, s)
                          : launch_moments_binned<T, 1, 8>(a, g, nbins, s);
    return d.bin == 4 ? launch_moments_binned<T, 2, 4>(a, g, nbins, s)
                      : launch_moments_binned<T, 2, 8>(a, g, nbins, s);
}

} // namespace rsol

namespace rsol {

template <typename T>
struct LossBinArgs {
    int64_t n;
    const uint32_t *cell;
    const T *o0, *o1, *o2, *u0, *u1, *u2;
    T *w;
    const T *nn;
    T coef;
    int nx, ny, nz;
    int *status;
    BinGeom g;
};

// Catastrophic losses (Sec. 2) for the last sort's output with a gathered
// n_n: one CTA per bin stages the bin's n_n tile (bin + 2-node halo) in shared
// memory and gathers each packet's n_n from it; packets whose stencil left the
// tile read the grid.  Same arithmetic as losses_kernel.  Bound by the latency of the
// packets' loads and by issue: FP32 at 64 registers keeps four CTAs on an SM, with
// three packets per thread in flight (2^24 packets, TSC: 164 -> 146 us; four packets at
// 80 registers, three CTAs, was the former; two packets at 64 took 150 us, at 48
// registers with spills 183 us).
template <typename T, int SHAPE, int B>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) losses_binned_kernel(LossBinArgs<T> a)
{
    constexpr int NP = SHAPE == 1 ? 2 : 3;
    constexpr int TE = B + 4;
    __shared__ T tile[TE * TE * TE];
    const int bin = blockIdx.x;
    const int bx = bin % a.g.nbx, by = (bin / a.g.nbx) % a.g.nby, bz = bin / (a.g.nbx * a.g.nby);
    const uint32_t lo = a.g.bin_start[bin], hi = a.g.bin_start[bin + 1];
    if (lo >= hi)
        return;
    const int ox = bx * B - 2, oy = by * B - 2, oz = bz * B - 2;
    // grid offsets of the tile's rows along each axis (periodic)
    __shared__ int s_axis[3 * TE];
    if (threadIdx.x < 3 * TE) {
        const int ax = threadIdx.x / TE, l = threadIdx.x % TE;
        const int o = ax == 0 ? ox : (ax == 1 ? oy : oz);
        const int n = ax == 0 ? a.nx : (ax == 1 ? a.ny : a.nz);
        const int stride = ax == 0 ? 1 : (ax == 1 ? a.nx : a.nx * a.ny);
        s_axis[threadIdx.x] = wrap_mod(o + l, n) * stride;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < TE * TE * TE; t += blockDim.x) {
        const int lx = t % TE, ly = (t / TE) % TE, lz = t / (TE * TE);
        tile[t] = a.nn[s_axis[lx] + s_axis[TE + ly] + s_axis[2 * TE + lz]];
    }
    __syncthreads();
    int flag = 0;
    constexpr uint32_t NT = 256;
    constexpr int U = sizeof(T) == 4 ? 3 : 4;  // packets per thread per pass: their loads are issued first
    for (uint32_t jb = lo + threadIdx.x; jb < hi; jb += U * NT) {
        uint32_t cc[U];
        T f0[U], f1[U], f2[U], v0[U], v1[U], v2[U], ww[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const size_t j = size_t(jb) + k * NT;
            const bool ok = j < hi;
            cc[k] = ok ? a.cell[j] : 0xFFFFFFFFu;
            f0[k] = ok ? a.o0[j] : T(0);
            f1[k] = ok ? a.o1[j] : T(0);
            f2[k] = ok ? a.o2[j] : T(0);
            v0[k] = ok ? a.u0[j] : T(0);
            v1[k] = ok ? a.u1[j] : T(0);
            v2[k] = ok ? a.u2[j] : T(0);
            ww[k] = ok ? a.w[j] : T(0);
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const size_t j = size_t(jb) + k * NT;
            if (j >= hi)
                continue;
            const T u[3] = {v0[k], v1[k], v2[k]};
            const T uu = dot3(u, u);
            const T beta = Math<T>::sqrt(uu) * Math<T>::rsqrt(T(1) + uu);
            const uint32_t c = cc[k];
            const int ix = cell_x(c), iy = cell_y(c), iz = cell_z(c);
            if (ix >= a.nx || iy >= a.ny || iz >= a.nz) {
                flag |= ST_BADCELL;
                continue;
            }
            T wx[3], wy[3], wz[3];
            const int rx = axis_weights<SHAPE>(f0[k], wx);
            const int ry = axis_weights<SHAPE>(f1[k], wy);
            const int rz = axis_weights<SHAPE>(f2[k], wz);
            // first stencil node, tile-local (periodic)
            int lx = ix + rx - ox, ly = iy + ry - oy, lz = iz + rz - oz;
            lx += lx < 0 ? a.nx : 0;
            ly += ly < 0 ? a.ny : 0;
            lz += lz < 0 ? a.nz : 0;
            lx -= lx >= a.nx ? a.nx : 0;
            ly -= ly >= a.ny ? a.ny : 0;
            lz -= lz >= a.nz ? a.nz : 0;
            const bool in_tile = lx >= 0 && ly >= 0 && lz >= 0 && lx + NP <= TE && ly + NP <= TE &&
                                 lz + NP <= TE;
            T dens = T(0);
            if (in_tile) {  // separable: rows along x, then y, then z
                const T *t0 = tile + (lz * TE + ly) * TE + lx;
#pragma unroll
                for (int cz = 0; cz < NP; ++cz) {
                    T dz = T(0);
#pragma unroll
                    for (int cy = 0; cy < NP; ++cy) {
                        const T *row = t0 + (cz * TE + cy) * TE;
                        T dy = wx[0] * row[0];
#pragma unroll
                        for (int cx = 1; cx < NP; ++cx)
                            dy += wx[cx] * row[cx];
                        dz += wy[cy] * dy;
                    }
                    dens += wz[cz] * dz;
                }
            } else {
                int kx[3], ky[3], kz[3];
                axis_nodes(ix, rx, a.nx, kx);
                axis_nodes(iy, ry, a.ny, ky);
                axis_nodes(iz, rz, a.nz, kz);
#pragma unroll
                for (int cz = 0; cz < NP; ++cz)
#pragma unroll
                    for (int cy = 0; cy < NP; ++cy) {
                        const T wyz = wy[cy] * wz[cz];
                        const int64_t row = (int64_t(kz[cz]) * a.ny + ky[cy]) * a.nx;
#pragma unroll
                        for (int cx = 0; cx < NP; ++cx)
                            dens += wx[cx] * wyz * a.nn[row + kx[cx]];
                    }
            }
            a.w[j] = ww[k] * exp(-a.coef * beta * dens);
        }
    }
    if (flag)
        atomicOr(a.status, flag);
}

template <typename T>
cudaError_t losses_binned_dispatch(const LossDesc &d, cudaStream_t s)
{
    LossBinArgs<T> a;
    a.n = d.n;
    a.cell = d.cell;
    a.o0 = static_cast<const T *>(d.off[0]);
    a.o1 = static_cast<const T *>(d.off[1]);
    a.o2 = static_cast<const T *>(d.off[2]);
    a.u0 = static_cast<const T *>(d.u[0]);
    a.u1 = static_cast<const T *>(d.u[1]);
    a.u2 = static_cast<const T *>(d.u[2]);
    a.w = static_cast<T *>(d.w);
    a.nn = static_cast<const T *>(d.nn);
    a.coef = T(d.coef);
    a.nx = d.nx;
    a.ny = d.ny;
    a.nz = d.nz;
    a.status = d.status;
    a.g.bin_start = d.bin_start;
    a.g.nbx = d.nbx;
    a.g.nby = d.nby;
    a.g.nbz = d.nbz;
    const unsigned nbins = unsigned(int64_t(d.nbx) * d.nby * d.nbz);
    if (d.shape == 1) {
        if (d.bin == 4) losses_binned_kernel<T, 1, 4><<<nbins, 256, 0, s>>>(a);
        else losses_binned_kernel<T, 1, 8><<<nbins, 256, 0, s>>>(a);
    } else {
        if (d.bin == 4) losses_binned_kernel<T, 2, 4><<<nbins, 256, 0, s>>>(a);
        else losses_binned_kernel<T, 2, 8><<<nbins, 256, 0, s>>>(a);
    }
    return cudaGetLastError();
}

} // namespace rsol
