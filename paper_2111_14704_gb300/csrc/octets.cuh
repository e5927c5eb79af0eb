// Octet order: where a CTA of the tiled FP32 kernels stages the deposit of its
// packets, and the deposit that the order makes cheap.
//
// The CTA takes its bin in chunks, in memory order, so that the packet arrays
// are read and written coalesced however far the packets have drifted since
// the sort.  Each packet's eight values are staged in shared memory at a place
// that groups the chunk's packets by stencil origin (the first node of their
// stencil, a slot of the bin's tile): a run is up to 32 packets of one
// origin, the runs of a chunk are sorted by length and taken eight at a time,
// and such an octet is laid out in rows, row i holding the i-th packet of each
// of its runs.  Runs of an octet have nearly equal lengths, so few places of a
// row stay empty.  Runs of one length are dealt out by slot mod 8, so that the
// sums of an octet's eight origins mostly go to different banks.
//
// A warp deposits an octet with four lanes per run, a pair of the eight values
// each, and a register accumulator per stencil node and pair: a row (eight
// packets) is an 8-byte load of values and three 4-byte loads of offsets per
// lane, from which the lane forms the weights, and a run reaches the shared
// tile once.  A deposit with a lane per stencil node, one run at a time, loads
// 36 bytes per lane and packet and is bound by the shared-memory pipe.
#pragma once

#include <cstdint>

#include "rsol_device.cuh"

namespace rsol {

constexpr uint16_t kOctNone = 0xFFFF;  // packet not in the tile; no run

// PLACES: staged places of a chunk; RUN: packets of one run
template <int SHAPE_, int TE_, int PLACES_, int RUN_>
struct OctetCfg {
    static constexpr int SHAPE = SHAPE_, TE = TE_, PLACES = PLACES_, RUN = RUN_;
    // packets of a chunk: its octets' (longest - shortest) add up to less than
    // RUN rows of empty places, and its last octet may lack runs
    static constexpr int CHUNK = PLACES - 8 * (2 * RUN - 1);
    static constexpr int KEYS = 2 * CHUNK;  // packets ordered at a time: two chunks
    static constexpr int NP = SHAPE == 1 ? 2 : 3;
    static constexpr int NS = NP * NP * NP;
    static constexpr int TT = TE * TE * TE;         // tile slots: (z TE + y) TE + x
    static_assert(TT < 2047, "a run holds its slot in 11 bits");
    static constexpr int OE = TE - NP + 1;          // stencil origins per axis
    static constexpr int NORG = OE * OE * OE;
    static constexpr int NCLS = RUN * 8;        // (run length, slot mod 8) classes
    // runs of a chunk: at most one remainder per origin, plus full runs
    static constexpr int NRUN = (NORG + CHUNK / RUN + 7) & ~7;
    static constexpr int NOCT = NRUN / 8;
    // kept while the two chunks are pushed: places, runs, octets' first rows
    static constexpr size_t place_bytes = (size_t(KEYS) * 2 + 15) & ~size_t(15);
    static constexpr size_t keep_bytes = place_bytes + 2 * size_t(NRUN) * 2 + 2 * size_t(NOCT) * 2;
    // staging: values [place][8], then offsets along x, y, z [place]
    static constexpr size_t stage_bytes = size_t(PLACES) * 11 * sizeof(float);
    // until the order is made, in the staging area
    static constexpr size_t temp_bytes = 2 * size_t(NCLS) * 4 + 2 * size_t(TT) * 4 + 2 * size_t(TT) * 4 +
                                         2 * size_t(TT) * 4 + 2 * size_t(KEYS) * 2;
    static_assert(temp_bytes <= stage_bytes, "the order's temporaries share the staging area");
};

template <typename Cfg>
struct OctetMem {
    using C = Cfg;
    // kept
    uint16_t *place;  // [C::KEYS] staged place of a packet of its chunk, or kOctNone
    uint16_t *run;    // [2][NRUN] slot | (length - 1) << 11, or kOctNone
    uint16_t *first;  // [2][NOCT] first row of an octet
    // staging
    float *q;         // [place][8]
    float *d;         // [3][place]
    // temporaries
    int *cls;         // [2][NCLS] runs of length C::RUN - (t >> 3) and slot residue t & 7
    int *hist;        // [2][TT] packets per origin
    uint32_t *runs;   // [2][TT] an origin's runs: remainder run | rank of the first full run
                      // in its class << 11 | number of full runs << 19
    float *scratch;   // [2 TT]
    uint16_t *key;    // [C::KEYS] origin slot of a packet; TT: not in the tile
    uint16_t *rank;   // [C::KEYS] its rank within the origin and chunk
    __device__ __forceinline__ OctetMem(unsigned char *keep, unsigned char *stage)
    {
        place = reinterpret_cast<uint16_t *>(keep);
        run = reinterpret_cast<uint16_t *>(keep + C::place_bytes);
        first = run + 2 * C::NRUN;
        q = reinterpret_cast<float *>(stage);
        d = q + size_t(C::PLACES) * 8;
        cls = reinterpret_cast<int *>(stage);
        hist = cls + 2 * C::NCLS;
        runs = reinterpret_cast<uint32_t *>(hist + 2 * C::TT);
        scratch = reinterpret_cast<float *>(runs + 2 * C::TT);
        key = reinterpret_cast<uint16_t *>(scratch + 2 * C::TT);
        rank = key + C::KEYS;
    }
};

// Place within its length class of the run of residue r and rank k among the
// class's runs of that residue: the residues are dealt out in turn.
__device__ __forceinline__ int octet_deal(const int *cls, int r, int k)
{
    const int4 a = reinterpret_cast<const int4 *>(cls)[0], b = reinterpret_cast<const int4 *>(cls)[1];
    const int c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    int p = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i)
        p += min(c[i], k) + (i < r && c[i] > k ? 1 : 0);
    return p;
}

// Clear what the counting and ordering of a part add to; before a barrier.
template <typename C, int NW>
__device__ __forceinline__ void octet_clear(const OctetMem<C> &m)
{
    for (int t = threadIdx.x; t < 2 * (C::NCLS + C::TT); t += NW * 32)  // cls, then hist
        m.cls[t] = 0;
    for (int t = threadIdx.x; t < C::NRUN; t += NW * 32)  // both chunks' runs, two at a time
        reinterpret_cast<uint32_t *>(m.run)[t] = 0xFFFFFFFFu;
}

// Ranks by packet index: the counters give a packet any rank within its origin
// and chunk; this gives it the number of earlier packets there, so that the
// order of every sum is that of the packets.  Each packet counts the earlier ones
// in its origin's list (a few, unless most packets crowd into few cells).
// Starts and ends synchronised.
template <typename C, int NW>
__device__ __forceinline__ void octet_stable_ranks(const OctetMem<C> &m, int n0, int n)
{
    constexpr int NT = NW * 32, N2 = 2 * C::TT, PER = (N2 + NT - 1) / NT;
    __shared__ int s_wsum[NW];
    uint32_t *at = m.runs;                                       // [N2] first list position of an origin
    uint16_t *list = reinterpret_cast<uint16_t *>(m.scratch);    // [KEYS]
    static_assert(size_t(C::KEYS) * 2 <= 2 * size_t(C::TT) * sizeof(float), "the lists fit the scratch");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int v[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int t = tid * PER + i;
        v[i] = t < N2 ? m.hist[t] : 0;
        sum += v[i];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        incl += lane >= o ? y : 0;
    }
    if (lane == 31)
        s_wsum[warp] = incl;
    __syncthreads();
    int run = incl - sum;
    for (int w = 0; w < warp; ++w)
        run += s_wsum[w];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int t = tid * PER + i;
        if (t < N2)
            at[t] = uint32_t(run);
        run += v[i];
    }
    __syncthreads();
    for (int r = tid; r < n; r += NT)
        if (m.key[r] < C::TT)
            list[at[(r >= n0 ? C::TT : 0) + m.key[r]] + m.rank[r]] = uint16_t(r);
    __syncthreads();
    for (int r = tid; r < n; r += NT)
        if (m.key[r] < C::TT) {
            const int t = (r >= n0 ? C::TT : 0) + m.key[r];
            const int lo = int(at[t]), c = m.hist[t];
            int before = 0;
            for (int k = 0; k < c; ++k)
                before += list[lo + k] < r ? 1 : 0;
            m.rank[r] = uint16_t(before);
        }
    __syncthreads();
}

// The octet order of n packets, the first n0 of them chunk 0 (n0, n - n0 <=
// C::CHUNK), from m.hist, m.key and m.rank.  Fills m.place, m.run and m.first;
// returns the octets of each chunk in noct.  Starts and ends synchronised.
// meanwhile(0), (1) and (2) are called, by all threads, between its barriers.
template <typename C, int NW, typename Meanwhile>
__device__ __forceinline__ void octet_order(const OctetMem<C> &m, int n0, int n, int (&noct)[2],
                                            Meanwhile meanwhile)
{
    constexpr int TE = C::TE;
    constexpr int NT = NW * 32;
    constexpr int PER = (2 * C::NORG + NT - 1) / NT;  // (chunk, origin) pairs per thread
    __shared__ int s_runs[2];
    __shared__ uint16_t s_cbase[2][C::RUN];          // first run of each length class
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // each origin's runs into classes: length (longest first), residue
    int slot[PER], cnt[PER], rk[PER], rf[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int o2 = tid + i * NT;
        cnt[i] = 0;
        if (o2 < 2 * C::NORG) {
            const int ch = o2 >= C::NORG, o = o2 - ch * C::NORG;
            const int x = o % C::OE, y = (o / C::OE) % C::OE, z = o / (C::OE * C::OE);
            slot[i] = ch * C::TT + (z * TE + y) * TE + x;
            cnt[i] = m.hist[slot[i]];
            int *cls = m.cls + ch * C::NCLS;
            const int nf = cnt[i] / C::RUN, rem = cnt[i] % C::RUN;
            rf[i] = nf ? atomicAdd(&cls[slot[i] & 7], nf) : 0;
            if (rem)
                rk[i] = atomicAdd(&cls[(C::RUN - rem) * 8 + (slot[i] & 7)], 1);
        }
    }
    meanwhile(0);
    __syncthreads();
    static_assert(C::TT % 8 == 0 && NW >= 2 && C::RUN <= 32, "residues of both chunks; a warp per chunk");
    static_assert(C::NRUN <= 2048 && C::CHUNK / C::RUN < 256, "fields of runs");
    if (warp < 2) {  // chunk `warp`, a lane per length class: runs of the class, and their prefix
        int sum = 0;
        if (lane < C::RUN)
#pragma unroll
            for (int r = 0; r < 8; ++r)
                sum += m.cls[warp * C::NCLS + lane * 8 + r];
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            incl += lane >= o ? y : 0;
        }
        if (lane < C::RUN)
            s_cbase[warp][lane] = uint16_t(incl - sum);
        if (lane == 31)
            s_runs[warp] = incl;
    }
    meanwhile(1);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (cnt[i]) {
            const int ch = slot[i] >= C::TT, sl = slot[i] - ch * C::TT;
            const int *cls = m.cls + ch * C::NCLS;
            uint16_t *run = m.run + ch * C::NRUN;
            const int nf = cnt[i] / C::RUN, rem = cnt[i] % C::RUN;
            for (int f = 0; f < nf; ++f)
                run[octet_deal(cls, sl & 7, rf[i] + f)] = uint16_t(sl | (C::RUN - 1) << 11);
            uint32_t last = 0;
            if (rem) {
                const int cl = C::RUN - rem;
                last = uint32_t(s_cbase[ch][cl] + octet_deal(cls + cl * 8, sl & 7, rk[i]));
                run[last] = uint16_t(sl | (rem - 1) << 11);
            }
            m.runs[slot[i]] = last | uint32_t(rf[i]) << 11 | uint32_t(nf) << 19;
        }
    meanwhile(2);
    __syncthreads();
    if (warp < 2) {  // rows of each octet of chunk `warp` (its first run is the longest), and their prefix
        constexpr int E = (C::NOCT + 31) / 32;
        const uint16_t *run = m.run + warp * C::NRUN;
        int rows[E], sum = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = lane * E + e;
            const uint16_t r = o < C::NOCT ? run[8 * o] : kOctNone;
            rows[e] = r == kOctNone ? 0 : (r >> 11) + 1;
            sum += rows[e];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            incl += lane >= o ? y : 0;
        }
        int row = incl - sum;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int o = lane * E + e;
            if (o < C::NOCT)
                m.first[warp * C::NOCT + o] = uint16_t(row);
            row += rows[e];
        }
    }
    __syncthreads();
    for (int r = tid; r < n; r += NT) {
        const int ch = r >= n0, sl = m.key[r], key = ch * C::TT + sl;
        int p = kOctNone;
        if (sl < C::TT) {
            const int rank = m.rank[r], row = rank % C::RUN;
            const uint32_t e = m.runs[key];
            int run = int(e & 2047u);
            if (rank < int(e >> 19) * C::RUN)  // in one of the origin's full runs
                run = octet_deal(m.cls + ch * C::NCLS, sl & 7, int(e >> 11 & 255u) + rank / C::RUN);
            // the eight places of a row are rotated by the row, so that a run's
            // packets, neighbours in memory, are staged to different banks
            p = (m.first[ch * C::NOCT + (run >> 3)] + row) * 8 + ((run + row) & 7);
        }
        m.place[r] = uint16_t(p);
    }
    noct[0] = (s_runs[0] + 7) >> 3;
    noct[1] = (s_runs[1] + 7) >> 3;
    __syncthreads();
}

// Stage the values Q and the one-axis positions of a packet (see octet_offset).
template <typename C>
__device__ __forceinline__ void octet_stage(const OctetMem<C> &m, int place, float dx, float dy,
                                            float dz, const float Q[8])
{
    float4 *q = reinterpret_cast<float4 *>(m.q + place * 8);
    q[0] = make_float4(Q[0], Q[1], Q[2], Q[3]);
    q[1] = make_float4(Q[4], Q[5], Q[6], Q[7]);
    m.d[place] = dx;
    m.d[C::PLACES + place] = dy;
    m.d[2 * C::PLACES + place] = dz;
}

// The staged position along one axis, from which axis_weights follow: the
// offset itself (CIC), or the distance from the nearest node (TSC).
template <int SHAPE>
__device__ __forceinline__ float octet_offset(float f)
{
    return SHAPE == 1 ? f : (f >= 0.5f ? f - 1.f : f);
}
template <int SHAPE>
__device__ __forceinline__ void octet_weights(float d, float w[3])
{
    if (SHAPE == 1) {
        w[0] = 1.f - d;
        w[1] = d;
    } else {
        const float a = 0.5f - d, b = 0.5f + d;
        w[0] = 0.5f * a * a;
        w[1] = 0.75f - d * d;
        w[2] = 0.5f * b * b;
    }
}

// Deposit of a staged chunk: warp w takes octets w, w + NW, ... (the longest
// first, so the warps' shares even out); each run's sums go to
// flush(origin slot, acc), four lanes a run, lane & 3 the pair of values.
template <typename C, int NW, bool MERGE, typename Flush>
__device__ __forceinline__ void octet_deposit(const OctetMem<C> &m, int chunk, int noct, Flush flush)
{
    constexpr int SHAPE = C::SHAPE, NP = C::NP;
    const int lane = threadIdx.x & 31, g = lane >> 2, pair = lane & 3;
    for (int o = threadIdx.x >> 5; o < noct; o += NW) {  // warp-uniform
        const uint32_t e = m.run[chunk * C::NRUN + 8 * o + g];
        const int mine = e == kOctNone ? 0 : int(e >> 11) + 1;
        const int rows = __shfl_sync(0xffffffffu, mine, 0);
        const int p0 = m.first[chunk * C::NOCT + o] * 8;
        f32x2 acc[C::NS];
#pragma unroll
        for (int k = 0; k < C::NS; ++k)
            acc[k] = 0;  // +0.0f in both halves
        float n_d[3];
        f32x2 n_Q;
        auto load = [&](int r) {  // the next row's loads are issued before this row's sums
            const int p = p0 + r * 8 + ((g + r) & 7);
            n_d[0] = n_d[1] = n_d[2] = 0.f;
            n_Q = 0;
            if (r < mine) {  // an empty place was never written
                n_d[0] = m.d[p];
                n_d[1] = m.d[C::PLACES + p];
                n_d[2] = m.d[2 * C::PLACES + p];
                n_Q = *reinterpret_cast<const f32x2 *>(m.q + p * 8 + 2 * pair);
            }
        };
        load(0);
#pragma unroll 1
        for (int r = 0; r < rows; ++r) {
            const float d[3] = {n_d[0], n_d[1], n_d[2]};
            const f32x2 Q2 = n_Q;
            load(r + 1);
            float wx[3], wy[3], wz[3];
            octet_weights<SHAPE>(d[0], wx);
            octet_weights<SHAPE>(d[1], wy);
            octet_weights<SHAPE>(d[2], wz);
            f32x2 c[NP];
#pragma unroll
            for (int x = 0; x < NP; ++x)
                c[x] = f2_mul(f2_pack(wx[x], wx[x]), Q2);
#pragma unroll
            for (int k = 0; k < NP * NP; ++k) {
                const float w = wy[k % NP] * wz[k / NP];
                const f32x2 w2 = f2_pack(w, w);
#pragma unroll
                for (int x = 0; x < NP; ++x)
                    acc[k * NP + x] = f2_fma(w2, c[x], acc[k * NP + x]);
            }
        }
        // eight runs of one origin (packets crowded into a cell): one sum, so that a
        // fixed-point tile rounds once for all of them (not where every sum has to be
        // the same from run to run: which runs meet in an octet may differ)
        const uint32_t e0 = __shfl_sync(0xffffffffu, e, 0);
        if (MERGE && __all_sync(0xffffffffu, e != kOctNone && ((e ^ e0) & 2047u) == 0)) {
#pragma unroll
            for (int k = 0; k < C::NS; ++k) {
                float x, y;
                f2_unpack(acc[k], x, y);
#pragma unroll
                for (int s = 4; s < 32; s <<= 1) {
                    x += __shfl_xor_sync(0xffffffffu, x, s);
                    y += __shfl_xor_sync(0xffffffffu, y, s);
                }
                acc[k] = f2_pack(x, y);
            }
            if (g == 0)
                flush(int(e & 2047u), acc);
        } else if (mine) {
            flush(int(e & 2047u), acc);
        }
    }
}

} // namespace rsol
