// gather.cuh -- the neighbour sums S_h(v) = sum over the neighbours u of v
// of c_h(u) (the inner sum over u of Eq. 1), the kernel shared by the
// translation units that instantiate it (gather_*.cu) and the table build.
#pragma once

#include "internal.h"

namespace mc {

enum : int { ERR_OVERFLOW = 1, ERR_INEXACT = 2, ERR_COLOUR = 4, ERR_SEARCH = 8 };

// ---------------------------------------------------------------------------
// Neighbour sums of level h >= 2 (the inner sum over u of Eq. 1):
//   S_h(v)[rho'', s] = sum_{u ~ v} c_h(u)[map(c_v, c_u, rho''), s].
// Rows are set-major, so the entries of one colour set (all r_h shapes) are
// contiguous, and a neighbour u contributes whole sets: the S sets holding
// c_u take u's sets that avoid c_v.  Only the first plane of a row is read
// (the low N bytes of its counts, common.cuh), in units of UB bytes: the
// widest of 16, 8, 4 that divides a set's bytes.  A lane owns the S units
// j, j + G, ... of its node and, per neighbour, loads the one source unit that
// feeds each (its offset from a map in shared memory), U neighbours in flight.
// Narrow rows (G < 8) take P neighbours of the node at once.  The G P lanes of
// a node load the ids and colours of as many neighbours together and hand
// them round by shuffles; the next ids are loaded while the rows are in
// flight.  Up to
// 64 low parts add up in 64 bits (N = 4) or 64 + 32 bits (N = 8) without a
// check.  If the level has wide rows at all, nodes with a wide neighbour add
// the upper parts in a second pass over those neighbours, exactly.
//   * nodes of degree <= HUB_CHUNK: G P lanes per node, 32 / (G P) nodes per
//     warp, taken in the order of `sched` (descending degree, so the nodes of a
//     warp have nearly equal degrees);
//   * hub chunks (HUB_CHUNK consecutive neighbours of a hub): a warp per
//     chunk, its 32 / G groups on different neighbours, summed by shuffles;
//     the partial row goes to `partial`, entry-major per hub.
// The first `chunk_blocks` blocks take the hub chunks, the rest the nodes.
// Bound by scattered reads from L2 and DRAM (k <= 6) and by instruction issue
// (k = 8).  Against reading whole 8- or 16-byte counts, ms per level: h = 2..6
// of R-MAT 22, k = 7, 128 bits 4.6 / 13.6 / 15.9 / 17.2 / 8.1 before, 2.1 / 4.6
// / 8.2 / 11.2 / 6.9 now; h = 2..7 of Chung-Lu 2M, k = 8 2.6 / 9.5 / 19.3 /
// 22.3 / 19.8 / 5.3 before, 1.4 / 2.9 / 7.2 / 10.0 / 8.2 / 3.4 now; h = 2..4 of
// Chung-Lu 1M, k = 5, 64 bits 0.26 / 0.27 / 0.21 before, 0.20 / 0.20 / 0.24
// now.
// ---------------------------------------------------------------------------
struct GatherArgs {
    const int64_t *row_ptr;
    const uint32_t *col;
    const uint8_t *colors;
    const uint8_t *ecol;
    const uint4 *sched;      // nodes of degree <= HUB_CHUNK, descending degree: (v, e0 lo, e0 hi, degree)
    int64_t n_small;
    const int32_t *node_chunk0;
    Rows src, dst;           // c_h, S_h
    void *partial;           // n_chunks x Ws counts
    const uint32_t *chunk_node;
    const int64_t *chunk_e0, *chunk_e1;
    const int16_t *gmap;
    int64_t n, nnz, n_chunks;
    int k, Bs;
    int ups;                 // units per colour set
    int ws_units;
    uint32_t *levels;        // the levels that have a wide row
    int chunk_blocks;
    int *err;
};

// UB bytes of a row's first plane: EPU counts of N bytes.
template <int N, int UB> struct Unit {
    static constexpr int EPU = UB / N;
    uint32_t w[UB / 4];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < UB / 4; ++i) w[i] = 0;
    }
    __device__ __forceinline__ void load(const uint8_t *p)
    {
        if constexpr (UB == 4) {
            w[0] = __ldg((const unsigned *)p);
        } else if constexpr (UB == 8) {
            const uint2 v = __ldg((const uint2 *)p);
            w[0] = v.x; w[1] = v.y;
        } else {
            const uint4 v = __ldg((const uint4 *)p);
            w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
        }
    }
    __device__ __forceinline__ uint64_t at(int e) const
    {
        if constexpr (N == 4) return w[e];
        else return ((uint64_t)w[2 * e + 1] << 32) | w[2 * e];
    }
};

// Sums of at most 64 first-plane counts: exact in 64 bits (N = 4) or 96
// (N = 8 of 128-bit counts); whole 64-bit counts (N = 8 of 64-bit ones) are
// checked.
template <typename CT, int N> struct LowSum {
    uint64_t lo;
    uint32_t hi;
    __device__ __forceinline__ void zero() { lo = 0; hi = 0; }
    __device__ __forceinline__ void add(uint64_t x)
    {
        lo += x;
        if constexpr (N == 8) hi += lo < x;
    }
    __device__ __forceinline__ void add_lane(int d)
    {
        const uint32_t h = N == 8 ? __shfl_xor_sync(0xffffffffu, hi, d) : 0u;
        add(__shfl_xor_sync(0xffffffffu, lo, d));
        hi += h;
    }
    __device__ __forceinline__ CT value(bool &ovf) const
    {
        if constexpr (sizeof(CT) == 16) return ((CT)(N == 8 ? hi : 0u) << 64) | lo;
        if constexpr (N == 8) ovf |= hi != 0;
        return (CT)lo;
    }
};

// The EPU low parts of a unit to its place in a first plane of nb-byte counts.
template <int EPU, typename CT> __device__ __forceinline__ void store_low(uint8_t *p, const CT *x, int nb)
{
    if (nb == 4) {
        if constexpr (EPU == 1) *(uint32_t *)p = (uint32_t)x[0];
        else if constexpr (EPU == 2) *(uint2 *)p = make_uint2((uint32_t)x[0], (uint32_t)x[1]);
        else *(uint4 *)p = make_uint4((uint32_t)x[0], (uint32_t)x[1], (uint32_t)x[2], (uint32_t)x[3]);
    } else {
        if constexpr (EPU == 1) *(uint64_t *)p = (uint64_t)x[0];
        else
#pragma unroll
            for (int i = 0; i < EPU; i += 2)
                *(ulonglong2 *)(p + 8 * i) = make_ulonglong2((uint64_t)x[i], (uint64_t)x[i + 1]);
    }
}

template <typename CT, int N, int UB, int G, int NU, int P, int U, int MB>
__global__ void __launch_bounds__(256, MB) gather_kernel(const __grid_constant__ GatherArgs a)
{
    // s_map[(c_v k + c_u) G NU + unit]: byte offset of the source unit in a
    // first-plane row of colour c_u, -1: none (also for the unit numbers past
    // the row's)
    extern __shared__ int16_t s_map[];
    for (int i = threadIdx.x; i < a.k * a.k * G * NU; i += blockDim.x) {
        const int cc = i / (G * NU), un = i - cc * (G * NU), set = un / a.ups;
        const int m = un < a.ws_units ? (int)a.gmap[cc * a.Bs + set] : -1;
        s_map[i] = (int16_t)(m < 0 ? -1 : (m * a.ups + (un - set * a.ups)) * UB);
    }
    __syncthreads();

    typedef Unit<N, UB> UT;
    constexpr int EPU = UT::EPU;
    constexpr int GW = G * P, NG = 32 / GW;  // lanes per node, nodes per warp
    const int lane = threadIdx.x & 31;
    const int grp = lane / GW, j = lane % G, par = lane % GW / G;
    const uint8_t *__restrict__ src = a.src.p0;
    const uint32_t stride = (uint32_t)a.src.s0;
    const int wpb = blockDim.x >> 5;
    const uint32_t *wide_of = a.src.wide;
    const uint32_t c_bit = a.src.bit;
    const bool lw = (*a.levels & c_bit) != 0;
    bool ovf = false, any_wide = false;
    LowSum<CT, N> acc[NU][EPU];

    auto fetch = [&](UT *x, uint32_t id, const int16_t *map) {
        const uint8_t *row = src + (uint64_t)id * stride;
#pragma unroll
        for (int i = 0; i < NU; ++i) {
            const int off = map[j + i * G];
            if (off >= 0) x[i].load(row + off);
            else x[i].zero();
        }
    };
    auto add = [&](const UT *x) {
#pragma unroll
        for (int i = 0; i < NU; ++i)
#pragma unroll
            for (int w = 0; w < EPU; ++w) acc[i][w].add(x[i].at(w));
    };
    auto clear = [&] {
#pragma unroll
        for (int i = 0; i < NU; ++i)
#pragma unroll
            for (int w = 0; w < EPU; ++w) acc[i][w].zero();
    };
    // the lanes with the same unit in `width` lanes add up
    auto reduce = [&](int width) {
        for (int d = G; d < width; d <<= 1)
#pragma unroll
            for (int i = 0; i < NU; ++i)
#pragma unroll
                for (int w = 0; w < EPU; ++w) acc[i][w].add_lane(d);
    };
    // the upper parts of the wide rows among neighbours [e0, e1)
    auto add_wide = [&](CT(*tot)[EPU], int64_t e0, int64_t e1, int cv) {
        for (int64_t e = e0; e < e1; ++e) {
            const uint32_t id = a.col[e];
            const int cu = a.ecol[e];
            if (cu == cv || !(wide_of[id] & c_bit)) continue;
            const uint8_t *high = a.src.high(id);
            const int16_t *map = s_map + (cv * a.k + cu) * (G * NU);
            for (int i = 0; i < NU; ++i) {
                const int off = map[j + i * G];
                if (off < 0) continue;
                for (int w = 0; w < EPU; ++w) ovf |= add_ovf(tot[i][w], row_rest<CT>(high, a.src.W, N, off / N + w));
            }
        }
    };

    if ((int)blockIdx.x < a.chunk_blocks) {
        // ---- hub chunks: a warp per chunk, its 32 / G groups on different neighbours
        constexpr int HG = 32 / G;
        constexpr int UC = U < G ? U : G;  // neighbours in flight per group: HG * UC <= 32
        const int hgrp = lane / G;
        for (int64_t t = (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5); t < a.n_chunks;
             t += (int64_t)a.chunk_blocks * wpb) {
            const int64_t v = a.chunk_node[t];
            const int64_t e0 = a.chunk_e0[t];
            const int cnt = (int)(a.chunk_e1[t] - e0);
            const int cv = a.colors[v];
            const int16_t *mapv = s_map + cv * a.k * (G * NU);
            bool near_wide = false;
            clear();
            uint32_t id[2];
            int cb[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const bool in = 32 * r + lane < cnt;
                id[r] = in ? a.col[e0 + 32 * r + lane] : 0u;
                const int cu = in ? (int)a.ecol[e0 + 32 * r + lane] : cv;
                cb[r] = cu * (G * NU);
                if (lw && cu != cv) near_wide |= (wide_of[id[r]] & c_bit) != 0;
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
                for (int b = 0; b < 32 && 32 * r + b < cnt; b += HG * UC) {
                    UT x[UC][NU];
#pragma unroll
                    for (int q = 0; q < UC; ++q) {
                        const int p = b + q * HG + hgrp;
                        fetch(x[q], __shfl_sync(0xffffffffu, id[r], p), mapv + __shfl_sync(0xffffffffu, cb[r], p));
                    }
#pragma unroll
                    for (int q = 0; q < UC; ++q) add(x[q]);
                }
            reduce(32);
            near_wide = lw && __any_sync(0xffffffffu, near_wide);
            if (hgrp == 0) {
                CT tot[NU][EPU];
#pragma unroll
                for (int i = 0; i < NU; ++i)
#pragma unroll
                    for (int w = 0; w < EPU; ++w) tot[i][w] = acc[i][w].value(ovf);
                if (near_wide) add_wide(tot, e0, e0 + cnt, cv);
                // partial row of the chunk, entry-major per hub:
                // [first chunk * Ws + entry * (chunks of the hub) + chunk]
                const int64_t c0 = a.node_chunk0[v];
                const int64_t nch = (a.row_ptr[v + 1] - a.row_ptr[v] + HUB_CHUNK - 1) / HUB_CHUNK;
                CT *out = (CT *)a.partial + c0 * a.dst.W + (t - c0);
#pragma unroll
                for (int i = 0; i < NU; ++i)
                    if (j + i * G < a.ws_units)
#pragma unroll
                        for (int w = 0; w < EPU; ++w)
                            out[(int64_t)((j + i * G) * EPU + w) * nch] = tot[i][w];
            }
            __syncwarp();
        }
        if (ovf) atomicOr(a.err, ERR_OVERFLOW);
        return;
    }

    // ---- nodes of degree <= HUB_CHUNK: GW lanes per node, which hold the ids
    // and colours of IB neighbours at a time, IPL per lane
    constexpr int IB = GW > U * P ? GW : U * P, IPL = IB / GW;
    const int64_t nblk = (int64_t)gridDim.x - a.chunk_blocks;
    const int64_t warp0 = ((int64_t)blockIdx.x - a.chunk_blocks) * wpb + (threadIdx.x >> 5);
    for (int64_t base = warp0 * NG; base < a.n_small; base += nblk * wpb * NG) {
        const int64_t idx = base + grp;
        const bool valid = idx < a.n_small;
        const uint4 rec = valid ? a.sched[idx] : make_uint4(0u, 0u, 0u, 0u);
        const int64_t v = rec.x;
        const int64_t e0 = (int64_t)(((uint64_t)rec.z << 32) | rec.y);
        const int d = (int)rec.w;
        const int cv = valid ? (int)a.colors[v] : 0;
        const int16_t *mapv = s_map + cv * a.k * (G * NU);
        const int dmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)d);
        bool near_wide = false;
        clear();
        uint32_t nid[IPL];
        int ncb[IPL];
        auto load_ids = [&](int off) {
#pragma unroll
            for (int p = 0; p < IPL; ++p) {
                const int pos = off + p * GW + lane % GW;
                const bool in = pos < d;
                nid[p] = in ? a.col[e0 + pos] : 0u;
                const int cu = in ? (int)a.ecol[e0 + pos] : cv;
                ncb[p] = cu * (G * NU);  // a neighbour of v's colour (or none) maps to nothing
                if (lw && cu != cv) near_wide |= (wide_of[nid[p]] & c_bit) != 0;
            }
        };
        load_ids(0);
        for (int off = 0; off < dmax; off += IB) {
            uint32_t id[IPL];
            int cb[IPL];
#pragma unroll
            for (int p = 0; p < IPL; ++p) { id[p] = nid[p]; cb[p] = ncb[p]; }
            if (off + IB < dmax) load_ids(off + IB);
            for (int t = 0; t < IB && off + t < dmax; t += U * P) {
                UT x[U][NU];
#pragma unroll
                for (int q = 0; q < U; ++q) {
                    // neighbour t + q P + par of the block, held by lane
                    // (that mod GW) of the node in its (that / GW)-th id
                    uint32_t u;
                    int c;
                    if constexpr (IPL > 1) {  // one round, t = 0
                        const int r = q * P / GW, at = q * P % GW;
                        u = __shfl_sync(0xffffffffu, id[r], grp * GW + at + par);
                        c = __shfl_sync(0xffffffffu, cb[r], grp * GW + at + par);
                    } else {
                        u = __shfl_sync(0xffffffffu, id[0], grp * GW + t + q * P + par);
                        c = __shfl_sync(0xffffffffu, cb[0], grp * GW + t + q * P + par);
                    }
                    fetch(x[q], u, mapv + c);
                }
#pragma unroll
                for (int q = 0; q < U; ++q) add(x[q]);
            }
        }
        if constexpr (P > 1) reduce(GW);
        const unsigned gmask = GW == 32 ? 0xffffffffu : ((1u << GW) - 1u) << (grp * GW);
        CT tot[NU][EPU];
#pragma unroll
        for (int i = 0; i < NU; ++i)
#pragma unroll
            for (int w = 0; w < EPU; ++w) tot[i][w] = acc[i][w].value(ovf);
        if (lw && (__ballot_sync(0xffffffffu, near_wide) & gmask)) add_wide(tot, e0, e0 + d, cv);
        bool wide = false;
        if (a.dst.N < (int)sizeof(CT)) {
#pragma unroll
            for (int i = 0; i < NU; ++i)
#pragma unroll
                for (int w = 0; w < EPU; ++w) wide |= above<CT>(tot[i][w], a.dst.N);
        }
        wide = (__ballot_sync(0xffffffffu, wide) & gmask) != 0;
        if (valid && par == 0) {
            uint8_t *low = a.dst.low(v), *high = a.dst.high(v);
#pragma unroll
            for (int i = 0; i < NU; ++i)
                if (j + i * G < a.ws_units) {
                    const int e = (j + i * G) * EPU;
                    store_low<EPU, CT>(low + e * a.dst.N, tot[i], a.dst.N);
                    if (wide)
                        for (int w = 0; w < EPU; ++w) store_rest<CT>(high, a.dst.W, a.dst.N, e + w, tot[i][w]);
                }
            if (wide) {
                any_wide = true;
                if (j == 0) atomicOr(a.dst.wide + v, a.dst.bit);
            }
        }
    }
    if (ovf) atomicOr(a.err, ERR_OVERFLOW);
    if (any_wide) atomicOr(a.levels, a.dst.bit);
}

typedef void (*GatherKernel)(GatherArgs);

// The instantiation for a count width (8 or 16 bytes), first-plane counts of
// N bytes, unit size, lanes per row G, units per lane NU, neighbours at once
// P, rows in flight U and blocks-per-SM target MB (gather_*.cu); NULL if it is
// not instantiated.
GatherKernel gather_kernel_ptr(size_t count_bytes, int N, int UB, int G, int NU, int P, int U, int MB);
GatherKernel gather_kernel_ptr_u64_4(int UB, int G, int NU, int P, int U, int MB);
GatherKernel gather_kernel_ptr_u64_8(int UB, int G, int NU, int P, int U, int MB);
GatherKernel gather_kernel_ptr_u128_4(int UB, int G, int NU, int P, int U, int MB);
GatherKernel gather_kernel_ptr_u128_8(int UB, int G, int NU, int P, int U, int MB);

// The schedules (rows in flight, blocks per SM) of one lane layout.
#define MC_GATHER_LAYOUT(CT, N, UB_, G_, NU_, P_)                                               \
    if (UB == UB_ && G == G_ && NU == NU_ && P == P_) {                                         \
        if (U == 2 && MB == 8) return gather_kernel<CT, N, UB_, G_, NU_, P_, 2, 8>;             \
        if (U == 2 && MB == 4) return gather_kernel<CT, N, UB_, G_, NU_, P_, 2, 4>;             \
        if (U == 1 && MB == 4) return gather_kernel<CT, N, UB_, G_, NU_, P_, 1, 4>;             \
        if (U == 2 && MB == 6) return gather_kernel<CT, N, UB_, G_, NU_, P_, 2, 6>;             \
        if (U == 4 && MB == 8) return gather_kernel<CT, N, UB_, G_, NU_, P_, 4, 8>;             \
        return nullptr;                                                                         \
    }
// A layout of fewer lanes than units (schedules 4 and 5).
#define MC_GATHER_FOLDED(CT, N, UB_, G_, NU_, P_)                                               \
    if (UB == UB_ && G == G_ && NU == NU_ && P == P_ && U == 2 && MB == 8)                      \
        return gather_kernel<CT, N, UB_, G_, NU_, P_, 2, 8>;

}  // namespace mc
