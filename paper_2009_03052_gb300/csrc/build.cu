// build.cu -- the colourful treelet count tables (Section 2.1, Eq. 1).
//
// Per level h the dynamic program runs as two kernels:
//   gather: S_h(v)[T'', C''] = sum_{u ~ v} c_h(u)[T'', C'']      (HBM bound)
//   merge : c_h(v)[T, C] = (1/beta_T) sum_{C' + C'' = C} c_{|T'|}(v)[T', C'] S_{|T''|}(v)[T'', C'']
// with T -> (T', T'') the canonical decomposition (T'' the subtree of the
// root's first child).  Rows are colour-relative: at node v only colour sets
// containing c_v (for c) or avoiding it (for S) are stored, indexed by the
// colex rank of the set with c_v deleted from the palette, so the merge's
// index structure is the same at every node and the gather reads only live
// entries of the neighbour's row.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <tuple>
#include <type_traits>

#include "gather.cuh"

namespace mc {

GatherKernel gather_kernel_ptr(size_t count_bytes, int N, int UB, int G, int NU, int P, int U, int MB)
{
    if (count_bytes == 16)
        return N == 4 ? gather_kernel_ptr_u128_4(UB, G, NU, P, U, MB) : gather_kernel_ptr_u128_8(UB, G, NU, P, U, MB);
    return N == 4 ? gather_kernel_ptr_u64_4(UB, G, NU, P, U, MB) : gather_kernel_ptr_u64_8(UB, G, NU, P, U, MB);
}

// The neighbour-sum kernel and its instantiations live in gather.cuh and
// gather_*.cu.
// Sum the chunk partials of each hub into its S row.  The chunk sums of a
// (hub, S entry) pair are contiguous; they become their inclusive prefix
// (the sampler binary-searches it) and the last prefix is the hub's
// neighbour sum.  Any overflowing partial sum means the total overflows too.
// A hub's S row is written in both planes; it is marked wide when an entry
// needs its upper part.
// Hubs of at most HUB_SERIAL chunks: a thread per (hub, entry) scans them in
// order (the threads of a warp take consecutive entries of one hub, whose
// chunk sums are adjacent); larger hubs: a warp per (hub, entry), 32 chunks
// per warp scan.

template <typename CT>
__device__ __forceinline__ void store_hub_entry(const Rows &dst, uint32_t v, int e, CT x, bool &wide)
{
    store_low<1, CT>(dst.low(v) + e * dst.N, &x, dst.N);
    store_rest<CT>(dst.high(v), dst.W, dst.N, e, x);
    if (above<CT>(x, dst.N)) {
        atomicOr(dst.wide + v, dst.bit);
        wide = true;
    }
}

// One launch: the first `big_blocks` blocks take the larger hubs.
template <typename CT>
__global__ void __launch_bounds__(256) hub_reduce_kernel(CT *__restrict__ partial, Rows dst, uint32_t *levels,
                                                         const uint32_t *__restrict__ hub_node,
                                                         const int64_t *__restrict__ hub_chunk0, int64_t n_hubs,
                                                         const uint32_t *__restrict__ big_hub, int64_t n_big, int big_blocks,
                                                         int *err)
{
    bool ovf = false, wide = false;
    const int Ws = dst.W;
    if ((int)blockIdx.x < big_blocks) {
        const int lane = threadIdx.x & 31;
        const int64_t nwarps = ((int64_t)big_blocks * blockDim.x) >> 5;
        for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < n_big * Ws; i += nwarps) {
            const int64_t bi = i / Ws;
            const int e = (int)(i - bi * Ws);
            const int64_t hub = big_hub[bi];
            const int64_t c0 = hub_chunk0[hub], nch = hub_chunk0[hub + 1] - c0;
            CT *p = partial + c0 * Ws + e * nch;
            CT carry = 0;
            for (int64_t b = 0; b < nch; b += 32) {
                const int64_t c = b + lane;
                CT x = c < nch ? p[c] : (CT)0;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const CT y = shfl_up(x, d);
                    if (lane >= d) ovf |= add_ovf(x, y);
                }
                ovf |= add_ovf(x, carry);
                if (c < nch) p[c] = x;
                carry = shfl(x, 31);
            }
            if (lane == 0) store_hub_entry<CT>(dst, hub_node[hub], e, carry, wide);
        }
    } else {
        const int64_t step = (int64_t)(gridDim.x - big_blocks) * blockDim.x;
        for (int64_t i = (int64_t)(blockIdx.x - big_blocks) * blockDim.x + threadIdx.x; i < n_hubs * Ws; i += step) {
            const int64_t hub = i / Ws;
            const int e = (int)(i - hub * Ws);
            const int64_t c0 = hub_chunk0[hub], nch = hub_chunk0[hub + 1] - c0;
            if (nch > HUB_SERIAL) continue;
            CT *p = partial + c0 * Ws + e * nch;
            CT run = 0;
            for (int64_t c = 0; c < nch; c += 4) {  // four loads in flight
                CT x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) x[q] = c + q < nch ? p[c + q] : (CT)0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    ovf |= add_ovf(run, x[q]);
                    if (c + q < nch) p[c + q] = run;
                }
            }
            store_hub_entry<CT>(dst, hub_node[hub], e, run, wide);
        }
    }
    if (ovf) atomicOr(err, ERR_OVERFLOW);
    if (wide) atomicOr(levels, dst.bit);
}

// ---------------------------------------------------------------------------
// merge of level h.  Output o carries (beta, #terms) and a list of (index
// into the c_{|T'|} row, index into the S_{|T''|} row) pairs, one per split of
// the colour set; c_1 is the constant 1.
//
// The merge by tiles of TN nodes, TN = 8 .. 128.  Each lower level pairs with
// one other level only -- c_{h1} with S_{h - h1} -- so a block stages the
// rows of one such pair at a time (cp.async, rows padded to an odd stride),
// computes the outputs of that pair, and goes on to the next; the output rows
// gather in shared memory and leave in one coalesced pass.  A thread keeps
// one node (tid mod TN) and takes every (threads / TN)-th output, so the
// threads that share an output run one program and read one entry of
// neighbouring rows: no divergence, no bank conflicts, and every lower row
// crosses the memory bus once.  Bound by latency at the few warps that shared
// memory allows (30 - 36%): issue slots are idle 38 - 46% of the time, and the
// stalls are fixed-latency waits, staging and barriers, in that order.  Staging
// the next pair while one is computed needs more shared memory and was slower
// (k = 7 levels 6 / 7: 4.8 / 5.5 against 3.9 / 4.8 ms), two nodes per thread
// gave nothing.  Against a thread per (node, output) reading whole counts
// through L1, ms per level 5 / 6 / 7 on R-MAT 22, k = 7, 128-bit counts: 10.6 /
// 15.0 / 12.5 before, 2.95 / 4.05 / 4.5 now; levels 6 / 7 / 8 on Chung-Lu 2M,
// k = 8: 20.8 / 27.8 / 21.1 before, 10.8 / 14.6 / 12.4 now; level 5 / 6 on a
// 994k-node grid, k = 6, 64-bit counts: 0.69 / 0.47 before, 0.34 / 0.26 now.
// Rows are read and written by their first planes (common.cuh): operands of 4
// or 8 bytes, with products of 64 to 128 bits.  A node with a wide row among a
// pair's operands reads that pair's operands from memory instead, in full;
// an output that exceeds its first plane writes its upper part at once, and
// the rest of such a row is zeroed when the tile leaves.
struct TilePair {
    int h1, h2;         // sizes of T' and T''
    int wa;             // row width of c_{h1} (0 for h1 = 1: implicit)
    int ca, cb;         // 8-byte pieces of their first planes
    int sa, sb;         // strides in shared memory (odd), in 8-byte pieces
    uint32_t ma, mb;    // ceil(2^32 / pieces): division by the row's pieces
    uint32_t bits;      // the pair's bits in the nodes' wide words
    int rec0, rec1;     // the pair's outputs in the record list
};
struct MergeTileArgs {
    Rows c[MAXK + 1], S[MAXK + 1];
    ExactDiv div[MAXK + 1];
    TilePair pair[MAXK];
    int npair;
    const uint2 *rec;       // output records: (o | beta << 16 | nterms << 24, first term)
    const uint32_t *terms;  // entries of the pair's rows: c_{h1} | S_{h2} << 16
    int nrec, nterms;
    const uint32_t *order;  // the nodes to do, NULL: 0 .. n_do - 1
    int64_t n_do;
    Rows out;
    int so, cw;             // output row: stride in shared memory and pieces of its first plane
    uint32_t mw;            // ceil(2^32 / cw)
    int log_tn, in_pieces;  // log2 TN; staging room of a node in 8-byte pieces
    uint32_t *levels;       // the levels that have a wide row
    const uint8_t *zero_root_colors;
    int *err;
};

// i / w for i < 2^16 by the precomputed m = ceil(2^32 / w)
__device__ __forceinline__ int div_width(int i, int w, uint32_t m) { return w == 1 ? i : (int)__umulhi((uint32_t)i, m); }

// The first-plane rows of a tile's nodes, in 8-byte pieces.
__device__ __forceinline__ void stage_rows(uint64_t *dst, const Rows &src, int pieces, int stride, uint32_t m, int tn,
                                           const uint32_t *node, int nthreads)
{
    for (int i = threadIdx.x; i < tn * pieces; i += nthreads) {
        const int r = div_width(i, pieces, m), e = i - r * pieces;
        const uint32_t v = node[r];
        if (v == 0xffffffffu) continue;
        const unsigned sa = (unsigned)__cvta_generic_to_shared(dst + r * stride + e);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(src.low(v) + 8 * e) : "memory");
    }
}

// Exact sums of products, as limbs with an explicit carry: no comparison per
// term.  `ovf` is set when the sum does not fit CT.
//   4 x 4 bytes: 64-bit products, 64 bits and a carry count;
//   4 x 8: the two 64-bit partial products on sums of their own;
//   8 x 8: 128-bit products, 128 bits and a carry count.
// At most 35 terms.  (With a 128-bit sum compared after each addition: 16.9
// against 14.3 ms at level 7 of Chung-Lu 2M, k = 8.)
template <typename CT, int NA, int NB> struct ProductSum {
    uint64_t lo = 0, hi = 0;
    uint32_t c = 0, c2 = 0;
    __device__ __forceinline__ void add(uint64_t x, uint64_t y)
    {
        if constexpr (NA == 8 && NB == 8) {
            asm("mad.lo.cc.u64 %0, %3, %4, %0;\n\tmadc.hi.cc.u64 %1, %3, %4, %1;\n\taddc.u32 %2, %2, 0;"
                : "+l"(lo), "+l"(hi), "+r"(c)
                : "l"(x), "l"(y));
        } else if constexpr (NA == 4 && NB == 4) {
            add1(lo, c, (uint64_t)(uint32_t)x * (uint32_t)y);
        } else {
            const uint32_t s = (uint32_t)(NA == 4 ? x : y);  // the 4-byte operand
            const uint64_t w = NA == 4 ? y : x;
            add1(lo, c, (uint64_t)s * (uint32_t)w);
            add1(hi, c2, (uint64_t)s * (uint32_t)(w >> 32));  // at 2^32
        }
    }
    static __device__ __forceinline__ void add1(uint64_t &l, uint32_t &carry, uint64_t p)
    {
        asm("add.cc.u64 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+l"(l), "+r"(carry) : "l"(p));
    }
    __device__ __forceinline__ CT value(bool &ovf) const
    {
        if constexpr (sizeof(CT) == 16) {
            if constexpr (NA == 8 && NB == 8) {
                ovf |= c != 0;
                return ((CT)hi << 64) | lo;
            } else if constexpr (NA == 4 && NB == 4) {
                return ((CT)c << 64) | lo;
            } else {
                return (((CT)c << 64) | lo) + ((((CT)c2 << 64) | hi) << 32);
            }
        } else {
            if constexpr (NA == 8 && NB == 8) {
                ovf |= (hi | c) != 0;
                return lo;
            } else if constexpr (NA == 4 && NB == 4) {
                ovf |= c != 0;
                return lo;
            } else {
                const u128 t = (((u128)c << 64) | lo) + ((((u128)c2 << 64) | hi) << 32);
                ovf |= (uint64_t)(t >> 64) != 0;
                return (uint64_t)t;
            }
        }
    }
};

// Sum over the terms of A[ia] * B[ib] (HA = false: of B[ib]), the operands
// first-plane counts of NA and NB bytes.
template <typename CT, bool HA, int NA, int NB>
__device__ __forceinline__ CT merge_sum(const uint8_t *A, const uint8_t *B, const uint32_t *term, int nt, bool &ovf)
{
    typedef typename std::conditional<NA == 4, uint32_t, uint64_t>::type TA;
    typedef typename std::conditional<NB == 4, uint32_t, uint64_t>::type TB;
    if constexpr (HA) {
        ProductSum<CT, NA, NB> s;
#pragma unroll 2
        for (int i = 0; i < nt; ++i) {
            const uint32_t tm = term[i];
            s.add(((const TA *)A)[tm & 0xffffu], ((const TB *)B)[tm >> 16]);
        }
        return s.value(ovf);
    } else {
        uint64_t lo = 0;
        uint32_t hi = 0;
        for (int i = 0; i < nt; ++i) {
            const uint64_t x = ((const TB *)B)[term[i] >> 16];
            lo += x;
            hi += lo < x;
        }
        if constexpr (sizeof(CT) == 16) return ((CT)hi << 64) | lo;
        ovf |= hi != 0;
        return (CT)lo;
    }
}

// The same from the rows in memory, upper parts included.
template <typename CT>
__device__ __noinline__ CT merge_sum_wide(const Rows &A, const Rows &B, bool has_a, int64_t v, const uint32_t *term, int nt,
                                          bool &ovf)
{
    CT sum = 0;
    for (int i = 0; i < nt; ++i) {
        CT p = entry_at<CT>(B, v, term[i] >> 16);
        if (has_a) {
            CT q;
            ovf |= mul_ovf(entry_at<CT>(A, v, term[i] & 0xffffu), p, q);
            p = q;
        }
        ovf |= add_ovf(sum, p);
    }
    return sum;
}

template <typename CT, int THREADS>
__global__ void __launch_bounds__(THREADS) merge_tile_kernel(const __grid_constant__ MergeTileArgs a)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int tn = 1 << a.log_tn, W = a.out.W, N = a.out.N, wpn = (W + 31) >> 5;
    uint64_t *s_in = (uint64_t *)s_raw;
    uint64_t *s_out = s_in + tn * a.in_pieces;
    uint2 *s_rec = (uint2 *)(s_out + tn * a.so);
    uint32_t *s_terms = (uint32_t *)(s_rec + a.nrec);
    uint32_t *s_src = s_terms + a.nterms;  // nodes whose rows are read (0xffffffff: none)
    uint32_t *s_dst = s_src + tn;          // nodes whose row is written
    uint32_t *s_big = s_dst + tn;          // per node, a bit per output above its first plane
    for (int i = threadIdx.x; i < a.nrec; i += THREADS) s_rec[i] = a.rec[i];
    for (int i = threadIdx.x; i < a.nterms; i += THREADS) s_terms[i] = a.terms[i];
    const int node = threadIdx.x & (tn - 1), grp = threadIdx.x >> a.log_tn, ngrp = THREADS >> a.log_tn;
    bool ovf = false, inexact = false, any_wide = false;
    const int64_t ntiles = (a.n_do + tn - 1) >> a.log_tn;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        if (threadIdx.x < tn) {
            const int64_t i = (tile << a.log_tn) + threadIdx.x;
            const uint32_t u = i < a.n_do ? (a.order ? a.order[i] : (uint32_t)i) : 0xffffffffu;
            s_dst[threadIdx.x] = u;
            s_src[threadIdx.x] = (u != 0xffffffffu && a.zero_root_colors && a.zero_root_colors[u] != 0) ? 0xffffffffu : u;
        }
        for (int i = threadIdx.x; i < tn * wpn; i += THREADS) s_big[i] = 0;
        __syncthreads();
        const uint32_t v = s_src[node];
        const bool live = v != 0xffffffffu;
        const uint32_t wide = live ? a.out.wide[v] : 0u;
        bool big = false;
        for (int p = 0; p < a.npair; ++p) {
            const TilePair &P = a.pair[p];
            uint64_t *s_b = s_in + tn * P.sa;
            if (P.wa) stage_rows(s_in, a.c[P.h1], P.ca, P.sa, P.ma, tn, s_src, THREADS);
            stage_rows(s_b, a.S[P.h2], P.cb, P.sb, P.mb, tn, s_src, THREADS);
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            __syncthreads();
            const uint8_t *A = (const uint8_t *)(s_in + node * P.sa);
            const uint8_t *B = (const uint8_t *)(s_b + node * P.sb);
            const int na = a.c[P.h1].N, nb = a.S[P.h2].N;
            const bool full = (wide & P.bits) != 0;
            auto outputs = [&](auto sum_of) {
                for (int r = P.rec0 + grp; r < P.rec1; r += ngrp) {
                    const uint2 rc = s_rec[r];
                    const uint32_t *term = s_terms + rc.y;
                    const int o = rc.x & 0xffffu, beta = (rc.x >> 16) & 255, nt = rc.x >> 24;
                    CT sum = 0;
                    if (live) {
                        if (!full) sum = sum_of(term, nt);
                        else sum = merge_sum_wide<CT>(a.c[P.h1], a.S[P.h2], P.wa != 0, v, term, nt, ovf);
                        if (beta != 1) {
                            CT q = 0;
                            if (!exact_div(sum, a.div[beta], q)) inexact = true;
                            sum = q;
                        }
                        if (above<CT>(sum, N)) {
                            store_rest<CT>(a.out.high(v), W, N, o, sum);
                            atomicOr(&s_big[node * wpn + (o >> 5)], 1u << (o & 31));
                            big = true;
                        }
                    }
                    uint8_t *row = (uint8_t *)(s_out + node * a.so);
                    if (N == 4) ((uint32_t *)row)[o] = (uint32_t)sum;
                    else ((uint64_t *)row)[o] = (uint64_t)sum;
                }
            };
#define MC_MERGE(HA, NA, NB) \
    outputs([&](const uint32_t *t, int nt) { return merge_sum<CT, HA, NA, NB>(A, B, t, nt, ovf); })
            if (!P.wa) {
                if (nb == 4) MC_MERGE(false, 4, 4);
                else MC_MERGE(false, 4, 8);
            } else if (na == 4) {
                if (nb == 4) MC_MERGE(true, 4, 4);
                else MC_MERGE(true, 4, 8);
            } else {
                if (nb == 4) MC_MERGE(true, 8, 4);
                else MC_MERGE(true, 8, 8);
            }
#undef MC_MERGE
            __syncthreads();
        }
        for (int i = threadIdx.x; i < tn * a.cw; i += THREADS) {
            const int r = div_width(i, a.cw, a.mw), e = i - r * a.cw;
            const uint32_t u = s_dst[r];
            if (u != 0xffffffffu) ((uint64_t *)a.out.low(u))[e] = s_out[r * a.so + e];
        }
        if (__syncthreads_or(big)) {
            any_wide = true;
            for (int r = 0; r < tn; ++r) {
                bool has = false;
                for (int w = 0; w < wpn; ++w) has |= s_big[r * wpn + w] != 0;
                if (!has) continue;
                uint8_t *high = a.out.high(s_dst[r]);
                for (int e = threadIdx.x; e < W; e += THREADS)
                    if (!((s_big[r * wpn + (e >> 5)] >> (e & 31)) & 1u)) store_rest<CT>(high, W, N, e, (CT)0);
                if (threadIdx.x == 0) atomicOr(a.out.wide + s_dst[r], a.out.bit);
            }
            __syncthreads();
        }
    }
    if (ovf) atomicOr(a.err, ERR_OVERFLOW);
    if (inexact) atomicOr(a.err, ERR_INEXACT);
    if (any_wide && threadIdx.x == 0) atomicOr(a.levels, a.out.bit);
}

// First-plane rows of the nodes in list[0 .. cnt) set to zero, a warp per row.
__global__ void __launch_bounds__(256) zero_rows_kernel(Rows out, const uint32_t *__restrict__ list, int64_t cnt)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = warp; i < cnt; i += nwarps)
        for (int e = lane; e < out.s0 / 8; e += 32) ((uint64_t *)out.low(list[i]))[e] = 0;
}

// ---------------------------------------------------------------------------
// per-node totals of a level over a set of shapes, and an inclusive u128
// prefix over the nodes (the cumulative counts of Section 3.2.1, taken over
// nodes for the root draw).
// ---------------------------------------------------------------------------
template <typename CT, int G>
__global__ void __launch_bounds__(256) row_totals_kernel(Rows c, int64_t n, int W, int R,
                                                         uint64_t allow0, uint64_t allow1,
                                                         u128 *__restrict__ tot, int *err)
{
    // groups of G lanes per node, 32/G nodes per warp
    const int lane = threadIdx.x & 31;
    const int grp = lane / G, j = lane % G;
    constexpr int NG = 32 / G;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool ovf = false;
    for (int64_t v0 = warp * NG; v0 < n; v0 += nwarps * NG) {
        const int64_t v = v0 + grp;
        u128 s = 0;
        const bool wide = v < n && (c.wide[v] & c.bit);
        if (v < n)
            for (int eb = j; eb < W; eb += 8 * G) {  // up to 8 loads in flight per lane
                CT x[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int e = eb + i * G;
                    const int sh = e % R;  // set-major row: entry e is (set e / R, shape e % R)
                    const bool ok = e < W && (sh < 64 ? (allow0 >> sh) & 1 : (allow1 >> (sh - 64)) & 1);
                    x[i] = ok ? row_low<CT>(c.low(v), c.N, e) : (CT)0;
                    if (ok && wide) x[i] |= row_rest<CT>(c.high(v), W, c.N, e);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) ovf |= add_ovf(s, widen(x[i]));
            }
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            const u128 o = shfl_xor(s, d);
            ovf |= add_ovf(s, o);
        }
        if (j == 0 && v < n) tot[v] = s;
    }
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}

// The rooted shapes of each unrooted treelet at one level: treelet j owns
// shape[off[j] .. off[j + 1]).
struct TreeletShapes {
    int16_t off[32];
    uint8_t shape[128];
};

// Per node and unrooted treelet T_j: the sum of the node's level-h counts
// over the rooted shapes of T_j and all colour sets, tot[j * n + v].  One
// thread per (node, treelet), treelet fastest, so a warp reads a few whole
// rows.  Overflow of a sum is flagged.
template <typename CT>
__global__ void __launch_bounds__(256) treelet_totals_kernel(Rows c, int64_t n, int R, int Bc,
                                                             int nu, const __grid_constant__ TreeletShapes ts,
                                                             u128 *__restrict__ tot, int *err)
{
    bool ovf = false;
    const int64_t total = n * nu;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = i / nu;
        const int j = (int)(i - v * nu);
        u128 s = 0;
        for (int q = ts.off[j]; q < ts.off[j + 1]; ++q) {
            const int sh = ts.shape[q];
            for (int b = 0; b < Bc; ++b) ovf |= add_ovf(s, widen(entry_at<CT>(c, v, b * R + sh)));
        }
        tot[(int64_t)j * n + v] = s;
    }
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}

constexpr int SCAN_THREADS = 512, SCAN_ITEMS = 8, SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T> __device__ __forceinline__ T warp_prefix(T x)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T y = shfl_up(x, d);
        if (lane >= d) x += y;
    }
    return x;
}

template <typename T> __device__ __forceinline__ T block_exclusive_scan(T x, T *smem, T &block_total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const T inc = warp_prefix(x);
    if (lane == 31) smem[w] = inc;
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        T y = lane < nw ? smem[lane] : (T)0;
        y = warp_prefix(y);
        if (lane < nw) smem[lane] = y;
    }
    __syncthreads();
    const T before = w > 0 ? smem[w - 1] : (T)0;
    block_total = smem[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before + inc - x;
}

// Inclusive 64- or 128-bit prefix of m arrays of n entries, `stride` entries apart
// (blockIdx.y picks one): tile sums, then each block adds up the sums of the
// tiles before its own and scans its tile.  One tile (n <= 4096) needs the
// second kernel only; beyond SCAN_DIRECT tiles the sums are scanned by a
// kernel of their own first, since every block would read all of them (at
// most 32 KB here; a tile is 64 KB).  Launches 3 -> 2 (1 for small arrays).
constexpr int64_t SCAN_DIRECT = 2048;

template <typename T> __global__ void __launch_bounds__(SCAN_THREADS) scan_tiles_kernel(const T *__restrict__ x, int64_t n, int64_t stride,
                                                                  T *__restrict__ tile_sum, int *err)
{
    __shared__ T smem[32];
    x += blockIdx.y * stride;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T s = 0;
    bool ovf = false;
    for (int i = 0; i < SCAN_ITEMS; ++i)
        if (base + i < n) ovf |= add_ovf(s, x[base + i]);
    T tot;
    const T ex = block_exclusive_scan(s, smem, tot);
    // the block total is exact iff no prefix wrapped
    if (ex + s < ex) ovf = true;
    if (threadIdx.x == blockDim.x - 1) tile_sum[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = tot;
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}

template <typename T> __global__ void __launch_bounds__(1024) scan_tile_sums_kernel(T *tile_sum, int64_t ntiles, int *err)
{
    __shared__ T smem[32];
    tile_sum += blockIdx.y * ntiles;
    T carry = 0;
    bool ovf = false;
    for (int64_t b = 0; b < ntiles; b += blockDim.x) {
        const int64_t i = b + threadIdx.x;
        const T x = i < ntiles ? tile_sum[i] : 0;
        T tot;
        const T ex = block_exclusive_scan(x, smem, tot);
        const T before = carry + ex;
        if (before < carry || before + x < before) ovf = true;
        if (i < ntiles) tile_sum[i] = before;  // exclusive
        const T nc = carry + tot;
        if (nc < carry) ovf = true;
        carry = nc;
    }
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}

// `scanned`: tile_sum holds the sums before each tile, else the tiles' own
template <typename T> __global__ void __launch_bounds__(SCAN_THREADS) scan_apply_kernel(T *__restrict__ x, int64_t n, int64_t stride,
                                                                  const T *__restrict__ tile_sum, bool scanned, int *err)
{
    __shared__ T smem[32];
    bool ovf = false;
    x += blockIdx.y * stride;
    T before = 0;
    if (scanned) {
        before = tile_sum[(int64_t)blockIdx.y * gridDim.x + blockIdx.x];
    } else if (blockIdx.x > 0) {
        tile_sum += (int64_t)blockIdx.y * gridDim.x;
        T s = 0;
        for (int t = threadIdx.x; t < (int)blockIdx.x; t += SCAN_THREADS) ovf |= add_ovf(s, tile_sum[t]);
        const T ex = block_exclusive_scan(s, smem, before);
        if (ex + s < ex) ovf = true;
    }
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T v[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = base + i < n ? x[base + i] : 0;
        ovf |= add_ovf(s, v[i]);
    }
    T tot;
    const T ex = block_exclusive_scan(s, smem, tot);
    T run = before + ex;
    if (run < before || run + s < run) ovf = true;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        run += v[i];
        if (base + i < n) x[base + i] = run;
    }
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}

// Sum over the nodes [lo, hi) of the level-h counts of unrooted treelet
// first + blockIdx.y: per block its part, then the parts added up.
template <typename CT>
__global__ void __launch_bounds__(256) treelet_sum_kernel(Rows c, int64_t lo, int64_t hi, int R, int Bc, int first,
                                                          const __grid_constant__ TreeletShapes ts, u128 *__restrict__ part,
                                                          int *err)
{
    __shared__ u128 smem[32];
    bool ovf = false;
    u128 s = 0;
    const int j = first + blockIdx.y;
    for (int64_t v = lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < hi; v += (int64_t)gridDim.x * blockDim.x)
        for (int q = ts.off[j]; q < ts.off[j + 1]; ++q)
            for (int b = 0; b < Bc; ++b) ovf |= add_ovf(s, widen(entry_at<CT>(c, v, b * R + ts.shape[q])));
    u128 tot;
    const u128 ex = block_exclusive_scan(s, smem, tot);
    if (ex + s < ex) ovf = true;
    if (threadIdx.x == 0) part[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = tot;
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}
__global__ void __launch_bounds__(256) part_sum_kernel(const u128 *__restrict__ part, int np, u128 *__restrict__ out, int *err)
{
    __shared__ u128 smem[32];
    bool ovf = false;
    u128 s = 0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) ovf |= add_ovf(s, part[(int64_t)blockIdx.x * np + i]);
    u128 tot;
    const u128 ex = block_exclusive_scan(s, smem, tot);
    if (ex + s < ex) ovf = true;
    if (threadIdx.x == 0) out[blockIdx.x] = tot;
    if (ovf) atomicOr(err, ERR_OVERFLOW);
}

// Colours of the edges' far ends (ecol, so that neighbour loops read colours
// contiguously) and colour blocks: every node's neighbour list stably
// partitioned by the neighbours' colours (scol), with the block starts (coff,
// k + 1 per node).  The per-colour counts are also the level-1 neighbour sums
// S_1(v)[{a}] (c of a single node is 1 at its own colour), written here too: rows
// of 4-byte first-plane counts (a degree is below 2^32), never wide.
//   Nodes of degree <= HUB_CHUNK: L = 8 lanes per node (4 below an average
// degree of 8: grid 0.067 against 0.055 ms with 8), in node order (the lists of
// neighbouring nodes are adjacent; in the gather's degree order 0.19 ms), each
// with ceil(d / L) consecutive neighbours; per-colour counts are packed one byte
// per colour (at most 64 each), so a prefix over the lanes and one over the
// bytes (a multiplication) give every lane its cursors.
//   Hubs, spread over their 64-neighbour chunks so no warp walks a whole hub:
// here the chunks' colours and per-colour counts, a warp per chunk (the first
// `chunk_blocks` blocks); then per hub the exclusive prefix of those counts over
// its chunks (each chunk's start inside every colour block), the block starts
// and S_1; then per chunk the scatter.
// Bound by the random colour reads and the lists' bytes.  Chung-Lu 1M, k = 5:
// 0.13 ms, against 0.072 + 0.086 + 0.020 for the edge colours, a thread per
// node and the chunk counts on their own.
static_assert(HUB_CHUNK == 64, "16 neighbours per lane, byte counters; two 32-edge rounds per chunk");

template <int L>
__global__ void __launch_bounds__(256) colour_blocks_kernel(const int64_t *__restrict__ row_ptr,
                                                            const uint32_t *__restrict__ col,
                                                            const uint8_t *__restrict__ colors,
                                                            int64_t n, const int64_t *__restrict__ chunk_e0,
                                                            const int64_t *__restrict__ chunk_e1, int64_t n_chunks,
                                                            int chunk_blocks, int k, uint8_t *__restrict__ ecol,
                                                            uint32_t *__restrict__ scol, int32_t *__restrict__ coff, Rows S1,
                                                            uint32_t *__restrict__ ccnt)
{
    const int lane = threadIdx.x & 31;
    if ((int)blockIdx.x < chunk_blocks) {
        const int64_t nwarps = ((int64_t)chunk_blocks * blockDim.x) >> 5;
        for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < n_chunks; c += nwarps) {
            const int64_t e0 = chunk_e0[c], e1 = chunk_e1[c];
            int cc[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int64_t e = e0 + 32 * r + lane;
                cc[r] = e < e1 ? (int)colors[col[e]] : -1;
                if (e < e1) ecol[e] = (uint8_t)cc[r];
            }
            uint32_t mine = 0;
#pragma unroll
            for (int a = 0; a < MAXK; ++a)
                if (a < k) {
                    const uint32_t x = __popc(__ballot_sync(0xffffffffu, cc[0] == a)) +
                                       __popc(__ballot_sync(0xffffffffu, cc[1] == a));
                    if (lane == a) mine = x;
                }
            if (lane < k) ccnt[c * k + lane] = mine;
        }
        return;
    }
    const int j = lane & (L - 1);
    constexpr int NG = 32 / L;
    const int64_t warp0 = ((int64_t)(blockIdx.x - chunk_blocks) * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)(gridDim.x - chunk_blocks) * blockDim.x) >> 5;
    for (int64_t base = warp0 * NG; base < n; base += nwarps * NG) {
        const int64_t v = base + (lane / L);
        const int64_t e0 = v < n ? row_ptr[v] : 0, deg = v < n ? row_ptr[v + 1] - e0 : 0;
        const bool small = v < n && deg <= HUB_CHUNK;
        const int d = small ? (int)deg : 0, m = (d + L - 1) / L;
        const int lo = min(d, j * m), hi = min(d, lo + m);
        uint64_t cols = 0;  // four bits per own neighbour
        uint64_t cnt = 0;
        for (int i = lo; i < hi; ++i) {
            const int c = colors[col[e0 + i]];
            ecol[e0 + i] = (uint8_t)c;
            cols |= (uint64_t)c << (4 * (i - lo));
            cnt += 1ull << (8 * c);
        }
        __syncwarp();
        uint64_t inc = cnt;
#pragma unroll
        for (int s = 1; s < L; s <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, inc, s, L);
            if (j >= s) inc += y;
        }
        const uint64_t tot = __shfl_sync(0xffffffffu, inc, L - 1, L);
        const uint64_t start = (tot * 0x0101010101010101ull) << 8;  // exclusive prefix over the bytes
        uint64_t cur = start + inc - cnt;
        for (int i = lo; i < hi; ++i) {
            const int c = (int)(cols >> (4 * (i - lo)) & 15u);
            scol[e0 + (int64_t)((cur >> (8 * c)) & 0xffu)] = col[e0 + i];
            cur += 1ull << (8 * c);
        }
        if (small) {
            for (int a = j; a <= k; a += L)
                coff[v * (k + 1) + a] = a < k ? (int32_t)((start >> (8 * a)) & 0xffu) : d;
            const int cv = colors[v];
            for (int a = j; a < k - 1; a += L)
                ((uint32_t *)S1.low(v))[a] = (uint32_t)((tot >> (8 * (a < cv ? a : a + 1))) & 0xffu);
        }
        __syncwarp();
    }
}

__global__ void hub_chunk_prefix_kernel(const uint8_t *__restrict__ colors, const uint32_t *__restrict__ hub_node,
                                        const int64_t *__restrict__ hub_chunk0, int64_t n_hubs, int k,
                                        uint32_t *__restrict__ ccnt, int32_t *__restrict__ coff,
                                        Rows S1)
{
    // one warp per hub: lanes take 32 chunks at a time; a warp scan per
    // colour turns the counts, in place, into each chunk's start inside that
    // colour's block
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t hb = warp; hb < n_hubs; hb += nwarps) {
        const int64_t v = hub_node[hb];
        const int64_t c0 = hub_chunk0[hb], c1 = hub_chunk0[hb + 1];
        uint32_t tot[MAXK];
#pragma unroll
        for (int a = 0; a < MAXK; ++a) tot[a] = 0;
        for (int64_t b = c0; b < c1; b += 32) {
            const int64_t c = b + lane;
#pragma unroll
            for (int a = 0; a < MAXK; ++a)
                if (a < k) {
                    const uint32_t x = c < c1 ? ccnt[c * k + a] : 0u;
                    uint32_t inc = x;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
                        if (lane >= d) inc += y;
                    }
                    if (c < c1) ccnt[c * k + a] = tot[a] + inc - x;
                    tot[a] += __shfl_sync(0xffffffffu, inc, 31);
                }
        }
        if (lane == 0) {
            uint32_t run = 0;
#pragma unroll
            for (int a = 0; a < MAXK; ++a)
                if (a < k) {
                    coff[v * (k + 1) + a] = (int32_t)run;
                    run += tot[a];
                }
            coff[v * (k + 1) + k] = (int32_t)run;
            const int cv = colors[v];
#pragma unroll
            for (int a = 0; a < MAXK - 1; ++a)
                if (a < k - 1) ((uint32_t *)S1.low(v))[a] = tot[a < cv ? a : a + 1];
        }
    }
}

__global__ void hub_chunk_scatter_kernel(const uint32_t *__restrict__ col, const uint8_t *__restrict__ ecol,
                                         const int64_t *__restrict__ row_ptr,
                                         const uint32_t *__restrict__ chunk_node,
                                         const int64_t *__restrict__ chunk_e0, const int64_t *__restrict__ chunk_e1,
                                         int64_t n_chunks, int k, const uint32_t *__restrict__ cstart,
                                         const int32_t *__restrict__ coff, uint32_t *__restrict__ scol)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t c = warp; c < n_chunks; c += nwarps) {
        const int64_t v = chunk_node[c];
        const int64_t base = row_ptr[v];
        const int64_t e0 = chunk_e0[c], e1 = chunk_e1[c];
        int cc[2];
        uint32_t uu[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int64_t e = e0 + 32 * r + lane;
            cc[r] = e < e1 ? (int)ecol[e] : -1;
            uu[r] = e < e1 ? col[e] : 0u;
        }
        uint32_t pos[MAXK];
#pragma unroll
        for (int a = 0; a < MAXK; ++a)
            pos[a] = a < k ? (uint32_t)coff[v * (k + 1) + a] + cstart[c * k + a] : 0u;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            uint32_t my = 0;
#pragma unroll
            for (int a = 0; a < MAXK; ++a)
                if (a < k) {
                    const unsigned m = __ballot_sync(0xffffffffu, cc[r] == a);
                    if (cc[r] == a) my = pos[a] + __popc(m & lt);
                    pos[a] += __popc(m);
                }
            if (cc[r] >= 0) scol[base + my] = uu[r];
        }
    }
}

// Root-search buckets: X in [0, R) falls in bucket b = floor(X / D), D =
// ceil(R / nb); start[b] is the first node whose inclusive prefix exceeds
// b * D, so the node drawn for X lies in [start[b], start[b + 1]].
// (For m prefixes at once: blockIdx.y.)  A block's first and last bucket are
// searched over all nodes, the others between those two.
__global__ void __launch_bounds__(256) bucket_kernel(const u128 *__restrict__ prefix, int64_t n, int64_t nb, u128 *D_out,
                                                     uint32_t *__restrict__ start, int64_t pstride, int64_t bstride)
{
    __shared__ u128 s_D;
    __shared__ int64_t s_end[2];
    prefix += blockIdx.y * pstride;
    start += blockIdx.y * bstride;
    if (threadIdx.x == 0) {
        const u128 R = prefix[n - 1];
        const u128 d = (R >> 64) == 0 ? (u128)(((uint64_t)R + (uint64_t)nb - 1 >= (uint64_t)R)
                                                   ? ((uint64_t)R + (uint64_t)nb - 1) / (uint64_t)nb
                                                   : (uint64_t)R / (uint64_t)nb + ((uint64_t)R % (uint64_t)nb != 0))
                                      : R / (u128)nb + ((R % (u128)nb) != 0 ? 1 : 0);
        s_D = d ? d : 1;
        if (blockIdx.x == 0) D_out[blockIdx.y] = s_D;
    }
    __syncthreads();
    const u128 D = s_D;
    auto search = [&](int64_t b, int64_t lo, int64_t hi) {
        const u128 X = (u128)b * D;
        while (lo < hi) {  // first v with prefix[v] > X, else n
            const int64_t mid = (lo + hi) >> 1;
            if (prefix[mid] > X) hi = mid; else lo = mid + 1;
        }
        return lo;
    };
    for (int64_t b0 = blockIdx.x * (int64_t)blockDim.x; b0 <= nb; b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b1 = min(nb, b0 + blockDim.x - 1);
        if (threadIdx.x == 0) s_end[0] = search(b0, 0, n);
        if (threadIdx.x == 32) s_end[1] = search(b1, 0, n);
        __syncthreads();
        const int64_t b = b0 + threadIdx.x;
        if (b <= b1) {
            const int64_t v = search(b, s_end[0], s_end[1]);
            start[b] = (uint32_t)(v < n ? v : n - 1);
        }
        __syncthreads();
    }
}

void build_buckets(const u128 *prefix, int64_t n, int64_t nb, u128 *dD, uint32_t *start, cudaStream_t s, int m,
                   int64_t bstride)
{
    if (n <= 0) return;
    MC_LAUNCH("buckets", s, bucket_kernel<<<dim3((unsigned)grid_for(nb + 1, 256), (unsigned)m), 256, 0, s>>>(
                                prefix, n, nb, dD, start, n, bstride));
}

int64_t bucket_count(int64_t n) { return std::max<int64_t>(1, std::min<int64_t>(n, (int64_t)1 << 22)); }

// A colour >= k is reported and replaced by 0 in the tables' own copy, so
// the kernels after this one never index past a colour's slot; the build
// then fails when its error flags are read.  No row is wide yet.
__global__ void check_colours_kernel(uint8_t *colors, int64_t n, int k, uint32_t *wide, int *err)
{
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        wide[v] = 0;
        if (colors[v] >= k) {
            atomicOr(err, ERR_COLOUR);
            colors[v] = 0;
        }
    }
}

__global__ void fill_ones_kernel(void *dst, int64_t n, int bytes)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (bytes == 8) ((uint64_t *)dst)[i] = 1;
        else ((u128 *)dst)[i] = 1;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int64_t scan_tiles(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE; }

// the scan with a caller-provided tile-sum buffer of m * scan_tiles(n) entries
template <typename T>
static void inclusive_scan_buf(T *x, int64_t n, int64_t stride, int *err, T *ts, cudaStream_t s, int m)
{
    if (n <= 0) return;
    const int64_t ntiles = scan_tiles(n);
    const dim3 grid((unsigned)ntiles, (unsigned)m);
    const bool scanned = ntiles > SCAN_DIRECT;
    if (ntiles > 1) MC_LAUNCH("scan_tiles", s, scan_tiles_kernel<T><<<grid, SCAN_THREADS, 0, s>>>(x, n, stride, ts, err));
    if (scanned)
        MC_LAUNCH("scan_tile_sums", s, scan_tile_sums_kernel<T><<<dim3(1, (unsigned)m), 1024, 0, s>>>(ts, ntiles, err));
    MC_LAUNCH("scan_apply", s, scan_apply_kernel<T><<<grid, SCAN_THREADS, 0, s>>>(x, n, stride, ts, scanned, err));
}

void inclusive_scan_u128(u128 *x, int64_t n, int *err, Arena &scratch, cudaStream_t s, int m)
{
    if (n > 0) inclusive_scan_buf<u128>(x, n, n, err, scratch.get<u128>((size_t)scan_tiles(n) * m), s, m);
}

void inclusive_scan_u64(uint64_t *x, int64_t n, int64_t stride, int *err, uint64_t *sums, cudaStream_t s, int m)
{
    inclusive_scan_buf<uint64_t>(x, n, stride, err, sums, s, m);
}

void inclusive_scan_u64(uint64_t *x, int64_t n, int64_t stride, int *err, Arena &scratch, cudaStream_t s, int m)
{
    if (n > 0) inclusive_scan_buf<uint64_t>(x, n, stride, err, scratch.get<uint64_t>((size_t)scan_tiles(n) * m), s, m);
}

ExactDiv make_div(int beta)
{
    ExactDiv d{};
    int t = 0;
    while (!((beta >> t) & 1)) ++t;
    const uint64_t odd = (uint64_t)(beta >> t);
    // Newton iteration for the inverse of an odd number modulo 2^64 / 2^128
    uint64_t inv = odd;  // correct to 3 bits
    for (int i = 0; i < 6; ++i) inv *= 2 - odd * inv;
    u128 inv2 = inv;
    for (int i = 0; i < 2; ++i) inv2 *= (u128)2 - (u128)odd * inv2;
    d.shift = t;
    d.inv64 = inv;
    d.inv128 = inv2;
    d.qmax64 = ~0ull / odd;
    d.qmax128 = (~(u128)0) / (u128)odd;
    return d;
}

template <typename CT> size_t bytes_of() { return sizeof(CT); }

template <typename CT>
static void launch_row_totals_t(const Rows &c, int64_t n, int W, int R, uint64_t allow0, uint64_t allow1, u128 *tot,
                                int *err, cudaStream_t s)
{
    int G = 1;  // lanes per node: each covers up to 8 entries
    while (G * 8 < W && G < 32) G <<= 1;
    const int grid = grid_for((n * G + 31) / 32 * 32, 256);
    switch (G) {
    case 1: MC_LAUNCH("row_totals", s, row_totals_kernel<CT, 1><<<grid, 256, 0, s>>>(c, n, W, R, allow0, allow1, tot, err)); break;
    case 2: MC_LAUNCH("row_totals", s, row_totals_kernel<CT, 2><<<grid, 256, 0, s>>>(c, n, W, R, allow0, allow1, tot, err)); break;
    case 4: MC_LAUNCH("row_totals", s, row_totals_kernel<CT, 4><<<grid, 256, 0, s>>>(c, n, W, R, allow0, allow1, tot, err)); break;
    case 8: MC_LAUNCH("row_totals", s, row_totals_kernel<CT, 8><<<grid, 256, 0, s>>>(c, n, W, R, allow0, allow1, tot, err)); break;
    case 16: MC_LAUNCH("row_totals", s, row_totals_kernel<CT, 16><<<grid, 256, 0, s>>>(c, n, W, R, allow0, allow1, tot, err)); break;
    default: MC_LAUNCH("row_totals", s, row_totals_kernel<CT, 32><<<grid, 256, 0, s>>>(c, n, W, R, allow0, allow1, tot, err)); break;
    }
}

void launch_row_totals(const mc_tables *t, int h, uint64_t allow0, uint64_t allow1, u128 *tot, int *err,
                       cudaStream_t s)
{
    const int64_t n = t->g->n;
    if (n == 0) return;
    if (t->packed) {
        launch_packed_row_totals(t, h, allow0, allow1, tot, err, s);
        return;
    }
    const int W = t->geo.Wc[h], R = shape_catalog().r[h];
    if (t->bits == 64)
        launch_row_totals_t<uint64_t>(t->rows(h, 0), n, W, R, allow0, allow1, tot, err, s);
    else
        launch_row_totals_t<u128>(t->rows(h, 0), n, W, R, allow0, allow1, tot, err, s);
}

static TreeletShapes treelet_shapes(int h)
{
    const ShapeCatalog &cat = shape_catalog();
    TreeletShapes ts{};
    int q = 0;
    for (int j = 0; j < cat.n_unrooted[h]; ++j) {
        ts.off[j] = (int16_t)q;
        for (int i = 0; i < cat.r[h]; ++i)
            if (cat.shapes[cat.gid(h, i)].unrooted == j) ts.shape[q++] = (uint8_t)i;
    }
    ts.off[cat.n_unrooted[h]] = (int16_t)q;
    return ts;
}

// Dense tables: tot[j * n + v] for every unrooted treelet j of level h in
// one pass over the level's c rows.
void launch_treelet_totals(const mc_tables *t, int h, u128 *tot, int *err, cudaStream_t s)
{
    const int64_t n = t->g->n;
    const ShapeCatalog &cat = shape_catalog();
    const int nu = cat.n_unrooted[h], R = cat.r[h];
    if (n == 0 || nu == 0) return;
    MC_REQUIRE(!t->packed, "treelet totals read dense tables");
    const TreeletShapes ts = treelet_shapes(h);
    const int Bc = t->geo.Bc[h];
    const int grid = grid_for(n * nu, 256);
    if (t->bits == 64)
        MC_LAUNCH("treelet_totals", s, treelet_totals_kernel<uint64_t><<<grid, 256, 0, s>>>(
                                           t->rows(h, 0), n, R, Bc, nu, ts, tot, err));
    else
        MC_LAUNCH("treelet_totals", s, treelet_totals_kernel<u128><<<grid, 256, 0, s>>>(
                                           t->rows(h, 0), n, R, Bc, nu, ts, tot, err));
}

static const char *const kGatherName[MAXK + 1] = {"gather_h0", "gather_h1", "gather_h2", "gather_h3",
                                                  "gather_h4", "gather_h5", "gather_h6", "gather_h7",
                                                  "gather_h8"};
static const char *const kMergeName[MAXK + 1] = {"merge_h0", "merge_h1", "merge_h2", "merge_h3", "merge_h4",
                                                 "merge_h5", "merge_h6", "merge_h7", "merge_h8"};

// Schedules of the neighbour sums (the autotuner's choices): rows in flight,
// blocks of 256 threads per SM (4: at most 64 registers, 6: 40, 8: 32) and, for
// rows of 5 to 16 units, the lanes folded twice or four times: two or four
// units per lane, so that a warp takes more nodes and hands fewer ids round.
// Picked on GB300 (ms): folded four times at h = 2, 3, 5 of the grid, k = 6
// (0.070 / 0.095 / 0.095; twice 0.097 / 0.137 / 0.117, not 0.131 / 0.164 /
// 0.156) and at h = 2, 5 of the other k = 6 graphs (0.122 against 0.150, batch);
// 4 blocks per SM at h = 4..6 of k = 8 (8.2 against 12.2 at h = 6 of Chung-Lu
// 2M).
constexpr int GATHER_CANDIDATES = 7;
static const int kGatherU[GATHER_CANDIDATES] = {2, 2, 1, 2, 2, 2, 4};
static const int kGatherMB[GATHER_CANDIDATES] = {8, 4, 4, 6, 8, 8, 8};
static const int kGatherFold[GATHER_CANDIDATES] = {1, 1, 1, 1, 2, 4, 1};

// G lanes for a row: the smallest power of two that covers its units, at most
// 32, then NU units per lane.  Rows of fewer than 8 units take P neighbours
// of the node at once, 8 lanes per node (4 when the average degree is below
// 8: most of 8 would idle), so that the ids and colours of 8 neighbours are
// one coalesced read.
template <typename CT> static bool launch_gather(const GatherArgs &base, int r, int h, int cand, cudaStream_t s)
{
    if (cand < 0 || cand >= GATHER_CANDIDATES) return false;
    GatherArgs ga = base;
    const int N = ga.src.N, set_bytes = r * N;
    const int UB = set_bytes % 16 == 0 ? 16 : set_bytes % 8 == 0 ? 8 : 4;  // a unit never straddles two colour sets
    ga.ups = set_bytes / UB;
    ga.ws_units = ga.dst.W * N / UB;
    int G = 1;
    while (G < ga.ws_units && G < 32) G <<= 1;
    int NU = (ga.ws_units + 31) / 32;
    if (NU > 3) NU = 6;
    if (NU * 32 < ga.ws_units) throw Error(MC_E_INTERNAL, "gather: S row too wide");
    const int fold = kGatherFold[cand];
    if (fold > 1) {
        if (NU != 1 || G < 8 || G > 16 || (fold == 4 && UB == 16)) return false;
        G /= fold;
        NU = (ga.ws_units + G - 1) / G;
    }
    const int lanes = ga.nnz >= 8 * ga.n ? 8 : 4, P = G < lanes ? lanes / G : 1;
    auto kern = gather_kernel_ptr(sizeof(CT), N, UB, G, NU, P, kGatherU[cand], kGatherMB[cand]);
    if (!kern) {
        if (fold > 1) return false;
        throw Error(MC_E_INTERNAL, "gather: no kernel for this row layout");
    }
    const int NG = 32 / (G * P);
    const int wpb = 256 / 32;
    const int64_t cap = (int64_t)sm_count() * 32;
    ga.chunk_blocks = (int)std::min<int64_t>((ga.n_chunks + wpb - 1) / wpb, cap);
    const int64_t node_blocks = std::max<int64_t>(1, std::min<int64_t>((ga.n_small + NG * wpb - 1) / (NG * wpb), cap));
    const int grid = (int)(ga.chunk_blocks + node_blocks);
    const size_t smem = (size_t)ga.k * ga.k * NU * G * sizeof(int16_t);
    MC_LAUNCH(kGatherName[h], s, kern<<<grid, 256, smem, s>>>(ga));
    return true;
}

// The tiled merge's plan: TN nodes per tile, the largest power of two up to
// 128 whose rows fit 72 KB of shared memory (three blocks per SM) and that
// leaves two tiles per SM, at least 8; shifted by `shift` (the tuner's
// neighbours: twice the tile is 1.4x faster at level 6 of k = 6, half of it
// with 128 threads up to 10% at levels 3-5 of k = 7).  False when the plan
// does not exist.
static bool plan_merge_tile(MergeTileArgs &ta, const MergePairs &Q, int shift, size_t &smem)
{
    auto magic = [](int w) { return w > 1 ? (uint32_t)((((uint64_t)1 << 32) + w - 1) / w) : 0u; };
    ta.npair = Q.n;
    ta.in_pieces = 0;
    for (int p = 0; p < Q.n; ++p) {
        TilePair &P = ta.pair[p];
        P.h1 = Q.h1[p];
        P.h2 = Q.h2[p];
        P.wa = P.h1 == 1 ? 0 : ta.c[P.h1].W;
        P.ca = P.wa ? ta.c[P.h1].s0 / 8 : 0;
        P.cb = ta.S[P.h2].s0 / 8;
        P.sa = P.wa ? P.ca | 1 : 0;
        P.sb = P.cb | 1;
        P.ma = magic(P.ca);
        P.mb = magic(P.cb);
        P.bits = (P.wa ? 1u << P.h1 : 0u) | 1u << (16 + P.h2);
        P.rec0 = Q.rec0[p];
        P.rec1 = Q.rec0[p + 1];
        ta.in_pieces = std::max(ta.in_pieces, P.sa + P.sb);
    }
    ta.cw = ta.out.s0 / 8;
    ta.so = ta.cw | 1;
    ta.mw = magic(ta.cw);
    ta.nrec = (int)Q.rec.size() / 2;
    ta.nterms = (int)Q.terms.size();
    const size_t fixed = (size_t)ta.nrec * 8 + (size_t)ta.nterms * 4;
    const size_t node = (size_t)(ta.in_pieces + ta.so) * 8 + 8 + (size_t)(ta.out.W + 31) / 32 * 4;
    int lt = 7;
    while (lt > 3 && (fixed + (node << lt) > 72 * 1024 || (ta.n_do >> lt) < 2 * (int64_t)sm_count())) --lt;
    lt += shift;
    if (lt < 3 || lt > 7) return false;
    ta.log_tn = lt;
    smem = fixed + (node << lt);
    return smem <= 220 * 1024;
}

// Merge candidates: threads per block and the tile against the plan's (as a
// power of two).
constexpr int MERGE_CANDIDATES = 6;

template <typename CT, int THREADS>
static bool launch_merge_tile(const MergeTileArgs &base, const MergePairs &Q, int h, int shift, cudaStream_t s)
{
    MergeTileArgs ta = base;
    size_t smem = 0;
    if (!plan_merge_tile(ta, Q, shift, smem)) return false;
    if (smem > 48 * 1024) allow_shared((const void *)merge_tile_kernel<CT, THREADS>);
    const int64_t ntiles = (ta.n_do + (1 << ta.log_tn) - 1) >> ta.log_tn;
    const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(2048 / THREADS, (int64_t)(227 * 1024 / (smem + 1024))));
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>(ntiles, (int64_t)sm_count() * per_sm));
    MC_LAUNCH(kMergeName[h], s, merge_tile_kernel<CT, THREADS><<<g, THREADS, smem, s>>>(ta));
    return true;
}

template <typename CT>
static bool launch_merge(const MergeTileArgs &ta, const MergePairs &Q, int h, int cand, cudaStream_t s)
{
    switch (cand) {
    case 0: return launch_merge_tile<CT, 256>(ta, Q, h, 0, s);
    case 1: return launch_merge_tile<CT, 256>(ta, Q, h, -1, s);
    case 2: return launch_merge_tile<CT, 256>(ta, Q, h, 1, s);
    case 3: return launch_merge_tile<CT, 512>(ta, Q, h, 0, s);
    case 4: return launch_merge_tile<CT, 128>(ta, Q, h, 0, s);
    case 5: return launch_merge_tile<CT, 128>(ta, Q, h, -1, s);
    default: return false;
    }
}

// ---------------------------------------------------------------------------
// Autotuner: the schedule of each (kernel, k, count width, level, graph
// shape, layout) is chosen by timing every candidate once on the first build
// that meets it (the candidates compute identical tables, so which one runs
// does not change any result).  The graph's shape is reduced to a degree
// bucket: log2 n, log2 of the average degree in half steps, log2 of the largest
// degree.  The layout is what else decides which candidate is best, or whether
// it exists: the bytes of the first-plane counts, the node order and, at level
// k, the merge program.  Choices can be loaded from and appended to a cache file
// (mc_autotune, or the MC_AUTOTUNE_CACHE environment variable); a line names
// the set of schedules that it was chosen from (TUNE_SET, counted up whenever a
// schedule number changes its meaning), and only the present set's are used as
// they are.
// ---------------------------------------------------------------------------
namespace {
constexpr int TUNE_SET = 2;
struct TuneKey {
    int kind, k, bits, h, logn, logdeg, loghub;
    int layout = -1;  // -1: of any layout (pinned choices, lines without one)
    bool operator<(const TuneKey &o) const
    {
        return std::tie(kind, k, bits, h, logn, logdeg, loghub, layout) <
               std::tie(o.kind, o.k, o.bits, o.h, o.logn, o.logdeg, o.loghub, o.layout);
    }
    TuneKey any() const
    {
        TuneKey x = *this;
        x.layout = -1;
        return x;
    }
};
struct TuneState {
    std::mutex mu;
    std::map<TuneKey, int> choice;  // timed here or by another process
    std::map<TuneKey, int> pinned;  // by mc_autotune_set
    std::map<TuneKey, int> hint;    // file lines without a set: used where tuning is off
    std::map<TuneKey, int> latest;  // the last of these per key of any layout
    std::set<TuneKey> retuned;  // mode 2: keys tuned again in this process
    int mode = 1;               // 0 never tune, 1 tune unknown keys, 2 tune every key once more
    std::string file;
    bool env_read = false;
};
TuneState &tune_state()
{
    static TuneState st;
    return st;
}

int candidates(int kind) { return kind == 0 ? GATHER_CANDIDATES : MERGE_CANDIDATES; }

void tune_load_file_locked(TuneState &st, const std::string &path)
{
    FILE *f = std::fopen(path.c_str(), "r");
    if (!f) return;
    char line[256];
    while (std::fgets(line, sizeof(line), f)) {
        TuneKey k{};
        int v = 0, layout = -1, set = 0;
        const int got = std::sscanf(line, "%d %d %d %d %d %d %d %d %d %d", &k.kind, &k.k, &k.bits, &k.h, &k.logn,
                                    &k.logdeg, &k.loghub, &v, &layout, &set);
        if ((k.kind != 0 && k.kind != 1) || v < 0 || v >= candidates(k.kind)) continue;
        if (got == 8) {
            st.hint[k.any()] = v;
        } else if (got == 10 && set == TUNE_SET && layout >= 0) {
            k.layout = layout;
            st.choice[k] = v;
        } else {
            continue;
        }
        st.latest[k.any()] = v;
    }
    std::fclose(f);
}

void tune_env_locked(TuneState &st)
{
    if (st.env_read) return;
    st.env_read = true;
    const char *p = std::getenv("MC_AUTOTUNE_CACHE");
    if (p && *p) {
        st.file = p;
        tune_load_file_locked(st, st.file);
    }
}

int ilog2(double x) { return x < 1.0 ? 0 : (int)std::floor(std::log2(x)); }
}  // namespace

static TuneKey tune_key(int kind, int k, int count_bits, int h, int64_t n, int64_t nnz, int64_t max_degree)
{
    const double nn = (double)std::max<int64_t>(n, 1);
    return TuneKey{kind, k, count_bits, h, ilog2((double)n), ilog2((double)nnz * (double)nnz / (nn * nn)),
                   ilog2((double)max_degree + 1)};
}

// The key of a build's kernel of level h.  Widths grow with the level, so those
// of a merge's operands follow from the first level of 8-byte counts.
static TuneKey tune_key(int kind, const mc_tables *t, int h)
{
    TuneKey key = tune_key(kind, t->k, t->bits, h, t->g->n, t->g->nnz, t->g->max_degree);
    if (kind == 0) {
        key.layout = (t->Nc[h] == 8) | (t->Ns[h] == 8) << 1;
    } else {
        int first = 1;
        while (first <= h && t->Nc[first] == 4) ++first;
        key.layout = first | (t->g->order != nullptr) << 4 | (t->skip_round && h == t->k) << 5 |
                     (t->zero_root && h == t->k) << 6;
    }
    return key;
}

// Run `launch(candidate)` for the tuned candidate of `key`; when tuning is
// allowed and the key is new (or mode 2, or the stored candidate is refused),
// time every candidate first.
template <typename F>
static void run_tuned(TuneKey key, int ncand, bool allow, cudaStream_t s, F &&launch)
{
    TuneState &st = tune_state();
    int v = -1;
    bool tune = false, stored = false;
    {
        std::lock_guard<std::mutex> lock(st.mu);
        tune_env_locked(st);
        allow = allow && st.mode > 0;
        auto find = [&](const std::map<TuneKey, int> &m, const TuneKey &k) {
            auto it = m.find(k);
            if (it == m.end()) return false;
            v = it->second;
            return true;
        };
        stored = find(st.choice, key);
        if (!stored && !find(st.pinned, key.any())) {
            tune = allow;
            if (!tune) find(st.hint, key.any());
        }
        tune = tune || (allow && st.mode == 2 && !st.retuned.count(key));
    }
    if (!tune && v >= 0) {
        if (launch(v)) return;
        v = -1;
        tune = allow && stored;
    }
    if (tune) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        MC_CUDA(cudaStreamIsCapturing(s, &cs));
        if (cs != cudaStreamCaptureStatusNone) tune = false;
    }
    if (tune) {
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        MC_CUDA(cudaEventCreate(&e0));
        MC_CUDA(cudaEventCreate(&e1));
        // three rounds over the candidates, each candidate's best time
        // counts: every candidate meets the caches as the others left them
        float best[8];
        bool ok[8];
        for (int c = 0; c < ncand && c < 8; ++c) { best[c] = 0.f; ok[c] = true; }
        for (int rep = 0; rep < 3; ++rep)
            for (int c = 0; c < ncand && c < 8; ++c) {
                if (!ok[c]) continue;
                MC_CUDA(cudaEventRecord(e0, s));
                if (!launch(c)) { ok[c] = false; continue; }
                MC_CUDA(cudaEventRecord(e1, s));
                MC_CUDA(cudaEventSynchronize(e1));
                float ms = 0.f;
                MC_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                if (rep == 0 || ms < best[c]) best[c] = ms;
            }
        int bv = -1;
        for (int c = 0; c < ncand && c < 8; ++c)
            if (ok[c] && (bv < 0 || best[c] < best[bv])) bv = c;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        v = bv < 0 ? 0 : bv;
        std::lock_guard<std::mutex> lock(st.mu);
        st.choice[key] = v;
        st.latest[key.any()] = v;
        st.retuned.insert(key);
        if (!st.file.empty()) {
            if (FILE *f = std::fopen(st.file.c_str(), "a")) {
                std::fprintf(f, "%d %d %d %d %d %d %d %d %d %d\n", key.kind, key.k, key.bits, key.h, key.logn,
                             key.logdeg, key.loghub, v, key.layout, TUNE_SET);
                std::fclose(f);
            }
        }
    }
    if ((v < 0 || !launch(v)) && !launch(0)) throw Error(MC_E_INTERNAL, "no schedule runs this level");
}

template <typename CT> static void build_levels(mc_tables *t, int *err, cudaStream_t s, bool allow_tune)
{
    const mc_graph *g = t->g;
    const Geometry &G = t->geo;
    const int k = t->k;
    const int64_t n = g->n;
    if (n == 0) return;
    uint32_t *levels = (uint32_t *)err + 1;  // the levels with a wide row
    // level 1 neighbour sums
    // colour blocks of every adjacency list, and the level-1 neighbour sums
    const int cblocks = g->n_chunks ? grid_for(g->n_chunks * 32, 256) : 0;
    const bool sparse = g->nnz < 8 * n;
    const int nblocks = grid_for(n * (sparse ? 4 : 8), 256);
    auto blocks = sparse ? colour_blocks_kernel<4> : colour_blocks_kernel<8>;
    uint32_t *ccnt = t->ccnt;
    MC_LAUNCH("colour_blocks", s, blocks<<<cblocks + nblocks, 256, 0, s>>>(
                                      g->row_ptr, g->col, t->colors, n, g->chunk_e0, g->chunk_e1,
                                      g->n_chunks, cblocks, k, t->ecol, t->scol, t->coff, t->rows(1, 1), ccnt));
    if (g->n_hubs) {
        MC_LAUNCH("colour_blocks_hub", s, hub_chunk_prefix_kernel<<<grid_for(g->n_hubs * 32, 256), 256, 0, s>>>(
                                              t->colors, g->hub_node, g->hub_chunk0, g->n_hubs, k, ccnt, t->coff,
                                              t->rows(1, 1)));
        MC_LAUNCH("colour_blocks_hub", s, hub_chunk_scatter_kernel<<<grid_for(g->n_chunks * 32, 256), 256, 0, s>>>(
                                              g->col, t->ecol, g->row_ptr, g->chunk_node, g->chunk_e0, g->chunk_e1,
                                              g->n_chunks, k, ccnt, t->coff, t->scol));
    }
    MergeTileArgs ta{};
    for (int h = 1; h <= k; ++h) {
        ta.c[h] = t->rows(h, 0);
        ta.S[h] = t->rows(h, 1);
    }
    for (int b = 1; b <= MAXK; ++b) ta.div[b] = make_div(b);
    ta.order = g->order;
    ta.n_do = g->n_do;
    ta.levels = levels;
    ta.err = err;
    for (int h = 2; h <= k; ++h) {
        if (t->skip_round && h == k - 1) continue;  // round k-1 skipped: nothing reads it
        ta.rec = t->p_rec[h];
        ta.terms = t->p_terms[h];
        ta.out = t->rows(h, 0);
        ta.zero_root_colors = (t->zero_root && h == k) ? t->colors : nullptr;
        if (g->order)
            MC_LAUNCH("zero_rows", s, zero_rows_kernel<<<grid_for((n - g->n_do) * 32, 256), 256, 0, s>>>(
                                          ta.out, g->order + g->n_do, n - g->n_do));
        const TuneKey mkey = tune_key(1, t, h);
        run_tuned(mkey, MERGE_CANDIDATES, allow_tune, s, [&](int c) { return launch_merge<CT>(ta, programs(k, t->skip_round).pairs[h], h, c, s); });
        if (h <= k - 1) {
            GatherArgs ga{};
            ga.row_ptr = g->row_ptr;
            ga.col = g->col;
            ga.colors = t->colors;
            ga.ecol = t->ecol;
            ga.node_chunk0 = g->node_chunk0;
            ga.src = t->rows(h, 0);
            ga.dst = t->rows(h, 1);
            ga.levels = levels;
            ga.partial = t->Sp[h];
            ga.chunk_node = g->chunk_node;
            ga.chunk_e0 = g->chunk_e0;
            ga.chunk_e1 = g->chunk_e1;
            ga.gmap = t->g_map[h];
            ga.n = n;
            ga.nnz = g->nnz;
            ga.n_chunks = g->n_chunks;
            ga.k = k;
            ga.Bs = G.Bs[h];
            ga.err = err;
            ga.sched = g->sched;
            ga.n_small = g->n_small;
            const TuneKey gkey = tune_key(0, t, h);
            const int rh = shape_catalog().r[h];
            run_tuned(gkey, GATHER_CANDIDATES, allow_tune, s, [&](int c) { return launch_gather<CT>(ga, rh, h, c, s); });
            if (g->n_hubs) {
                const int big = g->n_big_hubs ? grid_for(g->n_big_hubs * G.Ws[h] * 32, 256) : 0;
                MC_LAUNCH("hub_reduce", s, hub_reduce_kernel<CT><<<big + grid_for(g->n_hubs * G.Ws[h], 256), 256, 0, s>>>(
                    (CT *)t->Sp[h], t->rows(h, 1), levels, g->hub_node, g->hub_chunk0, g->n_hubs, g->big_hub, g->n_big_hubs,
                    big, err));
            }
        }
    }
}

}  // namespace mc

using namespace mc;

// Bytes of the first-plane counts of each level: 4 where the counts of the
// level are expected below 2^30, so that (almost) no row is wide, else 8.
// Expected largest count: the star of the largest degree, (d_max / k)^(h-1),
// and the trees at the end of a random edge, (h-1)! (g / k)^(h-1) with g the
// sum of squared degrees / nnz.  S_h counts like c_{h+1}.  A level with some
// wide rows is exact but costs its readers a look at the node's word: with
// 0.3% wide rows at level 4 the sampler of the 1M-node, k = 5 workload was
// 20% slower than with none.
static void plan_widths(mc_tables *t)
{
    const double star = std::log2(std::max((double)t->g->max_degree / t->k, 1.0));
    const double walk = std::log2(std::max(t->g->walk_growth / t->k, 1e-3));
    auto width = [&](int h) {
        double fact = 0;
        for (int i = 2; i < h; ++i) fact += std::log2((double)i);
        return h <= 2 || ((h - 1) * star <= 30 && (h - 1) * walk + fact <= 30) ? 4 : 8;
    };
    for (int h = 1; h <= t->k; ++h) {
        t->Nc[h] = width(h);
        t->Ns[h] = h == 1 ? 4 : width(h + 1);
    }
}

// Every launch of a build for the colours in `colors`, on stream s, into the
// buffers of t: no allocation, no host read, no synchronisation (so a
// rebuild can be captured into a CUDA graph).
static void enqueue_build(mc_tables *t, const uint8_t *colors, cudaStream_t s, bool allow_tune)
{
    const mc_graph *g = t->g;
    const int64_t n = g->n;
    const int k = t->k;
    int *err = t->dev_err;
    MC_CUDA(cudaMemsetAsync(err, 0, 4 * sizeof(int), s));
    if (n) {
        // the tables' own copy of the colours, checked before any kernel reads them
        if (colors != t->colors)
            MC_CUDA(cudaMemcpyAsync(t->colors, colors, (size_t)n, cudaMemcpyDefault, s));
        MC_LAUNCH("check_colours", s, check_colours_kernel<<<grid_for(n, 256), 256, 0, s>>>(t->colors, n, k, t->wide, err));
    }
    if (t->bits == 64) build_levels<uint64_t>(t, err, s, allow_tune);
    else build_levels<u128>(t, err, s, allow_tune);
    // root index of the top level (the level sampled by default); the other
    // levels get theirs on first use
    if (n) {
        launch_row_totals(t, k, ~0ull, ~0ull, t->prefix[k], err, s);
        inclusive_scan_buf<u128>(t->prefix[k], n, n, err, t->scan_tmp, s, 1);
        build_buckets(t->prefix[k], n, t->nbucket, t->dev_D, t->bucket[k], s);
    }
}

// Read the level-k total, the bucket width and the error flags back.
static void finish_build(mc_tables *t, cudaStream_t s)
{
    const int64_t n = t->g->n;
    int flags[2] = {0, 0};
    u128 R = 0, D = 1;
    MC_CUDA(cudaMemcpyAsync(flags, t->dev_err, sizeof(flags), cudaMemcpyDeviceToHost, s));
    if (n) {
        MC_CUDA(cudaMemcpyAsync(&R, t->prefix[t->k] + (n - 1), sizeof(u128), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaMemcpyAsync(&D, t->dev_D, sizeof(u128), cudaMemcpyDeviceToHost, s));
    }
    MC_CUDA(cudaStreamSynchronize(s));
    const int herr = flags[0];
    t->wide_levels = (uint32_t)flags[1];
    if (herr & ERR_COLOUR) throw Error(MC_E_INVALID, "a colour is >= k");
    if (herr & ERR_OVERFLOW)
        throw Error(MC_E_OVERFLOW, "a count does not fit in " + std::to_string(t->bits) + " bits");
    if (herr & ERR_INEXACT) throw Error(MC_E_INTERNAL, "a merge numerator is not divisible by beta");
    t->R[t->k] = R;
    t->bucketD[t->k] = D;
}

extern "C" mc_status mc_build_tables(const mc_graph *g, const uint8_t *colors, int k, int count_bits,
                                     uint32_t flags, const mc_allocator *alloc, void *stream,
                                     mc_tables **out)
{
    if (out) *out = nullptr;
    mc_tables *t = nullptr;
    mc_status st = guarded([&] {
        MC_REQUIRE(out && g, "graph or out is NULL");
        MC_REQUIRE(colors || g->n == 0, "colors is NULL");
        if (k < 2 || k > MAXK) throw Error(MC_E_UNSUPPORTED, "k must be in 2..8");
        MC_REQUIRE(count_bits == 64 || count_bits == 128, "count_bits must be 64 or 128");
        MC_REQUIRE((flags & ~(MC_BUILD_ZERO_ROOT | MC_BUILD_SKIP_ROUND | MC_BUILD_SUCCINCT | MC_BUILD_VARLEN)) == 0,
                   "unknown flags");
        if (flags & MC_BUILD_SKIP_ROUND) {
            MC_REQUIRE(k >= 4, "round skipping needs k >= 4");
            MC_REQUIRE(!(flags & MC_BUILD_ZERO_ROOT), "round skipping and zero-rooting do not combine");
        }
        cudaStream_t s = (cudaStream_t)stream;
        t = new mc_tables();
        t->g = g;
        t->k = k;
        t->bits = count_bits;
        t->zero_root = flags & MC_BUILD_ZERO_ROOT;
        t->skip_round = flags & MC_BUILD_SKIP_ROUND;
        t->varlen = flags & MC_BUILD_VARLEN;
        const bool pack = (flags & (MC_BUILD_SUCCINCT | MC_BUILD_VARLEN)) != 0;
        t->geo = make_geometry(k);
        t->arena.stream = s;
        if (alloc) { t->arena.alloc.a = *alloc; t->arena.alloc.custom = true; }
        const int64_t n = g->n;
        const Geometry &G = t->geo;
        const size_t cb = count_bits / 8;
        // every buffer a build writes, kept for rebuilds
        t->dev_err = t->arena.get<int>(4);
        t->dev_D = t->arena.get<u128>(1);
        t->scan_tmp = t->arena.get<u128>((size_t)std::max<int64_t>(scan_tiles(n), 1));
        if (g->n_hubs) t->ccnt = t->arena.get<uint32_t>((size_t)g->n_chunks * k);
        t->colors = t->arena.get<uint8_t>((size_t)n);
        t->wide = t->arena.get<uint32_t>((size_t)n);
        plan_widths(t);
        t->ecol = t->arena.get<uint8_t>((size_t)g->nnz);
        t->scol = t->arena.get<uint32_t>((size_t)g->nnz);
        t->coff = t->arena.get<int32_t>((size_t)n * (k + 1));
        // programs
        const Programs &P = programs(k, t->skip_round);
        for (int j = 0; j < 32; ++j) t->copies_k[j] = P.copies[j];
        uint8_t *prog = t->arena.get<uint8_t>(P.blob.size());
        MC_CUDA(cudaMemcpyAsync(prog, P.blob.data(), P.blob.size(), cudaMemcpyHostToDevice, s));
        for (int h = 1; h <= k; ++h) {
            t->p_rec[h] = (uint2 *)(prog + P.rec_at[h]);
            t->p_terms[h] = (uint32_t *)(prog + P.terms_at[h]);
            t->g_map[h] = (int16_t *)(prog + P.map_at[h]);
        }
        // tables
        for (int h = 2; h <= k; ++h)
            if (!t->level_missing(h)) t->c[h] = t->arena.get<uint8_t>(t->level_bytes(h, 0, n));
        for (int h = 1; h <= k - 1; ++h)
            if (!t->level_missing(h)) t->S[h] = t->arena.get<uint8_t>(t->level_bytes(h, 1, n));
        for (int h = 2; h <= k - 1; ++h)
            if (!t->level_missing(h)) t->Sp[h] = t->arena.get<uint8_t>((size_t)g->n_chunks * G.Ws[h] * cb);
        t->nbucket = bucket_count(n);
        t->prefix[k] = t->arena.get<u128>((size_t)n);
        t->bucket[k] = t->arena.get<uint32_t>((size_t)t->nbucket + 1);
        enqueue_build(t, colors, s, true);
        finish_build(t, s);
        if (pack) {
            pack_tables(t, s);
            t->packed = true;
        }
    });
    if (st != MC_OK) { delete t; return st; }
    *out = t;
    return MC_OK;
}

extern "C" mc_status mc_rebuild_tables(mc_tables *t, const uint8_t *colors, void *stream)
{
    return guarded([&] {
        MC_REQUIRE(t, "tables is NULL");
        MC_REQUIRE(colors || t->g->n == 0, "colors is NULL");
        if (t->packed) throw Error(MC_E_UNSUPPORTED, "packed (succinct) tables cannot be rebuilt in place");
        std::lock_guard<std::mutex> lock(t->idx_mu);
        enqueue_build(t, colors, (cudaStream_t)stream, false);
        t->stale = true;
        t->broken.clear();
        for (int h = 2; h < t->k; ++h) t->level_stale[h] = t->prefix[h] != nullptr;
    });
}

void mc::refresh_tables(const mc_tables *tc, cudaStream_t s, bool force)
{
    mc_tables *t = const_cast<mc_tables *>(tc);
    std::lock_guard<std::mutex> lock(t->idx_mu);
    if (force) {
        // a replayed capture runs no host code: treat the device state as new
        t->stale = true;
        t->broken.clear();
        for (int h = 2; h < t->k; ++h) t->level_stale[h] = t->prefix[h] != nullptr;
    }
    if (!t->broken.empty()) throw Error(MC_E_INVALID, "the last rebuild failed: " + t->broken);
    if (!t->stale) return;
    try {
        finish_build(t, s);
    } catch (const Error &e) {
        t->broken = e.what();
        throw;
    }
    t->stale = false;
}

extern "C" mc_status mc_tables_status(const mc_tables *t, void *stream)
{
    return guarded([&] {
        MC_REQUIRE(t, "tables is NULL");
        refresh_tables(t, (cudaStream_t)stream, true);
    });
}

void mc::ensure_level_index(const mc_tables *tc, int h, cudaStream_t s)
{
    mc_tables *t = const_cast<mc_tables *>(tc);
    refresh_tables(t, s);
    std::lock_guard<std::mutex> lock(t->idx_mu);
    if (h < 2 || (t->prefix[h] && !t->level_stale[h])) return;
    if (t->level_missing(h)) throw Error(MC_E_INVALID, "level h was skipped (round skipping)");
    const int64_t n = t->g->n;
    Arena scratch(true);
    scratch.alloc = t->arena.alloc;
    scratch.stream = s;
    int *err = scratch.get<int>(1);
    u128 *dD = scratch.get<u128>(1);
    MC_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    // a stale index (from an older colouring) is rebuilt in its own buffers
    u128 *p = t->prefix[h] ? t->prefix[h] : t->arena.get<u128>((size_t)n);
    uint32_t *bk = t->bucket[h] ? t->bucket[h] : t->arena.get<uint32_t>((size_t)t->nbucket + 1);
    launch_row_totals(t, h, ~0ull, ~0ull, p, err, s);
    inclusive_scan_u128(p, n, err, scratch, s);
    build_buckets(p, n, t->nbucket, dD, bk, s);
    u128 R = 0, D = 1;
    int herr = 0;
    if (n) {
        MC_CUDA(cudaMemcpyAsync(&R, p + (n - 1), sizeof(u128), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaMemcpyAsync(&D, dD, sizeof(u128), cudaMemcpyDeviceToHost, s));
    }
    MC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    MC_CUDA(cudaStreamSynchronize(s));
    if (herr) throw Error(MC_E_OVERFLOW, "a level total does not fit in 128 bits");
    t->R[h] = R;
    t->bucketD[h] = D;
    t->bucket[h] = bk;
    t->prefix[h] = p;  // published last
    t->level_stale[h] = false;
}

extern "C" void mc_free_tables(mc_tables *t)
{
    if (!t) return;
    mc_graph *owned = t->owned_graph;
    delete t;
    mc_free_graph(owned);
}

// Rooted totals of level h over the nodes [lo, hi): of all shapes (j0 < 0, one
// value, from the cached root index) or of the rootings of the unrooted
// shapes j0 .. j0 + nj.
static std::vector<u128> level_rooted_totals(const mc_tables *t, int h, int j0, int nj, int64_t lo, int64_t hi,
                                             cudaStream_t s)
{
    const ShapeCatalog &cat = shape_catalog();
    const int64_t n = t->g->n;
    std::vector<u128> out((size_t)nj, 0);
    if (h == 1) {
        if (j0 <= 0) out[0] = (u128)(hi - lo);
        return out;
    }
    if (hi <= lo) return out;
    if (j0 < 0) {
        ensure_level_index(t, h, s);
        if (lo == 0 && hi == n) {  // read back with the index
            out[0] = t->R[h];
            return out;
        }
    }
    Arena scratch(true);
    scratch.alloc = t->arena.alloc;
    scratch.stream = s;
    int *err = scratch.get<int>(1);
    MC_CUDA(cudaMemsetAsync(err, 0, sizeof(int), s));
    int herr = 0;
    if (j0 >= 0 && !t->packed) {
        // one pass over the rows for all shapes, added up on the device
        const int64_t cap = (int64_t)sm_count() * 4;
        u128 *part = scratch.get<u128>((size_t)std::min<int64_t>((n + 255) / 256, cap) * nj);
        u128 *sum = scratch.get<u128>((size_t)nj);
        const TreeletShapes ts = treelet_shapes(h);
        auto pass = [&](int64_t a, int64_t b) {
            const int blocks = (int)std::min<int64_t>((b - a + 255) / 256, cap);
            const dim3 grid((unsigned)blocks, (unsigned)nj);
            if (t->bits == 64)
                MC_LAUNCH("treelet_sum", s, treelet_sum_kernel<uint64_t><<<grid, 256, 0, s>>>(
                                                t->rows(h, 0), a, b, cat.r[h], t->geo.Bc[h], j0, ts, part, err));
            else
                MC_LAUNCH("treelet_sum", s, treelet_sum_kernel<u128><<<grid, 256, 0, s>>>(
                                                t->rows(h, 0), a, b, cat.r[h], t->geo.Bc[h], j0, ts, part, err));
            MC_LAUNCH("treelet_sum", s, part_sum_kernel<<<nj, 256, 0, s>>>(part, blocks, sum, err));
        };
        // a total that does not fit is an error for its ranges too (the build
        // has checked level k)
        if (h < t->k && hi - lo < n) pass(0, n);
        pass(lo, hi);
        MC_CUDA(cudaMemcpyAsync(out.data(), sum, (size_t)nj * sizeof(u128), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaStreamSynchronize(s));
        if (herr) throw Error(MC_E_OVERFLOW, "level total does not fit in 128 bits");
        return out;
    }
    // the level's node prefix, read at the range's ends
    for (int i = 0; i < nj; ++i) {
        const u128 *pre = nullptr;
        if (j0 < 0) {
            pre = t->prefix[h];
        } else {
            uint64_t a0 = 0, a1 = 0;
            for (int q = 0; q < cat.r[h]; ++q)
                if (cat.shapes[cat.gid(h, q)].unrooted == j0 + i) {
                    if (q < 64) a0 |= 1ull << q; else a1 |= 1ull << (q - 64);
                }
            u128 *tot = scratch.get<u128>((size_t)n);
            launch_row_totals(t, h, a0, a1, tot, err, s);
            inclusive_scan_u128(tot, n, err, scratch, s);
            pre = tot;
        }
        u128 top = 0, base = 0;
        MC_CUDA(cudaMemcpyAsync(&top, pre + (hi - 1), sizeof(u128), cudaMemcpyDeviceToHost, s));
        if (lo > 0) MC_CUDA(cudaMemcpyAsync(&base, pre + (lo - 1), sizeof(u128), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaStreamSynchronize(s));
        if (herr) throw Error(MC_E_OVERFLOW, "level total does not fit in 128 bits");
        out[(size_t)i] = top - base;
    }
    return out;
}

// Copies of unrooted shape j from its rooted total: R / h (one rooted copy
// per node), R at a zero-rooted level k, R / a_j at a round-skipped level k
// (a_j = 0: the star, not counted).
u128 mc::unrooted_from_rooted(const mc_tables *t, int h, int j, u128 R)
{
    u128 div = (u128)t->copies_div(h);
    if (t->skip_round && h == t->k) {
        div = (u128)t->copies_k[j];
        if (div == 0) {
            if (R != 0) throw Error(MC_E_INTERNAL, "an uncounted shape has counts");
            return 0;
        }
    }
    if (R % div != 0) throw Error(MC_E_INTERNAL, "rooted total not divisible by h");
    return R / div;
}

extern "C" mc_status mc_total_range(const mc_tables *t, int h, int32_t unrooted_shape, int64_t node_lo,
                                    int64_t node_hi, uint64_t rooted[2], uint64_t unrooted_count[2], void *stream)
{
    return guarded([&] {
        MC_REQUIRE(t && rooted && unrooted_count, "NULL argument");
        refresh_tables(t, (cudaStream_t)stream);
        MC_REQUIRE(h >= 1 && h <= t->k, "h must be in 1..k");
        MC_REQUIRE(!t->level_missing(h), "level h was skipped (round skipping)");
        const ShapeCatalog &cat = shape_catalog();
        MC_REQUIRE(unrooted_shape >= -1 && unrooted_shape < cat.n_unrooted[h], "unrooted shape out of range");
        const int64_t n = t->g->n;
        int64_t lo = node_lo, hi = node_hi;
        if (hi <= 0 && lo <= 0) { lo = 0; hi = n; }
        if (hi <= 0) hi = n;
        MC_REQUIRE(lo >= 0 && lo <= hi && hi <= n, "node range out of bounds");
        cudaStream_t s = (cudaStream_t)stream;
        const u128 R = level_rooted_totals(t, h, unrooted_shape, 1, lo, hi, s)[0];
        u128 U = 0;
        if (unrooted_shape >= 0) {
            U = unrooted_from_rooted(t, h, unrooted_shape, R);
        } else if (t->skip_round && h == t->k) {
            // per-shape divisors differ: t = sum_j R_j / a_j
            const std::vector<u128> Rj = level_rooted_totals(t, h, 0, cat.n_unrooted[h], lo, hi, s);
            for (int j = 0; j < cat.n_unrooted[h]; ++j) U += unrooted_from_rooted(t, h, j, Rj[(size_t)j]);
        } else {
            const u128 div = (u128)t->copies_div(h);
            if (R % div != 0) throw Error(MC_E_INTERNAL, "rooted total not divisible by h");
            U = R / div;
        }
        rooted[0] = (uint64_t)R;
        rooted[1] = (uint64_t)(R >> 64);
        unrooted_count[0] = (uint64_t)U;
        unrooted_count[1] = (uint64_t)(U >> 64);
    });
}

extern "C" mc_status mc_total(const mc_tables *t, int h, int32_t unrooted_shape, uint64_t rooted[2],
                              uint64_t unrooted_count[2], void *stream)
{
    return mc_total_range(t, h, unrooted_shape, 0, 0, rooted, unrooted_count, stream);
}

// ---------------------------------------------------------------------------
// batches: several (graph, colouring) instances side by side as one disjoint
// union, built in one pass (one launch per kernel for the whole batch)
// ---------------------------------------------------------------------------
struct ConcatPart {
    const int64_t *row_ptr;
    const uint32_t *col;
    const uint8_t *colors;
    int64_t noff, eoff;
};

// All instances in one launch (32 launches of 7 us each before, most of them
// a few blocks): a thread finds its element's instance by a binary search of
// the offsets.
__global__ void __launch_bounds__(256) concat_kernel(const ConcatPart *__restrict__ part, int count, int64_t N, int64_t NNZ,
                                                     int64_t *__restrict__ urp, uint32_t *__restrict__ ucol,
                                                     uint8_t *__restrict__ ucolors)
{
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    auto find = [&](auto off, int64_t i) {  // the last instance that starts at or before i
        int lo = 0, hi = count;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off(part[mid]) <= i) lo = mid; else hi = mid;
        }
        return lo;
    };
    for (int64_t i = t0; i < NNZ; i += step) {
        const ConcatPart p = part[find([](const ConcatPart &q) { return q.eoff; }, i)];
        ucol[i] = p.col[i - p.eoff] + (uint32_t)p.noff;
    }
    for (int64_t i = t0; i < N; i += step) {
        const ConcatPart p = part[find([](const ConcatPart &q) { return q.noff; }, i)];
        urp[i] = p.eoff + p.row_ptr[i - p.noff];
        if (ucolors) ucolors[i] = p.colors[i - p.noff];
    }
    if (t0 == 0) urp[N] = NNZ;
}

extern "C" mc_status mc_build_tables_batch(int count, const mc_graph *const *graphs, const uint8_t *const *colors,
                                           int k, int count_bits, uint32_t flags, const mc_allocator *alloc,
                                           void *stream, mc_tables **out, int64_t *node_offsets)
{
    if (out) *out = nullptr;
    mc_graph *ug = nullptr;
    mc_tables *t = nullptr;
    mc_status st = guarded([&] {
        MC_REQUIRE(out && node_offsets && graphs && colors && count >= 1, "bad batch arguments");
        cudaStream_t s = (cudaStream_t)stream;
        std::vector<int64_t> noff(count + 1, 0), eoff(count + 1, 0);
        for (int i = 0; i < count; ++i) {
            MC_REQUIRE(graphs[i] && (colors[i] || graphs[i]->n == 0), "NULL graph or colours in batch");
            noff[i + 1] = noff[i] + graphs[i]->n;
            eoff[i + 1] = eoff[i] + graphs[i]->nnz;
        }
        const int64_t N = noff[count], NNZ = eoff[count];
        MC_REQUIRE(N < (int64_t)0xffffffffLL, "batch has too many nodes");
        Arena scratch(true);
        if (alloc) { scratch.alloc.a = *alloc; scratch.alloc.custom = true; }
        scratch.stream = s;
        int64_t *urp = scratch.get<int64_t>((size_t)N + 1);
        uint32_t *ucol = scratch.get<uint32_t>((size_t)(NNZ > 0 ? NNZ : 1));
        uint8_t *ucolors = scratch.get<uint8_t>((size_t)(N > 0 ? N : 1));
        std::vector<ConcatPart> parts((size_t)count);
        bool on_device = true;  // colours elsewhere (host, another device) are copied one by one
        int dev = 0;
        MC_CUDA(cudaGetDevice(&dev));
        for (int i = 0; i < count; ++i) {
            parts[(size_t)i] = {graphs[i]->row_ptr, graphs[i]->col, colors[i], noff[i], eoff[i]};
            if (graphs[i]->n == 0) continue;
            cudaPointerAttributes at{};
            if (cudaPointerGetAttributes(&at, colors[i]) != cudaSuccess) cudaGetLastError();
            on_device &= (at.type == cudaMemoryTypeDevice && at.device == dev) || at.type == cudaMemoryTypeManaged;
        }
        ConcatPart *dparts = scratch.get<ConcatPart>((size_t)count);
        MC_CUDA(cudaMemcpyAsync(dparts, parts.data(), (size_t)count * sizeof(ConcatPart), cudaMemcpyHostToDevice, s));
        MC_LAUNCH("concat_csr", s, concat_kernel<<<grid_for(std::max(N, NNZ), 256), 256, 0, s>>>(
                                       dparts, count, N, NNZ, urp, ucol, on_device ? ucolors : nullptr));
        if (!on_device)
            for (int i = 0; i < count; ++i)
                if (graphs[i]->n)
                    MC_CUDA(cudaMemcpyAsync(ucolors + noff[i], colors[i], (size_t)graphs[i]->n, cudaMemcpyDefault, s));
        mc_status s2 = mc_load_graph(N, NNZ, urp, ucol, MC_GRAPH_DEVICE_PTRS | MC_GRAPH_TRUSTED, alloc, stream, &ug);
        if (s2 != MC_OK) throw Error(s2, std::string("batch graph: ") + mc_last_error());
        s2 = mc_build_tables(ug, ucolors, k, count_bits, flags, alloc, stream, &t);
        if (s2 != MC_OK) throw Error(s2, std::string("batch build: ") + mc_last_error());
        t->owned_graph = ug;
        ug = nullptr;
        for (int i = 0; i <= count; ++i) node_offsets[i] = noff[i];
    });
    if (st != MC_OK) {
        delete t;
        mc_free_graph(ug);
        return st;
    }
    *out = t;
    return MC_OK;
}

// Number of non-zero entries of a level's n rows.  The first plane is counted
// as one run of 8-byte words, eight in flight per thread; the place in the row
// matters only where rows end in half a word of padding (PAD) and is kept by
// addition.  Where the level has wide rows, a warp then looks up the entries of
// such rows whose low part is zero.  (A division and a look at the row's word per
// entry: 2.14 ms for level 6 of R-MAT 22, k = 7; whole 16-byte counts 1.14.)
template <typename CT, int N, bool PAD>
__global__ void __launch_bounds__(256) nonzeros_kernel(Rows x, int64_t n, bool wide, unsigned long long *count)
{
    constexpr int NW = 8;
    const int wpr = x.s0 / 8;  // words per row
    const int64_t step = (int64_t)gridDim.x * blockDim.x, t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t total = n * wpr;
    int e = PAD ? (int)(t0 % wpr) : 0;
    const int de = PAD ? (int)(step % wpr) : 0;
    unsigned long long c = 0;
    for (int64_t i = t0; i < total; i += NW * step) {
        uint64_t w[NW];
#pragma unroll
        for (int q = 0; q < NW; ++q) w[q] = i + q * step < total ? ((const uint64_t *)x.p0)[i + q * step] : 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            if constexpr (N == 8) {
                c += w[q] != 0;
            } else {
                c += (uint32_t)w[q] != 0;
                if (!PAD || e + 1 < wpr) c += (w[q] >> 32) != 0;
                if (PAD) {
                    e += de;
                    if (e >= wpr) e -= wpr;
                }
            }
        }
    }
    const int lane = threadIdx.x & 31;
    if (wide && N < (int)sizeof(CT)) {
        for (int64_t base = (t0 >> 5) * 32; base < n; base += step) {
            unsigned rows = __ballot_sync(0xffffffffu, base + lane < n && (x.wide[base + lane] & x.bit));
            for (; rows; rows &= rows - 1) {
                const int64_t v = base + __ffs(rows) - 1;
                for (int k = lane; k < x.W; k += 32)
                    c += row_low<CT>(x.low(v), N, k) == 0 && row_rest<CT>(x.high(v), x.W, N, k) != 0;
            }
        }
    }
    for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if (lane == 0 && c) atomicAdd(count, c);
}

template <typename CT> static void launch_nonzeros(const Rows &x, int64_t n, bool wide, unsigned long long *d, cudaStream_t s)
{
    const int grid = grid_for((n * (x.s0 / 8) + 7) / 8, 256);
    auto kern = x.N == 8 ? nonzeros_kernel<CT, 8, false> : x.W % 2 ? nonzeros_kernel<CT, 4, true> : nonzeros_kernel<CT, 4, false>;
    MC_LAUNCH("nonzeros", s, kern<<<grid, 256, 0, s>>>(x, n, wide, d));
}

extern "C" mc_status mc_table_nonzeros(const mc_tables *t, int h, int which, int64_t *count, void *stream)
{
    return guarded([&] {
        MC_REQUIRE(t && count, "NULL argument");
        refresh_tables(t, (cudaStream_t)stream);
        MC_REQUIRE(which == 0 || which == 1, "which must be 0 (c) or 1 (S)");
        MC_REQUIRE(h >= 1 && h <= (which ? t->k - 1 : t->k), "h out of range");
        MC_REQUIRE(!t->level_missing(h), "level h was skipped (round skipping)");
        const int64_t n = t->g->n;
        if (which == 0 && h == 1) { *count = n; return; }
        cudaStream_t s = (cudaStream_t)stream;
        if (t->packed) {  // the packed level holds exactly its non-zero entries
            int64_t c = 0;
            if (n) {
                MC_CUDA(cudaMemcpyAsync(&c, (which ? t->ps : t->pc)[h].off + n, sizeof(int64_t),
                                        cudaMemcpyDeviceToHost, s));
                MC_CUDA(cudaStreamSynchronize(s));
            }
            *count = c;
            return;
        }
        Arena scratch(true);
        scratch.alloc = t->arena.alloc;
        scratch.stream = s;
        unsigned long long *d = scratch.get<unsigned long long>(1), hc = 0;
        MC_CUDA(cudaMemsetAsync(d, 0, sizeof(*d), s));
        const Rows src = t->rows(h, which);
        if (n > 0) {
            const bool wide = t->wide_levels & src.bit;
            if (t->bits == 64) launch_nonzeros<uint64_t>(src, n, wide, d, s);
            else launch_nonzeros<u128>(src, n, wide, d, s);
        }
        MC_CUDA(cudaMemcpyAsync(&hc, d, sizeof(hc), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaStreamSynchronize(s));
        *count = (int64_t)hc;
    });
}

extern "C" mc_status mc_table_layout(const mc_tables *t, int h, int which, int64_t *row_entries,
                                     int *entry_bytes)
{
    return guarded([&] {
        MC_REQUIRE(t, "tables is NULL");
        MC_REQUIRE(which == 0 || which == 1, "which must be 0 (c) or 1 (S)");
        MC_REQUIRE(h >= 1 && h <= (which ? t->k - 1 : t->k), "h out of range");
        MC_REQUIRE(!t->level_missing(h), "level h was skipped (round skipping)");
        if (row_entries) *row_entries = which ? t->geo.Ws[h] : t->geo.Wc[h];
        if (entry_bytes) *entry_bytes = t->bits / 8;
    });
}

// Rows v0 .. v0 + cnt of a dense level as plain counts.
template <typename CT>
__global__ void __launch_bounds__(256) expand_kernel(Rows x, int64_t v0, int64_t total, CT *__restrict__ dst)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = total <= 0xffffffffll ? (int64_t)((uint32_t)i / (uint32_t)x.W) : i / x.W;
        dst[i] = entry_at<CT>(x, v0 + v, (int)(i - v * x.W));
    }
}

static void launch_expand(const mc_tables *t, int h, int which, int64_t v0, int64_t cnt, void *dst, cudaStream_t s)
{
    const Rows x = t->rows(h, which);
    const int64_t total = cnt * x.W;
    if (total == 0) return;
    if (t->bits == 64)
        MC_LAUNCH("expand", s, expand_kernel<uint64_t><<<grid_for(total, 256), 256, 0, s>>>(x, v0, total, (uint64_t *)dst));
    else
        MC_LAUNCH("expand", s, expand_kernel<u128><<<grid_for(total, 256), 256, 0, s>>>(x, v0, total, (u128 *)dst));
}

// Rows v0 .. v0 + rows of a dense level put together from their planes on the
// host, into host memory.
static void read_planes(const mc_tables *t, int h, int which, int64_t v0, int64_t rows, uint8_t *dst, cudaStream_t s)
{
    const Rows x = t->rows(h, which);
    const int cb = t->bits / 8;
    const int64_t end = v0 + rows, step = std::max<int64_t>(1, ((int64_t)16 << 20) / (x.s0 + x.s1 + 4));
    std::vector<uint8_t> low, high;
    std::vector<uint32_t> wide;
    for (; v0 < end; v0 += step) {
        const int64_t cnt = std::min(step, end - v0);
        low.resize((size_t)(cnt * x.s0));
        high.resize((size_t)(cnt * x.s1) + 1);
        wide.resize((size_t)cnt);
        MC_CUDA(cudaMemcpyAsync(low.data(), x.low(v0), (size_t)(cnt * x.s0), cudaMemcpyDeviceToHost, s));
        if (x.s1) MC_CUDA(cudaMemcpyAsync(high.data(), x.high(v0), (size_t)(cnt * x.s1), cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaMemcpyAsync(wide.data(), x.wide + v0, (size_t)cnt * 4, cudaMemcpyDeviceToHost, s));
        MC_CUDA(cudaStreamSynchronize(s));
        for (int64_t v = 0; v < cnt; ++v)
            for (int e = 0; e < x.W; ++e, dst += cb) {
                const uint8_t *up = high.data() + v * x.s1;
                std::memset(dst, 0, (size_t)cb);
                std::memcpy(dst, low.data() + v * x.s0 + e * x.N, (size_t)x.N);
                if (!(wide[(size_t)v] & x.bit) || x.N == cb) continue;
                if (cb == 16) std::memcpy(dst + 8, up + 8 * e, 8);
                if (x.N == 4) std::memcpy(dst + 4, up + (cb == 16 ? 8 * x.W : 0) + 4 * e, 4);
            }
    }
}

// Whether kernels may store whole counts at dst: memory of this device,
// aligned to a count.  Other device destinations (any address, memory of
// another device) are reached by copies.
static bool stores_counts(const void *dst, size_t count_bytes)
{
    int dev = 0;
    MC_CUDA(cudaGetDevice(&dev));
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, dst) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return ((at.type == cudaMemoryTypeDevice && at.device == dev) || at.type == cudaMemoryTypeManaged) &&
           (uintptr_t)dst % count_bytes == 0;
}

extern "C" mc_status mc_read_table(const mc_tables *t, int h, int which, void *dst, size_t dst_bytes,
                                   int dst_on_device, void *stream)
{
    return guarded([&] {
        MC_REQUIRE(t && dst, "NULL argument");
        refresh_tables(t, (cudaStream_t)stream);
        MC_REQUIRE(which == 0 || which == 1, "which must be 0 (c) or 1 (S)");
        MC_REQUIRE(h >= 1 && h <= (which ? t->k - 1 : t->k), "h out of range");
        MC_REQUIRE(!t->level_missing(h), "level h was skipped (round skipping)");
        const int64_t W = which ? t->geo.Ws[h] : t->geo.Wc[h], n = t->g->n;
        const size_t cb = t->bits / 8, bytes = (size_t)n * W * cb;
        MC_REQUIRE(dst_bytes >= bytes, "dst too small");
        cudaStream_t s = (cudaStream_t)stream;
        if (bytes == 0) return;
        const bool ones = which == 0 && h == 1, dense = !ones && !t->packed;
        const Rows x = t->rows(h, which);
        const cudaMemcpyKind kind = dst_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
        Arena scratch(true);
        scratch.alloc = t->arena.alloc;
        scratch.stream = s;
        if (dst_on_device && stores_counts(dst, cb)) {
            if (ones)
                MC_LAUNCH("fill_ones", s, fill_ones_kernel<<<grid_for(n, 256), 256, 0, s>>>(dst, n, (int)cb));
            else if (t->packed)
                launch_unpack(t, h, which, dst, s);
            else
                launch_expand(t, h, which, 0, n, dst, s);
        } else if (dense && x.N == (int)cb) {  // the first plane is the rows as they are
            MC_CUDA(cudaMemcpyAsync(dst, x.p0, bytes, kind, s));
        } else if (ones) {
            std::vector<uint8_t> one;
            uint8_t *at = (uint8_t *)dst;
            if (dst_on_device) {
                one.resize(bytes);
                at = one.data();
            }
            std::memset(at, 0, bytes);
            for (int64_t v = 0; v < n; ++v) at[v * (int64_t)cb] = 1;
            if (dst_on_device) {
                MC_CUDA(cudaMemcpyAsync(dst, at, bytes, cudaMemcpyHostToDevice, s));
                MC_CUDA(cudaStreamSynchronize(s));
            }
        } else if (t->packed) {
            void *tmp = scratch.get<uint8_t>(bytes);
            launch_unpack(t, h, which, tmp, s);
            MC_CUDA(cudaMemcpyAsync(dst, tmp, bytes, kind, s));
        } else if (!dst_on_device && bytes <= 256 * 1024 && !(t->wide_levels & x.bit)) {
            // a small level: its first plane copied and widened here, without
            // scratch and a launch (0.020 against 0.027 ms for a 1k-node graph)
            std::vector<uint8_t> low((size_t)(n * x.s0));
            MC_CUDA(cudaMemcpyAsync(low.data(), x.p0, low.size(), cudaMemcpyDeviceToHost, s));
            MC_CUDA(cudaStreamSynchronize(s));
            uint8_t *at = (uint8_t *)dst;
            auto widen_rows = [&](auto from) {
                for (int64_t v = 0; v < n; ++v)
                    for (int e = 0; e < x.W; ++e, at += cb) {
                        std::memcpy(&from, low.data() + v * x.s0 + e * sizeof(from), sizeof(from));
                        const uint64_t y[2] = {from, 0};
                        if (cb == 8) std::memcpy(at, y, 8);
                        else std::memcpy(at, y, 16);
                    }
            };
            if (x.N == 4) widen_rows((uint32_t)0);
            else widen_rows((uint64_t)0);
        } else {
            // through a scratch buffer of up to 256 MB (each further copy into host
            // pages not touched before costs some 0.5 ms beside its bytes), without
            // one from the planes as they are
            const int64_t row = W * (int64_t)cb;
            const int64_t step = std::max<int64_t>(1, std::min<int64_t>(n, ((int64_t)256 << 20) / row));
            void *tmp = nullptr;
            std::vector<uint8_t> host;
            try {
                tmp = scratch.get<uint8_t>((size_t)(step * row));
            } catch (const Error &) {
                if (dst_on_device) host.resize((size_t)(step * row));
            }
            for (int64_t v = 0; v < n; v += step) {
                const int64_t cnt = std::min(step, n - v);
                uint8_t *at = (uint8_t *)dst + v * row;
                if (tmp) {
                    launch_expand(t, h, which, v, cnt, tmp, s);
                    MC_CUDA(cudaMemcpyAsync(at, tmp, (size_t)(cnt * row), kind, s));
                } else {
                    read_planes(t, h, which, v, cnt, dst_on_device ? host.data() : at, s);
                    if (dst_on_device) {
                        MC_CUDA(cudaMemcpyAsync(at, host.data(), (size_t)(cnt * row), cudaMemcpyHostToDevice, s));
                        MC_CUDA(cudaStreamSynchronize(s));
                    }
                }
            }
        }
        MC_CUDA(cudaStreamSynchronize(s));
    });
}

extern "C" mc_status mc_autotune(int mode, const char *cache_file)
{
    return guarded([&] {
        MC_REQUIRE(mode >= 0 && mode <= 2, "mode must be 0, 1 or 2");
        TuneState &st = tune_state();
        std::lock_guard<std::mutex> lock(st.mu);
        tune_env_locked(st);
        st.mode = mode;
        if (mode == 2) st.retuned.clear();
        if (cache_file) {  // "" stops appending
            st.file = cache_file;
            if (!st.file.empty()) tune_load_file_locked(st, st.file);
        }
    });
}

extern "C" int mc_autotune_choice(int kind, int k, int count_bits, int h, int64_t n, int64_t nnz, int64_t max_degree)
{
    const TuneKey key = tune_key(kind, k, count_bits, h, n, nnz, max_degree);
    TuneState &st = tune_state();
    std::lock_guard<std::mutex> lock(st.mu);
    tune_env_locked(st);
    auto it = st.latest.find(key);
    return it == st.latest.end() ? -1 : it->second;
}

extern "C" mc_status mc_autotune_set(int kind, int k, int count_bits, int h, int64_t n, int64_t nnz,
                                     int64_t max_degree, int choice)
{
    return guarded([&] {
        MC_REQUIRE(kind == 0 || kind == 1, "kind must be 0 (neighbour sums) or 1 (merge)");
        MC_REQUIRE(choice >= 0 && choice < candidates(kind), "no such schedule");
        const TuneKey key = tune_key(kind, k, count_bits, h, n, nnz, max_degree);
        TuneState &st = tune_state();
        std::lock_guard<std::mutex> lock(st.mu);
        tune_env_locked(st);
        for (auto it = st.choice.lower_bound(key); it != st.choice.end() && !(key < it->first.any());)
            it = st.choice.erase(it);  // every layout's
        st.pinned[key] = st.latest[key] = choice;
    });
}
