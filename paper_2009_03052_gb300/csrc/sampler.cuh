// sampler.cuh -- the treelet samplers (Section 2.2; sample(T) of Section 4.1)
// and the classification of their samples (Section 4.4.3): kernels shared by
// the translation units that instantiate them (sampler_*.cu) and the host code.
#pragma once

#include "internal.h"

namespace mc {

enum : int { SERR_SEARCH = 1, SERR_CLASS = 2 };

// Position of the pair (i, j), i < j, in the adjacency word of an h-node graph.
__host__ __device__ __forceinline__ int pair_pos(int h, int i, int j)
{
    const int P = h * (h - 1) / 2;
    return P - 1 - (i * (2 * h - i - 1) / 2 + (j - i - 1));
}

// ---------------------------------------------------------------------------
// Sampler.
//   step 0  X = uniform(R); v = first node whose inclusive prefix exceeds X;
//           (T, C) = first entry of v's level-h row, in (shape id, colour
//           mask) order, whose running sum exceeds the remainder;
//   step s  for each decomposition node (T, C, x) in pre-order (T' before
//           T''): Y = uniform(beta_T c(T_C, x)); the block of colour sets
//           C'' (ascending mask) is found from the block weights
//           c(T'_{C\C''}, x) S(T'', C'', x); inside it, the neighbour u
//           (ascending) is the first whose running sum of c(T''_{C''}, u)
//           exceeds floor(Y' / c(T'_{C\C''}, x)) -- the same pair as a flat
//           scan over (C'', u) with weights c(T') c(T'').
// The h leaves of the decomposition are the sample's nodes; their induced
// subgraph is classified by the lookup table.
// ---------------------------------------------------------------------------
// One treelet's part of a launch that draws from several treelets: samples
// [end of the previous part, end) come from this root index, the first with
// sample index first_index.
struct SampleSeg {
    int64_t end;
    uint64_t first_index;
    const u128 *prefix;
    const uint32_t *bucket;
    u128 R, Xbase, D;
    uint64_t allow0, allow1;
};
static_assert(sizeof(SampleSeg) <= 128, "request admission charges 128 bytes per part");

struct SampleArgs {
    const int64_t *row_ptr;
    const uint32_t *col;
    const uint8_t *colors;
    const uint8_t *ecol;
    const uint32_t *scol;
    const int32_t *coff;
    int64_t n;
    Rows c[MAXK + 1], S[MAXK + 1];  // the levels of dense tables
    const uint32_t *wide;       // per node, the levels at which its row is wide
    uint32_t levels;            // the levels that have wide rows
    PackedView pc[MAXK + 1], ps[MAXK + 1];  // the levels of packed (succinct) tables
    const void *Sp[MAXK + 1];   // per level: inclusive prefix of each hub's chunk sums
    const int32_t *node_chunk0; // first chunk of a hub, -1 for other nodes
    int Bc[MAXK + 1], Bs[MAXK + 1], Wc[MAXK + 1], Ws[MAXK + 1];
    int R_[MAXK + 1];           // rooted shapes per size: rows are set-major, entry (set, shape) at set * R_ + shape
    int k, h;
    const u128 *prefix;
    u128 R;                     // total of the node range sampled from
    u128 Xbase;                 // prefix before that range (0 for the whole graph)
    const uint32_t *bucket;     // root-search buckets (nb + 1 entries)
    u128 D;                     // bucket width
    uint64_t allow0, allow1;
    const SampleSeg *seg;       // nseg > 0: the launch's parts, each with its own root index and
    int nseg;                   // index stream (prefix .. allow1 above unused)
    int first[MAXK + 2];
    uint8_t sz[MAX_SHAPES], loc[MAX_SHAPES], lft[MAX_SHAPES], rgt[MAX_SHAPES], beta[MAX_SHAPES];
    uint8_t crank[1 << (MAXK - 1)];        // colex rank of a set of the k-1 relative colours
    uint8_t unrank[MAXK][36];              // i-th m-subset (ascending masks)
    uint8_t pi[28], pj[28];
    uint64_t seed, first_index;
    int64_t begin, count;       // samples [begin, count) of the call
    uint32_t *found, *par;      // split sampling: nodes and parents of the samples from `begin` on
    const uint16_t *lut;
    uint32_t *nodes, *roots;
    int32_t *shapes, *classes;
    unsigned long long *hist;
    unsigned long long *bytes;  // when set: data bytes read and written, counted item by item
    unsigned long long *next;   // when set: warps take batches of 32 samples from this counter
                                // (zero at launch) as they finish; else a fixed grid stride
    int ncls;
    bool long_rows;             // adjacency offsets beyond 32 bits
    int *err;
};

// What the descent looks up by shape and by level, in shared memory: the
// lanes of a warp are at different shapes and levels, and constant memory
// serves one address at a time.
struct SampleSmem {
    uint8_t crank[1 << (MAXK - 1)];
    uint8_t unrank[MAXK][36];
    uint8_t pair[32];                   // per bit of the adjacency word: i | j << 4
    uint2 shape[MAX_SHAPES];            // size | local id << 8 | beta << 16; T' | T'' << 8
    uint4 level[2][MAXK + 1];           // c, S: first-plane base, row stride, N | has wide rows << 8
    uint4 upper[2][MAXK + 1];           // their second planes: base, row stride, counts per row
    int r[MAXK + 1];                    // rooted shapes per size
};

template <int T> __device__ __forceinline__ void fill_sample_smem(const SampleArgs &a, SampleSmem &sm)
{
    for (int i = threadIdx.x; i < (1 << (MAXK - 1)); i += T) sm.crank[i] = a.crank[i];
    for (int i = threadIdx.x; i < MAXK * 36; i += T) (&sm.unrank[0][0])[i] = (&a.unrank[0][0])[i];
    for (int i = threadIdx.x; i < MAX_SHAPES; i += T)
        sm.shape[i] = make_uint2((uint32_t)a.sz[i] | (uint32_t)a.loc[i] << 8 | (uint32_t)a.beta[i] << 16,
                                 (uint32_t)a.lft[i] | (uint32_t)a.rgt[i] << 8);
    for (int i = threadIdx.x; i < 2 * (MAXK + 1); i += T) {
        const int l = i % (MAXK + 1);
        const Rows &r = i > MAXK ? a.S[l] : a.c[l];
        sm.level[i / (MAXK + 1)][l] = make_uint4((uint32_t)(uint64_t)r.p0, (uint32_t)((uint64_t)r.p0 >> 32), (uint32_t)r.s0,
                                                 (uint32_t)r.N | ((a.levels & r.bit) ? 256u : 0u));
        sm.upper[i / (MAXK + 1)][l] = make_uint4((uint32_t)(uint64_t)r.p1, (uint32_t)((uint64_t)r.p1 >> 32), (uint32_t)r.s1,
                                                 (uint32_t)r.W);
        if (i <= MAXK) sm.r[l] = a.R_[l];
    }
    const int h = a.h, P = h * (h - 1) / 2;
    if (threadIdx.x < P)
        sm.pair[pair_pos(h, a.pi[threadIdx.x], a.pj[threadIdx.x])] = (uint8_t)(a.pi[threadIdx.x] | a.pj[threadIdx.x] << 4);
}

// Row x of level h of c (which = 0) or S (1): entry get(idx) of dense rows, or
// (PK) by a binary search of the packed row's keys.  full(idx) adds the upper
// part of a row that is wide, in line, so that the items of a scan are in flight
// together.  (Reading the upper part before the row is known to be wide, for a
// shorter chain of loads, was slower at every launch size: 20k samples of R-MAT
// 22, k = 7, 0.444 against 0.409 ms, 1M 3.13 against 2.56.)
template <typename CT, bool PK> struct RowRef {
    const SampleArgs &a;
    const SampleSmem &sm;
    const uint8_t *low;
    int64_t x;
    int h, N, which;
    bool wide;
    __device__ __forceinline__ RowRef(const SampleArgs &a_, const SampleSmem &sm_, int which_, int h_, int64_t x_)
        : a(a_), sm(sm_), low(nullptr), x(x_), h(h_), N(8), which(which_), wide(false)
    {
        if constexpr (!PK) {
            const uint4 l = sm.level[which][h];
            low = (const uint8_t *)(((uint64_t)l.y << 32) | l.x) + x * (uint64_t)l.z;
            N = (int)(l.w & 255u);
            if (l.w >> 8) wide = (a.wide[x] >> (which ? 16 + h : h)) & 1u;
        }
    }
    // entry idx of a row that is not wide
    __device__ __forceinline__ CT get(int idx) const
    {
        if constexpr (PK) return (CT)packed_get(which ? a.ps[h] : a.pc[h], x, idx);
        else return row_low_any<CT>(low, N, idx);
    }
    // of one entry (byte counting)
    __device__ __forceinline__ int bytes() const { return wide ? (int)sizeof(CT) : N; }
    __device__ __forceinline__ CT rest(int idx) const
    {
        const uint4 u = sm.upper[which][h];
        return row_rest<CT>((const uint8_t *)(((uint64_t)u.y << 32) | u.x) + x * (uint64_t)u.z, (int)u.w, N, idx);
    }
    __device__ __forceinline__ CT full(int idx) const
    {
        CT v = row_low_any<CT>(low, N, idx);
        if (wide) v |= rest(idx);
        return v;
    }
};

// Entries of rows that may be wide (dense tables), out of line: few levels of
// few tables have any, and the sampler is large for the instruction cache.
template <typename CT> __device__ __noinline__ CT entry_wide(const SampleArgs &a, int which, int h, int64_t x, int idx)
{
    return entry_at<CT>(which ? a.S[h] : a.c[h], x, idx);
}

__device__ __forceinline__ uint64_t quotient(uint64_t a, uint64_t b) { return a / b; }
__device__ __forceinline__ u128 quotient(u128 a, u128 b)
{
    return ((a >> 64) == 0 && (b >> 64) == 0) ? (u128)((uint64_t)a / (uint64_t)b) : a / b;
}

// The positions of a mask's set bits, four bits each, and the set bits that an
// index mask selects (bit i of im: the i-th lowest).
__device__ __forceinline__ uint32_t bit_positions(unsigned m)
{
    uint32_t p = 0;
    for (int i = 0; m; ++i, m &= m - 1) p |= (uint32_t)(__ffs(m) - 1) << (4 * i);
    return p;
}
__device__ __forceinline__ unsigned select_bits(unsigned im, uint32_t pos)
{
    unsigned out = 0;
    for (; im; im &= im - 1) out |= 1u << ((pos >> (4 * (__ffs(im) - 1))) & 15u);
    return out;
}

// Per-lane search: over items 0 .. len-1 in order, the first whose running
// sum of val(i) exceeds q (-1 if none), `before` the running sum before it.
// Items are loaded NW at a time so that their loads are in flight together.
template <int NW, typename V, typename F>
__device__ __forceinline__ int lane_first_exceeding(int len, V q, F val, V &before)
{
    V run = 0;
    for (int b = 0; b < len; b += NW) {
        V v[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) v[i] = b + i < len ? val(b + i) : (V)0;
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            if (b + i < len && run + v[i] > q) { before = run; return b + i; }
            run += v[i];
        }
    }
    return -1;
}

// The first index i in [lo, hi) with pred(i) true, for a predicate that is
// false then true along the range (hi if it is never true).  K = 1: binary
// search; K > 1: K probes per round, evenly spaced, all loads in flight
// together (about log_{K+1} of the range in dependent rounds).  on_probe()
// runs once per evaluated probe.
template <int K, typename P, typename F>
__device__ __forceinline__ int64_t first_true(int64_t lo, int64_t hi, P pred, F on_probe)
{
    if constexpr (K == 1) {
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            on_probe();
            if (pred(mid)) hi = mid; else lo = mid + 1;
        }
        return lo;
    } else {
        while (hi - lo > K) {
            const int64_t step = (hi - lo) / (K + 1);
            bool t[K];
#pragma unroll
            for (int i = 0; i < K; ++i) { t[i] = pred(lo + (i + 1) * step); on_probe(); }
            int64_t nlo = lo + K * step + 1, nhi = hi;
#pragma unroll
            for (int i = K - 1; i >= 0; --i)
                if (t[i]) { nhi = lo + (i + 1) * step; nlo = i ? lo + i * step + 1 : lo; }
            lo = nlo;
            hi = nhi;
        }
        bool t[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            t[i] = lo + i < hi ? pred(lo + i) : true;
            if (lo + i < hi) on_probe();
        }
#pragma unroll
        for (int i = K - 1; i >= 0; --i)
            if (t[i]) hi = lo + i;
        return hi;
    }
}

// Byte counts of the sampler's accesses, compiled in only when CNT: rb the
// bytes of the data items, rs the same accesses in 32-byte sectors (32 bytes
// per random access, contiguous runs by their bytes).
#define MC_COUNT(item, sector)           \
    do {                                 \
        if constexpr (CNT) {             \
            rb += (uint64_t)(item);      \
            rs += (uint64_t)(sector);    \
        }                                \
    } while (0)

// Lane-per-sample sampler: the 32 lanes of a warp draw 32 samples and walk
// their h-1 decomposition steps in lockstep (every h-treelet has h-1 internal
// decomposition nodes).  A lane does its own scalar work, short scans and
// binary searches (a hub's chunk by the prefix sums of its chunks).  CT: the
// tables' count type; V: the type of the descent's weights, draws and
// running sums (64 bits when every level total leaves room for beta, else
// 128 bits).
//
// A sample's node list, its stack of decomposition nodes (one word each:
// shape, colour set, root colour, root's place in the node list) and the
// adjacency offsets of its nodes live in shared memory, one column per
// thread: indexed per lane, they would be local memory, whose 464 bytes per
// thread times 1536 threads per SM passed through L1 and L2 beside the
// tables (half a gigabyte of DRAM writes per million samples).
//
// Bound by the latency of dependent random reads.  Occupancy target: 3 blocks
// of 512 per SM, 2 for 128-bit counts in dense tables (a wider state: 15.7
// against 22.7 ms for the launches of a 2M-sample adaptive run at k = 7 on
// R-MAT 19; packed rows 0.83 against 1.05 ms the other way, 200k samples,
// k = 6).  Items of a scan in flight: 2 for the narrower states (0.75 ms per 1M
// samples of Chung-Lu 1M, k = 5; 4: 0.88, 1: 0.82, 3: 0.80), 4 for 128-bit
// counts in dense tables (12.9 ms for the adaptive run; 2: 13.6, 8: 19.9).
// LAT (launches too small to fill the GPU): no register cap, 16 items of a scan
// (4 of packed rows, each a search of its own) and 8 adjacency searches in flight
// per lane, so each sample's chain of dependent loads is shorter.  FEW (packed
// rows, launches of at most 2 blocks per SM): registers for 2 blocks, the third
// would not run.  Packed rows, k = 6, Chung-Lu 200k, 128 bits, ms with estimates:
// 20k samples 0.744 in the latency mode, 0.880 without either (0.777 with the
// state in local memory), 100k 0.772 with FEW, 0.870 without (0.769).  The samples
// are the same in every mode.  SPLIT: the nodes and their parents go to memory and
// classify_kernel takes over, so that the searches of the classification neither
// hold the sampler's registers nor wait in the divergence of its warps (ms with
// estimates, split / one kernel: 10M samples at k = 6 14.1 / 15.1, 1M at k = 7,
// R-MAT 19, 1.99 / 2.20, 1M at k = 5 1.00 / 1.01; with the state in local memory
// 1.21).
// WD > 0 (128-bit dense tables with wide rows below level h): counts above 64 bits
// carry most of the weight, so most samples pass through wide rows; their entries
// are read in line, low and upper parts and the wide words of WD neighbours in
// flight, where the other kernels call entry_wide one at a time.  R-MAT 22, k = 7,
// ms with estimates (by calls / in line / whole 16-byte counts): 10M samples 31.6
// / 22.6 / 27.9, 1M 3.25 / 2.56 / 2.92, all split; 100k 0.58 / 0.518 / 0.516; 20k
// (latency mode) 0.465 / 0.413 / 0.413; without split scratch 1M 4.03 / 3.42 /
// 3.11.  WD: 3 where split sampling fills the GPU more than once (10M: 4 in flight
// 23.5), else 4 (100k: 3 in flight 0.569; latency mode: 8 0.455, 16 0.485; without
// split scratch 1M: 3 3.66, 5 3.71).
constexpr int SAMPLE_WORDS = 3 * MAXK;  // shared words per thread
constexpr int SAMPLE_BLOCK = 512, SAMPLE_BLOCK_LAT = 64;

template <typename CT, typename V, bool PK, bool LAT, bool CNT, bool SPLIT, int WD = 0, bool FEW = false>
__global__ void __launch_bounds__(LAT ? SAMPLE_BLOCK_LAT : SAMPLE_BLOCK, LAT ? 1 : ((sizeof(CT) == 16 && !PK) || FEW ? 2 : 3))
    sample_kernel(const __grid_constant__ SampleArgs a)
{
    constexpr int NW = WD ? WD : LAT ? (PK ? 4 : 16) : sizeof(CT) == 16 && !PK ? 4 : 2;  // items of a scan in flight
    constexpr int NQ = LAT ? 8 : 4;   // adjacency searches in flight
    constexpr int KS = LAT ? 8 : 1;   // probes per round of the root and hub chunk searches
    constexpr int T = LAT ? SAMPLE_BLOCK_LAT : SAMPLE_BLOCK;
    extern __shared__ uint32_t s_dyn[];
    uint32_t *const stk = s_dyn + threadIdx.x;             // entry i at i * T; after the descent the degrees
    uint32_t *const nod = s_dyn + MAXK * T + threadIdx.x;  // the nodes, in order of discovery
    uint32_t *const off = s_dyn + 2 * MAXK * T + threadIdx.x;  // their adjacency offsets (low words)
    unsigned int *const s_hist = s_dyn + SAMPLE_WORDS * T;
    __shared__ SampleSmem sm;
    const int h = a.h, P = h * (h - 1) / 2;
    fill_sample_smem<T>(a, sm);
    if (a.hist && !SPLIT)
        for (int i = threadIdx.x; i < a.ncls; i += T) s_hist[i] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)T + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * T) >> 5;
    constexpr int CB = (int)sizeof(CT);
    bool bad = false;
    uint64_t rb = 0, rs = 0;  // byte counts (CNT): data items, 32-byte sectors
    // a warp's next batch of 32 samples: from the shared counter (the warps
    // that draw cheap samples take more batches, so they end together), or
    // every nwarps-th batch
    auto take = [&](int64_t after) -> int64_t {
        if (!a.next) return after < 0 ? warp * 32 : after + nwarps * 32;
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(a.next, 32ull);
        return (int64_t)__shfl_sync(0xffffffffu, b, 0);
    };
    auto entry = [](int g, unsigned C, int cx, int at) {
        return (uint32_t)g | C << 8 | (uint32_t)cx << 16 | (uint32_t)at << 20;
    };
    for (int64_t base = a.begin + take(-1); base < a.count; base = a.begin + take(base - a.begin)) {
        const int64_t sid = base + lane;
        bool ok = sid < a.count;
        uint64_t index = a.first_index + (uint64_t)sid;
        uint32_t v = 0;
        int s0 = 0, sp = 0, nn = 0;
        uint32_t par = 0;  // per node, four bits: its parent's place in the node list
        {
            const u128 *prefix = a.prefix;
            const uint32_t *bucket = a.bucket;
            u128 R = a.R, Xbase = a.Xbase, D = a.D;
            uint64_t allow0 = a.allow0, allow1 = a.allow1;
            if (a.nseg > 0 && ok) {  // the part this sample falls in
                int g = 0;
                while (g + 1 < a.nseg && sid >= a.seg[g].end) ++g;
                const SampleSeg &sg = a.seg[g];
                index = sg.first_index + (uint64_t)(sid - (g ? a.seg[g - 1].end : 0));
                prefix = sg.prefix;
                bucket = sg.bucket;
                R = sg.R;
                Xbase = sg.Xbase;
                D = sg.D;
                allow0 = sg.allow0;
                allow1 = sg.allow1;
            }
            // ---- root: X = uniform(R); v = first node with prefix[v] > X, found
            // by binary search inside the bucket of X
            V X = 0;
            if (ok && !draw_below(a.seed, index, 0, (V)R, X)) { ok = false; bad = true; }
            X += (V)Xbase;  // a node range: the draw lands inside its part of the prefix
            if (ok) {
                const uint64_t bk = (uint64_t)(X / (V)D);
                const int64_t blo = bucket[bk], bhi = bucket[bk + 1];
                MC_COUNT(8, 32);
                const int64_t lo = first_true<KS>(
                    blo, bhi, [&](int64_t i) { return prefix[i] > (u128)X; }, [&] { MC_COUNT(16, 32); });
                MC_COUNT(32, 32);  // the check below and prefix[v - 1]
                v = (uint32_t)lo;
                if (!(prefix[v] > (u128)X)) { ok = false; bad = true; }
            }
            // ---- entry of v's level-h row, in (shape id, colour mask) order
            if (ok) {
                const V rem = X - (v ? (V)prefix[v - 1] : (V)0);
                const int Bc = a.Bc[h], Rh = a.R_[h];
                const RowRef<CT, PK> row(a, sm, 0, h, v);
                V bf;
                // e runs in (shape id, colour mask) order; the row is set-major
                auto scan = [&](auto at) {
                    return lane_first_exceeding<NW, V>(a.Wc[h], rem, [&](int e) -> V {
                        const int sh = e / Bc;
                        const bool al = sh < 64 ? (allow0 >> sh) & 1 : (allow1 >> (sh - 64)) & 1;
                        MC_COUNT(al ? row.bytes() : 0, al ? row.bytes() : 0);  // one contiguous row
                        return al ? (V)at((e - sh * Bc) * Rh + sh) : (V)0;
                    }, bf);
                };
                int found;
                if (!PK && CB == 16 && sm.level[0][h].w >> 8) found = scan([&](int i) { return row.full(i); });
                else if (!PK && row.wide) found = scan([&](int i) { return entry_wide<CT>(a, 0, h, v, i); });
                else found = scan([&](int i) { return row.get(i); });
                if (found < 0) { ok = false; bad = true; }
                else {
                    const int cv = a.colors[v];
                    s0 = found / Bc;
                    const unsigned C = (1u << cv) | insert_colour_gap(sm.unrank[h - 1][found % Bc], cv);
                    stk[0] = entry(a.first[h] + s0, C, cv, 0);
                    nod[0] = v;
                    sp = nn = 1;
                }
            }
        }
        // ---- descent: decomposition nodes in pre-order (T' before T'')
        for (uint32_t step = 1; step < (uint32_t)h; ++step) {
            uint2 sg = make_uint2(0, 0);
            uint32_t en = 0, x = 0;
            if (ok) {  // leaves on top of the stack are done
                for (;;) {
                    if (sp <= 0 || nn >= MAXK) { ok = false; bad = true; break; }
                    en = stk[--sp * T];
                    sg = sm.shape[en & 255u];
                    if ((sg.x & 255u) > 1) break;
                }
            }
            const int cx = (int)(en >> 16 & 15u), at = (int)(en >> 20);
            const unsigned C = en >> 8 & 255u;
            int ga = 0, gb = 0, hb = 1, lb = 0, sidx = 0, chunk0 = -1;
            unsigned C2 = 0;
            int64_t e0 = 0, deg = 0;
            CT q = 0;
            if (ok) {
                x = nod[at * T];
                ga = (int)(sg.y & 255u);
                gb = (int)(sg.y >> 8 & 255u);
                const uint32_t sa = sm.shape[ga].x, sb = sm.shape[gb].x;
                const int hg = (int)(sg.x & 255u), ha = (int)(sa & 255u), la = (int)(sa >> 8 & 255u);
                hb = (int)(sb & 255u);
                lb = (int)(sb >> 8 & 255u);
                e0 = a.row_ptr[x];
                deg = a.row_ptr[x + 1] - e0;
                chunk0 = a.node_chunk0[x];
                // colour sets relative to x: c_x deleted from the palette
                const unsigned rest = drop_colour(C & ~(1u << cx), cx);
                V Y = 0;
                const RowRef<CT, PK> rg(a, sm, 0, hg, x);
                MC_COUNT(16 + 4 + rg.bytes(), 96);  // row offsets, first chunk, c(T_C, x)
                const int ig = sm.crank[rest] * sm.r[hg] + (int)(sg.x >> 8 & 255u);
                const V W = (V)(sg.x >> 16 & 255u) *
                            (V)(WD ? rg.full(ig) : !PK && rg.wide ? entry_wide<CT>(a, 0, hg, x, ig) : rg.get(ig));
                if (!draw_below(a.seed, index, step, W, Y)) { ok = false; bad = true; }
                if (ok) {
                    // block of C'' (ascending mask), weights c(T'_{C\C''}, x) S(T'', C'', x)
                    const uint32_t pos = bit_positions(rest);
                    const int nr = __popc(rest);
                    int nsub = 1;
                    for (int i = 1; i <= hb; ++i) nsub = nsub * (nr - hb + i) / i;
                    const int Ra = sm.r[ha], Rb = sm.r[hb];
                    const RowRef<CT, PK> ra(a, sm, 0, ha, x), rb_(a, sm, 1, hb, x);
                    const bool wide = WD ? true : !PK && (ra.wide || rb_.wide);
                    auto index_a = [&](unsigned c2) { return sm.crank[rest & ~c2] * Ra + la; };
                    V before;
                    auto scan = [&](auto at_a, auto at_b) {
                        return lane_first_exceeding<NW, V>(nsub, Y, [&](int i) -> V {
                            const unsigned c2 = select_bits(sm.unrank[hb][i], pos);
                            MC_COUNT((ha == 1 ? 0 : ra.bytes()) + rb_.bytes(), ha == 1 ? 32 : 64);
                            return (ha == 1 ? (V)1 : (V)at_a(index_a(c2))) * (V)at_b(sm.crank[c2] * Rb + lb);
                        }, before);
                    };
                    const int blk = wide ? scan(
                                               [&](int i) {
                                                   if constexpr (WD > 0) return ra.full(i);
                                                   else return entry_wide<CT>(a, 0, ha, x, i);
                                               },
                                               [&](int i) {
                                                   if constexpr (WD > 0) return rb_.full(i);
                                                   else return entry_wide<CT>(a, 1, hb, x, i);
                                               })
                                         : scan([&](int i) { return ra.get(i); }, [&](int i) { return rb_.get(i); });
                    if (blk < 0) { ok = false; bad = true; }
                    else {
                        const unsigned c2 = select_bits(sm.unrank[hb][blk], pos);
                        C2 = insert_colour_gap(c2, cx);
                        const V x1 = ha == 1 ? (V)1
                                     : WD    ? (V)ra.full(index_a(c2))
                                             : (V)(wide ? entry_wide<CT>(a, 0, ha, x, index_a(c2)) : ra.get(index_a(c2)));
                        q = (CT)quotient(Y - before, x1);  // < S(T'', C'', x): fits CT
                        sidx = sm.crank[c2] * Rb + lb;
                    }
                }
            }
            uint32_t u = 0;
            int cu = 0;
            if (ok && hb == 1) {
                // T'' one node: c(T''_{C''}, u) is 1 for the neighbours of the one
                // colour of C'' and 0 otherwise, so the answer is the (q+1)-th
                // neighbour of that colour in ascending id order: position q of
                // that colour's block in the colour-sorted adjacency
                cu = __ffs(C2) - 1;
                const int32_t b0 = a.coff[(int64_t)x * (a.k + 1) + cu];
                const int32_t b1 = a.coff[(int64_t)x * (a.k + 1) + cu + 1];
                MC_COUNT(8 + 4, 64);
                if ((uint64_t)q >= (uint64_t)(b1 - b0)) { ok = false; bad = true; }
                else u = a.scol[e0 + b0 + (int64_t)q];
            } else if (ok) {
                // ---- hub: the 64-neighbour chunk holding the answer, from the
                // inclusive prefix of its chunk sums (contiguous per hub and entry):
                // the first chunk whose prefix exceeds q
                int64_t lo_e = e0;
                int64_t len = deg;
                if (chunk0 >= 0) {
                    const int64_t nch = (deg + HUB_CHUNK - 1) / HUB_CHUNK;
                    const CT *spp = (const CT *)a.Sp[hb] + (int64_t)chunk0 * a.Ws[hb] + (int64_t)sidx * nch;
                    const int64_t ci = first_true<KS>(
                        0, nch - 1, [&](int64_t i) { return spp[i] > q; }, [&] { MC_COUNT(CB, 32); });
                    MC_COUNT(2 * CB, 32);
                    if (!(spp[ci] > q)) { ok = false; bad = true; }
                    else {
                        lo_e = e0 + ci * HUB_CHUNK;
                        len = min((int64_t)HUB_CHUNK, deg - ci * HUB_CHUNK);
                        q -= ci ? spp[ci - 1] : (CT)0;
                    }
                }
                // ---- neighbour: first u (ascending) whose running sum of
                // c(T''_{C''}, u) exceeds q (at most HUB_CHUNK neighbours)
                int r = -1;
                if (ok) {
                    const int rcb = sm.r[hb];
                    const uint32_t *ids = a.col + lo_e;
                    const uint8_t *cols = a.ecol + lo_e;
                    auto index_of = [&](int ci) { return sm.crank[drop_colour(C2 & ~(1u << ci), ci)] * rcb + lb; };
                    CT bn;
                    if constexpr (PK) {
                        r = lane_first_exceeding<NW, CT>((int)len, q, [&](int i) -> CT {
                            const int ci = cols[i];
                            return ((C2 >> ci) & 1u) ? RowRef<CT, PK>(a, sm, 0, hb, ids[i]).get(index_of(ci)) : (CT)0;
                        }, bn);
                    } else if (!WD && sm.level[0][hb].w >> 8) {  // the level has wide rows
                        r = lane_first_exceeding<NW, CT>((int)len, q, [&](int i) -> CT {
                            const int ci = cols[i];
                            MC_COUNT(5, 5);  // contiguous edge colours and ids
                            if ((C2 >> ci) & 1u) MC_COUNT((int)(sm.level[0][hb].w & 255u) + 4, 64);  // entry, wide word
                            return ((C2 >> ci) & 1u) ? entry_wide<CT>(a, 0, hb, ids[i], index_of(ci)) : (CT)0;
                        }, bn);
                    } else {
                        // ids and colours of NW neighbours together, then the entries of
                        // those whose colour is in C'', all in flight
                        const uint4 lv = sm.level[0][hb];
                        const uint8_t *p0 = (const uint8_t *)(((uint64_t)lv.y << 32) | lv.x);
                        const int n = (int)len, N = (int)(lv.w & 255u);
                        CT run = 0;
                        for (int b = 0; b < n && r < 0; b += NW) {
                            uint32_t id[NW];
                            int ci[NW];
                            uint32_t ww[NW];
                            CT y[NW];
#pragma unroll
                            for (int i = 0; i < NW; ++i) {
                                const int k2 = min(b + i, n - 1);
                                ci[i] = cols[k2];
                                id[i] = ids[k2];
                            }
#pragma unroll
                            for (int i = 0; i < NW; ++i) {
                                const bool in = b + i < n && ((C2 >> ci[i]) & 1u);
                                MC_COUNT(5, 5);  // contiguous edge colours and ids
                                if (in) MC_COUNT(N, 32);  // the neighbour's row entry
                                y[i] = in ? row_low_any<CT>(p0 + id[i] * (uint64_t)lv.z, N, index_of(ci[i])) : (CT)0;
                                if constexpr (WD > 0) ww[i] = in && lv.w >> 8 ? (a.wide[id[i]] >> hb) & 1u : 0u;
                            }
                            if constexpr (WD > 0) {
                                const uint4 uv = sm.upper[0][hb];
                                const uint8_t *p1 = (const uint8_t *)(((uint64_t)uv.y << 32) | uv.x);
                                uint32_t any = 0;
#pragma unroll
                                for (int i = 0; i < NW; ++i) any |= ww[i];
                                if (any) {
#pragma unroll
                                    for (int i = 0; i < NW; ++i)
                                        if (ww[i])
                                            y[i] |= row_rest<CT>(p1 + id[i] * (uint64_t)uv.z, (int)uv.w, N, index_of(ci[i]));
                                }
                            }
#pragma unroll
                            for (int i = 0; i < NW; ++i)
                                if (r < 0) {
                                    if (run + y[i] > q) { r = b + i; u = id[i]; cu = ci[i]; }
                                    else run += y[i];
                                }
                        }
                    }
                }
                if (r < 0) { ok = false; bad = true; }
                else if (PK || (!WD && sm.level[0][hb].w >> 8)) {
                    u = a.col[lo_e + r];
                    cu = a.ecol[lo_e + r];
                }
            }
            if (ok) {
                if (sp + 2 > MAXK) { ok = false; bad = true; }
                else {
                    nod[nn * T] = u;
                    par |= (uint32_t)at << (4 * nn);
                    stk[sp * T] = entry(gb, C2, cu, nn);
                    stk[(sp + 1) * T] = entry(ga, C & ~C2, cx, at);
                    sp += 2;
                    ++nn;
                }
            }
        }
        if (ok && nn != h) { ok = false; bad = true; }
        if constexpr (SPLIT) {  // classify_kernel does the rest
            if (sid < a.count) {
                const int64_t at = sid - a.begin;
                a.par[at] = ok ? par : 0xffffffffu;
                if (ok)
                    for (int i = 0; i < h; ++i) a.found[at * h + i] = nod[i * T];
                if (ok && a.roots) a.roots[sid] = v;
                if (ok && a.shapes) a.shapes[sid] = s0;
            }
            continue;
        }
        int cls = -1;
        if (ok) {
            // induced subgraph, its nodes in order of discovery (the class does
            // not depend on the labels): the treelet's edges are known; the other
            // pairs are searched in the shorter adjacency list, NQ at a time
            uint32_t word = 0;
            for (int i = 1; i < h; ++i) word |= 1u << pair_pos(h, (int)(par >> (4 * i) & 15u), i);
            for (int i = 0; i < h; ++i) {
                const uint32_t x = nod[i * T];
                const int64_t lo = a.row_ptr[x];
                off[i * T] = (uint32_t)lo;
                stk[i * T] = (uint32_t)(a.row_ptr[x + 1] - lo);
                MC_COUNT(16, 32);
            }
            uint32_t todo = ((1u << P) - 1u) & ~word;
            while (todo) {
                const uint32_t *row[NQ];
                uint32_t lo[NQ], hi[NQ], key[NQ], bit[NQ];
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    lo[q] = hi[q] = key[q] = 0;
                    row[q] = a.col;
                    bit[q] = todo & (0u - todo);
                    if (!bit[q]) continue;
                    todo &= todo - 1;
                    const unsigned ij = sm.pair[__ffs(bit[q]) - 1];
                    int x = (int)(ij & 15u), y = (int)(ij >> 4);
                    uint32_t dx = stk[x * T];
                    const uint32_t dy = stk[y * T];
                    if (dy < dx) { const int t = x; x = y; y = t; dx = dy; }
                    hi[q] = dx;
                    key[q] = nod[y * T];
                    row[q] = a.col + (a.long_rows ? a.row_ptr[nod[x * T]] : (int64_t)off[x * T]);
                }
                bool more = true;
                while (more) {
                    more = false;
#pragma unroll
                    for (int q = 0; q < NQ; ++q)
                        if (lo[q] < hi[q]) {
                            const uint32_t mid = (lo[q] + hi[q]) >> 1;
                            const uint32_t w = row[q][mid];
                            MC_COUNT(4, 32);
                            if (w == key[q]) { word |= bit[q]; hi[q] = lo[q]; }
                            else if (w < key[q]) lo[q] = mid + 1;
                            else hi[q] = mid;
                            more |= lo[q] < hi[q];
                        }
                }
            }
            cls = a.lut[word];
            MC_COUNT(2, 32);
            if (cls == 0xffff) { cls = -1; bad = true; }
            if (a.nodes) {
                // ascending: an odd-even merge sort of 8, absent nodes last
                uint32_t n_[MAXK];
#pragma unroll
                for (int i = 0; i < MAXK; ++i) n_[i] = i < h ? nod[i * T] : 0xffffffffu;
                auto order = [&](int i, int j) {
                    const uint32_t lo = min(n_[i], n_[j]), hi = max(n_[i], n_[j]);
                    n_[i] = lo;
                    n_[j] = hi;
                };
#pragma unroll
                for (int p = 1; p < MAXK; p <<= 1)
#pragma unroll
                    for (int k2 = p; k2 >= 1; k2 >>= 1)
#pragma unroll
                        for (int j = k2 % p; j + k2 < MAXK; j += 2 * k2)
#pragma unroll
                            for (int i = 0; i < k2; ++i)
                                if (i + j + k2 < MAXK && (i + j) / (2 * p) == (i + j + k2) / (2 * p)) order(i + j, i + j + k2);
#pragma unroll
                for (int i = 0; i < MAXK; ++i)
                    if (i < h) a.nodes[sid * h + i] = n_[i];
            }
            if (a.roots) a.roots[sid] = v;
            if (a.shapes) a.shapes[sid] = s0;
            {
                const int ob = (a.nodes ? 4 * h : 0) + (a.roots ? 4 : 0) + (a.shapes ? 4 : 0) + (a.classes ? 4 : 0);
                MC_COUNT(ob, ob);
            }
            if (a.hist && cls >= 0) atomicAdd(&s_hist[cls], 1u);
        }
        if (sid < a.count && a.classes) a.classes[sid] = cls;
    }
    if (bad) atomicOr(a.err, SERR_SEARCH);
    if (CNT && a.bytes) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
            rb += __shfl_xor_sync(0xffffffffu, rb, d);
            rs += __shfl_xor_sync(0xffffffffu, rs, d);
        }
        if (lane == 0) {
            atomicAdd(a.bytes, (unsigned long long)rb);
            atomicAdd(a.bytes + 1, (unsigned long long)rs);
        }
    }
    if (a.hist && !SPLIT) {
        __syncthreads();
        for (int i = threadIdx.x; i < a.ncls; i += T)
            if (s_hist[i]) atomicAdd(&a.hist[i], (unsigned long long)s_hist[i]);
    }
}

// Warp-per-sample sampler, for requests of a few samples per resident warp: a
// warp draws one sample at a time, so that its chain of dependent loads is as
// short as it gets.  Lane i holds the sample's i-th node and i-th stack entry;
// scans run 32 M items at a time (each lane M consecutive items, a prefix over
// the lanes), searches probe 32 places at a time, the first random words of all
// steps are drawn side by side, and the classification's pairs are one per
// lane.  Bound by the latency of that chain: 1000 samples at k = 8 (Chung-Lu
// 300k, 128-bit counts) 0.052 ms against 0.355 with a lane per sample.  For
// large requests the lanes' repeated scalar work loses (1M samples at k = 5:
// 7.6 against 1.1 ms; with 8 lanes per sample 3.5).
template <typename T> __device__ __forceinline__ T warp_get(T x, int src)
{
    if constexpr (sizeof(T) == 16) return shfl(x, src);
    else return __shfl_sync(0xffffffffu, x, src);
}

// Over items 0 .. len-1 in order, the first whose running sum of val(i)
// exceeds q (-1 if none or !act), `before` the running sum before it.
template <int M, typename V, typename F>
__device__ __forceinline__ int warp_first_exceeding(bool act, int len, V q, F val, V &before)
{
    const int j = threadIdx.x & 31;
    V run = 0;
    int found = -1;
    for (int b = 0; __any_sync(0xffffffffu, act && b < len); b += 32 * M) {
        V x[M], s = 0;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int i = b + j * M + m;
            x[m] = act && i < len ? val(i) : (V)0;
        }
#pragma unroll
        for (int m = 0; m < M; ++m) s += x[m];
        V inc = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const V y = shfl_up(inc, d);
            if (j >= d) inc += y;
        }
        V r = run + inc - s;
        const unsigned hit = __ballot_sync(0xffffffffu, act && run + inc > q);
        int mf = M - 1;
#pragma unroll
        for (int m = 0; m < M - 1; ++m)
            if (mf == M - 1) {
                if (r + x[m] > q) mf = m - M;  // found: stop adding
                else r += x[m];
            }
        if (mf < 0) mf += M;
        const int src = hit ? __ffs(hit) - 1 : 0;
        const int at = warp_get(b + j * M + mf, src);
        const V rb = warp_get(r, src);
        if (hit && act) { found = at; before = rb; act = false; }
        run += warp_get(inc, 31);
    }
    return found;
}

// The first i in [lo, hi) with pred(i), false then true along the range (hi if
// never true): 32 evenly spaced probes per round.
template <typename P>
__device__ __forceinline__ int64_t warp_first_true(bool act, int64_t lo, int64_t hi, P pred)
{
    const int j = threadIdx.x & 31;
    while (__any_sync(0xffffffffu, act && lo < hi)) {
        const bool go = act && lo < hi;
        const int64_t step = (hi - lo + 31) / 32, p = lo + (j + 1) * step - 1;
        const bool t = go && (p >= hi || pred(p));
        const unsigned b = __ballot_sync(0xffffffffu, t);
        if (go) {
            const int f = b ? __ffs(b) - 1 : 32;
            const int64_t nlo = f ? lo + f * step : lo;
            hi = f < 32 ? min(hi, lo + (f + 1) * step - 1) : hi;
            lo = min(nlo, hi);
            if (f == 32) lo = hi;
        }
    }
    return lo;
}

template <typename CT, typename V, bool PK>
__global__ void __launch_bounds__(256, 2) sample_warp_kernel(const __grid_constant__ SampleArgs a)
{
    constexpr int T = 256, M = 4;
    extern __shared__ uint32_t s_dyn[];
    unsigned int *const s_hist = s_dyn;
    __shared__ SampleSmem sm;
    const int h = a.h, P = h * (h - 1) / 2;
    fill_sample_smem<T>(a, sm);
    if (a.hist)
        for (int i = threadIdx.x; i < a.ncls; i += T) s_hist[i] = 0;
    __syncthreads();
    const int j = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)T + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * T) >> 5;
    bool bad = false;
    auto full = [&](const RowRef<CT, PK> &r, int idx) -> CT {
        return !PK && r.wide ? entry_wide<CT>(a, r.which, r.h, r.x, idx) : r.get(idx);
    };
    auto entry = [](int g, unsigned C, int cx, int at) {
        return (uint32_t)g | C << 8 | (uint32_t)cx << 16 | (uint32_t)at << 20;
    };
    for (int64_t sid = warp; sid < a.count; sid += nwarps) {
        bool ok = true;
        uint64_t index = a.first_index + (uint64_t)sid;
        const u128 *prefix = a.prefix;
        const uint32_t *bucket = a.bucket;
        u128 R = a.R, Xbase = a.Xbase, D = a.D;
        uint64_t allow0 = a.allow0, allow1 = a.allow1;
        if (a.nseg > 0) {  // the part this sample falls in
            int g = 0;
            while (g + 1 < a.nseg && sid >= a.seg[g].end) ++g;
            const SampleSeg &sg = a.seg[g];
            index = sg.first_index + (uint64_t)(sid - (g ? a.seg[g - 1].end : 0));
            prefix = sg.prefix;
            bucket = sg.bucket;
            R = sg.R;
            Xbase = sg.Xbase;
            D = sg.D;
            allow0 = sg.allow0;
            allow1 = sg.allow1;
        }
        // the first attempt's words of every step, lane s for step s
        uint32_t pw[4] = {(uint32_t)index, (uint32_t)(index >> 32), (uint32_t)j, 0u};
        philox(pw, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
        // uniform(W) of step `step` (the words of draw_below), false after 128 rejections
        auto draw = [&](bool act, int step, V W, V &out) -> bool {
            const V wm1 = W - 1;
            V mask;
            if constexpr (sizeof(V) == 16) {
                const uint64_t hi = (uint64_t)(wm1 >> 64), lo = (uint64_t)wm1;
                const int bits = hi ? 128 - __clzll(hi) : 64 - __clzll(lo);
                mask = bits >= 128 ? ~(V)0 : (((V)1) << bits) - 1;
            } else {
                const int bits = 64 - __clzll(wm1);
                mask = bits >= 64 ? ~0ull : (1ull << bits) - 1;
            }
            auto value = [&](const uint32_t *w) -> V {
                V r = (V)w[0] | (V)((uint64_t)w[1] << 32);
                if constexpr (sizeof(V) == 16) r |= (V)w[2] << 64 | (V)w[3] << 96;
                return r & mask;
            };
            V r = warp_get(value(pw), step);
            // (each lane masked its own words with this step's mask)
            {
                bool need = act && W != 0 && !(r < W);
                for (uint32_t att = 1; att < 128 && __any_sync(0xffffffffu, need); att += 32) {
                    uint32_t c[4] = {(uint32_t)index, (uint32_t)(index >> 32), (uint32_t)step, att + j};
                    philox(c, (uint32_t)a.seed, (uint32_t)(a.seed >> 32));
                    const V y = value(c);
                    const unsigned b = __ballot_sync(0xffffffffu, y < W);
                    const V z = warp_get(y, b ? __ffs(b) - 1 : 0);
                    if (need && b) { r = z; need = false; }
                }
                out = r;
                return act && W != 0 && !need;
            }
        };
        // ---- root: X = uniform(R); v = first node with prefix[v] > X
        V X = 0;
        {
            const bool d = draw(ok, 0, (V)R, X);
            if (ok && !d) { ok = false; bad = true; }
        }
        X += (V)Xbase;  // a node range: the draw lands inside its part of the prefix
        int64_t blo = 0, bhi = 0;
        if (ok) {
            const uint64_t bk = (uint64_t)(X / (V)D);
            blo = bucket[bk];
            bhi = bucket[bk + 1];
        }
        const uint32_t v = (uint32_t)warp_first_true(ok, blo, bhi, [&](int64_t i) { return prefix[i] > (u128)X; });
        V rem = 0;
        if (ok) {
            if (!(prefix[v] > (u128)X)) { ok = false; bad = true; }
            else rem = X - (v ? (V)prefix[v - 1] : (V)0);
        }
        // ---- entry of v's level-h row, in (shape id, colour mask) order
        int s0 = 0, sp = 0, nn = 0;
        uint32_t par = 0;  // per node, four bits: its parent's place in the node list
        uint32_t mynode = 0, mystk = 0;
        {
            const int Bc = a.Bc[h], Rh = a.R_[h];
            const RowRef<CT, PK> row(a, sm, 0, h, ok ? v : 0);
            V bf;
            const int found = warp_first_exceeding<M, V>(ok, a.Wc[h], rem, [&](int e) -> V {
                const int sh = e / Bc;
                const bool al = sh < 64 ? (allow0 >> sh) & 1 : (allow1 >> (sh - 64)) & 1;
                return al ? (V)full(row, (e - sh * Bc) * Rh + sh) : (V)0;
            }, bf);
            if (ok && found < 0) { ok = false; bad = true; }
            if (ok) {
                const int cv = a.colors[v];
                s0 = found / Bc;
                const unsigned C = (1u << cv) | insert_colour_gap(sm.unrank[h - 1][found % Bc], cv);
                if (j == 0) { mystk = entry(a.first[h] + s0, C, cv, 0); mynode = v; }
                sp = nn = 1;
            }
        }
        // ---- descent: decomposition nodes in pre-order (T' before T'')
        for (int step = 1; step < h; ++step) {
            uint2 sg = make_uint2(0, 0);
            uint32_t en = 0;
            bool look = ok;
            while (__any_sync(0xffffffffu, look)) {  // leaves on top of the stack are done
                if (look && (sp <= 0 || nn >= MAXK)) { ok = look = false; bad = true; }
                if (look) --sp;
                const uint32_t e = warp_get(mystk, sp & 31);
                if (look) {
                    en = e;
                    sg = sm.shape[en & 255u];
                    if ((sg.x & 255u) > 1) look = false;
                }
            }
            const int cx = (int)(en >> 16 & 15u), at = (int)(en >> 20);
            const unsigned C = en >> 8 & 255u;
            const uint32_t x = warp_get(mynode, at & 31);
            const int ga = (int)(sg.y & 255u), gb = (int)(sg.y >> 8 & 255u);
            const uint32_t sa = sm.shape[ga].x, sb = sm.shape[gb].x;
            const int hg = (int)(sg.x & 255u), ha = (int)(sa & 255u), la = (int)(sa >> 8 & 255u);
            const int hb = (int)(sb & 255u), lb = (int)(sb >> 8 & 255u);
            int64_t e0 = 0, deg = 0;
            int chunk0 = -1;
            // colour sets relative to x: c_x deleted from the palette
            const unsigned rest = drop_colour(C & ~(1u << cx), cx);
            V W = 0, Y = 0;
            if (ok) {
                e0 = a.row_ptr[x];
                deg = a.row_ptr[x + 1] - e0;
                chunk0 = a.node_chunk0[x];
                W = (V)(sg.x >> 16 & 255u) *
                    (V)full(RowRef<CT, PK>(a, sm, 0, hg, x), sm.crank[rest] * sm.r[hg] + (int)(sg.x >> 8 & 255u));
            }
            {
                const bool d = draw(ok, step, W, Y);
                if (ok && !d) { ok = false; bad = true; }
            }
            // block of C'' (ascending mask), weights c(T'_{C\C''}, x) S(T'', C'', x)
            const uint32_t pos = bit_positions(rest);
            const int nr = __popc(rest);
            int nsub = 1;
            for (int i = 1; i <= hb; ++i) nsub = nsub * (nr - hb + i) / i;
            const int Ra = sm.r[ha], Rb = sm.r[hb];
            unsigned c2 = 0;
            CT q = 0;
            {
                const RowRef<CT, PK> ra(a, sm, 0, ha, ok ? x : 0), rb_(a, sm, 1, hb, ok ? x : 0);
                auto count_a = [&](unsigned m) -> V {
                    return ha == 1 ? (V)1 : (V)full(ra, sm.crank[rest & ~m] * Ra + la);
                };
                V before = 0;
                const int blk = warp_first_exceeding<2, V>(ok, nsub, Y, [&](int i) -> V {
                    const unsigned m = select_bits(sm.unrank[hb][i], pos);
                    return count_a(m) * (V)full(rb_, sm.crank[m] * Rb + lb);
                }, before);
                if (ok && blk < 0) { ok = false; bad = true; }
                if (ok) {
                    c2 = select_bits(sm.unrank[hb][blk], pos);
                    q = (CT)quotient(Y - before, count_a(c2));  // < S(T'', C'', x): fits CT
                }
            }
            const unsigned C2 = insert_colour_gap(c2, cx);
            uint32_t u = 0;
            int cu = 0;
            const bool single = ok && hb == 1, scan = ok && hb != 1;
            if (single) {
                // T'' one node: the (q+1)-th neighbour of the one colour of C'', at
                // position q of that colour's block in the colour-sorted adjacency
                cu = __ffs(C2) - 1;
                const int32_t b0 = a.coff[(int64_t)x * (a.k + 1) + cu];
                const int32_t b1 = a.coff[(int64_t)x * (a.k + 1) + cu + 1];
                if ((uint64_t)q >= (uint64_t)(b1 - b0)) { ok = false; bad = true; }
                else u = a.scol[e0 + b0 + (int64_t)q];
            }
            if (__any_sync(0xffffffffu, scan)) {
                // ---- hub: the first 64-neighbour chunk whose prefix of the chunk sums
                // (contiguous per hub and entry) exceeds q
                int64_t lo_e = e0, len = deg;
                bool act = scan;
                const bool hub = scan && chunk0 >= 0;
                const int64_t nch = (deg + HUB_CHUNK - 1) / HUB_CHUNK;
                const CT *spp = nullptr;
                if (hub)
                    spp = (const CT *)a.Sp[hb] + (int64_t)chunk0 * a.Ws[hb] + (int64_t)(sm.crank[c2] * Rb + lb) * nch;
                const int64_t ci = warp_first_true(hub, 0, nch - 1, [&](int64_t i) { return spp[i] > q; });
                if (hub) {
                    if (!(spp[ci] > q)) { ok = act = false; bad = true; }
                    else {
                        lo_e = e0 + ci * HUB_CHUNK;
                        len = min((int64_t)HUB_CHUNK, deg - ci * HUB_CHUNK);
                        q -= ci ? spp[ci - 1] : (CT)0;
                    }
                }
                // ---- neighbour: first u (ascending) whose running sum of
                // c(T''_{C''}, u) exceeds q (at most HUB_CHUNK neighbours)
                CT bn;
                const int r = warp_first_exceeding<2, CT>(act, (int)len, q, [&](int i) -> CT {
                    const int ci2 = a.ecol[lo_e + i];
                    if (!((C2 >> ci2) & 1u)) return (CT)0;
                    const uint32_t w = a.col[lo_e + i];
                    return full(RowRef<CT, PK>(a, sm, 0, hb, w), sm.crank[drop_colour(C2 & ~(1u << ci2), ci2)] * Rb + lb);
                }, bn);
                if (act) {
                    if (r < 0) { ok = false; bad = true; }
                    else {
                        u = a.col[lo_e + r];
                        cu = a.ecol[lo_e + r];
                    }
                }
            }
            if (ok) {
                if (sp + 2 > MAXK) { ok = false; bad = true; }
                else {
                    if (j == nn) mynode = u;
                    par |= (uint32_t)at << (4 * nn);
                    if (j == sp) mystk = entry(gb, C2, cu, nn);
                    if (j == sp + 1) mystk = entry(ga, C & ~C2, cx, at);
                    sp += 2;
                    ++nn;
                }
            }
        }
        if (ok && nn != h) { ok = false; bad = true; }
        // induced subgraph, its nodes in order of discovery (the class does not
        // depend on the labels): the treelet's edges are known; the other pairs
        // are searched in the shorter adjacency list, spread over the lanes
        uint32_t word = 0;
        for (int i = 1; i < h; ++i) word |= 1u << pair_pos(h, (int)(par >> (4 * i) & 15u), i);
        int64_t mylo = 0;
        uint32_t mydeg = 0;
        if (ok && j < h) {
            mylo = a.row_ptr[mynode];
            mydeg = (uint32_t)(a.row_ptr[mynode + 1] - mylo);
        }
        {
            const unsigned ij = j < P ? sm.pair[j] : 0u;
            const int x = (int)(ij & 15u), y = (int)(ij >> 4);
            const uint32_t dx = warp_get(mydeg, x), dy = warp_get(mydeg, y);
            const bool sw = dy < dx;
            const uint32_t key = warp_get(mynode, sw ? x : y);
            const uint32_t *row = a.col + warp_get(mylo, sw ? y : x);
            uint32_t lo = 0, hi = (ok && j < P && !((word >> j) & 1u)) ? (sw ? dy : dx) : 0u;
            bool mine = false;
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1, w = row[mid];
                if (w == key) { mine = true; hi = lo; }
                else if (w < key) lo = mid + 1;
                else hi = mid;
            }
            __syncwarp();
            word |= __ballot_sync(0xffffffffu, mine);
        }
        int cls = -1;
        if (ok) {
            cls = a.lut[word];
            if (cls == 0xffff) { cls = -1; bad = true; }
        }
        if (a.nodes) {  // ascending: a lane's node goes to its rank
            int rank = 0;
            for (int i = 0; i < h; ++i) rank += warp_get(mynode, i) < mynode;
            if (ok && j < h) a.nodes[sid * h + rank] = mynode;
        }
        if (j == 0) {
            if (ok) {
                if (a.roots) a.roots[sid] = v;
                if (a.shapes) a.shapes[sid] = s0;
                if (a.hist && cls >= 0) atomicAdd(&s_hist[cls], 1u);
            }
            if (a.classes) a.classes[sid] = cls;
        }
    }
    if (bad) atomicOr(a.err, SERR_SEARCH);
    if (a.hist) {
        __syncthreads();
        for (int i = threadIdx.x; i < a.ncls; i += T)
            if (s_hist[i]) atomicAdd(&a.hist[i], (unsigned long long)s_hist[i]);
    }
}

// Classification of split samples: a block takes tiles of 64 samples, loads
// their nodes and adjacency offsets together, spreads the pairs that are not
// treelet edges over its threads (a binary search of the shorter adjacency list
// each; more in flight per thread is slower: 0.25 against 0.17 ms per 1M
// samples at k = 5), looks the words up and writes the nodes in ascending
// order.  Inside the sampler the same searches run at its registers' occupancy
// and in the divergence of its 32 samples per warp.  `found` and `par` may be
// the output arrays themselves: a tile reads its samples before it writes them.
struct ClassifyArgs {
    const int64_t *row_ptr;
    const uint32_t *col;
    const uint32_t *found, *par;  // per sample: h nodes in order of discovery; four bits per node: its parent
    int64_t count;
    int h;
    const uint16_t *lut;
    uint32_t *nodes;
    int32_t *classes;
    unsigned long long *hist;
    int ncls;
    int *err;
};
constexpr int CLASSIFY_TILE = 64;

static __global__ void __launch_bounds__(256) classify_kernel(const __grid_constant__ ClassifyArgs a)
{
    constexpr int S = CLASSIFY_TILE, T = 256;
    extern __shared__ unsigned int s_hist[];
    __shared__ int64_t s_lo[S * MAXK];
    __shared__ uint32_t s_node[S * MAXK], s_deg[S * MAXK], s_word[S];
    __shared__ bool s_ok[S];
    __shared__ uint8_t s_i[32], s_j[32];
    const int h = a.h, P = h * (h - 1) / 2;
    if (threadIdx.x == 0)
        for (int i = 0; i < h; ++i)
            for (int j = i + 1; j < h; ++j) {
                s_i[pair_pos(h, i, j)] = (uint8_t)i;
                s_j[pair_pos(h, i, j)] = (uint8_t)j;
            }
    if (a.hist)
        for (int i = threadIdx.x; i < a.ncls; i += T) s_hist[i] = 0;
    bool bad = false;
    for (int64_t base = blockIdx.x * (int64_t)S; base < a.count; base += gridDim.x * (int64_t)S) {
        const int ns = (int)min((int64_t)S, a.count - base);
        __syncthreads();
        if (threadIdx.x < ns) {
            const uint32_t par = a.par[base + threadIdx.x];
            const bool ok = par != 0xffffffffu;
            uint32_t word = 0;
            if (ok)
                for (int i = 1; i < h; ++i) word |= 1u << pair_pos(h, (int)(par >> (4 * i) & 15u), i);
            s_word[threadIdx.x] = word;
            s_ok[threadIdx.x] = ok;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < ns * h; i += T) {
            const int s = i / h;
            if (!s_ok[s]) continue;
            const uint32_t x = a.found[base * h + i];
            const int64_t lo = a.row_ptr[x];
            s_node[i] = x;
            s_lo[i] = lo;
            s_deg[i] = (uint32_t)(a.row_ptr[x + 1] - lo);
        }
        __syncthreads();
        for (int it = threadIdx.x; it < ns * P; it += T) {
            const int s = it / P, b = it - s * P;
            // (the known edges' bits never change; the others are set below)
            if (!s_ok[s] || ((s_word[s] >> b) & 1u)) continue;
            int x = s * h + s_i[b], y = s * h + s_j[b];
            if (s_deg[y] < s_deg[x]) { const int t = x; x = y; y = t; }
            const uint32_t *row = a.col + s_lo[x];
            const uint32_t key = s_node[y];
            uint32_t lo = 0, hi = s_deg[x];
            while (lo < hi) {
                const uint32_t mid = (lo + hi) >> 1, w = row[mid];
                if (w == key) { atomicOr(&s_word[s], 1u << b); break; }
                if (w < key) lo = mid + 1;
                else hi = mid;
            }
        }
        __syncthreads();
        if (threadIdx.x < ns) {
            int cls = -1;
            if (s_ok[threadIdx.x]) {
                cls = a.lut[s_word[threadIdx.x]];
                if (cls == 0xffff) { cls = -1; bad = true; }
            }
            if (a.classes) a.classes[base + threadIdx.x] = cls;
            if (a.hist && cls >= 0) atomicAdd(&s_hist[cls], 1u);
        }
        if (a.nodes)
            for (int i = threadIdx.x; i < ns * h; i += T) {
                const int s = i / h;
                if (!s_ok[s]) continue;
                int rank = 0;
                for (int j = 0; j < h; ++j) rank += s_node[s * h + j] < s_node[i];
                a.nodes[(base + s) * h + rank] = s_node[i];
            }
    }
    if (bad) atomicOr(a.err, SERR_SEARCH);
    if (a.hist) {
        __syncthreads();
        for (int i = threadIdx.x; i < a.ncls; i += T)
            if (s_hist[i]) atomicAdd(&a.hist[i], (unsigned long long)s_hist[i]);
    }
}

typedef void (*SampleKernel)(SampleArgs);
enum class SampleMode { Lanes, Latency, Counted, Split, Warps };
// The kernel for tables of bits-bit counts with 64-bit descent arithmetic
// (narrow) or 128-bit, dense (sampler_dense.cu; all modes; `wide`, 128-bit counts
// only: rows below level h are wide, 3 or 4 of their items in flight) or packed
// (sampler_packed.cu; all but Counted; `few`: at most 2 blocks per SM).
SampleKernel sample_kernel_dense(SampleMode mode, int bits, bool narrow, int wide);
SampleKernel sample_kernel_packed(SampleMode mode, int bits, bool narrow, bool few);

}  // namespace mc
