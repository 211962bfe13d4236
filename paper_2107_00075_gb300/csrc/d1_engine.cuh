// d1_engine.cuh -- distance-1 coloring engine (kernels + host driver),
// templated on the graph view so that one engine colors a single graph
// (SingleView) or a flattened batch of independent graphs (BatchView).
//
// Method (Bogle et al., Sec. 3.2-3.3, Alg. 1-4), round-synchronous form:
//   round 1       every vertex holds tentative color 1; detection decides;
//   round r >= 2  assign: each worklist vertex takes the smallest color not
//                 committed in its neighborhood (first fit, Alg. 1);
//                 detect: a worklist vertex loses if a neighbor holds the
//                 same color and has priority (Alg. 3 + Alg. 4); winners
//                 commit, losers form the next worklist.
//
// How the GPU computes exactly that, with less work than re-reading every
// worklist vertex's adjacency each round:
//   * Detection only needs the neighbors that have priority over v (Alg. 4
//     recolors the lower-priority end of a conflict), so setup builds, per
//     vertex, the list H(v) = {u in N(v) : key(u) > key(v)}.  Every edge is
//     in exactly one list, and hubs -- which stay on the worklist for many
//     rounds -- have short lists.  A committed neighbor never holds v's
//     tentative color (first fit excluded it), so v loses iff some u in H(v)
//     currently holds v's tentative color.
//   * First fit reads a per-vertex set of forbidden colors: one 64-bit word
//     for colors 1..64 and, for vertices of degree >= 64, an overflow bitmap
//     up to color deg(v)+1 (a first-fit color never exceeds deg(v)+1).  When
//     a vertex commits color c it sets bit c in its neighbors' sets ("push");
//     each vertex pushes once, so the total push work is one pass over the
//     adjacency.
//
// Color encoding in col[]: > 0 committed; < 0 tentative (-t) for a vertex
// on the current worklist.  Every uncolored vertex is on the worklist, so
// |col[u]| is u's current color during detection; a winner flips its own
// sign in place without disturbing concurrent readers.
//
// Work decomposition (no result depends on it):
//   detect, by |H(v)| (options mid_degree / hub_degree): two worklists of
//   vertices whose lists a warp searches together (up to 64 entries, up to
//   16384), and one block per vertex for longer lists.  A loser stops at the
//   step that finds its conflict.  In round 1 every vertex holds color 1, so v
//   loses exactly when H(v) is not empty and no list is read.  Losers keep
//   their worklist entry: they are re-appended by source index (the list
//   counters are the hottest atomics of the kernel).  Setup cuts long rows into
//   512-entry items and push into 128-entry items, one warp each.
// The round loop runs on the device: a CUDA graph with a conditional WHILE
// node around {assign, detect, push}; the last block of detect updates the
// round state and sets the loop condition.  Once the worklist has at most
// mid_w vertices the rounds run in one cooperative launch with grid barriers
// (the mid loop), and the last ones of a dense core on the subgraph the
// worklist induces, in one thread-block cluster (the core phase).  Their
// waits are the only ones in the engine: the mid loop's barriers and the
// cluster's first meeting poll with a limit; the core's rounds use the hardware
// cluster barrier, which has none, between CTAs that have all met and do
// finite work.
//
// Batches: graph g owns global vertices [vtx_off[g], vtx_off[g+1]); ids,
// the priority hash and degrees are graph-local, so every graph is colored
// exactly as it would be alone; the rounds of all graphs run together and a
// graph simply has no worklist vertices once it is done.
#pragma once
#include "runtime.h"
#include "device_common.cuh"

#include <algorithm>
#include <cstring>
#include <functional>
#include <memory>
#include <type_traits>
#include <unordered_map>

namespace pgc {
std::vector<std::function<void()>>& release_hooks();

namespace d1 {

// ---------------------------------------------------------------------------
// graph views
// ---------------------------------------------------------------------------
// One graph: int32 CSR.
struct SingleView {
    const int* rp;
    const int* ci;
    __device__ __forceinline__ int graph(int) const { return 0; }
    __device__ __forceinline__ int base(int) const { return 0; }
    __device__ __forceinline__ void row(int v, int, long long& b, int& d) const {
        const int r0 = __ldg(rp + v);
        b = r0;
        d = __ldg(rp + v + 1) - r0;
    }
    __device__ __forceinline__ int nbr(long long e, int) const { return __ldg(ci + e); }
    // row start as entries hold it, and degree
    __device__ __forceinline__ void local_row(int v, int, int& r0, int& d) const {
        r0 = __ldg(rp + v);
        d = __ldg(rp + v + 1) - r0;
    }
    // absolute start of v's row from an entry's row start
    __device__ __forceinline__ int begin(int, int r0) const { return r0; }
    using Off = int;
    // first overflow word of v, whose row starts at b: v owns deg/32 + 1 words (colors
    // 65 .. deg + 1, the last that first fit can reach), so consecutive vertices never
    // overlap and the total is nnz/32 + n + 1
    __device__ __forceinline__ long long bm(int v, long long b) const { return (b >> 5) + v; }
    // the degree in v's priority, from its row length d
    __device__ __forceinline__ int degree(int, int d) const { return d; }
    static constexpr bool kSetup = true;   // the engine builds the lists from the rows
};

// A batch: graph-local row_ptr blocks (n_g + 1 entries each) and graph-local
// column ids; int64 offsets into the flattened arrays.
struct BatchView {
    const long long* vtx_off;
    const long long* nnz_off;
    const int* rp;
    const int* ci;
    const int* gid;   // graph of each global vertex
    int absolute;     // entries hold absolute row starts (fewer than 2^32 entries in the
                      // batch): two dependent loads less per entry
    __device__ __forceinline__ int graph(int v) const { return __ldg(gid + v); }
    __device__ __forceinline__ int base(int g) const { return (int)__ldg(vtx_off + g); }
    __device__ __forceinline__ void row(int v, int g, long long& b, int& d) const {
        const int r0 = __ldg(rp + v + g);
        b = __ldg(nnz_off + g) + r0;
        d = __ldg(rp + v + g + 1) - r0;
    }
    __device__ __forceinline__ int nbr(long long e, int base_g) const {
        return base_g + __ldg(ci + e);
    }
    __device__ __forceinline__ void local_row(int v, int g, int& r0, int& d) const {
        r0 = __ldg(rp + v + g);
        d = __ldg(rp + v + g + 1) - r0;
        if (absolute) r0 = (int)(unsigned)(__ldg(nnz_off + g) + r0);
    }
    __device__ __forceinline__ long long begin(int v, int r0) const {
        return absolute ? (long long)(unsigned)r0 : __ldg(nnz_off + graph(v)) + r0;
    }
    using Off = long long;
    __device__ __forceinline__ long long bm(int v, long long b) const { return (b >> 5) + v; }
    __device__ __forceinline__ int degree(int, int d) const { return d; }
    static constexpr bool kSetup = true;
};

// A conflict graph given by lists the caller has built (distance-2 and
// partial distance-2, net.cu): v's row is ci[beg .. beg + len), the vertices
// with priority over v first, so the rows are the priority lists as well.
// The rows may lie in any order.
struct ListView {
    const int2* rows;   // {beg, len} per vertex
    const int* ci;
    const int* r_ptr;   // the degree in v's priority is r_ptr[v + 1] - r_ptr[v]
    int bm_words;       // overflow words per vertex
    __device__ __forceinline__ int graph(int) const { return 0; }
    __device__ __forceinline__ int base(int) const { return 0; }
    __device__ __forceinline__ void row(int v, int, long long& b, int& d) const {
        const int2 x = __ldg(rows + v);
        b = x.x;
        d = x.y;
    }
    __device__ __forceinline__ int nbr(long long e, int) const { return __ldg(ci + e); }
    __device__ __forceinline__ int begin(int, int r0) const { return r0; }
    using Off = int;
    __device__ __forceinline__ long long bm(int v, long long) const {
        return (long long)v * bm_words;
    }
    __device__ __forceinline__ int degree(int v, int) const {
        return __ldg(r_ptr + v + 1) - __ldg(r_ptr + v);
    }
    static constexpr bool kSetup = false;
};

constexpr int kBuildS = 32;     // setup: degree up to this: one thread
constexpr int kBuildM = 512;    // setup: degree up to this: one warp
constexpr int kBuildItem = 512; // setup: adjacency items of this length
constexpr int kPushItem = 128;  // push: adjacency items of this length
// round-varying priorities: longer lists take a block.  With few long lists a
// warp on one is what a round waits for; with enough of them to fill the grid,
// blocks on the shorter ones wait at their barriers.  n stands in for their
// number, which nothing has counted when the line is drawn; measured on R-MAT
// graphs of edge factor 16 only, where the two grow together.
// Dynamic degree, with blocks from 1024 / 2048 / 4096 entries up: R-MAT 18 4.2 / 5.3 / 5.3 ms, R-MAT 20 12.7 / 11.1 / 16.0 ms, R-MAT 21
// 22.0 / 19.0 / 18.9 ms, R-MAT 22 39.3 / 38.6 / 34.0 ms, R-MAT 24 191 / 190 / 152 ms
// (from 16,384 up: R-MAT 22 55 ms, R-MAT 24 155 ms)
inline int varying_hub(int n) { return std::clamp(n >> 9, 1024, 4096); }
// winners up to this degree push inline: 32 / 128 / 512 take 58.1 / 46.8 / 46.7 ms
// for the 4096-graph batch, 3.0 / 3.1 / 3.9 for R-MAT 20, 11.5 / 11.5 / 13.6 for PD2
// 4M x 1M and 12.8 / 13.7 / 13.7 for the 27-point mesh 128^3 (rows of 124)
constexpr int kInlinePush = 128;

enum : int {
    ST_OK = 0, ST_NO_PROGRESS = 1, ST_MAX_ROUNDS = 2, ST_TIMEOUT = 3, ST_BARRIER = 4,
    ST_LISTS = 5,  // ListView: the lists did not fit their buffer
    ST_MID_BARRIER = 6   // (ST_BARRIER: the core phase's meeting)
};

// What every block of a round's kernel reads, in one place: a block reads it
// once (see enter()), because thousands of warps reading one line of L2 at the
// same time wait for one another (10,000 to 20,000 cycles for a handful of
// fields, more than a small round's work).
struct Hot {
    int round;        // round being executed (1-based)
    int done;         // 1 once the loop has ended
    int mid;          // 1: the graph loop handed the remaining rounds to the mid loop
    int tail;         // 1: the mid loop handed the remaining rounds to the core phase
    int ns[2];        // S-tier worklist sizes per parity
    int nm[2];        // M-tier worklist sizes
    int nl[2];        // L-tier worklist sizes
    int push_cnt;     // push work items queued this round
    int max_color;
    int stop;         // mid loop: round before which the time limit had passed (0: none)
    int pend;         // round 1's queued pushes still wait (setup queues them)
    __host__ __device__ int count(int p) const { return ns[p] + nm[p] + nl[p]; }
};

struct State : Hot {
    int status;       // ST_*
    int bs, bm, bc;   // setup: vertices (S, M) and items (C) per degree class
    int lists_full;   // ListView: the lists did not fit their buffer
    unsigned blocks_done;
    int bar_timeout;            // mid loop: a barrier wait gave up
    unsigned long long s_next;  // sum of degrees of the next worklist
    unsigned long long h_next;  // sum of |H(v)| over the next worklist
    unsigned long long h_first; // sum of |H(v)| over all vertices
    unsigned long long t0;      // globaltimer at start
    int core_k;       // core phase: vertices of the induced subgraph
    int core_par;     // core phase: parity whose worklist buffers hold its arrays
    alignas(128) unsigned bar_count;   // mid loop grid barrier: arrivals, a line of its own
};

template <class V>
struct Problem {
    V g;
    int* col;
    int* deg;
    int* hlen;
    int* hadj;                 // H(v) stored at hadj[row start of v ...]
    unsigned long long* bm0;   // forbidden colors 1..64, one word per vertex
    unsigned* bmx;             // forbidden colors 65..deg+1 (deg >= 64)
    unsigned* live;            // bit v set while v is uncolored
    // worklists per parity; an entry is {v, |H(v)|, deg(v), row start of v
    // within its graph}, so a scan needs no further lookup to begin
    int4* ws[2];               // S tier
    int4* wm[2];               // M tier
    int4* wl[2];               // L tier
    int2* items;               // setup: (vertex, item) list for long rows
    int2* push_q;              // (vertex, item) push work
    unsigned* core_mat;        // core phase: adjacency bits, k x ceil(k / 32) words
    int* g_rounds;             // batch: rounds per graph (nullable)
    int* g_colors;             // batch: colors per graph (nullable)
    long long* trace_w;
    long long* trace_s;
    long long* trace_h;
    State* st;
    unsigned long long seed;
    unsigned long long timeout_ns;
    long long nnz;
    int trace_cap;
    int n;
    int use_deg;
    int async_mode;    // PGC_ASYNC: first fit also avoids tentative colors written this round
    int prio_mode;     // 0: static degree; 1: dynamic degree; 2: saturation degree
    int* prio;         // prio_mode != 0: each vertex's priority this round
    int max_rounds;
    int det_s;
    int det_m;
    int mid_w;         // hand over to the mid loop once the worklist is this small (0: never)
    int tail_w;        // core phase for worklists up to this size (0: never)
    // a wait's limit, and the test hook's late block
    struct Wait {
        unsigned polls;     // polls before giving up
        int slow_block;     // this block is late (-1: none)
        unsigned slow_ns;   // ... by this much
        int slow_at;        // ... at its slow_at-th barrier (mid loop)
    } mid_wait, core_wait;  // the mid loop's barriers, the core phase's meeting
};

// A block's copy of the problem and of the round's counters.  Kernels take
// the state's address beside the problem's, so both loads start at once.
template <class V>
struct Ctx {
    Problem<V> P;
    Hot h;
};
__device__ __forceinline__ void read_hot(Hot& h, const State* st) {
    if (threadIdx.x < sizeof(Hot) / 4)
        reinterpret_cast<int*>(&h)[threadIdx.x] =
            reinterpret_cast<const volatile int*>(st)[threadIdx.x];
}
template <class V>
__device__ __forceinline__ const Problem<V>& enter(Ctx<V>& c, const Problem<V>* Pp,
                                                   const State* st) {
    static_assert(sizeof(Problem<V>) % 4 == 0, "copied by words");
    read_hot(c.h, st);
    for (int i = threadIdx.x; i < (int)(sizeof(Problem<V>) / 4); i += blockDim.x)
        reinterpret_cast<int*>(&c.P)[i] = __ldg(reinterpret_cast<const int*>(Pp) + i);
    __syncthreads();
    return c.P;
}

// Appends entries to the worklists of two tiers, a block's at once: one
// atomic per block and tier instead of one per warp (the list counters are
// single addresses that the whole grid hits).  Every thread of the block
// calls; s_n: 2 x 33 ints of shared memory.
__device__ __forceinline__ void block_append(bool a, bool b, int4 e, int4* la, int* ca, int4* lb,
                                             int* cb, int (*s_n)[33]) {
    const int lane = lane_id(), warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const unsigned ma = __ballot_sync(kFullMask, a), mb = __ballot_sync(kFullMask, b);
    if (lane == 0) {
        s_n[0][warp] = __popc(ma);
        s_n[1][warp] = __popc(mb);
    }
    __syncthreads();
    if (warp < 2) {   // warp 0 places the first tier, warp 1 the second
        const int x = lane < wpb ? s_n[warp][lane] : 0;
        int incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFullMask, incl, o);
            if (lane >= o) incl += y;
        }
        int base = 0;
        if (lane == 31 && incl) base = atomicAdd(warp ? cb : ca, incl);
        base = __shfl_sync(kFullMask, base, 31);
        if (lane < wpb) s_n[warp][lane] = base + incl - x;
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    if (a) la[s_n[0][warp] + __popc(ma & lt)] = e;
    if (b) lb[s_n[1][warp] + __popc(mb & lt)] = e;
    __syncthreads();
}

// key(u) > key(v) for u, v of the same graph, key = (deg, -h, -id) (hash of
// graph-local ids), hashing only when the degree term does not decide.  This is
// Alg. 4 read as one comparison: of two equal-colored vertices the one that does
// NOT have priority is recolored.
__device__ __forceinline__ bool higher(int du, int u, int dv, uint64_t hv, int v, int base,
                                       unsigned long long seed, bool use_deg) {
    if (use_deg && du != dv) return du > dv;
    const uint64_t hu = prio_hash(seed, (uint32_t)(u - base));
    if (hu != hv) return hu < hv;
    return u < v;
}

__device__ __forceinline__ int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Forbid color c for u (a vertex of graph g).  Setting bits of an already
// colored vertex is harmless (its set is never read again), so colors 1..64
// need no check and the update is a fire-and-forget reduction.
// VARYING (a priority that changes each round): also keep u's priority for
// the next round: the dynamic degree drops by one per adjacency entry of a
// newly colored neighbor; the saturation degree grows when c is a color u
// had not yet seen among its colored neighbors and c <= deg(u) + 1.
template <bool VARYING, class V>
__device__ __forceinline__ void push_color_live(const Problem<V>& P, int u, int g, int c) {
    if (VARYING && P.prio_mode == 1) atomicSub(P.prio + u, 1);
    if (c <= 64) {
        const unsigned long long bit = 1ull << (c - 1);
        if (VARYING && P.prio_mode == 2) {
            const unsigned long long old = atomicOr(P.bm0 + u, bit);
            if (!(old & bit) && c - 1 <= P.deg[u]) atomicAdd(P.prio + u, 1);
        } else {
            atomicOr(P.bm0 + u, bit);
        }
        return;
    }
    long long bu;
    int du;
    P.g.row(u, g, bu, du);
    if (c - 1 > du) return;   // u's own first fit never reaches c
    const int b = c - 65;
    if (VARYING && P.prio_mode == 2) {
        const unsigned old = atomicOr(P.bmx + P.g.bm(u, bu) + (b >> 5), 1u << (b & 31));
        if (!(old & (1u << (b & 31)))) atomicAdd(P.prio + u, 1);
    } else {
        atomicOr(P.bmx + P.g.bm(u, bu) + (b >> 5), 1u << (b & 31));
    }
}
template <class V>
__device__ __forceinline__ void push_color(const Problem<V>& P, int u, int g, int c) {
    // most neighbors of a late winner are colored already: skip them
    if ((P.live[u >> 5] >> (u & 31)) & 1u) {
        if (P.prio_mode) push_color_live<true>(P, u, g, c);
        else push_color_live<false>(P, u, g, c);
    }
}

// Batch bookkeeping: arr[g] = max(arr[g], val) over the lanes with pred,
// one atomic per (warp, graph).  All 32 lanes call.
__device__ __forceinline__ void graph_max(int* arr, bool pred, int g, int val) {
    const int key = pred ? g : -1 - (int)lane_id();
    const unsigned peers = __match_any_sync(kFullMask, key);
    const int m = __reduce_max_sync(peers, pred ? val : 0);
    if (pred && (int)lane_id() == __ffs(peers) - 1) atomicMax(arr + g, m);
}

// ---------------------------------------------------------------------------
// setup 1: degrees, tentative color 1, empty forbidden sets, degree classes
// ---------------------------------------------------------------------------
template <class V>
__global__ void d1_classify(const Problem<V>* __restrict__ Pp) {
    __shared__ int s_n[2][33];
    const Problem<V>& P = *Pp;
    State* st = P.st;
    const int n = P.n;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < n; base += stride) {
        const long long wbase = base + (threadIdx.x & ~31u), i = wbase + lane_id();
        const bool valid = i < n;
        int d = -1, r0 = 0;
        if (valid) {
            const int v = (int)i;
            const int g = P.g.graph(v);
            P.g.local_row(v, g, r0, d);
            const long long b = P.g.begin(v, r0);
            P.deg[v] = d;
            P.col[v] = P.async_mode ? 0 : -1;
            if (P.prio_mode) P.prio[v] = P.prio_mode == 1 ? d : 0;
            P.hlen[v] = 0;
            P.bm0[v] = 0ull;
            if (d >= 64) {
                unsigned* w = P.bmx + P.g.bm(v, b);
                for (int k = 0; k <= (d >> 5); ++k) w[k] = 0u;
            }
            if (d > kBuildM) {
                const int nit = ceil_div(d, kBuildItem);
                const int base = atomicAdd(&st->bc, nit);
                for (int k = 0; k < nit; ++k) P.items[base + k] = make_int2(v, k);
            }
        }
        const unsigned vm = __ballot_sync(kFullMask, valid);
        // wbase is a multiple of 32 (past n only in the last block's spare warps)
        if (lane_id() == 0 && vm) P.live[wbase >> 5] = vm;
        block_append(valid && d <= kBuildS, valid && d > kBuildS && d <= kBuildM,
                     make_int4((int)i, 0, d, r0), P.ws[0], &st->bs, P.wm[0], &st->bm, s_n);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->round = 1;
        st->t0 = global_ns();
        if (P.trace_cap > 0) {
            P.trace_w[0] = n;
            P.trace_s[0] = P.nnz;
        }
    }
}

// ---------------------------------------------------------------------------
// setup 2: H(v) = neighbors with higher priority, stored at v's row start.
// Only the vertices in [lo, hi) (one launch may cover a part of the graph,
// so the rest of the adjacency can still be on its way to the device).
// ---------------------------------------------------------------------------
template <class V>
__global__ void __maxnreg__(40) d1_build(const Problem<V>* __restrict__ Pp, int lo, int hi) {
    const Problem<V>& P = *Pp;
    State* st = P.st;
    const int* __restrict__ dg = P.deg;
    const unsigned long long seed = P.seed;
    const bool use_deg = P.use_deg != 0;
    const int lane = lane_id(), warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int gw = blockIdx.x * wpb + warp, nw = gridDim.x * wpb;
    const int nS = st->bs, nM = st->bm, nC = st->bc;
    // priorities that change each round: the lists hold every neighbor
    const bool all = P.prio_mode != 0;
    unsigned long long my_h = 0ull;

    // long rows: one warp per 512-entry item; positions by atomicAdd
    for (int q = gw; q < nC; q += nw) {
        const int2 it = P.items[q];
        const int v = it.x;
        if (v < lo || v >= hi) continue;
        const int g = P.g.graph(v), base = P.g.base(g);
        long long beg;
        int d;
        P.g.row(v, g, beg, d);
        const uint64_t hv = prio_hash(seed, (uint32_t)(v - base));
        const int e0 = it.y * kBuildItem, e1 = min(d, e0 + kBuildItem);
        for (int b0 = e0; b0 < e1; b0 += 32) {
            const int e = b0 + lane;
            int u = -1;
            bool keep = false;
            if (e < e1) {
                u = P.g.nbr(beg + e, base);
                keep = u != v && (all || higher(__ldg(dg + u), u, d, hv, v, base, seed, use_deg));
            }
            const unsigned m = __ballot_sync(kFullMask, keep);
            if (m == 0u) continue;
            int pos = 0;
            if (lane == 0) pos = atomicAdd(P.hlen + v, __popc(m));
            pos = __shfl_sync(kFullMask, pos, 0);
            if (keep) P.hadj[beg + pos + __popc(m & ((1u << lane) - 1u))] = u;
            if (lane == 0) my_h += (unsigned long long)__popc(m);
        }
    }

    // medium rows: one warp per vertex, ordered compaction by ballot
    for (int i = gw; i < nM; i += nw) {
        const int4 ent = P.wm[0][i];
        const int v = ent.x, d = ent.z;
        if (v < lo || v >= hi) continue;
        const int g = P.g.graph(v), base = P.g.base(g);
        const long long beg = P.g.begin(v, ent.w);
        const uint64_t hv = prio_hash(seed, (uint32_t)(v - base));
        int pos = 0;
        for (int b0 = 0; b0 < d; b0 += 32) {
            const int e = b0 + lane;
            int u = -1;
            bool keep = false;
            if (e < d) {
                u = P.g.nbr(beg + e, base);
                keep = u != v && (all || higher(__ldg(dg + u), u, d, hv, v, base, seed, use_deg));
            }
            const unsigned m = __ballot_sync(kFullMask, keep);
            if (keep) P.hadj[beg + pos + __popc(m & ((1u << lane) - 1u))] = u;
            pos += __popc(m);
        }
        if (lane == 0) {
            P.hlen[v] = pos;
            my_h += (unsigned long long)pos;
        }
    }

    // short rows: one thread per vertex
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nS; i += stride) {
        const int4 ent = P.ws[0][i];
        const int v = ent.x, d = ent.z;
        if (v < lo || v >= hi) continue;
        const int g = P.g.graph(v), base = P.g.base(g);
        const long long beg = P.g.begin(v, ent.w);
        const uint64_t hv = prio_hash(seed, (uint32_t)(v - base));
        int pos = 0;
        for (int e0 = 0; e0 < d; e0 += 4) {
            int u[4], du[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) u[j] = e0 + j < d ? P.g.nbr(beg + e0 + j, base) : v;
#pragma unroll
            for (int j = 0; j < 4; ++j) du[j] = u[j] != v ? __ldg(dg + u[j]) : 0;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (u[j] != v && (all || higher(du[j], u[j], d, hv, v, base, seed, use_deg)))
                    P.hadj[beg + pos++] = u[j];
        }
        P.hlen[v] = pos;
        my_h += (unsigned long long)pos;
    }
    my_h = warp_sum(my_h);
    if (lane == 0 && my_h) atomicAdd(&st->h_first, my_h);
}

// ---------------------------------------------------------------------------
// assign: first fit from the forbidden-color set
// ---------------------------------------------------------------------------
// First fit for worklist entry e = {v, |H(v)|, deg(v), local row start}.
// The forbidden set only grows from round to round (committed colors are
// final), so the first free color never decreases: the scan starts at the
// previous round's tentative color tp = -col[v].  w0: v's first 64 colors,
// loaded by the caller together with tp (neither waits for the other).
template <class V>
__device__ __forceinline__ int first_fit(const Problem<V>& P, int4 e, int tp,
                                         unsigned long long w0) {
    const int v = e.x;
    int t;
    if (w0 != ~0ull) {
        t = __ffsll((long long)~w0);
    } else {   // colors 1..64 all taken: deg(v) >= 64, scan the overflow bitmap
        const long long b = P.g.begin(v, e.w);
        const int words = (e.z >> 5) + 1;
        const unsigned* w = P.bmx + P.g.bm(v, b);
        // four words per step, from the word that holds the previous color
        int k = tp > 64 ? (tp - 65) >> 5 : 0;
        for (;;) {
            unsigned x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = k + j < words ? w[k + j] : 0u;
            int j = 0;
            unsigned y = x[0];
            if (y == kFullMask) {
                j = 1;
                y = x[1];
                if (y == kFullMask) {
                    j = 2;
                    y = x[2];
                    if (y == kFullMask) {
                        j = 3;
                        y = x[3];
                    }
                }
            }
            if (y != kFullMask || k + 4 >= words) {
                t = 64 + (k + j) * 32 + __ffs(~y);
                break;
            }
            k += 4;
        }
    }
    return t;
}

template <class V>
__device__ __forceinline__ void assign_phase(const Problem<V>& P, const Hot& h, int r) {
    const int cp = r & 1;
    const int n0 = h.ns[cp], n1 = h.nm[cp], n2 = h.nl[cp];
    const long long total = (long long)n0 + n1 + n2;
    const long long stride = (long long)gridDim.x * blockDim.x;
    // two vertices per thread and step, their loads side by side
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < total;
         i0 += 2 * stride) {
        int4 e[2];
        int tp[2];
        unsigned long long w0[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const long long i = i0 + j * stride;
            e[j] = make_int4(-1, 0, 0, 0);
            if (i < total)
                e[j] = i < n0 ? P.ws[cp][i]
                     : (i < n0 + n1 ? P.wm[cp][i - n0] : P.wl[cp][i - n0 - n1]);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            tp[j] = e[j].x >= 0 ? -P.col[e[j].x] : 0;
            w0[j] = e[j].x >= 0 ? P.bm0[e[j].x] : 0ull;
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (e[j].x >= 0) {
                const int t = first_fit(P, e[j], tp[j], w0[j]);
                if (t != tp[j]) P.col[e[j].x] = -t;
            }
    }
}

// Asynchronous speculation (PGC_ASYNC; the in-place coloring of VB_BIT in
// KokkosKernels, Sec. 3.2): first fit avoids the committed colors of N(v)
// and also every tentative color a neighbor has already written in this
// round (losers were reset to 0 at the end of the previous round, so a
// negative color is this round's).  One warp per worklist vertex scans its
// adjacency once per 64-color window.  Which tentative colors a vertex sees
// depends on timing, so the result is a proper coloring but not a
// deterministic one; detection is the same snapshot rule as always.
template <class V>
__device__ __forceinline__ void assign_async_phase(const Problem<V>& P, const Hot& h) {
    const int cp = h.round & 1;
    const int n0 = h.ns[cp], n1 = h.nm[cp], n2 = h.nl[cp];
    const long long total = (long long)n0 + n1 + n2;
    const int lane = lane_id(), wpb = blockDim.x >> 5;
    const long long gw = (long long)blockIdx.x * wpb + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * wpb;
    for (long long i = gw; i < total; i += nw) {
        const int4 e = i < n0 ? P.ws[cp][i]
                     : (i < n0 + n1 ? P.wm[cp][i - n0] : P.wl[cp][i - n0 - n1]);
        const int v = e.x, d = e.z;
        const int g = P.g.graph(v), base = P.g.base(g);
        const long long beg = P.g.begin(v, e.w);
        int t = 0;
        for (int w = 0; t == 0; ++w) {
            unsigned long long f = 0ull;
            if (w == 0) {
                f = P.bm0[v];
            } else {   // overflow bitmap words for colors 64w+1 .. 64w+64
                const unsigned* x = P.bmx + P.g.bm(v, beg);
                const int k = 2 * (w - 1), words = (d >> 5) + 1;
                const unsigned lo = k < words ? x[k] : 0u;
                const unsigned hi = k + 1 < words ? x[k + 1] : 0u;
                f = ((unsigned long long)hi << 32) | lo;
            }
            unsigned long long tb = 0ull;
            for (int j = lane; j < d; j += 32) {
                const int u = P.g.nbr(beg + j, base);
                const int c = u != v ? *(volatile const int*)(P.col + u) : 0;
                if (c < 0) {
                    const int b = -c - 1 - 64 * w;
                    if (b >= 0 && b < 64) tb |= 1ull << b;
                }
            }
            const unsigned tlo = __reduce_or_sync(kFullMask, (unsigned)tb);
            const unsigned thi = __reduce_or_sync(kFullMask, (unsigned)(tb >> 32));
            f |= ((unsigned long long)thi << 32) | tlo;
            if (f != ~0ull) t = 64 * w + __ffsll((long long)~f);
        }
        if (lane == 0) *(volatile int*)(P.col + v) = -t;
    }
}

template <class V>
__global__ void d1_assign(const Problem<V>* __restrict__ Pp, State* st,
                          cudaGraphConditionalHandle h, int use_cond) {
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        // The loop continues only if this round's detect says so: should its
        // round control ever not run, the device loop ends instead of spinning.
        if (use_cond) cudaGraphSetConditional(h, 0u);
        st->push_cnt = 0;   // the previous round's push kernel has finished
    }
    if (P.async_mode) assign_async_phase(P, ctx.h);
    else assign_phase(P, ctx.h, ctx.h.round);
}

// ---------------------------------------------------------------------------
// detect + commit + compact + inline push (+ round control in the last block)
// ---------------------------------------------------------------------------
// End of round r: record the trace, decide whether to go on, set up round
// r+1.  cur: the round's worklist.  Returns 1 when the coloring is finished (or
// has failed).
template <class V>
__device__ int round_decide(const Problem<V>& P, long long cur) {
    State* st = P.st;
    const int r = st->round;
    const int cp = r & 1, np = cp ^ 1;
    const long long nxt = (long long)*(volatile int*)&st->ns[np] + *(volatile int*)&st->nm[np] +
                          *(volatile int*)&st->nl[np];
    if (r < P.trace_cap) {
        P.trace_w[r] = nxt;
        P.trace_s[r] = (long long)*(volatile unsigned long long*)&st->s_next;
        P.trace_h[r] = (long long)*(volatile unsigned long long*)&st->h_next;
    }
    if (r == 1 && P.trace_cap > 0) P.trace_h[0] = (long long)st->h_first;
    int done = 0, status = ST_OK;
    if (nxt == 0) {
        done = 1;
    } else if (nxt >= cur) {
        done = 1;
        status = ST_NO_PROGRESS;
    } else if (r >= P.max_rounds) {
        done = 1;
        status = ST_MAX_ROUNDS;
    } else if (global_ns() - st->t0 > P.timeout_ns) {
        done = 1;
        status = ST_TIMEOUT;
    }
    if (!done) {
        st->ns[cp] = st->nm[cp] = st->nl[cp] = 0;
        st->round = r + 1;
        st->s_next = 0ull;
        st->h_next = 0ull;
    }
    st->status = status;
    st->done = done;
    st->blocks_done = 0u;
    st->mid = (!done && nxt <= P.mid_w) ? 1 : 0;
    __threadfence();
    return done;
}

// Round control of the launch-per-round loop: the WHILE node repeats while
// the coloring is unfinished and the worklist is larger than mid_w; the
// remaining rounds go to the mid loop.
template <class V>
__device__ void round_control(const Problem<V>& P, cudaGraphConditionalHandle h, int use_cond) {
    const int cp = P.st->round & 1;
    const int done = round_decide(P, (long long)P.st->ns[cp] + P.st->nm[cp] + P.st->nl[cp]);
    if (use_cond) cudaGraphSetConditional(h, (done || P.st->mid) ? 0u : 1u);
}

// Queue the pushes of the lanes with pred (all 32 call): ceil(deg / kPushItem)
// work items each, one atomic for all of them.
template <class V>
__device__ __forceinline__ void queue_push(const Problem<V>& P, bool pred, int v, int d) {
    if (!__any_sync(kFullMask, pred)) return;
    const int lane = lane_id(), nit = pred ? ceil_div(d, kPushItem) : 0;
    int incl = nit;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += y;
    }
    int base = 0;
    if (lane == 31) base = atomicAdd(&P.st->push_cnt, incl);
    base = __shfl_sync(kFullMask, base, 31) + incl - nit;
    for (int k = 0; k < nit; ++k) P.push_q[base + k] = make_int2(v, k);
}

// The vertex v whose list is being checked, with what a priority that
// changes each round needs: its priority this round and its hash.
struct Me {
    int v, p, base;
    uint64_t h;
};
struct NoMe {};   // the static order needs nothing about v
template <bool DYN>
using MeOf = typename std::conditional<DYN, Me, NoMe>::type;

template <class V>
__device__ __forceinline__ Me round_me(const Problem<V>& P, int v, int g) {
    const int base = P.g.base(g);
    return Me{v, P.prio[v], base, prio_hash(P.seed, (uint32_t)(v - base))};
}

// Priorities that change each round (Sec. 3.3, closing paragraph): u beats v
// when its priority this round is larger; ties go to the smaller hash, then
// the smaller id (Alg. 4 with the priority in place of the degree).
template <class V>
__device__ __forceinline__ bool beats(const Problem<V>& P, int u, const Me& me) {
    const int pu = P.prio[u];
    if (pu != me.p) return pu > me.p;
    const uint64_t hu = prio_hash(P.seed, (uint32_t)(u - me.base));
    if (hu != me.h) return hu < me.h;
    return u < me.v;
}

// u (an entry of v's list, < 0: none) holds v's tentative color t and, with
// DYN, beats v this round.  Without DYN the list holds only neighbors with
// priority over v (a static order), so the color alone decides.
template <bool DYN, class V>
__device__ __forceinline__ bool conflict(const Problem<V>& P, int u, int t, MeOf<DYN> me) {
    if constexpr (DYN) return u >= 0 && abs(P.col[u]) == t && beats(P, u, me);
    else return u >= 0 && abs(P.col[u]) == t;
}

// What detection adds up per lane over a round.
struct RoundSums {
    int max_color = 0;
    unsigned long long s = 0ull, h = 0ull;   // degrees and list lengths of the losers
};

// A step over the rows of the lanes in `open` (not empty): 128 places, the
// same power of two of consecutive entries for each row, at least four.  Place
// f = 32 j + lane (j = 0..3) is entry f % per of the row with rank f / per.
struct Deal {
    int n, log;   // rows; log2 of the entries per row
};
__device__ __forceinline__ Deal deal_rows(unsigned open, unsigned char* slot) {
    const int lane = lane_id();
    Deal d;
    d.n = __popc(open);
    d.log = d.n == 1 ? 7 : __clz(d.n - 1) - 25;
    __syncwarp();
    if (open >> lane & 1u) slot[__popc(open & ((1u << lane) - 1u))] = (unsigned char)lane;
    __syncwarp();
    return d;
}
// The lane whose row has place 32 j + lane (-1: none).
__device__ __forceinline__ int deal_lane(const Deal& d, const unsigned char* slot, int j) {
    const int i = (32 * j + (int)lane_id()) >> d.log;
    return i < d.n ? slot[i] : -1;
}
// Does the row with this rank have a place in the four ballots?
__device__ __forceinline__ bool deal_any(const Deal& d, int rank, const unsigned (&b)[4]) {
    if (d.log >= 7) return (b[0] | b[1] | b[2] | b[3]) != 0u;
    if (d.log == 6) return (rank ? b[2] | b[3] : b[0] | b[1]) != 0u;
    const int from = rank << d.log, j = from >> 5;
    const unsigned w = j == 0 ? b[0] : j == 1 ? b[1] : j == 2 ? b[2] : b[3];
    return (w >> (from & 31) & (kFullMask >> (32 - (1 << d.log)))) != 0u;
}

// ---------------------------------------------------------------------------
// setup 3: worklists by |H(v)|, and round 1
// ---------------------------------------------------------------------------
// In round 1 every vertex holds color 1, so v wins exactly when H(v) is empty,
// and no list is read: the winners commit here and the others are round 2's
// worklists (a pass over all entries less: 5.0 of 52 ms for the 4096-graph
// batch).  None of a winner's neighbors wins, so its pushes ask nobody.  With
// PGC_ASYNC or a round-varying priority round 1 is a round like any other.
template <class V>
__device__ __forceinline__ bool round1_in_setup(const Problem<V>& P) {
    return !P.async_mode && !P.prio_mode;
}

// The last block to finish ends round 1 (all threads call).
template <class V>
__device__ __forceinline__ void end_round1(const Problem<V>& P, State* st) {
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(&st->blocks_done, 1u) == gridDim.x - 1;
        if (s_last) {
            __threadfence();
            st->max_color = 1;
            st->pend = 1;
            round_decide(P, P.n);
            if (*(volatile int*)&st->lists_full) {
                st->status = ST_LISTS;
                st->done = 1;
                st->mid = 0;
            }
        }
    }
}

template <class V>
__global__ void d1_tier(const Problem<V>* __restrict__ Pp, State* st) {
    __shared__ int s_n[2][33];
    __shared__ unsigned char s_slot[32][32];
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    const int n = P.n, lane = lane_id();
    const bool first = round1_in_setup(P), traced = P.trace_cap > 0;
    const int p = first ? 0 : 1;   // parity of the worklists made here
    unsigned char* const slot = s_slot[threadIdx.x >> 5];
    unsigned long long sum_s = 0ull, sum_h = 0ull;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long base = (long long)blockIdx.x * blockDim.x; base < n; base += stride) {
        const long long i = base + threadIdx.x;
        const bool valid = i < n;
        int4 e = make_int4((int)i, 0, 0, 0);   // {v, |H(v)|, deg(v), row start}
        if (valid) {
            int r0, d;
            P.g.local_row((int)i, P.g.graph((int)i), r0, d);
            e = make_int4((int)i, P.hlen[i], d, r0);
        }
        const bool win = valid && first && e.y == 0, go_on = valid && !win;
        block_append(go_on && e.y <= P.det_s, go_on && e.y > P.det_s && e.y <= P.det_m, e, P.ws[p],
                     &st->ns[p], P.wm[p], &st->nm[p], s_n);
        if (go_on && e.y > P.det_m) P.wl[p][atomicAdd(&st->nl[p], 1)] = e;
        if (!first) continue;
        if (traced && go_on) {
            sum_s += (unsigned long long)e.z;
            sum_h += (unsigned long long)e.y;
        }
        const unsigned wins = __ballot_sync(kFullMask, win);
        if (!wins) continue;
        int g = 0;
        if (win) {
            P.col[e.x] = 1;
            if (P.g_rounds != nullptr) g = P.g.graph(e.x);
        }
        if (lane == __ffs(wins) - 1) P.live[e.x >> 5] &= ~wins;   // 32 vertices, one word
        if (P.g_rounds != nullptr) graph_max(P.g_colors, win, g, 1);
        queue_push(P, win && e.z > kInlinePush, e.x, e.z);
        const long long beg = win ? P.g.begin(e.x, e.w) : 0;
        const int nb = win ? P.g.base(P.g.graph(e.x)) : 0;
        unsigned open = __ballot_sync(kFullMask, win && e.z > 0 && e.z <= kInlinePush);
        for (int pos = 0; open;) {   // the neighbors' bit for color 1
            const Deal deal = deal_rows(open, slot);
            const int per = 1 << deal.log;
            int u[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int src = deal_lane(deal, slot, j), from = src < 0 ? lane : src;
                const int x = pos + ((32 * j + lane) & (per - 1));
                const int len = __shfl_sync(kFullMask, e.z, from);
                const int v = __shfl_sync(kFullMask, e.x, from);
                const int ub = __shfl_sync(kFullMask, nb, from);
                const long long b = __shfl_sync(kFullMask, beg, from);
                u[j] = src >= 0 && x < len ? P.g.nbr(b + x, ub) : -1;
                if (u[j] == v) u[j] = -1;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (u[j] >= 0) atomicOr(P.bm0 + u[j], 1ull);
            pos += per;
            open = __ballot_sync(kFullMask, (open >> lane & 1u) && pos < e.z);
        }
    }
    if (first) {
        if (traced) {
            sum_s = warp_sum(sum_s);
            sum_h = warp_sum(sum_h);
            if (lane == 0 && (sum_s || sum_h)) {
                atomicAdd(&st->s_next, sum_s);
                atomicAdd(&st->h_next, sum_h);
            }
        }
        end_round1(P, st);
    } else if (blockIdx.x == 0 && threadIdx.x == 0 && n <= P.mid_w) {
        st->mid = 1;   // all rounds in the mid loop
    }
}

// One tier's worklist: conflict search, commit, inline push and re-append.
//
// A warp takes up to 32 worklist vertices and searches their lists together:
// in each step the lists still undecided get the same number of places, so a
// step has up to 128 independent gathers in flight and costs two dependent
// loads however many lists it serves.  Losers meet their conflict within the
// first entries (a mean of 2 to 12 on meshes, patterns and R-MAT) and leave;
// their places go to those that must read on, at last 128 entries per step
// for one winner.  Consecutive lanes take consecutive entries: an instruction
// then touches one line per row instead of one per lane, and lines per
// instruction are what the first-level cache is bound by here (random gathers:
// 290 G/s measured, one line per SM and cycle).  Small worklists are spread
// over the warps first (fewer vertices per warp, more places for each).  The
// winners' pushes deal their rows in the same way.
//
// One thread or one warp per vertex with lists read alone, in turn, waited for
// the longest list of a warp; with the shared counters read once per block
// (Hot) and appended to once per block, detection of R-MAT 20's first 13
// rounds went from 0.86 to 0.57 ms, of PD2 4M x 1M's 51 rounds from 9.6 to
// 4.6 ms, of the 4096-graph batch from 56 to 31 ms.  64 registers (4 blocks
// per SM) beat 48 with spills (whole colorings: 46.8 against 50.9 ms for the
// batch, 28.0 against 28.6 for R-MAT 24, 11.5 against 11.7 for PD2 4M x 1M).
template <bool DYN, class V>
__device__ __forceinline__ void detect_tier(const Problem<V>& P, const int4* list, int n, int4* next,
                                            int* next_cnt, IdxAppend& app, unsigned char* slot,
                                            int r, RoundSums& sum) {
    const int* __restrict__ ha = P.hadj;
    int* const col = P.col;
    const bool batch = P.g_rounds != nullptr, traced = P.trace_cap > 0;
    const int lane = lane_id(), wpb = blockDim.x >> 5;
    const long long gw = (long long)blockIdx.x * wpb + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * wpb;
    int take = 32;   // vertices per warp: the smallest power of two that is one pass
    while (take > 1 && (take >> 1) * nw >= n) take >>= 1;
    using Off = typename V::Off;
    int4 ahead = make_int4(0, 0, 0, 0);   // the next vertex's entry, one step ahead
    if (lane < take && gw * take + lane < n) ahead = list[gw * take + lane];
    for (long long i0 = gw * take; i0 < n; i0 += nw * take) {
        const long long i = i0 + lane;
        const bool valid = lane < take && i < n;
        const int4 ent = ahead;
        if (i + nw * take < n && lane < take) ahead = list[i + nw * take];
        int t = 0;
        Off beg = 0;
        MeOf<DYN> me{};
        if (valid) {
            beg = P.g.begin(ent.x, ent.w);
            t = -col[ent.x];
            if constexpr (DYN) me = round_me(P, ent.x, P.g.graph(ent.x));
        }
        const int v = ent.x, hl = ent.y, d = ent.z;
        bool lose = false;
        int pos = 0;   // entries read of every list still open
        unsigned open = __ballot_sync(kFullMask, valid && hl > 0);
        while (open) {   // warp-uniform
            const Deal deal = deal_rows(open, slot);
            const int per = 1 << deal.log;
            int u[4], ut[4];
            MeOf<DYN> ume[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int src = deal_lane(deal, slot, j), from = src < 0 ? lane : src;
                const int x = pos + ((32 * j + lane) & (per - 1));
                const int len = __shfl_sync(kFullMask, hl, from);
                const Off b = __shfl_sync(kFullMask, beg, from);
                ut[j] = __shfl_sync(kFullMask, t, from);
                if constexpr (DYN) {
                    ume[j].v = __shfl_sync(kFullMask, me.v, from);
                    ume[j].p = __shfl_sync(kFullMask, me.p, from);
                    ume[j].base = __shfl_sync(kFullMask, me.base, from);
                    ume[j].h = __shfl_sync(kFullMask, me.h, from);
                }
                u[j] = src >= 0 && x < len ? __ldg(ha + b + x) : -1;
            }
            bool hit[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) hit[j] = conflict<DYN>(P, u[j], ut[j], ume[j]);
            unsigned hits[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) hits[j] = __ballot_sync(kFullMask, hit[j]);
            bool mine = open >> lane & 1u;
            if (mine) {
                lose = deal_any(deal, __popc(open & ((1u << lane) - 1u)), hits);
                mine = !lose && pos + per < hl;
            }
            pos += per;
            open = __ballot_sync(kFullMask, mine);
        }
        const bool win = valid && !lose;
        const int g = batch && win ? P.g.graph(v) : 0;
        if (lose) {
            sum.s += (unsigned long long)(V::kSetup ? d : traced ? P.g.degree(v, d) : 0);
            sum.h += (unsigned long long)hl;
        }
        if (win) {
            col[v] = t;
            atomicAnd(P.live + (v >> 5), ~(1u << (v & 31)));
            sum.max_color = max(sum.max_color, t);
        }
        // with DYN every push is queued: an inline one would change
        // neighbors' priorities while others still compare them
        queue_push(P, win && (d > kInlinePush || DYN), v, d);
        if (batch) {
            graph_max(P.g_rounds, win, g, r);
            graph_max(P.g_colors, win, g, t);
        }
        if (!DYN) {
            pos = 0;
            open = __ballot_sync(kFullMask, win && d <= kInlinePush && d > 0);
            while (open) {
                const Deal deal = deal_rows(open, slot);
                const int per = 1 << deal.log;
                int u[4], from[4];
                unsigned lw[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int src = deal_lane(deal, slot, j);
                    from[j] = src < 0 ? lane : src;
                    const int x =
                        __shfl_sync(kFullMask, pos, from[j]) + ((32 * j + lane) & (per - 1));
                    const int len = __shfl_sync(kFullMask, d, from[j]);
                    const Off b = __shfl_sync(kFullMask, beg, from[j]);
                    const int uv = __shfl_sync(kFullMask, v, from[j]);
                    const int ug = __shfl_sync(kFullMask, g, from[j]);
                    u[j] = src >= 0 && x < len ? P.g.nbr(b + x, P.g.base(ug)) : -1;
                    if (u[j] == uv) u[j] = -1;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) lw[j] = u[j] >= 0 ? P.live[u[j] >> 5] : 0u;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int ug = __shfl_sync(kFullMask, g, from[j]);
                    const int uc = __shfl_sync(kFullMask, t, from[j]);
                    if ((lw[j] >> (u[j] & 31)) & 1u) push_color_live<false>(P, u[j], ug, uc);
                }
                bool mine = open >> lane & 1u;
                if (mine) {
                    pos += per;
                    mine = pos < d;
                }
                open = __ballot_sync(kFullMask, mine);
            }
        }
        ia_push(app, lose, (int)i, list, next, next_cnt);
    }
}

// Detection, commit, compaction and inline push for one round (every block
// of the grid takes part).  DYN: priorities that change each round -- the
// lists then hold every neighbor, and a neighbor holding v's color must also
// beat v this round.
template <class V, bool DYN>
__device__ __forceinline__ void detect_phase(const Problem<V>& P, const Hot& hot, int r,
                                             int* smem) {
    __shared__ unsigned char s_slot[32][32];
    __shared__ int s_n[2][33], s_max;
    State* st = P.st;
    const int cp = r & 1, np = cp ^ 1;
    const int nS = hot.ns[cp], nM = hot.nm[cp], nL = hot.nl[cp];
    const int* __restrict__ ha = P.hadj;
    int* col = P.col;
    const int lane = lane_id();
    const int warp = threadIdx.x >> 5;
    RoundSums sum;
    // losers keep their entry and tier: appended by source index
    IdxAppend app_s = {smem + warp * 2 * kIdxSlots, 0};
    IdxAppend app_m = {smem + warp * 2 * kIdxSlots + kIdxSlots, 0};

    // --- L tier: one block per vertex (static assignment), four entries per
    // thread and step ---
    for (int i = blockIdx.x; i < nL; i += gridDim.x) {
        const int4 ent = P.wl[cp][i];
        const int v = ent.x, hl = ent.y, d = ent.z;
        const int g = P.g.graph(v);
        const long long beg = P.g.begin(v, ent.w);
        const int t = -col[v];
        MeOf<DYN> me{};
        if constexpr (DYN) me = round_me(P, v, g);
        bool lose = false;
        for (int b0 = 0; b0 < hl && !lose; b0 += 4 * blockDim.x) {
            int u[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int e = b0 + j * blockDim.x + threadIdx.x;
                u[j] = e < hl ? __ldg(ha + beg + e) : -1;
            }
            bool hit = false;
#pragma unroll
            for (int j = 0; j < 4; ++j) hit |= conflict<DYN>(P, u[j], t, me);
            lose = __syncthreads_or(hit);
        }
        if (threadIdx.x == 0) {
            if (lose) {
                P.wl[np][atomicAdd(&st->nl[np], 1)] = ent;
                sum.s += (unsigned long long)P.g.degree(v, d);
                sum.h += (unsigned long long)hl;
            } else {
                col[v] = t;
                atomicAnd(P.live + (v >> 5), ~(1u << (v & 31)));
                sum.max_color = max(sum.max_color, t);
                if (P.g_rounds != nullptr) {
                    atomicMax(P.g_rounds + g, r);
                    atomicMax(P.g_colors + g, t);
                }
            }
        }
        if (warp == 0) queue_push(P, lane == 0 && !lose, v, d);
        __syncthreads();
    }

    // --- M tier, then S tier: longer lists first ---
    detect_tier<DYN>(P, P.wm[cp], nM, P.wm[np], &st->nm[np], app_m, s_slot[warp], r, sum);
    detect_tier<DYN>(P, P.ws[cp], nS, P.ws[np], &st->ns[np], app_s, s_slot[warp], r, sum);

    // --- what is left in the appenders, and the totals, once per block: one
    // atomic per warp on the same address would take as long as a small round
    if (threadIdx.x == 0) s_max = 0;
    if (lane == 0) {
        s_n[0][warp] = app_s.count;
        s_n[1][warp] = app_m.count;
    }
    __syncthreads();
    const int my_max = warp_max(sum.max_color);
    if (lane == 0 && my_max > hot.max_color) atomicMax(&s_max, my_max);
    if (warp < 2) {
        const int x = lane < (int)(blockDim.x >> 5) ? s_n[warp][lane] : 0;
        int incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFullMask, incl, o);
            if (lane >= o) incl += y;
        }
        int base = 0;
        if (lane == 31 && incl) base = atomicAdd(warp ? &st->nm[np] : &st->ns[np], incl);
        base = __shfl_sync(kFullMask, base, 31);
        if (lane < (int)(blockDim.x >> 5)) s_n[warp][lane] = base + incl - x;
    }
    __syncthreads();
    for (int k = lane; k < app_s.count; k += 32)
        P.ws[np][s_n[0][warp] + k] = P.ws[cp][app_s.buf[k]];
    for (int k = lane; k < app_m.count; k += 32)
        P.wm[np][s_n[1][warp] + k] = P.wm[cp][app_m.buf[k]];
    if (threadIdx.x == 0 && s_max > 0) atomicMax(&st->max_color, s_max);
    if (P.trace_cap > 0) {
        const unsigned long long my_s = warp_sum(sum.s), my_h = warp_sum(sum.h);
        if (lane == 0 && (my_s || my_h)) {
            atomicAdd(&st->s_next, my_s);
            atomicAdd(&st->h_next, my_h);
        }
    }
}

template <class V, bool DYN = false>
__global__ void __maxnreg__(64) d1_detect(const Problem<V>* __restrict__ Pp, State* st,
                                          cudaGraphConditionalHandle h, int use_cond) {
    extern __shared__ int smem[];
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    if (ctx.h.mid || ctx.h.done) return;   // handed over before round 1, or no lists
    detect_phase<V, DYN>(P, ctx.h, ctx.h.round, smem);

    // --- last block runs the round control ---
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned ticket = atomicAdd(&st->blocks_done, 1u);
        s_last = ticket == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last && threadIdx.x == 0) {
        __threadfence();
        round_control(P, h, use_cond);
    }
}

// ---------------------------------------------------------------------------
// push: winners' colors into the forbidden sets of their neighbors
// ---------------------------------------------------------------------------
template <class V>
__device__ __forceinline__ void push_phase(const Problem<V>& P, int nq) {
    const int lane = lane_id(), wpb = blockDim.x >> 5;
    for (int q = blockIdx.x * wpb + (threadIdx.x >> 5); q < nq; q += gridDim.x * wpb) {
        const int2 item = P.push_q[q];
        const int v = item.x;
        const int c = P.col[v];
        const int g = P.g.graph(v), base = P.g.base(g);
        long long beg;
        int d;
        P.g.row(v, g, beg, d);
        const int e0 = item.y * kPushItem, e1 = min(e0 + kPushItem, d);
        for (int b0 = e0; b0 < e1; b0 += 128) {
            int u[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int e = b0 + j * 32 + lane;
                u[j] = e < e1 ? P.g.nbr(beg + e, base) : -1;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (u[j] >= 0 && u[j] != v) push_color(P, u[j], g, c);
        }
    }
}

// PGC_ASYNC: the next round's worklist vertices start uncolored (0), so that
// a negative color seen during its first fit is one written in that round.
template <class V>
__device__ __forceinline__ void reset_next_worklist(const Problem<V>& P, const Hot& h) {
    if (h.done) return;
    const int p = h.round & 1;
    const int n0 = h.ns[p], n1 = h.nm[p], n2 = h.nl[p];
    const long long total = (long long)n0 + n1 + n2;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += stride) {
        const int v = i < n0 ? P.ws[p][i].x
                    : (i < n0 + n1 ? P.wm[p][i - n0].x : P.wl[p][i - n0 - n1].x);
        P.col[v] = 0;
    }
}

template <class V>
__global__ void d1_push(const Problem<V>* __restrict__ Pp, State* st,
                        cudaGraphConditionalHandle h, int use_cond) {
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->pend = 0;
        // before the loop: round 1 has ended, does another one follow?
        if (use_cond) cudaGraphSetConditional(h, ctx.h.done || ctx.h.mid ? 0u : 1u);
    }
    push_phase(P, ctx.h.push_cnt);
    if (P.async_mode) reset_next_worklist(P, ctx.h);
}

// ---------------------------------------------------------------------------
// mid loop: the rounds of a worklist that does not fill the GPU
// ---------------------------------------------------------------------------
// Test hook: the calling thread waits ns nanoseconds (the host sets at most 2 s).
__device__ __forceinline__ void be_late(unsigned ns) {
    const unsigned long long t_end = global_ns() + ns;
    while (global_ns() < t_end) __nanosleep(1000);
}

// Grid-wide barrier for a cooperative launch (all blocks co-resident), then
// the block's copy of the counters.  Arrivals only count up and everyone polls
// the count itself, so nobody waits for an atomic's answer or for a second
// word to be written.  `phase`: barriers passed so far.  A wait that exceeds
// max_polls polls (2^22: about a second) gives up, records the failure and
// lets the kernel return with an error.
__device__ __forceinline__ bool grid_barrier(State* st, Hot& h, unsigned& phase,
                                             unsigned max_polls) {
    __shared__ int s_ok;
    __syncthreads();
    ++phase;
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) {
            const unsigned target = phase * gridDim.x;
            int ok = 1;
            asm volatile("red.release.gpu.add.u32 [%0], 1;" ::"l"(&st->bar_count) : "memory");
            unsigned polls = 0, now;
            for (;;) {
                asm volatile("ld.acquire.gpu.u32 %0, [%1];"
                             : "=r"(now) : "l"(&st->bar_count) : "memory");
                if (now >= target) break;
                ++polls;
                if (polls > max_polls || ((polls & 15u) == 0u && *(volatile int*)&st->bar_timeout)) {
                    atomicExch(&st->bar_timeout, 1);
                    ok = 0;
                    break;
                }
                if (polls > 64u) __nanosleep(64);
            }
            s_ok = ok;
        }
        __syncwarp();
        read_hot(h, st);
    }
    __syncthreads();
    return s_ok != 0;
}

constexpr int kMidMax = 65536;     // worklists up to this size
constexpr int kCoreRounds = 8;    // core phase: at this pace, rounds ahead
constexpr int kMidShared = 8;      // blocks when several colorings share the GPU (the server) ...
constexpr int kMidSharedMax = 16384;  // ... and their worklists

// The rounds (assign, detect, push) in one cooperative launch, one block per
// SM, grid barriers in place of launches.  Every block takes the same round
// decisions from the counters, so there is no last block to wait for; block 0
// prepares the next round's counters while everyone assigns.  What bounds a
// round is its chain of dependent loads (about 10,000 cycles in detection for
// any worklist) and two or three barriers of 2 to 3 us.
//
// kMidMax: on GB300 the loop is even with launched rounds at 262,144 vertices
// (PD2 4M x 1M 12.13 ms against 11.98) and ahead below (a 7-point mesh of
// 32^3 vertices 0.175 ms with 16,384 here, 0.150 with 65,536).
//
// The remaining rounds go to the core phase when the worklist fits it and
// shrinks slowly (a dense core: many rounds ahead; R-MAT 24 30.6 ms when the
// core phase takes over at 1,024 vertices, 28.7 at 4,096); a worklist that is
// about to run out finishes here.
//
// A server colors on many streams: 8 blocks per request leave the SMs to the
// others (32 requests: 38.7 ms with a block per SM, 22.7 with 8 blocks up to
// 8,192 vertices, 20.9 up to 16,384).
//
// T threads per block: 1024 for worklists that come from the launched rounds
// (R-MAT 24 27.8 ms against 29.1 with 512), 512 for problems that are small
// from the start and for round-varying priorities, whose code then does not
// spill (PD2 40K x 10K 1.02 -> 0.97 ms, R-MAT 18 with the dynamic degree 4.44
// -> 4.13).
template <class V, bool DYN, int T>
__global__ void __launch_bounds__(T, 1) d1_mid(const Problem<V>* __restrict__ Pp, State* st) {
    extern __shared__ int smem[];
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    Hot& h = ctx.h;
    if (h.done || !h.mid) return;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    unsigned phase = 0u;
    auto barrier = [&] {
        if ((int)blockIdx.x == P.mid_wait.slow_block && (int)phase + 1 == P.mid_wait.slow_at &&
            threadIdx.x == 0)
            be_late(P.mid_wait.slow_ns);
        return grid_barrier(st, h, phase, P.mid_wait.polls);
    };
    int r = h.round, cur = h.count(r & 1), status = ST_OK, done = 0, tail = 0;
    const int first = r;   // (the round before it looked at the clock itself)
    const unsigned long long t0 = lead ? st->t0 : 0ull, timeout_ns = P.timeout_ns;
    bool ok = true;
    if (h.pend && h.push_cnt > 0) {   // round 1's
        push_phase(P, h.push_cnt);
        ok = barrier();
    }
    while (ok) {
        const int np = (r & 1) ^ 1;
        unsigned long long now = 0ull;
        if (lead) {
            st->push_cnt = 0;
            st->ns[np] = st->nm[np] = st->nl[np] = 0;
            st->s_next = st->h_next = 0ull;
            // the end of the last round; the timer is slow to read, so its value
            // is used behind the barrier only
            now = global_ns();
        }
        if (!DYN || r > 1) assign_phase(P, h, r);
        if (!barrier()) break;
        if (lead && r > first && now - t0 > timeout_ns) st->stop = r;
        detect_phase<V, DYN>(P, h, r, smem);
        if (!barrier()) break;
        const int nxt = h.count(np), pushes = h.push_cnt;
        if (lead && P.trace_cap > 0) {
            if (r < P.trace_cap) {
                P.trace_w[r] = nxt;
                P.trace_s[r] = (long long)*(volatile unsigned long long*)&st->s_next;
                P.trace_h[r] = (long long)*(volatile unsigned long long*)&st->h_next;
            }
            if (r == 1) P.trace_h[0] = (long long)st->h_first;
        }
        if (h.stop) status = ST_TIMEOUT;   // passed before this round began
        else if (nxt == 0) done = 1;
        else if (nxt >= cur) status = ST_NO_PROGRESS;
        else if (r >= P.max_rounds) status = ST_MAX_ROUNDS;
        if (done || status != ST_OK) break;
        tail = nxt <= P.tail_w && (long long)(cur - nxt) * kCoreRounds < nxt;
        cur = nxt;
        ++r;
        if (pushes > 0) push_phase(P, pushes);
        if (tail) break;
        if (pushes > 0 && !barrier()) break;   // the next assign reads what they wrote
    }
    if (lead) {   // the counters of round r are in place for the core phase
        const int gave_up = *(volatile int*)&st->bar_timeout;
        st->round = r;
        st->status = gave_up ? ST_MID_BARRIER : status;
        st->done = gave_up || done || status != ST_OK;
        st->tail = tail;
        st->mid = 0;
    }
}

// ---------------------------------------------------------------------------
// core: the last rounds on the subgraph induced by the worklist
// ---------------------------------------------------------------------------
// Once the worklist W is small (at most tail_w vertices), the remaining
// rounds only ever involve W: a vertex outside W is committed, so it can no
// longer conflict (first fit avoids committed colors) and its forbidden set
// is never read again.  R-MAT's dense core needs hundreds of such rounds with
// little work in each, so what counts is the time of an empty round.  The
// core phase therefore
//   1. ranks W by priority (Alg. 4's order; rank 0 wins every conflict) and
//      writes the induced adjacency as a bit matrix over the ranks;
//   2. runs the rounds in ONE thread-block cluster: CTA c of C owns the ranks
//      congruent to c modulo C and keeps their matrix rows, forbidden colors
//      and state in its shared memory.  Every CTA holds all tentative colors;
//      what changes in a round (new tentative colors, the winners) is stored
//      into the other CTAs' shared memory, and a round has two cluster
//      barriers: nothing in it waits for global memory;
//   3. writes the colors back.
// The rounds are the same rounds the per-round kernels would run (same
// first fit on the same forbidden sets, same loser rule, same snapshot), so
// colors, round count and trace are unchanged.
//
// Scratch: the rank of v in hlen[v] (the list lengths are dead after setup),
// per-vertex arrays in the other parity's worklist buffers (3 x 16n bytes),
// the bit matrix in its own buffer.

constexpr int kCoreMax = 4096;      // vertices: at 16 CTAs, 256 rows of 512 bytes each in shared memory
constexpr int kCoreCluster = 16;    // CTAs of the cluster (non-portable size)
constexpr int kCoreThreads = 512;
constexpr int kCoreWin = 16;        // per row: forbidden-color words held (512 colors)
constexpr int kUploadChunks = 8;    // host adjacency uploaded in this many row ranges

// Adjacency still in (pinned) host memory when a coloring starts: it is
// copied in kUploadChunks row ranges on a second stream, and the list build
// of each range starts as soon as its rows have arrived, so the transfer
// overlaps the build.
struct Upload {
    const int* h_ci;   // host adjacency
    const int* h_rp;   // host row offsets (chunk boundaries)
    int* d_ci;         // device copy (the view's adjacency)
};
constexpr int kCoreWarpList = 2048; // lists up to this length: one warp; longer: one block

struct CoreArrays {
    int4* lent;    // [k] by rank: worklist entry {v, |H(v)|, deg, local row start}
    int* vid;      // [k] by rank: global id
    int* tent;     // [k] by rank: last tentative color
    ulonglong2* key;   // [k] by worklist position: smaller = higher priority
};

template <class V>
__device__ __forceinline__ CoreArrays core_arrays(const Problem<V>& P, int par, int k) {
    CoreArrays a;
    a.lent = P.ws[par];
    int* m = reinterpret_cast<int*>(P.wm[par]);
    a.vid = m;
    a.tent = m + k;
    a.key = reinterpret_cast<ulonglong2*>(P.wl[par]);
    return a;
}

template <class V>
__device__ __forceinline__ int4 core_entry(const Problem<V>& P, int cp, int nS, int nM, int i) {
    return i < nS ? P.ws[cp][i] : (i < nS + nM ? P.wm[cp][i - nS] : P.wl[cp][i - nS - nM]);
}

__device__ __forceinline__ bool is_live(const unsigned* live, int u) {
    return (live[u >> 5] >> (u & 31)) & 1u;
}

__device__ __forceinline__ int core_words(int k) { return (k + 31) >> 5; }

// Phase 1a: a sortable priority key per worklist vertex; the matrix cleared.
template <class V>
__global__ void d1_core_keys(const Problem<V>* __restrict__ Pp, State* st) {
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    const Hot& h = ctx.h;
    if (h.done || !h.tail) return;
    const int cp = h.round & 1, np = cp ^ 1;
    const int nS = h.ns[cp], nM = h.nm[cp], k = h.count(cp);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->core_k = k;
        st->core_par = np;
        // A block of the mid loop may have given up at its last barrier just as the
        // others passed it, too late for their report: its pushes are missing.
        // (Asked here and not in the loop, whose rounds took 0.8 us longer with it.)
        if (*(volatile int*)&st->bar_timeout) {
            st->status = ST_MID_BARRIER;
            st->done = 1;
        }
    }
    const CoreArrays A = core_arrays(P, np, k);
    const int t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    for (int i = t; i < k; i += nt) {
        const int4 e = core_entry(P, cp, nS, nM, i);
        const int v = e.x;
        const uint64_t h =
            prio_hash(P.seed, (uint32_t)(v - P.g.base(P.g.graph(v))));
        const unsigned nd = P.use_deg ? ~(unsigned)P.g.degree(v, e.z) : 0u;
        A.key[i] = make_ulonglong2(((unsigned long long)nd << 32) | (h >> 32),
                                   (h << 32) | (unsigned)v);
    }
    const int total = k * core_words(k);
    for (int i = t; i < total; i += nt) P.core_mat[i] = 0u;
}

// Phase 1b: rank by counting (k <= 4096 keys, a tile of them in shared
// memory at a time; each warp ranks four vertices), arrays in rank order.
constexpr int kRankTile = 1024;
template <class V>
__global__ void d1_core_rank(const Problem<V>* __restrict__ Pp, State* st) {
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    const Hot& h = ctx.h;
    if (h.done || !h.tail) return;
    __shared__ ulonglong2 tile[kRankTile];
    const int cp = h.round & 1;
    const int nS = h.ns[cp], nM = h.nm[cp], k = h.count(cp);
    const CoreArrays A = core_arrays(P, cp ^ 1, k);
    const int lane = lane_id(), warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int per = wpb * 4;
    for (int b0 = blockIdx.x * per; b0 < k; b0 += gridDim.x * per) {
        const int i0 = b0 + warp * 4;
        ulonglong2 me[4];
        int cnt[4] = {0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < 4; ++q)
            me[q] = i0 + q < k ? A.key[i0 + q] : make_ulonglong2(0ull, 0ull);
        for (int t0 = 0; t0 < k; t0 += kRankTile) {
            const int m = min(kRankTile, k - t0);
            __syncthreads();
            for (int i = threadIdx.x; i < m; i += blockDim.x) tile[i] = A.key[t0 + i];
            __syncthreads();
            for (int i = lane; i < m; i += 32) {
                const ulonglong2 o = tile[i];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    cnt[q] += o.x < me[q].x || (o.x == me[q].x && o.y < me[q].y);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int rank = (int)__reduce_add_sync(kFullMask, (unsigned)cnt[q]);
            if (lane == 0 && i0 + q < k) {
                const int4 e = core_entry(P, cp, nS, nM, i0 + q);
                A.lent[rank] = e;
                A.vid[rank] = e.x;
                A.tent[rank] = -P.col[e.x];
                P.hlen[e.x] = rank;
            }
        }
    }
}

// Phase 1c: the induced adjacency.  Every edge is in the list H of its
// lower-priority end, and both ends of an induced edge are uncolored, so the
// lists of W (shorter than its rows) give both bits of each edge.
template <class V>
__device__ __forceinline__ void core_edge(const Problem<V>& P, int i, int u, int words) {
    if (!is_live(P.live, u)) return;
    const int j = P.hlen[u];
    atomicOr(P.core_mat + (size_t)i * words + (j >> 5), 1u << (j & 31));
    atomicOr(P.core_mat + (size_t)j * words + (i >> 5), 1u << (i & 31));
}

template <class V>
__global__ void d1_core_bits(const Problem<V>* __restrict__ Pp, State* st) {
    __shared__ Ctx<V> ctx;
    const Problem<V>& P = enter(ctx, Pp, st);
    const Hot& h = ctx.h;
    if (h.done || !h.tail) return;
    const int k = h.count(h.round & 1), words = core_words(k);
    const CoreArrays A = core_arrays(P, (h.round & 1) ^ 1, k);
    const int lane = lane_id(), wpb = blockDim.x >> 5;
    const int gw = blockIdx.x * wpb + (threadIdx.x >> 5), nw = gridDim.x * wpb;
    for (int i = gw; i < k; i += nw) {
        const int4 e = A.lent[i];
        if (e.y > kCoreWarpList) continue;
        const int* list = P.hadj + P.g.begin(e.x, e.w);
        for (int b0 = lane; b0 < e.y; b0 += 128) {
            int u[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) u[q] = b0 + 32 * q < e.y ? __ldg(list + b0 + 32 * q) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (u[q] >= 0) core_edge(P, i, u[q], words);
        }
    }
    for (int i = blockIdx.x; i < k; i += gridDim.x) {
        const int4 e = A.lent[i];
        if (e.y <= kCoreWarpList) continue;   // block-uniform
        const int* list = P.hadj + P.g.begin(e.x, e.w);
        for (int b = threadIdx.x; b < e.y; b += blockDim.x)
            core_edge(P, i, __ldg(list + b), words);
    }
}

// Word w (32 colors, from 32w + 1) of v's forbidden set in global memory.
template <class V>
__device__ __forceinline__ unsigned forbidden_word(const Problem<V>& P, int4 e, int w) {
    if (w < 2) return __ldcg(reinterpret_cast<const unsigned*>(P.bm0 + e.x) + w);
    if (e.z < 64 || w - 2 > (e.z >> 5)) return 0u;
    const long long b = P.g.begin(e.x, e.w);
    return __ldcg(P.bmx + P.g.bm(e.x, b) + (w - 2));
}

// Shared memory of one CTA of the core loop: R = ceil(k / C) rows, row x of
// CTA c being rank x * C + c.
struct CoreSmem {
    int R;
    uint4* rows;           // [R][words4] adjacency bits over the ranks
    uint4* cls;            // [kCoreClasses][words4] ranks by tentative color modulo kCoreClasses
    uint4* won;            // [2][words4] ranks that committed, by parity of the round
    unsigned short* tarr;  // [C][Rt] tentative color of every rank, by owner (0: committed)
    unsigned short* wcol;  // [C][Rt] color of the ranks that committed, by owner
    unsigned* forb;        // [R][kCoreWin + 1] forbidden colors from word fbase
    int* fbase;            // [R] first color word of forb
    int* frnd;             // [R] round of the commit
    unsigned short* open;  // [2][R] uncolored rows, by parity of the round
    unsigned short* fcol;  // [R] committed color (0: none)
};
constexpr int kCoreClasses = 64;

// log2 of the rows of one CTA in tarr: padded to a power of two, at least the
// 32 rows (64 bytes) of a warp
__host__ __device__ inline int core_rt_log(int k) {
    int l = 5;
    while ((kCoreCluster << l) < k) ++l;
    return l;
}

__host__ __device__ inline size_t core_smem_bytes(int k) {
    const size_t C = kCoreCluster;
    const size_t R = ((size_t)k + C - 1) / C, words4 = ((size_t)k + 127) / 128;
    return 16 * words4 * (R + kCoreClasses + 2) + 2 * 2 * (C << core_rt_log(k)) +
           4 * (R * (kCoreWin + 1) + 2 * R) + 2 * 3 * R;
}

__device__ __forceinline__ CoreSmem core_smem(uint4* base, int k) {
    constexpr int C = kCoreCluster;
    CoreSmem S;
    const int words4 = (k + 127) >> 7;
    S.R = (k + C - 1) / C;
    S.rows = base;
    S.cls = S.rows + S.R * words4;
    S.won = S.cls + kCoreClasses * words4;
    S.tarr = reinterpret_cast<unsigned short*>(S.won + 2 * words4);
    S.wcol = S.tarr + (C << core_rt_log(k));
    S.forb = reinterpret_cast<unsigned*>(S.wcol + (C << core_rt_log(k)));
    S.fbase = reinterpret_cast<int*>(S.forb + S.R * (kCoreWin + 1));
    S.frnd = S.fbase + S.R;
    S.open = reinterpret_cast<unsigned short*>(S.frnd + S.R);
    S.fcol = S.open + 2 * S.R;
    return S;
}

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// the same shared-memory location in CTA `cta` of the cluster
__device__ __forceinline__ unsigned peer_u32(const void* p, int cta) {
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(cta));
    return r;
}
__device__ __forceinline__ void st_peer(unsigned a, unsigned x) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ void st_peer(unsigned a, uint4 x) {
    asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x.x), "r"(x.y),
                 "r"(x.z), "r"(x.w)
                 : "memory");
}
__device__ __forceinline__ void st_peer(unsigned a, unsigned short x) {
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(x) : "memory");
}
__device__ __forceinline__ void or_peer(unsigned a, unsigned x) {
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(x)
                 : "memory");
}
__device__ __forceinline__ void add_peer(unsigned a, unsigned x) {
    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(x)
                 : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\t"
                 "barrier.cluster.wait.acquire;" ::: "memory");
}

// State of a CTA that its peers write.
struct CoreShared {
    unsigned long long bar;  // mbarrier of the meeting: one arrival per CTA
    unsigned n_won[2];       // commits of the round in all CTAs, by parity of the round
    int stop;                // CTA 0: the time limit has passed
    int gave_up;             // a CTA's wait ran out
    int n_open[2];           // uncolored rows of this CTA, by parity of the round
    unsigned moved;          // warps' worth of rows with a new tentative color
};

// The CTAs meet once before the first round, with a bounded wait: every CTA
// arrives at every CTA's mbarrier; thread 0 polls its own.  A wait that runs
// out sets gave_up in all CTAs.  The rounds then use the hardware cluster
// barrier: all CTAs are resident and each round's work is finite.
__device__ __forceinline__ void core_meet(CoreShared& X, int C, unsigned max_polls) {
    __syncthreads();
    if ((int)threadIdx.x < C) {
        asm volatile("fence.acq_rel.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                         peer_u32(&X.bar, threadIdx.x))
                     : "memory");
    }
    if (threadIdx.x == 0) {
        const unsigned a = smem_u32(&X.bar);
        unsigned polls = 0, done = 0;
        for (;;) {
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t}"
                : "=r"(done)
                : "r"(a)
                : "memory");
            if (done) break;
            if (++polls > max_polls || *(volatile int*)&X.gave_up) {
                for (int c = 0; c < C; ++c) st_peer(peer_u32(&X.gave_up, c), 1u);
                break;
            }
            if (polls > 256u) __nanosleep(200);
        }
    }
    __syncthreads();
}

// Forbid color c for row x (rank `rank`) of this CTA.
template <class V>
__device__ __forceinline__ void core_forbid(const Problem<V>& P, const CoreSmem& S, const int4* lent,
                                            int x, int rank, int c) {
    const int w = ((c - 1) >> 5) - S.fbase[x];
    const unsigned bit = 1u << ((c - 1) & 31);
    if (w < 0) return;   // below the row's current color: never considered again
    if (w < kCoreWin) {
        atomicOr(S.forb + x * (kCoreWin + 1) + w, bit);
        return;
    }
    const int4 e = lent[rank];
    if (c - 1 > e.z) return;   // the row's own first fit never reaches c
    const int gw = (c - 1) >> 5;
    if (gw < 2) {
        atomicOr(reinterpret_cast<unsigned*>(P.bm0 + e.x) + gw, bit);
    } else {
        const long long b = P.g.begin(e.x, e.w);
        atomicOr(P.bmx + P.g.bm(e.x, b) + (gw - 2), bit);
    }
}

// First free color of row x at or after t (the forbidden set only grows, so
// it never decreases); the window moves up when it is used up.
template <class V>
__device__ __forceinline__ int core_first_fit(const Problem<V>& P, const CoreSmem& S,
                                              const int4* lent, int x, int rank, int t) {
    int w = ((t - 1) >> 5) - S.fbase[x];
    unsigned* f = S.forb + x * (kCoreWin + 1);
    for (;;) {
        for (; w < kCoreWin; ++w)
            if (f[w] != kFullMask) return (S.fbase[x] + w) * 32 + __ffs(~f[w]);
        const int nb = S.fbase[x] + kCoreWin;
        for (int j = 0; j < kCoreWin; ++j) f[j] = forbidden_word(P, lent[rank], nb + j);
        S.fbase[x] = nb;
        w = 0;
    }
}

// What is left of a uint4 of row bits (ranks 128 i .. 128 i + 127) below rank.
__device__ __forceinline__ uint4 bits_below(uint4 b, int i, int rank) {
    auto keep = [&](unsigned x, int w) {
        const int d = rank - 32 * w;
        return d >= 32 ? x : d <= 0 ? 0u : x & ((1u << d) - 1u);
    };
    return make_uint4(keep(b.x, 4 * i), keep(b.y, 4 * i + 1), keep(b.z, 4 * i + 2),
                      keep(b.w, 4 * i + 3));
}
__device__ __forceinline__ uint4 and4(uint4 a, uint4 b) {
    return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w);
}
__device__ __forceinline__ bool any4(uint4 b) { return (b.x | b.y | b.z | b.w) != 0u; }
// takes the lowest set bit out of b (not zero): its index, 0..127
__device__ __forceinline__ int pop_bit(uint4& b) {
    const bool x = b.x != 0u, y = !x && b.y != 0u, z = !x && !y && b.z != 0u;
    const unsigned w = x ? b.x : y ? b.y : z ? b.z : b.w, rest = w & (w - 1u);
    const int at = (x ? 0 : y ? 32 : z ? 64 : 96) + __ffs(w) - 1;
    if (x) b.x = rest;
    else if (y) b.y = rest;
    else if (z) b.z = rest;
    else b.w = rest;
    return at;
}

// Phase 2: the rounds (one cluster of C CTAs x kCoreThreads).
//
// A round's time is latency: two cluster barriers and what happens between
// them.  (1) The ranks that committed last round, met with a row's bits,
// give the colors to forbid; then first fit; 32 rows' new colors go to each
// CTA as one 64-byte store.  (2) Every CTA sorts all tentative colors into
// kCoreClasses bit sets over the ranks (by color modulo kCoreClasses); a row
// loses if its bits below its own rank (the neighbors with priority) meet
// its class in a rank of the same color.  Both steps take eight lanes per row
// and 128 ranks per lane at a time, whatever the row's degree is, so a warp
// has four rows in flight and a round of 1000 vertices is one pass.
//
// Measured on R-MAT 20 (136 rounds from 3,940 vertices): 2.68 ms for the
// whole phase as a cooperative launch of 32 blocks over induced lists in L2
// with three grid barriers per round, 0.98 ms here, of which the loop takes
// 14,300 cycles per round (the two barriers 3,300 with their waiting).  512
// threads beat 1024 (19,300 cycles: issue slots and block barriers).
template <class V>
__global__ void __launch_bounds__(kCoreThreads, 1) d1_core_loop(const Problem<V>* __restrict__ Pp) {
    extern __shared__ uint4 core_sm[];
    __shared__ CoreShared X;
    const Problem<V>& P = *Pp;
    State* st = P.st;
    // uniform over the cluster: nothing has been shared yet
    if (*(volatile int*)&st->done || !*(volatile int*)&st->tail) return;
    const int cta = blockIdx.x;
    constexpr int C = kCoreCluster;
    const int k = st->core_k, words = core_words(k), words4 = (k + 127) >> 7;
    const int rtl = core_rt_log(k), Rt = 1 << rtl;
    const CoreArrays A = core_arrays(P, st->core_par, k);
    const CoreSmem S = core_smem(core_sm, k);
    const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const int grp = lane >> 3, sub = lane & 7;
    const unsigned gmask = 0xffu << (grp * 8);
    const int own = cta < k ? (k - cta + C - 1) / C : 0;   // rows of this CTA
    unsigned short* mine = S.tarr + cta * Rt;              // their tentative colors
    int r = st->round;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&X.bar)), "r"(C));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        X.stop = X.gave_up = 0;
        X.n_won[0] = X.n_won[1] = 0u;
        X.n_open[r & 1] = own;
        X.n_open[(r & 1) ^ 1] = 0;
        X.moved = 0u;
    }
    for (int x = warp; x < own; x += kCoreThreads / 32) {
        const unsigned* src = P.core_mat + (size_t)(x * C + cta) * words;
        unsigned* dst = reinterpret_cast<unsigned*>(S.rows + x * words4);
        for (int w = lane; w < words4 * 4; w += 32) dst[w] = w < words ? __ldcg(src + w) : 0u;
    }
    for (int i = tid; i < 2 * words4; i += kCoreThreads)
        S.won[i] = make_uint4(0u, 0u, 0u, 0u);   // both parities
    for (int p = tid; p < C * Rt; p += kCoreThreads) {
        const int j = (p & (Rt - 1)) * C + (p >> rtl);
        S.tarr[p] = j < k ? (unsigned short)A.tent[j] : 0;
    }
    if (tid < own) {
        const int rank = tid * C + cta;
        const int4 e = A.lent[rank];
        const int fb = (A.tent[rank] - 1) >> 5;
        S.fbase[tid] = fb;
        S.fcol[tid] = 0;
        S.open[(r & 1) * S.R + tid] = (unsigned short)tid;
#pragma unroll 4
        for (int j = 0; j < kCoreWin; ++j)
            S.forb[tid * (kCoreWin + 1) + j] = forbidden_word(P, e, fb + j);
    }
    // traced (CTA 0, warp 0): degrees and list lengths of the worklist
    unsigned long long sum_s = 0ull, sum_h = 0ull;
    const bool traced = P.trace_cap > 0 && cta == 0 && warp == 0;
    const unsigned long long t0_ns = st->t0;
    if (traced) {
        for (int j = lane; j < k; j += 32) {
            const int4 e = A.lent[j];
            sum_s += (unsigned long long)P.g.degree(e.x, e.z);   // per lane, see below
            sum_h += (unsigned long long)e.y;
        }
    }
    __syncthreads();
    cluster_sync();   // every CTA's shared memory is ready for its peers
    if (cta == P.core_wait.slow_block && tid == 0) be_late(P.core_wait.slow_ns);
    // what a round needs of the problem, kept in registers: after a cluster
    // barrier a global load is an L2 round trip
    const int max_rounds = P.max_rounds, trace_cap = P.trace_cap;
    const unsigned long long timeout_ns = P.timeout_ns;
    int cur = k, status = ST_OK;
    core_meet(X, C, P.core_wait.polls);
    cluster_sync();
    // a CTA may have given up after this one met everyone: all decide by the
    // flag, which every CTA holds by now
    const bool go = X.gave_up == 0;
    while (go) {
        const int now = r & 1, old = now ^ 1;
        // the end of the last round; the timer is slow to read, so its value is
        // used behind the cluster barrier only
        const unsigned long long at_ns = cta == 0 && tid == 0 ? global_ns() : 0ull;
        const int n_open = X.n_open[now];
        uint4* const won = S.won + old * words4;
        unsigned short* const open = S.open + now * S.R;
        // --- commits of the last round into the forbidden sets, first fit ---
        for (int i = tid; i < kCoreClasses * words4; i += kCoreThreads)
            S.cls[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int q0 = warp * 4; q0 < n_open; q0 += kCoreThreads / 8) {
            const int q = q0 + grp;
            const int x = q < n_open ? open[q] : -1, rank = x * C + cta;
            if (x >= 0) {
                for (int i0 = 0; i0 < words4; i0 += 32) {
                    uint4 b[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + 8 * u + sub;
                        b[u] = i < words4 ? and4(S.rows[x * words4 + i], won[i])
                                          : make_uint4(0u, 0u, 0u, 0u);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        while (any4(b[u])) {
                            const int j = 128 * (i0 + 8 * u + sub) + pop_bit(b[u]);
                            core_forbid(P, S, A.lent, x, rank, S.wcol[((j % C) << rtl) + j / C]);
                        }
                }
            }
            __syncwarp();
            if (x >= 0 && sub == 0) {
                const int t0 = mine[x];
                const int t = core_first_fit(P, S, A.lent, x, rank, t0);
                if (t != t0) {
                    mine[x] = (unsigned short)t;
                    atomicOr(&X.moved, 1u << (x >> 5));
                }
            }
        }
        __syncthreads();
        // --- committed ranks leave tarr; 32 rows with a new color go out ---
        if (warp < Rt >> 5) {   // (a row that is sent has left tarr here already)
            const unsigned rank = tid * C + cta;
            const unsigned* const w = reinterpret_cast<const unsigned*>(won);
            if (tid < own && (w[rank >> 5] >> (rank & 31) & 1u)) mine[tid] = 0;
            if (X.moved >> warp & 1u) {
                __syncwarp();
                const uint4* from = reinterpret_cast<const uint4*>(mine + warp * 32);
                for (int c = lane >> 2; c < C; c += 8)
                    if (c != cta) st_peer(peer_u32(from + (lane & 3), c), from[lane & 3]);
            }
        }
        for (int i = kCoreThreads - 1 - tid; i < words; i += kCoreThreads)
            for (unsigned m = reinterpret_cast<const unsigned*>(won)[i]; m; m &= m - 1u) {
                const int j = 32 * i + __ffs(m) - 1;
                if (j % C != cta) S.tarr[((j % C) << rtl) + j / C] = 0;
            }
        cluster_sync();
        // --- detect ---
        if (tid == 0) {
            X.moved = 0u;
            X.n_open[old] = 0;
            X.n_won[old] = 0u;
            if (cta == 0 && at_ns - t0_ns > timeout_ns)
                for (int c = 0; c < C; ++c) st_peer(peer_u32(&X.stop, c), 1u);
        }
        for (int i = tid; i < words4; i += kCoreThreads) won[i] = make_uint4(0u, 0u, 0u, 0u);
        unsigned* cls = reinterpret_cast<unsigned*>(S.cls);
        for (int p = tid * 8; p < C * Rt; p += kCoreThreads * 8) {
            // eight ranks of one owner
            const uint4 t8 = *reinterpret_cast<const uint4*>(S.tarr + p);
            if (!any4(t8)) continue;
            const unsigned h[4] = {t8.x, t8.y, t8.z, t8.w};
            const int j0 = (p & (Rt - 1)) * C + (p >> rtl);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const unsigned t = u & 1 ? h[u >> 1] >> 16 : h[u >> 1] & 0xffffu;
                const int j = j0 + u * C;
                if (t)
                    atomicOr(cls + (t % kCoreClasses) * (words4 * 4) + (j >> 5), 1u << (j & 31));
            }
        }
        __syncthreads();
        for (int q0 = warp * 4; q0 < n_open; q0 += kCoreThreads / 8) {
            const int q = q0 + grp;
            const int x = q < n_open ? open[q] : -1, rank = x * C + cta;
            const unsigned short t = x >= 0 ? mine[x] : 0;
            bool hit = false;
            if (x >= 0) {
                const uint4* cl = S.cls + (t % kCoreClasses) * words4;
                const int n4 = (rank >> 7) + 1;   // uint4s holding ranks below
                for (int i0 = 0; i0 < n4; i0 += 32) {
                    uint4 b[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + 8 * u + sub;
                        b[u] = i < n4 ? bits_below(and4(S.rows[x * words4 + i], cl[i]), i, rank)
                                      : make_uint4(0u, 0u, 0u, 0u);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        while (!hit && any4(b[u])) {   // another color of the class: next
                            const int j = 128 * (i0 + 8 * u + sub) + pop_bit(b[u]);
                            hit = S.tarr[((j % C) << rtl) + j / C] == t;
                        }
                }
            }
            const bool lose = (__ballot_sync(kFullMask, hit) & gmask) != 0u;
            const unsigned again = __ballot_sync(kFullMask, x >= 0 && lose && sub == 0);
            int at = 0;
            if (lane == 0 && again) at = atomicAdd(&X.n_open[old], __popc(again));
            at = __shfl_sync(kFullMask, at, 0);
            if (again >> lane & 1u)
                S.open[old * S.R + at + __popc(again & ((1u << lane) - 1u))] = (unsigned short)x;
            if (x >= 0 && !lose) {   // commits; the group's lanes tell the CTAs
                if (sub == 0) {
                    S.fcol[x] = t;
                    S.frnd[x] = r;
                }
                const unsigned* w = reinterpret_cast<const unsigned*>(S.won + now * words4) + (rank >> 5);
                for (int c = sub; c < C; c += 8) {
                    st_peer(peer_u32(S.wcol + cta * Rt + x, c), t);
                    or_peer(peer_u32(w, c), 1u << (rank & 31));
                    add_peer(peer_u32(&X.n_won[now], c), 1u);
                }
            }
        }
        cluster_sync();
        // --- round control, the same decision in every thread ---
        const int n_won = (int)X.n_won[now], nxt = cur - n_won;
        if (traced) {
            for (int j = lane; j < k; j += 32)
                if (reinterpret_cast<const unsigned*>(S.won + now * words4)[j >> 5] >> (j & 31) & 1u) {
                    const int4 e = A.lent[j];
                    sum_s -= (unsigned long long)P.g.degree(e.x, e.z);
                    sum_h -= (unsigned long long)e.y;
                }
            const unsigned long long ts = warp_sum(sum_s), th = warp_sum(sum_h);
            if (lane == 0 && r < trace_cap) {
                P.trace_w[r] = nxt;
                P.trace_s[r] = (long long)ts;
                P.trace_h[r] = (long long)th;
            }
        }
        if (X.stop) status = ST_TIMEOUT;   // passed before this round began
        else if (nxt == 0) break;
        else if (n_won == 0) status = ST_NO_PROGRESS;
        else if (r >= max_rounds) status = ST_MAX_ROUNDS;
        if (status != ST_OK) break;
        cur = nxt;
        ++r;
    }
    cluster_sync();   // no CTA leaves while a peer may still store here
    // --- write back: committed colors, tentative ones of an unfinished run ---
    int my_max = 0;
    if (tid < own) {
        const int rank = tid * C + cta, v = A.vid[rank], c = S.fcol[tid];
        P.col[v] = c ? c : -(int)mine[tid];
        my_max = c;
        if (P.g_rounds != nullptr) {
            const int g = P.g.graph(v);
            atomicMax(P.g_rounds + g, c ? S.frnd[tid] : r + 1);
            if (c) atomicMax(P.g_colors + g, c);
        }
    }
    my_max = warp_max(my_max);
    if (lane == 0 && my_max > 0) atomicMax(&st->max_color, my_max);
    if (cta == 0 && tid == 0) {
        st->round = r;
        st->status = X.gave_up ? ST_BARRIER : status;
        st->done = 1;
    }
}

// ---------------------------------------------------------------------------
// host side: scratch layout and one engine instance per (device, view type)
// ---------------------------------------------------------------------------
// Device scratch of one coloring (n vertices, nnz adjacency entries).
struct Scratch {
    int* deg;
    int* hlen;
    int* hadj;
    unsigned long long* bm0;
    unsigned* bmx;
    unsigned* live;
    int4* ws;    // 2n entries: both parities
    int4* wm;
    int4* wl;
    int2* items;
    int2* pushq;
    int* prio = nullptr;   // n ints, only for priorities that change each round
    unsigned* core_mat = nullptr;   // core_mat_bytes(n); none: no core phase
};

// The core phase's adjacency bits: a worklist of k vertices takes k x ceil(k / 32) words.
inline size_t core_mat_bytes(long long n) {
    const size_t k = (size_t)std::min<long long>(n, kCoreMax);
    return k * ((k + 31) / 32) * 4;
}

struct ScratchSizes {
    size_t deg, hlen, hadj, bm0, bmx, live, list, items, pushq;
    size_t total() const {   // with 256-byte alignment of every buffer
        auto a = [](size_t x) { return (x + 255) / 256 * 256; };
        return a(deg) + a(hlen) + a(hadj) + a(bm0) + a(bmx) + a(live) + 3 * a(list) + a(items) +
               a(pushq);
    }
};

inline ScratchSizes scratch_sizes(long long n, long long nnz) {
    ScratchSizes z;
    z.deg = z.hlen = (size_t)n * 4;
    z.hadj = (size_t)std::max<long long>(nnz, 1) * 4;
    z.bm0 = (size_t)n * 8;
    z.bmx = ((size_t)(nnz >> 5) + (size_t)n + 1) * 4;
    z.live = ((size_t)n / 32 + 2) * 4;
    z.list = (size_t)n * sizeof(int4) * 2;
    z.items = ((size_t)n + (size_t)(nnz / kBuildItem) + 1) * sizeof(int2);
    z.pushq = ((size_t)n + (size_t)(nnz / kPushItem) + 1) * sizeof(int2);
    return z;
}

// Carves a scratch of scratch_sizes(n, nnz).total() bytes at base.
inline Scratch carve_scratch(void* base, long long n, long long nnz) {
    const ScratchSizes z = scratch_sizes(n, nnz);
    char* p = static_cast<char*>(base);
    auto take = [&](size_t bytes) {
        char* q = p;
        p += (bytes + 255) / 256 * 256;
        return q;
    };
    Scratch sc;
    sc.deg = reinterpret_cast<int*>(take(z.deg));
    sc.hlen = reinterpret_cast<int*>(take(z.hlen));
    sc.hadj = reinterpret_cast<int*>(take(z.hadj));
    sc.bm0 = reinterpret_cast<unsigned long long*>(take(z.bm0));
    sc.bmx = reinterpret_cast<unsigned*>(take(z.bmx));
    sc.live = reinterpret_cast<unsigned*>(take(z.live));
    sc.ws = reinterpret_cast<int4*>(take(z.list));
    sc.wm = reinterpret_cast<int4*>(take(z.list));
    sc.wl = reinterpret_cast<int4*>(take(z.list));
    sc.items = reinterpret_cast<int2*>(take(z.items));
    sc.pushq = reinterpret_cast<int2*>(take(z.pushq));
    return sc;
}
template <class V>
struct Engine {
    std::mutex mu;
    DeviceInfo dev;
    DevBuf deg, hlen, hadj, bm0, bmx, live, ws, wm, wl, items, pushq, prio, state, problem, trace,
        core_mat;
    HostBuf h_problem, h_state, h_misc;
    int trace_cap = 0;
    int last_want_trace = 0, last_tcap = 1;
    // [0]: setup + rounds; [1]: rounds only (setup enqueued by the host:
    // while the adjacency is still being uploaded, or lists built elsewhere);
    // [2], [3]: the same for problems of at most mid_w vertices, which have no
    // launch-per-round rounds
    static constexpr int kGraphs = 4;
    cudaGraph_t graph[kGraphs] = {};
    cudaGraphExec_t exec[kGraphs] = {};
    int g_grid = 0, g_block = 0, g_det = 0, g_async = 0, g_dyn = 0;
    int occ_block = 0, occ_per_sm = 0, occ_det = 0;   // occupancy of the last block size
    int mid_grid = -1;    // blocks of the mid loop (-1: not asked yet)
    bool shares_gpu = false;   // others color on the same GPU: a small mid loop (set once)
    int core_grid = -1;   // CTAs of the core loop's cluster (-1: not asked yet)
    cudaStream_t up_stream = nullptr;             // adjacency upload
    cudaEvent_t up_fork = nullptr, up_done[kUploadChunks] = {};

    void destroy_graph() {
        for (int k = 0; k < kGraphs; ++k) {
            if (exec[k]) cudaGraphExecDestroy(exec[k]);
            if (graph[k]) cudaGraphDestroy(graph[k]);
            exec[k] = nullptr;
            graph[k] = nullptr;
        }
        g_grid = 0;
    }

    void destroy_upload() {
        if (up_stream) cudaStreamDestroy(up_stream);
        if (up_fork) cudaEventDestroy(up_fork);
        for (cudaEvent_t& e : up_done)
            if (e) cudaEventDestroy(e);
        up_stream = nullptr;
        up_fork = nullptr;
        for (cudaEvent_t& e : up_done) e = nullptr;
    }
    void release() {
        destroy_graph();
        destroy_upload();
        for (DevBuf* b : {&deg, &hlen, &hadj, &bm0, &bmx, &live, &ws, &wm, &wl, &items, &pushq,
                          &prio, &state, &problem, &trace, &core_mat})
            b->release();
        for (HostBuf* b : {&h_problem, &h_state, &h_misc}) b->release();
        trace_cap = 0;
    }

    struct Geometry {
        int grid, block;
        size_t smem;   // two warp appenders per warp
        int mid_grid;  // co-resident blocks of the mid loop (0: no cooperative launch)
        int core_grid; // CTAs of the core loop's cluster (0: no cluster fits, no core phase)
        int det_grid;  // detect: its own occupancy
    };

    pgc_status geometry(const Opts& o, Geometry* g) {
        g->block = o.block;
        g->smem = (size_t)(o.block / 32) * 2 * kIdxSlots * sizeof(int);
        if (g->smem > 48 * 1024) {   // 1024-thread blocks: 64 KB of append buffers
            std::vector<const void*> fs = {(const void*)d1_detect<V>};
            if constexpr (V::kSetup) {
                fs.push_back((const void*)d1_detect<V, true>);
            }
            for (const void* f : fs)
                PGC_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)g->smem));
        }
        int per_sm = o.grid_per_sm;
        g->det_grid = dev.num_sms * per_sm;
        if (per_sm == 0 && occ_block == o.block) {
            per_sm = occ_per_sm;
            g->det_grid = dev.num_sms * occ_det;
        } else if (per_sm == 0) {
            int a = 0, b = 0;
            PGC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, d1_detect<V>, o.block, g->smem));
            if constexpr (V::kSetup)
                PGC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, d1_build<V>, o.block, 0));
            else
                PGC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, d1_assign<V>, o.block, 0));
            occ_block = o.block;
            occ_per_sm = per_sm = std::max(1, b);
            occ_det = std::max(1, a);
            g->det_grid = dev.num_sms * occ_det;
        }
        g->grid = dev.num_sms * per_sm;
        if (core_grid < 0) {   // once per engine: does the device take the cluster?
            PGC_CUDA(cudaFuncSetAttribute(d1_core_loop<V>,
                                          cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            PGC_CUDA(cudaFuncSetAttribute(d1_core_loop<V>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)core_smem_bytes(kCoreMax)));
            cudaLaunchAttribute at;
            cudaLaunchConfig_t lc = core_config(nullptr, &at);
            int clusters = 0;
            const cudaError_t e = cudaOccupancyMaxActiveClusters(&clusters, d1_core_loop<V>, &lc);
            if (e != cudaSuccess) cudaGetLastError();
            core_grid = e == cudaSuccess && clusters > 0 ? kCoreCluster : 0;
        }
        g->core_grid = core_grid;
        if (mid_grid < 0) {
            int fits = 1, coop = 0;   // every variant runs with one block per SM
            for (int v = 0; v < 4; ++v) {
                const MidKernel m = mid_kernel(v & 1, v & 2);
                int per = 0;
                PGC_CUDA(cudaFuncSetAttribute(m.f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)m.smem()));
                PGC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, m.f, m.threads,
                                                                       m.smem()));
                fits = std::min(fits, per);
            }
            PGC_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev.device));
            mid_grid = coop && fits > 0 ? (shares_gpu ? std::min(kMidShared, dev.num_sms)
                                                      : dev.num_sms) : 0;
        }
        g->mid_grid = mid_grid;
        return PGC_OK;
    }

    struct MidKernel {
        void* f;
        int threads;
        size_t smem() const { return (size_t)(threads / 32) * 2 * kIdxSlots * sizeof(int); }
    };
    // (a server's requests share the GPU: few blocks, each with all its threads)
    MidKernel mid_kernel(bool dyn, bool small) const {
        if constexpr (V::kSetup) {
            if (dyn) return {(void*)d1_mid<V, true, 512>, 512};
        }
        if (small && !shares_gpu) return {(void*)d1_mid<V, false, 512>, 512};
        return {(void*)d1_mid<V, false, 1024>, 1024};
    }

    // launch configuration of the core loop: one cluster
    static cudaLaunchConfig_t core_config(cudaStream_t stream, cudaLaunchAttribute* at) {
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = kCoreCluster;
        at->val.clusterDim.y = at->val.clusterDim.z = 1;
        cudaLaunchConfig_t lc = {};
        lc.gridDim = dim3(kCoreCluster);
        lc.blockDim = dim3(kCoreThreads);
        lc.dynamicSmemBytes = core_smem_bytes(kCoreMax);
        lc.stream = stream;
        lc.attrs = at;
        lc.numAttrs = 1;
        return lc;
    }

    static cudaKernelNodeParams knode(void* func, const Geometry& g, size_t smem, void** args) {
        cudaKernelNodeParams k = {};
        k.func = func;
        k.gridDim = dim3(g.grid);
        k.blockDim = dim3(g.block);
        k.sharedMemBytes = (unsigned)smem;
        k.kernelParams = args;
        return k;
    }

    // Graph k for this geometry and mode, built when a call first needs it (the
    // four together take 0.05 ms of a first call's 0.48).
    pgc_status ensure_graph(int k, const Geometry& g, int async, int dyn) {
        if (g_grid != g.grid || g_block != g.block || g_det != g.det_grid || g_async != async ||
            g_dyn != dyn) {
            destroy_graph();
            g_dyn = dyn;
            g_grid = g.grid;
            g_det = g.det_grid;
            g_block = g.block;
            g_async = async;
        }
        if (exec[k]) return PGC_OK;
        if (graph[k]) cudaGraphDestroy(graph[k]);   // of a call that failed
        graph[k] = nullptr;
        return build_one_graph(g, k % 2 == 0, k >= 2, async, dyn, &graph[k], &exec[k]);
    }

    // Setup (optional, with round 1), round 1 when it is not part of the setup
    // (PGC_ASYNC, round-varying priorities; else its queued pushes) and the WHILE
    // node of the later rounds (both unless small), the mid loop and the core
    // phase.
    pgc_status build_one_graph(const Geometry& g, bool setup, bool small, int async, int dyn,
                               cudaGraph_t* graph_out, cudaGraphExec_t* exec_out) {
        Problem<V>* dP = problem.as<Problem<V>>();
        PGC_CUDA(cudaGraphCreate(graph_out, 0));
        cudaGraph_t graph = *graph_out;
        cudaGraphConditionalHandle handle = 0;
        if (!small)
            PGC_CUDA(cudaGraphConditionalHandleCreate(&handle, graph, 0u,
                                                      cudaGraphCondAssignDefault));
        int use_cond = 1;
        cudaGraphConditionalHandle hnd = handle;
        int lo = 0, hi = INT32_MAX;
        State* dS = state.as<State>();
        void* p_args[] = {&dP};
        int no_cond = 0;
        void* s_args[] = {&dP, &dS};
        void* n_args[] = {&dP, &dS, &hnd, &no_cond};
        void* b_args[] = {&dP, &lo, &hi};
        void* c_args[] = {&dP, &dS, &hnd, &use_cond};
        cudaMemsetParams ms = {};
        ms.dst = state.ptr;
        ms.value = 0;
        ms.elementSize = 4;
        ms.width = sizeof(State) / 4;
        ms.height = 1;
        cudaGraphNode_t n_ms, n_cls, n_build, n_tier = nullptr, n_asg1, n_det, n_push, n_loop;
        if (setup) PGC_CUDA(cudaGraphAddMemsetNode(&n_ms, graph, nullptr, 0, &ms));
        void* detect = (void*)d1_detect<V>;
        if constexpr (V::kSetup) {
            if (dyn) detect = (void*)d1_detect<V, true>;
        }
        cudaKernelNodeParams k_det = knode(detect, g, g.smem, c_args);
        k_det.gridDim = dim3(g.det_grid);
        cudaKernelNodeParams k_push = knode((void*)d1_push<V>, g, 0, n_args);
        cudaKernelNodeParams k_push1 = knode((void*)d1_push<V>, g, 0, c_args);
        cudaKernelNodeParams k_asg = knode((void*)d1_assign<V>, g, 0, c_args);
        if constexpr (V::kSetup) {
            if (setup) {
                cudaKernelNodeParams k_cls = knode((void*)d1_classify<V>, g, 0, p_args);
                cudaKernelNodeParams k_build = knode((void*)d1_build<V>, g, 0, b_args);
                cudaKernelNodeParams k_tier = knode((void*)d1_tier<V>, g, 0, s_args);
                PGC_CUDA(cudaGraphAddKernelNode(&n_cls, graph, &n_ms, 1, &k_cls));
                PGC_CUDA(cudaGraphAddKernelNode(&n_build, graph, &n_cls, 1, &k_build));
                PGC_CUDA(cudaGraphAddKernelNode(&n_tier, graph, &n_build, 1, &k_tier));
            }
        }
        cudaGraphNode_t last = nullptr;   // what the next node waits for (none: starts at once)
        if (setup) last = n_tier;
        auto after = [&](cudaGraphNode_t* node, cudaGraph_t gr, const cudaKernelNodeParams& k) {
            const cudaError_t e = cudaGraphAddKernelNode(node, gr, last ? &last : nullptr,
                                                         last ? 1 : 0, &k);
            last = *node;
            return e;
        };
        if (!small) {
            if (async) PGC_CUDA(after(&n_asg1, graph, k_asg));
            if (async || dyn) PGC_CUDA(after(&n_det, graph, k_det));
            PGC_CUDA(after(&n_push, graph, async || dyn ? k_push : k_push1));
            cudaGraphNodeParams cp = {};
            cp.type = cudaGraphNodeTypeConditional;
            cp.conditional.handle = handle;
            cp.conditional.type = cudaGraphCondTypeWhile;
            cp.conditional.size = 1;
            PGC_CUDA(cudaGraphAddNode(&n_loop, graph, &n_push, nullptr, 1, &cp));
            cudaGraph_t body = cp.conditional.phGraph_out[0];
            cudaGraphNode_t b_asg, b_det, b_push;
            PGC_CUDA(cudaGraphAddKernelNode(&b_asg, body, nullptr, 0, &k_asg));
            PGC_CUDA(cudaGraphAddKernelNode(&b_det, body, &b_asg, 1, &k_det));
            PGC_CUDA(cudaGraphAddKernelNode(&b_push, body, &b_det, 1, &k_push));
            last = n_loop;
        }
        if (g.mid_grid > 0 && !async) {
            const MidKernel m = mid_kernel(dyn, small);
            cudaKernelNodeParams k_mid = knode(m.f, g, m.smem(), s_args);
            k_mid.gridDim = dim3(g.mid_grid);
            k_mid.blockDim = dim3(m.threads);
            cudaGraphNode_t n_mid;
            PGC_CUDA(after(&n_mid, graph, k_mid));
            cudaLaunchAttributeValue coop = {};
            coop.cooperative = 1;
            PGC_CUDA(cudaGraphKernelNodeSetAttribute(n_mid, cudaLaunchAttributeCooperative, &coop));
        }
        // no-ops unless the mid loop stopped with st->tail set (as a conditional
        // node, the four launches cost no less when not taken, more when taken)
        if (g.core_grid > 0 && g.mid_grid > 0 && !async && !dyn) {
            cudaKernelNodeParams k_ckeys = knode((void*)d1_core_keys<V>, g, 0, s_args);
            k_ckeys.gridDim = dim3(dev.num_sms);
            cudaKernelNodeParams k_crank = knode((void*)d1_core_rank<V>, g, 0, s_args);
            k_crank.gridDim = dim3(dev.num_sms);
            cudaKernelNodeParams k_cbits = knode((void*)d1_core_bits<V>, g, 0, s_args);
            k_cbits.gridDim = dim3(dev.num_sms);
            cudaKernelNodeParams k_cloop =
                knode((void*)d1_core_loop<V>, g, core_smem_bytes(kCoreMax), p_args);
            k_cloop.gridDim = dim3(g.core_grid);
            k_cloop.blockDim = dim3(kCoreThreads);
            cudaGraphNode_t n_ckeys, n_crank, n_cbits, n_cloop;
            PGC_CUDA(after(&n_ckeys, graph, k_ckeys));
            PGC_CUDA(after(&n_crank, graph, k_crank));
            PGC_CUDA(after(&n_cbits, graph, k_cbits));
            PGC_CUDA(after(&n_cloop, graph, k_cloop));
            cudaLaunchAttributeValue dim = {};
            dim.clusterDim.x = (unsigned)g.core_grid;
            dim.clusterDim.y = dim.clusterDim.z = 1;
            PGC_CUDA(cudaGraphKernelNodeSetAttribute(n_cloop, cudaLaunchAttributeClusterDimension,
                                                     &dim));
        }
        PGC_CUDA(cudaGraphInstantiate(exec_out, graph, 0));
        return PGC_OK;
    }

    // Colors n vertices (nnz adjacency entries in total) described by view,
    // with scratch owned by this engine; waits for the result.
    pgc_status run(const V& view, int n, long long nnz, int* d_col, int* g_rounds,
                   int* g_colors, uint64_t seed, const Opts& o, cudaStream_t stream,
                   int* rounds, int* num_colors, const Upload* up = nullptr) {
        pgc_status s = run_scratch(view, n, nnz, d_col, g_rounds, g_colors, seed, o, stream,
                                   rounds, num_colors, up);
        // out of device memory: keep no half-grown scratch (the next call
        // allocates again)
        if (s == PGC_ERR_OOM) release();
        return s;
    }

    pgc_status run_scratch(const V& view, int n, long long nnz, int* d_col, int* g_rounds,
                           int* g_colors, uint64_t seed, const Opts& o, cudaStream_t stream,
                           int* rounds, int* num_colors, const Upload* up) {
        // scratch grows, never shrinks; pointers travel in the Problem struct,
        // so the captured graph stays valid across calls
        const ScratchSizes z = scratch_sizes(n, nnz);
        if (pgc_status s = deg.ensure(z.deg)) return s;
        if (pgc_status s = hlen.ensure(z.hlen)) return s;
        if (pgc_status s = hadj.ensure(z.hadj)) return s;
        if (pgc_status s = bm0.ensure(z.bm0)) return s;
        if (pgc_status s = bmx.ensure(z.bmx)) return s;
        if (pgc_status s = live.ensure(z.live)) return s;
        if (pgc_status s = ws.ensure(z.list)) return s;
        if (pgc_status s = wm.ensure(z.list)) return s;
        if (pgc_status s = wl.ensure(z.list)) return s;
        if (pgc_status s = items.ensure(z.items)) return s;
        if (pgc_status s = pushq.ensure(z.pushq)) return s;
        const bool varying = (o.flags & (PGC_PRIORITY_DYNAMIC | PGC_PRIORITY_SATURATION)) != 0;
        if (varying)
            if (pgc_status s = prio.ensure((size_t)std::max(n, 1) * 4)) return s;
        Scratch sc;
        sc.deg = deg.as<int>();
        sc.hlen = hlen.as<int>();
        sc.hadj = hadj.as<int>();
        sc.bm0 = bm0.as<unsigned long long>();
        sc.bmx = bmx.as<unsigned>();
        sc.live = live.as<unsigned>();
        sc.ws = ws.as<int4>();
        sc.wm = wm.as<int4>();
        sc.wl = wl.as<int4>();
        sc.items = items.as<int2>();
        sc.pushq = pushq.as<int2>();
        sc.prio = varying ? prio.as<int>() : nullptr;
        if (pgc_status s = core_mat.ensure(core_mat_bytes(n))) return s;
        sc.core_mat = core_mat.as<unsigned>();
        if (pgc_status s = launch(sc, view, n, nnz, d_col, g_rounds, g_colors, seed, o, stream,
                                  up))
            return s;
        PGC_CUDA(cudaStreamSynchronize(stream));
        return finish(o, rounds, num_colors);
    }

    // ListView: enqueues the kernel that builds the lists (and what
    // d1_classify, d1_build and d1_tier leave behind) for the problem.
    using Setup = std::function<pgc_status(const Problem<V>*)>;

    // Enqueues one coloring on `stream` with caller-provided scratch (the
    // device loop in graph mode; host-loop mode drives the rounds and
    // therefore blocks).  The round state and trace are copied to pinned
    // host memory on the same stream; call finish() once the stream is done.
    pgc_status launch(const Scratch& sc, const V& view, int n, long long nnz, int* d_col,
                      int* g_rounds, int* g_colors, uint64_t seed, const Opts& o,
                      cudaStream_t stream, const Upload* up = nullptr,
                      const Setup* setup = nullptr) {
        const uint32_t pflags = o.flags & (PGC_PRIORITY_DYNAMIC | PGC_PRIORITY_SATURATION);
        if (pflags == (PGC_PRIORITY_DYNAMIC | PGC_PRIORITY_SATURATION))
            return fail(PGC_ERR_INVALID_ARG, "PGC_PRIORITY_DYNAMIC and PGC_PRIORITY_SATURATION "
                                             "exclude each other");
        if (pflags && (o.flags & (PGC_NO_DEGREE_RULE | PGC_ASYNC)))
            return fail(PGC_ERR_INVALID_ARG, "a round-varying priority excludes "
                                             "PGC_NO_DEGREE_RULE and PGC_ASYNC");
        if (pflags && !sc.prio)
            return fail(PGC_ERR_INVALID_ARG, "round-varying priorities need their scratch");
        if (pgc_status s = state.ensure(sizeof(State))) return s;
        if (pgc_status s = problem.ensure(sizeof(Problem<V>))) return s;
        if (pgc_status s = h_problem.ensure(sizeof(Problem<V>))) return s;
        if (pgc_status s = h_state.ensure(sizeof(State))) return s;
        const int want_trace = o.profile && o.profile->trace_cap > 0 ? o.profile->trace_cap : 0;
        const int tcap = std::max(want_trace, 1);
        if (trace_cap < tcap) {
            if (pgc_status s = trace.ensure((size_t)tcap * 3 * sizeof(long long))) return s;
            if (pgc_status s = h_misc.ensure((size_t)tcap * 3 * sizeof(long long))) return s;
            trace_cap = tcap;
        }
        last_want_trace = want_trace;
        last_tcap = tcap;

        Geometry g;
        if (pgc_status s = geometry(o, &g)) return s;

        Problem<V>* hp = h_problem.as<Problem<V>>();
        std::memset(hp, 0, sizeof(Problem<V>));
        hp->g = view;
        hp->col = d_col;
        hp->deg = sc.deg;
        hp->hlen = sc.hlen;
        hp->hadj = sc.hadj;
        hp->bm0 = sc.bm0;
        hp->bmx = sc.bmx;
        hp->live = sc.live;
        for (int p = 0; p < 2; ++p) {
            hp->ws[p] = sc.ws + (size_t)p * n;
            hp->wm[p] = sc.wm + (size_t)p * n;
            hp->wl[p] = sc.wl + (size_t)p * n;
        }
        hp->items = sc.items;
        hp->push_q = sc.pushq;
        hp->core_mat = sc.core_mat;
        hp->g_rounds = g_rounds;
        hp->g_colors = g_colors;
        hp->trace_w = trace.as<long long>();
        hp->trace_s = hp->trace_w + tcap;
        hp->trace_h = hp->trace_s + tcap;
        hp->trace_cap = want_trace;
        hp->st = state.as<State>();
        hp->seed = seed;
        hp->timeout_ns = (unsigned long long)o.timeout_ms * 1000000ull;
        hp->nnz = nnz;
        hp->n = n;
        hp->use_deg = (o.flags & PGC_NO_DEGREE_RULE) ? 0 : 1;
        hp->async_mode = (o.flags & PGC_ASYNC) ? 1 : 0;
        hp->prio_mode = (pflags & PGC_PRIORITY_DYNAMIC) ? 1 : (pflags ? 2 : 0);
        hp->prio = sc.prio;
        hp->max_rounds = o.max_rounds > 0 ? o.max_rounds : (n < INT32_MAX ? n + 1 : n);
        hp->det_s = o.mid_degree;
        // lists that hold whole rows: hubs' lists are long, and a block reads 1024
        // entries per step where a warp reads 128
        hp->det_m = pflags ? std::max(o.mid_degree, std::min(o.hub_degree, varying_hub((int)n)))
                           : o.hub_degree;
        hp->mid_w = hp->async_mode || g.mid_grid == 0 ? 0 : shares_gpu ? kMidSharedMax : kMidMax;
        hp->tail_w = hp->mid_w == 0 || pflags || g.core_grid == 0 || !sc.core_mat
                         ? 0 : std::min(o.tail_vertices, kCoreMax);
        const int small = n <= hp->mid_w ? 2 : 0;
        const TestHooks th = test_hooks();
        hp->mid_wait = {th.mid.polls, th.mid.slow_block, th.mid.slow_us * 1000u, th.mid.at};
        hp->core_wait = {th.core.polls, th.core.slow_block, th.core.slow_us * 1000u, th.core.at};
        PGC_CUDA(cudaMemcpyAsync(problem.ptr, hp, sizeof(Problem<V>), cudaMemcpyHostToDevice,
                                 stream));
        Problem<V>* dP = problem.as<Problem<V>>();

        State* hs = h_state.as<State>();
        if (!(o.flags & PGC_HOST_LOOP)) {
            const int which = !V::kSetup ? small + 1 : up ? 1 : small;
            if (pgc_status s = ensure_graph(which, g, hp->async_mode, hp->prio_mode != 0))
                return s;
            if constexpr (!V::kSetup) {
                PGC_CUDA(cudaMemsetAsync(state.ptr, 0, sizeof(State), stream));
                if (pgc_status s = (*setup)(dP)) return s;
                PGC_CUDA(cudaGraphLaunch(exec[which], stream));
            } else if (!up) {
                PGC_CUDA(cudaGraphLaunch(exec[which], stream));
            } else {
                // setup by hand: classify needs only the row offsets; the
                // build of row range k waits for that range's copy
                if (!up_stream) {
                    PGC_CUDA(cudaStreamCreateWithFlags(&up_stream, cudaStreamNonBlocking));
                    PGC_CUDA(cudaEventCreateWithFlags(&up_fork, cudaEventDisableTiming));
                    for (cudaEvent_t& e : up_done)
                        PGC_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
                }
                int cut[kUploadChunks + 1];
                cut[0] = 0;
                cut[kUploadChunks] = n;
                for (int k = 1; k < kUploadChunks; ++k) {   // first row past k/K of the entries
                    const long long want = nnz * k / kUploadChunks;
                    cut[k] = (int)(std::lower_bound(up->h_rp, up->h_rp + n, (int)want) - up->h_rp);
                    cut[k] = std::max(cut[k], cut[k - 1]);
                }
                PGC_CUDA(cudaEventRecord(up_fork, stream));
                PGC_CUDA(cudaStreamWaitEvent(up_stream, up_fork, 0));
                for (int k = 0; k < kUploadChunks; ++k) {
                    const size_t e0 = (size_t)up->h_rp[cut[k]], e1 = (size_t)up->h_rp[cut[k + 1]];
                    if (e1 > e0)
                        PGC_CUDA(cudaMemcpyAsync(up->d_ci + e0, up->h_ci + e0, (e1 - e0) * 4,
                                                 cudaMemcpyHostToDevice, up_stream));
                    PGC_CUDA(cudaEventRecord(up_done[k], up_stream));
                }
                PGC_CUDA(cudaMemsetAsync(state.ptr, 0, sizeof(State), stream));
                d1_classify<V><<<g.grid, g.block, 0, stream>>>(dP);
                for (int k = 0; k < kUploadChunks; ++k) {
                    PGC_CUDA(cudaStreamWaitEvent(stream, up_done[k], 0));
                    d1_build<V><<<g.grid, g.block, 0, stream>>>(dP, cut[k], cut[k + 1]);
                }
                d1_tier<V><<<g.grid, g.block, 0, stream>>>(dP, state.as<State>());
                PGC_CUDA(cudaGetLastError());
                PGC_CUDA(cudaGraphLaunch(exec[which], stream));
            }
        } else {
            KernelTimer kt;
            kt.prof = o.profile;
            kt.stream = stream;
            const cudaGraphConditionalHandle none = 0;
            State* dS = state.as<State>();
            PGC_CUDA(cudaMemsetAsync(state.ptr, 0, sizeof(State), stream));
#define PGC_TIMED(slot, name, launch_)                        \
    do {                                                      \
        if (pgc_status s_ = kt.begin(slot, name)) return s_;  \
        launch_;                                              \
        PGC_CUDA(cudaGetLastError());                         \
        if (pgc_status s_ = kt.end()) return s_;              \
    } while (0)
            if constexpr (V::kSetup) {
                PGC_TIMED(0, "d1_classify",
                          (d1_classify<V><<<g.grid, g.block, 0, stream>>>(dP)));
                PGC_TIMED(1, "d1_build",
                          (d1_build<V><<<g.grid, g.block, 0, stream>>>(dP, 0, INT32_MAX)));
                PGC_TIMED(2, "d1_tier",
                          (d1_tier<V><<<g.grid, g.block, 0, stream>>>(dP, state.as<State>())));
            } else {   // slot 0 is the caller's
                if (pgc_status s_ = kt.begin(1, "net_lists")) return s_;
                if (pgc_status s_ = (*setup)(dP)) return s_;
                if (pgc_status s_ = kt.end()) return s_;
            }
            for (int round = 1; !small; ++round) {
                const bool whole = round > 1 || hp->async_mode || hp->prio_mode;
                if (round > 1 || hp->async_mode)
                    PGC_TIMED(3, "d1_assign",
                              (d1_assign<V><<<g.grid, g.block, 0, stream>>>(dP, dS, none, 0)));
                if (whole) {   // otherwise round 1 was part of the setup
                    if (pgc_status s_ = kt.begin(4, "d1_detect")) return s_;
                    bool dyn_detect = false;
                    if constexpr (V::kSetup) {
                        if (hp->prio_mode) {
                            dyn_detect = true;
                            d1_detect<V, true>
                                <<<g.det_grid, g.block, g.smem, stream>>>(dP, dS, none, 0);
                        }
                    }
                    if (!dyn_detect)
                        d1_detect<V><<<g.det_grid, g.block, g.smem, stream>>>(dP, dS, none, 0);
                    PGC_CUDA(cudaGetLastError());
                    if (pgc_status s_ = kt.end()) return s_;
                }
                PGC_TIMED(5, "d1_push",
                          (d1_push<V><<<g.grid, g.block, 0, stream>>>(dP, dS, none, 0)));
                PGC_CUDA(cudaMemcpyAsync(hs, state.ptr, sizeof(State), cudaMemcpyDeviceToHost,
                                         stream));
                PGC_CUDA(cudaStreamSynchronize(stream));
                if (hs->done || hs->mid) break;
                if (round > hp->max_rounds + 1)
                    return fail(PGC_ERR_CUDA, "device round control did not finish the loop");
            }
            if (hp->mid_w > 0) {   // no-ops once the coloring is done
                void* args[] = {&dP, &dS};
                const MidKernel m = mid_kernel(hp->prio_mode != 0, small != 0);
                if (pgc_status s_ = kt.begin(7, "d1_mid")) return s_;
                PGC_CUDA(cudaLaunchCooperativeKernel(m.f, dim3(g.mid_grid), dim3(m.threads), args,
                                                     m.smem(), stream));
                if (pgc_status s_ = kt.end()) return s_;
            }
            if (hp->tail_w > 0) {
                if (pgc_status s_ = kt.begin(6, "d1_core")) return s_;
                d1_core_keys<V><<<dev.num_sms, g.block, 0, stream>>>(dP, dS);
                d1_core_rank<V><<<dev.num_sms, g.block, 0, stream>>>(dP, dS);
                d1_core_bits<V><<<dev.num_sms, g.block, 0, stream>>>(dP, dS);
                PGC_CUDA(cudaGetLastError());
                cudaLaunchAttribute at;
                cudaLaunchConfig_t lc = core_config(stream, &at);
                PGC_CUDA(cudaLaunchKernelEx(&lc, d1_core_loop<V>, (const Problem<V>*)dP));
                if (pgc_status s_ = kt.end()) return s_;
            }
#undef PGC_TIMED
            kt.destroy();
        }
        PGC_CUDA(cudaMemcpyAsync(hs, state.ptr, sizeof(State), cudaMemcpyDeviceToHost, stream));
        if (want_trace) {
            PGC_CUDA(cudaMemcpyAsync(h_misc.ptr, trace.ptr, (size_t)tcap * 3 * sizeof(long long),
                                     cudaMemcpyDeviceToHost, stream));
        }
        return PGC_OK;
    }

    // Reads the result of the last launch() (its stream must be complete).
    pgc_status finish(const Opts& o, int* rounds, int* num_colors) {
        State* hs = h_state.as<State>();
        const int want_trace = last_want_trace, tcap = last_tcap;
        if (want_trace && o.profile) {
            const long long* tw = h_misc.as<long long>();
            const long long* ts = tw + tcap;
            const long long* th = ts + tcap;
            const int nr = std::min(hs->round, want_trace);
            for (int i = 0; i < want_trace; ++i) {
                if (o.profile->trace_w) o.profile->trace_w[i] = i < nr ? tw[i] : 0;
                if (o.profile->trace_s) o.profile->trace_s[i] = i < nr ? ts[i] : 0;
                if (o.profile->trace_h) o.profile->trace_h[i] = i < nr ? th[i] : 0;
            }
        }
        *rounds = hs->round;
        *num_colors = hs->max_color;
        switch (hs->status) {
            case ST_OK: return PGC_OK;
            case ST_NO_PROGRESS:
                return fail(PGC_ERR_NO_CONVERGE, "a round committed no vertex (input not symmetric?)");
            case ST_MAX_ROUNDS: return fail(PGC_ERR_NO_CONVERGE, "max_rounds reached");
            case ST_TIMEOUT: return fail(PGC_ERR_TIMEOUT, "device round loop exceeded timeout_ms");
            case ST_BARRIER:
                return fail(PGC_ERR_TIMEOUT, "a grid barrier of the core loop timed out");
            case ST_MID_BARRIER:
                return fail(PGC_ERR_TIMEOUT, "a grid barrier of the mid loop timed out");
            default: return fail(PGC_ERR_CUDA, "unexpected device status");
        }
    }
};

// One engine per device and view type, created on first use.
template <class V>
Engine<V>* engine_for(int device) {
    static std::mutex mu;
    static std::unordered_map<int, std::unique_ptr<Engine<V>>> m;
    std::lock_guard<std::mutex> lk(mu);
    auto it = m.find(device);
    if (it != m.end()) return it->second.get();
    if (m.empty()) {
        release_hooks().push_back([] {
            std::lock_guard<std::mutex> lk2(mu);
            int cur = 0;
            cudaGetDevice(&cur);
            auto f = m.find(cur);
            if (f != m.end()) {
                std::lock_guard<std::mutex> lk3(f->second->mu);
                f->second->release();
            }
        });
    }
    auto e = std::make_unique<Engine<V>>();
    Engine<V>* p = e.get();
    m.emplace(device, std::move(e));
    return p;
}

}  // namespace d1
}  // namespace pgc
