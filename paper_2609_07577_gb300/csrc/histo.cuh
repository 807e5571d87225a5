// Per-vertex integer histograms keyed by a vertex id (coarsening: score and
// shared inbound count per neighbour) or a partition id (refinement:
// connection weight and inbound overlap per adjacent partition), followed by
// an argmax over the keys. Sums are integer atomics, so results do not
// depend on the order of updates.
//
// Vertices are first binned by their work (total length of the segments
// their incidences contribute), which bounds their number of distinct keys:
//   warp tier   work <= 3/4 of a 512-slot table: one warp, shared memory;
//               cannot overflow.
//   block tier  work <= 2^16: one 256-thread block, 2048-slot shared table;
//               a vertex with more than 1536 distinct keys is handed on.
//   big tier    work <= 2^22 or hand-overs: one 512-thread block per SM with
//               a 16384-slot shared table; overflow is handed on.
//   split tier  the rest: the incidences are cut into items of about 16384
//               elements processed by warps all over the GPU, all adding into
//               one global-memory table per vertex sized to twice its bound
//               of distinct keys (so it cannot overflow); one block per
//               vertex then reduces the table.
// Key spaces of up to 24,576 keys take arrays instead of the tables of the
// block tier (up to 4,096 keys) and of the big and split tiers (k_ht_dense).
// In the warp tier a warp flattens 32 incidences at a time (warp_visit); in
// the others a group of 4 to 32 lanes (the vertex's mean segment) takes an
// incidence (group_visit).
//
// A Policy supplies:
//   typedef S (score type), struct Acc (per-thread sums, with add(Acc) and
//   __device__ Acc reduce over a warp)
//   int32_t V (vertices), key space bound `keys`
//   static constexpr bool kMasks                    segments carry HRec's run masks
//   static constexpr bool kOptimistic               try the warp tier even when the
//                                                   bound exceeds its table (few keys expected)
//   __device__ bool skip(n)                         n needs no histogram (result
//                                                   written by write(n, 0, -1, 0, Acc()))
//   __device__ int64_t seg_len(int64_t i)           segment length of incidence i
//   __device__ int64_t vb(n), ve(n)                 incidence range of vertex n
//   __device__ uint32_t inc(int64_t i)              incidence i's word (hyperedge, source bit)
//   __device__ Seg<S> seg(uint32_t inc, Acc&)       its segment
//   __device__ void fetch(uint32_t inc)             brings what seg reads into the L1 cache
//   struct Own, Own own(n)                          what load reads of the visiting vertex
//   struct Item, Item load(n, Own, const Seg<S>&, off)  one element's reads; none() an empty Item
//   __device__ bool put(n, const Item&, table, Acc&)  its table update
//   (apart, so that several elements' loads are in flight per thread)
//   __device__ void consider(n, key, int64 sc, uint32 ov, const Acc& total,
//                            int64_t& best, int32_t& bkey, uint32_t& bov)
//   __device__ void write(n, best, bkey, bov, const Acc& total)
#pragma once
#include "common.cuh"
#include "histo_tiers.cuh"
#include "table_slot.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <type_traits>

namespace snn {

// (s1, m1) beats (s2, m2): larger value, ties to the lower id; id < 0 = none
__device__ __forceinline__ bool better(int64_t s1, int32_t m1, int64_t s2, int32_t m2)
{
    if (m1 < 0) return false;
    if (m2 < 0) return true;
    return s1 > s2 || (s1 == s2 && m1 < m2);
}

// Open-addressing slots: key (-1 empty), summed weight, summed overlap.
template <typename S>
struct Table {
    static constexpr bool kFills = true;   // an insert can fail
    int32_t* key;
    S* sc;
    uint32_t* ov;
    uint32_t mask;     // capacity - 1
    uint32_t probes;   // probe limit of add()

    // returns false if m finds no slot within the probe limit (tables that
    // must never fail use the full capacity as the limit)
    __device__ __forceinline__ bool add(int32_t m, S w, uint32_t o) const
    {
        return try_add(m, w, o, probes);
    }

    // returns false if m has no slot within the first max_probes probed
    __device__ __forceinline__ bool try_add(int32_t m, S w, uint32_t o, uint32_t max_probes) const
    {
        uint32_t slot = table_slot(m, mask);
        for (uint32_t probe = 0; probe < max_probes; probe++) {
            int32_t k = *(volatile int32_t*)&key[slot];
            if (k == -1) {
                int32_t prev = atomicCAS(&key[slot], -1, m);
                k = prev == -1 ? m : prev;
            }
            if (k == m) {
                atomicAdd(&sc[slot], w);
                if (o) atomicAdd(&ov[slot], o);
                return true;
            }
            slot = (slot + 1) & mask;
        }
        return false;
    }
};

__device__ __forceinline__ void prefetch_l1(const void* p)
{
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

template <typename S>
__host__ __device__ constexpr size_t slot_bytes()
{
    return 2 * sizeof(int32_t) + sizeof(S);
}

template <typename S>
__device__ __forceinline__ Table<S> carve_table(unsigned char* base, int64_t cap)
{
    Table<S> t;
    t.key = (int32_t*)base;
    t.sc = (S*)(base + (size_t)cap * sizeof(int32_t));
    t.ov = (uint32_t*)(base + (size_t)cap * (sizeof(int32_t) + sizeof(S)));
    t.mask = (uint32_t)(cap - 1);
    t.probes = (uint32_t)cap;
    return t;
}

// What the histograms read of a hyperedge, in one 32-byte sector: a vertex's
// incidences name hyperedges all over the level, so offsets, weight,
// multiplicity and flags in arrays of their own cost a sector each (the
// gains of the 262,144-neuron conv network's first round read 20 million
// segments of about nine partitions).
struct alignas(32) HRec {
    int64_t b;       // first element
    int64_t w;
    uint32_t k;
    uint32_t len;    // elements; bit 31: selfdst
    uint32_t dm;     // pin counts: bit r set when run r (r < 32) has destinations
    uint32_t sm;     // pin counts: bit r set when run r (r < 32) is a single pin
    __device__ int32_t n() const { return (int32_t)(len & 0x7fffffffu); }
    __device__ int sd() const { return (int)(len >> 31); }
};

// One incidence's segment: elements [b, b+len) of a per-hyperedge array,
// with the hyperedge's weight w, multiplicity k, whether the visiting vertex
// is one of its destinations (nd) and its selfdst flag (sd).
template <typename S>
struct Seg {
    int64_t b;
    int32_t len;
    S w;
    uint32_t k;
    int nd, sd;
    uint32_t dm, sm;   // as HRec (refinement)
};

// the segment of an incidence word (hyperedge id and source bit)
template <typename S>
__device__ __forceinline__ Seg<S> rec_seg(const HRec& r, uint32_t inc)
{
    Seg<S> g;
    g.sd = r.sd();
    g.nd = !(inc & SRC_BIT) || g.sd;
    g.b = r.b;
    g.len = r.n();
    g.w = (S)r.w;
    g.k = r.k;
    g.dm = r.dm;
    g.sm = r.sm;
    return g;
}

// Slots whose weight and overlap share one word, value = weight << sb |
// overlap, for vertices whose sums over all incidences bound both within 32
// bits: one shared-memory atomic an element instead of two. LIST: the slots
// in use are listed, so the result of a large table costs a read per key
// instead of one per slot.
// CLAIM: a slot is tried by compare-and-swap at once instead of being read
// first, for vertices of few long incidences, whose keys are mostly new
// (power-law level 0: 24.3 -> 23.0 ms; the conv network's, whose pins repeat,
// 31.4 -> 32.7 ms that way).
template <bool LIST, bool CLAIM = false>
struct PackedTable {
    static constexpr bool kFills = true;
    int32_t* key;
    uint32_t* val;
    uint16_t* used;    // LIST: slots in use, *nused of them
    int32_t* nused;
    uint32_t mask;
    uint32_t probes;
    int sb;
    __device__ __forceinline__ bool add(int32_t m, uint32_t w, uint32_t o) const
    {
        uint32_t slot = table_slot(m, mask);
        for (uint32_t probe = 0; probe < probes; probe++) {
            int32_t k = CLAIM ? -1 : *(volatile int32_t*)&key[slot];
            if (k == -1) {
                int32_t prev = atomicCAS(&key[slot], -1, m);
                k = prev == -1 ? m : prev;
                if (LIST && prev == -1) {
                    const unsigned am = __activemask();
                    const int leader = __ffs(am) - 1;
                    int32_t at = 0;
                    if ((int)(threadIdx.x & 31) == leader) at = atomicAdd(nused, __popc(am));
                    at = __shfl_sync(am, at, leader);
                    used[at + __popc(am & lanemask_lt())] = (uint16_t)slot;
                }
            }
            if (k == m) {
                atomicAdd(&val[slot], (w << sb) + o);
                return true;
            }
            slot = (slot + 1) & mask;
        }
        return false;
    }
};

// One warp visits incidences [vb, ve) of vertex n, 32 at a time with their
// segments flattened into one range, so that all 32 lanes load consecutive
// elements even when segments are short or uneven; two steps' loads are in
// flight. Returns false if an insert failed.
template <typename S, class Pol, class Tb>
__device__ bool warp_visit(const Pol& pol, int32_t n, int64_t vb, int64_t ve, const Tb& t,
                           typename Pol::Acc& acc)
{
    int lane = threadIdx.x & 31;
    bool ok = true;
    const typename Pol::Own own = pol.own(n);
    for (int64_t ib = vb; ib < ve; ib += 32) {
        int64_t i = ib + lane;
        Seg<S> sg{};
        if (i < ve) sg = pol.seg(pol.inc(i), acc);
        int32_t pre = sg.len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t t2 = __shfl_up_sync(FULL, pre, o);
            if (lane >= o) pre += t2;
        }
        int32_t total = __shfl_sync(FULL, pre, 31);
        pre -= sg.len;
        const int flags = sg.nd << 1 | sg.sd;
        // nonempty segments in order (src: lane of the r-th), so that within a
        // window of 32 elements the segment of one is the number of segments
        // starting at or before it, less one
        const unsigned some = __ballot_sync(FULL, sg.len > 0);
        int src = lane;
        if (some != FULL) {
            src = 0;
            unsigned rest = some;
            for (int r = 0; rest; r++) {
                if (lane == r) src = __ffs(rest) - 1;
                rest &= rest - 1;
            }
        }
        int before = 0;   // nonempty segments that start before the window
        constexpr int U = 2;
        for (int32_t vbase = 0; vbase < total; vbase += 32 * U) {
            typename Pol::Item it[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int32_t w0 = vbase + 32 * u, v = w0 + lane;
                const int32_t d = pre - w0;
                const unsigned starts =
                    __reduce_or_sync(FULL, sg.len > 0 && d >= 0 && d < 32 ? 1u << d : 0u);
                int r = before + __popc(starts & (lanemask_lt() | (1u << lane))) - 1;
                before += __popc(starts);
                const int lo = __shfl_sync(FULL, src, r & 31);
                Seg<S> g;
                g.b = __shfl_sync(FULL, sg.b, lo);
                g.len = 0;
                g.w = __shfl_sync(FULL, sg.w, lo);
                g.k = __shfl_sync(FULL, sg.k, lo);
                int f = __shfl_sync(FULL, flags, lo);
                g.nd = f >> 1;
                g.sd = f & 1;
                if (Pol::kMasks) {
                    g.dm = __shfl_sync(FULL, sg.dm, lo);
                    g.sm = __shfl_sync(FULL, sg.sm, lo);
                }
                int32_t pt = __shfl_sync(FULL, pre, lo);
                it[u] = v < total ? pol.load(n, own, g, v - pt) : Pol::none();
            }
#pragma unroll
            for (int u = 0; u < U; u++) ok = pol.put(n, it[u], t, acc) && ok;
        }
    }
    return __all_sync(FULL, ok);
}

// lanes (log2) that take one incidence of a vertex with this many incidences
// and elements: its mean segment, a power of two in [4, 32]
__device__ __forceinline__ int group_log(int64_t deg, int64_t work)
{
    int64_t mean = deg > 0 ? (work + deg - 1) / deg : 32;
    return mean <= 4 ? 2 : (mean <= 8 ? 3 : (mean <= 16 ? 4 : 5));
}

// T threads (whole warps; tid 0..T-1) visit incidences [vb, ve) of vertex n,
// a group of 2^glog lanes per incidence and U incidences in flight per group.
// The group's lanes hold the same segment in registers, so an element costs
// its load and its table update; the flattened form before (tiles of
// incidences, a shared-memory prefix and a search per element) spent most of
// its instructions on finding the segment. Segments longer than eight rounds
// of their group are finished by its whole warp; those longer than T go to
// slong (if any) for the whole block, which would otherwise wait for one of
// its warps (a vertex of the 1,048,576-neuron power-law network meets 47
// pins a hyperedge on average, but up to 16,384). AHEAD: the next pass's
// records are brought into the L1 cache and the words of the one after it are
// read while a pass runs, for blocks that have an SM to themselves, where a
// pass is a chain of three gathers (word, record, element). Returns false in
// lanes whose insert failed.
constexpr int HT_NLONG = 256;

template <typename S, int T, int U, bool AHEAD, class Pol, class Tb>
__device__ __forceinline__ bool group_visit(const Pol& pol, int32_t n, int64_t vb, int64_t ve,
                                            int glog, int tid, const Tb& t,
                                            typename Pol::Acc& acc, int64_t* slong = nullptr,
                                            int32_t* nlong = nullptr)
{
    const int lane = tid & 31, G = 1 << glog, gl = lane & (G - 1);
    const int grp = tid >> glog, ngrp = T >> glog;
    const bool longs = pol.L.maxlen > 8 * G || pol.L.maxlen > T;   // else no segment needs others' lanes
    bool ok = true;
    const typename Pol::Own own = pol.own(n);
    typename Pol::Acc other;   // a segment's own terms count once, in its first lane
    uint32_t wd[AHEAD ? U : 1], wd2[AHEAD ? U : 1];   // words of this pass and the next
    if (AHEAD) {
#pragma unroll
        for (int u = 0; u < U; u++) {
            int64_t i = vb + (int64_t)u * ngrp + grp;
            wd[u] = i < ve ? pol.inc(i) : 0u;
            wd2[u] = i + (int64_t)U * ngrp < ve ? pol.inc(i + (int64_t)U * ngrp) : 0u;
        }
    }
    for (int64_t base = vb; base < ve; base += (int64_t)U * ngrp) {
        Seg<S> g[U];
        typename Pol::Item it[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            int64_t i = base + (int64_t)u * ngrp + grp;
            g[u] = Seg<S>{};
            if (i < ve) g[u] = pol.seg(AHEAD ? wd[u] : pol.inc(i), gl == 0 ? acc : other);
        }
        if (AHEAD) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                int64_t i = base + (int64_t)(U + u) * ngrp + grp;
                wd[u] = wd2[u];
                if (i < ve) pol.fetch(wd[u]);
                i += (int64_t)U * ngrp;
                wd2[u] = i < ve ? pol.inc(i) : 0u;
            }
        }
        if (slong && longs) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                bool lg = g[u].len > T;
                int32_t at = HT_NLONG;
                if (lg && gl == 0) at = atomicAdd(nlong, 1);
                if (!__any_sync(FULL, lg)) continue;
                at = __shfl_sync(FULL, at, lane & ~(G - 1));
                if (lg && at < HT_NLONG) {
                    if (gl == 0) slong[at] = base + (int64_t)u * ngrp + grp;
                    g[u].len = 0;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            it[u] = gl < g[u].len ? pol.load(n, own, g[u], gl) : Pol::none();
#pragma unroll
        for (int u = 0; u < U; u++) ok = pol.put(n, it[u], t, acc) && ok;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const bool lg = longs && G < 32 && g[u].len > 8 * G;
            if (!lg) {
                for (int32_t off = gl + G; off < g[u].len; off += 2 * G) {
                    typename Pol::Item a = pol.load(n, own, g[u], off);
                    typename Pol::Item b =
                        off + G < g[u].len ? pol.load(n, own, g[u], off + G) : Pol::none();
                    ok = pol.put(n, a, t, acc) && ok;
                    ok = pol.put(n, b, t, acc) && ok;
                }
            }
            unsigned m = longs && G < 32 ? __ballot_sync(FULL, lg && gl == 0) : 0u;
            while (m) {
                int src = __ffs(m) - 1;
                m &= m - 1;
                Seg<S> w;
                w.b = __shfl_sync(FULL, g[u].b, src);
                w.len = __shfl_sync(FULL, g[u].len, src);
                w.w = __shfl_sync(FULL, g[u].w, src);
                w.k = __shfl_sync(FULL, g[u].k, src);
                w.nd = __shfl_sync(FULL, g[u].nd, src);
                w.sd = __shfl_sync(FULL, g[u].sd, src);
                if (Pol::kMasks) {
                    w.dm = __shfl_sync(FULL, g[u].dm, src);
                    w.sm = __shfl_sync(FULL, g[u].sm, src);
                }
                for (int32_t off = G + lane; off < w.len; off += 32)
                    ok = pol.put(n, pol.load(n, own, w, off), t, acc) && ok;
            }
        }
        if (Tb::kFills && !__all_sync(FULL, ok)) break;
    }
    return ok;
}

template <typename S>
__device__ __forceinline__ void clear_slots(const Table<S>& t, int64_t from, int64_t to,
                                            int64_t stride)
{
    for (int64_t i = from; i < to; i += stride) {
        t.key[i] = -1;
        t.sc[i] = 0;
        t.ov[i] = 0;
    }
}

// best over slots [from, to) by `stride`, resetting them
template <typename S, class Pol>
__device__ void scan_slots(const Pol& pol, int32_t n, const Table<S>& t, int64_t from, int64_t to,
                           int64_t stride, const typename Pol::Acc& tot, int64_t& bs, int32_t& bk,
                           uint32_t& bo)
{
    for (int64_t i = from; i < to; i += stride) {
        int32_t k = t.key[i];
        if (k < 0) continue;
        int64_t s = (int64_t)t.sc[i];
        uint32_t o = t.ov[i];
        t.key[i] = -1;
        t.sc[i] = 0;
        t.ov[i] = 0;
        pol.consider(n, k, s, o, tot, bs, bk, bo);
    }
}

__device__ __forceinline__ void warp_argmax(int64_t& bs, int32_t& bm, uint32_t& bo)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        int64_t s2 = __shfl_xor_sync(FULL, bs, o);
        int32_t m2 = __shfl_xor_sync(FULL, bm, o);
        uint32_t o2 = __shfl_xor_sync(FULL, bo, o);
        if (better(s2, m2, bs, bm)) {
            bs = s2;
            bm = m2;
            bo = o2;
        }
    }
}

constexpr int HT_WARPS = 8;
constexpr int HT_WCAP = 512;            // warp table slots
constexpr int HT_WLOAD = HT_WCAP * 3 / 4;
constexpr int HT_BTHREADS = 256;
constexpr int HT_BCAP = 2048;           // block table slots
constexpr int HT_GTHREADS = 512;        // big-block tier
enum : int { HT_TIER_WARP = 0, HT_TIER_BLOCK = 1, HT_TIER_BIG = 2, HT_TIER_SPLIT = 3, HT_NTIER = 4 };
// counters of run_histogram: per-tier vertex counts, then the summed work and
// the number of vertices given a histogram (not skipped)
// and the next list positions the block and big tiers hand out (dynamic
// scheduling: a block takes the next vertex when it is done with one)
enum : int {
    HT_CNT_WORK = HT_NTIER, HT_CNT_VERTS = HT_NTIER + 1, HT_CNT_NEXT = HT_NTIER + 2,
    HT_CNT_TODO = HT_NTIER + 2 + HT_NTIER,   // vertices not skipped (k_ht_skip)
    HT_NCNT = HT_CNT_TODO + 1
};

template <typename S>
__host__ __device__ constexpr int big_cap()
{
    return sizeof(S) == 4 ? 16384 : 8192;
}

__host__ __device__ inline int64_t pow2_ceil(int64_t x)
{
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Work of each vertex: total segment length over its incidences, or -1 when
// the policy decides it without a histogram. One thread per vertex tests
// skip() and lists the vertices to count (warp-aggregated appends); then one
// warp per listed vertex sums its segments. Rounds that evaluate few
// vertices pay a thread, not a warp, per skipped vertex, while full passes
// keep a warp per vertex.
template <class Pol>
__global__ void __launch_bounds__(256) k_ht_skip(Pol pol, int64_t* work, int32_t* todo, int64_t* ntodo)
{
    after_previous();
    int lane = threadIdx.x & 31;
    unsigned lt = lanemask_lt();
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < pol.V;
         base += (int64_t)gridDim.x * blockDim.x) {
        int64_t n = base + threadIdx.x;
        bool count = false;
        if (n < pol.V) {
            if (pol.skip((int32_t)n)) work[n] = -1;
            else count = true;
        }
        unsigned m = __ballot_sync(FULL, count);
        if (!m) continue;
        int leader = __ffs(m) - 1;
        int32_t pos = 0;
        if (lane == leader) pos = (int32_t)atomicAdd((unsigned long long*)ntodo, (unsigned long long)__popc(m));
        pos = __shfl_sync(FULL, pos, leader);
        if (count) todo[pos + __popc(m & lt)] = (int32_t)n;
    }
}

// (A vertex of more than HT_WORK_LONG incidences is summed by its whole
// block: on a tail level one super-node may be in most hyperedges, and one
// warp took 78 us for its 10,000 incidences.)
constexpr int64_t HT_WORK_LONG = 1024;

template <class Pol>
__global__ void __launch_bounds__(256)
    k_ht_work(Pol pol, int64_t* work, const int32_t* __restrict__ todo, const int64_t* __restrict__ ntodo)
{
    after_previous();
    __shared__ unsigned long long part;
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t nt = *ntodo;
    // consecutive vertices go to different blocks: few vertices (a tail level's
    // merged ones) then have a block each
    for (int64_t base = blockIdx.x; base < nt; base += (int64_t)gridDim.x * 8) {
        const int64_t mine = base + (int64_t)warp * gridDim.x;
        bool longer = false;
        if (mine < nt) {
            int32_t n = todo[mine];
            int64_t vb = pol.vb(n), ve = pol.ve(n);
            longer = ve - vb > HT_WORK_LONG;
            if (!longer) {
                int64_t w = 0;
#pragma unroll 4
                for (int64_t i = vb + lane; i < ve; i += 32) w += pol.seg_len(i);
                w = warp_sum(w);
                if (lane == 0) work[n] = w;
            }
        }
        if (!__syncthreads_or(longer)) continue;
        for (int x = 0; x < 8 && base + (int64_t)x * gridDim.x < nt; x++) {
            int32_t n = todo[base + (int64_t)x * gridDim.x];
            int64_t vb = pol.vb(n), ve = pol.ve(n);
            if (ve - vb <= HT_WORK_LONG) continue;
            if (threadIdx.x == 0) part = 0;
            __syncthreads();
            int64_t w = 0;
#pragma unroll 4
            for (int64_t i = vb + threadIdx.x; i < ve; i += 256) w += pol.seg_len(i);
            w = warp_sum(w);
            if (lane == 0) atomicAdd(&part, (unsigned long long)w);
            __syncthreads();
            if (threadIdx.x == 0) work[n] = (int64_t)part;
        }
    }
}

// lists: tier t's vertices at lists + t*V; cnt[t] their number; the split
// tier also records each vertex's table capacity
template <class Pol>
__device__ __forceinline__ void ht_push(const Pol& pol, int tier, int32_t n, int64_t work,
                                        int32_t* lists, int64_t* cnt, int64_t* scap)
{
    int64_t p = (int64_t)atomicAdd((unsigned long long*)&cnt[tier], 1ull);
    lists[(int64_t)tier * pol.V + p] = n;
    if (tier == HT_TIER_SPLIT) {
        int64_t bound = work < pol.keys ? work : pol.keys;
        scap[p] = pow2_ceil(2 * (bound > 16 ? bound : 16));
    }
}

// vertex n (of this thread; n >= V: none) into its tier's list, or its result
// when there is nothing to count; whole warps
template <class Pol>
__device__ __forceinline__ void ht_place(const Pol& pol, int64_t n, int64_t work, int32_t* lists,
                                         int64_t* cnt, int64_t* scap, const HtTiers& tiers, bool dense)
{
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    int tier = -1;
    if (n < pol.V) {
        if (work <= 0) {
            // skipped, or nothing to count: the empty table's result (no key,
            // zero sums) without a histogram
            pol.write((int32_t)n, 0, -1, 0, typename Pol::Acc());
        } else {
            int64_t bound = work < pol.keys ? work : pol.keys;
            // few keys but much work: many warps into one small table, or
            // (dense) a block's arrays
            if (bound <= HT_WLOAD && (work <= tiers.wwork || !dense))
                tier = work <= tiers.wwork ? HT_TIER_WARP : HT_TIER_SPLIT;
            else if (Pol::kOptimistic && work <= tiers.wwork) tier = HT_TIER_WARP;
            else if (work <= tiers.bwork) tier = HT_TIER_BLOCK;
            else if (work <= tiers.gwork) tier = HT_TIER_BIG;
            else tier = HT_TIER_SPLIT;
        }
    }
    for (int t = 0; t < HT_NTIER; t++) {
        unsigned m = __ballot_sync(FULL, tier == t);
        if (!m) continue;
        int leader = __ffs(m) - 1;
        int64_t pos = 0;
        if (lane == leader) pos = (int64_t)atomicAdd((unsigned long long*)&cnt[t], (unsigned long long)__popc(m));
        pos = __shfl_sync(FULL, pos, leader);
        if (tier == t) {
            int64_t p = pos + __popc(m & lt);
            lists[(int64_t)t * pol.V + p] = (int32_t)n;
            if (t == HT_TIER_SPLIT) {
                int64_t bound = work < pol.keys ? work : pol.keys;
                scap[p] = pow2_ceil(2 * (bound > 16 ? bound : 16));
            }
        }
    }
    int64_t ws = warp_sum(tier >= 0 ? work : 0);
    int64_t vs = __popc(__ballot_sync(FULL, tier >= 0));
    if (lane == 0 && vs) {
        atomicAdd((unsigned long long*)&cnt[HT_CNT_WORK], (unsigned long long)ws);
        atomicAdd((unsigned long long*)&cnt[HT_CNT_VERTS], (unsigned long long)vs);
    }
}

template <class Pol>
__global__ void __launch_bounds__(256)
    k_ht_classify(Pol pol, const int64_t* __restrict__ workv, int32_t* lists, int64_t* cnt,
                  int64_t* scap, HtTiers tiers, bool dense)
{
    after_previous();
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < pol.V;
         base += (int64_t)gridDim.x * blockDim.x) {
        int64_t n = base + threadIdx.x;
        ht_place(pol, n, n < pol.V ? workv[n] : -1, lists, cnt, scap, tiers, dense);
    }
}

// The three passes above in one launch, for levels of up to HT_PLAN_V
// vertices, where launches cost more than the work: a block takes 32 vertices
// a grid apart, a warp per listed one sums its segments (the block those of a
// long list), then the first warp classifies them. (Not 32 consecutive ones:
// super-nodes of like size have consecutive ids, and a block that got the
// largest of a 60,000-neuron layered network took 83 us.)
constexpr int32_t HT_PLAN_V = 1 << 16;

template <class Pol>
__global__ void __launch_bounds__(256)
    k_ht_plan(Pol pol, int64_t* workv, int32_t* lists, int64_t* cnt, int64_t* scap, HtTiers tiers,
              bool dense)
{
    after_previous();
    __shared__ int64_t work[32];
    __shared__ unsigned smask;
    __shared__ unsigned long long part;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t mine = blockIdx.x + (int64_t)lane * gridDim.x;
    if (warp == 0) {
        work[lane] = -1;
        unsigned m = __ballot_sync(FULL, mine < pol.V && !pol.skip((int32_t)mine));
        if (lane == 0) smask = m;
    }
    __syncthreads();
    unsigned m = smask, lng = 0;
    // the r-th listed vertex to warp r % 8
    for (int r = 0; m; r++) {
        int t = __ffs(m) - 1;
        m &= m - 1;
        int32_t n = (int32_t)(blockIdx.x + (int64_t)t * gridDim.x);
        int64_t vb = pol.vb(n), ve = pol.ve(n);
        if (ve - vb > HT_WORK_LONG) {
            lng |= 1u << t;
        } else if ((r & 7) == warp) {
            int64_t w = 0;
#pragma unroll 4
            for (int64_t i = vb + lane; i < ve; i += 32) w += pol.seg_len(i);
            w = warp_sum(w);
            if (lane == 0) work[t] = w;
        }
    }
    while (lng) {   // the same in every thread
        int t = __ffs(lng) - 1;
        lng &= lng - 1;
        int32_t n = (int32_t)(blockIdx.x + (int64_t)t * gridDim.x);
        int64_t vb = pol.vb(n), ve = pol.ve(n);
        if (threadIdx.x == 0) part = 0;
        __syncthreads();
        int64_t w = 0;
#pragma unroll 4
        for (int64_t i = vb + threadIdx.x; i < ve; i += 256) w += pol.seg_len(i);
        w = warp_sum(w);
        if (lane == 0) atomicAdd(&part, (unsigned long long)w);
        __syncthreads();
        if (threadIdx.x == 0) work[t] = (int64_t)part;
    }
    __syncthreads();
    if (warp != 0) return;
    if (mine < pol.V) workv[mine] = work[lane];
    ht_place(pol, mine, work[lane], lists, cnt, scap, tiers, dense);
}

template <class Pol>
__global__ void __launch_bounds__(HT_WARPS * 32)
    k_ht_warp(Pol pol, int32_t* lists, int64_t* cnt, const int64_t* __restrict__ workv,
              int64_t* scap)
{
    after_previous();
    using S = typename Pol::S;
    using Acc = typename Pol::Acc;
    extern __shared__ __align__(16) unsigned char ht_dyn[];
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t* list = lists + (int64_t)HT_TIER_WARP * pol.V;
    int64_t nl = cnt[HT_TIER_WARP];
    int64_t gw = blockIdx.x * (int64_t)HT_WARPS + warp, nw = (int64_t)gridDim.x * HT_WARPS;
    Table<S> full = carve_table<S>(ht_dyn + (size_t)warp * HT_WCAP * slot_bytes<S>(), HT_WCAP);
    clear_slots(full, lane, HT_WCAP, 32);
    __syncwarp();
    for (int64_t idx = gw; idx < nl; idx += nw) {
        int32_t n = list[idx];
        int64_t vb = pol.vb(n), ve = pol.ve(n);
        Acc acc;
        int64_t work = workv[n];
        int64_t bound = work < pol.keys ? work : pol.keys;
        int64_t cap = pow2_ceil(2 * (bound > 8 ? bound : 8));
        if (cap > HT_WCAP) cap = HT_WCAP;
        Table<S> t = full;
        t.mask = (uint32_t)(cap - 1);
        // a vertex whose bound fits the table cannot overflow it; others
        // (policies that expect few keys) try it and move on if it fills
        bool sure = bound <= HT_WLOAD;
        t.probes = sure ? (uint32_t)cap : 32u;
        bool ok = warp_visit<S>(pol, n, vb, ve, t, acc);
        __syncwarp();
        if (!ok) {
            clear_slots(t, lane, cap, 32);
            if (lane == 0) ht_push(pol, HT_TIER_BLOCK, n, work, lists, cnt, scap);
            __syncwarp();
            continue;
        }
        Acc tot = Pol::warp_reduce(acc);
        int64_t bs = 0;
        int32_t bk = -1;
        uint32_t bo = 0;
        scan_slots<S>(pol, n, t, lane, cap, 32, tot, bs, bk, bo);
        warp_argmax(bs, bk, bo);
        if (lane == 0) pol.write(n, bs, bk, bo, tot);
        __syncwarp();
    }
}

// the last index lo in [from, n) with spre[lo] <= v (spre non-decreasing,
// spre[from] <= v): one probe while v stays in the same segment, a binary
// search when it moved on
__device__ __forceinline__ int32_t seg_find(const int32_t* spre, int32_t n, int32_t from, int32_t v)
{
    if (from + 1 >= n || spre[from + 1] > v) return from;
    int32_t lo = from + 1, hi = n - 1;
    while (lo < hi) {
        int32_t mid = (lo + hi + 1) >> 1;
        if (spre[mid] <= v) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Block (T threads) per vertex with a CAP-slot shared table; vertices whose
// keys do not fit are pushed to tier `next`. What bounds it is the stream of
// shared-memory operations and the instructions around them, so a vertex
// whose summed weights and multiplicities fit one 32-bit word together uses
// packed sums.
//
// Vertices of more than T / 4 incidences are visited by groups of lanes
// (group_visit): with enough incidences per warp their uneven lengths even
// out, and an element needs no search (level 0 of the 1,048,576-neuron conv
// network: 40.1 -> 29.7 ms, packed sums included). Vertices of fewer keep
// the flattened form (their segments' prefix in shared memory, a search per
// element): on level 0 of the 1,048,576-neuron power-law network, 16
// incidences of 8 to 16,384 pins each, the groups left most of the block
// waiting for the longest (12.7 ms flattened, 15.3 by groups).
//
// Held to 32 registers so that eight blocks share an SM: at 6 blocks (40
// registers) the two networks above take 36.8 and 20.1 ms, at 5 39.5 and
// 21.5, at 8 31.9 and 19.2, a few spilled words included.
// (Their scratch is shared so that it fits: with quads in the table's scan,
// one segment a group in flight and no checks for long segments where the
// level has none, 28.1 and 17.0 ms; 29.2 and 17.2 with ids folded into the
// slots, table_slot.cuh.)
constexpr int HT_BLOCKS = 8;

template <class Pol, int T, int CAP, int TIER, int NEXT>
__global__ void __launch_bounds__(T, CAP <= 2048 ? HT_BLOCKS : 1)
    k_ht_block(Pol pol, int32_t* lists, int64_t* cnt, int64_t* scap, const int64_t* __restrict__ workv,
               int64_t leave)
{
    after_previous();
    using S = typename Pol::S;
    using Acc = typename Pol::Acc;
    extern __shared__ __align__(16) unsigned char ht_dyn[];
    __shared__ int sfail;
    __shared__ int32_t nlong;
    constexpr int FLAT = T / 4;   // most incidences of the flattened form
    // a vertex is flattened or visited by groups: one of the two is in use
    constexpr size_t SEG_BYTES = sizeof(Seg<S>) * FLAT, LONG_BYTES = sizeof(int64_t) * HT_NLONG;
    __shared__ __align__(16) unsigned char sseg_raw[SEG_BYTES > LONG_BYTES ? SEG_BYTES : LONG_BYTES];
    int64_t* slong = (int64_t*)sseg_raw;
    __shared__ int32_t spre[FLAT];
    __shared__ int32_t swarp[FLAT / 32];
    Seg<S>* sseg = (Seg<S>*)sseg_raw;
    __shared__ unsigned long long ssum[2];
    __shared__ __align__(16) unsigned char wacc_raw[sizeof(Acc) * (T / 32)];
    __shared__ int64_t rs[T / 32];
    __shared__ int32_t rk[T / 32];
    __shared__ uint32_t ro[T / 32];
    Acc* wacc = (Acc*)wacc_raw;
    const int nwarps = T / 32;
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (cnt[TIER] <= leave) return;   // so few that the big tier's blocks take them
    // pt shares t's slots: its sums take the place of the weights, its list
    // that of the overlaps, which are cleared when an unpacked vertex follows
    Table<S> t = carve_table<S>(ht_dyn, CAP);
    t.probes = 64;   // a vertex that clusters the table this much moves on
    constexpr bool LIST = CAP > 4096;
    __shared__ int32_t nused;
    PackedTable<LIST> pt;
    pt.key = t.key;
    pt.val = (uint32_t*)t.sc;
    pt.used = (uint16_t*)t.ov;
    pt.nused = &nused;
    pt.mask = t.mask;
    pt.probes = t.probes;
    bool listed = false;   // the list has overwritten overlaps
    clear_slots(t, threadIdx.x, CAP, T);
    const int32_t* list = lists + (int64_t)TIER * pol.V;
    int64_t nl = cnt[TIER];
    __shared__ int64_t snext;
    for (;;) {
        if (threadIdx.x == 0) {
            snext = (int64_t)atomicAdd((unsigned long long*)&cnt[HT_CNT_NEXT + TIER], 1ull);
            sfail = 0;
            nlong = 0;
            nused = 0;
            ssum[0] = ssum[1] = 0;
        }
        __syncthreads();
        int64_t idx = snext;
        if (idx >= nl) break;
        int32_t n = list[idx];
        int64_t vb = pol.vb(n), ve = pol.ve(n);
        const int deg = ve - vb < (int64_t)INT_MAX ? (int)(ve - vb) : INT_MAX;
        const bool flat = deg <= FLAT;
        const int glog = group_log(ve - vb, workv[n]);
        Acc acc;
        bool ok;
        int sb = -1;
        int32_t total = 0;
        unsigned long long wsum = 0, ksum = 0;
        if (flat) {
            if (threadIdx.x < FLAT) {   // whole warps
                Seg<S> g{};
                if ((int)threadIdx.x < deg) g = pol.seg(pol.inc(vb + threadIdx.x), acc);
                sseg[threadIdx.x] = g;
                wsum = g.w;
                ksum = g.k;
                int32_t inc = g.len;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    int32_t t2 = __shfl_up_sync(FULL, inc, o);
                    if (lane >= o) inc += t2;
                }
                spre[threadIdx.x] = inc - g.len;
                if (lane == 31) swarp[warp] = inc;
            }
        } else if (sizeof(S) == 4) {
            Acc other;
            for (int64_t i = vb + threadIdx.x; i < ve; i += T) {
                Seg<S> g = pol.seg(pol.inc(i), other);
                wsum += g.w;
                ksum += g.k;
            }
        }
        // bounds of a key's weight and overlap: the sums over all incidences
        if (sizeof(S) == 4 && vb + (threadIdx.x & ~31) < ve) {
            wsum = warp_sum(wsum);
            ksum = warp_sum(ksum);
            if (lane == 0) {
                atomicAdd(&ssum[0], wsum);
                atomicAdd(&ssum[1], ksum);
            }
        }
        __syncthreads();
        if (flat) {
            int32_t before = 0;
#pragma unroll
            for (int w = 0; w < FLAT / 32; w++) {
                if (w < warp) before += swarp[w];
                total += swarp[w];
            }
            if (threadIdx.x < FLAT && before) spre[threadIdx.x] += before;
            __syncthreads();
        }
        if constexpr (sizeof(S) == 4) {
            int wb = 64 - __clzll((long long)ssum[0]), kb = 64 - __clzll((long long)ssum[1]);
            if (wb + kb <= 32) sb = kb;
            if (LIST && sb < 0 && listed) {   // the same for the whole block
                clear_slots(t, threadIdx.x, CAP, T);
                listed = false;
                __syncthreads();
            }
            if (LIST && sb >= 0) listed = true;
            pt.sb = sb;
        }
        const typename Pol::Own own = pol.own(n);
        auto visit_flat = [&](const auto& tb) {
            constexpr int U = 4;   // elements in flight per thread
            bool k = true;
            int32_t lo = 0;
            for (int32_t v0 = threadIdx.x; v0 < total && k; v0 += U * T) {
                typename Pol::Item it[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    int32_t v = v0 + u * T;
                    if (v < total) {
                        lo = seg_find(spre, deg, lo, v);
                        it[u] = pol.load(n, own, sseg[lo], v - spre[lo]);
                    } else {
                        it[u] = Pol::none();
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) k = pol.put(n, it[u], tb, acc) && k;
            }
            return k;
        };
        auto visit_groups = [&](const auto& tb) {
            bool k = group_visit<S, T, 1, false>(pol, n, vb, ve, glog, threadIdx.x, tb, acc, slong, &nlong);
            __syncthreads();
            const int nlg = nlong < HT_NLONG ? nlong : HT_NLONG;
            Acc other;   // the segments' own terms are in already
            for (int x = 0; x < nlg && k; x++) {
                Seg<S> g = pol.seg(pol.inc(slong[x]), other);
                for (int32_t off = threadIdx.x; off < g.len && k; off += 2 * T) {
                    typename Pol::Item a = pol.load(n, own, g, off);
                    typename Pol::Item b = off + T < g.len ? pol.load(n, own, g, off + T) : Pol::none();
                    k = pol.put(n, a, tb, acc) && k;
                    k = pol.put(n, b, tb, acc) && k;
                }
            }
            return k;
        };
        if (sizeof(S) == 4 && sb >= 0) {
            if (flat) ok = visit_flat(PackedTable<LIST, !LIST>{pt.key, pt.val, pt.used, pt.nused, pt.mask, pt.probes, sb});
            else ok = visit_groups(pt);
        } else {
            ok = flat ? visit_flat(t) : visit_groups(t);
        }
        if (!ok) sfail = 1;
        Acc wa = Pol::warp_reduce(acc);
        if (lane == 0) wacc[warp] = wa;
        __syncthreads();
        if (sfail) {
            clear_slots(t, threadIdx.x, CAP, T);
            if (threadIdx.x == 0) ht_push(pol, NEXT, n, workv[n], lists, cnt, scap);
            __syncthreads();
            continue;
        }
        Acc tot = wacc[0];
        for (int w = 1; w < nwarps; w++) tot.add(wacc[w]);
        int64_t bs = 0;
        int32_t bk = -1;
        uint32_t bo = 0;
        if (sb >= 0) {
            const uint32_t omask = (1u << sb) - 1;   // sb < 32: multiplicities sum below 2^31
            if (LIST) {
                const int nk = nused;
                for (int x = threadIdx.x; x < nk; x += T) {
                    int i = pt.used[x];
                    int32_t k = pt.key[i];
                    uint32_t v = pt.val[i];
                    pt.key[i] = -1;
                    pt.val[i] = 0;
                    pol.consider(n, k, (int64_t)(v >> sb), v & omask, tot, bs, bk, bo);
                }
            } else {
                for (int i = 4 * threadIdx.x; i < CAP; i += 4 * T) {
                    int4* kp = reinterpret_cast<int4*>(pt.key + i);
                    uint4* vp = reinterpret_cast<uint4*>(pt.val + i);
                    const int4 k4 = *kp;
                    if ((k4.x & k4.y & k4.z & k4.w) == -1) continue;
                    const uint4 v4 = *vp;
                    *kp = make_int4(-1, -1, -1, -1);
                    *vp = make_uint4(0, 0, 0, 0);
                    const int32_t ks[4] = {k4.x, k4.y, k4.z, k4.w};
                    const uint32_t vs[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (ks[u] >= 0)
                            pol.consider(n, ks[u], (int64_t)(vs[u] >> sb), vs[u] & omask, tot, bs, bk, bo);
                }
            }
        } else {
            scan_slots<S>(pol, n, t, threadIdx.x, CAP, T, tot, bs, bk, bo);
        }
        warp_argmax(bs, bk, bo);
        if (lane == 0) {
            rs[warp] = bs;
            rk[warp] = bk;
            ro[warp] = bo;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < nwarps; w++)
                if (better(rs[w], rk[w], bs, bk)) {
                    bs = rs[w];
                    bk = rk[w];
                    bo = ro[w];
                }
            pol.write(n, bs, bk, bo, tot);
        }
        __syncthreads();
    }
}

// Dense tier: where the key space is small enough for one word pair per key
// in shared memory, a block counts a vertex straight into arrays indexed by
// key: no hashing, no probing, no table that can fill up, hence no vertex
// handed on, no split tier and no wait for its sizes. Presence of a key is a
// nonzero sum, so every weight has to be positive (the callers know).
//
// Four incidences are in flight per group, since a block walking one heavy
// super-node's incidences is a chain of gathers (incidence -> hyperedge ->
// pins).
//
// Clearing, scanning and occupancy bound it from above: a vertex costs the
// whole key range once, so vertices of little work stay on the hash tiers
// unless the range itself is small (HT_DENSE_SMALL).
constexpr int64_t HT_DENSE_KEYS = 24 * 1024;   // 192 KB of 32-bit sum pairs
constexpr int64_t HT_DENSE_SMALL = 4 * 1024;   // 32 KB: several 256-thread blocks per SM
constexpr int64_t HT_DENSE_BWORK = 8192;       // most elements a 256-thread block takes there

template <typename S>
struct DenseTable {
    static constexpr bool kFills = false;
    S* sc;
    uint32_t* ov;
    __device__ __forceinline__ bool add(int32_t m, S w, uint32_t o) const
    {
        atomicAdd(&sc[m], w);
        if (o) atomicAdd(&ov[m], o);
        return true;
    }
};


// one vertex by one block: its elements into the arrays, the sums of the
// policy's per-vertex terms into wacc[0..T/32)
template <class Pol, int T>
__device__ __forceinline__ void dense_count(const Pol& pol, int32_t n, int64_t vb, int64_t ve, int glog,
                                            const DenseTable<typename Pol::S>& t,
                                            typename Pol::Acc* wacc, int64_t* slong, int32_t* nlong)
{
    using S = typename Pol::S;
    using Acc = typename Pol::Acc;
    const typename Pol::Own own = pol.own(n);
    Acc acc, other;
    group_visit<S, T, 2, true>(pol, n, vb, ve, glog, threadIdx.x, t, acc, slong, nlong);
    __syncthreads();
    const int nlg = *nlong < HT_NLONG ? *nlong : HT_NLONG;
    for (int x = 0; x < nlg; x++) {
        Seg<S> g = pol.seg(pol.inc(slong[x]), other);   // its own terms are in already
        for (int32_t off = threadIdx.x; off < g.len; off += T)
            pol.put(n, pol.load(n, own, g, off), t, acc);
    }
    Acc wa = Pol::warp_reduce(acc);
    if ((threadIdx.x & 31) == 0) wacc[threadIdx.x >> 5] = wa;
    __syncthreads();
}

struct HtBest {
    int64_t s;
    int32_t k;
    uint32_t o;
};

// best of the block's threads, valid in thread 0
template <int T>
__device__ __forceinline__ HtBest block_best(int64_t bs, int32_t bk, uint32_t bo, HtBest* wbest)
{
    warp_argmax(bs, bk, bo);
    if ((threadIdx.x & 31) == 0) wbest[threadIdx.x >> 5] = HtBest{bs, bk, bo};
    __syncthreads();
    HtBest b = wbest[0];
    if (threadIdx.x == 0)
        for (int w = 1; w < T / 32; w++)
            if (better(wbest[w].s, wbest[w].k, b.s, b.k)) b = wbest[w];
    return b;
}

// one vertex by one block, to its result
template <class Pol, int T>
__device__ __forceinline__ void dense_vertex(const Pol& pol, int32_t n, int64_t work, int32_t keys,
                                             const DenseTable<typename Pol::S>& t,
                                             typename Pol::Acc* wacc, HtBest* wbest, int64_t* slong,
                                             int32_t* nlong)
{
    using S = typename Pol::S;
    const int64_t vb = pol.vb(n), ve = pol.ve(n);
    dense_count<Pol, T>(pol, n, vb, ve, group_log(ve - vb, work), t, wacc, slong, nlong);
    typename Pol::Acc tot = wacc[0];
    for (int w = 1; w < T / 32; w++) tot.add(wacc[w]);
    int64_t bs = 0;
    int32_t bk = -1;
    uint32_t bo = 0;
    for (int32_t k = threadIdx.x; k < keys; k += T) {
        S v = t.sc[k];
        if (v == 0) continue;
        uint32_t o = t.ov[k];
        t.sc[k] = 0;
        t.ov[k] = 0;
        pol.consider(n, k, (int64_t)v, o, tot, bs, bk, bo);
    }
    HtBest b = block_best<T>(bs, bk, bo, wbest);
    if (threadIdx.x == 0) pol.write(n, b.s, b.k, b.o, tot);
    __syncthreads();
}

template <class Pol, int T, int TIER>
__global__ void __launch_bounds__(T)
    k_ht_dense(Pol pol, const int32_t* __restrict__ lists, int64_t* cnt, int32_t keys,
               const int64_t* __restrict__ workv)
{
    after_previous();
    using S = typename Pol::S;
    using Acc = typename Pol::Acc;
    extern __shared__ __align__(16) unsigned char ht_dyn[];
    __shared__ int64_t slong[HT_NLONG];
    __shared__ int32_t nlong;
    __shared__ __align__(16) unsigned char wacc_raw[sizeof(Acc) * (T / 32)];
    __shared__ HtBest wbest[T / 32];
    __shared__ int64_t snext;
    DenseTable<S> t{(S*)ht_dyn, (uint32_t*)(ht_dyn + (size_t)keys * sizeof(S))};
    const int32_t* list = lists + (int64_t)TIER * pol.V;
    const int64_t nl = cnt[TIER];
    if (nl == 0) return;
    for (int32_t k = threadIdx.x; k < keys; k += T) {
        t.sc[k] = 0;
        t.ov[k] = 0;
    }
    for (;;) {
        if (threadIdx.x == 0) {
            snext = (int64_t)atomicAdd((unsigned long long*)&cnt[HT_CNT_NEXT + TIER], 1ull);
            nlong = 0;
        }
        __syncthreads();
        const int64_t idx = snext;
        if (idx >= nl) break;
        const int32_t n = list[idx];
        dense_vertex<Pol, T>(pol, n, workv[n], keys, t, (Acc*)wacc_raw, wbest, slong, &nlong);
    }
}

// The big tier. While it holds few vertices (a tail level has a handful for
// the whole GPU), a cluster of eight blocks takes one, each block counting an
// eighth of its incidences into its own arrays; the sums are joined through
// distributed shared memory, an eighth of the keys per block. One block alone
// is bound by its SM's shared-memory atomics (67 to 177 us for the one merged
// super-node of a level of the 12,007-neuron power-law network, 23 with the
// cluster). With more than HT_SOLO vertices every block takes its own (the
// 60,052-neuron layered network: 65 us a level, 113 with clusters). A block
// tier of at most `leave` vertices is taken here as well: their latency on
// 256 threads each would be the level's (79 us).
constexpr int HT_DENSE_CTAS = 8;
constexpr int64_t HT_SOLO = 38;       // two waves of clusters
constexpr int64_t HT_LEAVE = 304;     // two waves of blocks

template <class Pol, int T>
__global__ void __cluster_dims__(HT_DENSE_CTAS, 1, 1) __launch_bounds__(T)
    k_ht_dense_big(Pol pol, const int32_t* __restrict__ lists, int64_t* cnt, int32_t keys,
                   const int64_t* __restrict__ workv, int64_t leave)
{
    after_previous();
    namespace cg = cooperative_groups;
    using S = typename Pol::S;
    using Acc = typename Pol::Acc;
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char ht_dyn[];
    __shared__ int64_t slong[HT_NLONG];
    __shared__ int32_t nlong;
    __shared__ __align__(16) unsigned char wacc_raw[sizeof(Acc) * (T / 32)];
    __shared__ HtBest wbest[T / 32];
    __shared__ HtBest sbest;
    __shared__ int64_t snext;
    Acc* wacc = (Acc*)wacc_raw;
    DenseTable<S> t{(S*)ht_dyn, (uint32_t*)(ht_dyn + (size_t)keys * sizeof(S))};
    const int rank = (int)cl.block_rank();
    const int64_t nb = cnt[HT_TIER_BLOCK] <= leave ? cnt[HT_TIER_BLOCK] : 0;
    const int64_t nl = nb + cnt[HT_TIER_BIG];
    if (nl == 0) return;   // every block
    auto vertex = [&](int64_t idx) {
        return idx < nb ? lists[(int64_t)HT_TIER_BLOCK * pol.V + idx]
                        : lists[(int64_t)HT_TIER_BIG * pol.V + (idx - nb)];
    };
    unsigned long long* next = (unsigned long long*)&cnt[HT_CNT_NEXT + HT_TIER_BIG];
    for (int32_t k = threadIdx.x; k < keys; k += T) {
        t.sc[k] = 0;
        t.ov[k] = 0;
    }
    if (nl > HT_SOLO) {
        for (;;) {
            if (threadIdx.x == 0) {
                snext = (int64_t)atomicAdd(next, 1ull);
                nlong = 0;
            }
            __syncthreads();
            const int64_t idx = snext;
            if (idx >= nl) return;
            const int32_t n = vertex(idx);
            dense_vertex<Pol, T>(pol, n, workv[n], keys, t, wacc, wbest, slong, &nlong);
        }
    }
    for (;;) {
        if (threadIdx.x == 0) {
            if (rank == 0) snext = (int64_t)atomicAdd(next, 1ull);
            nlong = 0;
        }
        cl.sync();
        const int64_t idx = *cl.map_shared_rank(&snext, 0);
        if (idx >= nl) break;
        const int32_t n = vertex(idx);
        const int64_t v0 = pol.vb(n), deg = pol.ve(n) - v0;
        dense_count<Pol, T>(pol, n, v0 + deg * rank / HT_DENSE_CTAS, v0 + deg * (rank + 1) / HT_DENSE_CTAS,
                            group_log(deg, workv[n]), t, wacc, slong, &nlong);
        if (threadIdx.x == 0)
            for (int w = 1; w < T / 32; w++) wacc[0].add(wacc[w]);
        cl.sync();   // counts and sums of all blocks are in
        Acc tot = *cl.map_shared_rank(&wacc[0], 0);
        for (int r = 1; r < HT_DENSE_CTAS; r++) tot.add(*cl.map_shared_rank(&wacc[0], r));
        int64_t bs = 0;
        int32_t bk = -1;
        uint32_t bo = 0;
        const S* sc[HT_DENSE_CTAS];
        const uint32_t* ov[HT_DENSE_CTAS];
#pragma unroll
        for (int r = 0; r < HT_DENSE_CTAS; r++) {
            sc[r] = cl.map_shared_rank(t.sc, r);
            ov[r] = cl.map_shared_rank(t.ov, r);
        }
        for (int32_t k = rank * T + threadIdx.x; k < keys; k += HT_DENSE_CTAS * T) {
            S v = 0;
#pragma unroll
            for (int r = 0; r < HT_DENSE_CTAS; r++) v += sc[r][k];
            if (v == 0) continue;
            uint32_t o = 0;
#pragma unroll
            for (int r = 0; r < HT_DENSE_CTAS; r++) o += ov[r][k];
            pol.consider(n, k, (int64_t)v, o, tot, bs, bk, bo);
        }
        HtBest b = block_best<T>(bs, bk, bo, wbest);
        if (threadIdx.x == 0) sbest = b;
        cl.sync();   // every block has read the arrays
        if (rank == 0 && threadIdx.x == 0) {
            for (int r = 1; r < HT_DENSE_CTAS; r++) {
                HtBest c = *cl.map_shared_rank(&sbest, r);
                if (better(c.s, c.k, b.s, b.k)) b = c;
            }
            pol.write(n, b.s, b.k, b.o, tot);
        }
        for (int32_t k = threadIdx.x; k < keys; k += T) {
            if (t.sc[k]) {
                t.sc[k] = 0;
                t.ov[k] = 0;
            }
        }
    }
    cl.sync();   // no block leaves while another reads its shared memory
}

// Split tier. The incidences of the split vertices are laid out flat
// (vertex j owns flat positions [od[j], od[j+1])) and cut into work items of
// about `item` elements: an item starts at a vertex's first incidence or
// where the running element count crosses a multiple of `item`. The item
// size is chosen so that the items outnumber the resident warps.

__device__ __forceinline__ int64_t find_owner(const int64_t* od, int64_t ns, int64_t f)
{
    int64_t lo = 0, hi = ns - 1;
    while (lo < hi) {
        int64_t mid = (lo + hi + 1) >> 1;
        if (od[mid] <= f) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// degree, table capacity (twice the key bound, at most twice `limit` when
// limit > 0) and total work of the split vertices
template <class Pol>
__global__ void k_ht_split_deg(Pol pol, const int32_t* __restrict__ slist, int64_t ns, int64_t* deg,
                               const int64_t* __restrict__ workv, int64_t* total_work,
                               int64_t* scap, int64_t limit)
{
    after_previous();
    int64_t w = 0;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < ns;
         j += (int64_t)gridDim.x * blockDim.x) {
        int32_t n = slist[j];
        deg[j] = pol.ve(n) - pol.vb(n);
        int64_t work = workv[n];
        w += work;
        int64_t bound = work < pol.keys ? work : pol.keys;
        if (limit > 0 && bound > limit) bound = limit;
        scap[j] = pow2_ceil(2 * (bound > 16 ? bound : 16));
    }
    w = warp_sum(w);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd((unsigned long long*)total_work, (unsigned long long)w);
}

template <class Pol>
__global__ void k_ht_split_len(Pol pol, const int32_t* __restrict__ slist, int64_t ns,
                               const int64_t* __restrict__ od, int64_t D, int64_t* len)
{
    after_previous();
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < D;
         f += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = find_owner(od, ns, f);
        len[f] = pol.seg_len(pol.vb(slist[j]) + (f - od[j]));
    }
}

static __global__ void k_ht_split_starts(int64_t ns, const int64_t* __restrict__ od, int64_t D,
                                  const int64_t* __restrict__ x, const int64_t* __restrict__ len,
                                  int32_t* start, int64_t item)
{
    after_previous();
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < D;
         f += (int64_t)gridDim.x * blockDim.x) {
        int64_t j = find_owner(od, ns, f);
        int64_t base = x[od[j]];
        int s = 0;
        if (f == od[j]) s = 1;
        else {
            int64_t b0 = (x[f - 1] - base) / item, b1 = (x[f] - base) / item;
            s = b1 != b0;
        }
        start[f] = s;
    }
}

static __global__ void k_ht_split_items(int64_t D, const int32_t* __restrict__ start,
                                 const int32_t* __restrict__ pos, int64_t* item_f0)
{
    after_previous();
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < D;
         f += (int64_t)gridDim.x * blockDim.x)
        if (start[f]) item_f0[pos[f]] = f;
}

// adds the used slots of a warp-private table into the global table g and
// clears them
template <typename S>
__device__ bool flush_private(const Table<S>& p, int64_t cap, const Table<S>& g)
{
    int lane = threadIdx.x & 31;
    bool ok = true;
    for (int64_t i = lane; i < cap; i += 32) {
        int32_t k = p.key[i];
        if (k < 0) continue;
        if (!g.add(k, p.sc[i], p.ov[i])) ok = false;
        p.key[i] = -1;
        p.sc[i] = 0;
        p.ov[i] = 0;
    }
    __syncwarp();
    return __all_sync(FULL, ok);
}

// Items of vertices with few possible keys (table capacity <= HT_WCAP) are
// counted in a warp-private shared table first and flushed once per item,
// so many warps working for one vertex do not all hit the same few global
// slots; other items add straight into the global table.
template <class Pol>
__global__ void __launch_bounds__(HT_WARPS * 32)
    k_ht_split_visit(Pol pol, const int32_t* __restrict__ slist, int64_t ns,
                     const int64_t* __restrict__ od, int64_t D,
                     const int64_t* __restrict__ item_f0, int64_t nitems,
                     const int64_t* __restrict__ toff, const int64_t* __restrict__ scap,
                     unsigned char* pool, typename Pol::Acc* gacc, int32_t* ovf, uint32_t probes,
                     const int64_t* __restrict__ workv)
{
    after_previous();
    using S = typename Pol::S;
    using Acc = typename Pol::Acc;
    extern __shared__ __align__(16) unsigned char ht_dyn[];
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Table<S> priv = carve_table<S>(ht_dyn + (size_t)warp * HT_WCAP * slot_bytes<S>(), HT_WCAP);
    clear_slots(priv, lane, HT_WCAP, 32);
    __syncwarp();
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = gw; it < nitems; it += nw) {
        int64_t f0 = item_f0[it];
        int64_t f1 = it + 1 < nitems ? item_f0[it + 1] : D;
        int64_t j = find_owner(od, ns, f0);
        if (f1 > od[j + 1]) f1 = od[j + 1];
        int32_t n = slist[j];
        int64_t vb = pol.vb(n) + (f0 - od[j]);
        int64_t ve = pol.vb(n) + (f1 - od[j]);
        Table<S> g = carve_table<S>(pool + toff[j] * slot_bytes<S>(), scap[j]);
        if (probes) g.probes = probes;
        Acc acc;
        bool ok;
        const int glog = group_log(od[j + 1] - od[j], workv[n]);
        if (scap[j] <= HT_WCAP) {
            Table<S> p = priv;
            p.mask = (uint32_t)(scap[j] - 1);
            p.probes = (uint32_t)scap[j];
            ok = __all_sync(FULL, (group_visit<S, 32, 2, false>(pol, n, vb, ve, glog, lane, p, acc)));
            __syncwarp();
            ok = flush_private(p, scap[j], g) && ok;
        } else {
            ok = __all_sync(FULL, (group_visit<S, 32, 2, false>(pol, n, vb, ve, glog, lane, g, acc)));
        }
        if (!ok && lane == 0) ovf[j] = 1;
        Acc wa = Pol::warp_reduce(acc);
        if (lane == 0) wa.atomic_into(&gacc[j]);
    }
}

template <class Pol>
__global__ void __launch_bounds__(1024)
    k_ht_split_scan(Pol pol, const int32_t* __restrict__ slist, int64_t ns,
                    const int64_t* __restrict__ toff, const int64_t* __restrict__ scap,
                    unsigned char* pool, const typename Pol::Acc* gacc,
                    const int32_t* __restrict__ ovf)
{
    after_previous();
    using S = typename Pol::S;
    __shared__ int64_t rs[32];
    __shared__ int32_t rk[32];
    __shared__ uint32_t ro[32];
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int nwarps = blockDim.x >> 5;
    for (int64_t j = blockIdx.x; j < ns; j += gridDim.x) {
        if (ovf[j]) continue;   // redone with a larger table
        int32_t n = slist[j];
        Table<S> t = carve_table<S>(pool + toff[j] * slot_bytes<S>(), scap[j]);
        typename Pol::Acc tot = gacc[j];
        int64_t bs = 0;
        int32_t bk = -1;
        uint32_t bo = 0;
        scan_slots<S>(pol, n, t, threadIdx.x, scap[j], blockDim.x, tot, bs, bk, bo);
        warp_argmax(bs, bk, bo);
        if (lane == 0) {
            rs[warp] = bs;
            rk[warp] = bk;
            ro[warp] = bo;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < nwarps; w++)
                if (better(rs[w], rk[w], bs, bk)) {
                    bs = rs[w];
                    bk = rk[w];
                    bo = ro[w];
                }
            pol.write(n, bs, bk, bo, tot);
        }
        __syncthreads();
    }
}

static __global__ void k_ht_collect_ovf(const int32_t* __restrict__ slist, int64_t ns,
                                        const int32_t* __restrict__ ovf, int32_t* out, int64_t* cnt)
{
    after_previous();
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < ns;
         j += (int64_t)gridDim.x * blockDim.x)
        if (ovf[j]) out[atomicAdd((unsigned long long*)cnt, 1ull)] = slist[j];
}

template <typename S>
__global__ void k_ht_pool_clear(unsigned char* pool, const int64_t* __restrict__ toff,
                                const int64_t* __restrict__ scap, int64_t ns)
{
    after_previous();
    for (int64_t j = blockIdx.x; j < ns; j += gridDim.x) {
        Table<S> t = carve_table<S>(pool + toff[j] * slot_bytes<S>(), scap[j]);
        clear_slots(t, threadIdx.x, scap[j], blockDim.x);
    }
}

template <typename K>
inline Status set_smem(K kernel, size_t bytes)
{
    if (bytes > 48 * 1024)
        SNN_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return Status{};
}

constexpr int64_t HT_SPLIT_CAP = 1 << 16;

// Split tier for the vertices slist[0..ns). limit > 0 caps the tables and
// appends the vertices that overflowed to `again` at the device counter
// *nagain (the caller clears it; h_cnt[0] receives its new value);
// limit == 0 sizes every table to its exact bound, which cannot overflow.
template <class Pol>
Status run_split(const Pol& pol, Arena& ar, cudaStream_t s, const int32_t* sl, int64_t ns,
                 const int64_t* workv, int64_t limit, int32_t* again, int64_t* nagain,
                 int64_t* h_cnt)
{
    using S = typename Pol::S;
    int64_t *toff, *deg, *od, *tot, *scap;
    int32_t* ovf;
    SNN_TRY(ar.alloc(&toff, ns + 1));
    SNN_TRY(ar.alloc(&deg, ns));
    SNN_TRY(ar.alloc(&od, ns + 1));
    SNN_TRY(ar.alloc(&tot, 4));
    SNN_TRY(ar.alloc(&scap, ns));
    SNN_TRY(ar.alloc(&ovf, ns));
    SNN_CUDA(cudaMemsetAsync(tot, 0, 4 * sizeof(int64_t), s));
    SNN_CUDA(cudaMemsetAsync(ovf, 0, (size_t)ns * sizeof(int32_t), s));
    enqueue(k_ht_split_deg<Pol>, grid_for(ns, 256), 256, 0, s, pol, sl, ns, deg, workv, tot + 2, scap,
            limit);
    SNN_CUDA(cudaGetLastError());
    SNN_TRY(scan_exclusive_i64(scap, toff, ns, tot, ar, s));
    SNN_TRY(scan_exclusive_i64(deg, od, ns, od + ns, ar, s));
    SNN_CUDA(cudaMemcpyAsync(h_cnt, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SNN_CUDA(cudaMemcpyAsync(h_cnt + 1, od + ns, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SNN_CUDA(cudaMemcpyAsync(h_cnt + 2, tot + 2, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SNN_CUDA(cudaStreamSynchronize(s));
    int64_t slots = h_cnt[0], D = h_cnt[1];
    int64_t item = pow2_ceil(h_cnt[2] / (152 * 64 * 2) + 1);
    item = item < 1024 ? 1024 : (item > 16384 ? 16384 : item);
    int64_t *len, *x, *item_f0;
    int32_t *start, *pos;
    SNN_TRY(ar.alloc(&len, D));
    SNN_TRY(ar.alloc(&x, D));
    SNN_TRY(ar.alloc(&start, D));
    SNN_TRY(ar.alloc(&pos, D));
    SNN_TRY(ar.alloc(&item_f0, D));
    enqueue(k_ht_split_len<Pol>, grid_for(D, 256), 256, 0, s, pol, sl, ns, od, D, len);
    SNN_CUDA(cudaGetLastError());
    SNN_TRY(scan_exclusive_i64(len, x, D, nullptr, ar, s));
    enqueue(k_ht_split_starts, grid_for(D, 256), 256, 0, s, ns, od, D, x, len, start, item);
    SNN_CUDA(cudaGetLastError());
    SNN_TRY(scan_exclusive_i32(start, pos, D, (int32_t*)(tot + 1), ar, s));
    enqueue(k_ht_split_items, grid_for(D, 256), 256, 0, s, D, start, pos, item_f0);
    SNN_CUDA(cudaGetLastError());
    SNN_CUDA(cudaMemcpyAsync(h_cnt, tot + 1, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SNN_CUDA(cudaStreamSynchronize(s));
    int64_t items = h_cnt[0];
    unsigned char* pool;
    typename Pol::Acc* gacc;
    SNN_TRY(ar.alloc(&pool, slots * (int64_t)slot_bytes<S>()));
    SNN_TRY(ar.alloc(&gacc, ns));
    SNN_CUDA(cudaMemsetAsync(gacc, 0, (size_t)ns * sizeof(typename Pol::Acc), s));
    enqueue(k_ht_pool_clear<S>, (int)std::min<int64_t>(ns, 152 * 8), 256, 0, s, pool, toff, scap, ns);
    SNN_CUDA(cudaGetLastError());
    size_t wsm = (size_t)HT_WARPS * HT_WCAP * slot_bytes<S>();
    SNN_TRY(set_smem(k_ht_split_visit<Pol>, wsm));
    enqueue(k_ht_split_visit<Pol>, (int)std::min<int64_t>(ceil_div(items, HT_WARPS), 152 * 8),
            HT_WARPS * 32, wsm, s, pol, sl, ns, od, D, item_f0, items, toff, scap, pool, gacc, ovf,
            limit > 0 ? 256u : 0u, workv);
    SNN_CUDA(cudaGetLastError());
    enqueue(k_ht_split_scan<Pol>, (int)std::min<int64_t>(ns, 152 * 4), 1024, 0, s, pol, sl, ns, toff,
            scap, pool, gacc, ovf);
    SNN_CUDA(cudaGetLastError());
    if (limit > 0) {
        enqueue(k_ht_collect_ovf, grid_for(ns, 256), 256, 0, s, sl, ns, ovf, again, nagain);
        SNN_CUDA(cudaGetLastError());
        SNN_CUDA(cudaMemcpyAsync(h_cnt, nagain, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        SNN_CUDA(cudaStreamSynchronize(s));
    }
    return Status{};
}

// table capacity of each split-tier vertex (as k_ht_split_deg sizes it)
template <class Pol>
__global__ void k_ht_split_caps(Pol pol, const int32_t* __restrict__ slist, int64_t ns,
                                const int64_t* __restrict__ workv, int64_t limit, int64_t* caps)
{
    after_previous();
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < ns;
         j += (int64_t)gridDim.x * blockDim.x) {
        int64_t work = workv[slist[j]];
        int64_t bound = work < pol.keys ? work : pol.keys;
        if (limit > 0 && bound > limit) bound = limit;
        caps[j] = pow2_ceil(2 * (bound > 16 ? bound : 16));
    }
}

// cuts[c] .. cuts[c+1]: consecutive runs of slist whose tables hold at most
// pool_slots slots together (a single larger vertex forms its own run)
template <class Pol>
Status split_cuts(const Pol& pol, Arena& ar, cudaStream_t s, const int32_t* sl, int64_t ns,
                  const int64_t* workv, int64_t limit, int64_t pool_slots,
                  std::vector<int64_t>& cuts)
{
    cuts.assign(1, 0);
    if (ns <= 0) return Status{};
    Arena::Mark m = ar.mark();
    int64_t *caps, *pre;
    SNN_TRY(ar.alloc(&caps, ns));
    SNN_TRY(ar.alloc(&pre, ns));
    enqueue(k_ht_split_caps<Pol>, grid_for(ns, 256), 256, 0, s, pol, sl, ns, workv, limit, caps);
    SNN_CUDA(cudaGetLastError());
    SNN_TRY(scan_inclusive_i64(caps, pre, ns, ar, s));
    std::vector<int64_t> hp((size_t)ns);
    SNN_CUDA(cudaMemcpyAsync(hp.data(), pre, (size_t)ns * 8, cudaMemcpyDeviceToHost, s));
    SNN_CUDA(cudaStreamSynchronize(s));
    ar.rewind(m);
    int64_t start = 0;
    while (start < ns) {
        int64_t base = start > 0 ? hp[(size_t)start - 1] : 0;
        int64_t j = std::upper_bound(hp.begin() + start, hp.end(), base + pool_slots) - hp.begin();
        if (j <= start) j = start + 1;
        cuts.push_back(j);
        start = j;
    }
    return Status{};
}

// Host driver: work, classification and the warp, block and big-block tiers
// run without host synchronization; the split tier follows reads of its
// sizes. d_cnt: >= HT_NCNT device int64 (per-tier counts, summed work, vertices
// histogrammed); h_cnt: a pinned host int64[>=3].
template <class Pol>
Status run_histogram(const Pol& pol, Arena& ar, cudaStream_t s, int64_t* d_cnt, int64_t* h_cnt,
                     HtTiers tiers, int32_t key_space, bool positive)
{
    using S = typename Pol::S;
    int32_t V = pol.V;
    if (V <= 0) return Status{};
    // forms of the block and the big tier: arrays over the whole key space
    // where they fit (see k_ht_dense), else hash tables
    const bool dense_big = positive && sizeof(S) == 4 && key_space <= HT_DENSE_KEYS;
    const bool dense_block = dense_big && key_space <= HT_DENSE_SMALL;
    if (dense_block && tiers.bwork > HT_DENSE_BWORK && tiers.bwork < tiers.gwork)
        tiers.bwork = HT_DENSE_BWORK;
    // a vertex meets every pin of the level at most once
    const bool split = !dense_big || tiers.gwork < pol.L.P;
    int32_t* lists;
    int64_t *scap, *workv;
    SNN_TRY(ar.alloc(&lists, (int64_t)HT_NTIER * V));
    SNN_TRY(ar.alloc(&scap, V));
    SNN_TRY(ar.alloc(&workv, V));
    SNN_CUDA(cudaMemsetAsync(d_cnt, 0, HT_NCNT * sizeof(int64_t), s));
    if (V <= HT_PLAN_V) {
        enqueue(k_ht_plan<Pol>, (int)ceil_div(V, 32), 256, 0, s, pol, workv, lists, d_cnt, scap, tiers,
                dense_big);
    } else {
        int32_t* todo;
        int64_t* ntodo = d_cnt + HT_CNT_TODO;
        SNN_TRY(ar.alloc(&todo, V));
        enqueue(k_ht_skip<Pol>, grid_for(V, 256), 256, 0, s, pol, workv, todo, ntodo);
        enqueue(k_ht_work<Pol>, grid_for(V, 8, 152 * 16), 256, 0, s, pol, workv, todo, ntodo);
        SNN_CUDA(cudaGetLastError());
        enqueue(k_ht_classify<Pol>, grid_for(V, 256), 256, 0, s, pol, workv, lists, d_cnt, scap, tiers,
                dense_big);
    }
    SNN_CUDA(cudaGetLastError());
    size_t wsm = (size_t)HT_WARPS * HT_WCAP * slot_bytes<S>();
    size_t bsm = (size_t)HT_BCAP * slot_bytes<S>();
    size_t gsm = (size_t)big_cap<S>() * slot_bytes<S>();
    auto kb = k_ht_block<Pol, HT_BTHREADS, HT_BCAP, HT_TIER_BLOCK, HT_TIER_BIG>;
    auto kg = k_ht_block<Pol, HT_GTHREADS, big_cap<S>(), HT_TIER_BIG, HT_TIER_SPLIT>;
    // set on every call: the attribute is per device, and handles on other
    // host threads may reach this point concurrently
    SNN_TRY(set_smem(k_ht_warp<Pol>, wsm));
    enqueue(k_ht_warp<Pol>, (int)std::min<int64_t>(ceil_div(V, HT_WARPS), 152 * 8), HT_WARPS * 32, wsm,
            s, pol, lists, d_cnt, workv, scap);
    SNN_CUDA(cudaGetLastError());
    const size_t dsm = (size_t)key_space * (sizeof(S) + sizeof(uint32_t));
    if constexpr (sizeof(S) == 4) {
        if (dense_block) {
            auto kd = k_ht_dense<Pol, HT_BTHREADS, HT_TIER_BLOCK>;
            enqueue(kd, (int)std::min<int64_t>(V, 152 * 6), HT_BTHREADS, dsm, s, pol, lists, d_cnt,
                    key_space, workv);
        }
        if (dense_big) {
            auto kd = k_ht_dense_big<Pol, 1024>;
            const int64_t leave = dense_block ? 0 : HT_LEAVE;
            if (!dense_block) {
                SNN_TRY(set_smem(kb, bsm));
                enqueue(kb, (int)std::min<int64_t>(V, 152 * 8), HT_BTHREADS, bsm, s, pol, lists, d_cnt,
                        scap, workv, leave);
            }
            SNN_TRY(set_smem(kd, (size_t)HT_DENSE_KEYS * 8));
            enqueue(kd, 19 * HT_DENSE_CTAS, 1024, dsm, s, pol, lists, d_cnt, key_space, workv, leave);
        }
    }
    if (!dense_big) {
        SNN_TRY(set_smem(kb, bsm));
        enqueue(kb, (int)std::min<int64_t>(V, 152 * 8), HT_BTHREADS, bsm, s, pol, lists, d_cnt, scap,
                workv, 0);
        SNN_TRY(set_smem(kg, gsm));
        enqueue(kg, 152, HT_GTHREADS, gsm, s, pol, lists, d_cnt, scap, workv, 0);
    }
    SNN_CUDA(cudaGetLastError());
    if (!split) return Status{};
    SNN_CUDA(cudaMemcpyAsync(h_cnt, d_cnt + HT_TIER_SPLIT, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    SNN_CUDA(cudaStreamSynchronize(s));
    int64_t ns = h_cnt[0];
    if (ns == 0) return Status{};
    const int32_t* sl = lists + (int64_t)HT_TIER_SPLIT * V;
    // first pass with tables capped at 2 * HT_SPLIT_CAP slots; vertices that
    // overflow them are redone with tables sized to their exact key bound
    // Both passes run over chunks of vertices whose tables fit in a pool of
    // max(64 MiB, 4 bytes per pin of the level), so the scratch of this tier
    // stays bounded whatever the degree distribution; chunks are cut from
    // the vertices' actual table sizes.
    int32_t* again;
    int64_t* nagain;
    SNN_TRY(ar.alloc(&again, ns));
    SNN_TRY(ar.alloc(&nagain, 1));
    SNN_CUDA(cudaMemsetAsync(nagain, 0, sizeof(int64_t), s));
    const int64_t pool_slots =
        std::max<int64_t>((int64_t)64 << 20, 4 * pol.L.P) / (int64_t)slot_bytes<S>();
    std::vector<int64_t> cuts;
    SNN_TRY(split_cuts(pol, ar, s, sl, ns, workv, HT_SPLIT_CAP, pool_slots, cuts));
    h_cnt[0] = 0;
    for (size_t c = 0; c + 1 < cuts.size(); c++) {
        Arena::Mark m = ar.mark();
        SNN_TRY(run_split(pol, ar, s, sl + cuts[c], cuts[c + 1] - cuts[c], workv, HT_SPLIT_CAP,
                          again, nagain, h_cnt));
        ar.rewind(m);
    }
    int64_t n2 = h_cnt[0];
    if (n2 == 0) return Status{};
    SNN_TRY(split_cuts(pol, ar, s, again, n2, workv, 0, pool_slots, cuts));
    for (size_t c = 0; c + 1 < cuts.size(); c++) {
        Arena::Mark m = ar.mark();
        SNN_TRY(run_split(pol, ar, s, again + cuts[c], cuts[c + 1] - cuts[c], workv, 0, nullptr,
                          nullptr, h_cnt));
        ar.rewind(m);
    }
    return Status{};
}

}  // namespace snn
