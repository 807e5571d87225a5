// Uncoarsening and refinement (Sec. 4.1).
//
// Projection: rho_l(n) = rho_{l+1}(cid(n)).
//
// One refinement round:
//  S6  pins(p, e): per hyperedge, the sorted keys rho(q)*2 + [q is a
//      destination] are run-length encoded into (p, cnt, dcnt) entries;
//      e is inbound to p iff dcnt > 0. Partition state: size, inbound pins,
//      and distinct inbound axons (internal axons + k of inbound hyperedges).
//      Conn = sum omega(e) (lambda(e) - 1) comes out of the same pass.
//  S7  per vertex: save = omega of incident hyperedges where it is its
//      partition's last pin; for every other adjacent partition p the
//      connection weight conn(p) (loss = W - conn) and the k of hyperedges
//      where it is a destination and that are already inbound to p; gain =
//      save - loss; the best feasible move (ties to the lower p) is proposed
//      if its gain is positive.
//  S8  moves sorted by decreasing gain, ties by vertex id (stable radix sort
//      of compacted proposals, which are in vertex order).
//  S9  per hyperedge, its moved pins are replayed in move order: each
//      move's gain contribution omega([cnt(from)=1] - [cnt(to)=0]) is taken
//      with every earlier move applied, and when a destination leaves the
//      last / enters the first destination slot of a partition an inbound
//      event (p, move, -/+k) is emitted. Prefix sums give each prefix's gain.
//  S10 validity: per partition, its events (size/pins of every move, inbound
//      events) sorted by move and scanned; after each move that touches the
//      partition its limits are checked and changes of "violating" are added
//      to the move's violation delta. A prefix is valid iff the prefix sum of
//      violation deltas is zero.
//  S11 the valid prefix with the largest positive gain (shortest on ties) is
//      enacted.
#include "histo.cuh"
#include "internal.cuh"
#include "row_items.cuh"
#include "scan.cuh"

#include <algorithm>
#include <climits>
#include <memory>

namespace snn {

enum : int {
    RS_BEST = SC_C,    // best valid prefix gain
    RS_ISTAR = SC_D,   // index of its last move
    RS_COST = SC_E,    // Conn at round start
    RS_NEV = SC_F,     // inbound events emitted
    RS_NHV = SC_G,     // hyperedges replayed by the block tier
    RS_NHL = 11,       // listed hyperedges (int32)
};

// pinned host words the kernels of a round write (snnmap_hgraph::h_tier)
enum : int { HW_COST = 0, HW_BAD, HW_PROPS, HW_STATUS = HW_PROPS + 3, HW_BEST, HW_ISTAR };

constexpr int REPLAY_WARP_MAX = 32;
constexpr int PSTAR_MAX = 16;   // partitions of P* the column update takes

struct PinCounts {
    int32_t* p;
    int32_t* cnt;
    int32_t* dcnt;
    int32_t* lam;
    HRec* rec;     // per hyperedge: first entry, omega, k, lam and masks of its first 32 entries
};

struct PState {
    int64_t* size;
    int64_t* inpins;
    int64_t* pincnt;
};

// ---------------------------------------------------------------------------
// S5

__global__ void k_project(int32_t V, const int32_t* __restrict__ cid,
                          const int32_t* __restrict__ rc, int32_t* rf)
{
    after_previous();
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < V;
         n += (int64_t)gridDim.x * blockDim.x)
        rf[n] = rc[cid[n]];
}

Status project(snnmap_hgraph* h, int32_t level, const int32_t* rho_coarse, int32_t* rho_fine)
{
    Level& L = h->levels[level];
    if (L.V > 0) {
        enqueue(k_project, grid_for(L.V, 256), 256, 0, h->stream, L.V, L.cid, rho_coarse, rho_fine);
        SNN_CUDA(cudaGetLastError());
    }
    return Status{};
}

// ---------------------------------------------------------------------------
// S6

// Conn is summed into COST_SLOTS partial sums (hyperedge id modulo) rather
// than one word, so the per-hyperedge atomics do not all meet on one address
constexpr int COST_SLOTS = 256;

__global__ void k_cost_slots(const int64_t* __restrict__ slots, int64_t* out)
{
    after_previous();
    int64_t v = 0;
    for (int i = threadIdx.x; i < COST_SLOTS; i += blockDim.x) v += slots[i];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd((unsigned long long*)out, (unsigned long long)v);
}

// most partitions whose inbound sums a block keeps in shared memory (32 KB)
constexpr int32_t PC_SMEM_K = 8192;

struct PinCountJob {
    const int64_t* hoff;
    const int32_t* hpins;
    const uint8_t* hsd;
    const int32_t* hk;
    const int64_t* hw;
    const int32_t* rho;
    PinCounts pc;
    int64_t* pincnt;
    int64_t* cost;     // partial sums of Conn, by hyperedge id & cost_mask
    // inbound axons per partition summed per block first (a sum never passes
    // the number of input hyperedges, so 32 bits hold it): a level adds one
    // term per partition a hyperedge reaches, all on the K words of pincnt.
    // 45,039 hyperedges on 111 partitions: 67 us a level without.
    static constexpr bool kShared = true;
    int32_t K = 0;     // words kept per block; 0: add to pincnt directly
    int32_t cost_mask = COST_SLOTS - 1;
    uint32_t* acc = nullptr;
    static constexpr int kSharedWords = PC_SMEM_K;
    __host__ __device__ int shared_words() const { return K; }
    __device__ void attach(uint32_t* w) { acc = K > 0 ? w : nullptr; }
    __device__ void flush() const
    {
        for (int32_t p = threadIdx.x; p < K; p += blockDim.x)
            if (acc[p]) atomicAdd((unsigned long long*)&pincnt[p], (unsigned long long)acc[p]);
    }
    __device__ __forceinline__ void add_inbound(int32_t p, int32_t k) const
    {
        if (acc) atomicAdd(&acc[p], (uint32_t)k);
        else atomicAdd((unsigned long long*)&pincnt[p], (unsigned long long)k);
    }
    __device__ int len(int32_t a) const { return (int)(hoff[a + 1] - hoff[a]); }
    __device__ uint32_t load(int32_t a, int i) const
    {
        int64_t j = hoff[a] + i;
        uint32_t d = (i > 0 || hsd[a]) ? 1u : 0u;
        return ((uint32_t)rho[hpins[j]] << 1) | d;
    }
    __device__ void finish(int32_t a, const uint32_t* s, int n) const
    {
        int lane = threadIdx.x & 31;
        int64_t base = hoff[a];
        unsigned le = lanemask_lt() | (1u << lane);
        int R = 0;
        // pass 1: run starts (partition changes) and first destination of each run
        for (int c = 0; c < n; c += 32) {
            int i = c + lane;
            bool valid = i < n;
            uint32_t v = valid ? s[i] : KEY_PAD;
            uint32_t pv = (valid && i > 0) ? s[i - 1] : KEY_PAD;
            bool rs = valid && (i == 0 || (v >> 1) != (pv >> 1));
            bool ds = valid && (v & 1) && (i == 0 || v != pv);
            unsigned mr = __ballot_sync(FULL, rs);
            int r = R + __popc(mr & le) - 1;
            if (rs) {
                pc.p[base + r] = (int32_t)(v >> 1);
                pc.cnt[base + r] = i;
                pc.dcnt[base + r] = -1;
            }
            __syncwarp();
            if (ds) pc.dcnt[base + r] = i;
            __syncwarp();
            R += __popc(mr);
        }
        // pass 2: starts -> counts
        uint32_t dm = 0, sm = 0;
        for (int c = 0; c < R; c += 32) {
            int r = c + lane;
            int st = 0, nx = 0, dsx = -1;
            if (r < R) {
                st = pc.cnt[base + r];
                nx = (r + 1 < R) ? pc.cnt[base + r + 1] : n;
                dsx = pc.dcnt[base + r];
            }
            __syncwarp();
            int dc = r < R && dsx >= 0 ? nx - dsx : 0;
            if (r < R) {
                pc.cnt[base + r] = nx - st;
                pc.dcnt[base + r] = dc;
                if (dc > 0) add_inbound(pc.p[base + r], hk[a]);
            }
            unsigned md = __ballot_sync(FULL, dc > 0), ms = __ballot_sync(FULL, r < R && nx - st == 1);
            if (c == 0) {
                dm = md;
                sm = ms;
            }
        }
        if (lane == 0) {
            pc.lam[a] = R;
            pc.rec[a] = HRec{base, hw[a], (uint32_t)hk[a], (uint32_t)R | (uint32_t)hsd[a] << 31, dm, sm};
            if (R > 1) atomicAdd((unsigned long long*)&cost[a & cost_mask], (unsigned long long)(hw[a] * (R - 1)));
        }
    }
    __device__ void finish_thread(int32_t a, const uint32_t* s, int n, int st) const
    {
        int64_t base = hoff[a];
        uint32_t dm = 0, sm = 0;   // at most SEG_T_CAP runs
        int R = 0, c = 0, d = 0;
        for (int i = 0; i < n; i++) {
            uint32_t p = s[(i) * st] >> 1;
            if (i > 0 && p != (s[(i - 1) * st] >> 1)) {
                pc.p[base + R] = (int32_t)(s[(i - 1) * st] >> 1);
                pc.cnt[base + R] = c;
                pc.dcnt[base + R] = d;
                if (d > 0) add_inbound((int32_t)(s[(i - 1) * st] >> 1), hk[a]);
                dm |= (uint32_t)(d > 0) << R;
                sm |= (uint32_t)(c == 1) << R;
                R++;
                c = 0;
                d = 0;
            }
            c++;
            d += (int)(s[(i) * st] & 1);
        }
        if (n > 0) {
            pc.p[base + R] = (int32_t)(s[(n - 1) * st] >> 1);
            pc.cnt[base + R] = c;
            pc.dcnt[base + R] = d;
            if (d > 0) add_inbound((int32_t)(s[(n - 1) * st] >> 1), hk[a]);
            dm |= (uint32_t)(d > 0) << R;
            sm |= (uint32_t)(c == 1) << R;
            R++;
        }
        pc.lam[a] = R;
        pc.rec[a] = HRec{base, hw[a], (uint32_t)hk[a], (uint32_t)R | (uint32_t)hsd[a] << 31, dm, sm};
        if (R > 1) atomicAdd((unsigned long long*)&cost[a & cost_mask], (unsigned long long)(hw[a] * (R - 1)));
    }
};

__global__ void k_pstate_vertices(Level L, const int32_t* __restrict__ rho, PState ps)
{
    after_previous();
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < L.V;
         n += (int64_t)gridDim.x * blockDim.x) {
        int32_t p = rho[n];
        atomicAdd((unsigned long long*)&ps.size[p], (unsigned long long)L.vsize[n]);
        atomicAdd((unsigned long long*)&ps.inpins[p], (unsigned long long)L.vinpins[n]);
        if (L.vinint[n]) atomicAdd((unsigned long long*)&ps.pincnt[p], (unsigned long long)L.vinint[n]);
    }
}

__device__ __forceinline__ bool violates(int64_t sz, int64_t ip, int64_t pc, int32_t omega,
                                         int32_t delta, int32_t phi)
{
    return sz > omega || ip > phi || pc > delta;
}

// counts of partition p in hyperedge a at round start (entries sorted by p)
__device__ __forceinline__ void lookup_count(const PinCounts& pc, int64_t b, int32_t lam, int32_t p,
                                             int32_t& cnt, int32_t& dcnt)
{
    int32_t lo = 0, hi = lam;
    while (lo < hi) {
        int32_t mid = (lo + hi) >> 1;
        if (pc.p[b + mid] < p) lo = mid + 1;
        else hi = mid;
    }
    if (lo < lam && pc.p[b + lo] == p) {
        cnt = pc.cnt[b + lo];
        dcnt = pc.dcnt[b + lo];
    } else {
        cnt = 0;
        dcnt = 0;
    }
}

// save(n) = omega of incident hyperedges in which n is the last pin of its
// partition, W(n) = omega of all incident hyperedges. A move of n gains
// save(n) - W(n) + conn(n, p) <= save(n), so a vertex with save(n) = 0
// never proposes. A group of G lanes per hyperedge, lanes over its pins
// (both arrays cleared before).
template <int G>
__global__ void __launch_bounds__(256)
    k_save(Level L, PinCounts pc, const int32_t* __restrict__ rho, int64_t* savev, int64_t* Wv)
{
    after_previous();
    int lane = threadIdx.x & (G - 1);
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) / G;
    for (int64_t a = gw; a < L.E; a += nw) {
        int64_t b = L.hoff[a], e = L.hoff[a + 1];
        int32_t lam = pc.lam[a];
        unsigned long long w = (unsigned long long)L.hw[a];
        for (int64_t j = b + lane; j < e; j += G) {
            int32_t x = L.hpins[j];
            atomicAdd((unsigned long long*)&Wv[x], w);
            int32_t c, d;
            lookup_count(pc, b, lam, rho[x], c, d);
            if (c == 1) atomicAdd((unsigned long long*)&savev[x], w);
        }
    }
}

// The same with both sums kept per block in shared memory, for levels with
// few vertices: there a heavy super-node's two words take an atomic from most
// hyperedges. 32-bit sums (W and save are at most the summed omega).
constexpr int SAVE_SMEM_V = 24 * 1024;   // 192 KB
constexpr int SAVE_THREADS = 1024;

template <int G>
__global__ void __launch_bounds__(SAVE_THREADS)
    k_save_smem(Level L, PinCounts pc, const int32_t* __restrict__ rho, int64_t* savev, int64_t* Wv)
{
    after_previous();
    extern __shared__ uint32_t ssum[];   // W, then save
    uint32_t *sW = ssum, *sS = ssum + L.V;
    for (int32_t v = threadIdx.x; v < 2 * L.V; v += SAVE_THREADS) ssum[v] = 0;
    __syncthreads();
    int lane = threadIdx.x & (G - 1);
    int64_t a1 = (int64_t)L.E * (blockIdx.x + 1) / gridDim.x;
    for (int64_t a = (int64_t)L.E * blockIdx.x / gridDim.x + threadIdx.x / G; a < a1;
         a += SAVE_THREADS / G) {
        int64_t b = L.hoff[a], e = L.hoff[a + 1];
        int32_t lam = pc.lam[a];
        uint32_t w = (uint32_t)L.hw[a];
        for (int64_t j = b + lane; j < e; j += G) {
            int32_t x = L.hpins[j];
            atomicAdd(&sW[x], w);
            int32_t c, d;
            lookup_count(pc, b, lam, rho[x], c, d);
            if (c == 1) atomicAdd(&sS[x], w);
        }
    }
    __syncthreads();
    for (int32_t v = threadIdx.x; v < L.V; v += SAVE_THREADS) {
        if (sW[v]) atomicAdd((unsigned long long*)&Wv[v], (unsigned long long)sW[v]);
        if (sS[v]) atomicAdd((unsigned long long*)&savev[v], (unsigned long long)sS[v]);
    }
}

// ---------------------------------------------------------------------------
// S7: partition connection histogram per vertex

template <typename S_>
struct GainPol {
    using S = S_;
    // a vertex meets few partitions even when its bound is large
    static constexpr bool kOptimistic = true;
    static constexpr bool kMasks = true;
    struct Acc {
        int64_t W, save;   // summed omega of incident hyperedges; of those n is the last pin of
        __device__ Acc() : W(0), save(0) {}
        __device__ void add(const Acc& o)
        {
            W += o.W;
            save += o.save;
        }
        __device__ void atomic_into(Acc* g) const
        {
            if (W) atomicAdd((unsigned long long*)&g->W, (unsigned long long)W);
            if (save) atomicAdd((unsigned long long*)&g->save, (unsigned long long)save);
        }
    };
    static __device__ Acc warp_reduce(const Acc& a)
    {
        Acc r;
        r.W = warp_sum(a.W);
        r.save = warp_sum(a.save);
        return r;
    }

    Level L;
    PinCounts pc;
    PState ps;
    const int32_t* rho;
    int32_t V;
    int64_t keys;
    int32_t omega, delta, phi;
    int32_t* pto;
    int64_t* pgain;
    const int64_t* savev;
    const int32_t* dirty;   // vertices to evaluate; the others keep pto/pgain
    bool nonpos;            // propose the best feasible move whatever its gain

    __device__ bool skip(int32_t n) const { return (!nonpos && savev[n] == 0) || !dirty[n]; }
    __device__ int64_t vb(int32_t n) const { return L.voff[n]; }
    __device__ int64_t ve(int32_t n) const { return L.voff[n + 1]; }
    __device__ int64_t seg_len(int64_t i) const
    {
        return pc.lam[(int32_t)((uint32_t)L.vinc[i] & ~SRC_BIT)];
    }
    __device__ uint32_t inc(int64_t i) const { return (uint32_t)L.vinc[i]; }
    __device__ void fetch(uint32_t inc) const { prefetch_l1(pc.rec + (inc & ~SRC_BIT)); }
    __device__ Seg<S> seg(uint32_t inc, Acc& acc) const
    {
        HRec r = pc.rec[(int32_t)(inc & ~SRC_BIT)];
        acc.W += r.w;
        return rec_seg<S>(r, inc);
    }
    // one element: partition p (-1: nothing to add, -2: weight w to save)
    struct Item {
        int32_t p;
        S w;
        uint32_t o;
    };
    static __device__ Item none() { return Item{-1, 0, 0u}; }
    struct Own {
        int32_t part, size, inpins;
    };
    __device__ Own own(int32_t n) const { return Own{rho[n], L.vsize[n], L.vinpins[n]}; }
    __device__ Item load(int32_t, const Own& o, const Seg<S>& g, int32_t off) const
    {
        int64_t e = g.b + off;
        int32_t p = pc.p[e];
        if (p == o.part) {
            bool one = off < 32 ? (g.sm >> off) & 1 : pc.cnt[e] == 1;
            return Item{one ? -2 : -1, g.w, 0u};
        }
        // a partition that cannot take n by size or inbound pins is never
        // the chosen move: leave it out of the table
        if (ps.size[p] + o.size > omega || ps.inpins[p] + o.inpins > phi) return none();
        bool in = off < 32 ? (g.dm >> off) & 1 : pc.dcnt[e] > 0;
        return Item{p, g.w, (g.nd && in) ? g.k : 0u};
    }
    template <class Tb>
    __device__ bool put(int32_t, const Item& it, const Tb& t, Acc& acc) const
    {
        if (it.p >= 0) return t.add(it.p, it.w, it.o);
        if (it.p == -2) acc.save += (int64_t)it.w;
        return true;
    }
    // gain = save - loss with loss = W - conn(p); feasible if p stays within
    // Omega, Phi, and Delta on its inbound set grown by n's axons not yet
    // inbound to p
    __device__ void consider(int32_t n, int32_t p, int64_t conn, uint32_t o, const Acc& tot,
                             int64_t& bs, int32_t& bk, uint32_t& bo) const
    {
        int64_t gain = tot.save - tot.W + conn;
        bool feas = ps.size[p] + L.vsize[n] <= omega && ps.inpins[p] + L.vinpins[n] <= phi &&
                    ps.pincnt[p] + L.vincnt[n] - (int64_t)o <= delta;
        if (feas && better(gain, p, bs, bk)) {
            bs = gain;
            bk = p;
            bo = o;
        }
    }
    __device__ void write(int32_t n, int64_t bs, int32_t bk, uint32_t, const Acc&) const
    {
        if (!dirty[n]) return;
        bool prop = bk >= 0 && (bs > 0 || nonpos);
        pto[n] = prop ? bk : -1;
        pgain[n] = prop ? bs : 0;
    }
};

struct Moves {
    int32_t* n;
    int32_t* from;
    int32_t* to;
};

// Hyperedges holding a proposed move (k_prop_hedges builds the list): a
// round's replay, row updates, re-evaluation flags and pin-count updates
// iterate it instead of every hyperedge of the level.
struct HedgeList {
    const int32_t* a;   // hyperedge ids
    const int32_t* n;   // their number (device)
};

// ---------------------------------------------------------------------------
// Connection rows (refinement levels whose rows fit the memory budget)
//
// Row r of vertex n (r = rowid[n]) holds, for every partition p,
// C[r][p] = conn(n, p) = sum of omega(e) over incident e with cnt(p, e) > 0,
// and O[r][p] = sum of k(e) over e in which n is a destination and
// dcnt(p, e) > 0. A round then needs no histogram: the best move of n is a
// scan of its row against the partition state. Rows change only when a
// partition's count in a hyperedge crosses zero, which applied moves report
// (rows_cross). Projection to the next finer level leaves the rows of
// unmatched vertices exact (their hyperedges map one to one onto hyperedges
// of the same omega, k, destination role and partition set); the two
// members of each contracted pair get fresh rows (RowPol).

template <typename S_>
struct RowPol {
    using S = S_;
    // a row holds every adjacent partition: warp tables would overflow
    static constexpr bool kOptimistic = false;
    static constexpr bool kMasks = true;
    struct Acc {
        __device__ Acc() {}
        __device__ void add(const Acc&) {}
        __device__ void atomic_into(Acc*) const {}
    };
    static __device__ Acc warp_reduce(const Acc& a) { return a; }

    Level L;
    PinCounts pc;
    int32_t V;
    int64_t keys;
    const int32_t* fresh;
    const int32_t* rowid;
    RowTab tab;
    unsigned long long* M;
    int32_t cw;

    __device__ bool skip(int32_t n) const { return fresh[n] == 0; }
    __device__ int64_t vb(int32_t n) const { return L.voff[n]; }
    __device__ int64_t ve(int32_t n) const { return L.voff[n + 1]; }
    __device__ int64_t seg_len(int64_t i) const
    {
        return pc.lam[(int32_t)((uint32_t)L.vinc[i] & ~SRC_BIT)];
    }
    __device__ uint32_t inc(int64_t i) const { return (uint32_t)L.vinc[i]; }
    __device__ void fetch(uint32_t inc) const { prefetch_l1(pc.rec + (inc & ~SRC_BIT)); }
    __device__ Seg<S> seg(uint32_t inc, Acc&) const
    {
        return rec_seg<S>(pc.rec[(int32_t)(inc & ~SRC_BIT)], inc);
    }
    struct Item {
        int32_t p;
        S w;
        uint32_t o;
    };
    static __device__ Item none() { return Item{-1, 0, 0u}; }
    struct Own {};
    __device__ Own own(int32_t) const { return Own{}; }
    __device__ Item load(int32_t, const Own&, const Seg<S>& g, int32_t off) const
    {
        int64_t e = g.b + off;
        bool in = off < 32 ? (g.dm >> off) & 1 : pc.dcnt[e] > 0;
        return Item{pc.p[e], g.w, (g.nd && in) ? g.k : 0u};
    }
    template <class Tb>
    __device__ bool put(int32_t, const Item& it, const Tb& t, Acc&) const
    {
        return it.p < 0 || t.add(it.p, it.w, it.o);
    }
    // every key of the finished histogram lands in the row (stores, so a
    // vertex redone by a later tier overwrites its partial entries)
    __device__ void consider(int32_t n, int32_t p, int64_t conn, uint32_t o, const Acc&, int64_t&,
                             int32_t&, uint32_t&) const
    {
        int32_t row = rowid[n];
        tab.C(row)[p] = (int32_t)conn;
        tab.O(row)[p] = (int32_t)o;
        unsigned long long bit = 1ull << (p / cw);
        if (!(M[row] & bit)) atomicOr(&M[row], bit);   // a set bit is never cleared here
    }
    __device__ void write(int32_t, int64_t, int32_t, uint32_t, const Acc&) const {}
};

// best move per vertex from its row: largest gain = C - (W - save) over
// partitions p != rho(n) that can take n, ties to the lower p; proposed if
// positive. Only the chunks of the row that the mask M marks are read (an
// entry outside them is 0, and a partition with conn 0 is never taken);
// each lane still visits its partitions in increasing order.
__global__ void __launch_bounds__(256)
    k_dense_best(Level L, const int32_t* __restrict__ rho, PState ps,
                 const int64_t* __restrict__ savev, const int64_t* __restrict__ Wv,
                 const int32_t* __restrict__ rowid, RowTab tab,
                 const unsigned long long* __restrict__ M, int32_t cw, int32_t K, int32_t omega,
                 int32_t delta, int32_t phi,
                 int nonpos, int32_t* pto, int64_t* pgain, const int32_t* __restrict__ dirty)
{
    after_previous();
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t n = gw; n < L.V; n += nw) {
        if (dirty && !dirty[n]) continue;   // proposal kept from the previous round
        int64_t sv = savev[n];
        if (sv == 0 && !nonpos) {
            if (lane == 0) {
                pto[n] = -1;
                pgain[n] = 0;
            }
            continue;
        }
        int64_t T = Wv[n] - sv;
        int32_t own = rho[n];
        int64_t sz = L.vsize[n], ip = L.vinpins[n], ic = L.vincnt[n];
        int32_t rw = rowid[n];
        const int4* row = reinterpret_cast<const int4*>(tab.C(rw));
        const int32_t* ov = tab.O(rw);
        int64_t bs = 0;
        int32_t bk = -1;
        const int64_t nq = ((int64_t)K + 3) >> 2;
        ChunkDeal deal(M[rw], cw, lane);   // two loads a lane at a time
        while (__any_sync(FULL, deal.left())) {
            constexpr int U = 2;
            int4 c4[U];
            int64_t qq[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                qq[u] = deal.next(nq);
                c4[u] = qq[u] < nq ? row[qq[u]] : make_int4(0, 0, 0, 0);
            }
#pragma unroll
            for (int v = 0; v < U; v++) {
                int cv[4] = {c4[v].x, c4[v].y, c4[v].z, c4[v].w};
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    int32_t p = (int32_t)(4 * qq[v] + u);
                    int64_t g = (int64_t)cv[u] - T;
                    // default: positive gains only (bs starts at 0); variant:
                    // any adjacent partition (conn > 0), the first one found
                    // seeds bs
                    if (p < K && (g > bs || (nonpos && bk < 0 && cv[u] > 0)) && cv[u] > 0 &&
                        p != own && ps.size[p] + sz <= omega && ps.inpins[p] + ip <= phi &&
                        ps.pincnt[p] + ic - (int64_t)ov[p] <= delta) {
                        bs = g;
                        bk = p;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            int64_t s2 = __shfl_xor_sync(FULL, bs, o);
            int32_t m2 = __shfl_xor_sync(FULL, bk, o);
            if (better(s2, m2, bs, bk)) {
                bs = s2;
                bk = m2;
            }
        }
        if (lane == 0) {
            pto[n] = bk;
            pgain[n] = bk >= 0 ? bs : 0;
        }
    }
}

struct RowsRef {
    const int32_t* rowid;   // null: the level has no rows
    RowTab tab;
    unsigned long long* M;
    int32_t cw;
};

// Row updates of hyperedge a for the enacted prefix (one warp): the moves of
// its pins with index <= i* (buf[b .. b + m)) give each touched partition's
// count after the prefix; where cnt(p, e) crosses zero every pin's C[.][p]
// changes by omega(e), and where dcnt(p, e) crosses zero every
// destination's O[.][p] by k(e).
__device__ __forceinline__ void rows_cross(const Level& L, const PinCounts& pc, const Moves& mv,
                                           const RowsRef& R, int32_t a, int64_t b, int64_t e, int sd,
                                           int32_t lam, int64_t w, int32_t k, const uint32_t* buf,
                                           int m)
{
    const int lane = threadIdx.x & 31;
    const int32_t* rowid = R.rowid;
    unsigned long long* M = R.M;
    const int32_t cw = R.cw;
    {
        for (int ib = 0; ib < m; ib += 32) {
            int ii = ib + lane;
            // up to two crossing records per lane: partition, C sign, O sign
            int32_t rp[2] = {-1, -1};
            int rc[2] = {0, 0}, rd[2] = {0, 0};
            if (ii < m) {
                int32_t mi = (int32_t)(buf[b + ii] >> 1);
                int32_t cand[2] = {mv.from[mi], mv.to[mi]};
                for (int u = 0; u < 2; u++) {
                    int32_t p = cand[u];
                    bool first = true;
                    int nc = 0, nd = 0;
                    for (int jj = 0; jj < m; jj++) {
                        uint32_t rj = buf[b + jj];
                        int32_t mj = (int32_t)(rj >> 1);
                        int32_t fj = mv.from[mj], tj = mv.to[mj];
                        if (jj < ii && (fj == p || tj == p)) first = false;
                        int dlt = (tj == p) - (fj == p);
                        nc += dlt;
                        if (rj & 1) nd += dlt;
                    }
                    if (!first) continue;
                    int32_t c0, d0;
                    lookup_count(pc, b, lam, p, c0, d0);
                    int cs = ((c0 + nc) > 0) - (c0 > 0);
                    int ds = ((d0 + nd) > 0) - (d0 > 0);
                    if (cs || ds) {
                        rp[u] = p;
                        rc[u] = cs;
                        rd[u] = ds;
                    }
                }
            }
            for (int u = 0; u < 2; u++) {
                unsigned has = __ballot_sync(FULL, rp[u] >= 0);
                while (has) {
                    int src = __ffs(has) - 1;
                    has &= has - 1;
                    int32_t p = __shfl_sync(FULL, rp[u], src);
                    int cs = __shfl_sync(FULL, rc[u], src);
                    int ds = __shfl_sync(FULL, rd[u], src);
                    for (int64_t j = b + lane; j < e; j += 32) {
                        int32_t rw = rowid[L.hpins[j]];
                        if (cs) atomicAdd(R.tab.C(rw) + p, (int32_t)(cs * w));
                        unsigned long long bit = 1ull << (p / cw);
                        if (cs > 0 && !(M[rw] & bit)) atomicOr(&M[rw], bit);
                        if (ds && (j != b || sd)) atomicAdd(R.tab.O(rw) + p, ds * k);
                    }
                }
            }
        }
    }
}

// descent to the next finer level: the lower member of a pair keeps its
// super-node's row, the upper one takes row Vc + (its rank among the upper
// ones); both are to be computed afresh
struct UpperMember {
    const uint8_t* pr;
    __device__ int32_t operator()(int64_t n) const { return pr[n] == 2; }
};
struct RowIds {
    const uint8_t* pr;
    const int32_t *cid, *rowc;
    int32_t Vc;
    int32_t *rowf, *fresh;
    __device__ void operator()(int64_t n, int32_t before, int32_t upper) const
    {
        rowf[n] = upper ? Vc + before : rowc[cid[n]];
        fresh[n] = pr[n] != 0;
    }
};

// clears the rows of vertices flagged fresh (one warp per vertex)
__global__ void k_dense_zero(int32_t V, const int32_t* __restrict__ fresh,
                             const int32_t* __restrict__ rowid, RowTab tab,
                             unsigned long long* M)
{
    after_previous();
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t n = gw; n < V; n += nw) {
        if (!fresh[n]) continue;
        if (lane == 0) M[rowid[n]] = 0;
        int4* c = reinterpret_cast<int4*>(tab.C(rowid[n]));
        int4* o = reinterpret_cast<int4*>(tab.O(rowid[n]));
        for (int64_t q = lane; q < tab.Kp / 4; q += 32) {
            c[q] = make_int4(0, 0, 0, 0);
            o[q] = make_int4(0, 0, 0, 0);
        }
    }
}

// ---------------------------------------------------------------------------
// Incremental rounds on histogram levels. After an enacted prefix, a
// vertex's best move can change only if (a) one of its hyperedges holds a
// moved pin (its conn, overlap and save change only there), (b) it is
// adjacent to a partition that lost load (a source of an enacted move) and
// was tight before -- a partition with room for the largest vertex of the
// level in all three limits was feasible for every vertex before and still
// is, and partitions that only gained load lose feasibility, which matters
// only for (c) -- or (c) its proposed target changed state. Every other
// vertex keeps its proposal, which a full evaluation would reproduce.

__global__ void k_level_max(Level L, int32_t* vmax)
{
    after_previous();
    int32_t a = 0, b = 0, c = 0;
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < L.V;
         n += (int64_t)gridDim.x * blockDim.x) {
        a = max(a, L.vsize[n]);
        b = max(b, L.vinpins[n]);
        c = max(c, L.vincnt[n]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a = max(a, __shfl_xor_sync(FULL, a, o));
        b = max(b, __shfl_xor_sync(FULL, b, o));
        c = max(c, __shfl_xor_sync(FULL, c, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&vmax[0], a);
        atomicMax(&vmax[1], b);
        atomicMax(&vmax[2], c);
    }
}

// partitions touched by the enacted prefix (pchg) and the tight sources
// among them (prel), with the round-start state
__global__ void k_inc_parts(int32_t M, Moves mv, const int64_t* __restrict__ scal, PState ps,
                            const int32_t* __restrict__ vmax, int32_t omega, int32_t delta,
                            int32_t phi, uint8_t* pchg, uint8_t* prel,
                            const int32_t* __restrict__ pstar_n)
{
    after_previous();
    if (*pstar_n <= PSTAR_MAX) return;   // the column update below handles this round
    int64_t istar = scal[RS_BEST] > 0 ? scal[RS_ISTAR] : -1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= istar && i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t f = mv.from[i], t = mv.to[i];
        pchg[f] = 1;
        pchg[t] = 1;
        if (ps.size[f] + vmax[0] > omega || ps.inpins[f] + vmax[1] > phi ||
            ps.pincnt[f] + vmax[2] > delta)
            prel[f] = 1;
    }
}

// (a) and (b). A hyperedge holding enacted moved pins changes the other
// pins' conn, overlap or save only where a partition's count or
// destination count crosses zero or its count moves between 1 and 2; then
// all its pins are marked, otherwise only the moved pins. A hyperedge
// holding a partition of prel (round-start pin counts) marks all its pins.
// One warp per hyperedge; buf (one word per pin) collects the moves.
__global__ void __launch_bounds__(256)
    k_inc_hedges(Level L, PinCounts pc, const int32_t* __restrict__ moveidx, Moves mv,
                 const int64_t* __restrict__ scal, const uint8_t* __restrict__ prel, uint32_t* buf,
                 int32_t* dirty, const int32_t* __restrict__ pstar_n)
{
    after_previous();
    if (*pstar_n <= PSTAR_MAX) return;
    int64_t istar = scal[RS_BEST] > 0 ? scal[RS_ISTAR] : -1;
    if (istar < 0) return;
    int lane = threadIdx.x & 31;
    unsigned lt = lanemask_lt();
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t a = gw; a < L.E; a += nw) {
        int64_t b = L.hoff[a], e = L.hoff[a + 1];
        int sd = L.hsd[a];
        int m = 0;
        for (int64_t cb = b; cb < e; cb += 32) {
            int64_t j = cb + lane;
            int32_t mi = -1;
            if (j < e) mi = moveidx[L.hpins[j]];
            bool ap = mi >= 0 && mi <= istar;
            unsigned mk = __ballot_sync(FULL, ap);
            if (ap) buf[b + m + __popc(mk & lt)] = ((uint32_t)mi << 1) | ((j != b || sd) ? 1u : 0u);
            m += __popc(mk);
        }
        __syncwarp();
        int32_t lam = pc.lam[a];
        bool all = false;
        for (int32_t r = lane; r < lam && !all; r += 32)
            if (prel[pc.p[b + r]]) all = true;
        all = __any_sync(FULL, all);   // uniform before the warp-wide loop below
        for (int ib = 0; ib < m && !all; ib += 32) {
            int ii = ib + lane;
            if (ii < m) {
                int32_t mi = (int32_t)(buf[b + ii] >> 1);
                int32_t cand[2] = {mv.from[mi], mv.to[mi]};
                for (int u = 0; u < 2 && !all; u++) {
                    int32_t p = cand[u];
                    int nc = 0, nd = 0;
                    for (int jj = 0; jj < m; jj++) {
                        uint32_t rj = buf[b + jj];
                        int32_t mj = (int32_t)(rj >> 1);
                        int dlt = (mv.to[mj] == p) - (mv.from[mj] == p);
                        nc += dlt;
                        if (rj & 1) nd += dlt;
                    }
                    int32_t c0, d0;
                    lookup_count(pc, b, lam, p, c0, d0);
                    int c1 = c0 + nc, d1 = d0 + nd;
                    if ((c0 > 0) != (c1 > 0) || (d0 > 0) != (d1 > 0) || (c0 == 1) != (c1 == 1))
                        all = true;
                }
            }
            all = __any_sync(FULL, all);
        }
        all = __any_sync(FULL, all);
        if (all) {
            for (int64_t j = b + lane; j < e; j += 32) dirty[L.hpins[j]] = 1;
        } else {
            for (int ii = lane; ii < m; ii += 32) dirty[mv.n[buf[b + ii] >> 1]] = 1;
        }
    }
}

// (c)
__global__ void k_inc_targets(int32_t V, const int32_t* __restrict__ pto,
                              const uint8_t* __restrict__ pchg, int32_t* dirty,
                              const int32_t* __restrict__ pstar_n)
{
    after_previous();
    if (*pstar_n <= PSTAR_MAX) return;
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < V;
         n += (int64_t)gridDim.x * blockDim.x)
        if (pto[n] >= 0 && pchg[pto[n]]) dirty[n] = 1;
}


// ---------------------------------------------------------------------------
// Proposals after a short enacted prefix (at most PSTAR_MAX partitions
// touched). Moves change the state of their source and target partitions
// only (the set P*), and in every hyperedge only the counts of those
// partitions. For a vertex n that did not move, an option q outside P*
// therefore keeps conn(n, q), ov(n, q) and its feasibility, and its gain
// shifts by the change of save(n) alone; the previous best option outside
// P* stays the best outside P*. The options inside P* are recomputed from
// their columns conn(n, p), ov(n, p), summed over the hyperedges that hold
// a pin of p (found through p's members' incidence lists). n is evaluated
// in full (flagged for the next round's histogram) only if it moved, if its
// previous proposal targeted P*, or, when only positive gains are proposed,
// if it had no proposal and its save grew (its best option outside P* is
// then unknown). The other vertices get their exact proposal here.

struct PStar {
    int32_t* pslot = nullptr;   // [K] slot of a partition of P*; -1 none
    int32_t* slots = nullptr;   // [PSTAR_MAX] partition of each slot
    int32_t* cnt = nullptr;     // [0] distinct partitions of P*, [1] marked hyperedges,
                                // [2] value cnt[0] restarts from (> PSTAR_MAX: path off)
    uint32_t* hmask = nullptr;  // [E] slots whose partition has a pin in the hyperedge
    int32_t* hl = nullptr;      // [E] hyperedges with a nonzero mask
    int64_t* colc = nullptr;    // [PSTAR_MAX * V] conn(n, slot)
    int32_t* colo = nullptr;    // [PSTAR_MAX * V] ov(n, slot)
    uint32_t* vt = nullptr;     // [V] slots adjacent to n (some incident hyperedge has a pin there)
    int64_t* save0 = nullptr;   // [V] save at round start
};

__device__ __forceinline__ bool pstar_on(const int64_t* scal, const int32_t* cnt)
{
    return scal[RS_BEST] > 0 && cnt[0] <= PSTAR_MAX;
}

// P* from the enacted moves; the moved vertices are flagged for a full
// evaluation
__global__ void k_ps_slots(int32_t M, Moves mv, const int64_t* __restrict__ scal, PStar ps,
                           int32_t* dirty)
{
    after_previous();
    int64_t istar = scal[RS_BEST] > 0 ? scal[RS_ISTAR] : -1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= istar && i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        dirty[mv.n[i]] = 1;
        int32_t pp[2] = {mv.from[i], mv.to[i]};
        for (int u = 0; u < 2; u++) {
            int32_t p = pp[u];
            if (atomicCAS(&ps.pslot[p], -1, -2) != -1) continue;
            int32_t sl = atomicAdd(&ps.cnt[0], 1);
            if (sl < PSTAR_MAX) {
                ps.slots[sl] = p;
                ps.pslot[p] = sl;
            }
        }
    }
}

// every hyperedge incident to a member of a P* partition gets that slot's
// bit (warp over 32 consecutive vertices, then over each member's
// incidences)
__global__ void __launch_bounds__(256)
    k_ps_mark(Level L, const int32_t* __restrict__ rho, const int64_t* __restrict__ scal, PStar ps)
{
    after_previous();
    if (!pstar_on(scal, ps.cnt)) return;
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = gw * 32; base < L.V; base += nw * 32) {
        int64_t n = base + lane;
        int32_t sl = n < L.V ? ps.pslot[rho[n]] : -1;
        unsigned mem = __ballot_sync(FULL, sl >= 0);
        while (mem) {
            int src = __ffs(mem) - 1;
            mem &= mem - 1;
            int32_t m = (int32_t)__shfl_sync(FULL, (int32_t)n, src);
            uint32_t bit = 1u << __shfl_sync(FULL, sl, src);
            for (int64_t i = L.voff[m] + lane; i < L.voff[m + 1]; i += 32) {
                int32_t a = (int32_t)((uint32_t)L.vinc[i] & ~SRC_BIT);
                uint32_t old = atomicOr(&ps.hmask[a], bit);
                if (old == 0) ps.hl[atomicAdd(&ps.cnt[1], 1)] = a;
            }
        }
    }
}

// The same from the pin counts: every hyperedge looks its partitions up in the
// slot map. A heavy super-node of a P* partition is in most hyperedges, and
// one warp walking its incidence list took 60 to 170 us a round on tail
// levels; this reads one word per (hyperedge, partition) of the level, so it
// takes the levels of up to PS_MARK_PINS pins.
constexpr int64_t PS_MARK_PINS = 16 << 20;

template <int G>
__global__ void __launch_bounds__(256)
    k_ps_mark_counts(Level L, PinCounts pc, const int64_t* __restrict__ scal, PStar ps)
{
    after_previous();
    if (!pstar_on(scal, ps.cnt)) return;
    const int lane = threadIdx.x & (G - 1);
    const unsigned gmask = (G == 32 ? FULL : ((1u << (G & 31)) - 1)) << ((threadIdx.x & 31) & ~(G - 1));
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) / G;
    for (int64_t a = gw; a < L.E; a += nw) {
        int64_t b = L.hoff[a];
        int32_t lam = pc.lam[a];
        uint32_t m = 0;
        for (int32_t r = lane; r < lam; r += G) {
            int32_t sl = ps.pslot[pc.p[b + r]];
            if (sl >= 0) m |= 1u << sl;
        }
        m = __reduce_or_sync(gmask, m);
        if (lane == 0 && m) {
            ps.hmask[a] = m;
            ps.hl[atomicAdd(&ps.cnt[1], 1)] = (int32_t)a;
        }
    }
}

// columns: for each marked hyperedge and each of its slots p, every pin n
// outside p adds omega to conn(n, p) and, as a destination of a hyperedge
// inbound to p, k to ov(n, p) (counts after the moves); masks are cleared
__global__ void __launch_bounds__(256)
    k_ps_cols(Level L, PinCounts pc, const int32_t* __restrict__ rho,
              const int64_t* __restrict__ scal, PStar ps)
{
    after_previous();
    if (!pstar_on(scal, ps.cnt)) return;
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t nh = ps.cnt[1];
    int64_t V = L.V;
    for (int64_t idx = gw; idx < nh; idx += nw) {
        int32_t a = ps.hl[idx];
        uint32_t mask = ps.hmask[a];
        int64_t b = L.hoff[a], e = L.hoff[a + 1];
        int32_t lam = pc.lam[a];
        int64_t w = L.hw[a];
        int32_t k = L.hk[a];
        int sd = L.hsd[a];
        while (mask) {
            int sl = __ffs(mask) - 1;
            mask &= mask - 1;
            int32_t p = ps.slots[sl];
            int32_t c, d;
            lookup_count(pc, b, lam, p, c, d);
            int64_t* cc = ps.colc + (int64_t)sl * V;
            int32_t* co = ps.colo + (int64_t)sl * V;
            for (int64_t j = b + lane; j < e; j += 32) {
                int32_t n = L.hpins[j];
                if (rho[n] == p) continue;
                atomicAdd((unsigned long long*)&cc[n], (unsigned long long)w);
                if (d > 0 && (j != b || sd)) atomicAdd(&co[n], k);
                atomicOr(&ps.vt[n], 1u << sl);
            }
        }
        __syncwarp();
        if (lane == 0) ps.hmask[a] = 0;
    }
}

// each vertex's proposal for the next round (or its flag for a full
// evaluation); columns read are cleared
__global__ void k_ps_combine(Level L, const int32_t* __restrict__ rho,
                             const int64_t* __restrict__ scal, PStar ps, PState st,
                             const int64_t* __restrict__ savev, const int64_t* __restrict__ Wv,
                             int32_t omega, int32_t delta, int32_t phi, int nonpos, int32_t* pto,
                             int64_t* pgain, int32_t* dirty)
{
    after_previous();
    if (!pstar_on(scal, ps.cnt)) return;
    int32_t ns = ps.cnt[0];
    int64_t V = L.V;
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < V;
         n += (int64_t)gridDim.x * blockDim.x) {
        uint32_t adj = ps.vt[n];
        if (!dirty[n]) {
            int64_t ds = savev[n] - ps.save0[n];
            int32_t q = pto[n];
            if ((q >= 0 && ps.pslot[q] >= 0) || (!nonpos && q < 0 && ds > 0)) {
                dirty[n] = 1;
            } else {
                int64_t bs = q >= 0 ? pgain[n] + ds : 0;
                int32_t bk = q;
                if (adj) {
                    int64_t sw = savev[n] - Wv[n];
                    for (int sl = 0; sl < ns; sl++) {
                        if (!((adj >> sl) & 1u)) continue;
                        int32_t p = ps.slots[sl];
                        int64_t c = ps.colc[(int64_t)sl * V + n];
                        int64_t o = ps.colo[(int64_t)sl * V + n];
                        bool feas = st.size[p] + L.vsize[n] <= omega &&
                                    st.inpins[p] + L.vinpins[n] <= phi &&
                                    st.pincnt[p] + L.vincnt[n] - o <= delta;
                        if (feas && better(sw + c, p, bs, bk)) {
                            bs = sw + c;
                            bk = p;
                        }
                    }
                }
                bool prop = bk >= 0 && (bs > 0 || nonpos);
                pto[n] = prop ? bk : -1;
                pgain[n] = prop ? bs : 0;
            }
        }
        if (adj) {
            for (int sl = 0; sl < ns; sl++) {
                if (!((adj >> sl) & 1u)) continue;
                ps.colc[(int64_t)sl * V + n] = 0;
                ps.colo[(int64_t)sl * V + n] = 0;
            }
            ps.vt[n] = 0;
        }
    }
}

// The same update on levels refined from connection rows: a vertex's
// columns of P* are entries of its row (already updated by k_prefix_hedges;
// adjacency is a positive entry there, rows being used only when every
// omega is positive). With more than PSTAR_MAX partitions in P*, every
// vertex is flagged for a row scan.
__global__ void k_ps_rows(Level L, const int32_t* __restrict__ rho,
                          const int64_t* __restrict__ scal, PStar ps, PState st,
                          const int64_t* __restrict__ savev, const int64_t* __restrict__ Wv,
                          const int32_t* __restrict__ rowid, RowTab tab, int32_t omega,
                          int32_t delta, int32_t phi, int nonpos, int32_t* pto, int64_t* pgain,
                          int32_t* dirty)
{
    after_previous();
    if (scal[RS_BEST] <= 0) return;
    bool on = ps.cnt[0] <= PSTAR_MAX;
    int32_t ns = on ? ps.cnt[0] : 0;
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < L.V;
         n += (int64_t)gridDim.x * blockDim.x) {
        if (!on) {
            dirty[n] = 1;
            continue;
        }
        if (dirty[n]) continue;   // moved
        int64_t ds = savev[n] - ps.save0[n];
        int32_t q = pto[n];
        if ((q >= 0 && ps.pslot[q] >= 0) || (!nonpos && q < 0 && ds > 0)) {
            dirty[n] = 1;
            continue;
        }
        int64_t bs = q >= 0 ? pgain[n] + ds : 0;
        int32_t bk = q;
        const int32_t *C = tab.C(rowid[n]), *O = tab.O(rowid[n]);
        int64_t sw = savev[n] - Wv[n];
        int32_t own = rho[n];
        for (int sl = 0; sl < ns; sl++) {
            int32_t p = ps.slots[sl];
            int64_t c = C[p];
            if (p == own || c <= 0) continue;
            bool feas = st.size[p] + L.vsize[n] <= omega && st.inpins[p] + L.vinpins[n] <= phi &&
                        st.pincnt[p] + L.vincnt[n] - (int64_t)O[p] <= delta;
            if (feas && better(sw + c, p, bs, bk)) {
                bs = sw + c;
                bk = p;
            }
        }
        bool prop = bk >= 0 && (bs > 0 || nonpos);
        pto[n] = prop ? bk : -1;
        pgain[n] = prop ? bs : 0;
    }
}

// slot map and counters back to empty; the round's result to the host's words
__global__ void k_ps_reset(int32_t M, Moves mv, const int64_t* __restrict__ scal, PStar ps,
                           int64_t* host)
{
    after_previous();
    int64_t istar = scal[RS_BEST] > 0 ? scal[RS_ISTAR] : -1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= istar && i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        ps.pslot[mv.from[i]] = -1;
        ps.pslot[mv.to[i]] = -1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ps.cnt[0] = ps.cnt[2];
        ps.cnt[1] = 0;
        host[HW_STATUS] = scal[SC_STATUS];
        host[HW_BEST] = scal[RS_BEST];
        host[HW_ISTAR] = scal[RS_ISTAR];
    }
}

// ---------------------------------------------------------------------------
// S8

// (proposals, their incidences, vertices evaluated) before each vertex: one
// scan compacts the proposals in vertex order, keyed by bias - gain (gains
// lie within the summed omega, so no pass is needed to find their range),
// and counts what the round's buffers need
struct PropSums {
    int64_t m, deg, act;
    __host__ __device__ PropSums() : m(0), deg(0), act(0) {}
    __device__ PropSums(int64_t a, int64_t b, int64_t c) : m(a), deg(b), act(c) {}
    __device__ PropSums operator+(const PropSums& o) const
    {
        return PropSums(m + o.m, deg + o.deg, act + o.act);
    }
};
__device__ __forceinline__ PropSums scan_shfl_up(PropSums v, int o)
{
    return PropSums(__shfl_up_sync(FULL, v.m, o), __shfl_up_sync(FULL, v.deg, o),
                    __shfl_up_sync(FULL, v.act, o));
}
__device__ __forceinline__ PropSums scan_shfl(PropSums v, int src)
{
    return PropSums(__shfl_sync(FULL, v.m, src), __shfl_sync(FULL, v.deg, src),
                    __shfl_sync(FULL, v.act, src));
}
struct PropIn {
    const int32_t* pto;
    const int64_t* savev;
    const int32_t* dirty;
    const int64_t* voff;
    int nonpos;
    __device__ PropSums operator()(int64_t n) const
    {
        bool f = pto[n] >= 0;
        return PropSums(f, f ? voff[n + 1] - voff[n] : 0,
                        (nonpos || savev[n] > 0) && (!dirty || dirty[n]));
    }
};
struct PropOut {
    const int64_t* pgain;
    int64_t bias;
    uint64_t* keys;
    uint32_t* vals;
    __device__ void operator()(int64_t n, PropSums ex, PropSums v) const
    {
        if (!v.m) return;
        keys[ex.m] = (uint64_t)(bias - pgain[n]);
        vals[ex.m] = (uint32_t)n;
    }
};

// ---------------------------------------------------------------------------
// The list of hyperedges holding a proposed move, from the proposers'
// incidence lists.

__global__ void __launch_bounds__(256)
    k_prop_hedges(int32_t M, Moves mv, Level L, int32_t* hmark, int32_t* list, int32_t* n)
{
    after_previous();
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = gw; i < M; i += nw) {
        int32_t v = mv.n[i];
        for (int64_t j = L.voff[v] + lane; j < L.voff[v + 1]; j += 32) {
            int32_t a = (int32_t)((uint32_t)L.vinc[j] & ~SRC_BIT);
            if (atomicExch(&hmark[a], 1) == 0) list[atomicAdd(n, 1)] = a;
        }
    }
}

// ---------------------------------------------------------------------------
// S9 / S10 events

struct Events {
    uint64_t* key;   // partition << ibits | move
    uint32_t* idx;   // 0..n-1 (sort values)
    int32_t* dsize;
    int32_t* dinp;
    int32_t* dpc;
    int64_t cap;
    int ibits;
};

// the sorted moves: their arrays, cleared gains and violation changes, and
// their size and inbound-pin events; and what the rounds keep per vertex (no
// vertex flagged, the saves before the moves)
__global__ void k_moves(int32_t M, const uint32_t* __restrict__ vals, const int32_t* __restrict__ rho,
                        const int32_t* __restrict__ pto, Moves mv, int32_t* moveidx, Level L,
                        Events ev, int64_t* gp, int32_t* dv, int32_t* dirty,
                        const int64_t* __restrict__ savev, int64_t* save0)
{
    after_previous();
    const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t n = t0; n < L.V; n += step) {
        dirty[n] = 0;
        if (save0) save0[n] = savev[n];
    }
    for (int64_t i = t0; i < M; i += step) {
        int32_t n = (int32_t)vals[i];
        int32_t f = rho[n], t = pto[n];
        mv.n[i] = n;
        mv.from[i] = f;
        mv.to[i] = t;
        moveidx[n] = (int32_t)i;
        gp[i] = 0;
        dv[i] = 0;
        int64_t e0 = 2 * i, e1 = 2 * i + 1;
        ev.key[e0] = ((uint64_t)f << ev.ibits) | (uint64_t)i;
        ev.key[e1] = ((uint64_t)t << ev.ibits) | (uint64_t)i;
        ev.idx[e0] = (uint32_t)e0;
        ev.idx[e1] = (uint32_t)e1;
        ev.dsize[e0] = -L.vsize[n];
        ev.dsize[e1] = L.vsize[n];
        ev.dinp[e0] = -L.vinpins[n];
        ev.dinp[e1] = L.vinpins[n];
        ev.dpc[e0] = -L.vinint[n];
        ev.dpc[e1] = L.vinint[n];
    }
}

__device__ __forceinline__ void emit_inbound(const Events& ev, int64_t* scal, int64_t base,
                                             int32_t p, int32_t mi, int32_t d)
{
    int64_t pos = base + (int64_t)atomicAdd((unsigned long long*)&scal[RS_NEV], 1ull);
    if (pos >= ev.cap) {
        atomicOr((int*)&scal[SC_STATUS], ST_CAPACITY);
        return;
    }
    ev.key[pos] = ((uint64_t)p << ev.ibits) | (uint64_t)mi;
    ev.idx[pos] = (uint32_t)pos;
    ev.dsize[pos] = 0;
    ev.dinp[pos] = 0;
    ev.dpc[pos] = d;
}

// one moved pin's replay given the deltas of earlier moves of the same hyperedge
__device__ __forceinline__ void replay_one(const Level& L, const PinCounts& pc, int32_t a,
                                           int32_t mi, int32_t f, int32_t t, int d, int dcf_c,
                                           int dct_c, int dcf_d, int dct_d, int64_t* gp,
                                           const Events& ev, int64_t* scal, int64_t evbase)
{
    int64_t b = L.hoff[a];
    int32_t lam = pc.lam[a];
    int32_t c0f, d0f, c0t, d0t;
    lookup_count(pc, b, lam, f, c0f, d0f);
    lookup_count(pc, b, lam, t, c0t, d0t);
    int32_t cf = c0f + dcf_c, ct = c0t + dct_c;
    int64_t g = (int64_t)L.hw[a] * ((cf == 1 ? 1 : 0) - (ct == 0 ? 1 : 0));
    if (g) atomicAdd((unsigned long long*)&gp[mi], (unsigned long long)g);
    if (d) {
        if (d0f + dcf_d == 1) emit_inbound(ev, scal, evbase, f, mi, -L.hk[a]);
        if (d0t + dct_d == 0) emit_inbound(ev, scal, evbase, t, mi, L.hk[a]);
    }
}

__global__ void __launch_bounds__(256)
    k_replay_warp(Level L, PinCounts pc, const int32_t* __restrict__ moveidx, Moves mv,
                  uint32_t* mvbuf, int64_t* gp, Events ev, int64_t evbase, int32_t* heavy,
                  int32_t* heavycnt, int64_t* scal, HedgeList hl)
{
    after_previous();
    int lane = threadIdx.x & 31;
    unsigned lt = lanemask_lt();
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t nh = *hl.n;
    for (int64_t x = gw; x < nh; x += nw) {
        int32_t a = hl.a[x];
        int64_t b = L.hoff[a], e = L.hoff[a + 1];
        int sd = L.hsd[a];
        int cnt = 0;
        for (int64_t cb = b; cb < e; cb += 32) {
            int64_t j = cb + lane;
            int32_t mi = -1;
            if (j < e) mi = moveidx[L.hpins[j]];
            bool moved = mi >= 0;
            unsigned mk = __ballot_sync(FULL, moved);
            if (moved) {
                uint32_t d = (j != b || sd) ? 1u : 0u;
                mvbuf[b + cnt + __popc(mk & lt)] = ((uint32_t)mi << 1) | d;
            }
            cnt += __popc(mk);
        }
        if (cnt == 0) continue;
        __syncwarp();
        if (cnt > REPLAY_WARP_MAX) {
            if (lane == 0) {
                int32_t pos = atomicAdd((int*)&scal[RS_NHV], 1);
                heavy[pos] = (int32_t)a;
                heavycnt[pos] = cnt;
            }
            continue;
        }
        uint32_t rec = lane < cnt ? mvbuf[b + lane] : 0u;
        int32_t mi = (int32_t)(rec >> 1);
        int d = rec & 1;
        int32_t f = lane < cnt ? mv.from[mi] : -1;
        int32_t t = lane < cnt ? mv.to[mi] : -1;
        int dcf_c = 0, dct_c = 0, dcf_d = 0, dct_d = 0;
        for (int jj = 0; jj < cnt; jj++) {
            int32_t mj = __shfl_sync(FULL, mi, jj);
            int32_t fj = __shfl_sync(FULL, f, jj);
            int32_t tj = __shfl_sync(FULL, t, jj);
            int dj = __shfl_sync(FULL, d, jj);
            if (mj < mi) {
                int ef = (tj == f) - (fj == f), et = (tj == t) - (fj == t);
                dcf_c += ef;
                dct_c += et;
                if (dj) {
                    dcf_d += ef;
                    dct_d += et;
                }
            }
        }
        if (lane < cnt)
            replay_one(L, pc, (int32_t)a, mi, f, t, d, dcf_c, dct_c, dcf_d, dct_d, gp, ev, scal, evbase);
    }
}

__global__ void __launch_bounds__(256)
    k_replay_block(Level L, PinCounts pc, Moves mv, const uint32_t* __restrict__ mvbuf, int64_t* gp,
                   Events ev, int64_t evbase, const int32_t* __restrict__ heavy,
                   const int32_t* __restrict__ heavycnt, int64_t* scal)
{
    after_previous();
    int32_t nh = (int32_t)scal[RS_NHV];
    for (int32_t h = blockIdx.x; h < nh; h += gridDim.x) {
        int32_t a = heavy[h];
        int32_t cnt = heavycnt[h];
        int64_t b = L.hoff[a];
        for (int32_t x = threadIdx.x; x < cnt; x += blockDim.x) {
            uint32_t rec = mvbuf[b + x];
            int32_t mi = (int32_t)(rec >> 1);
            int d = rec & 1;
            int32_t f = mv.from[mi], t = mv.to[mi];
            int dcf_c = 0, dct_c = 0, dcf_d = 0, dct_d = 0;
            for (int32_t y = 0; y < cnt; y++) {
                uint32_t ry = mvbuf[b + y];
                int32_t mj = (int32_t)(ry >> 1);
                if (mj >= mi) continue;
                int32_t fj = mv.from[mj], tj = mv.to[mj];
                int ef = (tj == f) - (fj == f), et = (tj == t) - (fj == t);
                dcf_c += ef;
                dct_c += et;
                if (ry & 1) {
                    dcf_d += ef;
                    dct_d += et;
                }
            }
            replay_one(L, pc, a, mi, f, t, d, dcf_c, dct_c, dcf_d, dct_d, gp, ev, scal, evbase);
        }
    }
}

// ---------------------------------------------------------------------------
// S10

__global__ void k_part_bounds(int64_t T, const uint64_t* __restrict__ key, int ibits, int32_t* pbeg,
                              int32_t* pend)
{
    after_previous();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < T;
         e += (int64_t)gridDim.x * blockDim.x) {
        uint64_t p = key[e] >> ibits;
        if (e == 0 || (key[e - 1] >> ibits) != p) pbeg[p] = (int32_t)e;
        if (e == T - 1 || (key[e + 1] >> ibits) != p) pend[p] = (int32_t)(e + 1);
    }
}

__global__ void __launch_bounds__(256)
    k_part_validity(int32_t K, const int32_t* __restrict__ pbeg, const int32_t* __restrict__ pend,
                    Events ev, PState ps, int32_t omega, int32_t delta, int32_t phi, int32_t* dv)
{
    after_previous();
    int lane = threadIdx.x & 31;
    unsigned lt = lanemask_lt();
    uint64_t imask = (ev.ibits >= 64) ? ~0ull : ((1ull << ev.ibits) - 1);
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = gw; p < K; p += nw) {
        int32_t beg = pbeg[p], end = pend[p];
        if (beg >= end) continue;
        int64_t s0 = ps.size[p], i0 = ps.inpins[p], c0 = ps.pincnt[p];
        int64_t cs = 0, ci = 0, cc = 0;
        int prev_viol = 0;
        for (int32_t cb = beg; cb < end; cb += 32) {
            int32_t e = cb + lane;
            bool valid = e < end;
            int64_t mi = -1, ds = 0, di = 0, dc = 0;
            if (valid) {
                mi = (int64_t)(ev.key[e] & imask);
                uint32_t x = ev.idx[e];
                ds = ev.dsize[x];
                di = ev.dinp[x];
                dc = ev.dpc[x];
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int64_t a1 = __shfl_up_sync(FULL, ds, o);
                int64_t a2 = __shfl_up_sync(FULL, di, o);
                int64_t a3 = __shfl_up_sync(FULL, dc, o);
                if (lane >= o) {
                    ds += a1;
                    di += a2;
                    dc += a3;
                }
            }
            int64_t nmi = __shfl_down_sync(FULL, mi, 1);
            if (lane == 31) nmi = (e + 1 < end) ? (int64_t)(ev.key[e + 1] & imask) : -1;
            if (valid && e + 1 >= end) nmi = -1;
            bool gend = valid && nmi != mi;
            int viol = gend ? (violates(s0 + cs + ds, i0 + ci + di, c0 + cc + dc, omega, delta, phi) ? 1 : 0) : 0;
            unsigned gm = __ballot_sync(FULL, gend);
            unsigned below = gm & lt;
            int src = below ? 31 - __clz(below) : lane;
            int pv = __shfl_sync(FULL, viol, src);
            if (!below) pv = prev_viol;
            if (gend && viol != pv) atomicAdd(&dv[mi], viol - pv);
            if (gm) prev_viol = __shfl_sync(FULL, viol, 31 - __clz(gm));
            cs += __shfl_sync(FULL, ds, 31);
            ci += __shfl_sync(FULL, di, 31);
            cc += __shfl_sync(FULL, dc, 31);
        }
    }
}

// ---------------------------------------------------------------------------
// S11

__global__ void k_best1(int32_t M, const int64_t* __restrict__ G, const int32_t* __restrict__ nviol,
                        int64_t* scal)
{
    after_previous();
    int64_t best = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x)
        if (nviol[i] == 0 && G[i] > best) best = G[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        int64_t b2 = __shfl_xor_sync(FULL, best, o);
        best = b2 > best ? b2 : best;
    }
    if ((threadIdx.x & 31) == 0 && best > 0)
        atomicMax((unsigned long long*)&scal[RS_BEST], (unsigned long long)best);
}

__global__ void k_best2(int32_t M, const int64_t* __restrict__ G, const int32_t* __restrict__ nviol,
                        int64_t* scal)
{
    after_previous();
    int64_t best = scal[RS_BEST];
    if (best <= 0) return;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x)
        if (nviol[i] == 0 && G[i] == best) atomicMin((unsigned long long*)&scal[RS_ISTAR], (unsigned long long)i);
}

// S10 and S11 in one block, for rounds whose events and moves fit its shared
// memory: events sorted by (partition, move), each partition's limits after
// each of its moves from a segmented scan, violation changes and gains
// summed along the moves, and the best valid prefix. The event count stays
// on the device, so a round takes no wait between replay and prefix; as
// separate launches (sort, bounds, validity, two scans, two maxima, with the
// wait before them) this was about 70 us of a round.
struct Seg3 {
    int64_t s, i, c;   // size, inbound pins, inbound axons
    int head;          // the run started here
};
__device__ __forceinline__ Seg3 seg3_join(const Seg3& a, const Seg3& b)
{
    if (b.head) return b;
    return Seg3{a.s + b.s, a.i + b.i, a.c + b.c, a.head};
}
__device__ __forceinline__ Seg3 seg3_shfl_up(const Seg3& v, int o)
{
    return Seg3{__shfl_up_sync(FULL, v.s, o), __shfl_up_sync(FULL, v.i, o), __shfl_up_sync(FULL, v.c, o),
                __shfl_up_sync(FULL, v.head, o)};
}

constexpr int TAIL_EVENTS = SB_MAX;
constexpr int TAIL_PER = TAIL_EVENTS / SB_THREADS;   // consecutive events per thread

__global__ void __launch_bounds__(SB_THREADS)
    k_round_tail(int32_t M, Events ev, PState ps, int32_t omega, int32_t delta, int32_t phi,
                 const int64_t* __restrict__ gp, int64_t* scal)
{
    after_previous();
    __shared__ uint64_t w[TAIL_EVENTS];
    __shared__ int32_t dv[TAIL_EVENTS / 2];   // two events per move at least
    __shared__ Seg3 wseg[32];
    __shared__ int64_t wg[32];
    __shared__ int32_t wv[32];
    __shared__ unsigned long long sbest;
    __shared__ int simin;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int T = 2 * M + (int)scal[RS_NEV];   // <= TAIL_EVENTS (the events' capacity)
    constexpr int IB = 12;
    int N = 64;
    while (N < T) N <<= 1;
    for (int e = tid; e < N; e += SB_THREADS)
        w[e] = e < T ? (ev.key[e] << IB) | (uint64_t)e : ~0ull;
    for (int i = tid; i < M; i += SB_THREADS) dv[i] = 0;
    if (tid == 0) {
        sbest = 0;
        simin = INT_MAX;
    }
    __syncthreads();
    block_sort_words(w, N);
    const uint64_t imask = (1ull << ev.ibits) - 1;
    const int e0 = tid * TAIL_PER;
    Seg3 v[TAIL_PER];
    Seg3 run{0, 0, 0, 0};
#pragma unroll
    for (int r = 0; r < TAIL_PER; r++) {
        int e = e0 + r;
        Seg3 x{0, 0, 0, 0};
        if (e < T) {
            uint32_t o = (uint32_t)(w[e] & ((1u << IB) - 1));
            uint64_t p = w[e] >> IB >> ev.ibits;
            x = Seg3{ev.dsize[o], ev.dinp[o], ev.dpc[o], e == 0 || (w[e - 1] >> IB >> ev.ibits) != p};
        }
        run = r == 0 ? x : seg3_join(run, x);
        v[r] = run;
    }
    Seg3 inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        Seg3 t = seg3_shfl_up(inc, o);
        if (lane >= o) inc = seg3_join(t, inc);
    }
    if (lane == 31) wseg[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        Seg3 t = wseg[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            Seg3 u = seg3_shfl_up(t, o);
            if (lane >= o) t = seg3_join(u, t);
        }
        wseg[lane] = t;
    }
    __syncthreads();
    Seg3 before = seg3_shfl_up(inc, 1);
    if (lane == 0) before = Seg3{0, 0, 0, 0};
    if (warp > 0) before = lane == 0 ? wseg[warp - 1] : seg3_join(wseg[warp - 1], before);
#pragma unroll
    for (int r = 0; r < TAIL_PER; r++) {
        int e = e0 + r;
        if (e >= T) continue;
        uint64_t key = w[e] >> IB, nxt = e + 1 < T ? w[e + 1] >> IB : ~0ull;
        if (nxt == key) continue;   // the move has more events in this partition
        Seg3 a = seg3_join(before, v[r]);
        int32_t p = (int32_t)(key >> ev.ibits);
        if (!violates(ps.size[p] + a.s, ps.inpins[p] + a.i, ps.pincnt[p] + a.c, omega, delta, phi))
            continue;
        // violated after this move until the partition's next one
        atomicAdd(&dv[key & imask], 1);
        if (e + 1 < T && (nxt >> ev.ibits) == (uint64_t)p) atomicAdd(&dv[nxt & imask], -1);
    }
    __syncthreads();
    // prefix sums along the moves, two consecutive ones per thread
    int64_t g[2];
    int32_t d[2];
#pragma unroll
    for (int r = 0; r < 2; r++) {
        int i = 2 * tid + r;
        g[r] = i < M ? gp[i] : 0;
        d[r] = i < M ? dv[i] : 0;
    }
    int64_t gi = warp_inclusive(g[0] + g[1]);
    int32_t di = warp_inclusive(d[0] + d[1]);
    if (lane == 31) {
        wg[warp] = gi;
        wv[warp] = di;
    }
    __syncthreads();
    int64_t gb = gi - g[0] - g[1];
    int32_t db = di - d[0] - d[1];
    for (int x = 0; x < warp; x++) {
        gb += wg[x];
        db += wv[x];
    }
    int64_t G[2] = {gb + g[0], gb + g[0] + g[1]};
    bool ok[2] = {2 * tid < M && db + d[0] == 0, 2 * tid + 1 < M && db + d[0] + d[1] == 0};
    int64_t best = 0;
    if (ok[0] && G[0] > best) best = G[0];
    if (ok[1] && G[1] > best) best = G[1];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        int64_t b2 = __shfl_xor_sync(FULL, best, o);
        best = b2 > best ? b2 : best;
    }
    if (lane == 0 && best > 0) atomicMax(&sbest, (unsigned long long)best);
    __syncthreads();
    best = (int64_t)sbest;
    if (best <= 0) return;
    if (ok[1] && G[1] == best) atomicMin(&simin, 2 * tid + 1);
    if (ok[0] && G[0] == best) atomicMin(&simin, 2 * tid);
    __syncthreads();
    if (tid == 0) {
        scal[RS_BEST] = best;
        scal[RS_ISTAR] = simin;
    }
}

// The round's scalars: all zero but the prefix end (none). First round: Conn
// from its partial sums, and whether the partitions are within their limits
// (an enacted prefix is valid, so the state can only be broken at the start).
// Conn and that finding go straight to the host's words (pinned, HW_BAD
// cleared by the host, read after the proposals' wait), which saves a copy a
// round.
__global__ void __launch_bounds__(1024)
    k_round_begin(int64_t* scal, int64_t* costv, const int64_t* __restrict__ slots, int32_t K, PState ps,
                  int32_t omega, int32_t delta, int32_t phi, int64_t* host)
{
    after_previous();
    __shared__ unsigned long long sum;
    const int i = threadIdx.x;
    if (slots) {
        for (int64_t p = blockIdx.x * (int64_t)blockDim.x + i; p < K; p += (int64_t)gridDim.x * blockDim.x)
            if (violates(ps.size[p], ps.inpins[p], ps.pincnt[p], omega, delta, phi)) host[HW_BAD] = 1;
    }
    if (blockIdx.x != 0) return;
    if (i < SC_COUNT) scal[i] = i == RS_ISTAR ? INT64_MAX : 0;
    if (!slots) {
        if (i == 0) host[HW_COST] = *costv;
        return;
    }
    if (i == 0) sum = 0;
    __syncthreads();
    if (i < COST_SLOTS) {
        int64_t v = warp_sum(slots[i]);
        if ((i & 31) == 0) atomicAdd(&sum, (unsigned long long)v);
    }
    __syncthreads();
    if (i == 0) {
        *costv = (int64_t)sum;
        host[HW_COST] = (int64_t)sum;
    }
}

template <typename S>
static Status gains(snnmap_hgraph* h, Level& L, const PinCounts& pc, const int32_t* rho,
                    const PState& ps, int32_t K, int32_t* pto, int64_t* pgain,
                    const int64_t* savev, const int32_t* dirty)
{
    GainPol<S> pol;
    pol.savev = savev;
    pol.dirty = dirty;
    pol.nonpos = h->prm.refine_nonpositive != 0;
    pol.L = L;
    pol.pc = pc;
    pol.ps = ps;
    pol.rho = rho;
    pol.V = L.V;
    pol.keys = K;
    pol.omega = h->prm.omega;
    pol.delta = h->prm.delta;
    pol.phi = h->prm.phi;
    pol.pto = pto;
    pol.pgain = pgain;
    int64_t* cnt;
    SNN_TRY(h->scratch.alloc(&cnt, HT_NCNT));
    return run_histogram(pol, h->scratch, h->stream, cnt, h->h_scal + 12, h->tiers, K,
                         !h->wzero);
}

// rows of the vertices flagged fresh, from the round's pin counts
static Status dense_fresh(snnmap_hgraph* h, Level& L, const PinCounts& pc)
{
    DenseRows& D = h->dense;
    RowPol<uint32_t> pol;
    pol.L = L;
    pol.pc = pc;
    pol.V = L.V;
    pol.keys = D.K;
    pol.fresh = D.fresh;
    pol.rowid = D.rowid;
    pol.tab = D.tab;
    pol.M = D.M;
    pol.cw = D.cw;
    int64_t* cnt;
    SNN_TRY(h->scratch.alloc(&cnt, HT_NCNT));
    return run_histogram(pol, h->scratch, h->stream, cnt, h->h_scal + 12, h->tiers, D.K,
                         !h->wzero);
}

int64_t dense_row_budget(const snnmap_hgraph* h)
{
    if (h->row_budget >= 0) return h->row_budget;
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) return 0;
    return (int64_t)(tot / 4);
}

// rows per chunk: about 1 GB of C and O
constexpr int64_t ROW_CHUNK_BYTES = (int64_t)1 << 30;

Status dense_open(snnmap_hgraph* h, int32_t K, int64_t cap)
{
    dense_close(h);
    DenseRows& D = h->dense;
    cudaStream_t s = h->stream;
    D.K = K;
    D.Kp = ((int64_t)K + 3) & ~(int64_t)3;
    D.cap = cap > 0 ? cap : 1;
    D.tab.Kp = D.Kp;
    while (((int64_t)1 << D.tab.shift) < D.cap && ((int64_t)2 << D.tab.shift) * D.Kp * 8 <= ROW_CHUNK_BYTES)
        D.tab.shift++;
    const int64_t nchunks = ceil_div(D.cap, (int64_t)1 << D.tab.shift);
    SNN_CUDA(dev_malloc((void**)&D.tab.tab, (size_t)nchunks * 2 * sizeof(int32_t*), s));
    SNN_CUDA(dev_malloc(&D.rowid, (size_t)D.cap * 4, s));
    SNN_CUDA(dev_malloc(&D.rowid2, (size_t)D.cap * 4, s));
    SNN_CUDA(dev_malloc(&D.fresh, (size_t)D.cap * 4, s));
    SNN_CUDA(dev_malloc(&D.M, (size_t)D.cap * 8, s));
    D.cw = 32;
    while ((int64_t)D.cw * 64 < D.Kp) D.cw <<= 1;
    D.level = -1;
    D.pending = false;
    return Status{};
}

Status dense_grow(snnmap_hgraph* h, int64_t rows)
{
    DenseRows& D = h->dense;
    if (!D.rowid || rows > D.cap) return Status{SNNMAP_ERR_STATE, "connection rows: capacity"};
    if (rows > h->row_fault.rows) return Status{h->row_fault.code, "connection rows: refused"};
    const int64_t per = (int64_t)1 << D.tab.shift;
    const size_t had = D.chunks.size(), need = (size_t)ceil_div(std::max<int64_t>(rows - D.rows, 0), per);
    std::vector<int32_t*> ptrs;
    ptrs.reserve(2 * need);
    D.chunks.reserve(had + need);   // so that no chunk is lost to a failed host allocation
    while (D.rows < rows) {
        const int64_t n = std::min<int64_t>(per, D.cap - D.rows);
        int32_t* c = nullptr;
        SNN_CUDA(dev_malloc(&c, (size_t)(n * D.Kp) * 8, h->stream));
        D.chunks.push_back(c);
        ptrs.push_back(c);
        ptrs.push_back(c + n * D.Kp);
        D.rows += n;
    }
    if (!ptrs.empty())
        SNN_CUDA(cudaMemcpyAsync((void*)(D.tab.tab + 2 * had), ptrs.data(), ptrs.size() * sizeof(int32_t*),
                                 cudaMemcpyHostToDevice, h->stream));
    return Status{};
}

void dense_close(snnmap_hgraph* h)
{
    DenseRows& D = h->dense;
    for (int32_t* p : D.chunks) cudaFreeAsync(p, h->stream);
    for (int32_t* p : {D.rowid, D.rowid2, D.fresh})
        if (p) cudaFreeAsync(p, h->stream);
    if (D.M) cudaFreeAsync(D.M, h->stream);
    if (D.tab.tab) cudaFreeAsync((void*)D.tab.tab, h->stream);
    D = DenseRows{};
}

Status dense_begin(snnmap_hgraph* h, int32_t level)
{
    DenseRows& D = h->dense;
    const Level& L = h->levels[level];
    if (L.V > D.rows) return Status{SNNMAP_ERR_STATE, "connection rows: capacity"};
    SNN_TRY(iota_i32(D.rowid, L.V, h->stream));
    SNN_TRY(fill_i32(D.fresh, 1, L.V, h->stream));
    if (L.V > 0) {
        enqueue(k_dense_zero, grid_for((int64_t)L.V * 32, 256), 256, 0, h->stream, L.V, D.fresh,
                D.rowid, D.tab, D.M);
        SNN_CUDA(cudaGetLastError());
    }
    D.level = level;
    D.pending = true;
    return Status{};
}

Status dense_descend(snnmap_hgraph* h, int32_t level)
{
    DenseRows& D = h->dense;
    const Level& L = h->levels[level];
    int32_t Vc = h->levels[level + 1].V;
    if (D.level != level + 1 || L.V > D.rows)
        return Status{SNNMAP_ERR_STATE, "connection rows: descent out of order"};
    cudaStream_t s = h->stream;
    Arena& ar = h->scratch;
    if (L.V > 0) {
        SNN_TRY(scan_run<int32_t>(UpperMember{L.pr}, RowIds{L.pr, L.cid, D.rowid, Vc, D.rowid2, D.fresh}, L.V,
                                  (int32_t*)nullptr, ar, s));
        std::swap(D.rowid, D.rowid2);
        enqueue(k_dense_zero, grid_for((int64_t)L.V * 32, 256), 256, 0, s, L.V, D.fresh, D.rowid,
                D.tab, D.M);
        SNN_CUDA(cudaGetLastError());
    }
    D.level = level;
    D.pending = true;
    return Status{};
}

// pin counts + partition state + the COST_SLOTS partial sums of Conn for rho,
// into buffers the caller owns (state and sums cleared)
static Status pin_counts_into(snnmap_hgraph* h, Level& L, LevelExtra& X, int32_t K,
                              const int32_t* rho, PinCounts& pc, PState& ps, int64_t* slots)
{
    cudaStream_t s = h->stream;
    Arena& ar = h->scratch;
    if (L.V > 0) {
        enqueue(k_pstate_vertices, grid_for(L.V, 256), 256, 0, s, L, rho, ps);
        SNN_CUDA(cudaGetLastError());
    }
    PinCountJob job{L.hoff, L.hpins, L.hsd, L.hk, L.hw, rho, pc, ps.pincnt, slots};
    // with many hyperedges a partition, as every block clears and adds up K
    // words; where the line lies is of no consequence (2 and 128 hyperedges a
    // partition: within 0.5 % of this on eight passes of 4,096 to 1,048,576
    // neurons)
    if (K <= PC_SMEM_K && L.E >= 16 * (int64_t)K) job.K = K;
    return seg_run(job, X.seg, L.E, ar, s);
}

Status level_cost(snnmap_hgraph* h, int32_t level, int32_t K, const int32_t* rho, int64_t* cost)
{
    Level& L = h->levels[level];
    LevelExtra& X = h->extra[level];
    SNN_TRY(zero_scalars(h));
    PinCounts pc;
    PState ps;
    Arena& ar = h->scratch;
    SNN_TRY(ar.alloc(&pc.p, L.P));
    SNN_TRY(ar.alloc(&pc.cnt, L.P));
    SNN_TRY(ar.alloc(&pc.dcnt, L.P));
    SNN_TRY(ar.alloc(&pc.lam, L.E));
    SNN_TRY(ar.alloc(&pc.rec, L.E));
    int64_t* slots;
    Carver cv;
    cv.add(&ps.size, K);
    cv.add(&ps.inpins, K);
    cv.add(&ps.pincnt, K);
    cv.add(&slots, COST_SLOTS);
    char* base;
    SNN_TRY(ar.alloc(&base, (int64_t)cv.total));
    cv.assign(base);
    SNN_CUDA(cudaMemsetAsync(base, 0, cv.total, h->stream));
    SNN_TRY(pin_counts_into(h, L, X, K, rho, pc, ps, slots));
    enqueue(k_cost_slots, 1, 256, 0, h->stream, slots, h->d_scal + RS_COST);
    SNN_CUDA(cudaGetLastError());
    SNN_TRY(read_scalars(h));
    h->scratch.reset();
    *cost = h->h_scal[RS_COST];
    return Status{};
}

// ---------------------------------------------------------------------------
// Carried pin counts. Only hyperedges holding a pin of the enacted prefix
// change their counts; their old contributions (inbound k per partition,
// omega (lambda - 1) to Conn, omega to the save of a pin alone in its
// partition) are taken out before the moves, the moves' own size, inbound
// pins and internal axons move between partitions, the hyperedges are
// counted again, and their new contributions added back.

// One warp per listed hyperedge: its enacted moves; if it holds any, its row
// updates (levels with rows), its mark, and its old contributions out of the
// partition state, Conn and the saves (the count pass adds the new ones).
__global__ void __launch_bounds__(256)
    k_prefix_hedges(Level L, PinCounts pc, const int32_t* __restrict__ moveidx, Moves mv,
                    const int64_t* __restrict__ scal, RowsRef R, uint32_t* buf, int32_t* hdirty,
                    const int32_t* __restrict__ rho, PState ps, int64_t* savev, int64_t* costv,
                    HedgeList hl)
{
    after_previous();
    int64_t istar = scal[RS_BEST] > 0 ? scal[RS_ISTAR] : -1;
    if (istar < 0) return;   // nothing is marked (the marks are cleared every round)
    int lane = threadIdx.x & 31;
    unsigned lt = lanemask_lt();
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t nh = *hl.n;
    for (int64_t x = gw; x < nh; x += nw) {
        int32_t a = hl.a[x];
        int64_t b = L.hoff[a], e = L.hoff[a + 1];
        int sd = L.hsd[a];
        int m = 0;
        for (int64_t cb = b; cb < e; cb += 32) {
            int64_t j = cb + lane;
            int32_t mi = -1;
            if (j < e) mi = moveidx[L.hpins[j]];
            bool ap = mi >= 0 && mi <= istar;
            unsigned mk = __ballot_sync(FULL, ap);
            if (ap) buf[b + m + __popc(mk & lt)] = ((uint32_t)mi << 1) | ((j != b || sd) ? 1u : 0u);
            m += __popc(mk);
        }
        if (m == 0) continue;
        __syncwarp();
        int32_t lam = pc.lam[a];
        int64_t w = L.hw[a];
        int32_t k = L.hk[a];
        if (R.rowid) rows_cross(L, pc, mv, R, a, b, e, sd, lam, w, k, buf, m);
        if (lane == 0) hdirty[a] = 1;
        for (int32_t r = lane; r < lam; r += 32)
            if (pc.dcnt[b + r] > 0)
                atomicAdd((unsigned long long*)&ps.pincnt[pc.p[b + r]], (unsigned long long)(-(int64_t)k));
        if (lane == 0 && lam > 1)
            atomicAdd((unsigned long long*)costv, (unsigned long long)(-(w * (lam - 1))));
        for (int64_t j = b + lane; j < e; j += 32) {
            int32_t q = L.hpins[j];
            int32_t c, d;
            lookup_count(pc, b, lam, rho[q], c, d);
            if (c == 1) atomicAdd((unsigned long long*)&savev[q], (unsigned long long)(-w));
        }
    }
}

// new contributions of hyperedge a to the saves (one warp)
__device__ __forceinline__ void add_saves(const Level& L, const PinCounts& pc,
                                          const int32_t* __restrict__ rho, int64_t* savev, int32_t a)
{
    const int lane = threadIdx.x & 31;
    int64_t b = L.hoff[a], e = L.hoff[a + 1];
    int32_t lam = pc.lam[a];
    int64_t w = L.hw[a];
    for (int64_t j = b + lane; j < e; j += 32) {
        int32_t q = L.hpins[j];
        int32_t c, d;
        lookup_count(pc, b, lam, rho[q], c, d);
        if (c == 1) atomicAdd((unsigned long long*)&savev[q], (unsigned long long)w);
    }
}

// after the count pass over the size buckets: the saves of the marked
// hyperedges, and the listed ones' marks back to zero for the next round
__global__ void __launch_bounds__(256)
    k_prefix_saves(Level L, PinCounts pc, const int32_t* __restrict__ rho, int64_t* savev,
                   int32_t* hmark, int32_t* hdirty, HedgeList hl)
{
    after_previous();
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t nh = *hl.n;
    for (int64_t x = gw; x < nh; x += nw) {
        int32_t a = hl.a[x];
        if (hdirty[a]) add_saves(L, pc, rho, savev, a);
        __syncwarp();
        if (lane == 0) {
            hmark[a] = 0;
            hdirty[a] = 0;
        }
    }
}

// The count pass and the saves in one launch, a warp per listed hyperedge,
// for short lists on levels without hyperedges of more than SEG_B1_CAP pins:
// filtering the level's size buckets, counting them, and the two passes
// after it were six launches over mostly a few hundred hyperedges.
constexpr int64_t RECOUNT_MAX = 1 << 15;

__global__ void __launch_bounds__(256)
    k_prefix_recount(Level L, PinCountJob job, const int32_t* __restrict__ rho, int64_t* savev,
                     int32_t* hmark, int32_t* hdirty, HedgeList hl)
{
    after_previous();
    __shared__ __align__(16) uint32_t buf[8 * SEG_B1_CAP];
    const int lane = threadIdx.x & 31;
    uint32_t* s = buf + (threadIdx.x >> 5) * SEG_B1_CAP;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t nh = *hl.n;
    for (int64_t x = gw; x < nh; x += nw) {
        int32_t a = hl.a[x];
        if (hdirty[a]) {
            int n = job.len(a);
            if (n <= 32) {
                uint32_t v = lane < n ? job.load(a, lane) : KEY_PAD;
                s[lane] = warp_bitonic32(v);
                __syncwarp();
            } else if (n <= 64) {
                warp_sort_list<2>(job, a, n, s);
            } else if (n <= 128) {
                warp_sort_list<4>(job, a, n, s);
            } else {
                warp_sort_list<8>(job, a, n, s);
            }
            job.finish(a, s, n);
            __syncwarp();
            add_saves(L, job.pc, rho, savev, a);
        }
        __syncwarp();
        if (lane == 0) {
            hmark[a] = 0;
            hdirty[a] = 0;
        }
    }
}

// the enacted moves: rho, and their own size, inbound pins and internal axons
// change partition
__global__ void k_apply(int32_t M, Moves mv, Level L, const int64_t* __restrict__ scal, PState ps,
                        int32_t* rho, int32_t* moveidx)
{
    after_previous();
    int64_t istar = scal[RS_BEST] > 0 ? scal[RS_ISTAR] : -1;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < M;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t n = mv.n[i];
        moveidx[n] = -1;
        if (i > istar) continue;
        int32_t f = mv.from[i], t = mv.to[i];
        rho[n] = t;
        int64_t sz = L.vsize[n], ip = L.vinpins[n], ii = L.vinint[n];
        atomicAdd((unsigned long long*)&ps.size[f], (unsigned long long)(-sz));
        atomicAdd((unsigned long long*)&ps.size[t], (unsigned long long)sz);
        atomicAdd((unsigned long long*)&ps.inpins[f], (unsigned long long)(-ip));
        atomicAdd((unsigned long long*)&ps.inpins[t], (unsigned long long)ip);
        if (ii) {
            atomicAdd((unsigned long long*)&ps.pincnt[f], (unsigned long long)(-ii));
            atomicAdd((unsigned long long*)&ps.pincnt[t], (unsigned long long)ii);
        }
    }
}

// the level's size buckets restricted to marked hyperedges (each bucket keeps
// its start; counts by atomics, order irrelevant)
__global__ void k_seg_filter(const int32_t* __restrict__ list, const int32_t* __restrict__ meta,
                             int32_t E, const int32_t* __restrict__ hdirty, int32_t* out,
                             int32_t* meta2)
{
    after_previous();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < E;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = list[i];
        if (!hdirty[a]) continue;
        int b = 0;
        while (b + 1 < SEG_NB && i >= meta[b + 1]) b++;
        int32_t pos = atomicAdd(&meta2[SEG_NB + b], 1);
        out[meta[b] + pos] = a;
    }
}

__global__ void k_seg_meta_copy(const int32_t* __restrict__ meta, int32_t* meta2)
{
    after_previous();
    for (int b = threadIdx.x; b < SEG_NB; b += blockDim.x) meta2[b] = meta[b];
}

// Per-level buffers that outlive a round: proposals (kept by vertices the
// previous round did not touch), the vertices to evaluate, partition flags
// and the level's largest vertex state.
struct IncState {
    int32_t* pto = nullptr;
    int64_t* pgain = nullptr;
    int32_t* dirty = nullptr;
    uint8_t* pchg = nullptr;
    uint8_t* prel = nullptr;
    int32_t* vmax = nullptr;
    // pin counts, partition state, Conn (costv), save and W carried from
    // round to round: a round after the first starts from them, and the
    // enacted prefix updates them for the hyperedges holding a moved pin
    PinCounts pc;
    PState ps;
    int64_t* costv = nullptr;
    int64_t* slots = nullptr;    // partial sums of Conn of the first round
    int64_t* savev = nullptr;
    int64_t* Wv = nullptr;
    int32_t* hdirty = nullptr;   // per hyperedge
    int32_t* hmark = nullptr;    // per hyperedge: listed this round (k_prop_hedges)
    int32_t* hlist = nullptr;    // bucket lists filtered to dirty hyperedges
    int32_t* hmeta = nullptr;    // their bucket starts and counts (2 * SEG_NB)
    bool ready = false;          // set once the first round computed them
    PStar pst;                   // column update of proposals after short prefixes
    int64_t members = 0;         // members of pairs whose saves are to be computed (0: all vertices')
    int32_t* mlist = nullptr;
    int32_t* mcnt = nullptr;
};

// saves and W of the listed vertices (cleared before) from their hyperedges;
// the 4 to 64 blocks of a column share a vertex's incidences, so that the one
// heavy pair of a tail level is not a chain of gathers on a few warps (layered
// network of 60,000 neurons: 12.1 us a level with four blocks, 8.6 so)
__global__ void __launch_bounds__(256)
    k_save_members(Level L, PinCounts pc, const int32_t* __restrict__ rho,
                   const int32_t* __restrict__ list, const int32_t* __restrict__ nlist, int64_t* savev,
                   int64_t* Wv)
{
    after_previous();
    __shared__ unsigned long long sum[2];
    const int32_t nl = *nlist;
    for (int32_t x = blockIdx.x; x < nl; x += gridDim.x) {
        const int32_t n = list[x];
        const int64_t vb = L.voff[n], ve = L.voff[n + 1];
        if (vb + (int64_t)blockIdx.y * 256 >= ve) continue;   // the whole block
        if (threadIdx.x < 2) sum[threadIdx.x] = 0;
        __syncthreads();
        const int32_t p = rho[n];
        int64_t W = 0, save = 0;
        for (int64_t i = vb + (int64_t)blockIdx.y * 256 + threadIdx.x; i < ve; i += (int64_t)gridDim.y * 256) {
            HRec r = pc.rec[(int32_t)((uint32_t)L.vinc[i] & ~SRC_BIT)];
            W += r.w;
            int32_t c, d;
            lookup_count(pc, r.b, r.n(), p, c, d);
            if (c == 1) save += r.w;
        }
        W = warp_sum(W);
        save = warp_sum(save);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&sum[0], (unsigned long long)W);
            atomicAdd(&sum[1], (unsigned long long)save);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (sum[0]) atomicAdd((unsigned long long*)&Wv[n], sum[0]);
            if (sum[1]) atomicAdd((unsigned long long*)&savev[n], sum[1]);
        }
        __syncthreads();
    }
}

// One round; *applied = moves enacted, *gain = Conn removed, *cost = Conn at
// round start.
static Status refine_round(snnmap_hgraph* h, int32_t level, int32_t K, int32_t* rho,
                           int32_t* moveidx, const IncState& inc, int32_t* n_props,
                           int32_t* applied, int64_t* gain, int64_t* cost, int32_t* n_active,
                           int32_t* rows)
{
    cudaStream_t s = h->stream;
    Arena& ar = h->scratch;
    Level& L = h->levels[level];
    LevelExtra& X = h->extra[level];
    const snnmap_params& prm = h->prm;
    int32_t V = L.V;
    *n_props = 0;
    *n_active = 0;
    *rows = 0;
    *applied = 0;
    *gain = 0;
    PinCounts pc = inc.pc;
    PState ps = inc.ps;
    int64_t* host = h->h_tier + 2 * TIER_SLOTS;   // pinned, written by the kernels
    {
        ProfScope prof(h, PS_PINCOUNT);
        if (!inc.ready) SNN_TRY(pin_counts_into(h, L, X, K, rho, pc, ps, inc.slots));
        host[HW_BAD] = 0;
        enqueue(k_round_begin, inc.ready ? 1 : grid_for(K, 1024, 152), inc.ready ? 32 : 1024, 0, s,
                h->d_scal, inc.costv, inc.ready ? nullptr : inc.slots, K, ps, prm.omega, prm.delta,
                prm.phi, host);
        SNN_CUDA(cudaGetLastError());
    }
    DenseRows& D = h->dense;
    const bool dense = D.level == level;
    std::unique_ptr<ProfScope> prof;
    if (dense && D.pending) {
        prof.reset(new ProfScope(h, PS_ROWS));
        SNN_TRY(dense_fresh(h, L, pc));
        D.pending = false;
    }
    int32_t* pto = inc.pto;
    int64_t* pgain = inc.pgain;
    int64_t* savev = inc.savev;
    int64_t* Wv = inc.Wv;
    if (!inc.ready) {
        prof.reset(new ProfScope(h, PS_SAVE));
        if (inc.mlist) {
            if (inc.members > 0)
                enqueue(k_save_members,
                        dim3((unsigned)std::min<int64_t>(inc.members, 152 * 16),
                             (unsigned)std::min<int64_t>(std::max<int64_t>(152 * 8 / inc.members, 4), 64)),
                        256, 0, s, L, pc, rho, inc.mlist, inc.mcnt, savev, Wv);
            SNN_CUDA(cudaGetLastError());
        } else if (L.E > 0 && !h->wide && V <= SAVE_SMEM_V) {
            auto launch = [&](auto kern) -> Status {
                SNN_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              SAVE_SMEM_V * 8));
                enqueue(kern, grid_for(L.P, 4096, 152), SAVE_THREADS, (size_t)V * 8, s, L, pc, rho,
                        savev, Wv);
                return Status{};
            };
            switch (hedge_lanes(L.P, L.E)) {
            case 4: SNN_TRY(launch(k_save_smem<4>)); break;
            case 8: SNN_TRY(launch(k_save_smem<8>)); break;
            case 16: SNN_TRY(launch(k_save_smem<16>)); break;
            default: SNN_TRY(launch(k_save_smem<32>));
            }
            SNN_CUDA(cudaGetLastError());
        } else if (L.E > 0) {
            SNN_HEDGE_LAUNCH(hedge_lanes(L.P, L.E), k_save, L.E, s, L, pc, rho, savev, Wv);
            SNN_CUDA(cudaGetLastError());
        }
    }
    prof.reset(new ProfScope(h, PS_GAINS));
    if (dense) {
        if (V > 0) {
            enqueue(k_dense_best, grid_for((int64_t)V * 32, 256), 256, 0, s, L, rho, ps, savev, Wv,
                    D.rowid, D.tab, D.M, D.cw, K, prm.omega, prm.delta, prm.phi,
                    prm.refine_nonpositive, pto, pgain, inc.dirty);
            SNN_CUDA(cudaGetLastError());
        }
    } else if (h->wide) {
        SNN_TRY(gains<unsigned long long>(h, L, pc, rho, ps, K, pto, pgain, savev, inc.dirty));
    } else {
        SNN_TRY(gains<uint32_t>(h, L, pc, rho, ps, K, pto, pgain, savev, inc.dirty));
    }
    int gv = grid_for(V, 256);
    uint64_t *keys, *keys2;
    uint32_t *vals, *vals2;
    SNN_TRY(ar.alloc(&keys, V));
    SNN_TRY(ar.alloc(&vals, V));
    const int64_t bias = h->wsum;   // gains lie in [-wsum, wsum]
    for (int i = 0; i < 3; i++) host[HW_PROPS + i] = 0;
    if (V > 0)
        SNN_TRY(scan_run<PropSums>(PropIn{pto, savev, dense ? nullptr : inc.dirty, L.voff,
                                      prm.refine_nonpositive},
                               PropOut{pgain, bias, keys, vals}, V, (PropSums*)(host + HW_PROPS), ar, s));
    prof.reset();
    SNN_CUDA(cudaStreamSynchronize(s));
    const int64_t* hs = host + HW_PROPS;
    *cost = host[HW_COST];
    *n_active = (int32_t)hs[2];
    *rows = dense ? 1 : 0;
    if (host[HW_BAD])
        return Status{SNNMAP_ERR_INVALID, "refinement input breaks a per-core limit"};
    int32_t M = (int32_t)hs[0];
    int64_t deg = hs[1];
    *n_props = M;
    if (M == 0) return Status{};

    // S8
    prof.reset(new ProfScope(h, PS_SORTMOVES));
    SNN_TRY(ar.alloc(&keys2, M));
    SNN_TRY(ar.alloc(&vals2, M));
    SNN_TRY(radix_sort_pairs(keys, vals, keys2, vals2, M, bits_for(2 * (uint64_t)bias), ar, s));
    Moves mv;
    SNN_TRY(ar.alloc(&mv.n, M));
    SNN_TRY(ar.alloc(&mv.from, M));
    SNN_TRY(ar.alloc(&mv.to, M));
    int gm = grid_for(M, 256);
    int64_t *gp, *G;
    int32_t *dv, *nviol;
    SNN_TRY(ar.alloc(&gp, M));
    SNN_TRY(ar.alloc(&dv, M));
    Events ev;
    ev.cap = 2 * (int64_t)M + 2 * deg;
    ev.ibits = bits_for((uint64_t)M);
    SNN_TRY(ar.alloc(&ev.key, ev.cap));
    SNN_TRY(ar.alloc(&ev.idx, ev.cap));
    SNN_TRY(ar.alloc(&ev.dsize, ev.cap));
    SNN_TRY(ar.alloc(&ev.dinp, ev.cap));
    SNN_TRY(ar.alloc(&ev.dpc, ev.cap));
    enqueue(k_moves, std::max(gm, gv), 256, 0, s, M, vals, rho, pto, mv, moveidx, L, ev, gp, dv,
            inc.dirty, savev, inc.pst.save0);
    SNN_CUDA(cudaGetLastError());
    // the hyperedges holding a proposed move
    int64_t nhl = std::max<int64_t>(1, std::min<int64_t>(L.E, deg));
    int32_t* hla;
    int32_t* hln = (int32_t*)(h->d_scal + RS_NHL);
    SNN_TRY(ar.alloc(&hla, nhl));
    enqueue(k_prop_hedges, grid_for((int64_t)M * 32, 256), 256, 0, s, M, mv, L, inc.hmark, hla, hln);
    SNN_CUDA(cudaGetLastError());
    HedgeList hl{hla, hln};
    const int ghl = grid_for(nhl * 32, 256);

    // S9
    prof.reset(new ProfScope(h, PS_REPLAY));
    uint32_t* mvbuf;
    int32_t *hv, *hvc;
    SNN_TRY(ar.alloc(&mvbuf, L.P));
    SNN_TRY(ar.alloc(&hv, L.E));
    SNN_TRY(ar.alloc(&hvc, L.E));
    const bool heavy = X.seg.n[SEG_BB1] + X.seg.n[SEG_BB2] + X.seg.n[SEG_BB3] > 0;
    if (L.E > 0) {
        enqueue(k_replay_warp, ghl, 256, 0, s, L, pc, moveidx, mv, mvbuf, gp, ev, 2 * (int64_t)M, hv,
                hvc, h->d_scal, hl);
        // only a hyperedge of more than REPLAY_WARP_MAX pins holds more moves
        if (heavy)
            enqueue(k_replay_block, 152 * 2, 256, 0, s, L, pc, mv, mvbuf, gp, ev, 2 * (int64_t)M, hv,
                    hvc, h->d_scal);
        SNN_CUDA(cudaGetLastError());
    }
    if (ev.cap <= TAIL_EVENTS) {
        // S10, S11
        prof.reset(new ProfScope(h, PS_VALIDITY));
        enqueue(k_round_tail, 1, SB_THREADS, 0, s, M, ev, ps, prm.omega, prm.delta, prm.phi, gp,
                h->d_scal);
        SNN_CUDA(cudaGetLastError());
    } else {
        prof.reset();
        SNN_TRY(read_scalars(h));
        if (h->h_scal[SC_STATUS] & ST_CAPACITY) return Status{SNNMAP_ERR_CUDA, "event buffer overflow"};
        int64_t T = 2 * (int64_t)M + h->h_scal[RS_NEV];

        // S10
        prof.reset(new ProfScope(h, PS_VALIDITY));
        uint64_t* ekey2;
        uint32_t* eidx2;
        SNN_TRY(ar.alloc(&ekey2, T));
        SNN_TRY(ar.alloc(&eidx2, T));
        int kbits = bits_for((uint64_t)K);
        SNN_TRY(radix_sort_pairs(ev.key, ev.idx, ekey2, eidx2, T, ev.ibits + kbits, ar, s));
        int32_t *pbeg, *pend;
        SNN_TRY(ar.alloc(&pbeg, 2 * (int64_t)K));
        pend = pbeg + K;
        SNN_CUDA(cudaMemsetAsync(pbeg, 0, (size_t)K * 8, s));
        enqueue(k_part_bounds, grid_for(T, 256), 256, 0, s, T, ev.key, ev.ibits, pbeg, pend);
        SNN_CUDA(cudaGetLastError());
        enqueue(k_part_validity, grid_for((int64_t)K * 32, 256), 256, 0, s, K, pbeg, pend, ev, ps,
                prm.omega, prm.delta, prm.phi, dv);
        SNN_CUDA(cudaGetLastError());

        // S11
        prof.reset(new ProfScope(h, PS_APPLY));
        SNN_TRY(ar.alloc(&G, M));
        SNN_TRY(ar.alloc(&nviol, M));
        SNN_TRY(scan_inclusive_i64(gp, G, M, ar, s));
        SNN_TRY(scan_inclusive_i32(dv, nviol, M, ar, s));
        enqueue(k_best1, gm, 256, 0, s, M, G, nviol, h->d_scal);
        enqueue(k_best2, gm, 256, 0, s, M, G, nviol, h->d_scal);
    }
    prof.reset(new ProfScope(h, PS_APPLY));
    // P* of the enacted prefix; when it is short, the rows (k_ps_rows) or the
    // column update after the pin counts below decide the next round's
    // proposals, otherwise the flags of the three rules here do
    enqueue(k_ps_slots, gm, 256, 0, s, M, mv, h->d_scal, inc.pst, inc.dirty);
    SNN_CUDA(cudaGetLastError());
    if (!dense && (!inc.pst.colc || 2 * (int64_t)M > PSTAR_MAX)) {
        SNN_CUDA(cudaMemsetAsync(inc.pchg, 0, (size_t)(K > 0 ? K : 1), s));
        SNN_CUDA(cudaMemsetAsync(inc.prel, 0, (size_t)(K > 0 ? K : 1), s));
        enqueue(k_inc_parts, gm, 256, 0, s, M, mv, h->d_scal, ps, inc.vmax, prm.omega, prm.delta,
                prm.phi, inc.pchg, inc.prel, inc.pst.cnt);
        if (L.E > 0)
            enqueue(k_inc_hedges, grid_for((int64_t)L.E * 32, 256), 256, 0, s, L, pc, moveidx, mv,
                    h->d_scal, inc.prel, mvbuf, inc.dirty, inc.pst.cnt);
        enqueue(k_inc_targets, gv, 256, 0, s, V, pto, inc.pchg, inc.dirty, inc.pst.cnt);
        SNN_CUDA(cudaGetLastError());
    }
    // carried pin counts: take out the hyperedges the prefix touches (old
    // counts, old rho; on levels with rows the pass updates those as well, the
    // stage "cross"), move, count them again, add them back
    prof.reset(new ProfScope(h, dense ? PS_CROSS : PS_PINCOUNT));
    if (L.E > 0) {
        RowsRef R{dense ? D.rowid : nullptr, D.tab, D.M, D.cw};
        enqueue(k_prefix_hedges, ghl, 256, 0, s, L, pc, moveidx, mv, h->d_scal, R, mvbuf, inc.hdirty,
                rho, ps, savev, inc.costv, hl);
        SNN_CUDA(cudaGetLastError());
    }
    if (dense) prof.reset(new ProfScope(h, PS_PINCOUNT));
    enqueue(k_apply, gm, 256, 0, s, M, mv, L, h->d_scal, ps, rho, moveidx);
    SNN_CUDA(cudaGetLastError());
    if (L.E > 0) {
        PinCountJob job{L.hoff, L.hpins, L.hsd, L.hk, L.hw, rho, pc, ps.pincnt, inc.costv};
        job.cost_mask = 0;
        if (nhl <= RECOUNT_MAX && X.seg.n[SEG_BB2] + X.seg.n[SEG_BB3] == 0) {
            enqueue(k_prefix_recount, ghl, 256, 0, s, L, job, rho, savev, inc.hmark, inc.hdirty, hl);
        } else {
            SNN_CUDA(cudaMemsetAsync(inc.hmeta, 0, 2 * SEG_NB * sizeof(int32_t), s));
            enqueue(k_seg_meta_copy, 1, 32, 0, s, X.seg.meta, inc.hmeta);
            enqueue(k_seg_filter, grid_for(L.E, 256), 256, 0, s, X.seg.list, X.seg.meta, L.E,
                    inc.hdirty, inc.hlist, inc.hmeta);
            SNN_CUDA(cudaGetLastError());
            SegBuckets db = X.seg;
            db.list = inc.hlist;
            db.meta = inc.hmeta;
            int64_t* slots;
            SNN_TRY(ar.alloc(&slots, COST_SLOTS));
            SNN_CUDA(cudaMemsetAsync(slots, 0, COST_SLOTS * sizeof(int64_t), s));
            job.cost = slots;
            job.cost_mask = COST_SLOTS - 1;
            SNN_TRY(seg_run(job, db, L.E, ar, s));
            enqueue(k_cost_slots, 1, 256, 0, s, slots, inc.costv);
            enqueue(k_prefix_saves, ghl, 256, 0, s, L, pc, rho, savev, inc.hmark, inc.hdirty, hl);
        }
        SNN_CUDA(cudaGetLastError());
    }
    if (!dense) {
        prof.reset(new ProfScope(h, PS_GAINS));
        if (inc.pst.colc && V > 0) {
            if (L.P <= PS_MARK_PINS) {
                SNN_HEDGE_LAUNCH(hedge_lanes(L.P, 2 * (int64_t)L.E), k_ps_mark_counts, L.E, s, L, pc,
                                 h->d_scal, inc.pst);
            } else {
                enqueue(k_ps_mark, grid_for(V, 256), 256, 0, s, L, rho, h->d_scal, inc.pst);
            }
            enqueue(k_ps_cols, 152 * 8, 256, 0, s, L, pc, rho, h->d_scal, inc.pst);
            enqueue(k_ps_combine, gv, 256, 0, s, L, rho, h->d_scal, inc.pst, ps, savev, Wv, prm.omega,
                    prm.delta, prm.phi, prm.refine_nonpositive, pto, pgain, inc.dirty);
        }
        enqueue(k_ps_reset, gm, 256, 0, s, M, mv, h->d_scal, inc.pst, host);
        SNN_CUDA(cudaGetLastError());
    } else {
        prof.reset(new ProfScope(h, PS_GAINS));
        if (V > 0)
            enqueue(k_ps_rows, gv, 256, 0, s, L, rho, h->d_scal, inc.pst, ps, savev, Wv, D.rowid,
                    D.tab, prm.omega, prm.delta, prm.phi, prm.refine_nonpositive, pto, pgain, inc.dirty);
        enqueue(k_ps_reset, gm, 256, 0, s, M, mv, h->d_scal, inc.pst, host);
        SNN_CUDA(cudaGetLastError());
    }
    prof.reset();
    SNN_CUDA(cudaStreamSynchronize(s));
    if (host[HW_STATUS] & ST_CAPACITY) return Status{SNNMAP_ERR_CUDA, "event buffer overflow"};
    int64_t best = host[HW_BEST];
    int64_t istar = host[HW_ISTAR];
    if (best > 0 && istar < M) {
        *applied = (int32_t)(istar + 1);
        *gain = best;
    }
    return Status{};
}

__global__ void k_check_rho(int32_t V, const int32_t* __restrict__ rho, int32_t K, int64_t* scal)
{
    after_previous();
    int bad = 0;
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < V;
         n += (int64_t)gridDim.x * blockDim.x)
        if (rho[n] < 0 || rho[n] >= K) bad = 1;
    if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0) atomicOr((int*)&scal[SC_STATUS], ST_INVALID);
}

Status check_rho(snnmap_hgraph* h, int32_t level, int32_t K, const int32_t* rho)
{
    Level& L = h->levels[level];
    SNN_TRY(zero_scalars(h));
    if (L.V > 0) {
        enqueue(k_check_rho, grid_for(L.V, 256), 256, 0, h->stream, L.V, rho, K, h->d_scal);
        SNN_CUDA(cudaGetLastError());
    }
    SNN_TRY(read_scalars(h));
    if (h->h_scal[SC_STATUS] & ST_INVALID) return Status{SNNMAP_ERR_INVALID, "rho value outside [0, n_parts)"};
    return Status{};
}

// Proposals carried to the next finer level: an unmatched vertex keeps its
// super-node's proposal, gain and flag (its conn, overlap, save, W and the
// partition state are unchanged by projection); both members of a pair are
// evaluated.
__global__ void k_carry(int32_t V, const int32_t* __restrict__ cid, const uint8_t* __restrict__ pr,
                        const int32_t* __restrict__ pto_c, const int64_t* __restrict__ pgain_c,
                        const int32_t* __restrict__ dirty_c, int32_t* pto, int64_t* pgain,
                        int32_t* dirty)
{
    after_previous();
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < V;
         n += (int64_t)gridDim.x * blockDim.x) {
        int32_t c = cid[n];
        pto[n] = pto_c[c];
        pgain[n] = pgain_c[c];
        dirty[n] = (pr[n] || dirty_c[c]) ? 1 : 0;
    }
}

Status carry_open(snnmap_hgraph* h, int64_t cap)
{
    carry_close(h);
    Carry& C = h->carry;
    size_t n = (size_t)(cap > 0 ? cap : 1);
    for (int b = 0; b < 2; b++) {
        SNN_CUDA(dev_malloc(&C.pto[b], n * 4, h->stream));
        SNN_CUDA(dev_malloc(&C.pgain[b], n * 8, h->stream));
        SNN_CUDA(dev_malloc(&C.dirty[b], n * 4, h->stream));
        SNN_CUDA(dev_malloc(&C.save[b], n * 16, h->stream));
    }
    C.cap = cap;
    C.level = -1;
    C.slevel = -1;
    C.cur = 0;
    return Status{};
}

void carry_close(snnmap_hgraph* h)
{
    Carry& C = h->carry;
    for (int b = 0; b < 2; b++)
        for (void* p : {(void*)C.pto[b], (void*)C.pgain[b], (void*)C.dirty[b], (void*)C.save[b]})
            if (p) cudaFreeAsync(p, h->stream);
    C = Carry{};
}

// Saves and W inherited from the next coarser level (cid null: none). An
// unmatched vertex keeps its super-node's: its hyperedges map one to one onto
// that super-node's with the same summed omega, and it is its partition's last
// pin in the same ones. The members of pairs are listed and computed from
// their hyperedges (k_save_members), which took every vertex before.
struct SaveIn {
    const int32_t* cid;
    const uint8_t* pr;
    const int64_t *sc, *wc;
    int64_t *save, *W;
    int32_t *mlist, *mcnt;
};

// no move listed, every vertex to evaluate (unless inherited), no slot taken,
// saves inherited
__global__ void k_refine_init(int32_t V, int32_t K, int32_t* moveidx, int32_t* dirty, PStar ps,
                              int32_t base, SaveIn si)
{
    after_previous();
    int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t n = t0; n < V; n += step) {
        moveidx[n] = -1;
        if (dirty) dirty[n] = 1;
        if (si.cid) {
            bool pair = si.pr[n] != 0;
            int32_t c = si.cid[n];
            si.save[n] = pair ? 0 : si.sc[c];
            si.W[n] = pair ? 0 : si.wc[c];
            if (pair) si.mlist[atomicAdd(si.mcnt, 1)] = (int32_t)n;
        }
    }
    for (int64_t p = t0; p < K; p += step) ps.pslot[p] = -1;
    if (t0 < 4) ps.cnt[t0] = (t0 & 1) ? 0 : base;
}

Status refine_level(snnmap_hgraph* h, int32_t level, int32_t K, int32_t* rho, int64_t* cost,
                    int64_t* cost_start)
{
    Level& L = h->levels[level];
    cudaStream_t s = h->stream;
    int32_t* moveidx;
    IncState inc;
    PStar& pst = inc.pst;
    Carry& CA = h->carry;
    const bool dense_level = h->dense.level == level;
    const bool use_carry = CA.pto[0] && L.V <= CA.cap;
    const int64_t V = L.V, E = L.E;
    bool inherited = false;
    // the level's buffers, one allocation: the cleared ones first
    Carver cv;
    cv.add(&inc.hdirty, E);
    cv.add(&inc.hmark, E);
    cv.add(&inc.vmax, 3);
    cv.add(&inc.ps.size, K);
    cv.add(&inc.ps.inpins, K);
    cv.add(&inc.ps.pincnt, K);
    cv.add(&inc.slots, COST_SLOTS);
    // the members of pairs walk their incidence lists: while they are few. Pass
    // of the 1,048,576-neuron conv network: 585 ms with at most a quarter of the
    // vertices in pairs, 591 with all, 595 with a 32nd
    const bool inherit_save =
        use_carry && CA.slevel == level + 1 && 8 * (V - h->levels[level + 1].V) <= V;
    if (inherit_save) cv.add(&inc.mcnt, 1);
    if (!use_carry) {
        cv.add(&inc.savev, V);
        cv.add(&inc.Wv, V);
    }
    const size_t cleared = cv.total;
    cv.add(&moveidx, V);
    if (inherit_save) cv.add(&inc.mlist, 2 * (V - h->levels[level + 1].V));
    if (!use_carry) {
        cv.add(&inc.pto, V);
        cv.add(&inc.pgain, V);
        cv.add(&inc.dirty, V);
    }
    cv.add(&inc.pchg, K);
    cv.add(&inc.prel, K);
    cv.add(&inc.pc.p, L.P);
    cv.add(&inc.pc.cnt, L.P);
    cv.add(&inc.pc.dcnt, L.P);
    cv.add(&inc.pc.lam, E);
    cv.add(&inc.pc.rec, E);
    cv.add(&inc.costv, 1);
    cv.add(&inc.hlist, E);
    cv.add(&inc.hmeta, 2 * SEG_NB);
    cv.add(&pst.pslot, K);
    cv.add(&pst.slots, PSTAR_MAX);
    cv.add(&pst.cnt, 4);
    void* block = nullptr;
    SNN_CUDA(dev_malloc(&block, cv.total, s));
    cv.assign(block);
    // optional buffers. Rows levels need only the round-start saves besides
    // the slot map; the others the columns too: without them every round
    // takes the flag rules
    Carver co;
    size_t ccleared = 0;
    if (!dense_level) {
        co.add(&pst.hmask, E);
        co.add(&pst.vt, V);
        co.add(&pst.colc, (int64_t)PSTAR_MAX * V);
        co.add(&pst.colo, (int64_t)PSTAR_MAX * V);
        ccleared = co.total;
        co.add(&pst.hl, E);
    }
    co.add(&pst.save0, V);
    void* cols = nullptr;
    if (dev_malloc(&cols, co.total, s) == cudaSuccess) {
        co.assign(cols);
    } else {
        cudaGetLastError();
        cols = nullptr;
    }
    const int64_t mine = (int64_t)(cv.total + (cols ? co.total : 0));
    h->call_bytes += mine;
    auto give_back = [&]() {
        note_bytes(h);
        h->call_bytes -= mine;
        cudaFreeAsync(block, s);
        if (cols) cudaFreeAsync(cols, s);
    };
    SaveIn si{};
    auto setup = [&]() -> Status {
        SNN_CUDA(cudaMemsetAsync(block, 0, cleared, s));
        if (cols && ccleared) SNN_CUDA(cudaMemsetAsync(cols, 0, ccleared, s));
        if (use_carry) {
            int nb = 1 - CA.cur;
            inc.pto = CA.pto[nb];
            inc.pgain = CA.pgain[nb];
            inc.dirty = CA.dirty[nb];
            inc.savev = CA.save[nb];
            inc.Wv = CA.save[nb] + V;
            if (inherit_save) {
                inc.members = 2 * (V - h->levels[level + 1].V);
                const int64_t* from = CA.save[CA.cur];
                si = SaveIn{L.cid, L.pr, from, from + h->levels[level + 1].V, inc.savev, inc.Wv,
                            inc.mlist, inc.mcnt};
            } else {
                SNN_CUDA(cudaMemsetAsync(inc.savev, 0, (size_t)V * 16, s));
            }
            CA.slevel = -1;
            if (!dense_level && CA.level == level + 1 && L.V > 0) {
                enqueue(k_carry, grid_for(L.V, 256), 256, 0, s, L.V, L.cid, L.pr, CA.pto[CA.cur],
                        CA.pgain[CA.cur], CA.dirty[CA.cur], inc.pto, inc.pgain, inc.dirty);
                SNN_CUDA(cudaGetLastError());
                inherited = true;
            }
            CA.cur = nb;
            CA.level = -1;
        }
        // without the saves (and columns) the column update stays off
        enqueue(k_refine_init, grid_for(std::max<int64_t>(V, K), 256), 256, 0, s, L.V, K, moveidx,
                inherited ? nullptr : inc.dirty, pst, cols ? 0 : (1 << 30), si);
        if (!dense_level && L.V > 0) enqueue(k_level_max, grid_for(L.V, 256, 152 * 4), 256, 0, s, L,
                                             inc.vmax);
        SNN_CUDA(cudaGetLastError());
        return Status{};
    };
    Status st = setup();
    int64_t c = 0;
    bool have_cost = false;
    for (int32_t r = 0; st.ok() && r < h->prm.max_refine_rounds; r++) {
        int32_t props = 0, applied = 0, act = 0, rows = 0;
        int64_t g = 0, c0 = 0;
        st = refine_round(h, level, K, rho, moveidx, inc, &props, &applied, &g, &c0, &act, &rows);
        inc.ready = true;
        h->scratch.reset();
        if (!st.ok()) break;
        h->rlog.push_back(snnmap_round_log{level, r, props, applied, act, rows, g});
        if (!have_cost && cost_start) *cost_start = c0;
        c = c0 - g;
        have_cost = true;
        if (applied == 0) break;
    }
    give_back();
    if (use_carry && st.ok() && inc.ready) CA.slevel = level;   // saves, for the next finer level
    if (use_carry && st.ok() && !dense_level)
        CA.level = level;   // the next finer level may inherit these proposals
    if (!st.ok()) return st;
    if (!have_cost) {
        SNN_TRY(level_cost(h, level, K, rho, &c));
        if (cost_start) *cost_start = c;
    }
    *cost = c;
    return Status{};
}

}  // namespace snn
