// Neighbour scores as a dense matrix for the coarsening levels with few
// vertices (Sec. 4.1, Coarsening; Eq. neigh_histogram).
//
// When a level has at most about sqrt(budget / 16) vertices and few of them
// against its pair count (see mat_fits), score(n, m)
// (summed omega over hyperedges holding both) and the shared inbound count
// ov(n, m) (summed k over hyperedges where both are destinations) are kept
// for every pair in V x V int32 matrices. The candidate of n is then a scan
// of row n with the validity test of the histogram path, instead of a
// histogram over n's neighbourhood.
//
// Contraction keeps the entries of two unmatched vertices exact: their
// common hyperedges map one to one onto common hyperedges of the coarse
// level with the same summed omega and k and the same destination roles (a
// hyperedge can only vanish if all its pins fall into one super-node). So
// the next level's matrix is a gather of the previous one at the
// representatives, plus fresh rows (a histogram, ScorePol) for the merged
// super-nodes, stored into their columns as well.
#include "histo.cuh"
#include "internal.cuh"

namespace snn {

template <typename S_>
struct ScorePol {
    using S = S_;
    static constexpr bool kOptimistic = false;
    static constexpr bool kMasks = false;
    struct Acc {
        __device__ Acc() {}
        __device__ void add(const Acc&) {}
        __device__ void atomic_into(Acc*) const {}
    };
    static __device__ Acc warp_reduce(const Acc& a) { return a; }

    Level L;
    int32_t V;
    int64_t keys;
    const int32_t* fresh;   // rows to compute (null: every vertex)
    int32_t* Sm;
    int32_t* OVm;
    int64_t Vs;

    __device__ bool skip(int32_t n) const { return fresh && !fresh[n]; }
    __device__ int64_t vb(int32_t n) const { return L.voff[n]; }
    __device__ int64_t ve(int32_t n) const { return L.voff[n + 1]; }
    __device__ int64_t seg_len(int64_t i) const
    {
        int32_t a = (int32_t)((uint32_t)L.vinc[i] & ~SRC_BIT);
        return L.hoff[a + 1] - L.hoff[a];
    }
    __device__ uint32_t inc(int64_t i) const { return (uint32_t)L.vinc[i]; }
    __device__ void fetch(uint32_t inc) const
    {
        int32_t a = (int32_t)(inc & ~SRC_BIT);
        prefetch_l1(L.hoff + a);
        prefetch_l1(L.hw + a);
        prefetch_l1(L.hk + a);
        prefetch_l1(L.hsd + a);
    }
    __device__ Seg<S> seg(uint32_t inc, Acc&) const
    {
        int32_t a = (int32_t)(inc & ~SRC_BIT);
        Seg<S> g;
        g.sd = L.hsd[a];
        g.nd = !(inc & SRC_BIT) || g.sd;
        g.b = L.hoff[a];
        g.len = (int32_t)(L.hoff[a + 1] - g.b);
        g.w = (S)L.hw[a];
        g.k = (uint32_t)L.hk[a];
        return g;
    }
    struct Item {
        int32_t m;
        S w;
        uint32_t o;
    };
    static __device__ Item none() { return Item{-1, 0, 0u}; }
    struct Own {};
    __device__ Own own(int32_t) const { return Own{}; }
    __device__ Item load(int32_t n, const Own&, const Seg<S>& g, int32_t off) const
    {
        int32_t m = L.hpins[g.b + off];
        int md = off != 0 || g.sd;   // pin 0 is the source
        return Item{m == n ? -1 : m, g.w, (g.nd && md) ? g.k : 0u};
    }
    template <class Tb>
    __device__ bool put(int32_t, const Item& it, const Tb& t, Acc&) const
    {
        return it.m < 0 || t.add(it.m, it.w, it.o);
    }
    // every neighbour lands in the row and, mirrored, in the column (stores: a
    // vertex redone by a later tier overwrites its partial entries)
    __device__ void consider(int32_t n, int32_t m, int64_t s, uint32_t o, const Acc&, int64_t&,
                             int32_t&, uint32_t&) const
    {
        int64_t r = (int64_t)n * Vs + m, c = (int64_t)m * Vs + n;
        Sm[r] = Sm[c] = (int32_t)s;
        OVm[r] = OVm[c] = (int32_t)o;
    }
    __device__ void write(int32_t, int64_t, int32_t, uint32_t, const Acc&) const {}
};

// candidate of n: the valid neighbour with the largest score, ties to the
// lower id (the rules of the histogram path; its skip of vertices that cannot
// merge even with the smallest vertex finds nothing valid here either). A
// warp per row. What bounds it on late levels (2,500 vertices, a matrix that
// the L2 cache holds) is latency: MB_FLY loads a lane are in flight, and of
// their entries one state is read, the largest's (testing each larger entry
// as it came was a chain of gathers: 28.0 us a level of the conv network of
// 65,536 neurons, 13.2 so).
constexpr int MB_FLY = 4;

__global__ void __launch_bounds__(256)
    k_mat_best(Level L, const int32_t* __restrict__ Sm,
               const int32_t* __restrict__ OVm, int64_t Vs, int32_t omega, int32_t delta,
               int32_t phi, int32_t* cand, int64_t* cscore, int32_t* cov)
{
    after_previous();
    int lane = threadIdx.x & 31;
    int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t n = gw; n < L.V; n += nw) {
        int64_t sz = L.vsize[n], ip = L.vinpins[n], ic = L.vincnt[n];
        int64_t r0 = n * Vs;
        int64_t bs = 0;
        int32_t bk = -1;
        {
            const int4* row = reinterpret_cast<const int4*>(Sm + r0);
            for (int64_t q0 = lane; 4 * q0 < L.V; q0 += 32 * MB_FLY) {
                int4 c4[MB_FLY];
#pragma unroll
                for (int f = 0; f < MB_FLY; f++) {
                    int64_t q = q0 + 32 * f;
                    c4[f] = 4 * q < L.V ? row[q] : make_int4(0, 0, 0, 0);
                }
                for (;;) {
                    // the largest entry above the best so far, the first of
                    // equals, and only its state is read
                    int32_t top = 0, m = -1;
#pragma unroll
                    for (int f = 0; f < MB_FLY; f++) {
                        const int cv[4] = {c4[f].x, c4[f].y, c4[f].z, c4[f].w};
#pragma unroll
                        for (int u = 0; u < 4; u++) {
                            int32_t mm = (int32_t)(4 * (q0 + 32 * f) + u);
                            if (cv[u] > top && mm != n && mm < L.V) {
                                top = cv[u];
                                m = mm;
                            }
                        }
                    }
                    if (m < 0 || top <= bs) break;
                    const int32_t ms = L.vsize[m], mp = L.vinpins[m], mc = L.vincnt[m], mo = OVm[r0 + m];
                    if (sz + ms <= omega && ip + mp <= phi && ic + mc - (int64_t)mo <= delta) {
                        bs = top;
                        bk = m;
                        break;
                    }
                    // it cannot take n: the next one
                    const int32_t e = m - (int32_t)(4 * q0);
#pragma unroll
                    for (int f = 0; f < MB_FLY; f++) {
                        if (e == 128 * f) c4[f].x = 0;
                        if (e == 128 * f + 1) c4[f].y = 0;
                        if (e == 128 * f + 2) c4[f].z = 0;
                        if (e == 128 * f + 3) c4[f].w = 0;
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
        }
        if (lane == 0) {
            cand[n] = bk;
            cscore[n] = bk < 0 ? 0 : bs;
            cov[n] = bk < 0 ? 0 : OVm[r0 + bk];
        }
    }
}

// coarse vertex cid(n)'s representative (its smaller member) and whether it
// merged two vertices
__global__ void k_mat_reps(int32_t V, const int32_t* __restrict__ cid,
                           const int32_t* __restrict__ match, int32_t* repof, int32_t* fresh)
{
    after_previous();
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < V;
         n += (int64_t)gridDim.x * blockDim.x) {
        int32_t m = match[n];
        if (m >= 0 && m < (int32_t)n) continue;
        repof[cid[n]] = (int32_t)n;
        fresh[cid[n]] = m >= 0;
    }
}

// S2[i][j] = S[rep(i)][rep(j)] (one block per row); rows and columns of
// merged vertices are cleared for their fresh sums
__global__ void __launch_bounds__(256)
    k_mat_gather(int32_t V2, const int32_t* __restrict__ repof, const int32_t* __restrict__ fresh,
                 const int32_t* __restrict__ Sm,
                 const int32_t* __restrict__ OVm, int64_t Vs, int32_t* S2, int32_t* OV2, int64_t Vs2)
{
    after_previous();
    for (int64_t i = blockIdx.x; i < V2; i += gridDim.x) {
        int64_t src = (int64_t)repof[i] * Vs;
        int64_t dst = i * Vs2;
        if (fresh[i]) {
            for (int64_t j0 = 4 * threadIdx.x; j0 < Vs2; j0 += 4 * blockDim.x) {
                *reinterpret_cast<int4*>(S2 + dst + j0) = make_int4(0, 0, 0, 0);
                *reinterpret_cast<int4*>(OV2 + dst + j0) = make_int4(0, 0, 0, 0);
            }
            continue;
        }
        // Vs2 is V2 up to a multiple of four: quads of entries, the gathers of
        // one in flight together
        for (int64_t j0 = 4 * threadIdx.x; j0 < Vs2; j0 += 4 * blockDim.x) {
            int sv[4], ov[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                bool keep = j0 + u < V2 && !fresh[j0 + u];
                int64_t c = keep ? src + repof[j0 + u] : src;
                sv[u] = keep ? Sm[c] : 0;
                ov[u] = keep ? OVm[c] : 0;
            }
            *reinterpret_cast<int4*>(S2 + dst + j0) = make_int4(sv[0], sv[1], sv[2], sv[3]);
            *reinterpret_cast<int4*>(OV2 + dst + j0) = make_int4(ov[0], ov[1], ov[2], ov[3]);
        }
    }
}

static Status mat_rows(snnmap_hgraph* h, const Level& L, const int32_t* fresh)
{
    ScoreMat& M = h->mat;
    ScorePol<uint32_t> pol;
    pol.L = L;
    pol.V = L.V;
    pol.keys = L.V;
    pol.fresh = fresh;
    pol.Sm = M.S;
    pol.OVm = M.OV;
    pol.Vs = M.Vs;
    int64_t* cnt;
    SNN_TRY(h->scratch.alloc(&cnt, HT_NCNT));
    return run_histogram(pol, h->scratch, h->stream, cnt, h->h_scal + 12, h->tiers, L.V,
                         !h->wzero);
}

void mat_close(snnmap_hgraph* h)
{
    ScoreMat& M = h->mat;
    for (int32_t* p : {M.S, M.OV, M.S2, M.OV2})
        if (p) cudaFreeAsync(p, h->stream);
    M = ScoreMat{};
}

// The matrix is entered on a level when it fits the budget and pays: one
// level costs about 24 V^2 bytes of HBM traffic (gather 16, scan 8) against
// the histogram's pair_terms hash updates, which run roughly five times
// slower per item than bytes stream; so V^2 <= 5 * pair_terms. Once entered
// it stays (V shrinks while pair_terms barely does).
static bool mat_fits(const snnmap_hgraph* h, int32_t level)
{
    if (h->wide || h->wzero || h->wsum > INT32_MAX) return false;
    int64_t Vs = ((int64_t)h->levels[level].V + 3) & ~(int64_t)3;
    return 16 * Vs * Vs <= dense_row_budget(h) &&
           (double)Vs * (double)Vs <= 5.0 * (double)h->extra[level].pair_terms;
}

Status mat_affinity(snnmap_hgraph* h, int32_t level, bool* done)
{
    *done = false;
    ScoreMat& M = h->mat;
    const Level& L = h->levels[level];
    cudaStream_t s = h->stream;
    if (M.level != level) {
        mat_close(h);
        if (!mat_fits(h, level)) return Status{};
        int64_t Vs = ((int64_t)L.V + 3) & ~(int64_t)3;
        size_t bytes = (size_t)(Vs * Vs) * 4;
        cudaError_t e = dev_malloc(&M.S, bytes, s);
        if (e == cudaSuccess) e = dev_malloc(&M.OV, bytes, s);
        if (e == cudaSuccess) e = dev_malloc(&M.S2, bytes, s);
        if (e == cudaSuccess) e = dev_malloc(&M.OV2, bytes, s);
        if (e != cudaSuccess) {
            // no room: this level and the next ones use histograms
            cudaGetLastError();
            mat_close(h);
            return Status{};
        }
        M.cap = Vs * Vs;
        M.Vs = Vs;
        SNN_CUDA(cudaMemsetAsync(M.S, 0, bytes, s));
        SNN_CUDA(cudaMemsetAsync(M.OV, 0, bytes, s));
        SNN_TRY(mat_rows(h, L, nullptr));
        M.level = level;
    }
    if (L.V > 0) {
        enqueue(k_mat_best, grid_for((int64_t)L.V * 32, 256), 256, 0, s, L, M.S, M.OV, M.Vs,
                h->prm.omega, h->prm.delta, h->prm.phi, h->cand, h->cscore, h->cov);
        SNN_CUDA(cudaGetLastError());
    }
    h->extra[level].n_block = 0;
    h->extra[level].n_global = 0;
    h->extra[level].carried = 2;
    h->extra[level].n_full = 0;
    h->extra[level].hist_work = 0;
    *done = true;
    return Status{};
}

Status mat_descend(snnmap_hgraph* h, int32_t src)
{
    ScoreMat& M = h->mat;
    if (M.level != src) return Status{};
    const Level& F = h->levels[src];
    const Level& L = h->levels[src + 1];
    cudaStream_t s = h->stream;
    Arena& ar = h->scratch;
    int64_t Vs2 = ((int64_t)L.V + 3) & ~(int64_t)3;
    if (Vs2 * Vs2 > M.cap) {
        mat_close(h);
        return Status{};
    }
    int32_t *repof, *fresh;
    SNN_TRY(ar.alloc(&repof, L.V));
    SNN_TRY(ar.alloc(&fresh, L.V));
    if (F.V > 0) {
        enqueue(k_mat_reps, grid_for(F.V, 256), 256, 0, s, F.V, F.cid, h->match, repof, fresh);
        SNN_CUDA(cudaGetLastError());
    }
    if (L.V > 0) {
        enqueue(k_mat_gather, (int)std::min<int64_t>(L.V, 152 * 16), 256, 0, s, L.V, repof, fresh, M.S,
                M.OV, M.Vs, M.S2, M.OV2, Vs2);
        SNN_CUDA(cudaGetLastError());
    }
    std::swap(M.S, M.S2);
    std::swap(M.OV, M.OV2);
    M.Vs = Vs2;
    if (L.V > 0) {
        SNN_TRY(mat_rows(h, L, fresh));
    }
    M.level = src + 1;
    return Status{};
}

}  // namespace snn
