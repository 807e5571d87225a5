// Device-wide primitives: scratch arena, prefix scans and a stable LSD radix
// sort. Everything here is deterministic (no atomics on values whose order
// matters, no spin waits): the scans of scan.cuh, and for the sort a
// per-tile digit histogram, a scan of the digit-major histogram table and a
// stable scatter whose in-tile ranks come from warp match_any groups; short
// sorts run all their passes in one launch of one thread block cluster.
#include "common.cuh"
#include "scan.cuh"

#include <atomic>
#include <climits>
#include <mutex>

namespace snn {

static std::atomic<int64_t> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
int64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }

// ---------------------------------------------------------------------------
// Pool-backed device allocations

namespace {
constexpr int kMaxPoolDevices = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pools[kMaxPoolDevices] = {};
int g_live_handles = 0;
}  // namespace

static cudaError_t pool_of(int dev, cudaMemPool_t* out)
{
    if (dev < 0 || dev >= kMaxPoolDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pools[dev]) {
        cudaMemPoolProps pr{};
        pr.allocType = cudaMemAllocationTypePinned;
        pr.handleTypes = cudaMemHandleTypeNone;
        pr.location.type = cudaMemLocationTypeDevice;
        pr.location.id = dev;
        cudaMemPool_t p = nullptr;
        cudaError_t e = cudaMemPoolCreate(&p, &pr);
        if (e != cudaSuccess) return e;
        uint64_t keep = UINT64_MAX;
        e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        // handles on other streams (the batched and served forms) reuse
        // freed blocks only once their frees are known complete: no wait is
        // ever inserted between their streams
        int no = 0;
        if (e == cudaSuccess)
            e = cudaMemPoolSetAttribute(p, cudaMemPoolReuseAllowInternalDependencies, &no);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return e;
        }
        g_pools[dev] = p;
    }
    *out = g_pools[dev];
    return cudaSuccess;
}

cudaError_t dev_malloc(void** p, size_t bytes, cudaStream_t s)
{
    int dev = -1;
    cudaError_t e = cudaStreamGetDevice(s, &dev);
    if (e != cudaSuccess) return e;
    cudaMemPool_t pool = nullptr;
    e = pool_of(dev, &pool);
    if (e != cudaSuccess) return e;
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

int pool_handles(int delta)
{
    std::lock_guard<std::mutex> lk(g_pool_mu);
    g_live_handles += delta;
    if (g_live_handles < 0) g_live_handles = 0;
    if (g_live_handles == 0)
        for (cudaMemPool_t p : g_pools)
            if (p) cudaMemPoolTrimTo(p, 0);
    return g_live_handles;
}

cudaError_t pool_high(int dev, uint64_t* bytes)
{
    cudaMemPool_t pool = nullptr;
    cudaError_t e = pool_of(dev, &pool);
    if (e == cudaSuccess) e = cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemHigh, bytes);
    uint64_t zero = 0;
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrUsedMemHigh, &zero);
    return e;
}

// ---------------------------------------------------------------------------
// Arena

Status Arena::reserve(size_t bytes)
{
    if (!chunks.empty() && sizes.back() >= bytes && chunks.size() == 1) return Status{};
    release();
    void* p = nullptr;
    SNN_CUDA(dev_malloc(&p, bytes, stream));
    chunks.push_back(p);
    sizes.push_back(bytes);
    used = 0;
    return Status{};
}

Status Arena::take(size_t bytes, void** out)
{
    bytes = (bytes + 255) & ~(size_t)255;
    step_total += bytes;
    if (chunks.empty() || used + bytes > sizes.back()) {
        size_t want = bytes;
        if (chunks.empty() && peak > want) want = peak;
        if (want < ((size_t)64 << 20)) want = (size_t)64 << 20;
        void* p = nullptr;
        SNN_CUDA(dev_malloc(&p, want, stream));
        chunks.push_back(p);
        sizes.push_back(want);
        used = 0;
        if (held() > high) high = held();
    }
    *out = (char*)chunks.back() + used;
    used += bytes;
    return Status{};
}

void Arena::reset()
{
    if (step_total > peak) peak = step_total;
    if (chunks.size() > 1) {
        // consolidate: next step gets one chunk as large as this step needed
        for (void* p : chunks) cudaFreeAsync(p, stream);
        chunks.clear();
        sizes.clear();
        void* p = nullptr;
        size_t want = peak + ((size_t)16 << 20);
        if (dev_malloc(&p, want, stream) == cudaSuccess) {
            chunks.push_back(p);
            sizes.push_back(want);
        }
    }
    used = 0;
    step_total = 0;
}

void Arena::rewind(const Mark& m)
{
    if (step_total > peak) peak = step_total;
    while (chunks.size() > m.nchunks && !chunks.empty()) {
        cudaFreeAsync(chunks.back(), stream);
        chunks.pop_back();
        sizes.pop_back();
    }
    used = m.used;
    step_total = m.step_total;
}

void Arena::release()
{
    for (void* p : chunks) cudaFreeAsync(p, stream);
    chunks.clear();
    sizes.clear();
    used = 0;
}

size_t Arena::held() const
{
    size_t t = 0;
    for (size_t s : sizes) t += s;
    return t;
}

// ---------------------------------------------------------------------------
// Fills

template <typename T>
__global__ void k_fill(T* p, T v, int64_t n)
{
    after_previous();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

__global__ void k_iota(int32_t* p, int64_t n)
{
    after_previous();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        p[i] = (int32_t)i;
}

Status fill_i32(int32_t* p, int32_t v, int64_t n, cudaStream_t s)
{
    if (n <= 0) return Status{};
    enqueue(k_fill<int32_t>, grid_for(n, 256), 256, 0, s, p, v, n);
    SNN_CUDA(cudaGetLastError());
    return Status{};
}

Status iota_i32(int32_t* p, int64_t n, cudaStream_t s)
{
    if (n <= 0) return Status{};
    enqueue(k_iota, grid_for(n, 256), 256, 0, s, p, n);
    SNN_CUDA(cudaGetLastError());
    return Status{};
}

// ---------------------------------------------------------------------------
// Scans of plain arrays (scan.cuh)

namespace {

// running maximum as a "sum"
struct Max32 {
    int32_t v;
    __device__ Max32() : v(INT_MIN) {}
    __device__ explicit Max32(int32_t x) : v(x) {}
    __device__ Max32 operator+(const Max32& o) const { return Max32(v > o.v ? v : o.v); }
};
__device__ __forceinline__ Max32 scan_shfl_up(Max32 x, int o)
{
    return Max32(__shfl_up_sync(FULL, x.v, o));
}
__device__ __forceinline__ Max32 scan_shfl(Max32 x, int src)
{
    return Max32(__shfl_sync(FULL, x.v, src));
}
struct Max32Store {
    int32_t* p;
    __device__ void operator()(int64_t i, Max32 ex, Max32 x) const { p[i] = (ex + x).v; }
};

template <typename Tin, typename T, bool INCL>
Status scan_plain(const Tin* in, T* out, int64_t n, T* total, Arena& ar, cudaStream_t s)
{
    return scan_run<T>(ScanLoad<Tin, T>{in}, ScanStore<T, INCL>{out}, n, total, ar, s);
}

}  // namespace

Status scan_exclusive_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, int64_t* total,
                                 Arena& ar, cudaStream_t s)
{
    return scan_plain<int32_t, int64_t, false>(in, out, n, total, ar, s);
}

Status scan_exclusive_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* total, Arena& ar,
                          cudaStream_t s)
{
    return scan_plain<int64_t, int64_t, false>(in, out, n, total, ar, s);
}

Status scan_exclusive_i32(const int32_t* in, int32_t* out, int64_t n, int32_t* total, Arena& ar,
                          cudaStream_t s)
{
    return scan_plain<int32_t, int32_t, false>(in, out, n, total, ar, s);
}

Status scan_inclusive_i64(const int64_t* in, int64_t* out, int64_t n, Arena& ar, cudaStream_t s)
{
    return scan_plain<int64_t, int64_t, true>(in, out, n, (int64_t*)nullptr, ar, s);
}

Status scan_inclusive_i32(const int32_t* in, int32_t* out, int64_t n, Arena& ar, cudaStream_t s)
{
    return scan_plain<int32_t, int32_t, true>(in, out, n, (int32_t*)nullptr, ar, s);
}

Status scan_inclusive_max_i32(const int32_t* in, int32_t* out, int64_t n, Arena& ar,
                              cudaStream_t s)
{
    return scan_run<Max32>(ScanLoad<int32_t, Max32>{in}, Max32Store{out}, n, (Max32*)nullptr, ar, s);
}

// ---------------------------------------------------------------------------
// Radix sort: 8-bit digits, tiles of 4096 keys (8 warps x 16 rounds of 32).

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ROUNDS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;

// the bits of the digit at `shift` that lie below end_bit
__host__ __device__ __forceinline__ uint32_t digit_mask(int shift, int end_bit)
{
    return end_bit - shift < 8 ? (1u << (end_bit - shift)) - 1 : 255u;
}

__global__ void __launch_bounds__(RS_THREADS)
    k_rs_upsweep(const uint64_t* keys, int64_t n, int shift, uint32_t dmask, uint32_t* counts, int nblk)
{
    after_previous();
    __shared__ uint32_t hist[256];
    for (int i = threadIdx.x; i < 256; i += RS_THREADS) hist[i] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * RS_TILE;
    for (int i = threadIdx.x; i < RS_TILE; i += RS_THREADS) {
        int64_t j = base + i;
        if (j < n) atomicAdd(&hist[(keys[j] >> shift) & dmask], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += RS_THREADS) counts[(int64_t)i * nblk + blockIdx.x] = hist[i];
}

__global__ void __launch_bounds__(RS_THREADS)
    k_rs_downsweep(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout,
                   int64_t n, int shift, uint32_t dmask, const uint32_t* offs, int nblk)
{
    after_previous();
    __shared__ uint32_t wcnt[RS_WARPS][256];
    __shared__ uint32_t boff[256];
    __shared__ uint32_t tmp[RS_WARPS][32];
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < RS_WARPS * 256; i += RS_THREADS) (&wcnt[0][0])[i] = 0;
    for (int i = threadIdx.x; i < 256; i += RS_THREADS) boff[i] = offs[(int64_t)i * nblk + blockIdx.x];
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * RS_TILE + (int64_t)warp * (32 * RS_ROUNDS);
    uint64_t k[RS_ROUNDS];
    uint32_t rank[RS_ROUNDS];
    unsigned lt = lanemask_lt();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; r++) {
        int64_t j = base + r * 32 + lane;
        bool valid = j < n;
        k[r] = valid ? kin[j] : 0;
        uint32_t d = valid ? (uint32_t)((k[r] >> shift) & dmask) : 256u;
        unsigned peers = __match_any_sync(FULL, d);
        int leader = __ffs(peers) - 1;
        if (lane == leader && valid) {
            uint32_t c = wcnt[warp][d];
            tmp[warp][lane] = c;
            wcnt[warp][d] = c + __popc(peers);
        }
        __syncwarp();
        rank[r] = valid ? tmp[warp][leader] + __popc(peers & lt) : 0;
        __syncwarp();
    }
    __syncthreads();
    // exclusive prefix over warps per digit, plus the block's global offset
    for (int d = threadIdx.x; d < 256; d += RS_THREADS) {
        uint32_t acc = boff[d];
        for (int w = 0; w < RS_WARPS; w++) {
            uint32_t c = wcnt[w][d];
            wcnt[w][d] = acc;
            acc += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; r++) {
        int64_t j = base + r * 32 + lane;
        if (j < n) {
            uint32_t d = (uint32_t)((k[r] >> shift) & dmask);
            uint32_t pos = wcnt[warp][d] + rank[r];
            kout[pos] = k[r];
            vout[pos] = vin[j];
        }
    }
}

// The whole sort in one launch for short inputs: one cluster of 8 blocks
// runs every pass, with the cluster's hardware barrier between the phases
// and the blocks' digit counts read through distributed shared memory. A
// short sort is bound by its launches and by the latency of a pass, not by
// bytes: in the form above a pass of a few thousand keys is an upsweep, one
// to three scan kernels and a downsweep by one or a few blocks.
// Passes in which every key has the same digit move nothing and are skipped.
constexpr int RSC_CTAS = 8;
constexpr int RSC_THREADS = 1024;
constexpr int RSC_WARPS = RSC_THREADS / 32;
constexpr int RSC_ROUNDS = 12;
constexpr int64_t RSC_MAX = (int64_t)RSC_CTAS * RSC_THREADS * RSC_ROUNDS;   // 98,304

__global__ void __cluster_dims__(RSC_CTAS, 1, 1) __launch_bounds__(RSC_THREADS)
    k_rs_cluster(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt, uint32_t* vals_alt, int32_t n,
                 int end_bit)
{
    after_previous();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ uint32_t wcnt[RSC_WARPS][256];
    __shared__ uint32_t hist[256];
    __shared__ uint32_t goff[256];
    __shared__ uint32_t tmp[RSC_WARPS][32];
    __shared__ uint32_t wsum[8];
    __shared__ int same;
    const int rank = (int)cl.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    const int rounds = (n + RSC_CTAS * RSC_THREADS - 1) / (RSC_CTAS * RSC_THREADS);
    const int w0 = (rank * RSC_THREADS + warp * 32) * rounds;
    uint64_t *ki = keys, *ko = keys_alt;
    uint32_t *vi = vals, *vo = vals_alt;
    for (int shift = 0; shift < end_bit; shift += 8) {
        const uint32_t dmask = digit_mask(shift, end_bit);
        for (int i = threadIdx.x; i < RSC_WARPS * 256; i += RSC_THREADS) (&wcnt[0][0])[i] = 0;
        if (threadIdx.x == 0) same = 0;
        uint64_t k[RSC_ROUNDS];
        uint32_t rk[RSC_ROUNDS];
        // keys written by the other blocks in the pass before: read past L1
#pragma unroll
        for (int r = 0; r < RSC_ROUNDS; r++) {
            int j = w0 + r * 32 + lane;
            k[r] = r < rounds && j < n ? __ldcg((unsigned long long*)&ki[j]) : 0;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < RSC_ROUNDS; r++) {
            if (r >= rounds) continue;   // the same for the whole cluster
            bool valid = w0 + r * 32 + lane < n;
            uint32_t d = valid ? (uint32_t)((k[r] >> shift) & dmask) : 256u;
            unsigned peers = __match_any_sync(FULL, d);
            int leader = __ffs(peers) - 1;
            if (lane == leader && valid) {
                uint32_t c = wcnt[warp][d];
                tmp[warp][lane] = c;
                wcnt[warp][d] = c + __popc(peers);
            }
            __syncwarp();
            rk[r] = valid ? tmp[warp][leader] + __popc(peers & lt) : 0;
            __syncwarp();
        }
        __syncthreads();
        if (threadIdx.x < 256) {
            uint32_t acc = 0;
#pragma unroll 8
            for (int w = 0; w < RSC_WARPS; w++) {
                uint32_t c = wcnt[w][threadIdx.x];
                wcnt[w][threadIdx.x] = acc;
                acc += c;
            }
            hist[threadIdx.x] = acc;
        }
        cl.sync();
        uint32_t before = 0, tot = 0, inc = 0;
        if (threadIdx.x < 256) {
#pragma unroll
            for (int b = 0; b < RSC_CTAS; b++) {
                uint32_t c = cl.map_shared_rank(hist, b)[threadIdx.x];
                if (b < rank) before += c;
                tot += c;
            }
            if (tot == (uint32_t)n) same = 1;
            inc = warp_inclusive(tot);
            if (lane == 31) wsum[warp] = inc;
        }
        __syncthreads();
        if (threadIdx.x < 256) {
            uint32_t acc = inc - tot + before;
            for (int w = 0; w < warp; w++) acc += wsum[w];
            goff[threadIdx.x] = acc;
        }
        __syncthreads();
        if (!same) {   // the same in every block: all saw the same totals
#pragma unroll
            for (int r = 0; r < RSC_ROUNDS; r++) {
                int j = w0 + r * 32 + lane;
                if (r < rounds && j < n) {
                    uint32_t d = (uint32_t)((k[r] >> shift) & dmask);
                    uint32_t pos = goff[d] + wcnt[warp][d] + rk[r];
                    __stcg((unsigned long long*)&ko[pos], (unsigned long long)k[r]);
                    __stcg(&vo[pos], __ldcg(&vi[j]));
                }
            }
            uint64_t* tk = ki; ki = ko; ko = tk;
            uint32_t* tv = vi; vi = vo; vo = tv;
            __threadfence();
        }
        // the pass is complete, and hist may be written again
        cl.sync();
    }
    if (ki != keys) {
#pragma unroll
        for (int r = 0; r < RSC_ROUNDS; r++) {
            int j = w0 + r * 32 + lane;
            if (r < rounds && j < n) {
                keys[j] = __ldcg((unsigned long long*)&ki[j]);
                vals[j] = __ldcg(&vi[j]);
            }
        }
    }
}

// Up to SB_MAX items one block sorts in shared memory: a bitonic network over
// the words key << ibits | position, the key cut to the bits that order it,
// whose order is the stable order of the keys; whole keys and values then move
// by position. A refinement round sorts its moves and its events, mostly a few
// hundred to a few thousand of each, and there even one launch of the radix
// passes is a chain of barriers: 1,000 keys of 20 bits take 24 us in the
// cluster form.
__global__ void __launch_bounds__(SB_THREADS)
    k_sort_block(uint64_t* keys, uint32_t* vals, int32_t n, int N, int ibits, uint64_t kmask)
{
    after_previous();
    __shared__ uint64_t w[SB_MAX];
    uint64_t k[SB_MAX / SB_THREADS];
    uint32_t v[SB_MAX / SB_THREADS];
    const uint64_t imask = (1ull << ibits) - 1;
    for (int i = threadIdx.x; i < N; i += SB_THREADS)
        w[i] = i < n ? (keys[i] & kmask) << ibits | (uint64_t)i : ~0ull;
    __syncthreads();
    block_sort_words(w, N);
#pragma unroll
    for (int r = 0; r < SB_MAX / SB_THREADS; r++) {
        int i = r * SB_THREADS + threadIdx.x;
        if (i < n) {
            k[r] = keys[w[i] & imask];
            v[r] = vals[w[i] & imask];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SB_MAX / SB_THREADS; r++) {
        int i = r * SB_THREADS + threadIdx.x;
        if (i < n) {
            keys[i] = k[r];
            vals[i] = v[r];
        }
    }
}

Status radix_sort_pairs(uint64_t* keys, uint32_t* vals, uint64_t* keys_alt, uint32_t* vals_alt,
                        int64_t n, int end_bit, Arena& ar, cudaStream_t s)
{
    if (n <= 1 || end_bit <= 0) return Status{};
    if (n >= ((int64_t)1 << 32)) return Status{1, "radix sort: too many items"};
    if (n <= SB_MAX) {
        int N = 64, ib = bits_for((uint64_t)(n - 1));
        while (N < n) N <<= 1;
        if (end_bit + ib < 64) {   // the padding stays above every word
            enqueue(k_sort_block, 1, SB_THREADS, 0, s, keys, vals, (int32_t)n, N, ib,
                    ((uint64_t)1 << end_bit) - 1);
            SNN_CUDA(cudaGetLastError());
            return Status{};
        }
    }
    if (n <= RSC_MAX) {
        enqueue(k_rs_cluster, RSC_CTAS, RSC_THREADS, 0, s, keys, vals, keys_alt, vals_alt, (int32_t)n,
                end_bit);
        SNN_CUDA(cudaGetLastError());
        return Status{};
    }
    int nblk = (int)ceil_div(n, RS_TILE);
    uint32_t* counts = nullptr;
    SNN_TRY(ar.alloc(&counts, (int64_t)256 * nblk));
    uint64_t *ki = keys, *ko = keys_alt;
    uint32_t *vi = vals, *vo = vals_alt;
    for (int shift = 0; shift < end_bit; shift += 8) {
        const uint32_t dmask = digit_mask(shift, end_bit);
        enqueue(k_rs_upsweep, nblk, RS_THREADS, 0, s, ki, n, shift, dmask, counts, nblk);
        SNN_CUDA(cudaGetLastError());
        SNN_TRY((scan_plain<uint32_t, uint32_t, false>(counts, counts, (int64_t)256 * nblk,
                                                       (uint32_t*)nullptr, ar, s)));
        enqueue(k_rs_downsweep, nblk, RS_THREADS, 0, s, ki, vi, ko, vo, n, shift, dmask, counts,
                nblk);
        SNN_CUDA(cudaGetLastError());
        uint64_t* tk = ki; ki = ko; ko = tk;
        uint32_t* tv = vi; vi = vo; vo = tv;
    }
    if (ki != keys) {
        SNN_CUDA(cudaMemcpyAsync(keys, ki, (size_t)n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
        SNN_CUDA(cudaMemcpyAsync(vals, vi, (size_t)n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    }
    return Status{};
}

}  // namespace snn
