// Exclusive prefix sums with the elements computed on the fly (In) and the
// results consumed on the fly (Out), so that the kernels around a scan need
// no flag, length or index array of their own.
//
// Up to SCAN_BLOCK_MAX elements one block does the whole scan (k_scan_block),
// up to SCAN_CLUSTER_MAX one cluster of 8 blocks in one launch: a thread block cluster's barrier is a hardware one (no
// flag in memory to spin on or to clear) and the blocks' totals are
// exchanged through distributed shared memory. What bounds a scan of a
// level's arrays is not bandwidth but launches: the reduce/scan/tile form
// below for larger inputs takes three. Measured on a GB300 (int32 sums, back
// to back): 1k and 8k elements 6.2 us against 14.3 us, 64k 8.2 against 14.3,
// 128k 10.3 against 14.3, 256k 18.4 against 14.3: the line lies where eight
// SMs stop being enough.
#pragma once
#include "common.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace snn {

constexpr int SCAN_CTAS = 8;            // portable cluster size
constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ROUNDS = 8;          // elements per thread and sweep, at most
constexpr int64_t SCAN_CLUSTER_MAX = 1 << 17;
constexpr int SCAN_BLOCK_ROUNDS = 4;    // elements per thread of the one-block form, at most
constexpr int64_t SCAN_BLOCK_MAX = SCAN_BLOCK_ROUNDS * SCAN_THREADS;
constexpr int SCT_THREADS = 256;        // three-launch form
constexpr int SCT_ITEMS = 8;
constexpr int SCT_TILE = SCT_THREADS * SCT_ITEMS;

// two sums scanned together
struct Sum2 {
    int64_t a, b;
    __host__ __device__ Sum2() : a(0), b(0) {}
    __host__ __device__ Sum2(int64_t a_, int64_t b_) : a(a_), b(b_) {}
    __device__ Sum2 operator+(const Sum2& o) const { return Sum2(a + o.a, b + o.b); }
};

template <typename T>
__device__ __forceinline__ T scan_shfl_up(T v, int o)
{
    return __shfl_up_sync(FULL, v, o);
}
__device__ __forceinline__ Sum2 scan_shfl_up(Sum2 v, int o)
{
    return Sum2(__shfl_up_sync(FULL, v.a, o), __shfl_up_sync(FULL, v.b, o));
}
template <typename T>
__device__ __forceinline__ T scan_shfl(T v, int src)
{
    return __shfl_sync(FULL, v, src);
}
__device__ __forceinline__ Sum2 scan_shfl(Sum2 v, int src)
{
    return Sum2(__shfl_sync(FULL, v.a, src), __shfl_sync(FULL, v.b, src));
}

template <typename T>
__device__ __forceinline__ T warp_inclusive(T v)
{
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = scan_shfl_up(v, o);
        if (lane >= o) v = t + v;
    }
    return v;
}

// In: T operator()(int64_t i); Out: void operator()(int64_t i, T exclusive,
// T value). An element is read and written by the same thread, so the arrays
// behind In and Out may be the same. *total (device, may be null) = the sum.
template <typename T, class In, class Out>
__global__ void __cluster_dims__(SCAN_CTAS, 1, 1) __launch_bounds__(SCAN_THREADS)
    k_scan_cluster(In in, Out out, int64_t n, T* total)
{
    after_previous();
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ __align__(16) unsigned char raw[sizeof(T) * (2 * 32 + 2)];
    T* swarp = (T*)raw;          // [2][32]
    T* sblk = swarp + 2 * 32;    // [2]
    const int rank = (int)cl.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T carry = T();
    int par = 0;
    // the buffers of one sweep are written again two sweeps later, after the
    // cluster barrier of the sweep between
    for (int64_t base = 0; base < n; par ^= 1) {
        int64_t left = n - base;
        int rounds = left >= (int64_t)SCAN_CTAS * SCAN_THREADS * SCAN_ROUNDS
                         ? SCAN_ROUNDS
                         : (int)((left + SCAN_CTAS * SCAN_THREADS - 1) / (SCAN_CTAS * SCAN_THREADS));
        int64_t w0 = base + ((int64_t)rank * SCAN_THREADS + (int64_t)warp * 32) * rounds;
        T v[SCAN_ROUNDS], ex[SCAN_ROUNDS];
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) {
            int64_t i = w0 + r * 32 + lane;
            v[r] = r < rounds && i < n ? in(i) : T();
        }
        T run = T();
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) {
            if (r < rounds) {
                T inc = warp_inclusive(v[r]);
                T e = scan_shfl_up(inc, 1);
                ex[r] = lane == 0 ? run : run + e;
                run = run + scan_shfl(inc, 31);
            }
        }
        if (lane == 0) swarp[par * 32 + warp] = run;
        __syncthreads();
        if (warp == 0) {
            T t = swarp[par * 32 + lane];
            T inc = warp_inclusive(t);
            T e = scan_shfl_up(inc, 1);
            swarp[par * 32 + lane] = lane == 0 ? T() : e;
            if (lane == 31) sblk[par] = inc;
        }
        cl.sync();
        T off = carry, tot = T();
#pragma unroll
        for (int b = 0; b < SCAN_CTAS; b++) {
            T t = *cl.map_shared_rank(&sblk[par], b);
            if (b < rank) off = off + t;
            tot = tot + t;
        }
        off = off + swarp[par * 32 + warp];
#pragma unroll
        for (int r = 0; r < SCAN_ROUNDS; r++) {
            int64_t i = w0 + r * 32 + lane;
            if (r < rounds && i < n) out(i, off + ex[r], v[r]);
        }
        carry = carry + tot;
        base += (int64_t)SCAN_CTAS * SCAN_THREADS * rounds;
    }
    if (total && rank == 0 && threadIdx.x == 0) *total = carry;
    cl.sync();   // no block leaves while another reads its shared memory
}

// The same by one block, for the short scans of late levels: no cluster to
// place and no cluster barriers. Four elements a thread is where the block's
// own work has eaten that up (proposals' scan of the power-law networks'
// levels of 50 to 4,000 vertices: 9.4 us by a cluster, 4.1 by a block; counts
// of 6,000 take 10.9 by a cluster).
template <typename T, class In, class Out>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_block(In in, Out out, int32_t n, T* total)
{
    after_previous();
    __shared__ __align__(16) unsigned char raw[sizeof(T) * 33];
    T* swarp = (T*)raw;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int rounds = (n + (int)blockDim.x - 1) / (int)blockDim.x;   // <= SCAN_BLOCK_ROUNDS
    const int w0 = warp * 32 * rounds + lane;
    T v[SCAN_BLOCK_ROUNDS], ex[SCAN_BLOCK_ROUNDS];
#pragma unroll
    for (int r = 0; r < SCAN_BLOCK_ROUNDS; r++) v[r] = r < rounds && w0 + r * 32 < n ? in(w0 + r * 32) : T();
    T run = T();
#pragma unroll
    for (int r = 0; r < SCAN_BLOCK_ROUNDS; r++) {
        if (r < rounds) {
            T inc = warp_inclusive(v[r]);
            T e = scan_shfl_up(inc, 1);
            ex[r] = lane == 0 ? run : run + e;
            run = run + scan_shfl(inc, 31);
        }
    }
    if (lane == 0) swarp[warp] = run;
    __syncthreads();
    if (warp == 0) {
        T inc = warp_inclusive(lane < nw ? swarp[lane] : T());
        T e = scan_shfl_up(inc, 1);
        __syncwarp();
        swarp[lane] = lane == 0 ? T() : e;
        if (lane == 31) swarp[32] = inc;
    }
    __syncthreads();
    const T off = swarp[warp];
#pragma unroll
    for (int r = 0; r < SCAN_BLOCK_ROUNDS; r++)
        if (r < rounds && w0 + r * 32 < n) out(w0 + r * 32, off + ex[r], v[r]);
    if (total && threadIdx.x == 0) *total = swarp[32];
}

// exclusive prefix of each thread's value over the block of SCT_THREADS
template <typename T>
__device__ __forceinline__ T block_prefix(T v, T* sh, T* block_total)
{
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = SCT_THREADS / 32;
    T inc = warp_inclusive(v);
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    T before = T(), tot = T();
#pragma unroll
    for (int w = 0; w < NW; w++) {
        T t = sh[w];
        if (w < warp) before = before + t;
        tot = tot + t;
    }
    T e = scan_shfl_up(inc, 1);
    *block_total = tot;
    return lane == 0 ? before : before + e;
}

// a tile is 8 rows of SCT_THREADS consecutive elements; a warp owns 32 * 8
// consecutive ones
template <typename T, class In>
__global__ void __launch_bounds__(SCT_THREADS) k_scan_sums(In in, int64_t n, T* bsum)
{
    after_previous();
    __shared__ __align__(16) unsigned char raw[sizeof(T) * (SCT_THREADS / 32)];
    T acc = T();
    int64_t base = (int64_t)blockIdx.x * SCT_TILE;
#pragma unroll
    for (int r = 0; r < SCT_ITEMS; r++) {
        int64_t i = base + r * SCT_THREADS + threadIdx.x;
        if (i < n) acc = acc + in(i);
    }
    T tot;
    block_prefix(acc, (T*)raw, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

template <typename T, class In, class Out>
__global__ void __launch_bounds__(SCT_THREADS)
    k_scan_apply(In in, Out out, int64_t n, const T* boff, T* total)
{
    after_previous();
    __shared__ __align__(16) unsigned char raw[sizeof(T) * (SCT_THREADS / 32)];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t w0 = (int64_t)blockIdx.x * SCT_TILE + (int64_t)warp * 32 * SCT_ITEMS;
    T v[SCT_ITEMS], ex[SCT_ITEMS];
#pragma unroll
    for (int r = 0; r < SCT_ITEMS; r++) {
        int64_t i = w0 + r * 32 + lane;
        v[r] = i < n ? in(i) : T();
    }
    T run = T();
#pragma unroll
    for (int r = 0; r < SCT_ITEMS; r++) {
        T inc = warp_inclusive(v[r]);
        T e = scan_shfl_up(inc, 1);
        ex[r] = lane == 0 ? run : run + e;
        run = run + scan_shfl(inc, 31);
    }
    T* sh = (T*)raw;
    if (lane == 0) sh[warp] = run;
    __syncthreads();
    T off = boff[blockIdx.x], all = T();
#pragma unroll
    for (int w = 0; w < SCT_THREADS / 32; w++) {
        T t = sh[w];
        if (w < warp) off = off + t;
        all = all + t;
    }
#pragma unroll
    for (int r = 0; r < SCT_ITEMS; r++) {
        int64_t i = w0 + r * 32 + lane;
        if (i < n) out(i, off + ex[r], v[r]);
    }
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = boff[blockIdx.x] + all;
}

// Sort of w[0..N) (shared memory, N a power of two in [64, SB_MAX]) by one
// block of SB_THREADS, by a bitonic network; starts after and ends with a
// barrier.
constexpr int SB_MAX = 4096;
constexpr int SB_THREADS = 1024;

__device__ __forceinline__ void block_sort_words(uint64_t* w, int N)
{
    // a warp's 32 pairs of a step with stride <= 32 lie in one aligned run of
    // 64 words, so only longer strides need the whole block
    for (int k = 2; k <= N; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < N / 2; t += SB_THREADS) {
                int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
                uint64_t a = w[i], b = w[i + j];
                if ((a > b) == ((i & k) == 0)) {
                    w[i] = b;
                    w[i + j] = a;
                }
            }
            // the next step's stride is j / 2, or k after the last of these
            if (j > 32 || (j == 1 && k > 32)) __syncthreads();
            else __syncwarp();
        }
    }
    __syncthreads();
}

template <typename Tin, typename T>
struct ScanLoad {
    const Tin* p;
    __device__ T operator()(int64_t i) const { return (T)p[i]; }
};
template <typename T, bool INCL>
struct ScanStore {
    T* p;
    __device__ void operator()(int64_t i, T ex, T v) const { p[i] = INCL ? ex + v : ex; }
};

template <typename T, class In, class Out>
Status scan_run(const In& in, const Out& out, int64_t n, T* total, Arena& ar, cudaStream_t s)
{
    if (n <= 0) {
        if (total) SNN_CUDA(cudaMemsetAsync(total, 0, sizeof(T), s));
        return Status{};
    }
    if (n <= SCAN_BLOCK_MAX) {
        enqueue(k_scan_block<T, In, Out>, 1, (int)std::min<int64_t>((n + 31) & ~(int64_t)31, SCAN_THREADS), 0,
                s, in, out, (int32_t)n, total);
        SNN_CUDA(cudaGetLastError());
        return Status{};
    }
    if (n <= SCAN_CLUSTER_MAX) {
        enqueue(k_scan_cluster<T, In, Out>, SCAN_CTAS, SCAN_THREADS, 0, s, in, out, n, total);
        SNN_CUDA(cudaGetLastError());
        return Status{};
    }
    int64_t nb = ceil_div(n, SCT_TILE);
    T* bsum = nullptr;
    SNN_TRY(ar.alloc(&bsum, nb));
    enqueue(k_scan_sums<T, In>, (unsigned)nb, SCT_THREADS, 0, s, in, n, bsum);
    SNN_CUDA(cudaGetLastError());
    SNN_TRY((scan_run<T>(ScanLoad<T, T>{bsum}, ScanStore<T, false>{bsum}, nb, (T*)nullptr, ar, s)));
    enqueue(k_scan_apply<T, In, Out>, (unsigned)nb, SCT_THREADS, 0, s, in, out, n, bsum, total);
    SNN_CUDA(cudaGetLastError());
    return Status{};
}

}  // namespace snn
