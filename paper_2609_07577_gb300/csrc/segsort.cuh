// Segmented sort of small uint32 key lists, one list per hyperedge, followed
// by a per-hyperedge epilogue. Hyperedges are split into size buckets once
// per level (by pin count L):
//   T:  L <= 16      one thread, keys in registers
//   B0: L <= 32      one warp, keys in registers (shuffle bitonic network)
//   B1: L <= 256     one warp, 2, 4 or 8 keys a lane in registers
//   B2: L <= 16384   one block of 512 threads, keys in dynamic shared memory
//   B3: larger       one block of 1024 threads, keys in a global scratch slice
// Each kernel walks its bucket's list with a grid-stride loop whose bound is
// read on the device, so no host synchronization is needed to launch them.
// Sorted keys are padded with 0xffffffff, which no key may equal.
//
// A Job supplies:
//   __device__ int len(int32_t a)                number of keys of hyperedge a
//   __device__ uint32_t load(int32_t a, int i)   key i (0 <= i < len)
//   __device__ void finish(int32_t a, const uint32_t* s, int n)
//        run by one full warp on the n sorted keys s[0..n)
//   __device__ void finish_thread(int32_t a, const uint32_t* s, int n, int st)
//                                                   (key i at s[i * st])
//        the same, run by a single thread
// and optionally kShared = true with
//   static constexpr int kSharedWords            most 32-bit words of shared memory a block
//                                                keeps for it, over all jobs of the type
//   int shared_words() const                     those of this job (0: none), zero on entry
//   __device__ void attach(uint32_t* words)      that memory, before any finish
//   __device__ void flush() const                run by the whole block after its lists
#pragma once
#include "common.cuh"

#include <type_traits>

namespace snn {

constexpr int SEG_T_CAP = 16;
constexpr int SEG_B1_CAP = 256;
constexpr int SEG_B2_CAP = 16384;
constexpr int SEG_B2_THREADS = 512;
constexpr int SEG_B3_THREADS = 1024;
constexpr int SEG_B3_BLOCKS = 16;
constexpr uint32_t KEY_PAD = 0xffffffffu;

// Per-level bucket lists of hyperedge ids: one array of E ids holding the
// buckets (T, B0, B1, B2, B3) back to back; meta (device int32[10]) =
// start[5], count[5].
// n: the counts on the host, or -1 while they are not known there; a filtered
// copy of the lists keeps its level's counts as upper bounds (seg_run sizes
// its launches by them and leaves out empty buckets).
struct SegBuckets {
    int32_t* list = nullptr;
    int32_t* meta = nullptr;
    int64_t b3_cap = 0;        // power of two >= longest hyperedge if any is in B3
    int32_t n[5] = {-1, -1, -1, -1, -1};
};

__device__ __forceinline__ uint32_t warp_bitonic32(uint32_t v)
{
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            uint32_t o = __shfl_xor_sync(FULL, v, j);
            bool up = (lane & k) == 0;
            bool lower = (lane & j) == 0;
            uint32_t mn = v < o ? v : o, mx = v < o ? o : v;
            v = (lower == up) ? mn : mx;
        }
    }
    return v;
}

__device__ __forceinline__ int pow2_at_least(int n, int lo)
{
    int p = lo;
    while (p < n) p <<= 1;
    return p;
}

// bitonic sort of s[0..N) by the whole block (s in shared or global memory)
__device__ __forceinline__ void block_bitonic(uint32_t* s, int N)
{
    for (int k = 2; k <= N; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < N; i += blockDim.x) {
                int ixj = i ^ j;
                if (ixj > i) {
                    uint32_t a = s[i], b = s[ixj];
                    bool asc = (i & k) == 0;
                    if ((a > b) == asc) {
                        s[i] = b;
                        s[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
}

enum : int { SEG_BT = 0, SEG_BB0 = 1, SEG_BB1 = 2, SEG_BB2 = 3, SEG_BB3 = 4, SEG_NB = 5 };

// Ascending sort of the 32 R keys a warp holds in registers, key r of lane l
// at position l R + r: a bitonic network whose strides below R stay inside a
// lane and whose longer strides are one shuffle per key.
template <int R>
__device__ __forceinline__ void warp_bitonic_regs(uint32_t (&k)[R])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 2; w <= 32 * R; w <<= 1) {
#pragma unroll
        for (int j = w >> 1; j > 0; j >>= 1) {
            if (j >= R) {
                const bool lower = (lane & (j / R)) == 0;
#pragma unroll
                for (int r = 0; r < R; r++) {
                    uint32_t o = __shfl_xor_sync(FULL, k[r], j / R);
                    bool up = ((lane * R + r) & w) == 0;
                    k[r] = (lower == up) ? min(k[r], o) : max(k[r], o);
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; r++) {
                    if ((r & j) != 0) continue;
                    bool up = ((lane * R + r) & w) == 0;
                    uint32_t x = k[r], y = k[r | j];
                    k[r] = up ? min(x, y) : max(x, y);
                    k[r | j] = up ? max(x, y) : min(x, y);
                }
            }
        }
    }
}

// keys of hyperedge a (L <= 32 R) sorted into s by one warp
template <int R, class Job>
__device__ __forceinline__ void warp_sort_list(const Job& job, int32_t a, int L, uint32_t* s)
{
    const int lane = threadIdx.x & 31;
    uint32_t k[R];
#pragma unroll
    for (int r = 0; r < R; r++) {
        int i = r * 32 + lane;
        k[r] = i < L ? job.load(a, i) : KEY_PAD;
    }
    warp_bitonic_regs<R>(k);
#pragma unroll
    for (int r = 0; r < R; r++) s[lane * R + r] = k[r];
    __syncwarp();
}

// T: one thread per list of at most SEG_T_CAP keys: the keys are sorted in
// registers by a fully unrolled bitonic network (padding sorts last) and
// handed to the epilogue through shared memory, slot i of thread t at
// i * blockDim + t so that a warp's lanes touch consecutive banks.
template <class Job>
__device__ __forceinline__ void seg_thread_lists(const Job& job, const int32_t* __restrict__ list,
                                                 int n, int block, int nblocks, uint32_t* sk)
{
    for (int base = block * 256; base < n; base += nblocks * 256) {
        int idx = base + threadIdx.x;
        if (idx >= n) continue;
        int32_t a = list[idx];
        int L = job.len(a);
        uint32_t k[SEG_T_CAP];
#pragma unroll
        for (int i = 0; i < SEG_T_CAP; i++) k[i] = i < L ? job.load(a, i) : KEY_PAD;
#pragma unroll
        for (int w = 2; w <= SEG_T_CAP; w <<= 1) {
#pragma unroll
            for (int j = w >> 1; j > 0; j >>= 1) {
#pragma unroll
                for (int i = 0; i < SEG_T_CAP; i++) {
                    int l = i ^ j;
                    if (l > i) {
                        bool up = (i & w) == 0;
                        uint32_t x = k[i], y = k[l];
                        if ((x > y) == up) {
                            k[i] = y;
                            k[l] = x;
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < SEG_T_CAP; i++) sk[i * 256 + threadIdx.x] = k[i];
        job.finish_thread(a, sk + threadIdx.x, L, 256);
    }
}

template <class J, class = void>
struct seg_shared : std::false_type {};
template <class J>
struct seg_shared<J, std::enable_if_t<J::kShared>> : std::true_type {};

// The three small buckets in one launch: blocks [0, gt) take T, the next gb0
// blocks B0 and the rest B1, so a level pays one launch and one tail for
// them (three launches of mostly few blocks before).
//
// B0 and B1 sort in registers. B1 held its keys in shared memory, one
// compare-exchange a load pair, a store pair and a warp barrier: the
// partition hypergraph of the 1,048,576-neuron conv network (917,504 lists
// of 77 keys) took 2.14 ms there and takes 1.0 ms here.
template <class Job>
__global__ void __launch_bounds__(256) k_seg_small(Job job, const int32_t* __restrict__ lists,
                                                   const int32_t* __restrict__ meta, int gt, int gb0)
{
    after_previous();
    extern __shared__ uint32_t seg_dyn[];
    if constexpr (seg_shared<Job>::value) {
        for (int i = threadIdx.x; i < job.shared_words(); i += 256) seg_dyn[i] = 0;
        job.attach(seg_dyn);
        __syncthreads();
    }
    __shared__ __align__(16) uint32_t buf[SEG_T_CAP * 256];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int blk = blockIdx.x;
    if (blk < gt) {
        seg_thread_lists(job, lists + meta[SEG_BT], meta[SEG_NB + SEG_BT], blk, gt, buf);
    } else if (blk < gt + gb0) {
        const int32_t* list = lists + meta[SEG_BB0];
        int n = meta[SEG_NB + SEG_BB0];
        uint32_t* s = buf + warp * 32;
        for (int idx = (blk - gt) * 8 + warp; idx < n; idx += gb0 * 8) {
            int32_t a = list[idx];
            int L = job.len(a);
            uint32_t v = lane < L ? job.load(a, lane) : KEY_PAD;
            s[lane] = warp_bitonic32(v);
            __syncwarp();
            job.finish(a, s, L);
            __syncwarp();
        }
    } else {
        const int32_t* list = lists + meta[SEG_BB1];
        int n = meta[SEG_NB + SEG_BB1];
        const int g = gridDim.x - gt - gb0;
        uint32_t* s = buf + warp * SEG_B1_CAP;
        for (int idx = (blk - gt - gb0) * 8 + warp; idx < n; idx += g * 8) {
            int32_t a = list[idx];
            int L = job.len(a);
            if (L <= 64) warp_sort_list<2>(job, a, L, s);
            else if (L <= 128) warp_sort_list<4>(job, a, L, s);
            else warp_sort_list<8>(job, a, L, s);
            job.finish(a, s, L);
            __syncwarp();
        }
    }
    if constexpr (seg_shared<Job>::value) {
        __syncthreads();
        job.flush();
    }
}

// B2 (shared memory) and B3 (global scratch, gscratch != nullptr)
template <class Job>
__global__ void k_seg_big(Job job, const int32_t* __restrict__ lists,
                          const int32_t* __restrict__ meta, int bucket, uint32_t* gscratch,
                          int64_t cap)
{
    after_previous();
    extern __shared__ uint32_t sbuf[];
    uint32_t* s = gscratch ? gscratch + (int64_t)blockIdx.x * cap : sbuf;
    const int32_t* list = lists + meta[bucket];
    int n = meta[SEG_NB + bucket];
    for (int idx = blockIdx.x; idx < n; idx += gridDim.x) {
        int32_t a = list[idx];
        int L = job.len(a);
        int N = pow2_at_least(L, 32);
        for (int i = threadIdx.x; i < N; i += blockDim.x) s[i] = i < L ? job.load(a, i) : KEY_PAD;
        __syncthreads();
        block_bitonic(s, N);
        if (threadIdx.x < 32) job.finish(a, s, L);
        __syncthreads();
    }
}

__device__ __forceinline__ int seg_bucket(int64_t len)
{
    return len <= SEG_T_CAP ? SEG_BT
         : len <= 32 ? SEG_BB0 : (len <= SEG_B1_CAP ? SEG_BB1 : (len <= SEG_B2_CAP ? SEG_BB2 : SEG_BB3));
}

// Per-thread bucket counts and pair terms, added to device words by whole
// blocks (every thread of the block calls flush).
struct SegTally {
    int32_t c[SEG_NB] = {0, 0, 0, 0, 0};
    int64_t terms = 0;
    __device__ void add(int64_t len)
    {
        int b = seg_bucket(len);
#pragma unroll
        for (int i = 0; i < SEG_NB; i++) c[i] += b == i;
        terms += len * (len - 1);
    }
    __device__ void flush(int64_t* counts, int64_t* w2)
    {
        __shared__ int32_t sc[SEG_NB];
        __shared__ unsigned long long st;
        if (threadIdx.x < SEG_NB) sc[threadIdx.x] = 0;
        if (threadIdx.x == 0) st = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SEG_NB; i++) {
            int32_t t = warp_sum(c[i]);
            if ((threadIdx.x & 31) == 0 && t) atomicAdd(&sc[i], t);
        }
        int64_t t = warp_sum(terms);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(&st, (unsigned long long)t);
        __syncthreads();
        if (threadIdx.x < SEG_NB && sc[threadIdx.x])
            atomicAdd((unsigned long long*)&counts[threadIdx.x], (unsigned long long)sc[threadIdx.x]);
        if (threadIdx.x == 0 && st) atomicAdd((unsigned long long*)w2, st);
    }
};

// Builds the bucket lists of a level from the counts known on the host
// (b.n); cursor: SEG_NB device words, zero on entry. The order within a
// bucket follows the hyperedge ids up to the order in which blocks arrive
// (no result depends on it).
Status seg_lists(const int64_t* hoff, int32_t E, int32_t maxlen, SegBuckets& b, int32_t* cursor,
                 cudaStream_t s);

inline int seg_grid_big(int32_t E) { return grid_for(E, 1, 152 * 2); }

template <class Job>
Status seg_run(const Job& job, const SegBuckets& b, int32_t E, Arena& ar, cudaStream_t s)
{
    if (E <= 0) return Status{};
    auto count = [&](int k) { return b.n[k] >= 0 ? b.n[k] : E; };
    size_t dyn = 0;
    int cap = 152 * 16;
    if constexpr (seg_shared<Job>::value) {
        // every block clears and flushes its words: fewer, longer blocks
        dyn = (size_t)job.shared_words() * sizeof(uint32_t);
        if (dyn) cap = 152 * 4;
    }
    int gt = count(SEG_BT) > 0 ? grid_for(count(SEG_BT), 256, cap) : 0;
    int gb0 = count(SEG_BB0) > 0 ? grid_for(count(SEG_BB0), 8, cap) : 0;
    int gb1 = count(SEG_BB1) > 0 ? grid_for(count(SEG_BB1), 8, cap) : 0;
    if (gt + gb0 + gb1 > 0) {
        // the type's most, not this job's: the attribute is the kernel's, and a
        // handle on another host thread may set it between here and the launch
        if constexpr (seg_shared<Job>::value)
            SNN_CUDA(cudaFuncSetAttribute(k_seg_small<Job>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          Job::kSharedWords * (int)sizeof(uint32_t)));
        enqueue(k_seg_small<Job>, gt + gb0 + gb1, 256, dyn, s, job, b.list, b.meta, gt, gb0);
        SNN_CUDA(cudaGetLastError());
    }
    if (count(SEG_BB2) > 0) {
        size_t smem = SEG_B2_CAP * sizeof(uint32_t);
        SNN_CUDA(cudaFuncSetAttribute(k_seg_big<Job>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
        enqueue(k_seg_big<Job>, seg_grid_big(count(SEG_BB2)), SEG_B2_THREADS, smem, s, job, b.list,
                b.meta, SEG_BB2, nullptr, 0);
        SNN_CUDA(cudaGetLastError());
    }
    if (b.b3_cap > 0 && count(SEG_BB3) > 0) {
        uint32_t* g = nullptr;
        SNN_TRY(ar.alloc(&g, (int64_t)SEG_B3_BLOCKS * b.b3_cap));
        enqueue(k_seg_big<Job>, SEG_B3_BLOCKS, SEG_B3_THREADS, 0, s, job, b.list, b.meta, SEG_BB3, g,
                b.b3_cap);
        SNN_CUDA(cudaGetLastError());
    }
    return Status{};
}

}  // namespace snn
