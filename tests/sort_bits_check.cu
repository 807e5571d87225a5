// Harness of tests/test_gpu_sort_bits.py: the library's stable sort of keys
// that have bits at and above end_bit, for the sizes given on the command
// line. Prints one line per check: "<n> <end_bit> <ok|wrong>".
#include "common.cuh"

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <numeric>
#include <random>
#include <vector>

using namespace snn;

static bool check(int64_t n, int bits, std::mt19937_64& rng, Arena& ar, cudaStream_t s)
{
    std::vector<uint64_t> k(n), gk(n);
    std::vector<uint32_t> v(n), gv(n), order(n);
    for (int64_t i = 0; i < n; i++) {
        k[i] = rng();
        if (i % 3 == 0 && i) k[i] = (k[i] >> bits << bits) | (k[i / 2] & ((1ull << bits) - 1));
        v[i] = (uint32_t)rng();
    }
    std::iota(order.begin(), order.end(), 0u);
    const uint64_t m = (1ull << bits) - 1;
    std::stable_sort(order.begin(), order.end(), [&](uint32_t p, uint32_t q) { return (k[p] & m) < (k[q] & m); });
    uint64_t *dk, *dk2;
    uint32_t *dv, *dv2;
    cudaMalloc(&dk, n * 8);
    cudaMalloc(&dk2, n * 8);
    cudaMalloc(&dv, n * 4);
    cudaMalloc(&dv2, n * 4);
    cudaMemcpy(dk, k.data(), n * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dv, v.data(), n * 4, cudaMemcpyHostToDevice);
    bool ok = radix_sort_pairs(dk, dv, dk2, dv2, n, bits, ar, s).ok();
    ok = cudaStreamSynchronize(s) == cudaSuccess && ok;
    cudaMemcpy(gk.data(), dk, n * 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(gv.data(), dv, n * 4, cudaMemcpyDeviceToHost);
    for (int64_t i = 0; i < n; i++) ok = ok && gk[i] == k[order[i]] && gv[i] == v[order[i]];
    cudaFree(dk);
    cudaFree(dk2);
    cudaFree(dv);
    cudaFree(dv2);
    ar.reset();
    return ok;
}

int main(int argc, char** argv)
{
    cudaStream_t s;
    if (cudaStreamCreate(&s) != cudaSuccess) return 2;
    Arena ar;
    ar.stream = s;
    std::mt19937_64 rng(11);
    for (int i = 1; i < argc; i++)
        for (int bits : {1, 8, 13, 40, 53})
            printf("%s %d %s\n", argv[i], bits, check(atoll(argv[i]), bits, rng, ar, s) ? "ok" : "wrong");
    ar.release();
    return cudaStreamSynchronize(s) == cudaSuccess ? 0 : 3;
}
