// Harness of tests/test_gpu_prims.py: the library's scans and stable sort
// against the standard library's, for the sizes given on the command line.
// Prints one line per check: "<what> <n> <ok|wrong>".
#include "scan.cuh"

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <numeric>
#include <vector>

using namespace snn;

namespace {

struct PairIn {
    const int32_t* p;
    __device__ Sum2 operator()(int64_t i) const { return Sum2(p[i], (int64_t)p[i] << 33); }
};
struct PairOut {
    int64_t *a, *b;
    __device__ void operator()(int64_t i, Sum2 ex, Sum2 v) const
    {
        a[i] = ex.a;
        b[i] = ex.b + v.b;
    }
};

uint64_t g_rng = 88172645463325252ull;
uint64_t rnd()
{
    g_rng ^= g_rng << 13;
    g_rng ^= g_rng >> 7;
    g_rng ^= g_rng << 17;
    return g_rng;
}

template <typename T>
struct Buf {
    T* p = nullptr;
    explicit Buf(int64_t n) { cudaMalloc(&p, (n > 0 ? n : 1) * sizeof(T)); }
    ~Buf() { cudaFree(p); }
    void put(const std::vector<T>& v) { cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice); }
    std::vector<T> get(int64_t n)
    {
        std::vector<T> v(n);
        cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
        return v;
    }
};

void say(const char* what, int64_t n, bool ok) { printf("%s %lld %s\n", what, (long long)n, ok ? "ok" : "wrong"); }

void check(int64_t n, Arena& ar, cudaStream_t s)
{
    std::vector<int32_t> x(n);
    for (auto& v : x) v = (int32_t)(rnd() % 1000) - 200;
    Buf<int32_t> in(n), out(n);
    Buf<int64_t> a(n), b(n), total(2);
    in.put(x);
    bool ok = scan_exclusive_i32(in.p, out.p, n, (int32_t*)total.p, ar, s).ok();
    cudaStreamSynchronize(s);
    auto got = out.get(n);
    int64_t sum = 0;
    for (int64_t i = 0; i < n; i++) {
        ok = ok && got[i] == (int32_t)sum;
        sum += x[i];
    }
    ok = ok && (int32_t)total.get(1)[0] == (int32_t)sum;
    say("exclusive", n, ok);

    ok = scan_inclusive_max_i32(in.p, out.p, n, ar, s).ok();
    cudaStreamSynchronize(s);
    got = out.get(n);
    int32_t mx = INT32_MIN;
    for (int64_t i = 0; i < n; i++) {
        mx = std::max(mx, x[i]);
        ok = ok && got[i] == mx;
    }
    say("max", n, ok);

    ok = scan_run<Sum2>(PairIn{in.p}, PairOut{a.p, b.p}, n, (Sum2*)total.p, ar, s).ok();
    cudaStreamSynchronize(s);
    auto ga = a.get(n), gb = b.get(n), gt = total.get(2);
    int64_t sa = 0, sb = 0;
    for (int64_t i = 0; i < n; i++) {
        sb += (int64_t)x[i] << 33;
        ok = ok && ga[i] == sa && gb[i] == sb;
        sa += x[i];
    }
    say("pair", n, ok && gt[0] == sa && gt[1] == sb);

    // few, many and equal keys; 62 bits leave no room for a position
    for (int bits : {0, 3, 20, 48, 62}) {
        std::vector<uint64_t> k(n);
        std::vector<uint32_t> v(n), order(n);
        for (int64_t i = 0; i < n; i++) {
            k[i] = bits ? rnd() >> (64 - bits) : 0;
            if (i && i % 3 == 0) k[i] = k[i / 2];
            v[i] = (uint32_t)rnd();
        }
        std::iota(order.begin(), order.end(), 0u);
        std::stable_sort(order.begin(), order.end(), [&](uint32_t p, uint32_t q) { return k[p] < k[q]; });
        Buf<uint64_t> dk(n), dk2(n);
        Buf<uint32_t> dv(n), dv2(n);
        dk.put(k);
        dv.put(v);
        ok = radix_sort_pairs(dk.p, dv.p, dk2.p, dv2.p, n, bits, ar, s).ok();
        cudaStreamSynchronize(s);
        auto gk = dk.get(n);
        auto gv = dv.get(n);
        for (int64_t i = 0; i < n; i++) ok = ok && gk[i] == k[order[i]] && gv[i] == v[order[i]];
        say("sort", n, ok);
    }
    ar.reset();
}

}  // namespace

int main(int argc, char** argv)
{
    cudaStream_t s;
    if (cudaStreamCreate(&s) != cudaSuccess) return 2;
    Arena ar;
    ar.stream = s;
    for (int i = 1; i < argc; i++) check(atoll(argv[i]), ar, s);
    ar.release();
    return cudaStreamSynchronize(s) == cudaSuccess ? 0 : 3;
}
