// Harness of tests/test_gpu_memory.py: each network given by
// "V E P omega delta phi FILE" (FILE: off int64[E + 1], pins int32[P], w
// int32[E]) is run as a single batched job; prints its footprint, the peak it
// reports and the most the library's pool had in use.
#include "internal.cuh"

#include <cstdio>
#include <cstdlib>

int main(int argc, char** argv)
{
    for (int i = 1; i + 6 < argc; i += 7) {
        snnmap_job j{};
        j.n_vertices = atoi(argv[i]);
        j.n_hedges = atoi(argv[i + 1]);
        const int64_t P = atoll(argv[i + 2]);
        j.params = snnmap_default_params(atoi(argv[i + 3]), atoi(argv[i + 4]), atoi(argv[i + 5]));
        std::vector<int64_t> off(j.n_hedges + 1);
        std::vector<int32_t> pins(P), w(j.n_hedges), rho(j.n_vertices);
        FILE* f = fopen(argv[i + 6], "rb");
        if (!f || fread(off.data(), 8, off.size(), f) != off.size() ||
            fread(pins.data(), 4, pins.size(), f) != pins.size() || fread(w.data(), 4, w.size(), f) != w.size())
            return 2;
        fclose(f);
        j.offsets = off.data();
        j.pins = pins.data();
        j.w = w.data();
        j.rho_out = rho.data();
        j.on_host = 1;
        snnmap_serve_opts o{};
        o.slots = 1;
        o.mem_budget = 1;   // the footprint model's own row budget, nothing on top
        uint64_t high = 0;
        if (snn::pool_high(0, &high) != cudaSuccess) return 3;
        if (snnmap_batch_partition(&j, 1, &o)) return 4;
        if (snn::pool_high(0, &high) != cudaSuccess) return 3;
        printf("%lld %lld %llu\n", (long long)j.footprint, (long long)j.peak_bytes, (unsigned long long)high);
    }
    return 0;
}
