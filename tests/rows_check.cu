// Harness of tests/test_gpu_rows_refused.py: a pass, one with connection rows
// refused on the way down, as dense_grow would fail, and one more as the first.
//   rows_check V E P omega delta phi FILE NTH CODE
// The second pass's rows are refused from the NTH (0: coarsest, -1: finest) of
// the first pass's levels with rows on, with status CODE. FILE: off
// int64[E + 1], pins int32[P], w int32[E]; the partitions are appended to it.
// Prints "<status> <cost> <levels with rows> <levels without>" of each pass.
#include "internal.cuh"

#include <cstdio>
#include <cstdlib>

int main(int argc, char** argv)
{
    if (argc != 10) return 2;
    const int32_t V = atoi(argv[1]), E = atoi(argv[2]);
    const int64_t P = atoll(argv[3]);
    snnmap_params prm = snnmap_default_params(atoi(argv[4]), atoi(argv[5]), atoi(argv[6]));
    std::vector<int64_t> off(E + 1);
    std::vector<int32_t> pins(P), w(E), rho(V);
    FILE* f = fopen(argv[7], "r+b");
    if (!f || fread(off.data(), 8, E + 1, f) != (size_t)E + 1 || fread(pins.data(), 4, P, f) != (size_t)P ||
        fread(w.data(), 4, E, f) != (size_t)E)
        return 2;
    int64_t* d_off;
    int32_t *d_pins, *d_w, *d_rho;
    if (cudaMalloc(&d_off, (E + 1) * 8) || cudaMalloc(&d_pins, P * 4) || cudaMalloc(&d_w, E * 4) ||
        cudaMalloc(&d_rho, V * 4))
        return 3;
    cudaMemcpy(d_off, off.data(), (E + 1) * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(d_pins, pins.data(), P * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(d_w, w.data(), E * 4, cudaMemcpyHostToDevice);
    snnmap_hgraph* h = nullptr;
    if (snnmap_build_hgraph(&prm, V, E, d_off, d_pins, d_w, nullptr, &h)) return 4;
    const auto none = h->row_fault;
    std::vector<int32_t> on_rows;   // vertices of the first pass's levels with rows
    fseek(f, 0, SEEK_END);
    for (int pass = 0; pass < 3; pass++) {
        h->row_fault = none;
        if (pass == 1) {
            const int nth = atoi(argv[8]);
            const size_t at = nth < 0 ? on_rows.size() + nth : nth;
            if (at >= on_rows.size()) return 6;
            h->row_fault.rows = on_rows[at] - 1;
            h->row_fault.code = atoi(argv[9]);
        }
        int64_t cost = -1;
        int rc = snnmap_partition(h, nullptr, d_rho, &cost, nullptr);
        int with = 0, without = 0;
        for (const auto& r : h->rlog) {
            if (r.round != 0) continue;
            (r.rows ? with : without)++;
            if (pass == 0 && r.rows) on_rows.push_back(h->levels[r.level].V);
        }
        printf("%d %lld %d %d\n", rc, (long long)cost, with, without);
        if (h->dense.rowid || !h->dense.chunks.empty()) return 5;
        if (rc) continue;
        cudaMemcpy(rho.data(), d_rho, V * 4, cudaMemcpyDeviceToHost);
        fwrite(rho.data(), 4, V, f);
    }
    fclose(f);
    snnmap_free(h);
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 3;
}
