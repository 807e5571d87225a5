// First slot of a key in the histograms' open-addressing tables (histo.cuh).
// The header uses no CUDA type, so the rule also compiles as plain host code.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define TS_HD __host__ __device__ __forceinline__
#else
#define TS_HD inline
#endif

namespace snn {

// Key m's first slot in a table of mask + 1 slots: the high bits of a
// multiplicative hash (the golden ratio's), scaled to the table. Runs of
// consecutive ids, which a hyperedge's sorted pins often are, land spread over
// it, closer to even than a random function's. The multiplication alone keeps
// an arithmetic progression one: ids a stride apart whose multiple of the
// golden ratio is near a whole number (233, 987, 1597, ...) all met in a few
// slots, filled the table's probe limit and went on to a slower tier. Folding
// the id's high bits in first breaks that once the progression leaves 256 ids.
// Level 0 of the 262,144-neuron conv network, ids times 233: 25.8 ms without
// the fold, 8.1 with it (10.7 before tables were multiplicative); as generated
// 7.2 and 7.4; the 1,048,576-neuron network 28.1 and 29.1, 32.5 with a full
// mixing hash.
TS_HD uint32_t table_slot(int32_t m, uint32_t mask)
{
    const uint32_t x = (uint32_t)m;
    const uint32_t h = (x ^ (x >> 8)) * 0x9e3779b1u;
#ifdef __CUDA_ARCH__
    return __umulhi(h, mask + 1);
#else
    return (uint32_t)((uint64_t)h * (mask + 1) >> 32);
#endif
}

}  // namespace snn
