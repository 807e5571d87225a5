// Which quads (int4) of a connection row each lane of a warp reads: the quads
// of the chunks that the row's mask marks, dealt so that a step's 32 reads are
// a part of one chunk or (chunks of fewer than 32 quads) one lane group per
// chunk of 32 / cq consecutive marked ones. With one chunk a step, 8 of 32
// lanes loaded at the smallest chunk width (conv network of 65,536 neurons:
// 11.7 us a round, 7.3 so). A lane gets its quads in increasing order. The
// header uses no CUDA type, so the dealing also compiles as plain host code.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define ROW_HD __host__ __device__ __forceinline__
#else
#define ROW_HD inline
#endif

namespace snn {

struct ChunkDeal {
    uint64_t msk;   // marked chunks left to this lane's group
    int cq;         // quads a chunk (a power of two of at least 8)
    int per;        // steps a chunk
    int side;       // chunks a step
    int at;         // this lane's quad in a step's part of a chunk
    int part = 0;   // steps taken of the first chunk left

    // mask: bit c for chunk c, entries [c cw, (c + 1) cw) of the row
    ROW_HD ChunkDeal(uint64_t mask, int32_t cw, int lane)
        : msk(mask), cq(cw >> 2), per(cq > 32 ? (cq + 31) / 32 : 1), side(cq < 32 ? 32 / cq : 1), at(lane)
    {
        const int grp = cq < 32 ? lane / cq : 0;
        if (cq < 32) at = lane - grp * cq;
        for (int g = 0; g < grp; g++) msk &= msk - 1;   // this group's first chunk
    }
    ROW_HD bool left() const { return msk != 0; }
    // the quad of this lane's next step, `none` where it has none
    ROW_HD int64_t next(int64_t none)
    {
        int64_t quad = none;
        if (msk) {
            const int q = at + part * 32;
#ifdef __CUDA_ARCH__
            const int c = __ffsll((long long)msk) - 1;
#else
            const int c = __builtin_ctzll(msk);
#endif
            if (q < cq) quad = (int64_t)c * cq + q;
            if (++part == per) {
                part = 0;
                for (int g = 0; g < side; g++) msk &= msk - 1;
            }
        }
        return quad;
    }
};

}  // namespace snn
