// csrc/row_items.cuh on the host, for tests/test_row_deal.py.
#include "row_items.cuh"

// quads of a lane in the order it reads them; returns their number
extern "C" int row_deal(uint64_t mask, int32_t cw, int lane, int64_t* out, int cap)
{
    snn::ChunkDeal d(mask, cw, lane);
    int n = 0;
    while (d.left()) {
        int64_t q = d.next(-1);
        if (q >= 0 && n < cap) out[n++] = q;
    }
    return n;
}
