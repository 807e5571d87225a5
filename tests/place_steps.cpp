// The steps of csrc/place_items.cuh and csrc/initial_items.cuh that the
// placement kernels call, each beside the same sum written pin by pin, on host
// arrays. Test infrastructure only; built by tests/test_place_steps.py.
#include "initial_items.cuh"
#include "place_items.cuh"

#include <algorithm>
#include <cstring>
#include <vector>

using namespace snn::place;

extern "C" {

// Forces of node p (voff/vinc: its hyperedges, one entry per pin entry) by
// the kernels' steps and by force_terms; 0 past the border.
void steps_force(int32_t p, const int64_t* voff, const int32_t* vinc, const int64_t* off,
                 const int32_t* pins, const int64_t* eta, int32_t np, int32_t width, int32_t height,
                 const int32_t* g, int64_t got[4], int64_t want[4])
{
    std::vector<Cell> cell(np);
    for (int32_t q = 0; q < np; q++) cell[q] = cell_of(width, g[q]);
    std::fill(got, got + 4, 0);
    std::fill(want, want + 4, 0);
    int32_t nb[4];
    neighbours(width, height, g[p], nb);
    for (int64_t t = voff[p]; t < voff[p + 1]; t++) {
        int32_t a = vinc[t];
        side_forces(pins, off[a], off[a + 1], cell.data(), p, cell[p], eta[a], got);
        int64_t f[4] = {0, 0, 0, 0};
        force_terms(pins, off[a], off[a + 1], g, p, g[p], nb, width, f);
        for (int d = 0; d < 4; d++) want[d] += eta[a] * f[d];
    }
    for (int d = 0; d < 4; d++)
        if (!on_lattice(width, height, cell[p], d)) got[d] = 0;
}

// One hyperedge's re-evaluated share for p and its distances from pin entry j.
void steps_reeval_trd(const int32_t* pins, int64_t b, int64_t e, int64_t j, int32_t np, int32_t nh,
                      int32_t width, const int32_t* g, const int32_t* rank, const int32_t* mate,
                      int32_t p, int64_t got[2], int64_t want[2])
{
    std::vector<Cell> core(nh), cell(np);
    for (int32_t h = 0; h < nh; h++) core[h] = cell_of(width, h);
    for (int32_t q = 0; q < np; q++) cell[q] = cell_of(width, g[q]);
    const int32_t h = g[p], k = mate[h], r = rank[h];
    got[0] = reeval_cells(pins, b, e, g, rank, mate, core.data(), p, core[h], core[k], r);
    want[0] = reeval_terms(pins, b, e, g, rank, mate, p, h, k, r, width);
    got[1] = trd_cells(pins, j, e, cell.data());
    want[1] = trd_terms(pins, j, e, g, width);
}

// G(x) and the row of corrections of x (at position pos[x] of [lo, hi)) by
// the kernels' step and by single_gain and corr_row; row_*: hi - mid entries.
void steps_gain(int32_t x, const int64_t* voff, const int32_t* vinc, const int64_t* off,
                const int32_t* pins, const int64_t* eta, const int32_t* pos, int32_t lo, int32_t mid,
                int32_t hi, int64_t* g_got, int64_t* g_want, int64_t* row_got, int64_t* row_want)
{
    namespace ip = snn::initial;
    const int sd = ip::side_of(pos[x], lo, mid, hi);
    *g_got = 0;
    for (int64_t t = voff[x]; t < voff[x + 1]; t++) {
        int32_t a = vinc[t];
        *g_got += ip::gain_corr_hedge(pins, off[a], off[a + 1], pos, sd, lo, mid, hi, eta[a],
                                      [&](int32_t j, int64_t w) { row_got[j] += w; });
    }
    *g_want = ip::single_gain(vinc, voff[x], voff[x + 1], off, pins, eta, pos, sd, lo, mid, hi);
    if (sd == 1)
        ip::corr_row(vinc, voff[x], voff[x + 1], off, pins, eta, pos, lo, mid, hi,
                     [&](int32_t j, int64_t w) { row_want[j] += w; });
}
}
