/* The binning's short cell rule (nf_cell.cuh) over an array, on the host. */
#include <cstdint>

#include "nf_cell.cuh"

extern "C" void cell_rule(const float *x, int64_t n, double kl, unsigned char *ok_cell, int *cell, unsigned char *ok_off,
                          int *cell_off, float *off)
{
    const float hi = (float)kl, lo = (float)(kl - (double)hi);
    for (int64_t i = 0; i < n; ++i) {
        cell[i] = cell_off[i] = -1;
        off[i] = 0.0f;
        ok_cell[i] = nf::cell_short<false>(x[i], hi, lo, &cell[i], nullptr);
        ok_off[i] = nf::cell_short<true>(x[i], hi, lo, &cell_off[i], &off[i]);
    }
}
