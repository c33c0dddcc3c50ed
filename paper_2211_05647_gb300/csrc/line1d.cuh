// line1d.cuh -- interface of the 1-D cooperative stepping kernel (line1d.cu).
#pragma once

#include <algorithm>
#include <vector>

#include "internal.cuh"

namespace fp {

template <typename TA>
struct LineArgs {
    TA *E, *H, *mur, *jslot;   // mur == nullptr: PEC ends
    void *df;
    const TA *dens, *tab;      // tab: [alpha | beta | w'] each `pitch` long
    const int32_t *slot_cell, *cut, *slot_cut;
    uint64_t *mail;            // eight words a CTA
    int64_t *d_step;           // receives step0 + nsteps
    int *err;
    uint64_t seed;
    Source src;
    int64_t step0;             // steps done before the launch
    uint32_t seq;              // tag of the first step's messages
    int nsteps, nz, pitch, rows_max, nodes_max;
    TA ch, ce, cj, m;
};

struct LinePlan {
    std::vector<int32_t> cut, slot_cut;   // range starts, one more than there are CTAs
    int nodes_max = 0, rows_max = 0;
};
LinePlan line1d_plan(int64_t nz, const std::vector<int32_t> &cells, int ctas, double row_cost);
size_t line1d_smem_bytes(int f_dtype, int pitch, int rows, int nodes);
template <typename TA>
cudaError_t launch_line1d(cudaStream_t st, const LineArgs<TA> &a, int f_dtype, int ctas);

}  // namespace fp
