// line1d.cuh -- interface of the 1-D cooperative stepping kernel (line1d.cu).
#pragma once

#include "internal.cuh"
#include "line_plan.cuh"

namespace fp {

constexpr int kLineThreads = 512;

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

size_t line1d_smem_bytes(int f_dtype, int pitch, int rows, int nodes);
template <typename TA>
cudaError_t launch_line1d(cudaStream_t st, const LineArgs<TA> &a, int f_dtype, int ctas);

}  // namespace fp
