#pragma once
#include "common.cuh"
#include "ls.cuh"

namespace psps {

struct PenaltyDev {
    int nm;
    float beta[16];  // beta[k * 4 + k']
};

// What the last block does with the sums: nothing, close phi(0) (pobj: the
// data term's nobj block partials; history: the objective history), or set the
// line search up.  Saves the one-block kernels that would otherwise follow.
enum { kPenaltyOnly = 0, kPenaltyBegin = 1, kPenaltySearch = 2 };
struct PenaltyCtl {
    int then = kPenaltyOnly;
    DevLS *ls = nullptr;
    const dfloat *pobj = nullptr;
    int nobj = 0;
    double *history = nullptr;
};

int penalty_blocks(int64_t npix);
// rx_out (+)= R x (or |R| x with abs_mode); partials (3 per block, nullable):
// sum x.Rx, sum p.Rx, sum p.Rp.  x or p may be null (their terms are zero).
mbir_status launch_penalty(const PenaltyDev &pd, int nx, int ny, int nz, const float *x, const float *p, float *rx_out,
                           int accumulate, int abs_mode, dfloat *partials, int nblocks, const PenaltyCtl &ctl,
                           cudaStream_t s);

}  // namespace psps
