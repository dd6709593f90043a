// The one-launch solve of matrices that fit one tile (small_solve.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/svt.h"

namespace svt {

constexpr int kSmallDim = 128;    // both sides at most this
constexpr int kSmallIters = 128;  // steps whose coefficients fit the launch's parameters

// Launch parameters: the call's arguments and the solve's resolved schedule.
struct SmallSolve {
    const float *A;
    float *Y;
    int64_t lda, ldy;
    svt_status *d_status;
    float tau;
    int m, n;          // input shape
    int pairs;         // FP32 tier: every iterate a hi/lo pair
    int rank_r;        // Corollary 1: no P chain
    int iters;
    int hp_steps;      // leading S steps on hi/lo pairs
    int norm_fro;      // the chains start divided by their Frobenius norms
    int cubic;         // NS3 schedule
    double first[3];               // a, b, c of the first step (scaled by the chain's norm)
    float coef[3 * kSmallIters];   // a, b, c of each step
};

cudaError_t small_solve_launch(const SmallSolve &p, cudaStream_t s);

// Flops of the launch's products: algorithmic (symmetric ones at half, hi/lo segments not
// counted again) and executed by the tensor cores.
void small_solve_flops(const SmallSolve &p, double *alg, double *executed);

} // namespace svt
