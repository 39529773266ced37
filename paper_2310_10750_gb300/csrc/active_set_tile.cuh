// The beta2 > 0 solver on the paper's lattices (n = 64, 88, 128) with its FP32 correction solve on
// chip: interface between active_set.cu (which describes the method and the fallback kernel for
// other n) and active_set_tile.cu (the kernel).
#pragma once

#include "mfmc_internal.h"
#include "trace.cuh"

namespace mfmc {

// Constants of the correction solve shared by both kernels.
constexpr float AS_CG_RTOL = 1e-5f;   // max |J d + F| / max |F| that ends a correction (active_set_tile.cu:
                                      // one of its tolerances)
constexpr float AS_OMEGA = 0.8f;      // damping of the Jacobi sweeps

struct alignas(16) AsFactor {
    double x, y, z, w;  // a row of hf_product_table
};

struct AsTileArgs {
    const float *u0;
    float *uT;
    double *ubar, *ooi;
    const double *eps;   // per sample, or nullptr: eps_nominal
    double eps_nominal;
    double *buf;         // [ns][as_tile_per_sample(n)]
    int *status;         // set to 1 when an iteration bound is reached
    unsigned long long *iters;  // [2]: Newton and CG iterations, added by every CTA
    const double *wtab;  // Gaussian: FP64 weight / eps^2 by r^2; nullptr: constant kernel
    int widths[kMaxR + 1];
    int R, nsteps;
    int newton_max, cg_max;
    // the disc sums by FFT: product table and twiddles of half_fft.cuh; nullptr: the direct sum
    const AsFactor *tab;
    const double2 *tw;
    TraceBuf trace;
    size_t s0;
    double ahat, chat, tau, beta1, beta2, cF;
};

// Doubles of scratch per sample: u, g and w in FP64 and the correction d in FP32.
__host__ __device__ constexpr size_t as_tile_per_sample(int n) { return (size_t)3 * n * n + (size_t)n * n / 2; }
bool as_tile_supported(int n);
mfmc_status launch_active_set_tile(const AsTileArgs &a, int n, unsigned grid, cudaStream_t st);

}  // namespace mfmc
