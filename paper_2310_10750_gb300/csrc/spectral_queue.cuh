// The resident spectral queue: one launch over the (model, sample group) items of up to
// kSrMaxModels periodic beta2 = 0 models with n <= 128, each item a whole solve on chip.
//
// Items of a model on n = 128 and 88 (one sample) or n = 64 (four samples) run the tile-form solve
// (spectral_tile.cuh); items of any other n run the mixed-radix solve of smem_fft.cuh (one sample).
// The CTA's shared memory is the largest any of the launch's models needs; a launch with
// tile-form items has sixteen warps a CTA, one without them nine and two CTAs per SM.  Kernel and
// launcher in spectral.cu, host set-up in spectral_resident.cu.
#pragma once

#include "mfmc_internal.h"
#include "smem_fft.cuh"
#include "trace.cuh"

namespace mfmc {

enum : int { kSqGeneric = 0, kSqTile64 = 64, kSqTile88 = 88, kSqTile128 = 128 };  // item kinds
constexpr int kSqThreads = 288;      // nine warps: a launch of mixed-radix items alone
constexpr int kSqTileThreads = 512;  // sixteen warps: a launch with tile-form items

struct SqModelDev {
    const float *u0;       // [ns][n][n] initial fields
    float *uT;             // final fields, or nullptr
    double *ubar, *ooi;    // per sample, or nullptr
    const StepCoef *coef;  // per sample
    const int *steps_ps;   // per-sample step counts, or nullptr: nsteps for every sample
    const float *khat;     // mixed-radix: K^(ky, kx) / n^2 at [ky][n/2 + 1]
    const float4 *tab;     // tile form: the product table (hf_product_table)
    const float2 *tw;      // W_n^j, j < n (mixed-radix); hf_twiddles (tile form)
    FftPlan plan;
    int kind;              // kSqGeneric or kSqTile*
    int spc;               // samples per item
    int ns, nsteps;
};

struct SqArgs {
    SqModelDev m[kSrMaxModels];
    int begin[kSrMaxModels + 1];  // items of model k: [begin[k], begin[k + 1])
    int nm, total;
    int *counter;                 // zero at launch
    TraceBuf trace;
};

// Dynamic shared memory of one item kind on an n x n lattice, in a CTA of `warps` warps.
size_t spectral_queue_smem(int kind, int n, int warps);
// The tile form's tables of a model with n = 64, 88 or 128 (made once per model and device).
mfmc_status spectral_tile_tables(Model &m, const float4 **tab, const float2 **tw);
// CTAs of the queue kernel that fit on one SM with `smem` bytes of dynamic shared memory; tile:
// the launch has tile-form items (the kernel form that carries them).
int spectral_queue_blocks_per_sm(bool tile, size_t smem);
mfmc_status launch_spectral_queue(bool tile, const SqArgs &a, int grid, size_t smem, cudaStream_t st);

}  // namespace mfmc
