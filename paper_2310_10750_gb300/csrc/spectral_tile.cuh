// The whole solve of one sample on an N x N lattice (N = 64, 88, 128) by N / 8 warps, beta2 = 0, on
// the transforms of half_fft.cuh: the field stays in registers for every step (the inverse row
// transform ends in the layout the forward one starts from, so the update of Eq. nonl_CH_nm and the
// projection of Eq. potential_obstacle sit between them), the half spectrum in shared memory.
//
// What bounds it: the FMA pipe and shared memory, about evenly (per 128^2 step 1.26 M FP32
// operations, 9.8 K cycles at 128 a clock, and 6.1 K cycles of shared-memory traffic on an SM).
// 100 steps of 256 samples: 128^2 1.28 ms, 88^2 0.75; of 1000 samples of 64^2 1.03.  The forms
// before it (one complex transform per two rows, split and merged around the product, the field in
// shared memory; mixed radix at 88): 2.57, 3.21 and 2.34 ms.
#pragma once

#include "half_fft.cuh"
#include "mfmc_internal.h"

namespace mfmc {

// Shared memory of a lattice's transforms in bytes (T: float or double).
template <int N, typename T>
__host__ __device__ constexpr size_t hf_smem_bytes() {
    return (size_t)(HfCfg<N>::Z + HfCfg<N>::TW) * 2 * sizeof(T);
}

// Barrier of the lattice's warps (id 0: the whole CTA).
template <int NT>
__device__ __forceinline__ void tile_sync(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(NT) : "memory");
}

// tab: product table, tw: twiddles (global; hf_product_table, hf_twiddles); smem: hf_smem_bytes<N,
// float>() bytes, 16-byte aligned; red: N / 8 doubles of shared memory; warp: index among the
// lattice's warps; bar: their barrier.  Ends with the barrier, smem and red free.
template <int N>
__device__ __forceinline__ void tile_solve(const float *__restrict__ u0, float *__restrict__ uT, const StepCoef cf,
                                           const float4 *__restrict__ tab, const float2 *__restrict__ twg, int nsteps,
                                           double *ubar, double *ooi, float2 *smem, double *red, int warp, int bar) {
    using K = HfCfg<N>;
    Hf<N, float2> h;
    float2 *tw = smem + K::Z;
    h.z = smem;
    h.tw = tw;
    h.warp = warp;
    h.lane = threadIdx.x & 31;
    for (int i = warp * 32 + h.lane; i < K::TW; i += K::NT) tw[i] = twg[i];
    const size_t r0 = (size_t)(2 * h.my_row()) * N + h.n1();
    float2 u[K::A], v[K::A];
#pragma unroll
    for (int j = 0; j < K::A; ++j) u[j] = make_float2(__ldg(u0 + r0 + 8 * j), __ldg(u0 + r0 + N + 8 * j));
    tile_sync<K::NT>(bar);
#pragma unroll 1
    for (int k = 0; k < nsteps; ++k) {
#pragma unroll
        for (int j = 0; j < K::A; ++j) v[j] = u[j];
        h.rows_forward(v);
        tile_sync<K::NT>(bar);
        h.columns(tab);
        tile_sync<K::NT>(bar);
        h.rows_inverse(v);
#pragma unroll
        for (int j = 0; j < K::A; ++j) {
            const float a = u[j].x + fmaf(cf.c1, fmaf(-cf.c0, u[j].x, v[j].x), cf.c2 * u[j].x);
            const float b = u[j].y + fmaf(cf.c1, fmaf(-cf.c0, u[j].y, v[j].y), cf.c2 * u[j].y);
            u[j] = make_float2(fminf(1.f, fmaxf(-1.f, a)), fminf(1.f, fmaxf(-1.f, b)));
        }
    }
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < K::A; ++j) {
        s += (double)u[j].x + (double)u[j].y;
        if (uT) {
            uT[r0 + 8 * j] = u[j].x;
            uT[r0 + N + 8 * j] = u[j].y;
        }
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (h.lane == 0) red[warp] = s;
    tile_sync<K::NT>(bar);
    if (warp == 0 && h.lane == 0) {
        double t = 0.0;
        for (int i = 0; i < K::NW; ++i) t += red[i];
        const double mean = t / ((double)N * N);
        if (ubar) *ubar = mean;
        if (ooi) *ooi = 0.5 * (1.0 + mean);
    }
    tile_sync<K::NT>(bar);
}

}  // namespace mfmc
