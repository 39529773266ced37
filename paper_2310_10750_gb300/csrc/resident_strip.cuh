// The resident solve (R <= 4; R = 5, 6, 8 on n <= 112): one CTA per sample, the field in registers for
// every step.
//
// A group of n / 4 lanes owns a strip of NB blocks of four rows (eight for R > 4), a lane four
// columns, so a row's window comes from neighbour lanes by shuffles and the periodic wrap is a lane
// index.  Every row's segment sums are formed once per step, by its owner, and added to the 2R + 1
// output rows they belong to; sums for rows of the strips above and below go there as partial sums
// through shared memory (two buffers in turn, one CTA barrier per step).  Results do not depend on
// NB: an output row's sum is (its own block + the block above) + the block below, each block's rows in ascending
// order, whether the blocks lie in one thread or in two.
//
// What bounds it: the FMA pipe (R = 4: 5.5 adds per point for the segment sums, 8 for the disc
// rows, 4 for the update: 2.2K cycles of a 128^2 step on an SM) and the shuffles and exchanges
// (2.0K cycles).  The kernel it replaces formed one segment difference per (row, output row) and
// walked (16 + 2R) / 16 of the rows, at 7 warps an SM (195 registers): 1001 samples of 128^2,
// R = 4, 500 steps 9.48 -> 5.58 ms; 4096 of 64^2, R = 2, 1000 steps 12.72 -> 7.07 ms; 32 of 64^2,
// R = 4, 200 steps (NB = 1) 318 -> 123 us.
//
// NB = 2 for throughput.  NB = 1 halves a step's serial chain at twice the exchange traffic: taken
// when the batch leaves most of the chip idle (launch_resident_strip).
#pragma once

#include "step_kernels.cuh"

namespace mfmc {

// Rows of a block: a row's sums then reach no further than the adjacent blocks.
__host__ __device__ constexpr int strip_rows(int R) { return R <= 4 ? 4 : 8; }

// Lanes that hold the columns next to a lane's (one and two lanes to the left and right, periodic).
struct StripLanes {
    int l1, l2, r1, r2;
};

// The segment sums of a block of BR rows u (four columns a lane), added to the output rows of the
// block (own) and the R rows below (dn[k]: row BR + k); those of the R rows above go to
// put_up(k, sums) (row k - R) as soon as the block has no more rows for them.
template <int R, int BR, typename Up>
__device__ __forceinline__ void strip_block(const float (&u)[BR][4], const StripLanes &ln, float2 (&own)[BR][2],
                                            float2 (&dn)[R][2], Up put_up) {
    constexpr DiscClasses<R> cls{};
    constexpr int M = 2 + R;
    float2 up[R][2];
#pragma unroll
    for (int r = 0; r < BR; ++r) {
        float v[4 + 2 * R], p[5 + 2 * R];
#pragma unroll
        for (int k = 0; k < R; ++k) {  // columns -1 - k and 4 + k of the lane
            v[R - 1 - k] = __shfl_sync(0xffffffffu, u[r][3 - k % 4], k < 4 ? ln.l1 : ln.l2);
            v[R + 4 + k] = __shfl_sync(0xffffffffu, u[r][k % 4], k < 4 ? ln.r1 : ln.r2);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) v[R + k] = u[r][k];
        // centre sums: p[k] = sum of v[M .. k - 1] for k > M, of v[k .. M - 1] for k < M
        p[M] = 0.f;
        p[M + 1] = v[M];
        p[M - 1] = v[M - 1];
#pragma unroll
        for (int q = 1; q < M; ++q) {
            p[M + 1 + q] = p[M + q] + v[M + q];
            p[M - 1 - q] = p[M - q] + v[M - 1 - q];
        }
#pragma unroll
        for (int c = 0; c < cls.count; ++c) {
            const int hw = cls.width[c];
            float h[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int b = i + R - hw, e = i + R + hw + 1;
                h[i] = hw == 0 ? v[R + i] : (b >= M ? p[e] - p[b] : (e <= M ? p[b] - p[e] : p[e] + p[b]));
            }
            const float2 h01 = make_float2(h[0], h[1]), h23 = make_float2(h[2], h[3]);
            // packed adds halve the instructions, scalar ones leave the FMA pipe sooner: R <= 2 scalar (4096
            // samples of 64^2, R = 2, 1000 steps: 7.34 -> 7.04 ms), above it one pair each (32 of 64^2, R = 4:
            // 135 packed, 129 scalar, 126 us mixed; 128^2, R = 4 alike)
            auto add = [&](float2 (&s)[2], bool first) {
                s[0] = first ? h01 : (R <= 2 ? make_float2(s[0].x + h01.x, s[0].y + h01.y) : __fadd2_rn(s[0], h01));
                s[1] = first ? h23 : make_float2(s[1].x + h23.x, s[1].y + h23.y);
            };
#pragma unroll
            for (int y = -R; y < BR + R; ++y) {
                const int ady = r > y ? r - y : y - r;
                if (ady <= R && cls.of[ady <= R ? ady : 0] == c) {
                    const bool first = r == (y > R ? y - R : 0);  // the output row's first row in this block
                    if (y < 0)
                        add(up[y < 0 ? y + R : 0], first);
                    else if (y < BR)
                        add(own[y >= 0 && y < BR ? y : 0], first);
                    else
                        add(dn[y >= BR ? y - BR : 0], first);
                }
            }
        }
        if (r < R) put_up(r, up[r < R ? r : 0]);  // row r - R: the block's rows 0 .. r are all it gets
    }
}

__host__ __device__ constexpr int strip_groups(int n) { return 32 / (n / 4); }          // strips per warp
// warps of a sample in strips of `rows` rows
__host__ __device__ constexpr int strip_warps(int n, int rows) {
    return (n / rows + strip_groups(n) - 1) / strip_groups(n);
}
inline size_t strip_smem(int n, int R, int nb) {
    const int br = strip_rows(R);
    const size_t ex = (size_t)2 * (n / (br * nb)) * 2 * R * n * sizeof(float);
    const size_t red = (size_t)(n / br) * (n / 4) * sizeof(double);
    return ex > red ? ex : red;
}

template <int R, int NB>
__global__ void __launch_bounds__(R <= 4 ? 512 : 448) resident_strip_kernel(ResidentArgs a) {
    constexpr int BR = strip_rows(R);
    static_assert(R <= BR && R <= 8, "a block's sums reach the adjacent blocks only, a window two lanes");
    extern __shared__ float4 smem4[];
    const int n = a.n, L = n / 4, strips = n / (BR * NB), groups = strip_groups(n);
    const int lane = threadIdx.x & 31, g = lane / L, cg = lane - g * L;
    const int strip_w = (threadIdx.x >> 5) * groups + g;
    const bool act = g < groups && strip_w < strips;
    const int strip = act ? strip_w : 0;   // idle lanes follow strip 0 and store nothing
    const int base = lane - cg, lanes = g < groups ? L : 32 - groups * L;
    const StripLanes ln{base + (cg + lanes - 1) % lanes, base + (cg + 2 * lanes - 2) % lanes, base + (cg + 1) % lanes,
                        base + (cg + 2) % lanes};
    const int cc = act ? cg : 0;
    // exchange rows [buffer][strip][0: for the strip above, 1: for the strip below][R][L]
    const int ex_strip = 2 * R * L, ex_buf = strips * ex_strip;
    float4 *const mine = smem4 + strip * ex_strip + cc;
    const float4 *const from_up = smem4 + (strip == 0 ? strips - 1 : strip - 1) * ex_strip + R * L + cc;
    const float4 *const from_dn = smem4 + (strip == strips - 1 ? 0 : strip + 1) * ex_strip + cc;
    const size_t nn = (size_t)n * n, off = (size_t)strip * BR * NB * n + 4 * cc;
    for (int sample = blockIdx.x; sample < a.ns; sample += gridDim.x) {
        const float *__restrict__ src = a.u0 + (size_t)sample * nn + off;
        float u[NB][BR][4];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int r = 0; r < BR; ++r) {
                const float4 t = __ldg(reinterpret_cast<const float4 *>(src + (size_t)(BR * b + r) * n));
                u[b][r][0] = t.x, u[b][r][1] = t.y, u[b][r][2] = t.z, u[b][r][3] = t.w;
            }
        const StepCoef cf = a.coef[sample];
        const float2 nc0 = make_float2(-cf.c0, -cf.c0), c1 = make_float2(cf.c1, cf.c1), c2 = make_float2(cf.c2, cf.c2);
        const int nsteps = a.steps_ps ? a.steps_ps[sample] : a.nsteps;
#pragma unroll 1
        for (int step = 0; step < nsteps; ++step) {
            const int buf = (step & 1) * ex_buf;
            float2 up[NB][R][2], own[NB][BR][2], dn[NB][R][2];  // up: of blocks 1 .. (block 0's goes out)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                strip_block<R, BR>(u[b], ln, own[b], dn[b], [&](int k, const float2 (&v)[2]) {
                    if (b == 0) {
                        if (act) mine[buf + k * L] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
                    } else {
                        up[b][k][0] = v[0];
                        up[b][k][1] = v[1];
                    }
                });
                if (act && b == NB - 1) {
#pragma unroll
                    for (int k = 0; k < R; ++k)
                        mine[buf + (R + k) * L] = make_float4(dn[b][k][0].x, dn[b][k][0].y, dn[b][k][1].x, dn[b][k][1].y);
                }
            }
            __syncthreads();
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int r = 0; r < BR; ++r) {
                    float2 s0 = own[b][r][0], s1 = own[b][r][1];
                    if (r < R) {  // from the block above
                        float2 t0, t1;
                        if (b == 0) {
                            const float4 t = from_up[buf + r * L];
                            t0 = make_float2(t.x, t.y);
                            t1 = make_float2(t.z, t.w);
                        } else {
                            t0 = dn[b - 1 >= 0 ? b - 1 : 0][r < R ? r : 0][0];
                            t1 = dn[b - 1 >= 0 ? b - 1 : 0][r < R ? r : 0][1];
                        }
                        s0 = __fadd2_rn(s0, t0);
                        s1 = __fadd2_rn(s1, t1);
                    }
                    if (r >= BR - R) {  // from the block below
                        float2 t0, t1;
                        const int k = r - (BR - R) >= 0 ? r - (BR - R) : 0;
                        if (b == NB - 1) {
                            const float4 t = from_dn[buf + k * L];
                            t0 = make_float2(t.x, t.y);
                            t1 = make_float2(t.z, t.w);
                        } else {
                            t0 = up[b + 1 < NB ? b + 1 : 0][k][0];
                            t1 = up[b + 1 < NB ? b + 1 : 0][k][1];
                        }
                        s0 = __fadd2_rn(s0, t0);
                        s1 = __fadd2_rn(s1, t1);
                    }
                    const float2 x0 = make_float2(u[b][r][0], u[b][r][1]), x1 = make_float2(u[b][r][2], u[b][r][3]);
                    const float2 v0 = __fadd2_rn(x0, __ffma2_rn(c1, __ffma2_rn(nc0, x0, s0), __fmul2_rn(c2, x0)));
                    const float2 v1 = __fadd2_rn(x1, __ffma2_rn(c1, __ffma2_rn(nc0, x1, s1), __fmul2_rn(c2, x1)));
                    u[b][r][0] = fminf(1.f, fmaxf(-1.f, v0.x));
                    u[b][r][1] = fminf(1.f, fmaxf(-1.f, v0.y));
                    u[b][r][2] = fminf(1.f, fmaxf(-1.f, v1.x));
                    u[b][r][3] = fminf(1.f, fmaxf(-1.f, v1.y));
                }
        }
        // OoI: FP64 sums of the blocks of BR x 4 values, then in block order per column group, then
        // over the groups
        __syncthreads();  // the last step's exchange rows have been read
        double *red = reinterpret_cast<double *>(smem4);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            double part = 0.0;
#pragma unroll
            for (int r = 0; r < BR; ++r) {
                part += ((double)u[b][r][0] + (double)u[b][r][1]) + ((double)u[b][r][2] + (double)u[b][r][3]);
                if (a.uT && act)
                    *reinterpret_cast<float4 *>(a.uT + (size_t)sample * nn + off + (size_t)(BR * b + r) * n) =
                        make_float4(u[b][r][0], u[b][r][1], u[b][r][2], u[b][r][3]);
            }
            if (act) red[(strip * NB + b) * L + cc] = part;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            double t = 0.0;
            if (lane < L)
                for (int k = 0; k < n / BR; ++k) t += red[k * L + lane];
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) {
                const double mean = t / (double)nn;
                if (a.ubar) a.ubar[sample] = mean;
                if (a.ooi) a.ooi[sample] = 0.5 * (1.0 + mean);
            }
        }
        __syncthreads();
    }
}

template <int R, int NB>
mfmc_status launch_strip(const ResidentArgs &a, int sms, cudaStream_t st) {
    auto kern = resident_strip_kernel<R, NB>;
    const size_t smem = strip_smem(a.n, R, NB);
    MFMC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int nt = 32 * strip_warps(a.n, strip_rows(R) * NB);
    int per_sm = 0;
    MFMC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem));
    const int cap = (per_sm > 0 ? per_sm : 1) * sms;
    kern<<<a.ns < cap ? a.ns : cap, nt, smem, st>>>(a);
    MFMC_LAUNCHED("resident_strip launch");
    return MFMC_OK;
}

template <int R>
mfmc_status launch_resident_strip(const ResidentArgs &a, cudaStream_t st) {
    if (a.ns <= 0) return MFMC_OK;
    int dev = 0, sms = 0;
    MFMC_CUDA(cudaGetDevice(&dev));
    MFMC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if constexpr (R > 4) {  // blocks of eight rows fill the registers
        return launch_strip<R, 1>(a, sms, st);
    } else {
        // NB = 1 while all of the batch's four-row strips fit at 8 warps an SM (and 16 a CTA)
        const int w1 = strip_warps(a.n, 4);
        if (w1 <= 16 && (long long)a.ns * w1 <= 8LL * sms) return launch_strip<R, 1>(a, sms, st);
        return launch_strip<R, 2>(a, sms, st);
    }
}

}  // namespace mfmc
