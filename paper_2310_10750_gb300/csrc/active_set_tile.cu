// The beta2 > 0 step (MFMC_ALGO_ACTIVE_SET) on n = 64, 88 and 128: the method of active_set.cu,
// one CTA per sample, with the FP32 correction solve held in registers and shared memory.
//
// Layout.  Warp w owns lattice rows 8w .. 8w + 7 and a lane 2 or 4 consecutive columns of them
// (n = 64: 2 columns, 32 lanes, 8 warps; n = 88: 4 columns, 22 lanes, 11 warps; n = 128: 4
// columns, 32 lanes, 16 warps), so a row is one warp, its periodic wrap a shuffle, and only a
// warp's first and last row pass through shared memory when a stencil is applied.  The residual
// of the correction (f) and the V-cycle's iterate (v) are registers; p and q are shared memory,
// each thread reading back its own values; d is global scratch that is only added to (a vector
// reduction, no load).  The inactive set is one bit per point, a 32-bit mask per thread.
//
// The multigrid levels halve the thread's block: 4 x 8, 2 x 4 and 1 x 2 points (n = 64: 2 x 8
// and 1 x 4), each level's mask average a population count of the thread's bits, restriction
// and prolongation exchanging one row per warp.  The levels below one column a lane (16^2 and
// 8^2, or 11^2 for n = 88) are one warp's work, in its registers.  A pass costs one CTA barrier (the
// row exchange alternates two buffers) and no index arithmetic; the relaxation factors are divided once
// a Newton pass.  f and v are 32 registers each (n = 64: 16) where the launch allows 128, 80 and 64 a
// thread, so parts of them spill around the coarse levels (bytes of stores a thread: 128^2 580, 88^2
// 1448, 64^2 488; L1 holds them).
//
// What bounds it: the fallback kernel (fine-level vectors in L2, generic indices) issued 943
// instructions per point and CG iteration, and waited on L2 (long scoreboard 4.4 cycles an
// instruction).  Here the FP64 pipe (two lanes a clock an SM) takes the larger part of a step, 52 % busy
// over 128^2 solves and 69 % over 64^2: the disc sum's transforms (444 K cycles a step of 128^2) and 7
// operations per point of a Newton residual (88 K); a V-cycle is 20 K cycles.  beta2 = 0.05: 50
// samples of 128^2, 20 steps, 17.3 ms (fallback kernel 113), 1000 of 64^2, 10 steps, 11.3 ms (106), 304
// of 88^2, 8 steps, 8.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>

#include "active_set_tile.cuh"
#include "spectral_tile.cuh"

namespace mfmc {

namespace {

// Newton passes of a step (4 to 8 as a rule) under the default bound: loose corrections up to the first of
// these, then again from the beta2 = 0 step's w with tight ones, then once more, its first AT_DAMPED
// corrections halved, which ends most cycles of the active set.  (2400 samples of 4 steps, 5 lattices and
// horizons, eps 0.002 to 0.06, beta2 0.05 to 5: tight corrections alone end 1618 within 60 passes, loose ones
// alone 1620 but 5 of those not, with the restarts 2262 and none of those lost; 12, 32, 6 passes 2142.)
constexpr int AT_LOOSE_PASSES = 12, AT_TIGHT_PASSES = 24, AT_DAMPED = 10;
constexpr int AT_NU_COARSE = 8;  // coarsest sweeps (16, as the fallback kernel has: no CG iteration fewer)

template <int N>
struct AtCfg {
    static constexpr int CW = N == 64 ? 2 : 4;      // columns per lane
    static constexpr int LU = N / CW;               // lanes in use
    static constexpr int RW = 8;                    // rows per warp
    static constexpr int NW = N / RW, NT = 32 * NW;
    static constexpr int LEVELS = CW == 4 ? 3 : 2;  // levels held in registers: CW >> level columns a lane
    static constexpr int TN = N >> LEVELS;          // the first level of the one-warp part
    static constexpr int XP = 32 * CW;              // floats of an exchanged row
    // shared memory (floats): p, q, the exchange rows (two buffers of two rows a warp), the one-warp
    // part's right-hand side, result, diagonal, relaxation factors and 8^2 factors, then the relaxation
    // factors of levels 1 and 2
    static constexpr int P = 0, Q = N * N, X = 2 * N * N, T = X + 4 * NW * XP;
    static constexpr int RX1 = T + (4 * TN * TN + 64), RX2 = RX1 + N * N / 4;
    // N = 64 forms them in every sweep: four CTAs an SM bind on shared memory (11.45 ms held, 11.34 formed)
    static constexpr bool HOLD = N != 64;
    static constexpr size_t SMEM = (size_t)(HOLD ? RX2 + N * N / 16 : RX1) * sizeof(float);
    static_assert(LU <= 32 && N % RW == 0 && N % CW == 0, "one warp per row block");
};

// a / b rounded to nearest, from r = 1 / b rounded to nearest: one correction of the product a r by its
// exact remainder (Markstein, IBM J. Res. Dev. 34, 1990), three operations where a division takes about ten.
__device__ __forceinline__ double at_div(double a, double b, double r) {
    const double q = a * r;
    return fma(fma(-q, b, a), r, q);
}
__device__ __forceinline__ double at_clip(double v) { return v > 1.0 ? 1.0 : (v < -1.0 ? -1.0 : v); }

template <int C>
__device__ __forceinline__ void at_ld(float (&v)[C], const float *p) {
    if constexpr (C == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
    } else if constexpr (C == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x, v[1] = t.y;
    } else {
        v[0] = *p;
    }
}
template <int C>
__device__ __forceinline__ void at_st(float *p, const float (&v)[C]) {
    if constexpr (C == 4)
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (C == 2)
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    else
        *p = v[0];
}
template <int C>
__device__ __forceinline__ void at_ld64(double (&v)[C], const double *p) {
#pragma unroll
    for (int c = 0; c < C; c += 2) {
        const double2 t = *reinterpret_cast<const double2 *>(p + c);
        v[c] = t.x, v[c + 1] = t.y;
    }
}
template <int C>
__device__ __forceinline__ void at_st64(double *p, const double (&v)[C]) {
#pragma unroll
    for (int c = 0; c < C; c += 2) *reinterpret_cast<double2 *>(p + c) = make_double2(v[c], v[c + 1]);
}
// d += v at C consecutive floats of global memory that only this thread touches (no load; the
// values are read back past L1).
template <int C>
__device__ __forceinline__ void at_red(float *p, const float (&v)[C]) {
    if constexpr (C == 4)
        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                     : "memory");
    else
        asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v[0]), "f"(v[1]) : "memory");
}

// A thread's view of the CTA and the operator.  Level l: J v = (tb1 + 4 tb2[l] + m icg) v - tb2[l] (sum
// of the four neighbours), m the mean of the inactive set over the level's 2^l x 2^l points.
template <int N>
struct At {
    using K = AtCfg<N>;
    float *sm, *red;
    int warp, lane, left, right;  // lanes of the columns left and right of the lane's (periodic)
    int slot;                     // the lane's first column in a [row][warp][lane] layout (idle lanes: lane 0's)
    int par, rpar;                // the exchange and reduction buffers in turn
    unsigned mask;                // inactive set: bit row * CW + column
    float tb1, icg, tb2;          // tb2: level 0; level l has tb2 / 4^l
    float w0, w1, d0, d1;         // level 0: omega / diagonal and diagonal off and on the inactive set

    __device__ __forceinline__ float *xrow(int w, int which) const {
        return sm + K::X + ((par * K::NW + w) * 2 + which) * K::XP;
    }
    __device__ __forceinline__ int up() const { return warp == 0 ? K::NW - 1 : warp - 1; }
    __device__ __forceinline__ int down() const { return warp == K::NW - 1 ? 0 : warp + 1; }
    // Rows next to the warp's: the last row of the warp above and the first of the warp below.
    template <int C>
    __device__ __forceinline__ void exchange(const float (&top)[C], const float (&bot)[C], float (&above)[C],
                                             float (&below)[C]) {
        at_st<C>(xrow(warp, 0) + lane * C, top);
        at_st<C>(xrow(warp, 1) + lane * C, bot);
        __syncthreads();
        at_ld<C>(above, xrow(up(), 1) + lane * C);
        at_ld<C>(below, xrow(down(), 0) + lane * C);
        par ^= 1;
    }
    template <int C>
    __device__ __forceinline__ void from_above(const float (&bot)[C], float (&above)[C]) {
        at_st<C>(xrow(warp, 1) + lane * C, bot);
        __syncthreads();
        at_ld<C>(above, xrow(up(), 1) + lane * C);
        par ^= 1;
    }
    template <int C>
    __device__ __forceinline__ void from_below(const float (&top)[C], float (&below)[C]) {
        at_st<C>(xrow(warp, 0) + lane * C, top);
        __syncthreads();
        at_ld<C>(below, xrow(down(), 0) + lane * C);
        par ^= 1;
    }
    // CTA-wide sum in a fixed order: butterflies over the lanes, then over the warps' sums (the
    // same in every warp).  Idle lanes pass 0.
    __device__ __forceinline__ float sum(float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[rpar * 32 + warp] = v;
        __syncthreads();
        float t = lane < K::NW ? red[rpar * 32 + lane] : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        rpar ^= 1;
        return t;
    }
    // CTA-wide maximum of unsigned integers.
    __device__ __forceinline__ unsigned max_bits(unsigned v) {
        const unsigned m = __reduce_max_sync(0xffffffffu, v);
        if (lane == 0) red[rpar * 32 + warp] = __uint_as_float(m);
        __syncthreads();
        const unsigned t = __reduce_max_sync(0xffffffffu, lane < K::NW ? __float_as_uint(red[rpar * 32 + lane]) : 0u);
        rpar ^= 1;
        return t;
    }
    // CTA-wide maximum of non-negative values (their bit patterns order as unsigned integers).
    __device__ __forceinline__ float max(float v) { return __uint_as_float(max_bits(__float_as_uint(v))); }

    template <int L>
    __device__ __forceinline__ float tb2l() const { return tb2 * (1.0f / (1 << (2 * L))); }
    template <int L>
    __host__ __device__ static constexpr unsigned bits(int y, int c) {
        unsigned b = 0;
        for (int i = 0; i < (1 << L); ++i)
            for (int j = 0; j < (1 << L); ++j) b |= 1u << (((y << L) + i) * K::CW + (c << L) + j);
        return b;
    }
    // The diagonal of J at the lane's point (y, c) of level L.
    template <int L>
    __device__ __forceinline__ float diag(int y, int c) const {
        const float d = tb1 + 4.0f * tb2l<L>();
        if constexpr (L == 0)
            return (mask & bits<0>(y, c)) ? d1 : d0;
        else
            return fmaf((float)__popc(mask & bits<L>(y, c)), icg * (1.0f / (1 << (2 * L))), d);
    }
    // omega / diagonal of the lane's row y of level L.  Those of levels 1 and 2 hold for a Newton pass:
    // divided once (hold_relax) into shared memory, each thread reading back its own.
    template <int L>
    __device__ __forceinline__ float *relax_at(int y) const {
        return sm + (L == 1 ? K::RX1 : K::RX2) + y * (K::NW * K::LU * (K::CW >> L)) + (slot >> L);
    }
    template <int L, int C>
    __device__ __forceinline__ void relax(int y, float (&w)[C]) const {
        static_assert(C == K::CW >> L, "a level's columns");
        if constexpr (L == 0) {
#pragma unroll
            for (int c = 0; c < C; ++c) w[c] = (mask & bits<0>(y, c)) ? w1 : w0;
        } else if constexpr (K::HOLD) {
            at_ld<C>(w, relax_at<L>(y));
        } else {
#pragma unroll
            for (int c = 0; c < C; ++c) {  // the fast quotient corrected by its remainder
                const float d = diag<L>(y, c), r = __fdividef(1.0f, d), q = AS_OMEGA * r;
                w[c] = fmaf(fmaf(-q, d, AS_OMEGA), r, q);
            }
        }
    }
    template <int L>
    __device__ __forceinline__ void hold_relax() {
        constexpr int C = K::CW >> L;
        if (lane < K::LU) {
#pragma unroll
            for (int y = 0; y < (K::RW >> L); ++y) {
                float w[C];
#pragma unroll
                for (int c = 0; c < C; ++c) w[c] = AS_OMEGA / diag<L>(y, c);
                at_st<C>(relax_at<L>(y), w);
            }
        }
        if constexpr (L + 1 < K::LEVELS) hold_relax<L + 1>();
    }
};

// One row's neighbour sums: up + down + left + right.
template <int N, int C>
__device__ __forceinline__ void at_nb(const At<N> &t, const float (&up)[C], const float (&cur)[C], const float (&dn)[C],
                                      float (&S)[C]) {
    const float l = __shfl_sync(0xffffffffu, cur[C - 1], t.left), r = __shfl_sync(0xffffffffu, cur[0], t.right);
#pragma unroll
    for (int c = 0; c < C; ++c) S[c] = (up[c] + dn[c]) + ((c == 0 ? l : cur[c - 1]) + (c == C - 1 ? r : cur[c + 1]));
}

// One damped-Jacobi sweep of v in place: v + omega D^-1 (f - J v) = (1 - omega) v + omega D^-1 (f + tb2 S).
template <int N, int L, int C, int R>
__device__ __forceinline__ void at_sweep(At<N> &t, const float (&f)[R][C], float (&v)[R][C]) {
    float prev[C], below[C];
    t.template exchange<C>(v[0], v[R - 1], prev, below);
    const float tb2 = t.template tb2l<L>();
#pragma unroll
    for (int y = 0; y < R; ++y) {
        float S[C], w[C];
        at_nb<N, C>(t, prev, v[y], y == R - 1 ? below : v[y + 1 < R ? y + 1 : y], S);
        t.template relax<L, C>(y, w);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            prev[c] = v[y][c];
            v[y][c] = fmaf(w[c], fmaf(tb2, S[c], f[y][c]), (1.0f - AS_OMEGA) * v[y][c]);
        }
    }
}

// The horizontally weighted residual rows h (weights 1 2 1 over 4, at every second column) of
// v against f, for the full-weighting restriction.
template <int N, int L, int C, int R>
__device__ __forceinline__ void at_residual_rows(At<N> &t, const float (&f)[R][C], float (&v)[R][C],
                                                 float (&h)[R][C > 1 ? C / 2 : 1]) {
    float prev[C], below[C];
    t.template exchange<C>(v[0], v[R - 1], prev, below);
    const float tb2 = t.template tb2l<L>();
#pragma unroll
    for (int y = 0; y < R; ++y) {
        float S[C], r[C];
        at_nb<N, C>(t, prev, v[y], y == R - 1 ? below : v[y + 1 < R ? y + 1 : y], S);
#pragma unroll
        for (int c = 0; c < C; ++c) {
            prev[c] = v[y][c];
            r[c] = fmaf(-t.template diag<L>(y, c), v[y][c], fmaf(tb2, S[c], f[y][c]));
        }
        const float l = __shfl_sync(0xffffffffu, r[C - 1], t.left);
        if constexpr (C > 1) {
#pragma unroll
            for (int X = 0; X < C / 2; ++X) h[y][X] = 0.25f * ((X == 0 ? l : r[2 * X - 1]) + r[2 * X + 1]) + 0.5f * r[2 * X];
        } else {
            const float rr = __shfl_sync(0xffffffffu, r[0], t.right);
            h[y][0] = 0.25f * (l + rr) + 0.5f * r[0];
        }
    }
}

// ------------------------------------------------------------------- the one-warp levels
// A level of n x n (n = 16, 8 or 11) in one warp's registers: lane g n + x holds column x of the rows
// g R .. g R + R - 1 (G row groups, n = G R; lanes from G n on are idle and mirror lane 0).
template <int n>
struct TailCfg {
    static constexpr int G = n == 16 ? 2 : (n == 8 ? 4 : 1), R = n / G;
    static_assert(G * n <= 32 && G * R == n, "one warp");
};
template <int n>
struct TailLanes {
    int g, x, left, right, above, below;  // the lane's place and the lanes of its neighbours
    __device__ explicit TailLanes(int lane) {
        using T = TailCfg<n>;
        const int l = lane < T::G * n ? lane : 0;
        g = l / n;
        x = l - g * n;
        left = l + (x == 0 ? n - 1 : -1);
        right = l + (x == n - 1 ? 1 - n : 1);
        above = (g == 0 ? T::G - 1 : g - 1) * n + x;
        below = (g == T::G - 1 ? 0 : g + 1) * n + x;
    }
};

__device__ __forceinline__ float tail_shfl(float v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

// The neighbour sums of every point of the lane.
template <int n>
__device__ __forceinline__ void tail_nb(const TailLanes<n> &p, const float (&v)[TailCfg<n>::R], float (&S)[TailCfg<n>::R]) {
    constexpr int R = TailCfg<n>::R;
    const float a = TailCfg<n>::G == 1 ? v[R - 1] : tail_shfl(v[R - 1], p.above);
    const float b = TailCfg<n>::G == 1 ? v[0] : tail_shfl(v[0], p.below);
#pragma unroll
    for (int y = 0; y < R; ++y)
        S[y] = ((y == 0 ? a : v[y > 0 ? y - 1 : 0]) + (y == R - 1 ? b : v[y + 1 < R ? y + 1 : y])) +
               (tail_shfl(v[y], p.left) + tail_shfl(v[y], p.right));
}

// One damped-Jacobi sweep in place: w = omega / diagonal.
template <int n>
__device__ __forceinline__ void tail_sweep(const TailLanes<n> &p, const float (&f)[TailCfg<n>::R],
                                           const float (&w)[TailCfg<n>::R], float (&v)[TailCfg<n>::R], float tb2) {
    float S[TailCfg<n>::R];
    tail_nb<n>(p, v, S);
#pragma unroll
    for (int y = 0; y < TailCfg<n>::R; ++y) v[y] = fmaf(w[y], fmaf(tb2, S[y], f[y]), (1.0f - AS_OMEGA) * v[y]);
}

template <int n>
__device__ __forceinline__ void tail_coarsest(const TailLanes<n> &p, const float (&f)[TailCfg<n>::R],
                                              const float (&w)[TailCfg<n>::R], float (&v)[TailCfg<n>::R], float tb2) {
#pragma unroll
    for (int y = 0; y < TailCfg<n>::R; ++y) v[y] = w[y] * f[y];
#pragma unroll 1
    for (int k = 2; k <= AT_NU_COARSE; ++k) tail_sweep<n>(p, f, w, v, tb2);
}

// One cycle of the n x n level by one warp.  fs (shared memory): the right-hand side, then the result,
// the diagonals, omega / diagonal, and (n = 16) omega / diagonal of 8^2.
template <int n>
__device__ __noinline__ void tail_cycle(float *fs, float tb2, int lane) {
    constexpr int R = TailCfg<n>::R, G = TailCfg<n>::G;
    const TailLanes<n> p(lane);
    float f[R], w[R], v[R];
#pragma unroll
    for (int y = 0; y < R; ++y) {
        f[y] = fs[(p.g * R + y) * n + p.x];
        w[y] = fs[3 * n * n + (p.g * R + y) * n + p.x];
    }
    if constexpr (n != 16) {
        tail_coarsest<n>(p, f, w, v, tb2);
    } else {  // 16^2 over 8^2: lane 16 g + x of 16^2 holds rows 8 g .., lane 8 g + x of 8^2 rows 2 g, 2 g + 1
        const TailLanes<8> q(lane);
        float d[R], S[R], h[R], fc[2], wc[2], vc[2];
#pragma unroll
        for (int y = 0; y < R; ++y) {
            v[y] = w[y] * f[y];
        }
        tail_sweep<n>(p, f, w, v, tb2);
        tail_nb<n>(p, v, S);
        asm volatile("" ::: "memory");  // the diagonals are not loaded earlier: registers
#pragma unroll
        for (int y = 0; y < R; ++y) d[y] = fs[2 * n * n + (p.g * R + y) * n + p.x];
#pragma unroll
        for (int y = 0; y < R; ++y) {  // residual, weighted 1 2 1 along x
            const float r = fmaf(-d[y], v[y], fmaf(tb2, S[y], f[y]));
            h[y] = 0.25f * (tail_shfl(r, p.left) + tail_shfl(r, p.right)) + 0.5f * r;
        }
        const float ha = tail_shfl(h[R - 1], p.above);
        // coarse rows 4 g' .. of this lane's column (g' = its half), then to the 8^2 owners
        float cf[R / 2];
#pragma unroll
        for (int Y = 0; Y < R / 2; ++Y)
            cf[Y] = 0.25f * ((Y == 0 ? ha : h[Y > 0 ? 2 * Y - 1 : 0]) + h[2 * Y + 1]) + 0.5f * h[2 * Y];
        const int from = (q.g >> 1) * 16 + 2 * q.x;  // rows 2 q.g, 2 q.g + 1 = rows 2 (q.g & 1), + 1 of that half
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float f0 = tail_shfl(cf[i], from), f1 = tail_shfl(cf[2 + i], from);
            fc[i] = (q.g & 1) ? f1 : f0;
            wc[i] = fs[4 * n * n + (2 * q.g + i) * 8 + q.x];
        }
        tail_coarsest<8>(q, fc, wc, vc, 0.25f * tb2);
        // bilinear prolongation: coarse rows 4 g .. 4 g + 4 at columns x / 2 and (x odd) the next
        float e[R / 2 + 1];
        const int X = p.x >> 1, X1 = (p.x & 1) ? ((X + 1) & 7) : X;
#pragma unroll
        for (int Y = 0; Y <= R / 2; ++Y) {
            const int yc = (4 * p.g + Y) & 7, base = (yc >> 1) * 8;
            const float a0 = tail_shfl(vc[0], base + X), a1 = tail_shfl(vc[1], base + X);
            const float b0 = tail_shfl(vc[0], base + X1), b1 = tail_shfl(vc[1], base + X1);
            e[Y] = 0.5f * ((Y & 1) ? a1 + b1 : a0 + b0);  // 4 g is even: the row's parity is Y's
        }
#pragma unroll
        for (int y = 0; y < R; ++y) v[y] += (y & 1) ? 0.5f * (e[y >> 1] + e[(y >> 1) + 1]) : e[y >> 1];
        tail_sweep<n>(p, f, w, v, tb2);
        tail_sweep<n>(p, f, w, v, tb2);
    }
    if (lane < G * n) {
#pragma unroll
        for (int y = 0; y < R; ++y) fs[n * n + (p.g * R + y) * n + p.x] = v[y];
    }
}

// ------------------------------------------------------------------------- the register levels
// v = B f on level L and below: two damped-Jacobi sweeps (the first from zero), the coarse
// correction (full weighting, bilinear prolongation), two sweeps.
template <int N, int L, int C, int R>
__device__ __forceinline__ void at_cycle(At<N> &t, const float (&f)[R][C], float (&v)[R][C]) {
    using K = AtCfg<N>;
#pragma unroll
    for (int y = 0; y < R; ++y) {
        float w[C];
        t.template relax<L, C>(y, w);
#pragma unroll
        for (int c = 0; c < C; ++c) v[y][c] = w[c] * f[y][c];
    }
    at_sweep<N, L, C, R>(t, f, v);
    constexpr int HC = C > 1 ? C / 2 : 1;
    float cf[R / 2][HC];
    {
        float h[R][HC], ha[HC];
        at_residual_rows<N, L, C, R>(t, f, v, h);
        t.template from_above<HC>(h[R - 1], ha);
#pragma unroll
        for (int Y = 0; Y < R / 2; ++Y)
#pragma unroll
            for (int X = 0; X < HC; ++X)
                cf[Y][X] = 0.25f * ((Y == 0 ? ha[X] : h[Y == 0 ? 0 : 2 * Y - 1][X]) + h[2 * Y + 1][X]) + 0.5f * h[2 * Y][X];
    }
    if constexpr (C > 1) {
        float e[R / 2][HC], eb[HC], er[R / 2 + 1];
        at_cycle<N, L + 1, HC, R / 2>(t, cf, e);
        t.template from_below<HC>(e[0], eb);
#pragma unroll
        for (int Y = 0; Y < R / 2; ++Y) er[Y] = __shfl_sync(0xffffffffu, e[Y][0], t.right);
        er[R / 2] = __shfl_sync(0xffffffffu, eb[0], t.right);
#pragma unroll
        for (int Y = 0; Y < R / 2; ++Y) {
            float a[HC + 1], b[HC + 1];  // coarse rows Y and Y + 1 with the column to the right
#pragma unroll
            for (int X = 0; X < HC; ++X) {
                a[X] = e[Y][X];
                b[X] = Y + 1 < R / 2 ? e[Y + 1 < R / 2 ? Y + 1 : Y][X] : eb[X];
            }
            a[HC] = er[Y];
            b[HC] = er[Y + 1];
#pragma unroll
            for (int X = 0; X < HC; ++X) {
                const float m0 = 0.5f * (a[X] + a[X + 1]), m1 = 0.5f * (b[X] + b[X + 1]);
                v[2 * Y][2 * X] += a[X];
                v[2 * Y][2 * X + 1] += m0;
                v[2 * Y + 1][2 * X] += 0.5f * (a[X] + b[X]);
                v[2 * Y + 1][2 * X + 1] += 0.5f * (m0 + m1);
            }
        }
    } else {
        constexpr int TN = K::TN;
        float *tf = t.sm + K::T, *tv = tf + TN * TN;
        if ((t.lane & 1) == 0 && t.lane < K::LU) {
#pragma unroll
            for (int Y = 0; Y < R / 2; ++Y) tf[(t.warp * (R / 2) + Y) * TN + (t.lane >> 1)] = cf[Y][0];
        }
        __syncthreads();
        if (t.warp == 0) tail_cycle<TN>(tf, t.template tb2l<L + 1>(), t.lane);
        __syncthreads();
        const int x = t.lane < K::LU ? t.lane : 0, X = x >> 1, X1 = (x & 1) ? (X + 1 == TN ? 0 : X + 1) : X;
#pragma unroll
        for (int y = 0; y < R; ++y) {
            const int Y = t.warp * (R / 2) + (y >> 1), Y1 = (y & 1) ? (Y + 1 == TN ? 0 : Y + 1) : Y;
            v[y][0] += 0.25f * ((tv[Y * TN + X] + tv[Y * TN + X1]) + (tv[Y1 * TN + X] + tv[Y1 * TN + X1]));
        }
    }
    at_sweep<N, L, C, R>(t, f, v);
    at_sweep<N, L, C, R>(t, f, v);
}

// What holds of the one-warp levels for a Newton pass: the diagonals of the first from the threads'
// masks (the count over a 2^LEVELS square is the lane's block of 2^LEVELS rows and the right lane's), and
// the relaxation factors.
template <int N>
__device__ __forceinline__ void at_hold_tail(At<N> &t) {
    using K = AtCfg<N>;
    constexpr int TN = K::TN, LV = K::LEVELS, TR = K::RW >> LV;
    constexpr float area = 1.0f / (1 << (2 * LV));
    float *td = t.sm + K::T + 2 * TN * TN, *tw = td + TN * TN, *tw8 = tw + TN * TN;
    const float d0 = t.tb1 + 4.0f * t.tb2 * area;
#pragma unroll
    for (int Y = 0; Y < TR; ++Y) {
        const unsigned rows = t.mask & ((K::CW << LV) == 32 ? 0xffffffffu
                                                            : ((1u << ((K::CW << LV) & 31)) - 1u) << (Y * (K::CW << LV)));
        const int own = __popc(rows), both = own + __shfl_sync(0xffffffffu, own, t.right);
        if ((t.lane & 1) == 0 && t.lane < K::LU) {
            const float d = fmaf((float)both, t.icg * area, d0);
            td[(t.warp * TR + Y) * TN + (t.lane >> 1)] = d;
            tw[(t.warp * TR + Y) * TN + (t.lane >> 1)] = AS_OMEGA / d;
        }
    }
    if constexpr (TN == 16) {  // 8^2: the mean of m icg is the diagonals' mean less the stencil's part
        __syncthreads();
        if (threadIdx.x < 64) {
            const float *d = td + (threadIdx.x >> 3) * 32 + (threadIdx.x & 7) * 2;
            const float tb2 = t.tb2 * area, s16 = t.tb1 + 4.0f * tb2, s8 = t.tb1 + tb2;
            tw8[threadIdx.x] = AS_OMEGA / (0.25f * ((d[0] + d[16]) + (d[1] + d[17])) - s16 + s8);
        }
    }
}

// g = e2a (disc sums of u) + c_F u by the CTA: the transforms of half_fft.cuh in FP64.  smem:
// hf_smem_bytes<N, double>() bytes.  Begins and ends with a CTA barrier.
template <int N>
__device__ __noinline__ void at_disc_sums(const double *U, double *G, const AsFactor *tab, const double2 *twg,
                                          double2 *smem, double e2a, double cF) {
    using K = HfCfg<N>;
    Hf<N, double2> h;
    double2 *tw = smem + K::Z;
    h.z = smem;
    h.tw = tw;
    h.warp = threadIdx.x >> 5;
    h.lane = threadIdx.x & 31;
    __syncthreads();
    for (int i = threadIdx.x; i < K::TW; i += K::NT) tw[i] = twg[i];
    __syncthreads();
    const size_t r0 = (size_t)(2 * h.my_row()) * N + h.n1();
    double2 v[K::A];
#pragma unroll
    for (int j = 0; j < K::A; ++j) v[j] = make_double2(U[r0 + 8 * j], U[r0 + N + 8 * j]);
    h.rows_forward(v);
    __syncthreads();
    h.columns(tab);
    __syncthreads();
    h.rows_inverse(v);
#pragma unroll
    for (int j = 0; j < K::A; ++j) {
        G[r0 + 8 * j] = fma(e2a, v[j].x, cF * U[r0 + 8 * j]);
        G[r0 + N + 8 * j] = fma(e2a, v[j].y, cF * U[r0 + N + 8 * j]);
    }
    __syncthreads();
}

template <int N, int MINB>
__global__ void __launch_bounds__(AtCfg<N>::NT, MINB) active_set_tile_kernel(const __grid_constant__ AsTileArgs a) {
    using K = AtCfg<N>;
    constexpr int CW = K::CW, RW = K::RW, nn = N * N;
    extern __shared__ __align__(16) float at_smem[];
    __shared__ float red[64];
    __shared__ int widths[kMaxR + 1];
    __shared__ double red64[K::NW];
    const size_t smp = a.s0 + blockIdx.x;
    const unsigned long long t_start = a.trace.rec ? trace_clock() : 0ull;
    At<N> t;
    t.sm = at_smem;
    t.red = red;
    t.warp = threadIdx.x >> 5;
    t.lane = threadIdx.x & 31;
    const bool act = t.lane < K::LU;
    t.slot = (t.warp * K::LU + (act ? t.lane : 0)) * CW;
    t.left = t.lane == 0 ? K::LU - 1 : t.lane - 1;
    t.right = t.lane >= K::LU - 1 ? 0 : t.lane + 1;
    t.par = t.rpar = 0;
    t.mask = 0u;
    double *U = a.buf + smp * as_tile_per_sample(N), *G = U + nn, *W = G + nn;
    // the thread's slot of p, q and d: row y at + y * N * NW floats... [row][warp][lane] vectors
    constexpr int SROW = K::NW * K::LU * CW;
    float *D = reinterpret_cast<float *>(W + nn) + t.slot, *Pp = at_smem + K::P + t.slot, *Qp = at_smem + K::Q + t.slot;
    const int own = t.warp * RW * N + (act ? t.lane : 0) * CW;  // the thread's first point
    if (threadIdx.x <= a.R) widths[threadIdx.x] = a.widths[threadIdx.x];
    const double eps = a.eps ? a.eps[smp] : a.eps_nominal;
    const double e2a = eps * eps * a.ahat, cg = e2a * a.chat, icg = 1.0 / cg;
    const double tb1 = a.tau * a.beta1, tb2h = a.tau * a.beta2 * (double)N * (double)N;
    // the residual is formed as c_gamma F = (c_gamma tau A) w + P_[-c_gamma, c_gamma](w + g) - c_gamma u:
    // no quotient, and one operation fewer than with the product by 1 / c_gamma
    const double cgtb2 = cg * tb2h, cgdiag = fma(4.0, cgtb2, cg * tb1), ftol = 1e-11 * cg;
    const unsigned long long cgbits = (unsigned long long)__double_as_longlong(cg);
    t.tb1 = (float)tb1;
    t.icg = (float)icg;
    t.tb2 = (float)tb2h;
    t.d0 = t.tb1 + 4.0f * t.tb2;
    t.d1 = t.d0 + t.icg;
    t.w0 = AS_OMEGA / t.d0;
    t.w1 = AS_OMEGA / t.d1;
    for (int i = threadIdx.x; i < nn; i += K::NT) U[i] = (double)a.u0[smp * (size_t)nn + i];
    __syncthreads();
    const bool roomy = a.newton_max >= kAsNewtonMax;  // room for loose corrections and restarts
    bool failed = false;
    unsigned long long n_newton = 0, n_cg = 0;
    for (int step = 1; step <= a.nsteps && !failed; ++step) {
        // explicit part g = gamma * u + c_F u
        if (a.tab) {
            at_disc_sums<N>(U, G, a.tab, a.tw, reinterpret_cast<double2 *>(at_smem), e2a, a.cF);
        } else {
            for (int i = threadIdx.x; i < nn; i += K::NT) {
                const int y = i / N, x = i - y * N;
                double S = 0.0;
                for (int dy = -a.R; dy <= a.R; ++dy) {
                    const int ady = dy < 0 ? -dy : dy, w = widths[ady];
                    int yy = y + dy;
                    yy += yy < 0 ? N : 0;
                    yy -= yy >= N ? N : 0;
                    int xx = x - w;
                    xx += xx < 0 ? N : 0;
                    for (int dx = -w; dx <= w; ++dx) {
                        S += a.wtab ? a.wtab[ady * ady + dx * dx] * U[yy * N + xx] : U[yy * N + xx];
                        xx = xx == N - 1 ? 0 : xx + 1;
                    }
                }
                G[i] = e2a * S + a.cF * U[i];
            }
            __syncthreads();
        }
        for (int it = 1;; ++it) {
            // start: w of the previous step, or the beta2 = 0 step's, at the first step and where a step has
            // not come home (its active set cycles)
            if (it == 1 ? step == 1 : roomy && (it == AT_LOOSE_PASSES + 1 || it == AT_TIGHT_PASSES + 1)) {
                for (int i = threadIdx.x; i < nn; i += K::NT) {
                    const double u0 = at_clip((U[i] + tb1 * G[i]) / (1.0 + tb1 * cg));
                    W[i] = cg * u0 - G[i];
                }
                __syncthreads();
            }
            ++n_newton;
            // FP64 residual c_gamma F(w), the inactive set, and the right-hand side of J d = -F, which is
            // f = -(c_gamma F) / max |c_gamma F| with d scaled back by max |c_gamma F| / c_gamma
            float f[RW][CW];
            unsigned fhi = 0u;  // maximum of the high words of |c_gamma F|: a NaN's lies above every number's
            unsigned now = 0u;
            {
                double up[CW], cur[CW], dn[CW];
                at_ld64<CW>(up, W + (t.warp == 0 ? nn - N + own : own - N));
                at_ld64<CW>(cur, W + own);
#pragma unroll
                for (int y = 0; y < RW; ++y) {
                    const int i = own + y * N;
                    double g[CW], u[CW];
                    at_ld64<CW>(dn, W + (y == RW - 1 && t.warp == K::NW - 1 ? i + N - nn : i + N));
                    at_ld64<CW>(g, G + i);
                    at_ld64<CW>(u, U + i);
                    const double l = __shfl_sync(0xffffffffu, cur[CW - 1], t.left);
                    const double r = __shfl_sync(0xffffffffu, cur[0], t.right);
#pragma unroll
                    for (int c = 0; c < CW; ++c) {
                        const double S = (up[c] + dn[c]) + ((c == 0 ? l : cur[c > 0 ? c - 1 : 0]) +
                                                            (c == CW - 1 ? r : cur[c + 1 < CW ? c + 1 : c]));
                        const double z = cur[c] + g[c];
                        // |z| < c_gamma and the projection on the bit patterns (no FP64 compares)
                        const unsigned long long zb = (unsigned long long)__double_as_longlong(z);
                        const bool in = (zb & ~(1ull << 63)) < cgbits;
                        const double zc = in ? z : __longlong_as_double((long long)((zb & 1ull << 63) | cgbits));
                        const double F = fma(cgdiag, cur[c], fma(-cgtb2, S, fma(-cg, u[c], zc)));
                        now |= in ? 1u << (y * CW + c) : 0u;
                        f[y][c] = act ? -(float)F : 0.0f;
                        fhi = umax(fhi, (unsigned)__double2hiint(F) & 0x7fffffffu);
                    }
#pragma unroll
                    for (int c = 0; c < CW; ++c) {
                        up[c] = cur[c];
                        cur[c] = dn[c];
                    }
                }
            }
            const bool changed = __syncthreads_or(act && now != t.mask);
            t.mask = now;
            // the largest value with that high word: what passes meets the bound in full
            const double fbound = __hiloint2double((int)t.max_bits(act ? fhi : 0u), -1);
            if (it > 1 && !changed && fbound <= ftol) break;
            // the bound on the passes, or a residual that no pass mends (a NaN or an infinity, which the
            // correction would carry to every point): the sample's solve stops
            if (it > a.newton_max || !(fbound < INFINITY)) {
                failed = true;
                break;
            }
            const float fmax = (float)fbound;
            if (fmax < FLT_MIN) continue;  // F = 0 with a new active set: the next pass confirms it
            at_hold_tail<N>(t);
            if constexpr (K::HOLD) t.template hold_relax<1>();
            const float sc = 1.0f / fmax;  // scaled to max |f| = 1
#pragma unroll
            for (int y = 0; y < RW; ++y)
#pragma unroll
                for (int c = 0; c < CW; ++c) f[y][c] *= sc;
            // CG on J d = f from d = 0, preconditioned by one V-cycle, to a residual that matches what the
            // correction can be worth: while the active set still moves it limits the next residual, not
            // the solve, and on a settled set the next residual is this one times the tolerance (AS_CG_RTOL
            // throughout: 33.1 CG iterations a step of 128^2 samples, now 26.1).  The loose corrections
            // cost a pass here and there (4.8 -> 5.1), and where the active set is close to cycling they can
            // make it cycle: under a caller's tighter bound there are none, and a step that they do not
            // bring home starts over without them.
            const bool loose = roomy && it <= AT_LOOSE_PASSES;
            const float rtol = loose && it == 1 ? 3e-2f : (loose && changed ? 1e-3f : (changed || it == 1 ? AS_CG_RTOL : 1e-6f));
            float rz = 0.0f;
            for (int k = 1;; ++k) {
                float v[RW][CW];
                at_cycle<N, 0, CW, RW>(t, f, v);
                float dot = 0.0f;
#pragma unroll
                for (int y = 0; y < RW; ++y)
#pragma unroll
                    for (int c = 0; c < CW; ++c) dot = fmaf(f[y][c], v[y][c], dot);
                const float rz2 = t.sum(act ? dot : 0.0f), beta = k == 1 ? 0.0f : rz2 / rz;
                rz = rz2;
                // p = z + beta p, q = J z + beta q
                float pq = 0.0f;
                {
                    float prev[CW], below[CW];
                    t.template exchange<CW>(v[0], v[RW - 1], prev, below);
#pragma unroll
                    for (int y = 0; y < RW; ++y) {
                        float S[CW], p[CW], q[CW];
                        at_nb<N, CW>(t, prev, v[y], y == RW - 1 ? below : v[y + 1 < RW ? y + 1 : y], S);
                        if (k > 1 && act) {
                            at_ld<CW>(p, Pp + y * SROW);
                            at_ld<CW>(q, Qp + y * SROW);
                        } else {
#pragma unroll
                            for (int c = 0; c < CW; ++c) p[c] = q[c] = 0.0f;
                        }
#pragma unroll
                        for (int c = 0; c < CW; ++c) {
                            prev[c] = v[y][c];
                            const float jz = fmaf(t.template diag<0>(y, c), v[y][c], -t.tb2 * S[c]);
                            p[c] = fmaf(beta, p[c], v[y][c]);
                            q[c] = fmaf(beta, q[c], jz);
                            pq = fmaf(p[c], q[c], pq);
                        }
                        if (act) {
                            at_st<CW>(Pp + y * SROW, p);
                            at_st<CW>(Qp + y * SROW, q);
                        }
                    }
                }
                pq = t.sum(act ? pq : 0.0f);
                const float alpha = pq > 0.0f ? rz / pq : 0.0f;
                float rmax = 0.0f;
                if (act) {
#pragma unroll
                    for (int y = 0; y < RW; ++y) {
                        float p[CW], q[CW];
                        at_ld<CW>(p, Pp + y * SROW);
                        at_ld<CW>(q, Qp + y * SROW);
#pragma unroll
                        for (int c = 0; c < CW; ++c) {
                            p[c] *= alpha;
                            f[y][c] = fmaf(-alpha, q[c], f[y][c]);
                            rmax = fmaxf(rmax, fabsf(f[y][c]));
                        }
                        if (k == 1)
                            at_st<CW>(D + y * SROW, p);
                        else
                            at_red<CW>(D + y * SROW, p);
                    }
                }
                rmax = t.max(rmax);
                if (rmax <= rtol || !(pq > 0.0f) || !(rz > 0.0f) || k >= a.cg_max) {
                    n_cg += k;
                    break;
                }
            }
            if (act) {
                const bool damped = roomy && it > AT_TIGHT_PASSES && it <= AT_TIGHT_PASSES + AT_DAMPED;
                const double scale = (double)fmax * (damped ? 0.5 * icg : icg);
#pragma unroll
                for (int y = 0; y < RW; ++y) {
                    double w[CW];
                    at_ld64<CW>(w, W + own + y * N);
#pragma unroll
                    for (int c = 0; c < CW; ++c) w[c] = fma(scale, (double)__ldcg(D + y * SROW + c), w[c]);
                    at_st64<CW>(W + own + y * N, w);
                }
            }
            __syncthreads();
        }
        if (failed) break;
        if (act) {
#pragma unroll
            for (int y = 0; y < RW; ++y) {
                double w[CW], g[CW];
                at_ld64<CW>(w, W + own + y * N);
                at_ld64<CW>(g, G + own + y * N);
#pragma unroll
                for (int c = 0; c < CW; ++c) w[c] = at_clip(at_div(w[c] + g[c], cg, icg));
                at_st64<CW>(U + own + y * N, w);
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicAdd(&a.iters[0], n_newton);
        atomicAdd(&a.iters[1], n_cg);
        trace_put(a.trace, kTraceActiveSet, (uint32_t)smp, (uint32_t)a.nsteps, t_start);
    }
    if (failed) {
        if (threadIdx.x == 0) atomicExch(a.status, 1);
        return;
    }
    double s = 0.0;
    for (int i = threadIdx.x; i < nn; i += K::NT) {
        const double u = U[i];
        s += u;
        if (a.uT) a.uT[smp * (size_t)nn + i] = (float)u;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (t.lane == 0) red64[t.warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int i = 0; i < K::NW; ++i) tot += red64[i];
        const double mean = tot / (double)nn;
        if (a.ubar) a.ubar[smp] = mean;
        if (a.ooi) a.ooi[smp] = 0.5 * (1.0 + mean);
    }
}

template <int N, int MINB>
mfmc_status at_launch(const AsTileArgs &a, unsigned grid, cudaStream_t st) {
    using K = AtCfg<N>;
    size_t smem = K::SMEM;
    if (a.tab) smem = std::max(smem, hf_smem_bytes<N, double>());
    auto kern = active_set_tile_kernel<N, MINB>;
    MFMC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<grid, K::NT, smem, st>>>(a);
    MFMC_LAUNCHED("active_set_tile launch");
    return MFMC_OK;
}

}  // namespace

bool as_tile_supported(int n) { return n == 64 || n == 88 || n == 128; }

mfmc_status launch_active_set_tile(const AsTileArgs &a, int n, unsigned grid, cudaStream_t st) {
    switch (n) {
        case 64: return at_launch<64, 4>(a, grid, st);
        case 88: return at_launch<88, 2>(a, grid, st);
        case 128: return at_launch<128, 1>(a, grid, st);
        default: return fail(MFMC_EINVAL, "no on-chip active-set kernel for n = %d", n);
    }
}

}  // namespace mfmc
