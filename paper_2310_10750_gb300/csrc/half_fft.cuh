// Periodic disc sums of an N x N lattice (N = 64, 88, 128) by FFT, in registers and shared memory,
// FP32 or FP64: S = IFFT2(FFT2(u) K^) with K^ the (real, even) transform of the disc weights.
//
// Packing.  Rows 2p and 2p + 1 make one complex row, z[p][x] = u[2p][x] + i u[2p + 1][x], so the
// transforms run on N/2 x N complex values.  With Z = DFT2(z) (N/2 points over p, N over x), the
// transforms of the even and odd rows are E = (Z[q][k] + conj Z[-q][-k]) / 2 and
// O = (Z[q][k] - conj Z[-q][-k]) / 2i, the lattice's transform is E + W O at row frequency q and
// E - W O at q + N/2 (W = exp(-2 pi i q / N)), and the sums' even and odd rows have the transforms
//     Se = Kp E2 + T O2,   So = conj(T) E2 + Kp O2,   E2 = 2E, O2 = 2O,
//     Kp = (K^[q] + K^[q + N/2]) / (2 N^2),   T = W (K^[q] - K^[q + N/2]) / (2 N^2),
// so the product is local to the pair (q, k), (-q, -k).  Column k and column -k are transformed by
// the same threads, the second conjugated: its transform then holds conj Z[-q][-k] where the first
// holds Z[q][k], and the product needs no exchange.  (Columns 0 and N/2 are their own partners;
// they share a slot and exchange through shared memory.)
//
// Transforms.  A row transform is N = A x 8: 8 lanes transform A values each in registers
// (x = n1 + 8j), multiply by W_N^(n1 k2), and after an exchange inside the warp A items transform
// 8 values each; the inverse runs the same steps backwards, so it ends where the forward begins
// and the field can stay in registers between steps.  A column transform is N/2 = A2 x B2 the same
// way, in place in the column's own storage.  A warp takes four packed rows, then four column
// pairs: N/8 warps.  Every shared-memory access is free of bank conflicts at FP32 and FP64 but
// for a few lanes (row pitch RS, position k1 PA + k2 of frequency k = k2 + A k1, skewed column
// exchange).  Per complex value a step makes 12 shared-memory accesses; the unpacked form it
// replaces made about 25, with one 9-warp CTA per SM.
#pragma once

#include <cuda_runtime.h>

#include "smem_fft.cuh"

namespace mfmc {

template <int N>
struct HfCfg {
    static constexpr int H = N / 2;
    static constexpr int A = N / 8, B = 8;             // row transform: A values a lane, 8 lanes
    static constexpr int B2 = N == 128 ? 8 : 4, A2 = H / B2;
    static constexpr int PA = A % 2 ? A : A + 1;       // spacing of the lanes' runs in a row
    // row pitch in complex values: 4 or 12 mod 16
    static constexpr int RS = N == 128 ? 140 : (N == 88 ? 92 : 76);
    static constexpr int NW = N / 8, NT = 32 * NW;
    static constexpr int TR = (A + 1) / 2 * 2 + 2;      // pitch of the row twiddles (complex)
    static constexpr int TC = A2 + (A2 % 2 ? 2 : 1);    // pitch of the column twiddles
    static constexpr int TW = B * TR + B2 * TC;          // complex values of both twiddle tables
    static constexpr int Z = H * RS;                     // complex values of the packed lattice
    static_assert(A * B == N && A2 * B2 == H && (RS % 16 == 4 || RS % 16 == 12) && RS >= 7 * PA + A, "layout");
};

__host__ __device__ constexpr bool hf_supported(int n) { return n == 64 || n == 88 || n == 128; }

template <typename C>
using hf_real = decltype(C().x);

__device__ __forceinline__ float2 hadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 hsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ double2 hadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 hsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// a (c - i s), conjugated for the inverse: the twiddle of angle -theta with c = cos, s = sin.
template <bool INV, typename C>
__device__ __forceinline__ C hrot(C a, hf_real<C> c, hf_real<C> s) {
    C o;
    o.x = INV ? fma(-s, a.y, c * a.x) : fma(s, a.y, c * a.x);
    o.y = INV ? fma(s, a.x, c * a.y) : fma(-s, a.x, c * a.y);
    return o;
}
// a w, conjugated w for the inverse
template <bool INV, typename C>
__device__ __forceinline__ C hmul(C a, C w) {
    C o;
    o.x = INV ? fma(a.x, w.x, a.y * w.y) : fma(a.x, w.x, -(a.y * w.y));
    o.y = INV ? fma(a.y, w.x, -(a.x * w.y)) : fma(a.y, w.x, a.x * w.y);
    return o;
}

// P-point transforms in registers, natural order in and out.
template <bool INV, typename C>
__device__ __forceinline__ void hdft4(C &a, C &b, C &c, C &d) {
    const C s0 = hadd(a, c), d0 = hsub(a, c), s1 = hadd(b, d), e = hsub(b, d);
    const C d1 = frot<INV>(e);
    a = hadd(s0, s1);
    c = hsub(s0, s1);
    b = hadd(d0, d1);
    d = hsub(d0, d1);
}

template <int P, bool INV, typename C>
__device__ __forceinline__ void hdft(C (&v)[P]) {
    using T = hf_real<C>;
    constexpr T r2 = T(0.70710678118654752440);  // cos(pi / 4)
    if constexpr (P == 4) {
        hdft4<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (P == 8) {
        // even and odd points, W_8^k on the odd ones, then pairs k, k + 4
        C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        hdft4<INV>(e[0], e[1], e[2], e[3]);
        hdft4<INV>(o[0], o[1], o[2], o[3]);
        C t;
        t = o[1];  // (1 - i) / sqrt 2 (inverse: its conjugate)
        o[1].x = r2 * (INV ? t.x - t.y : t.x + t.y);
        o[1].y = r2 * (INV ? t.y + t.x : t.y - t.x);
        o[2] = frot<INV>(o[2]);
        t = o[3];  // (-1 - i) / sqrt 2
        o[3].x = r2 * (INV ? -t.x - t.y : t.y - t.x);
        o[3].y = r2 * (INV ? t.x - t.y : -t.y - t.x);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = hadd(e[k], o[k]);
            v[k + 4] = hsub(e[k], o[k]);
        }
    } else if constexpr (P == 16) {
        constexpr T c1 = T(0.92387953251128675613), s1 = T(0.38268343236508977173);  // cos, sin(pi / 8)
        // four transforms over points i + 4j, W_16^(ik), then four over i: X[k + 4m]
#pragma unroll
        for (int i = 0; i < 4; ++i) hdft4<INV>(v[i], v[i + 4], v[i + 8], v[i + 12]);
        // v[i + 4k] = y_i[k]
        v[5] = hrot<INV>(v[5], c1, s1);
        v[9] = hrot<INV>(v[9], r2, r2);
        v[13] = hrot<INV>(v[13], s1, c1);
        v[6] = hrot<INV>(v[6], r2, r2);
        v[10] = frot<INV>(v[10]);
        v[14] = hrot<INV>(v[14], -r2, r2);
        v[7] = hrot<INV>(v[7], s1, c1);
        v[11] = hrot<INV>(v[11], -r2, r2);
        v[15] = hrot<INV>(v[15], -c1, -s1);
#pragma unroll
        for (int k = 0; k < 4; ++k) hdft4<INV>(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        // X[k + 4m] is in v[4k + m]
        C o[16];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int m = 0; m < 4; ++m) o[k + 4 * m] = v[4 * k + m];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = o[k];
    } else {
        static_assert(P == 11, "radix");
        // conjugate pairs (q, 11 - q): X_k = a_0 + sum cos S_q, Y_k = sum sin D_q
        constexpr T cs[6] = {T(1), T(0.84125353283118116886), T(0.41541501300188642553),
                             T(-0.14231483827328514044), T(-0.65486073394528506406), T(-0.95949297361449738989)};
        constexpr T sn[6] = {T(0), T(0.54064081745559758211), T(0.90963199535451837141),
                             T(0.98982144188093273238), T(0.75574957435425828377), T(0.28173255684142969771)};
        C S[6], D[6], b0 = v[0];
#pragma unroll
        for (int q = 1; q < 6; ++q) {
            S[q] = hadd(v[q], v[11 - q]);
            D[q] = hsub(v[q], v[11 - q]);
            b0 = hadd(b0, S[q]);
        }
        const C a0 = v[0];
        v[0] = b0;
#pragma unroll
        for (int k = 1; k < 6; ++k) {
            C X = a0, Y;
            Y.x = Y.y = T(0);
#pragma unroll
            for (int q = 1; q < 6; ++q) {
                const int j = (q * k) % 11, m = j < 6 ? j : 11 - j;
                const T c = cs[m], s = j < 6 ? -sn[m] : sn[m];  // W^j = c + i s
                X.x = fma(c, S[q].x, X.x);
                X.y = fma(c, S[q].y, X.y);
                Y.x = fma(s, D[q].x, Y.x);
                Y.y = fma(s, D[q].y, Y.y);
            }
            C iY;
            iY.x = -Y.y;
            iY.y = Y.x;
            v[k] = INV ? hsub(X, iY) : hadd(X, iY);
            v[11 - k] = INV ? hadd(X, iY) : hsub(X, iY);
        }
    }
}

// A thread's place in the CTA's transforms (warp: index among the N / 8 warps of the lattice).
// tw: the twiddle tables (hf_twiddles) in shared memory; z: HfCfg<N>::Z complex values of it.
template <int N, typename C>
struct Hf {
    using K = HfCfg<N>;
    C *z;
    const C *tw;
    int warp, lane;
    // the four packed rows of a warp in the order 0, 2, 1, 3: lanes of a half warp then take rows
    // two apart, whose banks do not overlap
    __device__ __forceinline__ int row(int g) const { return 4 * warp + ((g & 1) << 1) + (g >> 1); }
    __device__ __forceinline__ int n1() const { return lane & 7; }
    __device__ __forceinline__ int my_row() const { return row(lane >> 3); }  // the lane's packed row
    __device__ __forceinline__ static int pos(int k) { return k / K::A * K::PA + k % K::A; }
    // place of (m1, q2) among the column's rows during its exchange
    __device__ __forceinline__ static int skew(int m1, int q2) {
        return K::A2 == 8 ? m1 * 8 + ((q2 + m1) & 7) : m1 * K::A2 + q2;
    }
    // the row twiddles W_N^(n1 k2) of the lane, two at a time (k2 even)
    __device__ __forceinline__ void row_tw(int k2, C &w0, C &w1) const {
        const C *p = tw + n1() * K::TR + k2;
        if constexpr (sizeof(C) == 8) {
            const float4 t = *reinterpret_cast<const float4 *>(p);
            w0 = C{t.x, t.y};
            w1 = C{t.z, t.w};
        } else {
            w0 = p[0];
            w1 = p[1];
        }
    }

    // v: the lane's A values of its packed row (x = n1 + 8j).  Leaves the row's transform in z.
    __device__ __forceinline__ void rows_forward(C (&v)[K::A]) const {
        hdft<K::A, false>(v);
        C *r = z + my_row() * K::RS + n1() * K::PA;
#pragma unroll
        for (int k2 = 0; k2 < K::A; k2 += 2) {
            C w0, w1;
            row_tw(k2, w0, w1);
            r[k2] = k2 == 0 ? v[0] : hmul<false>(v[k2], w0);
            if (k2 + 1 < K::A) r[k2 + 1] = hmul<false>(v[k2 + 1 < K::A ? k2 + 1 : 0], w1);
        }
        __syncwarp();
#pragma unroll
        for (int i0 = 0; i0 < 4 * K::A; i0 += 32) {
            const int i = i0 + lane;
            if (4 * K::A % 32 == 0 || i < 4 * K::A) {
                C *p = z + row(i / K::A) * K::RS + i % K::A;
                C y[8];
#pragma unroll
                for (int m = 0; m < 8; ++m) y[m] = p[m * K::PA];
                hdft<8, false>(y);
#pragma unroll
                for (int m = 0; m < 8; ++m) p[m * K::PA] = y[m];
            }
        }
    }

    // The inverse: v becomes the lane's A values of its packed row of sums.
    __device__ __forceinline__ void rows_inverse(C (&v)[K::A]) const {
#pragma unroll
        for (int i0 = 0; i0 < 4 * K::A; i0 += 32) {
            const int i = i0 + lane;
            if (4 * K::A % 32 == 0 || i < 4 * K::A) {
                C *p = z + row(i / K::A) * K::RS + i % K::A;
                C y[8];
#pragma unroll
                for (int m = 0; m < 8; ++m) y[m] = p[m * K::PA];
                hdft<8, true>(y);
#pragma unroll
                for (int m = 0; m < 8; ++m) p[m * K::PA] = y[m];
            }
        }
        __syncwarp();
        const C *r = z + my_row() * K::RS + n1() * K::PA;
#pragma unroll
        for (int k2 = 0; k2 < K::A; k2 += 2) {
            C w0, w1;
            row_tw(k2, w0, w1);
            v[k2] = k2 == 0 ? r[0] : hmul<true>(r[k2], w0);
            if (k2 + 1 < K::A) v[k2 + 1 < K::A ? k2 + 1 : 0] = hmul<true>(r[k2 + 1], w1);
        }
        hdft<K::A, true>(v);
    }

    // The product at one pair: a = Z[q][k], b = conj Z[-q][-k] -> the same of the sums' transform.
    // t: {Kp, Re T, Im T, what their FP32 rounding leaves of K^[q], added to Kp (FP64: not read)}.
    template <typename T4>
    __device__ __forceinline__ static void product(C &a, C &b, const T4 &t) {
        C e, o, se, so;
        e.x = a.x + b.x;
        e.y = a.y + b.y;
        o.x = a.y - b.y;  // -i (a - b)
        o.y = b.x - a.x;
        se.x = -(t.z * o.y);
        se.y = t.z * o.x;
        so.x = t.z * e.y;
        so.y = -(t.z * e.x);
        if constexpr (sizeof(T4) == 16) {
            se.x = fma(t.w, e.x, se.x);
            se.y = fma(t.w, e.y, se.y);
            so.x = fma(t.w, o.x, so.x);
            so.y = fma(t.w, o.y, so.y);
        }
        se.x = fma(t.x, e.x, fma(t.y, o.x, se.x));
        se.y = fma(t.x, e.y, fma(t.y, o.y, se.y));
        so.x = fma(t.x, o.x, fma(t.y, e.x, so.x));
        so.y = fma(t.x, o.y, fma(t.y, e.y, so.y));
        a.x = se.x - so.y;  // se + i so
        a.y = se.y + so.x;
        b.x = se.x + so.y;  // se - i so
        b.y = se.y - so.x;
    }

    // Column pass over the row transforms of all warps (a CTA barrier before and after it):
    // forward, product with tab[c][q] (c = 0 .. N/2), inverse.
    template <typename T4>
    __device__ __forceinline__ void columns(const T4 *__restrict__ tab) const {
        constexpr int A2 = K::A2, B2 = K::B2, RS = K::RS, I1 = 8 * B2, R1 = I1 / 32;
        static_assert(I1 % 32 == 0, "stage 1 fills the warp");
        const C *twc = tw + K::B * K::TR;
        {
            C v[R1][A2];
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const int i = 32 * r + lane, c = 4 * warp + (i & 3), m1 = (i >> 2) % B2, ab = (i >> 2) / B2;
                const C *p = z + pos(ab ? (c == 0 ? K::H : N - c) : c) + m1 * RS;
#pragma unroll
                for (int j = 0; j < A2; ++j) {
                    v[r][j] = p[j * B2 * RS];
                    if (ab) v[r][j].y = -v[r][j].y;
                }
                hdft<A2, false>(v[r]);
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const int i = 32 * r + lane, c = 4 * warp + (i & 3), m1 = (i >> 2) % B2, ab = (i >> 2) / B2;
                C *p = z + pos(ab ? (c == 0 ? K::H : N - c) : c);
#pragma unroll
                for (int q2 = 0; q2 < A2; ++q2)
                    p[skew(m1, q2) * RS] = q2 == 0 ? v[r][0] : hmul<false>(v[r][q2], twc[m1 * K::TC + q2]);
            }
            __syncwarp();
        }
        {
            constexpr int I2 = 4 * A2, R2 = (I2 + 31) / 32;
            C a[R2][B2], b[R2][B2];
#pragma unroll
            for (int r = 0; r < R2; ++r) {
                const int i = 32 * r + lane;
                if (I2 % 32 == 0 || i < I2) {
                    const int c = 4 * warp + (i & 3), q2 = i >> 2;
                    const C *pa = z + pos(c), *pb = z + pos(c == 0 ? K::H : N - c);
                    T4 tv[B2];  // in flight during the transforms (256 samples of 128^2: 1368 -> 1322 us)
#pragma unroll
                    for (int m = 0; m < B2; ++m) tv[m] = tab[c * K::H + q2 + A2 * m];
#pragma unroll
                    for (int m = 0; m < B2; ++m) {
                        a[r][m] = pa[skew(m, q2) * RS];
                        b[r][m] = pb[skew(m, q2) * RS];
                    }
                    hdft<B2, false>(a[r]);
                    hdft<B2, false>(b[r]);
                    if (c != 0) {
#pragma unroll
                        for (int m = 0; m < B2; ++m) product(a[r][m], b[r][m], tv[m]);
                    }
                }
            }
            if (warp == 0) {
                // slot 0: columns 0 (a) and N/2 (b, conjugated and reversed), each its own partner:
                // their values at -q through the columns' storage
                C *pa = z + pos(0), *pb = z + pos(K::H);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    const int i = 32 * r + lane;
                    if ((i & 3) == 0 && (I2 % 32 == 0 || i < I2)) {
#pragma unroll
                        for (int m = 0; m < B2; ++m) {
                            pa[((i >> 2) + A2 * m) * RS] = a[r][m];
                            pb[((i >> 2) + A2 * m) * RS] = b[r][m];
                        }
                    }
                }
                __syncwarp();
#pragma unroll
                for (int r = 0; r < R2; ++r) {
                    const int i = 32 * r + lane;
                    if ((i & 3) == 0 && (I2 % 32 == 0 || i < I2)) {
#pragma unroll
                        for (int m = 0; m < B2; ++m) {
                            const int q = (i >> 2) + A2 * m, nq = q == 0 ? 0 : K::H - q;
                            C am = pa[nq * RS], bm = pb[nq * RS];
                            am.y = -am.y;
                            bm.y = -bm.y;
                            product(a[r][m], am, tab[q]);
                            product(bm, b[r][m], tab[K::H * K::H + q]);
                        }
                    }
                }
                __syncwarp();
            }
#pragma unroll
            for (int r = 0; r < R2; ++r) {
                const int i = 32 * r + lane;
                if (I2 % 32 == 0 || i < I2) {
                    const int c = 4 * warp + (i & 3), q2 = i >> 2;
                    C *pa = z + pos(c), *pb = z + pos(c == 0 ? K::H : N - c);
                    hdft<B2, true>(a[r]);
                    hdft<B2, true>(b[r]);
#pragma unroll
                    for (int m = 0; m < B2; ++m) {
                        pa[skew(m, q2) * RS] = a[r][m];
                        pb[skew(m, q2) * RS] = b[r][m];
                    }
                }
            }
            __syncwarp();
        }
        {
            C v[R1][A2];
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const int i = 32 * r + lane, c = 4 * warp + (i & 3), m1 = (i >> 2) % B2, ab = (i >> 2) / B2;
                const C *p = z + pos(ab ? (c == 0 ? K::H : N - c) : c);
#pragma unroll
                for (int q2 = 0; q2 < A2; ++q2)
                    v[r][q2] = q2 == 0 ? p[skew(m1, 0) * RS]
                                       : hmul<true>(p[skew(m1, q2) * RS], twc[m1 * K::TC + q2]);
                hdft<A2, true>(v[r]);
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                const int i = 32 * r + lane, c = 4 * warp + (i & 3), m1 = (i >> 2) % B2, ab = (i >> 2) / B2;
                C *p = z + pos(ab ? (c == 0 ? K::H : N - c) : c) + m1 * RS;
#pragma unroll
                for (int j = 0; j < A2; ++j) {
                    if (ab) v[r][j].y = -v[r][j].y;
                    p[j * B2 * RS] = v[r][j];
                }
            }
        }
    }
};

// Host tables of a model on its n x n lattice: the product factors at [c][q], c = 0 .. n/2, q < n/2, and
// the twiddles as the kernels hold them in shared memory.  kh(kx, ky): K^ / n^2 in FP64.
//
// The fields vary slowly, so what a step sees of the table is K^ at the low frequencies q, where it is the
// sum of the two rounded factors Kp and conj(W) T; an error there acts the same way in every step.
// T is therefore taken from the rounded Kp, and a fourth factor holds what is left: 100 steps of the
// paper's nine models in FP32, mean field error against FP64 6.93e-8 rms without it, 6.83e-8 with it
// (one rounded K^ a frequency, the form before: 6.99e-8).
template <typename T, typename Kh>
void hf_product_table(int n, Kh kh, T *tab) {
    const int H = n / 2;
    for (int c = 0; c <= H; ++c)
        for (int q = 0; q < H; ++q) {
            const double k1 = kh(c, q), k2 = kh(c, q + H), th = 2.0 * M_PI * q / n;
            T *t = tab + 4 * ((size_t)c * H + q);
            t[0] = (T)(0.5 * (k1 + k2));
            const double d = k1 - (double)t[0];
            t[1] = (T)(d * std::cos(th));
            t[2] = (T)(-d * std::sin(th));
            t[3] = (T)(k1 - ((double)t[0] + (double)t[1] * std::cos(th) - (double)t[2] * std::sin(th)));
        }
}
template <int N, typename T>
void hf_twiddles_n(T *tw) {  // HfCfg<N>::TW complex values
    using K = HfCfg<N>;
    for (int i = 0; i < 2 * K::TW; ++i) tw[i] = T(0);
    for (int n1 = 0; n1 < K::B; ++n1)
        for (int k2 = 0; k2 < K::A; ++k2) {
            const double th = 2.0 * M_PI * (double)(n1 * k2) / N;
            tw[2 * (n1 * K::TR + k2)] = (T)std::cos(th);
            tw[2 * (n1 * K::TR + k2) + 1] = (T)-std::sin(th);
        }
    for (int m1 = 0; m1 < K::B2; ++m1)
        for (int q2 = 0; q2 < K::A2; ++q2) {
            const double th = 2.0 * M_PI * (double)(m1 * q2) / K::H;
            const int i = K::B * K::TR + m1 * K::TC + q2;
            tw[2 * i] = (T)std::cos(th);
            tw[2 * i + 1] = (T)-std::sin(th);
        }
}
inline int hf_tw_size(int n) { return n == 128 ? HfCfg<128>::TW : (n == 88 ? HfCfg<88>::TW : HfCfg<64>::TW); }
template <typename T>
void hf_twiddles(int n, T *tw) {
    if (n == 128)
        hf_twiddles_n<128>(tw);
    else if (n == 88)
        hf_twiddles_n<88>(tw);
    else
        hf_twiddles_n<64>(tw);
}

}  // namespace mfmc
