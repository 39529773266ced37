// The resident solve with the field in shared memory, a sample per CTA (n = 128) or per cluster of
// four CTAs (n = 256, 64 rows each): no field traffic and no launch between steps.
//
// A warp owns 8 rows of a 128-column strip (16 warps a CTA), a lane four columns.  Each of its rows
// is summed once per step: the window from shared memory, the centre sums, one segment sum per
// half-width class, added to the 2R + 1 output rows it belongs to.  Sums for rows of the strips above
// and below (R each) go to those strips' buffers, in the neighbour CTA's shared memory at the edge
// of a CTA's rows, and each strip then adds (own + from above) + from below, updates and stores its
// rows.  So no row is summed twice, where the row-streaming kernel walks 2R halo rows per range
// (half its walk and more for a batch of 64 samples) and streams the fields through HBM.
//
// A step has one cluster barrier, between the partial sums' writes and reads, and one of the CTA,
// between their reads and the next step's writes; the buffers that another CTA writes alternate, so
// that a write can only meet the reads of two steps before, which the cluster barrier of the step
// between has ordered.  The two column strips of a row (n = 256) meet at a 64-thread barrier once
// their row block is updated.
//
// What bounds it: shared memory, 44 wavefronts a row of 128 columns (window 20, partial sums 16,
// field 8): 5.6 K cycles a step of 64 x 256 points on an SM, the FMA pipe 4.0 K.  256^2, R = 8, 500
// steps: 512 samples 26.1 ms (row streaming 29.0), 64 samples 7.4 us a step (row streaming 26.3, the
// tile kernel 14.9); 36 clusters of four fit the 152 SMs at a time.
#include <cuda_runtime.h>

#include <algorithm>

#include "resident_cluster.cuh"
#include "tma_step.cuh"

namespace mfmc {

namespace {

constexpr int RC_ROWS = 8, RC_WARPS = 16, RC_NT = 32 * RC_WARPS;

template <int N, int R>
struct RcCfg {
    static constexpr int XS = N / 128;                  // column strips (warps per row block)
    static constexpr int STRIPS = RC_WARPS / XS;        // row blocks per CTA
    static constexpr int ROWS = STRIPS * RC_ROWS;       // rows per CTA
    static constexpr int CL = N / ROWS;                 // CTAs per sample
    static constexpr int FIELD = ROWS * N;              // floats
    static constexpr int IN = RC_WARPS * 2 * R * 128;   // floats: per warp R rows from above, R from below
    // the buffers that another CTA writes (top strip's "above", bottom strip's "below") alternate
    // between IN and this second copy from step to step
    static constexpr int FAR = CL > 1 ? 2 * XS * R * 128 : 0;  // floats: [above, below][column strip][R]
    static constexpr size_t SMEM = (size_t)(FIELD + IN + FAR) * sizeof(float);
};

__device__ __forceinline__ uint32_t rc_map(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void rc_st_remote(uint32_t addr, float2 a, float2 b) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y)
                 : "memory");
}

// Barrier of the sample's CTAs.
template <int CL>
__device__ __forceinline__ void rc_sync() {
    if constexpr (CL > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else {
        __syncthreads();
    }
}

template <int N, int R>
__global__ void __launch_bounds__(RC_NT, 1) resident_cluster_kernel(ResidentArgs a) {
    using K = RcCfg<N, R>;
    constexpr DiscClasses<R> cls{};
    constexpr int M = RowWin<R>::M, R4 = RowWin<R>::R4, NQ = RowWin<R>::WIN / 4, CL = K::CL;
    extern __shared__ __align__(16) float rc_smem[];
    __shared__ double red[RC_WARPS];
    __shared__ double cta_sum[CL];
    float *const u = rc_smem;                                              // [ROWS][N]
    float4 *const in = reinterpret_cast<float4 *>(rc_smem + K::FIELD);      // [warp][above, below][R][32]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int strip = warp / K::XS, xs = warp % K::XS, x = 128 * xs + 4 * lane;
    const int rank = CL > 1 ? (int)(blockIdx.x % CL) : 0, cluster = (int)blockIdx.x / CL, clusters = (int)gridDim.x / CL;
    // the lane's window: float4 q of it starts at column x - R4 + 4q, taken modulo N
    int wc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int c = x - R4 + 4 * q;
        wc[q] = c < 0 ? c + N : (c >= N ? c - N : c);
    }
    float *const mine = u + strip * RC_ROWS * N;  // the warp's rows
    // where the warp's sums for the strips above and below go: their "below" and "above" buffers
    const bool up_out = strip == 0, dn_out = strip == K::STRIPS - 1;
    const int up_warp = (up_out ? K::STRIPS - 1 : strip - 1) * K::XS + xs, dn_warp = (dn_out ? 0 : strip + 1) * K::XS + xs;
    float4 *const up_dst = in + ((up_warp * 2 + 1) * R) * 32 + lane, *const dn_dst = in + ((dn_warp * 2 + 0) * R) * 32 + lane;
    float4 *const far = reinterpret_cast<float4 *>(rc_smem + K::FIELD + K::IN) + xs * R * 32 + lane;  // [above, below]
    const uint32_t up_rank = CL > 1 ? (rank + CL - 1) % CL : 0, dn_rank = CL > 1 ? (rank + 1) % CL : 0;
    const uint32_t up_addr[2] = {rc_map(smem_u32(up_dst), up_rank), rc_map(smem_u32(far + K::XS * R * 32), up_rank)};
    const uint32_t dn_addr[2] = {rc_map(smem_u32(dn_dst), dn_rank), rc_map(smem_u32(far), dn_rank)};
    const bool up_far = CL > 1 && up_out, dn_far = CL > 1 && dn_out;
    const bool dn_far_in = up_far, up_far_in = dn_far;  // the top strip's "above" and the bottom's "below" come from afar
    const float4 *const from_up = in + ((warp * 2 + 0) * R) * 32 + lane, *const from_dn = in + ((warp * 2 + 1) * R) * 32 + lane;
    const size_t nn = (size_t)N * N, off = (size_t)(rank * K::ROWS + strip * RC_ROWS) * N + x;

    auto pair_sync = [&]() {  // the warps of one row block
        if constexpr (K::XS > 1)
            asm volatile("bar.sync %0, %1;" ::"r"(1 + strip), "n"(32 * K::XS) : "memory");
        else
            __syncwarp();
    };

    for (int sample = cluster; sample < a.ns; sample += clusters) {
        const float *__restrict__ src = a.u0 + (size_t)sample * nn + off;
#pragma unroll
        for (int y = 0; y < RC_ROWS; ++y)
            *reinterpret_cast<float4 *>(mine + y * N + x) = __ldg(reinterpret_cast<const float4 *>(src + (size_t)y * N));
        const StepCoef cf = a.coef[sample];
        const float2 nc0 = make_float2(-cf.c0, -cf.c0), c1 = make_float2(cf.c1, cf.c1), c2 = make_float2(cf.c2, cf.c2);
        const int nsteps = a.steps_ps ? a.steps_ps[sample] : a.nsteps;
        rc_sync<CL>();  // every CTA of the cluster runs and has left the sample before
        pair_sync();
#pragma unroll 1
        for (int step = 0; step < nsteps; ++step) {
            const int alt = step & 1;
            float2 own[RC_ROWS][2], up[R][2], dn[R][2];
#pragma unroll
            for (int r = 0; r < RC_ROWS; ++r) {
                RowWin<R> w;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float4 t = *reinterpret_cast<const float4 *>(mine + r * N + wc[q]);
                    w.v[4 * q + 0] = t.x;
                    w.v[4 * q + 1] = t.y;
                    w.v[4 * q + 2] = t.z;
                    w.v[4 * q + 3] = t.w;
                }
                row_prefix<R>(w);
#pragma unroll
                for (int c = 0; c < cls.count; ++c) {
                    const int hw = cls.width[c];
                    float h[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int b = i + R - hw, e = i + R + hw + 1;
                        h[i] = hw == 0 ? w.v[R4 + i]
                                       : (b >= M ? w.p[e] - w.p[b] : (e <= M ? w.p[b] - w.p[e] : w.p[e] + w.p[b]));
                    }
                    const float2 h01 = make_float2(h[0], h[1]), h23 = make_float2(h[2], h[3]);
                    auto add = [&](float2 (&s)[2], bool first) {
                        s[0] = first ? h01 : __fadd2_rn(s[0], h01);
                        s[1] = first ? h23 : __fadd2_rn(s[1], h23);
                    };
#pragma unroll
                    for (int y = -R; y < RC_ROWS + R; ++y) {
                        const int ady = r > y ? r - y : y - r;
                        if (ady <= R && cls.of[ady <= R ? ady : 0] == c) {
                            const bool first = r == (y > R ? y - R : 0);  // the output row's first row of this block
                            if (y < 0)
                                add(up[y < 0 ? y + R : 0], first);
                            else if (y < RC_ROWS)
                                add(own[y >= 0 && y < RC_ROWS ? y : 0], first);
                            else
                                add(dn[y >= RC_ROWS ? y - RC_ROWS : 0], first);
                        }
                    }
                }
                if (r == 0) __syncthreads();  // every strip of the CTA has read the last step's sums
                // output row r - R of the strip above has all of this strip's rows
                if (r < R) {
                    if (up_far)
                        rc_st_remote((alt ? up_addr[1] : up_addr[0]) + 512 * r, up[r < R ? r : 0][0], up[r < R ? r : 0][1]);
                    else
                        up_dst[32 * r] = make_float4(up[r < R ? r : 0][0].x, up[r < R ? r : 0][0].y,
                                                     up[r < R ? r : 0][1].x, up[r < R ? r : 0][1].y);
                }
            }
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (dn_far)
                    rc_st_remote((alt ? dn_addr[1] : dn_addr[0]) + 512 * k, dn[k][0], dn[k][1]);
                else
                    dn_dst[32 * k] = make_float4(dn[k][0].x, dn[k][0].y, dn[k][1].x, dn[k][1].y);
            }
            rc_sync<CL>();
            // (own + from above) + from below
            const float4 *const fu = dn_far_in && alt ? far : from_up, *const fd = up_far_in && alt ? far + K::XS * R * 32 : from_dn;
#pragma unroll
            for (int y = 0; y < RC_ROWS; ++y) {
                if (y < R) {
                    const float4 t = fu[32 * y];
                    own[y][0] = __fadd2_rn(own[y][0], make_float2(t.x, t.y));
                    own[y][1] = __fadd2_rn(own[y][1], make_float2(t.z, t.w));
                }
                if (y >= RC_ROWS - R) {
                    const float4 t = fd[32 * (y - (RC_ROWS - R))];
                    own[y][0] = __fadd2_rn(own[y][0], make_float2(t.x, t.y));
                    own[y][1] = __fadd2_rn(own[y][1], make_float2(t.z, t.w));
                }
            }
#pragma unroll
            for (int y = 0; y < RC_ROWS; ++y) {
                float4 *p = reinterpret_cast<float4 *>(mine + y * N + x);
                const float4 t = *p;
                const float2 x0 = make_float2(t.x, t.y), x1 = make_float2(t.z, t.w);
                const float2 v0 = __fadd2_rn(x0, __ffma2_rn(c1, __ffma2_rn(nc0, x0, own[y][0]), __fmul2_rn(c2, x0)));
                const float2 v1 = __fadd2_rn(x1, __ffma2_rn(c1, __ffma2_rn(nc0, x1, own[y][1]), __fmul2_rn(c2, x1)));
                *p = make_float4(fminf(1.f, fmaxf(-1.f, v0.x)), fminf(1.f, fmaxf(-1.f, v0.y)),
                                 fminf(1.f, fmaxf(-1.f, v1.x)), fminf(1.f, fmaxf(-1.f, v1.y)));
            }
            pair_sync();
        }
        // OoI: FP64, rows then lanes then warps then CTAs in order
        double part = 0.0;
#pragma unroll
        for (int y = 0; y < RC_ROWS; ++y) {
            const float4 t = *reinterpret_cast<const float4 *>(mine + y * N + x);
            part += ((double)t.x + (double)t.y) + ((double)t.z + (double)t.w);
            if (a.uT) *reinterpret_cast<float4 *>(a.uT + (size_t)sample * nn + off + (size_t)y * N) = t;
        }
        for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
        if (lane == 0) red[warp] = part;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int i = 0; i < RC_WARPS; ++i) t += red[i];
            if constexpr (CL > 1)
                asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(rc_map(smem_u32(&cta_sum[rank]), 0)), "d"(t)
                             : "memory");
            else
                cta_sum[0] = t;
        }
        rc_sync<CL>();
        if (rank == 0 && threadIdx.x == 0) {
            double t = 0.0;
            for (int i = 0; i < CL; ++i) t += cta_sum[i];
            const double mean = t / (double)nn;
            if (a.ubar) a.ubar[sample] = mean;
            if (a.ooi) a.ooi[sample] = 0.5 * (1.0 + mean);
        }
        __syncthreads();  // red and the sums are free (the next sample's barriers order the other CTAs)
    }
}

template <int N, int R>
mfmc_status rc_launch(const ResidentArgs &a, cudaStream_t st) {
    using K = RcCfg<N, R>;
    auto kern = resident_cluster_kernel<N, R>;
    MFMC_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)K::SMEM));
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(RC_NT);
    cfg.dynamicSmemBytes = K::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = K::CL;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(K::CL);
    int clusters = 0;
    MFMC_CUDA(cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg));
    cfg.gridDim = dim3((unsigned)(K::CL * std::max(1, std::min(a.ns, clusters))));
    MFMC_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
    MFMC_LAUNCHED("resident_cluster launch");
    return MFMC_OK;
}

}  // namespace

mfmc_status launch_resident_cluster(int R, const ResidentArgs &a, cudaStream_t st) {
    if (a.ns <= 0) return MFMC_OK;
    if (a.n == 128) return R == 5 ? rc_launch<128, 5>(a, st) : (R == 6 ? rc_launch<128, 6>(a, st) : rc_launch<128, 8>(a, st));
    return R == 4 ? rc_launch<256, 4>(a, st) : (R == 6 ? rc_launch<256, 6>(a, st) : rc_launch<256, 8>(a, st));
}

}  // namespace mfmc
