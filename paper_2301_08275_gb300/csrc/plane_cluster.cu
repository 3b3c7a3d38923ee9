// plane_cluster.cu - steps of small 2D grids (64 or 128 points per axis) with
// the whole plane on chip, spread over a thread-block cluster.
//
// A step of such a grid is bound by latency: as two sweeps it is two launches
// whose CTAs each fetch a tile, run a few hundred instructions and drain (11.7
// us per step of a 64^2 complex64 grid, 13 us per sweep with its reductions at
// 128^2 complex128).  Here one cluster of 8 or 16 CTAs keeps the plane in
// shared memory and registers for all steps of a launch.  CTA c owns n1/CS rows
// and n0/CS columns; a row sweep ends by writing every point into the shared
// memory of the CTA that owns its column, a column sweep into that of the CTA
// that owns its row, and one hardware cluster barrier follows each (what a
// buffer held has been read before the barrier that precedes its next writes).
//
// Sizes: 64 and 128 points per axis, the small grids of the batched and ground-state
// workloads.  32-point axes would leave a CTA of 8 with half a warp, and complex64
// columns of 256 points take the sweeps' 32-point plan, whose threads would not be
// those of the rows; 256 x 64 and 256 x 128 have not been tried.
//
// The lines run the same transforms, tables and pointwise code as the streaming
// sweeps (pass_kernels.cuh), so their results are the same bits.
// Measured, us per step on chip / as sweeps, one instance: 64^2 complex64 real
// 4.7 / 11.7, imaginary 5.3 / 22.7; 128^2 complex64 6.1 / 13.5 and 6.5 / 24.8;
// 64^2 complex128 9.0 / 17.4 and 14 / 31; 128^2 complex128 14 / 19 and 20 / 33.
// 8 instances of 128^2 complex128: 20.5 / 22 and 29 / 39 (PLANE_MAX_POINTS).
//
// In imaginary time the norm is summed over the cluster in the order of the
// streaming reduction (rows as group_sum and group_sum_df add them, then
// k_reduce_lines' warps of 32 rows), so these steps give the same bits too; the
// renormalisation, the last row sweep of a step and the first of the next stay
// in registers.
#include "pass_kernels.cuh"

namespace gpe {

namespace {

__device__ __forceinline__ unsigned pl_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ void pl_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ unsigned pl_map(unsigned a, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void pl_store(unsigned a, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void pl_store(unsigned a, double2 v)
{
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};\n" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void pl_store(unsigned a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(a), "d"(v) : "memory");
}

// Points per thread as in the streaming sweeps' pass plans (8 in complex64, 4
// in complex128); CTAs per cluster: 8 (the portable size), or 16 where that
// leaves more than two warps per scheduler (64 x 128: 6.5 us per step on 8 CTAs
// in complex64; complex128, whose sweeps run about three times the
// instructions, 13.4 us on 8).
template <typename R, int N0, int N1> struct PlaneCfg {
    static constexpr int CS = N0 * N1 * (sizeof(R) == 8 ? 2 : 1) > 8192 ? 16 : 8;
    static constexpr int E = sizeof(R) == 4 ? 8 : 4;
    static constexpr int L0 = N1 / CS, L1 = N0 / CS;         // rows and columns of a CTA
    using S = typename std::conditional<sizeof(R) == 4, float, fx>::type;
    using Rows = GTile<S, N0, L0, 1, false, E>;
    using Cols = GTile<S, N1, L1, 1, false, E>;
    using C = typename CT<R>::C;
    using U = typename Rows::U;
    static constexpr int NT = Rows::NT;
    static_assert(NT == Cols::NT, "one thread layout for both sweeps");
    static constexpr int POINTS = N0 * N1 / CS;
    static_assert(NT >= N1 && N1 <= 128, "the rows' norms are added by one thread each, four warps at most");
    static constexpr size_t smem = 2 * sizeof(C) * POINTS + 16 * (size_t)(N0 + N1) + 2 * sizeof(double) * N1 +
                                   sizeof(double) * NT + 2 * sizeof(unsigned) * (L0 > L1 ? L0 : L1);
};

template <typename R, int N0, int N1, bool IMAG>
__global__ void __launch_bounds__(PlaneCfg<R, N0, N1>::NT) k_plane(const PlaneArgs pa)
{
    using Cfg = PlaneCfg<R, N0, N1>;
    using Rows = typename Cfg::Rows;
    using Cols = typename Cfg::Cols;
    using C = typename Cfg::C;
    using U = typename Cfg::U;
    constexpr int E = Cfg::E, L0 = Cfg::L0, L1 = Cfg::L1, NT = Cfg::NT, CS = Cfg::CS;
    constexpr int T0 = Rows::TPL, T1 = Cols::TPL;
    extern __shared__ __align__(128) unsigned char smraw[];
    C *const bufa = reinterpret_cast<C *>(smraw);            // rows: point x of row l at x L0 + l
    C *const bufb = bufa + Cfg::POINTS;                      // columns: point y of column l at y L1 + l
    U *const tw0 = reinterpret_cast<U *>(bufb + Cfg::POINTS);
    U *const tw1 = tw0 + N0;
    double *const nrm = reinterpret_cast<double *>(tw1 + N1);    // [2][N1] norms of the rows
    double *const red = nrm + 2 * N1;                        // [NT] of the sums
    unsigned *const lsc = reinterpret_cast<unsigned *>(red + NT);
    const int t = threadIdx.x, lr = t % L0, tr = t / L0, lc = t % L1, tc = t / L1;
    if (pa.rows.stop && *reinterpret_cast<const volatile int *>(pa.rows.stop)) return;   // uniform over the grid
    Rows::load_twiddles(tw0, static_cast<const U *>(pa.rows.tw), t, NT);
    Cols::load_twiddles(tw1, static_cast<const U *>(pa.cols.tw), t, NT);
    const int c = (int)pl_rank();
    const int64_t inst = blockIdx.x / CS;
    C *const psi = pa.rows.inst_ptr ? static_cast<C *>(pa.rows.inst_ptr[inst])
                                    : static_cast<C *>(pa.rows.dst) + inst * (int64_t)(N0 * N1);
    LineGeom gr, gc;
    gr.inst = gc.inst = (int)inst;
    gr.ti = gc.ti = pa.rows.slot_of ? pa.rows.slot_of[inst] : (int)inst;
    gr.valid = gc.valid = true;
    gr.lg = gc.lg = gr.li = gc.li = 0;
    gr.c1 = gc.c1 = 0;
    gr.c0 = c * L0 + lr;             // this thread's row and column
    gr.off = (int64_t)gr.c0 * N0;
    gc.c0 = c * L1 + lc;
    gc.off = gc.c0;
    const unsigned a_addr = smem_addr(bufa), b_addr = smem_addr(bufb);

    C v[E];
    // point x of this thread's row to the owner of column x, and back
    auto to_columns = [&]() {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int x = tr + T0 * e;
            pl_store(pl_map(b_addr, (unsigned)(x / L1)) + (unsigned)((gr.c0 * L1 + x % L1) * (int)sizeof(C)), v[e]);
        }
    };
    auto to_rows = [&]() {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int y = tc + T1 * e;
            pl_store(pl_map(a_addr, (unsigned)(y / L0)) + (unsigned)((gc.c0 * L0 + y % L0) * (int)sizeof(C)), v[e]);
        }
    };
    // line scales of complex128 sweeps start from zero
    auto clear = [&]() {
        if (sizeof(R) == 8)
            for (int i = t; i < 2 * (L0 > L1 ? L0 : L1); i += NT) lsc[i] = 0;
    };
    // (scale: of complex128 values before OP_NIMAG, as OP_SCALE_NIMAG has it)
    auto row_sweep = [&](const PassArgs &a, int op_pre, int fft1, int op_mid, int fft2, double scale = 1.0) {
        if constexpr (sizeof(R) == 8) {
            fx_sweep<Rows, false>(v, a, gr, scale, bufa, bufa, tr, lr, tw0, lsc, op_pre, fft1, op_mid, fft2);
        } else {
            C w[1][E];
#pragma unroll
            for (int e = 0; e < E; ++e) w[0][e] = v[e];
            point_op<R, E, T0>(op_pre, w[0], a, gr.inst, gr.ti, gr.c0, 0, tr, gr.off);
            sweep_transforms<Rows, false>(w, bufa, bufa, tr, lr, tw0, fft1, fft2, [&]() {
                point_op<R, E, T0>(op_mid, w[0], a, gr.inst, gr.ti, gr.c0, 0, tr, gr.off);
            });
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = w[0][e];
        }
    };
    auto column_sweep = [&](const PassArgs &a, int op_mid) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = bufb[(tc + T1 * e) * L1 + lc];
        if constexpr (sizeof(R) == 8) {
            fx_sweep<Cols, false>(v, a, gc, 1.0, bufb, bufb, tc, lc, tw1, lsc, OP_NONE, -1, op_mid, 1);
        } else {
            C w[1][E];
#pragma unroll
            for (int e = 0; e < E; ++e) w[0][e] = v[e];
            sweep_transforms<Cols, false>(w, bufb, bufb, tc, lc, tw1, -1, 1, [&]() {
                point_op<R, E, T1>(op_mid, w[0], a, gc.inst, gc.ti, gc.c0, 0, tc, gc.off);
            });
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = w[0][e];
        }
        to_rows();
        __syncthreads();             // lsc has been read
        clear();
        pl_sync();
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = bufa[(tr + T0 * e) * L0 + lr];
    };
    auto exchange_to_columns = [&]() {
        to_columns();
        __syncthreads();
        clear();
        pl_sync();
    };

#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = psi[gr.off + tr + T0 * e];
    clear();
    pl_sync();                       // twiddles and cleared words; every CTA of the cluster runs

    if constexpr (!IMAG) {
        PassArgs r = pa.rows, k = pa.cols;
        if (pa.first) {
            r.vt_ax = pa.vh[0];
            r.vt_o0 = pa.vh[1];
            r.nl_c = 0.5 * pa.dt;
            r.vq_full = 0;
            r.dphi = 0.0f;
            r.nl_cf = pa.half_dtf;
            row_sweep(r, OP_NREAL, -1, OP_NONE, 0);
            __syncthreads();
            clear();
        }
#pragma unroll 1
        for (int s = 0; s < pa.nsteps; ++s) {
            exchange_to_columns();
            if (sizeof(R) == 4) {
                k.dither = pa.dither;
                if (pa.dither)
                    for (int q = 0; q < 4; ++q) k.dk[q] = pa.dk[s][q];
            }
            column_sweep(k, OP_KREAL);
            const bool last = pa.last && s == pa.nsteps - 1;
            r.vt_ax = last ? pa.vh[0] : pa.vf[0];
            r.vt_o0 = last ? pa.vh[1] : pa.vf[1];
            r.nl_c = last ? 0.5 * pa.dt : pa.dt;
            r.vq_full = last ? 0 : 1;
            r.dphi = sizeof(R) == 4 && pa.dither ? pa.dphi[s] : 0.0f;
            r.nl_cf = last ? pa.half_dtf : pa.dtf;
            row_sweep(r, OP_NONE, 1, OP_NREAL, last ? 0 : -1);
        }
    } else {
        PassArgs r = pa.rows;
        r.nl_c = 0.5 * pa.dt;
        r.vq_full = 0;
        r.nl_cf = pa.half_dtf;
        double sc = 1.0;             // renormalisation factor that v still lacks
        auto rescale = [&]() {
#pragma unroll
            for (int e = 0; e < E; ++e) v[e] = cscale(v[e], (R)sc);
        };
#pragma unroll 1
        for (int s = 0; s < pa.nsteps; ++s) {
            if constexpr (sizeof(R) == 4) rescale();
            row_sweep(r, OP_NIMAG, -1, OP_NONE, 0, sc);
            exchange_to_columns();
            column_sweep(pa.cols, OP_KIMAG);
            row_sweep(r, OP_NONE, 1, OP_NIMAG, 0);
            // every row's norm, to every CTA.  In complex64 the threads of a row's
            // first warp have its sum, in complex128 all of them.
            constexpr int SND = sizeof(R) == 8 ? CS : 32 / L0 < T0 ? 32 / L0 : T0;
            static_assert(SND <= T0 && CS % SND == 0, "senders of a row");
            double sn[1] = {0.0};
            if constexpr (sizeof(R) == 4) {
                float nh[1] = {0.0f}, nl[1] = {0.0f};
#pragma unroll
                for (int e = 0; e < E; ++e) df_acc(nh[0], nl[0], norm2(v[e]));
                group_sum_df<L0, T0, 1>(nh, nl, reinterpret_cast<float2 *>(red), lr, tr);
                sn[0] = (double)nh[0] + (double)nl[0];
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) sn[0] += norm2(v[e]);
                group_sum<L0, T0, 1>(sn, red, lr, tr);
                clear();
            }
            double *const slot = nrm + N1 * (s & 1);
            if (tr < SND) {
                const unsigned at = smem_addr(slot + gr.c0);
#pragma unroll
                for (int k = 0; k < CS; k += SND) pl_store(pl_map(at, (unsigned)(tr + k)), sn[0]);
            }
            pl_sync();
            // FP64 additions keep a sub-partition for 64 cycles each: a warp per 32
            // rows, then one warp for their sums and the factor
            if (t < N1) {
                double x = slot[t];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if ((t & 31) == 0) red[t >> 5] = x;
            }
            __syncthreads();
            if (t == 0) {
                const double tot = (N1 == 128 ? (red[0] + red[1]) + (red[2] + red[3]) : red[0] + red[1]) * pa.dv;
                double f = 1.0;
                if (!(tot > 0.0) || !isfinite(tot)) {
                    if (c == 0) atomicOr(pa.rows.err, (int)ERR_NUMERIC);
                } else {
                    f = sqrt(pa.target / tot);
                }
                red[N1 / 32] = f;
            }
            __syncthreads();
            sc = red[N1 / 32];
        }
        rescale();
    }
#pragma unroll
    for (int e = 0; e < E; ++e) psi[gr.off + tr + T0 * e] = v[e];
    pl_sync();                       // no CTA leaves while another may still write to it
}

struct PlaneState {
    std::mutex mu;
    int ok[64] = {};     // per device: 0 unknown, 1 usable, -1 no such cluster fits
};

template <typename R, int N0, int N1, bool IMAG> cudaError_t launch_plane_k(const PlaneArgs &a, cudaStream_t st)
{
    using Cfg = PlaneCfg<R, N0, N1>;
    static_assert(Cfg::Rows::layout_consistent() && Cfg::Cols::layout_consistent(), "shared layout of the exchanges");
    static PlaneState ps;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorNotSupported;
    auto *kern = k_plane<R, N0, N1, IMAG>;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(Cfg::NT);
    cfg.dynamicSmemBytes = Cfg::smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = Cfg::CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    {
        std::lock_guard<std::mutex> lk(ps.mu);
        if (ps.ok[dev] == 0) {
            if (Cfg::CS > 8) cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem);
            int ncl = 0;
            cfg.gridDim = dim3(Cfg::CS);
            const cudaError_t oe = cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg);
            if (oe != cudaSuccess) cudaGetLastError();
            ps.ok[dev] = oe == cudaSuccess && ncl >= 1 ? 1 : -1;
        }
        if (ps.ok[dev] < 0) return cudaErrorNotSupported;
    }
    if (a.count <= 0) return cudaSuccess;
    cfg.gridDim = dim3((unsigned)(a.count * Cfg::CS));
    return cudaLaunchKernelEx(&cfg, kern, a);
}
template <typename R, int N0, int N1> cudaError_t launch_plane_n(const PlaneArgs &a, cudaStream_t st)
{
    return a.imag ? launch_plane_k<R, N0, N1, true>(a, st) : launch_plane_k<R, N0, N1, false>(a, st);
}

}  // namespace

#ifndef GPE_PLANE_R
#define GPE_PLANE_R float
#define GPE_PLANE_LAUNCH launch_plane_f32
#endif

cudaError_t GPE_PLANE_LAUNCH(int n0, int n1, const PlaneArgs &a, cudaStream_t st)
{
    using R = GPE_PLANE_R;
    if (n0 == 64 && n1 == 64) return launch_plane_n<R, 64, 64>(a, st);
    if (n0 == 64 && n1 == 128) return launch_plane_n<R, 64, 128>(a, st);
    if (n0 == 128 && n1 == 64) return launch_plane_n<R, 128, 64>(a, st);
    if (n0 == 128 && n1 == 128) return launch_plane_n<R, 128, 128>(a, st);
    return cudaErrorInvalidValue;
}

}  // namespace gpe
