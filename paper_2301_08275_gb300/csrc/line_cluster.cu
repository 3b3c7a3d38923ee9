// line_cluster.cu - complex128 real-time steps of a few short lines (64, 128
// or 256 points), each line spread over a cluster of CTAs.
//
// A single line is bound by the chain of instructions that its busiest warp
// runs per step.  A line of N = 32 CS points is spread over a cluster of CS = 2,
// 4 or 8 CTAs of one warp, one point per lane: CTA c holds points CS i + c, i
// the lane.  The arithmetic is 64-bit fixed point with one scale for the line
// (fx.cuh): a complex addition takes two integer additions per lane, a complex
// product 12 integer multiply-adds, where FP64 takes 64 cycles per instruction.
//
// The transform is the four-step factorisation N = 32 x CS of the discrete
// Fourier transform (the split-step scheme's F and F^-1, Sec. 2 of the paper):
//   X[k1 + 32 k2] = sum_c W_CS^(c k2) W_N^(c k1) sum_i x[CS i + c] W_32^(i k1)
// Step A, the inner sums over i, is a 32-point transform within one warp
// (radix-2 stages across lanes, partners exchanged by shuffles, decimation in
// frequency: natural order in, bit-reversed out).  After the twiddle W_N^(c k1)
// the CTAs exchange their values (CTA j receives the rows k1 = j R .. j R +
// R - 1, R = 32 / CS, of every column): step B, the sums over c, is then
// again local, CS-point transforms over aligned lane groups.  The kinetic
// factor multiplies the spectrum in that layout; the inverse runs the same
// steps backwards (decimation in time: bit-reversed in, natural out) and ends
// in the layout it started from, where the nonlinear and potential factors
// of the next substep are pointwise.  Two exchanges per step, each an
// all-to-all of one 16-byte value per lane, written into the receiving CTA's
// shared memory by st.async and counted by that CTA's mbarrier.
//
// Scale: the growth of a step (N) is divided out by 4 at the forward four-step
// twiddle, N / 16 at the inverse one and 4 at the last stage of the inverse, so
// a step is unitary and the line keeps the scale it was loaded with; values
// stay below 2^3.5 |x|_2 throughout (16 |x|_2 is what the scale allows for).
//
// Measured: 1.55 us per step of a 256-point line (3.17 us with one real number
// per lane in FP64 over 16 CTAs), 1.5 us at 64 points; k_line1d_fx, one CTA per
// line, takes 2.8 and 2.3 us.  The two exchanges are 0.3 us each.
#include <mutex>

#include "pass_kernels.cuh"

namespace gpe {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ unsigned cl_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_map(unsigned a, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// write 16 bytes to a cluster address and count them on the barrier at bar
__device__ __forceinline__ void cl_send(unsigned dst, unsigned bar, fx2 v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];\n" ::"r"(dst),
                 "l"(v.x), "l"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ fx2 shfl_xor(fx2 v, int h)
{
    return mk(__shfl_xor_sync(FULL, v.x, h), __shfl_xor_sync(FULL, v.y, h));
}
// v w 2^-64 (w of 62 bits: divides by 4), half = 2^31 - 1 or 2^31: lanes whose
// factor is one meet ties, which alternate between the steps
__device__ __forceinline__ fx2 mul_quarter(fx2 v, int4 w, long long half)
{
    const Limbs x = limbs(v.x), y = limbs(v.y);
    long long mr = imad(x.h, w.y, half), mi = imad(x.h, w.w, half);
    mr = imad(x.l, w.x, mr);
    mi = imad(x.l, w.z, mi);
    mr = imad(-y.h, w.w, mr);
    mi = imad(y.h, w.y, mi);
    mr = imad(y.l, -w.z, mr);
    mi = imad(y.l, w.x, mi);
    long long hr = imul(x.h, w.x), hi = imul(x.h, w.z);
    hr = imad(-y.h, w.z, hr);
    hi = imad(y.h, w.x, hi);
    return mk(hr + (mr >> 32), hi + (mi >> 32));
}

// W_N^m (inverse: its conjugate) from the plan's table
template <int N> __device__ __forceinline__ int4 wtab(const int4 *tw, int m, bool inv)
{
    const fx2 w = fx_value(tw[m & (N - 1)]);
    return fx_pack(w.x, inv ? -w.y : w.y);
}
__device__ __forceinline__ int4 one62() { return make_int4(1 << 30, 0, 0, 0); }

__device__ __forceinline__ int brev(int x, int bits) { return (int)(__brev((unsigned)x) >> (32 - bits)); }

// Radix-2 stages across the lanes of aligned groups of G positions (index in
// the group i = lane & (G-1)).  Decimation in frequency: half-widths G/2 .. 1;
// the lower lane of a pair keeps the sum, the upper takes the difference times
// W_2H^(i mod H).  Decimation in time: the reverse.
template <int G> struct LaneDft {
    static constexpr int S = G == 32 ? 5 : (G == 8 ? 3 : (G == 4 ? 2 : 1));
    int4 w[S > 1 ? S - 1 : 1];          // stage twiddles of the upper lanes (stages with H > 1)
    long long neg[S];                   // all ones on the upper lanes of a stage

    template <int N> __device__ __forceinline__ void init(const int4 *tw, int lane, bool inv, bool dif)
    {
        const int i = lane & (G - 1);
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int H = dif ? (G >> (s + 1)) : (1 << s);
            const bool up = (i & H) != 0;
            neg[s] = up ? -1ll : 0ll;
            if (H > 1) w[dif ? s : s - 1] = up ? wtab<N>(tw, (i & (H - 1)) * (N / (2 * H)), inv) : one62();
        }
    }
    // own + other on the lower lane of a pair, other - own on the upper
    __device__ __forceinline__ static long long pair(long long v, long long o, long long n) { return ((v ^ n) - n) + o; }
    // natural order in, bit-reversed out
    __device__ __forceinline__ fx2 dif(fx2 v) const
    {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int H = G >> (s + 1);
            const fx2 o = shfl_xor(v, H);
            v = mk(pair(v.x, o.x, neg[s]), pair(v.y, o.y, neg[s]));
            if (H > 1) v = fx_mul<2>(v, w[s]);
        }
        return v;
    }
    // bit-reversed order in, natural out; QUARTER: the last stage's twiddle divides by 4
    template <bool QUARTER> __device__ __forceinline__ fx2 dit(fx2 v, long long half) const
    {
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int H = 1 << s;
            if (H > 1) v = QUARTER && s == S - 1 ? mul_quarter(v, w[s - 1], half) : fx_mul<2>(v, w[s - 1]);
            const fx2 o = shfl_xor(v, H);
            v = mk(pair(v.x, o.x, neg[s]), pair(v.y, o.y, neg[s]));
        }
        return v;
    }
};

template <int CS>
__global__ void __launch_bounds__(32) k_line1d_cluster(const Line1DArgs a)
{
    constexpr int N = 32 * CS, R = 32 / CS, LGCS = CS == 8 ? 3 : (CS == 4 ? 2 : 1);
    __shared__ __align__(16) fx2 xb[2][32];         // receive buffers of the two exchanges
    __shared__ __align__(8) uint64_t xbar[2];
    __shared__ unsigned lsc[2];
    const int lane = threadIdx.x;
    const int c = (int)cl_rank();
    const int64_t inst = blockIdx.x / CS;
    double2 *psi = a.inst_ptr ? static_cast<double2 *>(a.inst_ptr[inst]) : static_cast<double2 *>(a.psi) + inst * N;
    const int64_t ib = a.slot_of ? a.slot_of[inst] : inst;
    const int4 *tw = static_cast<const int4 *>(a.twx);

    if (lane == 0) {
        mbar_init(&xbar[0], 1);
        mbar_init(&xbar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (lane < 2) lsc[lane] = 0;
    __syncwarp();

    // the line's scale: every CTA reads the whole line (L2) and takes the same
    double2 whole[CS];
#pragma unroll
    for (int k = 0; k < CS; ++k) whole[k] = psi[lane + 32 * k];
    const LineScale ls = line_scale<1, 32, CS>(whole, lsc, lsc + 1, 0, 4);
    const int n = CS * lane + c;
    const double2 d = psi[n];
    fx2 v = mk(fx_from(d.x, ls.q), fx_from(d.y, ls.q));

    // per-lane constants: stage twiddles, four-step twiddles, kinetic factor
    LaneDft<32> fa, ia;     // step A forward (DIF) and inverse (DIT)
    LaneDft<CS> fb, ibt;    // step B forward and inverse
    fa.template init<N>(tw, lane, false, true);
    ia.template init<N>(tw, lane, true, false);
    fb.template init<N>(tw, lane, false, true);
    ibt.template init<N>(tw, lane, true, false);
    const int k1a = brev(lane, 5);                     // step A output: k1 at this lane
    const int4 t4f = wtab<N>(tw, c * k1a, false);
    const int rB = lane / CS, qB = lane & (CS - 1);    // step B layout: lane r CS + q
    const int k1b = c * R + rB;
    const fx2 ti = fx_value(wtab<N>(tw, qB * k1b, true));
    const int4 t4i = fx_pack(ti.x >> (LGCS - 1), ti.y >> (LGCS - 1));
    const int4 kin = static_cast<const int4 *>(a.ktx)[k1b + 32 * brev(qB, LGCS)];
    // destinations of this lane's value in the two exchanges
    const unsigned rankA = (unsigned)(k1a / R), rankB = (unsigned)qB;
    const unsigned dstA = cl_map(smem_addr(&xb[0][(k1a % R) * CS + c]), rankA), barA = cl_map(smem_addr(&xbar[0]), rankA);
    const unsigned dstB = cl_map(smem_addr(&xb[1][brev(k1b, 5)]), rankB), barB = cl_map(smem_addr(&xbar[1]), rankB);
    // potential angles at this lane's point and the interaction
    const long long *vq = static_cast<const long long *>(a.vq);
    const long long *vl = a.vq_last ? static_cast<const long long *>(a.vq_last) : vq;
    const long long vh = vq ? vq[ib * N + n] : 0, vlast = vl ? vl[ib * N + n] : 0;
    const FxCoupling *gq = static_cast<const FxCoupling *>(a.gq) + 2 * ib;
    const FxNonlinear nh = fx_nonlinear(gq, ls.q), nf = fx_nonlinear(gq + 1, ls.q);
    const double g = a.g[ib], ct = a.dt * 0.15915494309189533577;

    cl_sync();   // every CTA's barriers are initialised before any value is sent to it

    v = fx_rotate(v, fx_nl_angle(v, nh, g, 0.5 * ct) + vh);
    bool timed_out = false;
    for (int64_t st = 0; st < a.nsteps; ++st) {
        const unsigned par = (unsigned)(st & 1);
        const long long half = (1ll << 31) - (long long)par;
        if (lane == 0) {
            // 32 lanes x 16 bytes arrive per exchange (tx_extra: failure-handling test hook)
            mbar_expect_tx(&xbar[0], 512u + (unsigned)a.tx_extra);
            mbar_expect_tx(&xbar[1], 512u + (unsigned)a.tx_extra);
        }
        // forward transform, step A, and the exchange to the row layout
        v = fa.dif(v);
        v = mul_quarter(v, t4f, half);
        cl_send(dstA, barA, v);
        if (__any_sync(FULL, !mbar_wait_bounded(&xbar[0], par))) {
            timed_out = true;
            break;
        }
        v = xb[0][lane];
        // step B, kinetic factor, inverse step B
        v = fb.dif(v);
        v = fx_mul<2>(v, kin);
        v = ibt.template dit<false>(v, half);
        v = mul_quarter(v, t4i, half);
        cl_send(dstB, barB, v);
        if (__any_sync(FULL, !mbar_wait_bounded(&xbar[1], par))) {
            timed_out = true;
            break;
        }
        v = xb[1][lane];
        v = ia.template dit<true>(v, half);
        const bool last = st == a.nsteps - 1;
        const long long ang = last ? fx_nl_angle(v, nh, g, 0.5 * ct) + vlast
                                   : fx_nl_angle(v, nf, g, ct) + (long long)((unsigned long long)vh << 1);
        v = fx_rotate(v, ang);
    }
    if (timed_out && lane == 0 && a.err) atomicOr(a.err, (int)ERR_CLUSTER_TIMEOUT);
    // no CTA leaves while a value addressed to it can still be in flight
    cl_sync();
    psi[n] = ls.bad ? mk(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll))
                    : mk(fx_to(v.x, ls.q), fx_to(v.y, ls.q));
}

struct ClusterState {
    std::mutex mu;
    int ok[64][3] = {};    // per device and cluster size: 0 unknown, 1 usable, -1 not
};
ClusterState g_cl;

template <int CS> cudaError_t launch_cl(const Line1DArgs &a, cudaStream_t st)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorNotSupported;
    const int slot = CS == 8 ? 2 : (CS == 4 ? 1 : 0);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.batch * CS));
    cfg.blockDim = dim3(32);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    {
        std::lock_guard<std::mutex> lk(g_cl.mu);
        if (g_cl.ok[dev][slot] == 0) {
            int ncl = 0;
            cudaLaunchConfig_t probe = cfg;
            probe.gridDim = dim3(CS);
            const cudaError_t oe = cudaOccupancyMaxActiveClusters(&ncl, k_line1d_cluster<CS>, &probe);
            if (oe != cudaSuccess) cudaGetLastError();
            g_cl.ok[dev][slot] = (oe == cudaSuccess && ncl >= 1) ? 1 : -1;
        }
        if (g_cl.ok[dev][slot] < 0) return cudaErrorNotSupported;
    }
    if (a.nsteps <= 0) return cudaSuccess;
    return cudaLaunchKernelEx(&cfg, k_line1d_cluster<CS>, a);
}

}  // namespace

bool line1d_cluster_applies(const Line1DArgs &a)
{
    return !a.imag && (a.n == 64 || a.n == 128 || a.n == 256) && a.batch >= 1 && a.batch <= LINE_CLUSTER_MAX_BATCH;
}

cudaError_t launch_line1d_cluster(const Line1DArgs &a, cudaStream_t st)
{
    switch (a.n) {
    case 64: return launch_cl<2>(a, st);
    case 128: return launch_cl<4>(a, st);
    case 256: return launch_cl<8>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace gpe
