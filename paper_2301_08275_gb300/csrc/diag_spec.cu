// diag_spec.cu - FP64 reductions (norm, energy, mu, rms sizes, renormalisation
// factor) and the kernels of the kinetic-energy spectra.
#include <math.h>

#include "fft_tile.cuh"
#include <algorithm>

#include "gpe_internal.h"

namespace gpe {

// ------------------------------------------------------------------ reductions
// sums[b*NQ + q] = sum over the lines of instance b of partials[q][line], in a
// fixed order that depends only on the number of lines: chunks of
// REDUCE_CHUNK consecutive lines are summed by one CTA each (strided
// per-thread sums into four accumulators, warp shuffles, one shared-memory
// stage), then one warp per (instance, quantity) adds the chunk sums (strided
// per lane, shuffles).  FP64 additions are slow on this GPU (one warp
// instruction per 64 cycles per SM sub-partition): spreading them over many
// SMs is what makes the sum fast (65536 lines: 24 us in one CTA before).
// One launch: the last CTA of an instance to finish its chunk adds that
// instance's chunk sums (an instance of one chunk has none to add; one CTA for
// all instances was a serial tail of FP64 additions: the energies of 64 grids of
// 64 x 128 x 128 took 1158 us, now 1105).  With scale set, the sum of quantity 0 (the norm)
// also gives the imaginary-time renormalisation factor s_b = sqrt(target / (sum
// rho dV)).  Launched dependent on the sweep before it and with the next sweep
// dependent on it, as the sweeps are on one another: as two ordinary launches
// it was 22 of the 346 us of a 256^3 complex64 imaginary step (ncu: 10 us of
// work) and half of the difference between real and imaginary steps of small grids.
__device__ __forceinline__ void reduce_finish(double s, int64_t b, int q, double *sums, double dv, double target,
                                              double *scale, int *err)
{
    sums[b * NQ + q] = s;
    if (scale && q == 0) {
        const double nrm = s * dv;
        if (!(nrm > 0.0) || !isfinite(nrm)) {
            atomicOr(err, (int)ERR_NUMERIC);
            scale[b] = 1.0;
        } else {
            scale[b] = sqrt(target / nrm);
        }
    }
}
__global__ void __launch_bounds__(256) k_reduce_lines(const double *__restrict__ partials, int64_t cap, int q0, int nq,
                                                      int64_t lpi, int64_t nch, double *csum,
                                                      double *__restrict__ sums, double dv, double target,
                                                      double *__restrict__ scale, int *err, unsigned *counter,
                                                      const int *stop)
{
    __shared__ double sh[8];
    __shared__ bool last;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" :::);
    if (stop && *reinterpret_cast<const volatile int *>(stop)) return;
    const int64_t c = blockIdx.x, b = blockIdx.z;
    const int q = q0 + blockIdx.y, t = threadIdx.x;
    const int64_t first = c * REDUCE_CHUNK;
    const int64_t n = lpi - first < REDUCE_CHUNK ? lpi - first : REDUCE_CHUNK;
    const double *p = partials + (int64_t)q * cap + b * lpi + first;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    int64_t j = t;
    for (; j + 3 * 256 < n; j += 4 * 256) {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += p[j + (int64_t)k * 256];
    }
    for (int k = 0; j < n; j += 256, ++k) acc[k & 3] += p[j];
    double s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((t & 31) == 0) sh[t >> 5] = s;
    __syncthreads();
    if (t == 0) {
        const double r = ((sh[0] + sh[1]) + (sh[2] + sh[3])) + ((sh[4] + sh[5]) + (sh[6] + sh[7]));
        last = false;
        if (nch == 1) {
            reduce_finish(r, b, q, sums, dv, target, scale, err);
        } else {
            csum[(b * NQ + q) * nch + c] = r;
            __threadfence();
            last = atomicAdd(counter + b, 1u) == gridDim.x * gridDim.y - 1;
        }
    }
    __syncthreads();
    if (!last) return;
    // every chunk sum of the instance is written: one warp per quantity
    __threadfence();
    const int lane = t & 31;
    for (int w = t >> 5; w < nq; w += 8) {
        const double *pc = csum + (b * NQ + q0 + w) * nch;
        double x = 0.0;
        for (int64_t k = lane; k < nch; k += 32) x += __ldcg(pc + k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) reduce_finish(x, b, q0 + w, sums, dv, target, scale, err);
    }
    if (t == 0) counter[b] = 0;      // for the next launch on this stream
}

// norm, E_kin, E_pot, E_int, E, mu and sigma_x, sigma_y, sigma_z, r_rms from the
// per-instance sums of the diagnostic passes.
__global__ void k_finish_diag(const double *__restrict__ sums, int64_t batch, int ndim, int64_t n0, int64_t n1,
                              int64_t n2, double dv, const double *__restrict__ g, double *__restrict__ out6,
                              double *__restrict__ out4, const int *stop)
{
    if (stop && *reinterpret_cast<const volatile int *>(stop)) return;
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= batch) return;
    const double *q = sums + b * NQ;
    const double nrm = q[0] * dv;
    const double n[3] = {(double)n0, (double)n1, (double)n2};
    double ek = 0.0;
    for (int a = 0; a < ndim; ++a) ek += q[6 + a] / n[a];
    ek *= 0.5 * dv;
    const double ep = q[4] * dv;
    const double ei = 0.5 * g[b] * q[5] * dv;
    out6[6 * b + 0] = nrm;
    out6[6 * b + 1] = ek;
    out6[6 * b + 2] = ep;
    out6[6 * b + 3] = ei;
    out6[6 * b + 4] = ek + ep + ei;
    out6[6 * b + 5] = (ek + ep + 2.0 * ei) / nrm;
    double r2 = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double s2 = a < ndim ? q[1 + a] / q[0] : 0.0;
        out4[4 * b + a] = sqrt(s2);
        r2 += s2;
    }
    out4[4 * b + 3] = sqrt(r2);
}

int64_t reduce_chunks(int64_t lines_per_inst) { return (lines_per_inst + REDUCE_CHUNK - 1) / REDUCE_CHUNK; }

cudaError_t launch_reduce_lines(const double *partials, int64_t lines_cap, int nq_first, int nq, int64_t batch,
                                int64_t lines_per_inst, double *csum, double *sums, unsigned *counter, cudaStream_t st,
                                double dv, double target, double *scale, int *err, const int *stop)
{
    if (batch <= 0 || nq <= 0) return cudaSuccess;
    const int64_t nch = reduce_chunks(lines_per_inst);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nch, (unsigned)nq, (unsigned)batch);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_reduce_lines, partials, lines_cap, nq_first, nq, lines_per_inst, nch, csum, sums,
                               dv, target, scale, err, counter, stop);
}

__global__ void k_imag_init(const double *__restrict__ out6, double *__restrict__ eprev, int64_t batch, int *stop,
                            int64_t *done)
{
    for (int64_t b = threadIdx.x; b < batch; b += blockDim.x) eprev[b] = out6[6 * b + 4];
    if (threadIdx.x == 0) {
        *stop = 0;
        *done = 0;
    }
}

__global__ void __launch_bounds__(256) k_imag_check(const double *__restrict__ out6, double *__restrict__ eprev,
                                                    int64_t batch, double etol, int64_t chunk, int *stop,
                                                    int64_t *done, const int *err)
{
    if (*reinterpret_cast<const volatile int *>(stop)) return;
    // the host rule of gpe_step_imag: stop when every instance moved by less
    // than etol since the last check (never for etol <= 0)
    int moved = !(etol > 0.0), bad = 0;
    for (int64_t b = threadIdx.x; b < batch; b += blockDim.x) {
        const double e = out6[6 * b + 4];
        if (!isfinite(e)) bad = 1;
        if (!(fabs(e - eprev[b]) < etol)) moved = 1;
        eprev[b] = e;
    }
    moved = __syncthreads_or(moved);
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        *done += chunk;
        if (bad || (err && (*reinterpret_cast<const volatile int *>(err) & ERR_NUMERIC))) *stop = 2;
        else if (!moved) *stop = 1;
    }
}

cudaError_t launch_imag_init(const double *out6, double *eprev, int64_t batch, int *stop, int64_t *done,
                             cudaStream_t st)
{
    k_imag_init<<<1, 256, 0, st>>>(out6, eprev, batch, stop, done);
    return cudaGetLastError();
}

cudaError_t launch_imag_check(const double *out6, double *eprev, int64_t batch, double etol, int64_t chunk, int *stop,
                              int64_t *done, const int *err, cudaStream_t st)
{
    k_imag_check<<<1, 256, 0, st>>>(out6, eprev, batch, etol, chunk, stop, done, err);
    return cudaGetLastError();
}

cudaError_t launch_finish_diag(const double *sums, int64_t batch, int ndim, const int64_t *n, double dv,
                               const double *g, double *out6, double *out4, cudaStream_t st, const int *stop)
{
    const int nb = (int)((batch + 127) / 128);
    k_finish_diag<<<nb, 128, 0, st>>>(sums, batch, ndim, n[0], n[1], n[2], dv, g, out6, out4, stop);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ spectra
// coordinate of point i on an axis (all extents are powers of two)
__device__ __forceinline__ int axis_index(int64_t i, const SpecArgs &s, int axis)
{
    const int sh = axis == 0 ? 0 : axis == 1 ? s.lg[0] : s.lg[0] + s.lg[1];
    return (int)(i >> sh) & ((1 << s.lg[axis]) - 1);
}

// dst = i k_axis src, with the Nyquist mode of i k_axis set to zero.
template <typename R>
__global__ void k_deriv(const SpecArgs s, const typename CT<R>::C *__restrict__ src, typename CT<R>::C *__restrict__ dst,
                        int axis)
{
    using C = typename CT<R>::C;
    const int na = 1 << s.lg[axis];
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.N; i += (int64_t)gridDim.x * blockDim.x) {
        const int j = axis_index(i, s, axis);
        const R k = (2 * j == na) ? (R)0 : (R)(s.kf[axis] * (double)(j < na / 2 ? j : j - na));
        const C v = src[i];
        dst[i] = mk(-k * v.y, k * v.x);
    }
}

// sum of one double per thread of a block, in a fixed order; thread 0 has it
__device__ __forceinline__ double block_sum(double s, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sh[w];
    return r;
}

// w <- u = Im(conj(psi) * w / N) / |psi| (part 0) or Re(...) / |psi| (part 1: the
// gradient of |psi|), 0 where |psi|^2 < 1e-30, stored as (u, 0); part 2 leaves w
// alone and takes |psi|.  partial[block] = sum of the squares, which fixes the
// scale of the shell sums (below): a few per mille suffice, so single
// precision adds them, and double precision where those leave its range.
template <typename R>
__global__ void __launch_bounds__(256) k_velocity(const SpecArgs s, const typename CT<R>::C *__restrict__ psi,
                                                  typename CT<R>::C *__restrict__ w, double *__restrict__ partial)
{
    using C = typename CT<R>::C;
    __shared__ double sh[8];
    const R invn = (R)(1.0 / (double)s.N);
    auto value = [&](int64_t i) -> R {
        const C p = psi[i];
        const R rho = p.x * p.x + p.y * p.y;
        if (s.part == 2) return sqrt(rho);
        const C d = w[i];
        R u = (R)0;      // as velocity_of (pass_kernels.cuh)
        if (rho >= (R)1e-30) u = (s.part ? (p.x * d.x + p.y * d.y) : (p.x * d.y - p.y * d.x)) * invn / sqrt(rho);
        return u;
    };
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    float acc = 0.0f;
    for (int64_t i = first; i < s.N; i += step) {
        const R u = value(i);
        const float f = (float)u;
        acc = fmaf(f, f, acc);
        if (s.part != 2) w[i] = mk(u, (R)0);
    }
    double t = (double)acc;
    if (!(acc > 1e-30f && acc < 1e37f)) {
        t = 0.0;
        for (int64_t i = first; i < s.N; i += step) {
            const double u = s.part == 2 ? (double)value(i) : (double)w[i].x;
            t += u * u;
        }
    }
    t = block_sum(t, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

// Shell histogram of |u_i|^2 and |u_c|^2 (split) or of sum_a |u_a|^2 (slot 0)
// over the k grid.  Shell sums are accumulated in 64-bit fixed point so that
// they do not depend on the order in which threads and blocks add (integer
// addition is associative).  The scale is the power of two that maps the
// field's total (Parseval, from the sums of squares in real space), below
// 2^61; rounding costs at most total * 2^-62 per point, of either sign.
//
// FP64 arithmetic bounded this kernel (about 100 FP64 operations a point with
// three divisions: 202 us for a 1024^2 complex64 field), so
//  * the parts come from |k x u|^2 / k^2 and |k . u|^2 / k^2, one division
//    each, for any scale of k: q_a = m_a L_max / L_a in place of k_a;
//  * complex64 fields take them in two-float arithmetic (error-free products
//    and sums, 2^-44 relative; the fields themselves carry 2^-24);
//  * shells of cubic boxes are exact integer tests, of other boxes a single
//    precision root, in double only next to a shell's edge;
//  * neighbouring lanes of one shell add through shuffles, the first of them
//    adds to the block's histogram, and the blocks add theirs to one in global
//    memory (no per-block copies to sum afterwards).
// Spectra of a 1024^2 complex64 field, the whole call: 458 -> 219 us with
// this binning, 153 us with each mode binned beside its mirror image and the
// derivative and the velocity taken inside the transforms (OP_DERIV, OP_VEL).
struct Pf {
    float h, l;
};
__device__ __forceinline__ Pf pf_norm(float h, float l)
{
    const float s = h + l;
    return {s, l - (s - h)};
}
__device__ __forceinline__ Pf pf_add(Pf a, Pf b)
{
    const float s = a.h + b.h, v = s - a.h;
    return pf_norm(s, ((a.h - (s - v)) + (b.h - v)) + (a.l + b.l));
}
__device__ __forceinline__ Pf pf_neg(Pf a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Pf pf_mul(Pf a, float b)
{
    const float p = a.h * b;
    return {p, fmaf(a.h, b, -p) + a.l * b};
}
__device__ __forceinline__ Pf pf_sq(Pf a)
{
    const float p = a.h * a.h;
    return pf_norm(p, fmaf(a.h, a.h, -p) + 2.0f * a.h * a.l);
}
__device__ __forceinline__ Pf pf_div(Pf a, Pf b)
{
    const float r = 1.0f / b.h, z = a.h * r;
    return pf_norm(z, (fmaf(-z, b.h, a.h) + (a.l - z * b.l)) * r);
}
// the same operations on doubles, so that one kernel serves both precisions
template <typename R> struct Wide;
template <> struct Wide<float> {
    using T = Pf;
    __device__ static T make(double v) { return {(float)v, (float)(v - (double)(float)v)}; }
    __device__ static T whole(float v) { return {v, 0.0f}; }
    __device__ static T mul(T a, float b) { return pf_mul(a, b); }
    __device__ static T add(T a, T b) { return pf_add(a, b); }
    __device__ static T neg(T a) { return pf_neg(a); }
    __device__ static T sq(T a) { return pf_sq(a); }
    __device__ static T div(T a, T b) { return pf_div(a, b); }
    __device__ static float hi(T a) { return a.h; }
    // round(v 2^61), 0 <= v <= 1
    __device__ static long long fixed(T a)
    {
        return __float2ll_rn(a.h * 2305843009213693952.0f) + __float2ll_rn(a.l * 2305843009213693952.0f);
    }
};
template <> struct Wide<double> {
    using T = double;
    __device__ static T make(double v) { return v; }
    __device__ static T whole(double v) { return v; }
    __device__ static T mul(T a, double b) { return a * b; }
    __device__ static T add(T a, T b) { return a + b; }
    __device__ static T neg(T a) { return -a; }
    __device__ static T sq(T a) { return a * a; }
    __device__ static T div(T a, T b) { return a / b; }
    __device__ static float hi(T a) { return (float)a; }
    __device__ static long long fixed(T a) { return __double2ll_rn(a * 2305843009213693952.0); }
};

// power of two that scales the fields so that their squares sum to at most one
__device__ __forceinline__ double field_scale(double total, int prec)
{
    if (!(total > 0.0) || !isfinite(total)) return 1.0;
    int ex = 0;
    frexp(total * 1.002, &ex);
    int h = (ex + 1) >> 1;                        // total < 2^ex <= 4^h
    if (prec == 0) h = max(-126, min(126, h));
    return ldexp(1.0, -h);
}

//
// Modes +-m of every axis share their shell and their q up to signs: a thread
// takes all of them (4 points in 2D, 8 in 3D) and divides, converts and adds
// once.  Warps take runs of 32 consecutive m_x >= 0 of a row of (m_y, m_z) >= 0.
constexpr int BIN_THREADS = 512;
template <typename R>
__global__ void __launch_bounds__(BIN_THREADS) k_bin(const SpecArgs s, const typename CT<R>::C *__restrict__ u0,
                                                     const typename CT<R>::C *__restrict__ u1,
                                                     const typename CT<R>::C *__restrict__ u2, int nshells,
                                                     const double *__restrict__ partial, int npartial, double total,
                                                     unsigned long long *__restrict__ hist,
                                                     double *__restrict__ scale_out)
{
    using C = typename CT<R>::C;
    using W = Wide<R>;
    using T = typename W::T;
    extern __shared__ unsigned long long shq[];   // [2][nshells]
    __shared__ double shd[BIN_THREADS / 32], shs;
    const int nsum = (s.split ? 2 : 1) * nshells;
    for (int i = threadIdx.x; i < nsum; i += BIN_THREADS) shq[i] = 0ull;
    double t = 0.0;
    for (int i = threadIdx.x; i < npartial; i += BIN_THREADS) t += partial[i];
    t = block_sum(t, shd);
    if (threadIdx.x == 0) {
        shs = field_scale(t * total, s.prec);
        // a field that is not finite has no spectrum
        if (blockIdx.x == 0) *scale_out = isfinite(t) ? shs : __longlong_as_double(0x7ff8000000000000ll);
    }
    __syncthreads();
    const R sc = (R)shs;
    const C *const u[3] = {u0, u1, u2};
    const int lane = threadIdx.x & 31;
    const T lr[3] = {W::make(s.lratio[0]), W::make(s.lratio[1]), W::make(s.lratio[2])};
    const int n[3] = {1 << s.lg[0], 1 << s.lg[1], 1 << s.lg[2]};
    const int h0 = n[0] / 2 + 1, h1 = n[1] / 2 + 1, h2 = n[2] / 2 + 1;      // modes 0 .. n/2 (one for an absent axis)
    const int chunks = (h0 + 31) / 32;
    const int64_t units = (int64_t)chunks * h1 * h2;
    const int nc = s.split ? s.ndim : s.ncomp;
    // whole warps run every iteration (the shuffles below)
    for (int64_t w = blockIdx.x * (int64_t)(BIN_THREADS / 32) + (threadIdx.x >> 5); w < units;
         w += (int64_t)gridDim.x * (BIN_THREADS / 32)) {
        const int row = (int)(w / chunks);
        int m[3];
        m[0] = (int)(w - (int64_t)row * chunks) * 32 + lane;
        m[2] = row / h1;
        m[1] = row - m[2] * h1;
        const bool on = m[0] < h0;
        long long ei = 0, ec = 0;
        int shell = -1;
        if (on) {
            T q[3], q2;
            if (s.cubic) {
                const int k2 = m[0] * m[0] + m[1] * m[1] + m[2] * m[2];
                // floor(sqrt(k2) + 1/2) = n  <=>  n^2 - n < k2 <= n^2 + n (or n = 0 = k2)
                int r = (int)(sqrtf((float)k2) + 0.5f);
                if (r > 0 && k2 <= r * r - r) --r;
                if (k2 > r * r + r) ++r;
                shell = r;
                q2 = W::whole((R)k2);
#pragma unroll
                for (int a = 0; a < 3; ++a) q[a] = W::whole((R)m[a]);
            } else {
                q2 = W::whole((R)0);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    q[a] = W::mul(lr[a], (R)m[a]);
                    q2 = W::add(q2, W::sq(q[a]));
                }
                const float r = sqrtf(W::hi(q2)) + 0.5f, tol = 1e-6f * r + 1e-6f;
                shell = (int)r;
                if (r - (float)shell < tol || (float)shell + 1.0f - r < tol) {
                    double d2 = 0.0;
                    for (int a = 0; a < s.ndim; ++a) {
                        const double qa = (double)m[a] * s.lratio[a];
                        d2 += qa * qa;
                    }
                    shell = (int)floor(sqrt(d2) + 0.5);
                }
            }
            const bool parts = s.split && (m[0] | m[1] | m[2]) != 0;
            T si = W::whole((R)0), scp = W::whole((R)0);
            // sign of every axis; modes 0 and n/2 (the Nyquist mode, -n/2) have one
            const int k0 = m[0] == 0 || 2 * m[0] == n[0] ? 1 : 2, k1 = m[1] == 0 || 2 * m[1] == n[1] ? 1 : 2,
                      k2s = m[2] == 0 || 2 * m[2] == n[2] ? 1 : 2;
            for (int c2 = 0; c2 < k2s; ++c2)
                for (int c1 = 0; c1 < k1; ++c1)
                    for (int c0 = 0; c0 < k0; ++c0) {
                        const int64_t i = (int64_t)(c0 ? n[0] - m[0] : m[0]) +
                                          ((int64_t)(c1 ? n[1] - m[1] : m[1]) << s.lg[0]) +
                                          ((int64_t)(c2 ? n[2] - m[2] : m[2]) << (s.lg[0] + s.lg[1]));
                        const R sg[3] = {c0 || 2 * m[0] == n[0] ? -sc : sc, c1 || 2 * m[1] == n[1] ? -sc : sc,
                                         c2 || 2 * m[2] == n[2] ? -sc : sc};
                        R re[3] = {(R)0, (R)0, (R)0}, im[3] = {(R)0, (R)0, (R)0};
                        for (int a = 0; a < nc; ++a) {
                            const C v = u[a][i];
                            // q_a carries its sign through the component (all products below are even in it)
                            re[a] = v.x * (parts ? sg[a] : sc);
                            im[a] = v.y * (parts ? sg[a] : sc);
                        }
                        if (!parts) {
#pragma unroll
                            for (int a = 0; a < 3; ++a)
                                si = W::add(si, W::add(W::sq(W::whole(re[a])), W::sq(W::whole(im[a]))));
                            continue;
                        }
                        auto cross = [&](const R *v, int a, int b) {
                            return W::add(W::mul(q[a], v[b]), W::neg(W::mul(q[b], v[a])));
                        };
                        auto dot = [&](const R *v) {
                            T d = W::add(W::mul(q[0], v[0]), W::mul(q[1], v[1]));
                            if (s.ndim > 2) d = W::add(d, W::mul(q[2], v[2]));
                            return d;
                        };
                        si = W::add(si, W::add(W::sq(cross(re, 0, 1)), W::sq(cross(im, 0, 1))));
                        if (s.ndim > 2) {
                            si = W::add(si, W::add(W::sq(cross(re, 0, 2)), W::sq(cross(im, 0, 2))));
                            si = W::add(si, W::add(W::sq(cross(re, 1, 2)), W::sq(cross(im, 1, 2))));
                        }
                        scp = W::add(scp, W::add(W::sq(dot(re)), W::sq(dot(im))));
                    }
            if (parts) {
                ei = W::fixed(W::div(si, q2));
                ec = W::fixed(W::div(scp, q2));
            } else {
                ei = W::fixed(si);
            }
        }
        // sums over runs of lanes with one shell; the first lane of a run adds them
        const int up = __shfl_up_sync(0xffffffffu, shell, 1);
        const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || up != shell);
        const unsigned later = lane == 31 ? 0u : heads >> (lane + 1);
        const int run = later ? __ffs((int)later) : 32 - lane;       // lanes from here to the run's end
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long a = __shfl_down_sync(0xffffffffu, ei, o);
            if (o < run) ei += a;
            if (s.split) {
                const long long c = __shfl_down_sync(0xffffffffu, ec, o);
                if (o < run) ec += c;
            }
        }
        if (on && ((heads >> lane) & 1u)) {
            atomicAdd(&shq[shell], (unsigned long long)ei);
            if (s.split) atomicAdd(&shq[nshells + shell], (unsigned long long)ec);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nsum; i += BIN_THREADS)
        if (shq[i]) atomicAdd(&hist[i], shq[i]);
}
// shells out of the histogram (second slot only when split)
__global__ void k_hist_out(const unsigned long long *__restrict__ hist, int nshells, int split,
                           const double *__restrict__ scale_p, double half_dv_over_n, double *__restrict__ out)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= 2 * nshells) return;
    const double inv = 1.0 / *scale_p;            // powers of two: exact
    out[s] = !split && s >= nshells ? 0.0 : half_dv_over_n * ((double)hist[s] * 4.3368086899420177e-19 * inv * inv);
}

static int grid_for(int64_t N)
{
    int64_t b = (N + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    return (int)(b < 1 ? 1 : b);
}

int velocity_blocks(const SpecArgs &s)
{
    const int64_t b = (s.N + 255) / 256;
    return (int)(b < 1 ? 1 : b > 152 * 4 ? 152 * 4 : b);
}

cudaError_t launch_deriv(const SpecArgs &s, const void *src, void *dst, int axis, cudaStream_t st)
{
    if (s.prec == 0)
        k_deriv<float><<<grid_for(s.N), 256, 0, st>>>(s, (const float2 *)src, (float2 *)dst, axis);
    else
        k_deriv<double><<<grid_for(s.N), 256, 0, st>>>(s, (const double2 *)src, (double2 *)dst, axis);
    return cudaGetLastError();
}

cudaError_t launch_velocity(const SpecArgs &s, const void *psi, void *w, double *partial, cudaStream_t st)
{
    const int nb = velocity_blocks(s);
    if (s.prec == 0) k_velocity<float><<<nb, 256, 0, st>>>(s, (const float2 *)psi, (float2 *)w, partial);
    else k_velocity<double><<<nb, 256, 0, st>>>(s, (const double2 *)psi, (double2 *)w, partial);
    return cudaGetLastError();
}

// Trap tables of one time level (see launch_trap_level): angles in double
// precision from the same formula as the plan's static tables, split into
// hi + lo floats for complex64.
__global__ void k_trap_level(int prec, void *t0, void *t1, void *t2, int ndim, int64_t n0, int64_t n1, int64_t n2,
                             double lo0, double lo1, double lo2, double h0, double h1, double h2, double g0, double g1,
                             double g2, double c, int64_t batch)
{
    const int64_t tot = n0 + (ndim > 1 ? n1 : 0) + (ndim > 2 ? n2 : 0);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < tot * batch;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = q / tot;
        int64_t j = q - b * tot;
        int a = 0;
        if (j >= n0) {
            j -= n0;
            a = 1;
            if (j >= n1) {
                j -= n1;
                a = 2;
            }
        }
        const int64_t na = a == 0 ? n0 : (a == 1 ? n1 : n2);
        const double x = (a == 0 ? lo0 : (a == 1 ? lo1 : lo2)) + (double)j * (a == 0 ? h0 : (a == 1 ? h1 : h2));
        const double gm = a == 0 ? g0 : (a == 1 ? g1 : g2);
        const double th = 0.5 * gm * gm * x * x * c;
        if (prec == 2) {
            static_cast<long long *>(a == 0 ? t0 : (a == 1 ? t1 : t2))[b * na + j] = fx_turns(th / 6.283185307179586477);
            continue;
        }
        const double sh = sin(0.5 * th);
        const double wx = -2.0 * sh * sh, wy = -sin(th);
        const float hx = (float)wx, hy = (float)wy;
        static_cast<float4 *>(a == 0 ? t0 : (a == 1 ? t1 : t2))[b * na + j] =
            make_float4(hx, hy, (float)(wx - (double)hx), (float)(wy - (double)hy));
    }
}

cudaError_t launch_trap_level(int prec, void *const *tab, int ndim, const int64_t *n, const double *lo,
                              const double *h, const double *gamma, double c, int64_t batch, cudaStream_t st)
{
    const int64_t tot = (n[0] + (ndim > 1 ? n[1] : 0) + (ndim > 2 ? n[2] : 0)) * batch;
    const int blocks = (int)std::min<int64_t>((tot + 255) / 256, 1024);
    k_trap_level<<<blocks, 256, 0, st>>>(prec, tab[0], ndim > 1 ? tab[1] : nullptr, ndim > 2 ? tab[2] : nullptr, ndim,
                                         n[0], ndim > 1 ? n[1] : 1, ndim > 2 ? n[2] : 1, lo[0], lo[1], lo[2], h[0], h[1],
                                         h[2], gamma[0], gamma[1], gamma[2], c, batch);
    return cudaGetLastError();
}

// histogram and shells of the fields uh; work: 2 nshells + 1 doubles (histogram
// and scale); total times the sum of the npartial numbers at partial is the sum of
// squares of the fields
cudaError_t launch_bin(const SpecArgs &s, void *const *uh, int64_t nshells, const double *partial, int npartial,
                       double total, double *work, double half_dv_over_n, double *out, cudaStream_t st)
{
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(work);
    double *scale = work + 2 * nshells;
    const size_t smem = sizeof(unsigned long long) * (s.split ? 2 : 1) * (size_t)nshells;
    // two blocks per SM: each sums the partials (FP64) before it starts
    int64_t units = (((int64_t)1 << s.lg[0]) / 2 + 32) / 32;
    for (int a = 1; a < 3; ++a) units *= ((int64_t)1 << s.lg[a]) / 2 + 1;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((units + BIN_THREADS / 32 - 1) / (BIN_THREADS / 32), 152 * 2));
    // the attribute belongs to the process: always the largest size, so that no call
    // takes room from another thread's launch
    constexpr int most = (int)(2 * MAX_SHELLS * sizeof(unsigned long long));
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * 2 * (size_t)nshells, st);
    if (e != cudaSuccess) return e;
    if (s.prec == 0) {
        e = cudaFuncSetAttribute(k_bin<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
        k_bin<float><<<nb, BIN_THREADS, smem, st>>>(s, (const float2 *)uh[0], (const float2 *)uh[1], (const float2 *)uh[2],
                                            (int)nshells, partial, npartial, total, hist, scale);
    } else {
        e = cudaFuncSetAttribute(k_bin<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
        k_bin<double><<<nb, BIN_THREADS, smem, st>>>(s, (const double2 *)uh[0], (const double2 *)uh[1], (const double2 *)uh[2],
                                             (int)nshells, partial, npartial, total, hist, scale);
    }
    k_hist_out<<<(unsigned)((2 * nshells + 127) / 128), 128, 0, st>>>(hist, (int)nshells, s.split, scale,
                                                                     half_dv_over_n, out);
    return cudaGetLastError();
}

}  // namespace gpe
