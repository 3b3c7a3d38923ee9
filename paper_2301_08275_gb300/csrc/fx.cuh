// fx.cuh - 64-bit fixed-point line arithmetic of the complex128 sweeps.
//
// What bounds complex128 on this GPU is its FP64 pipe: one FP64 instruction
// keeps an SM sub-partition for 64 cycles per warp, a 32 x 32 + 64-bit integer
// multiply-add (IMAD.WIDE) for 2.0 and a 64-bit integer addition for 2.3 (both
// measured).  A transform along a line needs no floating point: after one
// common power-of-two scale per line every value fits a 64-bit integer, and an
// addition then costs 1/28 and a product by a unit factor about 1/6 of its
// FP64 form.  The state stays complex128 in memory; a sweep converts each line
// on load and store (integer instructions too).
//
// Precision.  A line is held as X = x 2^-q in signed 64-bit integers, with q
// the smallest exponent for which no value of the sweep can leave 62 bits:
// every partial sum of a unitary-factor transform over n points is at most
// sqrt(n) |x|_2 (Cauchy-Schwarz), and |x|_2 is bounded from the line itself
// (line_scale below).  That leaves 52 to 55 bits below the line's rms value in
// every stage, and integer additions are exact, so a line picks up a rounding
// error of at most a few 2^-54 of its rms value per multiplication stage
// against 2^-53 per addition and multiplication in FP64.  Twiddles are rounded to
// nearest at 62 fraction bits; kinetic factors are 1 + w for a w in double
// precision, as FP64 sweeps had them.  Measured against long double
// (2D and 3D grids, 30 to 100 steps, real and imaginary time): relative L2
// error 0.07 to 0.62 of the FP64 sweeps' it replaced, norm drift 0.03 to 0.6.
//
// Measured time of a 1024^2 complex128 real-time step: 451 us in FP64, 83 us
// in fixed point; of a 128^2 imaginary-time step as sweeps 66 and 33 us (4 in
// place of 8 points per thread among it), 20 us on chip (plane_cluster.cu).
//
// Products: a 64-bit value is split as a = ah 2^32 + al with a SIGNED low half
// (limbs), so every partial product is one signed IMAD.WIDE.  al * wl (at most
// a quarter of the result's last place, of either sign) is left out.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace gpe {

struct fx {};                                   // scalar tag of the tile engine (fft_tile.cuh)
struct __align__(16) fx2 {
    long long x, y;
};
// A unit factor w is held as the limbs of round(w 2^62): (re high, re low, im
// high, im low).

__host__ __device__ __forceinline__ fx2 mk(long long a, long long b)
{
    fx2 r;
    r.x = a;
    r.y = b;
    return r;
}

// c + a b, 32 x 32 + 64 bits
__device__ __forceinline__ long long imad(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ long long imul(int a, int b)
{
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
// a = h 2^32 + l, l signed (|a| < 2^63 - 2^31)
struct Limbs {
    int h, l;
};
__device__ __forceinline__ Limbs limbs(long long a)
{
    Limbs r;
    r.l = (int)a;
    r.h = (int)(a >> 32) + (int)((unsigned)r.l >> 31);
    return r;
}
__host__ __device__ __forceinline__ int4 fx_pack(long long re, long long im)
{
    int4 u;
    u.y = (int)re;
    u.x = (int)((re - u.y) >> 32);
    u.w = (int)im;
    u.z = (int)((im - u.w) >> 32);
    return u;
}
__device__ __forceinline__ fx2 fx_value(int4 u)
{
    return mk(((long long)u.x << 32) + u.y, ((long long)u.z << 32) + u.w);
}
__device__ __forceinline__ int4 fx_unit(fx2 w)
{
    const Limbs a = limbs(w.x), b = limbs(w.y);
    return make_int4(a.h, a.l, b.h, b.l);
}

// v w 2^(SH - 64) for w given by its limbs: SH = 0 divides by 4 what a factor
// held to 62 bits multiplies, SH = 64 - (fraction bits of w) keeps the scale.
// |v| < 2^62, |w| <= 2^62 (the cross sums then stay below 2^63).  Only high
// limbs are negated: a low limb can be -2^31, which has no negative.
template <int SH> __device__ __forceinline__ fx2 fx_mul(fx2 v, int4 w)
{
    const Limbs x = limbs(v.x), y = limbs(v.y);
    const int ih = w.z, il = w.w;
    constexpr long long half = 1ll << (31 - SH);
    long long mr = imad(x.h, w.y, half), mi = imad(x.h, il, half);
    mr = imad(x.l, w.x, mr);
    mi = imad(x.l, ih, mi);
    mr = imad(-y.h, il, mr);
    mi = imad(y.h, w.y, mi);
    mr = imad(y.l, -ih, mr);
    mi = imad(y.l, w.x, mi);
    long long hr = imul(x.h, w.x), hi = imul(x.h, ih);
    hr = imad(-y.h, ih, hr);
    hi = imad(y.h, w.x, hi);
    if constexpr (SH == 0) return mk(hr + (mr >> 32), hi + (mi >> 32));
    return mk((hr << SH) + (mr >> (32 - SH)), (hi << SH) + (mi >> (32 - SH)));
}
// a b 2^(SH - 64) for reals, plus c
template <int SH> __device__ __forceinline__ long long fx_mulr(long long a, Limbs b, long long c = 0)
{
    const Limbs x = limbs(a);
    long long m = imad(x.h, b.l, 1ll << (31 - SH));
    m = imad(x.l, b.h, m);
    if constexpr (SH == 0) return imad(x.h, b.h, c) + (m >> 32);
    return (imul(x.h, b.h) << SH) + (m >> (32 - SH)) + c;
}
// v + v w 2^-64, w small (offset of a unit factor from one, 64 fraction bits)
__device__ __forceinline__ fx2 fx_madd1(fx2 v, fx2 w)
{
    const Limbs x = limbs(v.x), y = limbs(v.y), a = limbs(w.x), b = limbs(w.y);
    constexpr long long half = 1ll << 31;
    long long mr = imad(x.h, a.l, half), mi = imad(x.h, b.l, half);
    mr = imad(x.l, a.h, mr);
    mi = imad(x.l, b.h, mi);
    mr = imad(-y.h, b.l, mr);
    mi = imad(y.h, a.l, mi);
    mr = imad(y.l, -b.h, mr);
    mi = imad(y.l, a.h, mi);
    long long hr = imad(x.h, a.h, v.x), hi = imad(x.h, b.h, v.y);
    hr = imad(-y.h, b.h, hr);
    hi = imad(y.h, a.h, hi);
    return mk(hr + (mr >> 32), hi + (mi >> 32));
}

// the tile engine's operations: a twiddle divides by 4 (the growth of the
// radix-8 pass that follows it is at most 8, sqrt(8) in the mean), so the
// butterfly's first input, which has no twiddle, is divided alike
// (radix-4 plans divide by 2)
template <bool CONJ = false, int SH = 0> __device__ __forceinline__ fx2 umul(fx2 v, int4 w)
{
    static_assert(!CONJ, "the sweeps run one copy of the forward transform");
    return fx_mul<SH>(v, w);
}
// (ties to even: rounding them up would shift every mode alike by 1/8 of the
// last place, which the inverse transform gathers at the line's first point)
template <int SH> __device__ __forceinline__ long long fx_down(long long a)
{
    constexpr int d = 2 - SH;
    return (a + ((1 << (d - 1)) - 1) + ((a >> d) & 1)) >> d;
}
template <int SH = 0> __device__ __forceinline__ fx2 tw_first(fx2 v) { return mk(fx_down<SH>(v.x), fx_down<SH>(v.y)); }
// x / sqrt(2) = x - x (1 - 1/sqrt(2)): the constant has 64 fraction bits, the result keeps the scale
__device__ __forceinline__ long long mul_rsqrt2(long long a)
{
    // round((1 - 1/sqrt(2)) 2^64) = 1257966796 2^32 + 102865788
    constexpr int dh = 1257966796, dl = 102865788;
    const Limbs x = limbs(a);
    long long m = imad(x.h, -dl, 1ll << 31);
    m = imad(x.l, -dh, m);
    return imad(x.h, -dh, a) + (m >> 32);
}

// ---------------------------------------------------------------- conversions
// Both directions round to nearest, ties to even: one to three bits are dropped
// from most values, so ties are common, and rounding them away from zero made
// the norm grow by 2e-17 per step.

// round(x 2^-q), |x| 2^-q < 2^62, q >= -1021 (zero and subnormal x give 0)
__device__ __forceinline__ long long fx_from(double x, int q)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int e = (hi >> 20) & 0x7ff;
    // the mantissa below bit 63; PTX shifts clamp: 64 or more gives 0
    const unsigned mh = 0x40000000u | (__funnelshift_l((unsigned)lo, (unsigned)hi, 10) & 0x3fffffffu);
    const unsigned long long m = ((unsigned long long)mh << 32) | (unsigned)(lo << 10);
    const int s = 1085 + q - e;
    unsigned long long t, h, y;
    asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(s));
    asm("shl.b64 %0, %1, %2;" : "=l"(h) : "l"(1ull), "r"(s - 1));
    asm("shr.u64 %0, %1, %2;" : "=l"(y) : "l"(m + (t & 1) + h - 1), "r"(s));
    const long long g = (long long)(hi >> 31);
    return (long long)(y ^ (unsigned long long)g) - g;
}
// X 2^q to the nearest double, -1021 <= q <= 959
__device__ __forceinline__ double fx_to(long long X, int q)
{
    const long long s = X >> 63;
    const unsigned long long m = (unsigned long long)((X ^ s) - s);
    const unsigned h = (unsigned)(m >> 32), l = (unsigned)m;
    const int lz = h ? __clz((int)h) : 32 + __clz((int)l);
    const unsigned long long M = m << (lz & 63);
    const unsigned low = (unsigned)M;
    unsigned long long r = (M >> 11) + (((low & 0x7ffu) + ((low >> 11) & 1u) + 0x3ffu) >> 11);
    // the mantissa's leading one adds the last unit of the exponent
    r += (unsigned long long)(unsigned)(1085 + q - lz) << 52;
    r = (m == 0 ? 0ull : r) | ((unsigned long long)s & 0x8000000000000000ull);
    return __longlong_as_double((long long)r);
}

// Line scale.  Every value of the line is bounded by its exponent, reduced to
// the line's largest; the squares of 9-bit truncations (rounded up) relative to
// that bound |x|_2 within a few per cent.  Both reductions are integer, so the
// scale does not depend on the order in which threads or tile shapes add.
// wmax, wsum: one word per line, zero on entry; returns q and marks lines that
// hold an infinity or a NaN (or whose values leave the range of fx_to).
struct LineScale {
    int q;
    bool bad;
};
template <int L, int NT, int E>
__device__ __forceinline__ LineScale line_scale(const double2 (&d)[E], unsigned *wmax, unsigned *wsum, int l, int gb)
{
    unsigned mx = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        mx = max(mx, (unsigned)__double2hiint(d[e].x) & 0x7fffffffu);
        mx = max(mx, (unsigned)__double2hiint(d[e].y) & 0x7fffffffu);
    }
    constexpr bool WARP = NT % 32 == 0 && L <= 16;
    const int lane = threadIdx.x & 31;
    if constexpr (WARP) {
        if constexpr (L == 1) {
            mx = __reduce_max_sync(0xffffffffu, mx);
        } else {
#pragma unroll
            for (int o = 16; o >= L; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane < L) atomicMax(&wmax[l], mx);
    } else {
        atomicMax(&wmax[l], mx);
    }
    __syncthreads();
    const int em = (int)(wmax[l] >> 20);
    unsigned s = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const unsigned hi = (unsigned)__double2hiint(c ? d[e].y : d[e].x);
            const unsigned t = ((hi & 0xfffffu) | 0x100000u) >> min(31, 12 + em - (int)((hi >> 20) & 0x7ffu));
            s += (t + 1) * (t + 1);
        }
    }
    if constexpr (WARP) {
        if constexpr (L == 1) {
            s = __reduce_add_sync(0xffffffffu, s);
        } else {
#pragma unroll
            for (int o = 16; o >= L; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        }
        if (lane < L) atomicAdd(&wsum[l], s);
    } else {
        atomicAdd(&wsum[l], s);
    }
    __syncthreads();
    s = wsum[l];
    // |x|_2 <= 2^(nb + em - 1031), 4^nb >= s
    const int nb = (33 - __clz((int)s)) >> 1;
    LineScale r;
    r.q = max(nb + em - 1031 + gb - 61, -1021);
    r.bad = em == 0x7ff || r.q > 800;
    return r;
}

// ---------------------------------------------------------------- phases
// v exp(-2 pi i t / 2^64).  Angles of at most 1/64 turn (the usual case) take a
// Maclaurin series of the offset from one, applied as v + v w; the others a
// full-circle form.  Each coefficient below is round(c_k scale^k 2^bits) of the
// series in the variable named with it.
//   short: z = t 2^-58 in [-1, 1], a = 2 pi / 64, u = z^2 / 16: cos a z - 1 and
//   sin a z / z, 64 fraction bits; first terms left out 2e-21 and 2e-19
//   long: z = r 2^-61 in [-1, 1] (r the angle less its nearest quarter turn),
//   a = pi / 4, u = z^2 / 16, 60 fraction bits; terms left out 3e-21 and 8e-20
__device__ __forceinline__ fx2 fx_small_offset(long long t)
{
    const long long z4 = t << 4;                       // z, 62 fraction bits
    const Limbs z = limbs(z4);
    const Limbs u = limbs(fx_mulr<0>(z4, z));          // z^2 / 16, 64 fraction bits
    long long c = (imul(443359018, u.h) >> 32) - 258748764451ll;
    c = fx_mulr<0>(c, u, 93960764191488ll);
    c = fx_mulr<0>(c, u, -18278814420134671ll);
    c = fx_mulr<0>(c, u, 1422359894497287770ll);
    c = fx_mulr<0>(-c, u);
    long long s = (long long)(((unsigned long long)2822511172u * (unsigned)u.h) >> 32) - 1317796636204ll;
    s = fx_mulr<0>(s, u, 358903681866414ll);
    s = fx_mulr<0>(s, u, -46546618701181590ll);
    s = fx_mulr<0>(s, u, 1811004864519280711ll);
    s = fx_mulr<2>(-s, z);
    return mk(c, s);
}
static __device__ __noinline__ fx2 fx_rotate_any(fx2 v, long long t)
{
    const int quad = (int)((unsigned long long)(t + (1ll << 61)) >> 62);
    const long long r = t - (long long)((unsigned long long)quad << 62);
    const long long z2 = r << 1;                       // z, 62 fraction bits
    const Limbs z = limbs(z2);
    const Limbs u = limbs(fx_mulr<0>(z2, z));
    long long c = fx_mulr<0>(-160013427551ll, u, 4961101462710ll);
    c = fx_mulr<0>(c, u, -120639521369162ll);
    c = fx_mulr<0>(c, u, 2224647716048689ll);
    c = fx_mulr<0>(c, u, -29753320050600495ll);
    c = fx_mulr<0>(c, u, 271317744433452895ll);
    c = fx_mulr<0>(c, u, -1539453160513337852ll);
    c = fx_mulr<0>(c, u, 4679376491554475725ll);
    c = fx_mulr<0>(c, u, -5689439577989151081ll);
    c = fx_mulr<0>(c, u, 1152921504606846976ll);
    long long s = fx_mulr<0>(155432976ll, u, -6614434322ll);
    s = fx_mulr<0>(s, u, 229202351602ll);
    s = fx_mulr<0>(s, u, -6316670567766ll);
    s = fx_mulr<0>(s, u, 134402633106998ll);
    s = fx_mulr<0>(s, u, -2124382083883464ll);
    s = fx_mulr<0>(s, u, 23676939797241351ll);
    s = fx_mulr<0>(s, u, -172726240700510392ll);
    s = fx_mulr<0>(s, u, 735034740462416105ll);
    s = fx_mulr<0>(s, u, -1489491798437810879ll);
    s = fx_mulr<0>(s, u, 905502432259640355ll);
    s = fx_mulr<2>(s, z);
    // exp(-i (quad pi/2 + a z)) = (-i)^quad (c - i s)
    fx2 w = mk(c, -s);
    if (quad & 1) w = mk(-s, -c);
    if (quad & 2) w = mk(-w.x, -w.y);
    return fx_mul<4>(v, fx_unit(w));
}
__device__ __forceinline__ fx2 fx_rotate(fx2 v, long long t)
{
    if (t + (1ll << 58) >= 0 && t <= (1ll << 58)) return fx_madd1(v, fx_small_offset(t));
    return fx_rotate_any(v, t);
}
// largest exponent of two that one term of an imaginary-time factor may have
// (three of them add up, see fx_nimag, and fx_exp2m takes less than 1024)
constexpr int FX_EXP_MAX = 340;
// 2^-a for a held to 53 fraction bits (|a| < 1024), as a double: the nearest
// whole number to the exponent, exp of the rest from its Maclaurin series to
// the 14th term (z = 2 rest in [-1, 1], variable z / 4, 60 fraction bits; the
// first term left out is below 1e-19)
__device__ __forceinline__ double fx_exp2m(long long a)
{
    const int n = (int)((a + (1ll << 52)) >> 53);
    const Limbs z = limbs(((long long)n << 53) - a << 10);
    long long p = (imul(1280465205, z.h) >> 32) + 12931245613ll;
    p = fx_mulr<0>(p, z, 121262985468ll);
    p = fx_mulr<0>(p, z, 1049673046670ll);
    p = fx_mulr<0>(p, z, 8328969544420ll);
    p = fx_mulr<0>(p, z, 60080815287248ll);
    p = fx_mulr<0>(p, z, 390052324203650ll);
    p = fx_mulr<0>(p, z, 2250906215263282ll);
    p = fx_mulr<0>(p, z, 11365799319932687ll);
    p = fx_mulr<0>(p, z, 49192146943818121ll);
    p = fx_mulr<0>(p, z, 177423166116318949ll);
    p = fx_mulr<0>(p, z, 511935043789664227ll);
    p = fx_mulr<0>(p, z, 1107849223398934356ll);
    p = fx_mulr<0>(p, z, 1598288580650331957ll);
    p = fx_mulr<0>(p, z, 1152921504606846976ll);
    if (n > 960) return 0.0;
    if (n < -900) return __longlong_as_double(0x7ff0000000000000ll);
    return fx_to(p, -60 - n);
}

// sqrt(|g| c / 2 pi) = m 2^e with m of 62 bits (0 for g = 0), and the sign of
// g: the nonlinear angle in turns is the square of |v| times it.  One entry
// per instance and substep length (half, full), built on the host.
struct FxCoupling {
    long long m;
    int e, neg;
};
// |v|^2 m^2 in 2^-64 turns for v = X 2^q: u = X m 2^e to 54 fraction bits,
// squared in 128 bits; sh = the shift from the product to that scale.  The
// angle is right modulo one turn for every |u| < 2^62, which sh <= 0 ensures.
__device__ __forceinline__ long long fx_angle(fx2 X, Limbs m, int sh)
{
    const int r = min(-sh, 63);
    const long long half = r > 0 ? 1ll << (r - 1) : 0;
    const Limbs a = limbs((fx_mulr<2>(X.x, m) + half) >> r), b = limbs((fx_mulr<2>(X.y, m) + half) >> r);
    const long long hh = imad(b.h, b.h, imul(a.h, a.h));
    const long long mid = imad(b.h, b.l, imul(a.h, a.l));
    const unsigned long long ll = (unsigned long long)imul(a.l, a.l) + (unsigned long long)imul(b.l, b.l);
    return (long long)((unsigned long long)hh << 20) + (mid >> 11) + (long long)(ll >> 44);
}
// a double in turns, reduced to [-1/2, 1/2], in 2^-64 turns
__device__ __forceinline__ long long fx_turns(double t)
{
    t -= rint(t);
    return (long long)((unsigned long long)(long long)(t * 9223372036854775808.0) << 1);
}

// The interaction's angle for values held as v 2^q: coupling entry gq (half or
// full step), g c / 2 pi as a double for angles that may pass a turn.
struct FxNonlinear {
    Limbs m;
    int sh, q;
    bool none, neg;
};
__device__ __forceinline__ FxNonlinear fx_nonlinear(const FxCoupling *gq, int q)
{
    FxNonlinear r;
    const long long m = gq->m;
    r.m = limbs(m);
    r.none = m == 0;
    r.neg = gq->neg != 0;
    r.sh = 62 + 54 + gq->e + q;
    r.q = q;
    return r;
}
__device__ __forceinline__ long long fx_nl_angle(fx2 v, const FxNonlinear &f, double g, double c_turn)
{
    if (f.none) return 0;
    if (f.sh <= 0) {
        const long long t = fx_angle(v, f.m, f.sh);
        return f.neg ? -t : t;
    }
    // in FP64, reduced there
    const double x = fx_to(v.x, f.q), y = fx_to(v.y, f.q);
    return fx_turns(g * c_turn * (x * x + y * y));
}

}  // namespace gpe
