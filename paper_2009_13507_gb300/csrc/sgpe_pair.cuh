// sgpe_pair.cuh -- the 2D step of the complex128 and double-float forms on the
// FP32 pipe: every substep as an increment in FP32 pairs, added to the state once
// per kernel.
//
// Why. GB300's FP64 pipe takes a warp instruction every 64 cycles, its FP32 pipe
// one per cycle, and the FP64 step (about 270 FP64 instructions a point) kept the
// FP64 pipe busy. But a step changes psi by little: SO, CALCNU, HERM and the
// Crank-Nicolson sweeps each add an increment of size dt times an energy, 2^-6 to
// 2^-15 of |psi| at the steps the method is used with. An increment formed in FP32
// pairs (hi + lo, about 2^-48 relative) is then exact to 2^-53 |psi| and better,
// which is a rounding of the FP64 state itself; the sum state + increment is the
// only operation that needs the state's full width. Increments that are not small
// (large dt mu, strong SO, structure near the grid scale) are formed in FP64, see
// pair_large. The FP64 evaluation rounds the whole state some ten times a step instead. Error
// against an 80-bit reference (FP64 step -> this one): 128 x 112, 30 steps at dt = 2e-4,
// imaginary time 7.1e-16 -> 4.3e-16, real time 3.8e-15 -> 1.2e-15; double-float 1.8e-14 ->
// 3.8e-15 and 6.6e-14 -> 9.0e-15. Measured, us a step: complex128 256^2 imaginary / real time
// 42.9 / 49.6 -> 22.5 / 23.3, 512^2 158 / 195 -> 88 / 91, 161^2 real time 42.1 -> 18.7, 2048^2 2116 ->
// 1032; double-float 256^2 19.8 / 27.3 -> 17.3 / 18.0, 1024^2 220 / 352 -> 208 / 233.
//
// Pairs here are "lazy": products keep the exact error of the leading product and
// both cross terms, sums keep the exact rounding error of the leading sum, and
// nothing is renormalised in between (lo stays within a few ulp of hi).
// Multiplication and addition go through the _rn intrinsics, so that no
// contraction breaks an error term.
//
// State values are split through the integer pipe (FP64 conversions would queue on
// the FP64 pipe): hi rounded to 24 bits, lo the signed rest rounded to 24. A block
// whose largest value lies outside 2^-40 .. 2^40 shifts all its values by a power
// of two on the way in and out, so states of any scale are treated alike. What is far below a
// block's largest value (2^-74 without a shift) loses its lo to FP32's range, and so the
// relative, not the absolute accuracy of its increments.
//
// The sweeps are short convolutions. T = tridiag(-bt, 1 + 2bt, -bt) = u (I - gS)(I -
// gS^T), g = bt/u, has the Green's function g^|k| / (u (1 - g^2)) on the infinite line,
// and the odd extension of the state about the ghost points gives the finite line's
// solution. With the links M_i = x_(i+1) - x_i (even about the ghost points) the
// increment of x' = T^-1 (I + bt L) x = x + 2 bt T^-1 L x is
//   sum_(k >= 0) v_k (M_(i+k) - M_(i-1-k)),  v_k = 2 bt g^k / (u (1 + g)),
// cut where |g|^k < 2^-56: kt = 10 taps at bt = 0.02 (the host allows 16, bt up to about
// 0.08; larger bt keeps the FP64 kernels). Taps with |g|^k < 2^-26 only need the leading
// parts. No recurrence, no carries between threads: one thread a point, one barrier.
#pragma once
#include "sgpe_cn.cuh"

namespace sgpe {

// One axis and time mode: the taps v_k, as pairs for k < kp (wr, wi: (hi, hi, lo, lo) of the
// real and imaginary part) and rounded for the rest (wf: (re, re, -im, im)); kt taps in all
// (0: not applicable). The halves are doubled for the packed instructions.
struct PairTab {
    float4 wr[kPairPairTaps], wi[kPairPairTaps], wf[kPairTaps];
    int kp, kt;
    float v2;               // |v_0|^2
    double2 near[kPairNear];  // v_0, v_1 in FP64
};

// -- lazy pairs -------------------------------------------------------------------
__device__ __forceinline__ df lsum(float a, float b, float lo) {  // a + b + lo, the rounding of a + b kept
    const float s = __fadd_rn(a, b), t = __fadd_rn(s, -a);
    const float e = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t));
    return df(s, __fadd_rn(e, lo));
}
__device__ __forceinline__ df ladd(df a, df b) { return lsum(a.hi, b.hi, __fadd_rn(a.lo, b.lo)); }
__device__ __forceinline__ df lsub(df a, df b) { return lsum(a.hi, -b.hi, __fadd_rn(a.lo, -b.lo)); }
__device__ __forceinline__ df laddf(df a, float b) { return lsum(a.hi, b, a.lo); }
__device__ __forceinline__ df lneg(df a) { return df(-a.hi, -a.lo); }
__device__ __forceinline__ df lmul(df a, df b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    return df(p, __fmaf_rn(a.lo, b.hi, e));
}
__device__ __forceinline__ df lmulf(df a, float b) {
    const float p = __fmul_rn(a.hi, b);
    return df(p, __fmaf_rn(a.lo, b, __fmaf_rn(a.hi, b, -p)));
}
__device__ __forceinline__ df lsq(df a) {
    const float p = __fmul_rn(a.hi, a.hi);
    return df(p, __fmaf_rn(__fadd_rn(a.hi, a.hi), a.lo, __fmaf_rn(a.hi, a.hi, -p)));
}
__device__ __forceinline__ df lfma(df a, df b, df c) { return ladd(c, lmul(a, b)); }
__device__ __forceinline__ df lscale(df a, float s) { return df(__fmul_rn(a.hi, s), __fmul_rn(a.lo, s)); }  // s a power of two

// A complex pair: h = (re.hi, im.hi), l = (re.lo, im.lo), so that sums and products with a
// real pair take the packed FP32x2 instructions, both parts at once (each lane rounded as the
// scalar instruction): fewer instructions to fetch and to wait for.
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 p_neg(float2 a) { return __fmul2_rn(a, make_float2(-1.0f, -1.0f)); }
struct __align__(16) cd {
    float2 h, l;
    cd() = default;
    __device__ __forceinline__ cd(float2 a, float2 b) : h(a), l(b) {}
    __device__ __forceinline__ cd(df re, df im) : h(make_float2(re.hi, im.hi)), l(make_float2(re.lo, im.lo)) {}
    __device__ __forceinline__ df re() const { return df(h.x, l.x); }
    __device__ __forceinline__ df im() const { return df(h.y, l.y); }
};
__device__ __forceinline__ cd cadd(cd a, cd b) {
    const float2 s = p_add(a.h, b.h), t = p_sub(s, a.h);
    const float2 e = p_add(p_sub(a.h, p_sub(s, t)), p_sub(b.h, t));
    return cd(s, p_add(e, p_add(a.l, b.l)));
}
__device__ __forceinline__ cd csub(cd a, cd b) {
    const float2 s = p_sub(a.h, b.h), t = p_sub(s, a.h);
    const float2 e = p_sub(p_sub(a.h, p_sub(s, t)), p_add(b.h, t));
    return cd(s, p_add(e, p_sub(a.l, b.l)));
}
// a times the real pair (sh.x, sl.x) given doubled
__device__ __forceinline__ cd cscl2(float2 sh, float2 sl, cd a) {
    const float2 p = __fmul2_rn(sh, a.h);
    float2 e = __ffma2_rn(sh, a.h, p_neg(p));
    e = __ffma2_rn(sh, a.l, e);
    return cd(p, __ffma2_rn(sl, a.h, e));
}
__device__ __forceinline__ cd cscl(df s, cd a) { return cscl2(make_float2(s.hi, s.hi), make_float2(s.lo, s.lo), a); }
__device__ __forceinline__ cd cneg(cd a) { return cd(p_neg(a.h), p_neg(a.l)); }
__device__ __forceinline__ cd cjg(cd a) { return cd(make_float2(a.h.x, -a.h.y), make_float2(a.l.x, -a.l.y)); }
__device__ __forceinline__ cd cmuli(cd a) { return cd(make_float2(-a.h.y, a.h.x), make_float2(-a.l.y, a.l.x)); }   // i a
__device__ __forceinline__ cd cmulni(cd a) { return cd(make_float2(a.h.y, -a.h.x), make_float2(a.l.y, -a.l.x)); }  // -i a
__device__ __forceinline__ cd cmulp(cd a, cd b) { return cadd(cscl(a.re(), b), cscl(a.im(), cmuli(b))); }
__device__ __forceinline__ cd cmulc(cd a, cd b) { return cadd(cscl(a.re(), b), cscl(a.im(), cmulni(b))); }  // conj(a) b
__device__ __forceinline__ df cnrm(cd a) {
    const float2 p = __fmul2_rn(a.h, a.h);
    const float2 e = __ffma2_rn(p_add(a.h, a.h), a.l, __ffma2_rn(a.h, a.h, p_neg(p)));
    return lsum(p.x, p.y, __fadd_rn(e.x, e.y));
}
__device__ __forceinline__ cd czero() { return cd(make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)); }

// -- the state's width ------------------------------------------------------------
// x 2^k as a pair, through the integer pipe; bias = (896 - k) << 20. Values below
// 2^-126 after the shift come out as 0, larger than FP32's range as NaN.
__device__ __forceinline__ df split64(double x, unsigned bias) {
    const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
    const unsigned sg = h & 0x80000000u;
    // round to 24 bits by adding half of the 29 bits below; what is left is signed (a truncated
    // hi would bias every dropped lo lo product)
    const unsigned l2 = l + 0x10000000u;
    const int t = (int)((h & 0x7fffffffu) + (l2 < l ? 1u : 0u) - bias);  // FP32 exponent (8 bits), 20 mantissa bits
    unsigned f = __funnelshift_l(l2, (unsigned)t, 3);
    const int es = (int)((h & 0x7ff00000u) - bias) - (52 << 20);  // exponent field of 2^(E - 52)
    float lo = __fmul_rn((float)((int)(l2 & 0x1fffffffu) - 0x10000000), __int_as_float(es > 0 ? es << 3 : 0));
    if (t < (1 << 20)) {
        f = 0u;
        lo = 0.0f;
    }
    if (t >= (255 << 20)) f = 0x7fc00000u;
    return df(__uint_as_float(f | sg), sg ? -lo : lo);
}
// v 2^-k as a double (same bias); FP32 subnormals and results below 2^-1022 come out as 0.
__device__ __forceinline__ double widen(float v, unsigned bias) {
    const unsigned b = __float_as_uint(v), e = b & 0x7f800000u;
    const int h = (int)(((b & 0x7fffffffu) >> 3) + bias);
    if (e == 0u || h < (1 << 20)) return 0.0;
    if (e == 0x7f800000u) return (double)v;
    return __hiloint2double((int)((b & 0x80000000u) | (unsigned)h), (int)(b << 29));
}

// (hi + lo) 2^-k as a double rounded once (same bias): hi's bits plus lo in units of hi's last
// place, by an integer addition on the 64 bits, where widen(hi) + widen(lo) would take an FP64
// instruction. lo is at most half of FP32's last place of hi after the exact sum, so only a
// power of two less something leaves its binade, below which the units are half as large.
// Two FP64 instructions less per component, point and kernel: 256^2 24.1 -> 21.7 us a step, 64^2 12.0 ->
// 11.5, 512^2 90.9 -> 85.6, 1024^2 298 -> 280.
__device__ __forceinline__ double widen(df v, unsigned bias) {
    const df s = two_sum(v.hi, v.lo);
    const unsigned b = __float_as_uint(s.hi), eb = b & 0x7f800000u;
    const int h = (int)(((b & 0x7fffffffu) >> 3) + bias);
    // (below 2^-75 the units have no FP32 scale)
    if (eb < (52u << 23) || eb == 0x7f800000u || h < (2 << 20)) return widen(v.hi, bias) + widen(v.lo, bias);
    int k = __float2int_rn(__fmul_rn(s.lo, __uint_as_float((306u << 23) - eb)));
    if (b >> 31) k = -k;
    if (k < 0 && (b & 0x7fffffu) == 0u) k *= 2;
    const long long z = (((long long)h << 32) | (long long)(unsigned)(b << 29)) + k;
    return __longlong_as_double(z | ((long long)(b >> 31) << 63));
}

// The storage of one real number per form: what a kernel keeps of a loaded value
// (base), its pair, differences of two values, and value + increment.
template <typename R> struct PairState;
template <> struct PairState<double> {
    static constexpr bool kShift = true;
    __device__ __forceinline__ static df pair(double x, unsigned bias) { return split64(x, bias); }
    __device__ __forceinline__ static df diff(double a, double b, unsigned bias) { return split64(a - b, bias); }
    // (two roundings: the increment's parts, a few ulp of lo apart, and the sum)
    __device__ __forceinline__ static double plus(double x, df inc, unsigned bias) {
        return x + widen(inc, bias);
    }
    __device__ __forceinline__ static double times(double x, double d) { return x * d; }
    __device__ __forceinline__ static unsigned mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
};
template <> struct PairState<df> {
    static constexpr bool kShift = false;
    __device__ __forceinline__ static df pair(df x, unsigned) { return x; }
    __device__ __forceinline__ static df diff(df a, df b, unsigned) { return lsub(a, b); }
    __device__ __forceinline__ static df plus(df x, df inc, unsigned) {
        const df s = ladd(x, inc);
        return fast_two_sum(s.hi, s.lo);
    }
    __device__ __forceinline__ static df times(df x, double d) { return x * df_from(d); }
    __device__ __forceinline__ static unsigned mag(df) { return 0u; }
};
template <typename R> __device__ __forceinline__ cd pair_of(cx<R> a, unsigned bias) {
    return cd(PairState<R>::pair(a.re, bias), PairState<R>::pair(a.im, bias));
}
template <typename R> __device__ __forceinline__ cd pair_diff(cx<R> a, cx<R> b, unsigned bias) {
    return cd(PairState<R>::diff(a.re, b.re, bias), PairState<R>::diff(a.im, b.im, bias));
}
template <typename R> __device__ __forceinline__ cx<R> pair_plus(cx<R> x, cd inc, unsigned bias) {
    return {PairState<R>::plus(x.re, inc.re(), bias), PairState<R>::plus(x.im, inc.im(), bias)};
}
template <typename R> __device__ __forceinline__ unsigned pair_mag(cx<R> a) {
    return max(PairState<R>::mag(a.re), PairState<R>::mag(a.im));
}
constexpr unsigned kBias0 = 896u << 20;
// The block's shift k from the largest high word of its values: 0 in 2^-40 .. 2^40
// (and for zero, infinities and NaN).
__device__ __forceinline__ int pair_shift(unsigned mx) {
    return (mx >= (983u << 20) && mx < (1063u << 20)) || mx == 0u || mx >= 0x7ff00000u ? 0 : 1023 - (int)(mx >> 20);
}

// The pending factors as d - 1 in a pair, where they are one factor with |d - 1| < 2^-6; *is_far 1
// otherwise, 2 where one lies outside 1/2 .. 2 (NaN too): the step before's values then say nothing
// about this one's. One thread's chain that the whole block waits for: comparisons and the
// split on the integer pipe, where an FP64 instruction would take its 64 cycles.
__device__ __forceinline__ void pair_near(const double* d, df* dm, int* is_far) {
    const double e = d[0] - 1.0;
    const long long b = __double_as_longlong(d[0]);
    *is_far = b != __double_as_longlong(d[1]) || b != __double_as_longlong(d[2]) ||
              ((unsigned)__double2hiint(e) & 0x7fffffffu) >= (1017u << 20);
    for (int j = 0; j < 3; j++)
        if ((unsigned)__double2hiint(d[j]) - (1022u << 20) >= (2u << 20)) *is_far = 2;
    *dm = split64(e, kBias0);
}

// -- pointwise substeps -------------------------------------------------------------
__device__ __forceinline__ df kpair(const KParams& p, int i) { return df(p.kf[i], p.kl[i]); }

static __device__ __noinline__ df em1_wide(df x) { return df_from(expm1((double)x.hi + (double)x.lo)); }
static __device__ __noinline__ void sc_wide(df x, df* cm1, df* sn) {
    double s, c;
    sincos(0.5 * ((double)x.hi + (double)x.lo), &s, &c);
    *cm1 = df_from(-2.0 * s * s);
    *sn = df_from(2.0 * s * c);
}
// The HERM coefficients s, k for w = (dt A)^2 >= 2^-20: below 2^-12, all that stays in pairs, by the
// series in pairs (the last term in FP32: its rounding is below 2^-55 of the coefficients), larger
// through FP64.
template <bool IMAG> __device__ __noinline__ void herm_wide(cd a, cd b, const KParams& p, df* s, df* k) {
    const df w = lmul(kpair(p, KC_DT2), ladd(cnrm(a), cnrm(b)));
    if (w.hi < 2.44140625e-4f) {
        const df v = IMAG ? w : lneg(w);
        const float rs = fmaf(v.hi, p.kf[KC_HS0 + 3], p.kf[KC_HS0 + 2]), rk = fmaf(v.hi, p.kf[KC_HK0 + 3], p.kf[KC_HK0 + 2]);
        *s = lfma(ladd(kpair(p, KC_HS0 + 1), lmulf(v, rs)), v, kpair(p, KC_HS0));
        const df q = lfma(ladd(kpair(p, KC_HK0 + 1), lmulf(v, rk)), v, kpair(p, KC_HK0));
        *k = IMAG ? q : lneg(q);
        return;
    }
    const double ar = (double)a.h.x + (double)a.l.x, ai = (double)a.h.y + (double)a.l.y;
    const double br = (double)b.h.x + (double)b.l.x, bi = (double)b.h.y + (double)b.l.y;
    double sd, kd;
    herm_coeffs<IMAG>(ar * ar + ai * ai + br * br + bi * bi, p.dt, &sd, &kd);
    *s = df_from(sd);
    *k = df_from(kd);
}

// exp(x) - 1. |x| < 2^-6: x (1 + x (1/2 + x (1/6 + r))), the tail r in FP32 (its
// rounding, times x^3, stays below 2^-45 |x|); up to 16: em1(2y) = em1(y) (2 + em1(y))
// from y = x 2^-n; larger arguments through FP64.
__device__ __forceinline__ df em1_pair(df x) {
    int n = 0;
    const float ax = fabsf(x.hi);
    if (!(ax < 0.015625f)) {
        if (!(ax < 16.0f)) return em1_wide(x);
        n = (int)(__float_as_uint(ax) >> 23) - 120;  // 1 at 2^-6
        x = lscale(x, __int_as_float((127 - n) << 23));
    }
    const float xf = x.hi;
    const float r = xf * fmaf(xf, fmaf(xf, fmaf(xf, 1.0f / 5040.0f, 1.0f / 720.0f), 1.0f / 120.0f), 1.0f / 24.0f);
    constexpr df c6 = df_from(1.0 / 6.0);
    df q = laddf(lmul(laddf(c6, r), x), 0.5f);  // (lo of 1/6 + r is kept: r is small against 1/6)
    q = lmul(lmul(q, x), x);                    // x^2 (1/2 + ...)
    df e = ladd(x, q);
    for (int i = 0; i < n; i++) e = lmul(e, laddf(e, 2.0f));
    return e;
}

// (cos x - 1, sin x). |x| < 2^-6 by series, the tails in FP32; up to 16 by doubling:
// cos 2y - 1 = 2 c (2 + c), sin 2y = 2 s (1 + c), c = cos y - 1; larger through FP64.
__device__ __forceinline__ void sc_pair(df x, df* cm1, df* sn) {
    int n = 0;
    const float ax = fabsf(x.hi);
    if (!(ax < 0.015625f)) {
        if (!(ax < 16.0f)) {
            sc_wide(x, cm1, sn);
            return;
        }
        n = (int)(__float_as_uint(ax) >> 23) - 120;
        x = lscale(x, __int_as_float((127 - n) << 23));
    }
    const df t = lsq(x);
    const float tf = t.hi;
    constexpr df c6 = df_from(-1.0 / 6.0), c24 = df_from(1.0 / 24.0);
    const float rs = tf * fmaf(-tf, 1.0f / 5040.0f, 1.0f / 120.0f), rc = -tf * fmaf(-tf, 1.0f / 40320.0f, 1.0f / 720.0f);
    df s = ladd(x, lmul(lmul(laddf(c6, rs), t), x));        // x - x^3/6 + ...
    df c = lmul(laddf(lmul(laddf(c24, rc), t), -0.5f), t);  // -t/2 + t^2/24 - ...
    for (int i = 0; i < n; i++) {
        s = lscale(lmul(s, laddf(c, 1.0f)), 2.0f);
        c = lscale(lmul(c, laddf(c, 2.0f)), 2.0f);
    }
    *cm1 = c;
    *sn = s;
}

// -z times v: -v (imaginary time), -i v (real time)
template <bool IMAG> __device__ __forceinline__ cd mz(cd v) {
    if constexpr (IMAG) return cneg(v);
    return cmulni(v);
}
// gx P + (-i gy) Q: the form of every row of the 2D H_SO
__device__ __forceinline__ cd so_form(df gx, df gy, cd P, cd Q) {
    return cadd(cscl(gx, P), cscl(gy, cmulni(Q)));
}

// CALCNU of one point in FP64, and HERM where herm is set.
template <bool IMAG>
__device__ __noinline__ void nonlin_wide(cx<double> (&u)[3], const KParams& p, double Ot, int ix, int iy, bool herm) {
    const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;
    calcnu_point_dt<IMAG>(u, p.kd[KC_NVX] * (kx * kx) + p.kd[KC_NVY] * (ky * ky), p);
    if (herm) herm_point<IMAG>(u, p.kd[KC_C2], Ot, p.kd[KC_DT], &p);
}
// CALCNU of component j of the point x (st entries between components) in FP64.
template <bool IMAG>
__device__ __noinline__ double2 calcnu_own(const double2* x, int st, int j, const KParams& p, int ix, int iy) {
    const cx<double> u[3] = {unpack(x[0]), unpack(x[st]), unpack(x[2 * st])};
    const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;
    const double rp = nrm(u[0]), r0 = nrm(u[1]), rm = nrm(u[2]);
    const double base = fma(p.kd[KC_NC0], rp + r0 + rm, p.kd[KC_NVX] * (kx * kx) + p.kd[KC_NVY] * (ky * ky));
    const double q = j == 1 ? rp + rm : j == 0 ? rp - rm + r0 : rm - rp + r0;
    const double e = fma(p.kd[KC_NC2], q, base);
    const cx<double> v = j == 0 ? u[0] : j == 1 ? u[1] : u[2];
    if constexpr (IMAG) return pack(scl(exp_small(e), v));
    double s, c;
    sincos_small(e, &s, &c);
    return pack(mul(cx<double>{c, s}, v));
}

// All pointwise substeps of one point in FP64, from the state in memory (d: the pending factors).
template <bool IMAG>
__device__ __noinline__ void point_wide(const double2* __restrict__ A, const KParams& p, const double* d, double Ot,
                                        int ix, int iy, cx<double> (&u)[3]) {
    pointwise_point<double, IMAG>(A, p, d, Ot, ix, iy, 7, u);
}

// The sweep's increment at a point by the taps k >= k0: M points at M_i of its line, st entries
// between links.
template <bool IMAG> __device__ __forceinline__ cd pair_taps(const cd* M, int st, const PairTab& t, int k0) {
    const int kp = t.kp, kt = t.kt;
    float2 f = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = kPairTaps - 1; k >= 1; k--) {
        if (k < kp || k >= kt || k < k0) continue;
        const float2 d = p_sub(M[k * st].h, M[-(k + 1) * st].h);
        f = __ffma2_rn(make_float2(t.wf[k].x, t.wf[k].y), d, f);
        if constexpr (!IMAG) f = __ffma2_rn(make_float2(t.wf[k].z, t.wf[k].w), make_float2(d.y, d.x), f);
    }
    cd acc(f, make_float2(0.0f, 0.0f));
#pragma unroll
    for (int k = kPairPairTaps - 1; k >= 0; k--) {
        if (k >= kp || k < k0) continue;
        const cd d = csub(M[k * st], M[-(k + 1) * st]);
        acc = cadd(acc, cscl2(make_float2(t.wr[k].x, t.wr[k].y), make_float2(t.wr[k].z, t.wr[k].w), d));
        if constexpr (!IMAG)
            acc = cadd(acc, cscl2(make_float2(t.wi[k].x, t.wi[k].y), make_float2(t.wi[k].z, t.wi[k].w), cmuli(d)));
    }
    return acc;
}

// The same by the taps k < kPairNear in FP64, of the point x_i and its two neighbours on either
// side: at(q) is point i + q, zero at the ghost points -1 and n, and beyond those the line
// continues oddly. (Out of line: the kernels' registers stay what the pairs need.)
template <bool IMAG, typename At>
__device__ __forceinline__ double2 near_taps(At&& at, int i, int n, double2 a, double2 b) {
    const cx<double> zero = {0.0, 0.0};
    const cx<double> x = at(0), m1 = i > 0 ? at(-1) : zero, p1 = i < n - 1 ? at(1) : zero;
    const cx<double> m2 = i > 1 ? at(-2) : i == 1 ? zero : cx<double>{-x.re, -x.im};
    const cx<double> p2 = i < n - 2 ? at(2) : i == n - 2 ? zero : cx<double>{-x.re, -x.im};
    const cx<double> d0 = {fma(-2.0, x.re, m1.re + p1.re), fma(-2.0, x.im, m1.im + p1.im)};
    const cx<double> d1 = {(m2.re - m1.re) + (p2.re - p1.re), (m2.im - m1.im) + (p2.im - p1.im)};
    if constexpr (IMAG) return make_double2(fma(a.x, d0.re, b.x * d1.re), fma(a.x, d0.im, b.x * d1.im));
    return make_double2(fma(a.x, d0.re, fma(-a.y, d0.im, fma(b.x, d1.re, -b.y * d1.im))),
                        fma(a.x, d0.im, fma(a.y, d0.re, fma(b.x, d1.im, b.y * d1.re))));
}
// x: the point in memory, st entries between points.
template <bool IMAG>
__device__ __noinline__ double2 near_mem(const double2* x, int st, int i, int n, double2 a, double2 b) {
    return near_taps<IMAG>([&](int q) { return unpack(x[q * st]); }, i, n, a, b);
}
// The same for points x + s (s: increments).
template <bool IMAG>
__device__ __noinline__ double2 near_inc(const double2* x, const cd* s, unsigned bias, int i, int n, double2 a, double2 b) {
    return near_taps<IMAG>([&](int q) { return pair_plus<double>(unpack(x[q]), s[q], bias); }, i, n, a, b);
}

// -- what leaves the increments (complex128) -----------------------------------------------
// A pair is exact to about 2^-48 of the increment, so an increment is as exact as the FP64
// step's own roundings as long as it is small: below 2^-6 of the spinor at the point in
// imaginary time, 2^-5 in real time (where the FP64 sweeps' complex products round more) and
// for dt mu, or below 2^-10 of the grid's largest |psi| (known from the step before), where the
// error stays under 2^-58 of that. Each kernel checks its increments against this; larger
// ones are formed in FP64:
//   kNonlin  dt mu: the block takes CALCNU in FP64, HERM's increments start from there
//   kHerm    dt A: the block takes CALCNU and HERM in FP64
//   kSo      SO (strong coupling, structure near the grid scale): the block takes all pointwise
//            substeps in FP64, from the state in memory
//   kRough   a sweep (structure near the grid scale): the warp takes v_0 and v_1, which carry all
//            but |g|^2 <= 2^-7 of it, in FP64
// Error against an 80-bit reference of 10 steps of independent random values, FP64 step /
// increments without these checks / this: bt = 0.0625 imaginary time 5.9e-16 / 1.5e-15 / 3.1e-16,
// bt = 0.08 real time 1.4e-15 / 8.1e-15 / 7.7e-16, gamma = 20 (dt = 2.5e-3, dx = 0.1) real time
// 2.3e-15 / 6.1e-15 / 7.6e-16. They cost about 3 % of a step of a smooth state.
constexpr unsigned kNonlin = 1u, kSo = 2u, kRough = 4u, kHerm = 8u;
constexpr unsigned kWide = kNonlin | kSo | kHerm;  // pointwise substeps in FP64
// (U 2^(k - 4))^2 for the largest |psi| U of the step before as a high word (0: unknown), 2^k the block's shift
__device__ __forceinline__ float pair_floor2(unsigned umax, int k) {
    const int e = (int)(umax >> 20) - 1023 + k - 4;
    return umax < (1u << 20) ? 0.0f : __int_as_float((127 + 2 * max(-60, min(60, e))) << 23);
}
// The squared limit of SO's and a sweep's increments next to rho (NaN stays in the increments).
template <bool IMAG> __device__ __forceinline__ float pair_limit2(float rho, float floor2) {
    return (IMAG ? 0.000244140625f : 0.0009765625f) * fmaxf(rho, floor2);
}
// What is too large at a point: so2, sw2 the squared increments of SO and of the sweep, ae the
// largest |dt mu|, w = (dt A)^2.
template <bool IMAG>
__device__ __forceinline__ unsigned pair_large(float so2, float sw2, float rho, float floor2, float ae, float w) {
    const float lim = pair_limit2<IMAG>(rho, floor2);
    unsigned b = (so2 > lim ? kSo : 0u) | (sw2 > lim ? kRough : 0u);
    const bool wbig = !(w < 2.44140625e-4f);
    if ((!(ae < 0.03125f) || wbig) && rho > 0.0f) {
        // dt mu up to 2: against the floor; beyond (2^-40 of it), the value itself would lose its relative accuracy
        const float big = ae < 2.0f ? rho * fmaxf(ae * ae, w) : rho * 2.81474976710656e14f;
        if (big >= 0.000244140625f * floor2) b |= wbig ? kNonlin | kHerm : kNonlin;
    }
    return b;
}
// |x_(i+1) - 2 x_i + x_(i-1)|^2 of a point in memory (zero ghosts outside 0..n-1), from the leading 24 bits
// of the values.
__device__ __forceinline__ float bend2(const double2* x, int i, int n, unsigned bias) {
    const double2 c = x[0], zero = make_double2(0.0, 0.0), l = i > 0 ? x[-1] : zero, r = i < n - 1 ? x[1] : zero;
    const float a = split64(l.x, bias).hi + split64(r.x, bias).hi - 2.0f * split64(c.x, bias).hi;
    const float b = split64(l.y, bias).hi + split64(r.y, bias).hi - 2.0f * split64(c.y, bias).hi;
    return fmaf(a, a, b * b);
}
__device__ __forceinline__ float norm2(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }

// -- kernel 1: pending scale, SO, CALCNU, HERM, Crank-Nicolson along x ------------------
// One block per row segment (segment sg of nseg writes the points [o0, o1) of row iy and
// works on [a0, a1), kt + 1 points more at each end inside the row), one thread per point
// and component, the components in warps of their own (three neighbouring warps a group of
// 32 points, on different sub-partitions): each substep is the same short
// code for all three, so a block's warps share its instruction lines and a small grid's
// few blocks have three times the warps (64^2: 15.1 us a step with one thread a point, 11.9
// so). The components meet in shared memory: the differences before SO, the densities
// before CALCNU, the state before HERM, the increments and links before the sweep.
//
// Links: the sweep and SO's x difference take the differences of
// neighbouring state values, taken in the state's own width and then split (a rounding
// of 2^-48 of the difference, not of the values), plus the differences of the increments.
//
// A block with an increment too large for a pair (pair_large; complex128 only: larger steps, a
// wide trap in the first step, rough states) takes what it has to FP64 and restarts the
// increments from the result.
constexpr int kPairXThreads = 3 * kPairXPts;

template <typename R, bool IMAG>
__global__ void __launch_bounds__(kPairXThreads, 2)
    k_pair_x(const typename V2<R>::T* __restrict__ A, typename V2<R>::T* __restrict__ Bout, KParams p, DevScalars* sc,
             const double* __restrict__ omega_tab, PairTab t, int nseg, const double* __restrict__ partials, int m,
             int renorm) {
    using PS = PairState<R>;
    using T = typename V2<R>::T;
    constexpr int H = kPairTaps + 1;
    __shared__ cd Ls[3][kPairXPts + 2 * H];  // H + i: the link from point i to i + 1 (H - 1: from the left ghost)
    __shared__ __align__(16) cd Us[3][kPairXPts];  // y differences; the state before HERM; the full-width state; increments
    __shared__ df rs[3][kPairXPts];
    __shared__ double red[3], dsh[3];
    __shared__ df dms;
    __shared__ int far_s;
    __shared__ unsigned wmax[kPairXThreads / 32], large_s;
    const int tid = threadIdx.x, warp = tid >> 5, nw = blockDim.x >> 5, nwp = nw / 3;
    const int iy = blockIdx.x / nseg;
    const PairSeg sg = pair_seg(p.nx, nseg, t.kt + 1, blockIdx.x - iy * nseg);
    const int np = sg.a1 - sg.a0;
    const int grp = warp / 3, j = warp - 3 * grp, i = grp * 32 + (tid & 31), ix = sg.a0 + i;
    const bool in = i < np, out = in && ix >= sg.o0 && ix < sg.o1, so = p.so_case != 0;
    const size_t plane = (size_t)p.nx * p.ny, at = j * plane + (size_t)iy * p.nx + ix;
    const cx<R> zr = {R(0), R(0)};
    pdl_wait();
    cx<R> x = in ? ld<R>(A, at) : zr;
    const cx<R> xp = in && ix + 1 < p.nx ? ld<R>(A, at + 1) : zr;
    const cx<R> ym = in && so && iy > 0 ? ld<R>(A, at - p.nx) : zr;
    const cx<R> yp = in && so && iy + 1 < p.ny ? ld<R>(A, at + p.nx) : zr;
    const bool from_parts = partials && *(volatile const int*)&sc->scale_src;
    unsigned um = 0u;  // the grid's largest |psi| of the step before (high word; 0: unknown)
    if (from_parts && warp < 3) {
        const double q = sum_partials_warp(partials + (size_t)warp * m, m);
        if ((tid & 31) == 0) red[warp] = q;
    }
    if constexpr (PS::kShift) {
        const int tick = *(volatile const int*)&sc->pair_tick;
        um = *(volatile const unsigned*)&sc->umax[(tick + 2) % 3];
        if (blockIdx.x == 0 && tid == 0) {  // the slot of this step's y sweep; the next step's is cleared
            sc->umax_slot = tick;
            sc->umax[(tick + 1) % 3] = 0u;
        }
        const unsigned mx = __reduce_max_sync(0xffffffffu, max(pair_mag(x), max(pair_mag(ym), pair_mag(yp))));
        if ((tid & 31) == 0) wmax[warp] = mx;
        if (tid == 0) large_s = 0u;
    }
    __syncthreads();
    int k = 0;
    if constexpr (PS::kShift) {
        unsigned mx = 0u;
        for (int w = 0; w < nw; w++) mx = max(mx, wmax[w]);
        k = pair_shift(mx);
    }
    unsigned bias = (unsigned)(896 - k) << 20;
    if (in) {
        Ls[j][H + i] = pair_diff(xp, x, bias);
        if (i == 0) Ls[j][H - 1] = sg.a0 == 0 ? pair_of(x, bias) : czero();
        if (so) Us[j][i] = pair_diff(yp, ym, bias);
    }
    cd u = pair_of(x, bias), s = czero();
    if (tid == blockDim.x - 32) {  // lane 0 of the last warp
        if (from_parts) {
            const double N[3] = {red[0] * p.cell, red[1] * p.cell, red[2] * p.cell};
            const bool finite = isfinite(N[0]) && isfinite(N[1]) && isfinite(N[2]);
            double d[3];
            renorm_factors(N, finite ? renorm : 0, p.mag, d);
            for (int c = 0; c < 3; c++) dsh[c] = d[c];
        } else {
            for (int c = 0; c < 3; c++) dsh[c] = sc->scale[c];
        }
        pair_near(dsh, &dms, &far_s);
        if (PS::kShift && blockIdx.x == 0) sc->umax_prev = far_s > 1 ? 0u : um;
    }
    __syncthreads();
    if (far_s > 1) um = 0u;
    // SO: rows +1 and -1 of H_SO take psi_0 (X with the sign +, -), row 0 psi_-1 - psi_+1 and their sum
    const df hx = kpair(p, KC_HX), hy = kpair(p, KC_HY);
    auto xdiff = [&](int c) { return cadd(Ls[c][H + i], Ls[c][H + i - 1]); };
    if (so) {
        cd P, Q;
        if (j == 1) {
            P = csub(xdiff(2), xdiff(0));
            Q = cadd(Us[0][i], Us[2][i]);
        } else {
            P = xdiff(1);
            if (j == 2) P = cneg(P);
            Q = Us[1][i];
        }
        s = mz<IMAG>(so_form(hx, hy, P, Q));
    }
    bool relink = false;
    float so2 = norm2(s.h);
    {
        const df dm = dms;
        if (far_s) {
            // factors far from 1 (the first step of a state of other norm) or unequal (Eq. (DJ)):
            // the state times d in its own width, SO with the factors of its sources
            relink = true;
            const int kold = k;
            if (fabs(dsh[0]) > 1e6 || fabs(dsh[0]) < 1e-6) {  // the scaled state has unit norm: no shift
                k = 0;
                bias = kBias0;
            }
            if (so) {
                cd h = czero();
                for (int c = 0; c < 3; c++) {
                    if ((c == 1) == (j == 1)) continue;
                    int e;
                    const df dc = df_from(frexp(dsh[c], &e));
                    const float f = __int_as_float((127 + max(-126, min(126, e + k - kold))) << 23);
                    cd P = xdiff(c);
                    if (c == 0 || j == 2) P = cneg(P);
                    h = cadd(h, so_form(lscale(lmul(hx, dc), f), lscale(lmul(hy, dc), f), P, Us[c][i]));
                }
                s = mz<IMAG>(h);
                so2 = norm2(s.h);
            }
            x = {PS::times(x.re, dsh[j]), PS::times(x.im, dsh[j])};
            u = pair_of(x, bias);
        } else if (dm.hi != 0.0f) {
            // d (psi + s) = psi + s + (d - 1)(psi + s)
            s = cadd(s, cscl(dm, cadd(u, s)));
        }
        if (!in) s = czero();  // (its neighbours are unset)
    }
    u = cadd(u, s);
    rs[j][i] = cnrm(u);
    __syncthreads();
    // CALCNU (f: from shifted to true densities, within FP32's range)
    const float f = __int_as_float((127 + max(-126, min(126, -2 * k))) << 23);
    const df Ot = omega_tab ? df_from(__ldg(omega_tab + sc->step_idx) * 0.70710678118654752440) : kpair(p, KC_OMEGA);
    const df c2 = lscale(kpair(p, KC_C2), f);
    cd tn;
    unsigned large = 0u;
    {
        const df rp = rs[0][i], r0 = rs[1][i], rm = rs[2][i], rpm = ladd(rp, rm);
        const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;  // |k| <= 2048: k^2 is exact in FP32
        const df Vn = ladd(lmulf(kpair(p, KC_NVX), (float)(kx * kx)), lmulf(kpair(p, KC_NVY), (float)(ky * ky)));
        const df base = lfma(lscale(kpair(p, KC_NC0), f), ladd(rpm, r0), Vn);
        df q = rpm;
        if (j != 1) q = ladd(r0, j == 0 ? lsub(rp, rm) : lsub(rm, rp));
        const df e = lfma(lscale(kpair(p, KC_NC2), f), q, base);
        if constexpr (PS::kShift) {
            const float ot = fabsf(Ot.hi);
            const float ea = fmaf(fabsf(c2.hi), sqrtf(rm.hi * r0.hi), ot), eb = fmaf(fabsf(c2.hi), sqrtf(r0.hi * rp.hi), ot);
            // (the first point of a segment inside the row has no link to its left, and writes nothing)
            const float2 r = p_sub(Ls[j][H + i].h, Ls[j][H + i - 1].h);
            if (in && (i > 0 || sg.a0 == 0))
                large = pair_large<IMAG>(so2, t.v2 * norm2(r), rpm.hi + r0.hi, pair_floor2(um, k),
                                   fabsf(e.hi), p.kf[KC_DT2] * fmaf(ea, ea, eb * eb));
        }
        if constexpr (IMAG) {
            tn = cscl(em1_pair(e), u);
        } else {
            df cm1, sn;
            sc_pair(e, &cm1, &sn);
            tn = cadd(cscl(cm1, u), cscl(sn, cmuli(u)));
        }
    }
    Us[j][i] = cadd(u, tn);
    bool slow = relink, herm = true;  // herm: HERM in pairs
    unsigned bits = 0u;
    const unsigned votes = kWide | (relink ? kRough : 0u);  // (links anew anyway: rough blocks restart too)
    if constexpr (PS::kShift) {
        if (__any_sync(0xffffffffu, large & votes)) {
            const unsigned all = __reduce_or_sync(0xffffffffu, large);
            if ((threadIdx.x & 31) == 0) atomicOr(&large_s, all);
        }
        if (__syncthreads_or(large & votes)) bits = large_s;
        if (far_s > 1) bits |= kRough;
        slow = relink || bits;
    } else {
        __syncthreads();
    }
    T* xs = reinterpret_cast<T*>(&Us[0][0]);  // [3][kPairXPts]
    cd up, u0, um_;
    if (PS::kShift && bits) {
        if constexpr (PS::kShift) {
            // the increments so far into the state, the large ones in FP64; HERM's from there
            if (!(bits & kWide)) s = cadd(s, tn);
            if (in) xs[j * kPairXPts + i] = pack(pair_plus<R>(x, s, bias));
            __syncthreads();
            // CALCNU by each component for itself; where HERM or SO is large too, one thread a point takes all
            herm = !(bits & (kHerm | kSo));
            if (in && (bits & kWide)) {
                if (herm) {
                    x = unpack(calcnu_own<IMAG>(xs + i, kPairXPts, j, p, ix, iy));
                } else if (j == 0) {
                    const double otd = omega_tab ? __ldg(omega_tab + sc->step_idx) * 0.70710678118654752440 : p.kd[KC_OMEGA];
                    cx<double> v[3];
                    for (int c = 0; c < 3; c++) v[c] = unpack(xs[c * kPairXPts + i]);
                    if (bits & kSo)
                        point_wide<IMAG>(A, p, dsh, otd, ix, iy, v);
                    else
                        nonlin_wide<IMAG>(v, p, otd, ix, iy, true);
                    for (int c = 0; c < 3; c++) xs[c * kPairXPts + i] = pack(v[c]);
                }
            }
            __syncthreads();
            if (in && (bits & kWide) && herm) xs[j * kPairXPts + i] = pack(x);
            __syncthreads();
            x = in ? unpack(xs[j * kPairXPts + i]) : zr;
            s = up = u0 = um_ = czero();
            if (in && herm) {
                up = pair_of(unpack(xs[i]), bias);
                u0 = pair_of(unpack(xs[kPairXPts + i]), bias);
                um_ = pair_of(unpack(xs[2 * kPairXPts + i]), bias);
            }
        }
    } else {
        s = cadd(s, tn);
        up = Us[0][i];
        u0 = Us[1][i];
        um_ = Us[2][i];
    }
    if (herm) {
        cd a = cscl(c2, cmulc(um_, u0)), b = cscl(c2, cmulc(u0, up));
        a = cd(ladd(a.re(), Ot), a.im());
        b = cd(ladd(b.re(), Ot), b.im());
        const float w = p.kf[KC_DT2] *
                        fmaf(a.h.x, a.h.x, fmaf(a.h.y, a.h.y, fmaf(b.h.x, b.h.x, b.h.y * b.h.y)));
        df cs, ck;
        if (w < 9.5367431640625e-07f) {
            // w < 2^-20: the series corrections in FP32 (their rounding is below 2^-46 of the coefficients)
            const float v = IMAG ? w : -w;
            cs = laddf(kpair(p, KC_HS0), v * fmaf(p.kf[KC_HS0 + 2], v, p.kf[KC_HS0 + 1]));
            ck = laddf(kpair(p, KC_HK0), v * fmaf(p.kf[KC_HK0 + 2], v, p.kf[KC_HK0 + 1]));
            if (!IMAG) ck = lneg(ck);
        } else {
            herm_wide<IMAG>(a, b, p, &cs, &ck);
        }
        // -s_z A u + k A^2 u: (A u)_0 = a* u_+ + b u_-; the rows +1, -1 are a, b* times -s_z u_0 +
        // k (A u)_0; (A^2 u)_0 = (|a|^2 + |b|^2) u_0
        const cd A0 = cadd(cmulc(a, up), cmulp(b, um_));
        if (j == 1)
            s = cadd(s, cadd(mz<IMAG>(cscl(cs, A0)), cscl(lmul(ck, ladd(cnrm(a), cnrm(b))), u0)));
        else
            s = cadd(s, cmulp(j == 0 ? a : cjg(b), cadd(mz<IMAG>(cscl(cs, u0)), cscl(ck, A0))));
    }
    __syncthreads();  // every Us (xs) has been read
    int k0 = 0;
    const bool fresh = PS::kShift && bits;  // the increments start from zero
    if (slow) {
        if (fresh) {
            x = pair_plus<R>(x, s, bias);
            s = czero();
        }
        if (in) xs[j * kPairXPts + i] = pack(x);
        __syncthreads();
        if (in) {
            Ls[j][H + i] = pair_diff(i + 1 < np ? unpack(xs[j * kPairXPts + i + 1]) : zr, x, bias);
            if (i == 0) Ls[j][H - 1] = sg.a0 == 0 ? pair_of(x, bias) : czero();
        }
        if constexpr (PS::kShift) {
            if (fresh) {
                if (__any_sync(0xffffffffu, out && t.v2 * bend2(xs + j * kPairXPts + i, ix, p.nx, bias) >
                                                       pair_limit2<IMAG>(norm2(pair_of(x, bias).h), pair_floor2(um, k)))) {
                    k0 = kPairNear;
                    if (out) x = add(x, unpack(near_mem<IMAG>(xs + j * kPairXPts + i, 1, ix, p.nx, t.near[0], t.near[1])));
                }
            }
        }
        __syncthreads();
    }
    // the links of the updated state, mirrored about the line's ghost points (zero past the
    // ends of a segment inside the row: those links weigh less than 2^-56)
    if (!fresh) {
        Us[j][i] = in ? s : czero();
        __syncthreads();
    }
    {
        cd* L = Ls[j] + H;
        if (in) {
            const cd M = fresh ? L[i] : cadd(L[i], csub(i + 1 < np ? Us[j][i + 1] : czero(), s));
            L[i] = M;
            if (sg.a0 == 0 && i < H - 2) L[-3 - i] = M;                      // M_(-2-k) = M_(-1+k)
            if (sg.a1 == p.nx && np - 1 - i < H) L[2 * np - 1 - i] = M;      // M_(n+k) = M_(n-1-k)
            if (i == 0) {
                const cd M1 = cadd(L[-1], s);
                L[-1] = M1;
                if (sg.a0 == 0) L[-2] = M1;
            }
        }
        if (sg.a0 != 0 && i < H - 1) L[-2 - i] = czero();
        if (sg.a1 != p.nx && i < H) L[np + i] = czero();
    }
    __syncthreads();
    if constexpr (PS::kShift) {
        if (!slow && __any_sync(0xffffffffu, large & kRough)) {
            k0 = kPairNear;
            if (out) x = add(x, unpack(near_inc<IMAG>(A + at, &Us[j][i], bias, ix, p.nx, t.near[0], t.near[1])));
        }
    }
    if (out) {
        const cd inc = cadd(s, pair_taps<IMAG>(Ls[j] + H + i, 1, t, k0));
        st<R>(Bout, at, pair_plus<R>(x, inc, bias));
    }
}

// The same with one thread per point, for grids that fill the GPU: the components meet in
// registers, which halves the instructions of the by-component kernel (no factor is formed
// three times: 4.9 M against 10.9 M at 256^2 when the two were first compared) and needs half the
// barriers (256^2: 41 -> 25 us a step then). Bound by latency and instruction fetch: at 256^2 30 % of the
// issue slots and 17 % of the FP64 pipe are used, 32 % of the fetches miss the instruction cache
// (3.2 stalls an issue), 256 blocks are 21 % of the warps. Segments of up to kPairPPts points.
template <typename R, bool IMAG>
__global__ void __launch_bounds__(kPairPPts, 2)
    k_pair_xp(const typename V2<R>::T* __restrict__ A, typename V2<R>::T* __restrict__ Bout, KParams p, DevScalars* sc,
              const double* __restrict__ omega_tab, PairTab t, int nseg, const double* __restrict__ partials, int m,
              int renorm) {
    using PS = PairState<R>;
    using T = typename V2<R>::T;
    constexpr int H = kPairTaps + 1;
    __shared__ cd Ls[3][kPairPPts + 2 * H];
    __shared__ __align__(16) cd Us[3][kPairPPts];  // the full-width state; the increments
    __shared__ double red[3], dsh[3];
    __shared__ df dms;
    __shared__ int far_s;
    __shared__ unsigned wmax[kPairPPts / 32], large_s;
    const int i = threadIdx.x, warp = i >> 5, nw = blockDim.x >> 5;
    const int iy = blockIdx.x / nseg;
    const PairSeg sg = pair_seg(p.nx, nseg, t.kt + 1, blockIdx.x - iy * nseg);
    const int np = sg.a1 - sg.a0, ix = sg.a0 + i;
    const bool in = i < np, out = in && ix >= sg.o0 && ix < sg.o1, so = p.so_case != 0;
    const size_t plane = (size_t)p.nx * p.ny, at = (size_t)iy * p.nx + ix;
    const cx<R> zr = {R(0), R(0)};
    pdl_wait();
    cx<R> x[3], xp[3], ym[3], yp[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        x[j] = in ? ld<R>(A, j * plane + at) : zr;
        xp[j] = in && ix + 1 < p.nx ? ld<R>(A, j * plane + at + 1) : zr;
        ym[j] = in && so && iy > 0 ? ld<R>(A, j * plane + at - p.nx) : zr;
        yp[j] = in && so && iy + 1 < p.ny ? ld<R>(A, j * plane + at + p.nx) : zr;
    }
    const bool from_parts = partials && *(volatile const int*)&sc->scale_src;
    unsigned um = 0u;
    if (from_parts)
        for (int j = warp; j < 3; j += nw) {
            const double q = sum_partials_warp(partials + (size_t)j * m, m);
            if ((i & 31) == 0) red[j] = q;
        }
    if constexpr (PS::kShift) {
        const int tick = *(volatile const int*)&sc->pair_tick;
        um = *(volatile const unsigned*)&sc->umax[(tick + 2) % 3];
        if (blockIdx.x == 0 && i == 0) {
            sc->umax_slot = tick;
            sc->umax[(tick + 1) % 3] = 0u;
        }
        unsigned mx = 0u;
#pragma unroll
        for (int j = 0; j < 3; j++) mx = max(mx, max(pair_mag(x[j]), max(pair_mag(ym[j]), pair_mag(yp[j]))));
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((i & 31) == 0) wmax[warp] = mx;
        if (i == 0) large_s = 0u;
    }
    __syncthreads();
    int k = 0;
    if constexpr (PS::kShift) {
        unsigned mx = 0u;
        for (int w = 0; w < nw; w++) mx = max(mx, wmax[w]);
        k = pair_shift(mx);
    }
    unsigned bias = (unsigned)(896 - k) << 20;
    cd u[3], s[3], L[3], Y[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        u[j] = pair_of(x[j], bias);
        s[j] = czero();
        L[j] = pair_diff(xp[j], x[j], bias);
        if (so) Y[j] = pair_diff(yp[j], ym[j], bias);
        if (in) Ls[j][H + i] = L[j];
        if (i == 0) Ls[j][H - 1] = sg.a0 == 0 ? u[j] : czero();
    }
    if (i == blockDim.x - 32) {  // lane 0 of the last warp
        if (from_parts) {
            const double N[3] = {red[0] * p.cell, red[1] * p.cell, red[2] * p.cell};
            const bool finite = isfinite(N[0]) && isfinite(N[1]) && isfinite(N[2]);
            double d[3];
            renorm_factors(N, finite ? renorm : 0, p.mag, d);
            for (int c = 0; c < 3; c++) dsh[c] = d[c];
        } else {
            for (int c = 0; c < 3; c++) dsh[c] = sc->scale[c];
        }
        pair_near(dsh, &dms, &far_s);
        if (PS::kShift && blockIdx.x == 0) sc->umax_prev = far_s > 1 ? 0u : um;
    }
    __syncthreads();
    if (far_s > 1) um = 0u;
    const df hx = kpair(p, KC_HX), hy = kpair(p, KC_HY);
    const bool relink = far_s != 0;
    float so2 = 0.0f, r2 = 0.0f;
    if (PS::kShift) {
#pragma unroll
        for (int j = 0; j < 3; j++) r2 += norm2(p_sub(L[j].h, Ls[j][H + i - 1].h));
    }
    if (so) {
        cd X[3];
#pragma unroll
        for (int j = 0; j < 3; j++) X[j] = in ? cadd(L[j], Ls[j][H + i - 1]) : czero();  // (unset past the end)
        df gx[3] = {hx, hx, hx}, gy[3] = {hy, hy, hy};
        if (relink) {  // (the shift's change below included)
            const int kn = fabs(dsh[0]) > 1e6 || fabs(dsh[0]) < 1e-6 ? 0 : k;
            for (int c = 0; c < 3; c++) {
                int e;
                const df dc = df_from(frexp(dsh[c], &e));
                const float f = __int_as_float((127 + max(-126, min(126, e + kn - k))) << 23);
                gx[c] = lscale(lmul(hx, dc), f);
                gy[c] = lscale(lmul(hy, dc), f);
            }
        }
        if (relink) {
            const cd n0 = cneg(X[0]), n1 = cneg(X[1]);
            s[0] = mz<IMAG>(so_form(gx[1], gy[1], X[1], Y[1]));
            s[2] = mz<IMAG>(so_form(gx[1], gy[1], n1, Y[1]));
            s[1] = mz<IMAG>(cadd(so_form(gx[0], gy[0], n0, Y[0]), so_form(gx[2], gy[2], X[2], Y[2])));
        } else {
            const cd ax = cscl(hx, X[1]), ay = cscl(hy, cmulni(Y[1]));
            s[0] = mz<IMAG>(cadd(ax, ay));
            s[2] = mz<IMAG>(csub(ay, ax));
            s[1] = mz<IMAG>(so_form(hx, hy, csub(X[2], X[0]), cadd(Y[0], Y[2])));
        }
        so2 = norm2(s[0].h) + norm2(s[1].h) + norm2(s[2].h);
    }
    if (relink) {
        if (fabs(dsh[0]) > 1e6 || fabs(dsh[0]) < 1e-6) {
            k = 0;
            bias = kBias0;
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
            x[j] = {PS::times(x[j].re, dsh[j]), PS::times(x[j].im, dsh[j])};
            u[j] = pair_of(x[j], bias);
        }
    } else if (dms.hi != 0.0f) {
        const df dm = dms;
#pragma unroll
        for (int j = 0; j < 3; j++) s[j] = cadd(s[j], cscl(dm, cadd(u[j], s[j])));
    }
#pragma unroll
    for (int j = 0; j < 3; j++) u[j] = cadd(u[j], s[j]);
    const float f = __int_as_float((127 + max(-126, min(126, -2 * k))) << 23);
    const df Ot = omega_tab ? df_from(__ldg(omega_tab + sc->step_idx) * 0.70710678118654752440) : kpair(p, KC_OMEGA);
    const df c2 = lscale(kpair(p, KC_C2), f);
    df e[3];
    unsigned large = 0u;
    {
        const df rp = cnrm(u[0]), r0 = cnrm(u[1]), rm = cnrm(u[2]), rpm = ladd(rp, rm), dpm = lsub(rp, rm);
        const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;
        const df Vn = ladd(lmulf(kpair(p, KC_NVX), (float)(kx * kx)), lmulf(kpair(p, KC_NVY), (float)(ky * ky)));
        const df base = lfma(lscale(kpair(p, KC_NC0), f), ladd(rpm, r0), Vn), nc2 = lscale(kpair(p, KC_NC2), f);
        e[0] = lfma(nc2, ladd(r0, dpm), base);
        e[1] = lfma(nc2, rpm, base);
        e[2] = lfma(nc2, lsub(r0, dpm), base);
        if constexpr (PS::kShift) {
            const float ae = fmaxf(fabsf(e[0].hi), fmaxf(fabsf(e[1].hi), fabsf(e[2].hi))), ot = fabsf(Ot.hi);
            const float ea = fmaf(fabsf(c2.hi), sqrtf(rm.hi * r0.hi), ot), eb = fmaf(fabsf(c2.hi), sqrtf(r0.hi * rp.hi), ot);
            if (in && (i > 0 || sg.a0 == 0))
                large = pair_large<IMAG>(so2, t.v2 * r2, rpm.hi + r0.hi, pair_floor2(um, k), ae,
                                   p.kf[KC_DT2] * fmaf(ea, ea, eb * eb));
        }
    }
    bool slow = relink, herm = true;
    unsigned bits = 0u;
    const unsigned votes = kWide | (relink ? kRough : 0u);
    if constexpr (PS::kShift) {
        if (__any_sync(0xffffffffu, large & votes)) {
            const unsigned all = __reduce_or_sync(0xffffffffu, large);
            if ((threadIdx.x & 31) == 0) atomicOr(&large_s, all);
        }
        if (__syncthreads_or(large & votes)) bits = large_s;
        if (far_s > 1) bits |= kRough;
        slow = relink || bits;
    }
    T* xs = reinterpret_cast<T*>(&Us[0][0]);  // [3][kPairPPts]
    int k0 = 0;
    if (!(bits & kWide)) {
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cd tn;
            if constexpr (IMAG) {
                tn = cscl(em1_pair(e[j]), u[j]);
            } else {
                df cm1, sn;
                sc_pair(e[j], &cm1, &sn);
                tn = cadd(cscl(cm1, u[j]), cscl(sn, cmuli(u[j])));
            }
            s[j] = cadd(s[j], tn);
            u[j] = cadd(u[j], tn);
        }
    } else {
        if constexpr (PS::kShift) {
            const double otd = omega_tab ? __ldg(omega_tab + sc->step_idx) * 0.70710678118654752440 : p.kd[KC_OMEGA];
            herm = !(bits & (kHerm | kSo));
            cx<double> v[3];
#pragma unroll
            for (int j = 0; j < 3; j++) v[j] = pair_plus<R>(x[j], s[j], bias);
            if (!(bits & kSo))
                nonlin_wide<IMAG>(v, p, otd, ix, iy, !herm);
            else if (in)
                point_wide<IMAG>(A, p, dsh, otd, ix, iy, v);
#pragma unroll
            for (int j = 0; j < 3; j++) {
                x[j] = v[j];
                u[j] = pair_of(v[j], bias);
                s[j] = czero();
            }
        }
    }
    if (herm) {
        cd a = cscl(c2, cmulc(u[2], u[1])), b = cscl(c2, cmulc(u[1], u[0]));
        a = cd(ladd(a.re(), Ot), a.im());
        b = cd(ladd(b.re(), Ot), b.im());
        const float w = p.kf[KC_DT2] *
                        fmaf(a.h.x, a.h.x, fmaf(a.h.y, a.h.y, fmaf(b.h.x, b.h.x, b.h.y * b.h.y)));
        df cs, ck;
        if (w < 9.5367431640625e-07f) {
            const float v = IMAG ? w : -w;
            cs = laddf(kpair(p, KC_HS0), v * fmaf(p.kf[KC_HS0 + 2], v, p.kf[KC_HS0 + 1]));
            ck = laddf(kpair(p, KC_HK0), v * fmaf(p.kf[KC_HK0 + 2], v, p.kf[KC_HK0 + 1]));
            if (!IMAG) ck = lneg(ck);
        } else {
            herm_wide<IMAG>(a, b, p, &cs, &ck);
        }
        // -s_z A u + k A^2 u = A (-s_z u + k A u) row by row, (A^2 u)_0 = (|a|^2 + |b|^2) u_0
        const cd A0 = cadd(cmulc(a, u[0]), cmulp(b, u[2]));
        const cd m0 = cadd(mz<IMAG>(cscl(cs, u[1])), cscl(ck, A0));  // rows +1, -1: a, b* times this
        s[0] = cadd(s[0], cmulp(a, m0));
        s[2] = cadd(s[2], cmulc(b, m0));
        s[1] = cadd(s[1], cadd(mz<IMAG>(cscl(cs, A0)), cscl(lmul(ck, ladd(cnrm(a), cnrm(b))), u[1])));
    }
    const bool fresh = PS::kShift && bits;  // the increments start from zero
    if (slow) {
        if (fresh) {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                if (herm) x[j] = pair_plus<R>(x[j], s[j], bias);
                s[j] = czero();
            }
        }
#pragma unroll
        for (int j = 0; j < 3; j++)
            if (in) xs[j * kPairPPts + i] = pack(x[j]);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 3; j++) {
            L[j] = pair_diff(i + 1 < np ? unpack(xs[j * kPairPPts + i + 1]) : zr, x[j], bias);
            if (i == 0) Ls[j][H - 1] = sg.a0 == 0 ? pair_of(x[j], bias) : czero();
        }
        if constexpr (PS::kShift) {
            if (fresh) {
                float b2 = 0.0f, rho = 0.0f;
                if (out) {
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        b2 += bend2(xs + j * kPairPPts + i, ix, p.nx, bias);
                        rho += norm2(pair_of(x[j], bias).h);
                    }
                }
                if (__any_sync(0xffffffffu, t.v2 * b2 > pair_limit2<IMAG>(rho, pair_floor2(um, k)))) {
                    k0 = kPairNear;
                    if (out) {
#pragma unroll
                        for (int j = 0; j < 3; j++)
                            x[j] = add(x[j], unpack(near_mem<IMAG>(xs + j * kPairPPts + i, 1, ix, p.nx, t.near[0], t.near[1])));
                    }
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 3; j++) Us[j][i] = in ? s[j] : czero();
    __syncthreads();
    if constexpr (PS::kShift) {
        if (!slow && __any_sync(0xffffffffu, large & kRough)) {
            k0 = kPairNear;
            if (out) {
#pragma unroll
                for (int j = 0; j < 3; j++)
                    x[j] = add(x[j], unpack(near_inc<IMAG>(A + j * plane + at, &Us[j][i], bias, ix, p.nx, t.near[0], t.near[1])));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 3; j++) {
        cd* Lj = Ls[j] + H;
        if (in) {
            const cd M = cadd(L[j], csub(i + 1 < np ? Us[j][i + 1] : czero(), s[j]));
            Lj[i] = M;
            if (sg.a0 == 0 && i < H - 2) Lj[-3 - i] = M;
            if (sg.a1 == p.nx && np - 1 - i < H) Lj[2 * np - 1 - i] = M;
            if (i == 0) {
                const cd M1 = cadd(Lj[-1], s[j]);
                Lj[-1] = M1;
                if (sg.a0 == 0) Lj[-2] = M1;
            }
        }
        if (sg.a0 != 0 && i < H - 1) Lj[-2 - i] = czero();
        if (sg.a1 != p.nx && i < H) Lj[np + i] = czero();
    }
    __syncthreads();
    if (out) {
        // (one copy of the taps' code; the increments of this thread's own points)
#pragma unroll 1
        for (int j = 0; j < 3; j++) Us[j][i] = cadd(Us[j][i], pair_taps<IMAG>(Ls[j] + H + i, 1, t, k0));
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const cd inc = Us[j][i];
            st<R>(Bout, j * plane + at, cx<R>{PS::plus(x[j].re, inc.re(), bias), PS::plus(x[j].im, inc.im(), bias)});
        }
    }
}

// -- kernel 2: Crank-Nicolson along y ---------------------------------------------------
// One block per tile of 8 adjacent columns (whole 128-byte lines) of one component and
// 64 rows [o0, o1); thread (column, row lane r of 32) takes the rows o0 + r and o0 + 32 +
// r, and of the 16 rows above and below, which only give links, row lane r < 16 the row
// o0 - 1 - r, the others o1 + r - 16. Norm partials per tile: pairs per thread and block,
// the tile's sum in FP64.
template <typename R, bool IMAG>
__global__ void __launch_bounds__(256, 4)
    k_pair_y(const typename V2<R>::T* __restrict__ in, typename V2<R>::T* __restrict__ out, KParams p, PairTab t, int nrt,
             double* __restrict__ part, DevScalars* sc, int head, int renorm, int advance) {
    using PS = PairState<R>;
    constexpr int CW = kPairCols, H = kPairTaps;
    __shared__ cd Ms[(kPairRows + 2 * H) * CW];  // (H + r) * CW + column: the link from row o0 + r to the next
    __shared__ typename PartT<R>::T red[8];
    __shared__ long long zred[8];
    __shared__ unsigned wmax[8];
    const int tid = threadIdx.x, cc = tid % CW, rl = tid / CW;
    const int nct = (p.nx + CW - 1) / CW;
    const int rt = blockIdx.x % nrt, rest = blockIdx.x / nrt, ct = rest % nct, j = rest / nct;
    const int n = p.ny, o0 = rt * kPairRows, col = ct * CW + cc;
    const bool colok = col < p.nx;
    const size_t base = (size_t)j * p.nx * n + (colok ? col : p.nx - 1);
    const cx<R> zr = {R(0), R(0)};
    pdl_wait();
    if (blockIdx.x == 0 && tid < 3) {
        if (tid == 0) sc->pair_tick = (sc->pair_tick + 1) % 3;
        if (head) {  // as k_cny_reg
            if (renorm) {
                if (tid == 0) sc->scale_src = 1;
            } else {
                sc->scale[tid] = 1.0;
                sc->scale_f[tid] = 1.0f;
                sc->scale_l[tid] = 0.0f;
            }
            if (advance && tid == 0) sc->step_idx += 1;
        }
    }
    auto row = [&](int r) { return r >= 0 && r < n ? ld<R>(in, base + (size_t)r * p.nx) : zr; };
    // the rows of this thread and the ones below them (the links go from a row to the next)
    const int rh = rl < 16 ? o0 - 1 - rl : o0 + kPairRows + rl - 16;
    const cx<R> x0 = row(o0 + rl), x1 = row(o0 + 32 + rl), y0 = row(o0 + rl + 1), y1 = row(o0 + 33 + rl);
    const cx<R> xh = row(rh), yh = row(rh + 1);
    int k = 0;
    unsigned umx = 0u;
    float floor2 = 0.0f;
    if constexpr (PS::kShift) {
        const unsigned um = *(volatile const unsigned*)&sc->umax_prev;
        unsigned mx = max(max(pair_mag(x0), pair_mag(x1)), pair_mag(xh));
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((tid & 31) == 0) wmax[tid >> 5] = mx;
        __syncthreads();
        mx = 0u;
        for (int w = 0; w < 8; w++) mx = max(mx, wmax[w]);
        k = pair_shift(mx);
        umx = mx;
        floor2 = pair_floor2(um, k);
        if (tid == 0) atomicMax(&sc->umax[sc->umax_slot], mx);
    }
    const unsigned bias = (unsigned)(896 - k) << 20;
    // link r (from row r to r + 1) of this column, and its mirror images about the ghost rows -1 and n:
    // M_(-2-k) = M_(-1+k), M_(n+k) = M_(n-1-k)
    cd* M = Ms + H * CW + cc;
    auto put = [&](int r, const cx<R>& a, const cx<R>& b) {
        if (r >= -1 && r < n) {
            const cd l = pair_diff(b, a, bias);
            M[(r - o0) * CW] = l;
            const int lo = -3 - r - o0, hi = 2 * n - 1 - r - o0;  // the images' places
            if (lo >= -H) M[lo * CW] = l;
            if (hi < kPairRows + H) M[hi * CW] = l;
        }
    };
    put(o0 + rl, x0, y0);
    put(o0 + 32 + rl, x1, y1);
    put(rh, xh, yh);
    __syncthreads();
    df acc = df(0.0f, 0.0f);
    float acc2 = 0.0f;
#pragma unroll 1
    for (int q = 0; q < 2; q++) {
        const int r = o0 + 32 * q + rl;
        const bool act = r < n && colok;
        const cd* Mr = M + (32 * q + rl) * CW;
        cx<R> x = q ? x1 : x0;
        cd xh = pair_of(x, bias);
        int k0 = 0;
        if constexpr (PS::kShift) {
            // (one component is at hand: the check is against its own value)
            const float2 d = p_sub(Mr[0].h, Mr[-CW].h);
            if (__any_sync(0xffffffffu, act && t.v2 * norm2(d) > pair_limit2<IMAG>(norm2(xh.h), floor2))) {
                k0 = kPairNear;
                if (act) x = add(x, unpack(near_mem<IMAG>(in + base + (size_t)r * p.nx, p.nx, r, n, t.near[0], t.near[1])));
                xh = pair_of(x, bias);
            }
        }
        if (act) {
            const cd inc = pair_taps<IMAG>(Mr, CW, t, k0);
            st<R>(out, base + (size_t)r * p.nx,
                  cx<R>{PS::plus(x.re, inc.re(), bias), PS::plus(x.im, inc.im(), bias)});
            // |o|^2: the squares of the low parts (all positive, below the rounding of the products'
            // error terms) are summed apart; dropped, they would bias the norm by 2^-49
            const cd o = cadd(xh, inc);
            acc = ladd(acc, cnrm(o));
            acc2 = fmaf(o.l.x, o.l.x, fmaf(o.l.y, o.l.y, acc2));
        }
    }
    if (!part) return;
    // the tile's sum. complex128: 64-bit integers in units of 2^-57 of the most a thread can hold
    // (pairs would round it to 2^-49, FP64 shuffle sums cost 7 FP64 instructions a warp), four FP64
    // instructions at the end (the warps' sums and the power of two in FP64 were some 30, one
    // after the other at the end of every block: with the pending factors' chain 256^2 25.2 -> 24.0 us a
    // step, 512^2 97.7 -> 90.9, 64^2 12.95 -> 12.0); double-float: in pairs
    double q;
    if constexpr (PS::kShift) {
        // |x 2^k| < 2^(E + 1): a thread's four squares stay below 2^(2E + 4)
        const int E = max(-50, min(50, (int)(umx >> 20) - 1023 + k));
        const float f = __int_as_float((127 + 26 - E) << 23), g = __int_as_float((127 + 27 - E) << 23);
        long long z = __float2ll_rn(acc.hi * f * g) + (__float2ll_rn(acc.lo * f * g) + __float2ll_rn(acc2 * f * g));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) z += __shfl_xor_sync(0xffffffffu, z, off);
        if ((tid & 31) == 0) zred[tid >> 5] = z;
        __syncthreads();
        q = 0.0;
        if (tid == 0) {
            // (the eight sums do not fit 64 bits: their high and low parts apart, one rounding at the end)
            long long zh = 0;
            int zl = 0;
#pragma unroll
            for (int w = 0; w < 8; w++) {
                zh += zred[w] >> 12;
                zl += (int)(zred[w] & 4095);
            }
            q = fma((double)zh, 4096.0, (double)zl) * __hiloint2double((1023 + 2 * E - 53) << 20, 0);
        }
    } else {
        const df ps = block_part(fast_two_sum(acc.hi, acc.lo + acc2), red);
        q = (double)ps.hi + (double)ps.lo;
    }
    if (tid == 0) {
        if (k != 0) q = q * exp2(-(double)k) * exp2(-(double)k);
        // (integers carry no NaN: infinities and NaN among the tile's values make its sum one, so that
        // the step sets the error flag and leaves the scale at 1)
        if (PS::kShift && umx >= 0x7ff00000u) q = __longlong_as_double(0x7ff8000000000000ll);
        part[blockIdx.x] = q;
    }
}

}  // namespace sgpe
