// sgpe_socn.cuh -- the SO substep by Crank-Nicolson (the unitary variant of
// the explicit-Euler SO substep of Appendix A Eqs. (p1)-(p2)).
//
// Along one grid line the SO operator of Sec. 2 is H = g S p, p = -i D (D the
// central first difference with zero ghosts, spacing h), S one of the spin-1
// matrices Sigma_x, Sigma_y, Sigma_z of Eq. (smat) and g a real strength (1D:
// gamma; 2D x lines: -gamma with S = Sigma_y; 2D y lines: eta gamma with S =
// Sigma_x). Crank-Nicolson: (I + z/2 H) psi' = (I - z/2 H) psi. S has the
// eigenvalues +1, 0, -1 with eigenvectors u_k (the columns of U, fixed 3x3),
// so in the rotated components phi = U^H psi the system splits into three
// scalar lines: phi_0 is unchanged, and phi_(+-1) solve
//   T phi' = (2 I - T) phi,  T = I + a_m (S+ - S-),  a_m = -i z g m / (4 h),
// a tridiagonal matrix with opposite off-diagonals (S+-: shift by one point).
// Each line is solved in increment form, phi' = phi + 2 e with
// T e = -a_m (phi_(i+1) - phi_(i-1)), by the lane-chunk scan of the kinetic
// sweeps with skew tables (k_coef, CoefJob::skew): u_0 = 1, u_i = 1 + a^2 / u_(i-1);
// forward y_i = fa_i x_i + fg_i y_(i-1) with fa = 1/u, fg = a/u; backward w_i = y_i -
// fg_i w_(i+1). The result is psi' = U phi'.
//
// One block of three warps per line (n <= 1024 points): the line's three
// components are loaded, rotated and staged in shared memory in the lanes'
// padded chunk layout; warps 0 and 2 solve phi_(+1) and phi_(-1); all threads
// rotate back and store.
#pragma once
#include "sgpe_cn.cuh"

namespace sgpe {

// One family of lines of one grid (x lines or y lines) for the SO-CN substep.
struct SoCnLines {
    double ur[9], ui[9];      // U[j][k] = ur[3j + k] + i ui[3j + k]: component j of the eigenvector of m_k
    double are, aim;          // a of m = +1 (m = -1 takes -a)
    int which;                // the spin matrix: 0 Sigma_x, 1 Sigma_y, 2 Sigma_z
    int n, nlines;            // points per line, lines
    long long stride, lstride;  // element distance between the points of a line, between lines
    long long plane;          // elements per spin component
};

constexpr int kSoCnThreads = 96;

// One product term u v (or conj(u) v) of the eigenbasis rotation. For the FP32
// state the rounding remainder ul of each entry of U (1/sqrt2 is not an FP32
// number) is added inside the fused multiply-adds, before the product is first
// rounded: each term is then rounded once from a value accurate to ~1e-15. Added
// after the rounded product the remainder would be lost, and the rounding of
// 1/sqrt2 would shrink the norm by ~1.3e-8 per rotation, four rotations a step.
template <bool CONJ, typename R>
__device__ __forceinline__ cx<R> rot_term(cx<R> u, cx<R> ul, cx<R> v) {
    if constexpr (is_f32<R>()) {
        const cx<R> c = CONJ ? cmul(ul, v) : mul(ul, v);
        if (CONJ)
            return {fma(u.re, v.re, fma(u.im, v.im, c.re)), fma(u.re, v.im, fma(-u.im, v.re, c.im))};
        return {fma(u.re, v.re, fma(-u.im, v.im, c.re)), fma(u.re, v.im, fma(u.im, v.re, c.im))};
    } else {
        return CONJ ? cmul(u, v) : mul(u, v);
    }
}

// The rotation phi = U^H psi and its inverse psi = U phi for complex128 and double-float
// from U's few distinct entries (1/2, 1/sqrt2, zeros, factors i): 14 real operations a
// point instead of the general product's 84. On the FP64 pipe that product was half of the
// kernel (161^2: 26.4 -> about 15 us a launch, four launches a Strang step: 164 -> 118 us).
template <typename R> __device__ __forceinline__ cx<R> times_i(cx<R> a) { return {-a.im, a.re}; }
template <typename R>
__device__ __forceinline__ void socn_rot(int which, bool inverse, const cx<R> (&v)[3], cx<R> (&o)[3]) {
    if (which == 2) {
        o[0] = v[0];
        o[1] = v[1];
        o[2] = v[2];
        return;
    }
    const R r = to_r<R>(0.70710678118654752440), half = to_r<R>(0.5);
    const cx<R> q = scl(r, v[1]);
    if (which == 0) {  // both ways: (h + q, r (v_+ - v_-), h - q), h = (v_+ + v_-)/2
        const cx<R> h = scl(half, add(v[0], v[2]));
        o[1] = scl(r, sub(v[0], v[2]));
        o[0] = add(h, q);
        o[2] = sub(h, q);
    } else if (!inverse) {  // (h - i q, r (v_+ + v_-), h + i q), h = (v_+ - v_-)/2
        const cx<R> h = scl(half, sub(v[0], v[2])), iq = times_i(q);
        o[1] = scl(r, add(v[0], v[2]));
        o[0] = sub(h, iq);
        o[2] = add(h, iq);
    } else {  // (q + h, i r (v_+ - v_-), q - h), h = (v_+ + v_-)/2
        const cx<R> h = scl(half, add(v[0], v[2]));
        o[1] = times_i(scl(r, sub(v[0], v[2])));
        o[0] = add(q, h);
        o[2] = sub(q, h);
    }
}

template <typename R, int C> constexpr size_t socn_smem_bytes() {
    return (size_t)3 * 32 * (C + 1) * sizeof(typename V2<R>::T);
}

// The SO-CN substep on one family of lines: in -> out (may be the same buffer).
// scale: apply the pending renormalisation scale of sc on load (the first
// kernel of a step). tp, tm: the skew tables of m = +1 and m = -1.
template <typename R, int C>
__global__ void __launch_bounds__(kSoCnThreads) k_socn(const typename V2<R>::T* in, typename V2<R>::T* out,
                                                      SoCnLines L, Tabs<R> tp, Tabs<R> tm,
                                                      const DevScalars* __restrict__ sc, int scale) {
    using T = typename V2<R>::T;
    extern __shared__ __align__(16) unsigned char socn_smem[];
    T* row = reinterpret_cast<T*>(socn_smem);
    constexpr int S = 32 * (C + 1);
    const int n = L.n;
    const size_t base = (size_t)blockIdx.x * (size_t)L.lstride;
    const size_t plane = (size_t)L.plane, stride = (size_t)L.stride;
    const cx<R> zero = {R(0), R(0)};
    pdl_wait();
    R ds[3];
#pragma unroll
    for (int j = 0; j < 3; j++) ds[j] = scale ? scale_of<R>(sc, j) : R(1);
    // U and, for the FP32 state, the rest of each entry after rounding to FP32 (Ul, see rot_term)
    cx<R> U[9], Ul[9];
    if constexpr (is_f32<R>()) {
#pragma unroll
        for (int q = 0; q < 9; q++) {
            U[q] = {to_r<R>(L.ur[q]), to_r<R>(L.ui[q])};
            Ul[q] = {to_r<R>(L.ur[q] - dbl(U[q].re)), to_r<R>(L.ui[q] - dbl(U[q].im))};
        }
    }
    for (int i = threadIdx.x; i < 32 * C; i += kSoCnThreads) {
        cx<R> v[3];
#pragma unroll
        for (int j = 0; j < 3; j++) v[j] = i < n ? scl(ds[j], ldc<R>(in, j * plane + base + (size_t)i * stride)) : zero;
        const int slot = (i / C) * (C + 1) + (i % C);
        cx<R> ph[3];
        if constexpr (is_f32<R>()) {
#pragma unroll
            for (int k = 0; k < 3; k++) {
                // phi_k = sum_j conj(U[j][k]) psi_j
                ph[k] = rot_term<true>(U[k], Ul[k], v[0]);
                ph[k] = add(ph[k], rot_term<true>(U[3 + k], Ul[3 + k], v[1]));
                ph[k] = add(ph[k], rot_term<true>(U[6 + k], Ul[6 + k], v[2]));
            }
        } else {
            socn_rot(L.which, false, v, ph);
        }
#pragma unroll
        for (int k = 0; k < 3; k++) row[k * S + slot] = pack(ph[k]);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp != 1) {
        const Tabs<R>& t = warp == 0 ? tp : tm;
        const R sg = warp == 0 ? R(1) : R(-1);
        const cx<R> a = {sg * to_r<R>(L.are), sg * to_r<R>(L.aim)};
        T* r = row + warp * S;
        const int i0 = lane * C;
        cx<R> x[C], e[C];
#pragma unroll
        for (int m = 0; m < C; m++) x[m] = unpack(r[lane * (C + 1) + m]);
        // e_i = -a (x_(i+1) - x_(i-1)); points past n hold zeros
        cx<R> prev = shup(x[C - 1], 1), last = shdn(x[0], 1);
        if (lane == 0) prev = zero;
        if (lane == 31) last = zero;
#pragma unroll
        for (int m = 0; m < C; m++) {
            const cx<R> nxt = (m + 1 < C) ? x[m + 1] : last;
            const cx<R> d = sub(nxt, prev);
            e[m] = {-(a.re * d.re - a.im * d.im), -(a.re * d.im + a.im * d.re)};
            prev = x[m];
        }
        LaneTabs<R, false, C> lt;
        lt.init(t, i0);
        solve_chunk<R, false, C, true>(e, lt);
#pragma unroll
        for (int m = 0; m < C; m++) {
            const cx<R> o = {fma(R(2), e[m].re, x[m].re), fma(R(2), e[m].im, x[m].im)};
            r[lane * (C + 1) + m] = pack(o);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kSoCnThreads) {
        const int slot = (i / C) * (C + 1) + (i % C);
        const cx<R> ph[3] = {unpack(row[slot]), unpack(row[S + slot]), unpack(row[2 * S + slot])};
        cx<R> o[3];
        if constexpr (is_f32<R>()) {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                // psi_j = sum_k U[j][k] phi_k
                o[j] = rot_term<false>(U[3 * j], Ul[3 * j], ph[0]);
                o[j] = add(o[j], rot_term<false>(U[3 * j + 1], Ul[3 * j + 1], ph[1]));
                o[j] = add(o[j], rot_term<false>(U[3 * j + 2], Ul[3 * j + 2], ph[2]));
            }
        } else {
            socn_rot(L.which, true, ph, o);
        }
#pragma unroll
        for (int j = 0; j < 3; j++) st<R>(out, j * plane + base + (size_t)i * stride, o[j]);
    }
}

}  // namespace sgpe
