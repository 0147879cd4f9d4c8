// sgpe_adjoint.cu -- hand-written adjoint of the real-time split step
// (arXiv:2009.13507, Sec. 3 and Appendix A) for the gradient of
//     L = dx dy sum_r (rho_N(r) - rho_tgt(r))^2,   rho = sum_j |psi_j|^2,
// with respect to the per-step Rabi strengths Omega_n and the trap
// frequencies (wx, wy), by checkpoint-and-recompute.
//
// Gradient convention: g = dL/dRe(psi) + i dL/dIm(psi), so dL = Re(conj(g) dpsi).
// One forward step is psi_{n+1} = CNy CNx HERM_n CALCNU SO (psi_n). Backwards:
//   CN along y and x are complex-linear maps M with M^H = the same sweep with
//   dt -> -dt (tables of bt = -i dt/(4h^2)); SO is I - i dt H_SO with H_SO
//   Hermitian, so its adjoint is the SO substep with dt -> -dt; CALCNU and HERM
//   are non-holomorphic (they depend on |psi|^2 and conj(psi)) and get explicit
//   reverse passes below, recomputing their inputs from the stored psi_n.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "../../include/sgpe.h"
#include "sgpe_cn.cuh"
#include "sgpe_kernels.cuh"
#include "sgpe_launch.h"

namespace sgpe {

// d s/d C^2 and d k/d C^2 of the real-time HERM coefficients
// s = sin(dt C)/C, k = (cos(dt C) - 1)/C^2 (series in v = -(dt C)^2 when small).
template <typename R> __device__ __forceinline__ void herm_coeff_derivs(R C2, R dt, R* ds, R* dk) {
    R w = dt * dt * C2;
    if (w <= R(1.0 / 1024.0)) {
        R v = -w;
        // s  = dt sum v^n/(2n+1)!    -> ds/dC2 = -dt^3 sum_{n>=1} n v^{n-1}/(2n+1)!
        // k  = -dt^2 sum v^n/(2n+2)! -> dk/dC2 = dt^4 sum_{n>=1} n v^{n-1}/(2n+2)!
        R ps = fma(fma(fma(R(4.0 / 362880.0), v, R(3.0 / 5040.0)), v, R(2.0 / 120.0)), v, R(1.0 / 6.0));
        R pk = fma(fma(fma(R(4.0 / 3628800.0), v, R(3.0 / 40320.0)), v, R(2.0 / 720.0)), v, R(1.0 / 24.0));
        *ds = -dt * dt * dt * ps;
        *dk = dt * dt * dt * dt * pk;
        return;
    }
    R C = sqrt(C2), x = dt * C;
    R sn = sin(x), cs = cos(x);
    *ds = (x * cs - sn) / (R(2) * C2 * C);
    *dk = (-x * sn - R(2) * (cs - R(1))) / (R(2) * C2 * C2);
}

template <typename R> __device__ __forceinline__ R re_cmul(cx<R> a, cx<R> b) {  // Re(conj(a) b)
    return fma(a.re, b.re, a.im * b.im);
}
template <typename R> __device__ __forceinline__ R im_cmul(cx<R> a, cx<R> b) {  // Im(conj(a) b)
    return fma(a.re, b.im, -a.im * b.re);
}

// Reverse pass of HERM (real time): u is the HERM input, g holds the gradient
// w.r.t. its output on entry and w.r.t. its input on exit; returns dL/dOt.
template <typename R>
__device__ __forceinline__ R herm_adjoint(const cx<R> (&u)[3], cx<R> (&g)[3], R c2, R Ot, R dt) {
    const cx<R> p = u[0], z = u[1], m = u[2];
    cx<R> a = cmul(m, z);
    a = {fma(c2, a.re, Ot), c2 * a.im};
    cx<R> b = cmul(z, p);
    b = {fma(c2, b.re, Ot), c2 * b.im};
    const R na = nrm(a), nb = nrm(b), C2 = na + nb;
    R s, k, ds, dk;
    herm_coeffs<false>(C2, dt, &s, &k);
    herm_coeff_derivs<R>(C2, dt, &ds, &dk);
    const cx<R> Ap = mul(a, z), A0 = add(cmul(a, p), mul(b, m)), Am = cmul(b, z);
    const cx<R> ab = mul(a, b);
    const cx<R> Bp = axpy(na, p, mul(ab, m)), B0 = scl(C2, z), Bm = axpy(nb, m, cmul(ab, p));
    const cx<R> gP = g[0], gZ = g[1], gM = g[2];
    cx<R> gp = gP, gz = gZ, gm = gM;
    // P = p - i s Ap + k Bp (and likewise Z, M)
    R gs = im_cmul(gP, Ap) + im_cmul(gZ, A0) + im_cmul(gM, Am);
    R gk = re_cmul(gP, Bp) + re_cmul(gZ, B0) + re_cmul(gM, Bm);
    const cx<R> is = {R(0), s};
    const cx<R> gAp = mul(is, gP), gA0 = mul(is, gZ), gAm = mul(is, gM);
    const cx<R> gBp = scl(k, gP), gB0 = scl(k, gZ), gBm = scl(k, gM);
    // Bp = na p + ab m
    gp = axpy(na, gBp, gp);
    R gna = re_cmul(gBp, p);
    cx<R> gab = cmul(m, gBp);
    gm = add(gm, cmul(ab, gBp));
    // B0 = C2 z
    gz = axpy(C2, gB0, gz);
    R gC2 = re_cmul(gB0, z);
    // Bm = conj(ab) p + nb m
    gp = add(gp, mul(ab, gBm));
    gab = add(gab, mul(p, cj(gBm)));
    gm = axpy(nb, gBm, gm);
    R gnb = re_cmul(gBm, m);
    // Ap = a z
    cx<R> ga = cmul(z, gAp);
    gz = add(gz, cmul(a, gAp));
    // A0 = conj(a) p + b m
    ga = add(ga, mul(p, cj(gA0)));
    gp = add(gp, mul(a, gA0));
    cx<R> gb = cmul(m, gA0);
    gm = add(gm, cmul(b, gA0));
    // Am = conj(b) z
    gb = add(gb, mul(z, cj(gAm)));
    gz = add(gz, mul(b, gAm));
    // ab = a b
    ga = add(ga, cmul(b, gab));
    gb = add(gb, cmul(a, gab));
    // s(C2), k(C2); C2 = |a|^2 + |b|^2
    gC2 = fma(gs, ds, fma(gk, dk, gC2));
    gna += gC2;
    gnb += gC2;
    ga = axpy(R(2) * gna, a, ga);
    gb = axpy(R(2) * gnb, b, gb);
    // a = c2 conj(m) z + Ot ; b = c2 conj(z) p + Ot
    gm = axpy(c2, mul(z, cj(ga)), gm);
    gz = axpy(c2, mul(m, ga), gz);
    gz = axpy(c2, mul(p, cj(gb)), gz);
    gp = axpy(c2, mul(z, gb), gp);
    g[0] = gp;
    g[1] = gz;
    g[2] = gm;
    return ga.re + gb.re;
}

// Reverse pass of CALCNU (real time): u1 is the CALCNU input, g the gradient
// w.r.t. its output on entry and w.r.t. u1 on exit; W = sum_j dt Im(conj(g_j) u2_j)
// is returned for the trap gradient (dmu_j/dV = 1).
template <typename R>
__device__ __forceinline__ R calcnu_adjoint(const cx<R> (&u1)[3], cx<R> (&g)[3], R V, R c0, R c2, R dt) {
    const R rp = nrm(u1[0]), r0 = nrm(u1[1]), rm = nrm(u1[2]);
    const R base = fma(c0, rp + r0 + rm, V);
    const R mu[3] = {fma(c2, rp - rm + r0, base), fma(c2, rp + rm, base), fma(c2, rm - rp + r0, base)};
    R w[3];
    cx<R> e[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        R s, c;
        sincos_small(dt * mu[j], &s, &c);
        e[j] = {c, -s};  // exp(-i dt mu_j)
        const cx<R> u2 = mul(e[j], u1[j]);
        w[j] = dt * im_cmul(g[j], u2);
    }
    const R cp = c0 + c2, cm = c0 - c2;
    const R a[3] = {cp * w[0] + cp * w[1] + cm * w[2], cp * w[0] + c0 * w[1] + cp * w[2],
                    cm * w[0] + cp * w[1] + cp * w[2]};
#pragma unroll
    for (int k = 0; k < 3; k++) g[k] = axpy(R(2) * a[k], u1[k], cmul(e[k], g[k]));
    return w[0] + w[1] + w[2];
}

// Per point: recompute SO and CALCNU of psi_n, reverse HERM and CALCNU; g returns the
// cotangent at the SO output, gOt the point's share of dL/dOt and W that of dL/dV.
template <typename R>
__device__ __forceinline__ void reverse_point(const typename V2<R>::T* __restrict__ psi,
                                              const typename V2<R>::T* G, const KParams& p, R Ot, int ix,
                                              int iy, size_t c, size_t plane, cx<R> (&g)[3], R* gOt, R* W) {
    const cx<R> zero = {R(0), R(0)};
    cx<R> u[3];
#pragma unroll
    for (int j = 0; j < 3; j++) u[j] = ld<R>(psi, j * plane + c);
    if (p.so_case) {
        cx<R> X[3], Y[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cx<R> xp = (ix + 1 < p.nx) ? ld<R>(psi, j * plane + c + 1) : zero;
            cx<R> xm = (ix > 0) ? ld<R>(psi, j * plane + c - 1) : zero;
            X[j] = sub(xp, xm);
            if (p.dim == 2) {
                cx<R> yp = (iy + 1 < p.ny) ? ld<R>(psi, j * plane + c + p.nx) : zero;
                cx<R> ym = (iy > 0) ? ld<R>(psi, j * plane + c - p.nx) : zero;
                Y[j] = sub(yp, ym);
            } else {
                Y[j] = zero;
            }
        }
        R gx[3] = {(R)p.hx, (R)p.hx, (R)p.hx}, gy[3] = {(R)p.hy, (R)p.hy, (R)p.hy};
        so_point<false>(u, X, Y, gx, gy, p.so_case);
    }
    const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;
    const R V = (R)p.vx * (R)(kx * kx) + (p.dim == 2 ? (R)p.vy * (R)(ky * ky) : R(0));
    const R dt = (R)p.dt;
    cx<R> u2[3] = {u[0], u[1], u[2]};
    calcnu_point<false>(u2, V, (R)p.c0, (R)p.c2, dt);
#pragma unroll
    for (int j = 0; j < 3; j++) g[j] = ld<R>(G, j * plane + c);
    *gOt = herm_adjoint<R>(u2, g, (R)p.c2, Ot, dt);
    *W = calcnu_adjoint<R>(u, g, V, (R)p.c0, (R)p.c2, dt);
}

// complex128: the reverse of HERM and CALCNU on g in place, with FP64 partial sums of dL/dOt
// and the trap sums; the reverse SO and the sum of the partials are launches of their own
// (the ring of ka_reverse would repeat a quarter to a half of this kernel's FP64 work, which bounds it).
// Block 32 x 4, one point per thread.
template <typename R>
__global__ void __launch_bounds__(128) ka_pointwise(const typename V2<R>::T* __restrict__ psi,
                                                    typename V2<R>::T* __restrict__ G, KParams p, double Ot,
                                                    double* part) {
    __shared__ double red[4 * 3];
    const int ix = blockIdx.x * blockDim.x + threadIdx.x;
    const int iy = blockIdx.y * blockDim.y + threadIdx.y;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    double acc[3] = {0.0, 0.0, 0.0};  // dL/dOt, sum W wx x^2, sum W wy y^2
    if (ix < p.nx && iy < p.ny) {
        const size_t plane = (size_t)p.nx * p.ny, c = (size_t)iy * p.nx + ix;
        const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;
        cx<R> g[3];
        R gOt, W;
        reverse_point<R>(psi, G, p, (R)Ot, ix, iy, c, plane, g, &gOt, &W);
#pragma unroll
        for (int j = 0; j < 3; j++) st<R>(G, j * plane + c, g[j]);
        acc[0] = (double)gOt;
        // dV/dwx = wx x^2, dV/dwy = wy y^2
        acc[1] = (double)W * p.wx * (double)(kx * kx) * p.dx * p.dx;
        acc[2] = p.dim == 2 ? (double)W * p.wy * (double)(ky * ky) * p.dy * p.dy : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 3; q++)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
    if ((tid & 31) == 0)
        for (int q = 0; q < 3; q++) red[(tid >> 5) * 3 + q] = acc[q];
    __syncthreads();
    if (tid == 0) {
        const int nw = (blockDim.x * blockDim.y) >> 5;
        const int blk = blockIdx.y * gridDim.x + blockIdx.x;
        for (int q = 0; q < 3; q++) {
            double s = 0.0;
            for (int w = 0; w < nw; w++) s += red[w * 3 + q];
            part[3 * blk + q] = s;
        }
    }
}

// dL/dpsi of the final-density loss and the loss partial sums: g_j = 4 cell (rho - rho_tgt) psi_j.
template <typename R>
__global__ void __launch_bounds__(128) ka_loss(const typename V2<R>::T* __restrict__ psi,
                                               const double* __restrict__ tgt, typename V2<R>::T* __restrict__ G,
                                               KParams p, double* part) {
    __shared__ double red[4];
    const int ix = blockIdx.x * blockDim.x + threadIdx.x;
    const int iy = blockIdx.y * blockDim.y + threadIdx.y;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    double acc = 0.0;
    if (ix < p.nx && iy < p.ny) {
        const size_t plane = (size_t)p.nx * p.ny, c = (size_t)iy * p.nx + ix;
        cx<R> u[3];
        double rho = 0.0;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            u[j] = ld<R>(psi, j * plane + c);
            rho += (double)u[j].re * (double)u[j].re + (double)u[j].im * (double)u[j].im;
        }
        const double d = rho - tgt[c];
        acc = p.cell * d * d;
        const R f = (R)(4.0 * p.cell * d);
#pragma unroll
        for (int j = 0; j < 3; j++) st<R>(G, j * plane + c, scl(f, u[j]));
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((tid & 31) == 0) red[tid >> 5] = acc;
    __syncthreads();
    if (tid == 0) {
        const int nw = (blockDim.x * blockDim.y) >> 5;
        double s = 0.0;
        for (int w = 0; w < nw; w++) s += red[w];
        part[blockIdx.y * gridDim.x + blockIdx.x] = s;
    }
}

// out[0] = sum of part[3b + 0] / sqrt2 (dL/dOmega_n) and dw[0..1] += sums of part[3b + 1..2],
// by one block in a fixed order. red: 3 doubles a warp.
__device__ __forceinline__ void reduce_partials(const double* part, int nblk, double* out, double* dw, double* red) {
    double s[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x)
        for (int q = 0; q < 3; q++) s[q] += part[3 * (size_t)b + q];
    block_reduce<3>(s, red);
    if (threadIdx.x == 0) {
        out[0] = s[0] * 0.70710678118654752440;
        dw[0] += s[1];
        dw[1] += s[2];
    }
}

// complex64: a whole reverse pointwise stage in one launch. Block b >= 1 owns a tile of
// 32 x 8 points (tile b - 1): it reverses HERM and CALCNU of its points and of the ring of
// neighbours that the SO stencil reads (a thread a point: 256 + 80 of the block's 352), keeps
// those cotangents in shared memory, and applies the reverse SO (dt -> -dt) from there; Gin
// and Gout differ. Block 0 sums the partials that the previous launch left in part_prev (the
// next-later step's, whose dL/dOmega goes to out_prev), which otherwise is a launch of its own
// between two steps: the partials have two halves that the launches use in turn.
//
// What bounds it: latency (256 tiles at 256^2 are one wave). The FP64 part is the sums of
// dL/dOt, W kx^2 and W ky^2: ten FP64 instructions a warp (fold_sum3; the factors
// wx dx^2, wy dy^2 are applied to the block's sums) instead of 25.
// Measured (256^2, 100 steps, a gradient by propagate_real): 5.62 -> 4.32 ms against three
// launches (in place 8.7 us, the sum 5.1, SO 2.9, and their gaps). The y sweep stays in place:
// on row tiles (to the other buffer) 4.12 ms, but the gradient's error against 64 bits grows
// from 1.1e-6 to 1.2e-6.
constexpr int kRevX = 32, kRevY = 8;
constexpr int kRevPts = kRevX * kRevY, kRevRing = 2 * (kRevX + kRevY);
constexpr int kRevThreads = 32 * ((kRevPts + kRevRing + 31) / 32);

// Sums of three values over the warp in six additions a lane: lanes 0, 8 and 16 return the
// sums of a, b and c. Each exchange halves the values a lane still holds.
__device__ __forceinline__ double fold_sum3(double a, double b, double c) {
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16, odd = lane & 8;
    double x = (up ? c : a) + __shfl_xor_sync(0xffffffffu, up ? a : c, 16);
    const double y = (up ? 0.0 : b) + __shfl_xor_sync(0xffffffffu, up ? b : 0.0, 16);
    const double send = up ? x : (odd ? x : y);
    const double got = __shfl_xor_sync(0xffffffffu, send, 8);
    x = ((odd && !up) ? y : x) + got;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

__global__ void __launch_bounds__(kRevThreads) ka_reverse(const float2* __restrict__ psi,
                                                          const float2* __restrict__ Gin, float2* __restrict__ Gout,
                                                          KParams p, float Ot, double* part, int tiles_x,
                                                          const double* part_prev, int nblk, double* out_prev,
                                                          double* dw) {
    constexpr int kW = kRevX + 2;
    __shared__ float2 gs[3][kRevY + 2][kW];
    __shared__ double red[(kRevThreads / 32) * 3];
    const int t = threadIdx.x;
    pdl_wait();
    if (blockIdx.x == 0) {
        if (part_prev) reduce_partials(part_prev, nblk, out_prev, dw, red);
        return;
    }
    const int tile = blockIdx.x - 1;
    const int x0 = (tile % tiles_x) * kRevX, y0 = (tile / tiles_x) * kRevY;
    int lx, ly;
    if (t < kRevPts) {
        lx = t % kRevX;
        ly = t / kRevX;
    } else if (t < kRevPts + 2 * kRevX) {
        lx = t % kRevX;
        ly = t < kRevPts + kRevX ? -1 : kRevY;
    } else {  // the last threads past the ring repeat its last point without storing it
        const int h = min(t - (kRevPts + 2 * kRevX), 2 * kRevY - 1);
        lx = h < kRevY ? -1 : kRevX;
        ly = h % kRevY;
    }
    const int ix = x0 + lx, iy = y0 + ly;
    const bool in = ix >= 0 && ix < p.nx && iy >= 0 && iy < p.ny;
    const size_t plane = (size_t)p.nx * p.ny;
    const cx<float> zero = {0.f, 0.f};
    cx<float> g[3] = {zero, zero, zero};
    float gOt = 0.f, W = 0.f;
    const int kx = ix - p.nx / 2, ky = iy - p.ny / 2;
    if (in) {
        const size_t c = (size_t)iy * p.nx + ix;
        reverse_point<float>(psi, Gin, p, Ot, ix, iy, c, plane, g, &gOt, &W);
    }
    if (t < kRevPts + kRevRing) {
#pragma unroll
        for (int j = 0; j < 3; j++) gs[j][ly + 1][lx + 1] = make_float2(g[j].re, g[j].im);
    }
    if (t < kRevPts) {  // whole warps
        const double w = (double)W;
        const double s = fold_sum3((double)gOt, w * (double)(kx * kx), w);
        const int lane = t & 31;
        if (!(lane & 7) && lane < 24) red[(t >> 5) * 3 + (lane >> 3)] = s;
    }
    __syncthreads();
    if (t < kRevPts && in) {
        if (p.so_case) {
            auto at = [&](int j, int y, int x) { return cx<float>{gs[j][y][x].x, gs[j][y][x].y}; };
            cx<float> X[3], Y[3];
#pragma unroll
            for (int j = 0; j < 3; j++) {
                X[j] = sub(at(j, ly + 1, lx + 2), at(j, ly + 1, lx));
                Y[j] = p.dim == 2 ? sub(at(j, ly + 2, lx + 1), at(j, ly, lx + 1)) : zero;
            }
            const float hx = -(float)p.hx, hy = -(float)p.hy;
            const float gx[3] = {hx, hx, hx}, gy[3] = {hy, hy, hy};
            so_point<false>(g, X, Y, gx, gy, p.so_case);
        }
#pragma unroll
        for (int j = 0; j < 3; j++) st<float>(Gout, j * plane + (size_t)iy * p.nx + ix, g[j]);
    } else if (t >= kRevPts && t < kRevPts + 3) {
        // dV/dwx = wx x^2, dV/dwy = wy y^2 (a warp's row has one ky)
        const int q = t - kRevPts;
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < kRevY; w++) {
            const int r = y0 + w - p.ny / 2;
            s = q < 2 ? s + red[w * 3 + q] : fma(red[w * 3 + 2], (double)(r * r), s);
        }
        if (q == 1) s *= p.wx * p.dx * p.dx;
        if (q == 2) s = p.dim == 2 ? s * p.wy * p.dy * p.dy : 0.0;
        part[3 * tile + q] = s;
    }
}

__global__ void __launch_bounds__(256) ka_reduce(const double* part, int nblk, double* out, double* dw) {
    __shared__ double red[8 * 3];
    reduce_partials(part, nblk, out, dw, red);
}

// One block: out[0] = sum of part[b] (the loss).
__global__ void __launch_bounds__(256) ka_sum(const double* part, int nblk, double* out) {
    __shared__ double red[8];
    double s[1] = {0.0};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) s[0] += part[b];
    block_reduce<1>(s, red);
    if (threadIdx.x == 0) out[0] = s[0];
}

}  // namespace sgpe

using namespace sgpe;

// ---------------------------------------------------------------------------
// Host driver
// ---------------------------------------------------------------------------
namespace {

struct AdjLayout {
    size_t ckpt, seg, g, g2, part, scal, total;
    int nck, K;
};

AdjLayout adj_layout(int nx, int ny, int esz, int nsteps, int K) {
    AdjLayout L;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t st = al((size_t)3 * nx * ny * esz);
    L.K = K;
    L.nck = (nsteps + K - 1) / K;
    size_t o = 0;
    L.ckpt = o;
    o += st * (size_t)(L.nck > 0 ? L.nck : 1);
    L.seg = o;
    o += st * (size_t)K;
    L.g = o;
    o += st;
    L.g2 = o;
    o += st;
    L.part = o;
    // the partials of two launches of 32 x 8 tiles, or of one of 32 x 4 points
    o = al(o + sizeof(double) * 3 * (size_t)ceil_div(nx, 32) * 2 * ceil_div(ny, 8));
    L.scal = o;
    o = al(o + sizeof(double) * 8);
    L.total = o;
    return L;
}

}  // namespace

template <typename R>
static cudaError_t adj_forward_step(const CtxView& v, const void* in, void* out, double omega) {
    KParams k = v.kp;
    k.omega_t = omega * 0.70710678118654752440;
    cudaError_t e;
    if (v.geo->fused && !std::is_same<R, double>::value) {
        // complex64, 2D rows of at most 1024 points: pointwise substeps and CN along
        // x in one kernel (real time: the pending scale is 1, flushed at entry and
        // kept by the y sweep). Same bits as the two kernels; 256^2, 500 steps:
        // 28.4 -> 27.6 ms per gradient (complex128 measured 101.1 -> 102.0, kept unfused).
        if ((e = Launcher<R>::pwx(v.stream, false, in, v.mid, k, v.sc, nullptr, v.tabs_real[0].t, nullptr, 0, 0)))
            return e;
        return Launcher<R>::cn_y(v.stream, false, v.mid, out, k, v.tabs_real[1], *v.geo, v.partials, v.sc, 0, 0, 0);
    }
    e = Launcher<R>::pointwise(v.stream, false, in, v.mid, k, v.sc, nullptr, 7);
    if (e) return e;
    if (v.dim == 2) {
        if ((e = Launcher<R>::cn_x(v.stream, false, false, v.mid, v.mid, k, v.tabs_real[0], *v.geo, v.partials, v.sc, 0,
                                   0)))
            return e;
        return Launcher<R>::cn_y(v.stream, false, v.mid, out, k, v.tabs_real[1], *v.geo, v.partials, v.sc, 0, 0, 0);
    }
    return Launcher<R>::cn_x(v.stream, false, false, v.mid, out, k, v.tabs_real[0], *v.geo, v.partials, v.sc, 0, 0);
}

// Marks the workspace as holding the checkpoints of a forward pass of nsteps
// steps with checkpoint_every = K (checked by the reverse entry point), and the
// states of its last segment (kSegHeld).
constexpr double kAdjTag = 7.0e7 + 13.0;
constexpr int kSegHeld = 7;  // scal[7]: 1 while the segment buffer holds the last segment's states
__global__ void ka_tag(double* scal, int nsteps, int K) {
    scal[4] = kAdjTag;
    scal[5] = (double)nsteps;
    scal[6] = (double)K;
    scal[kSegHeld] = 1.0;
}

// Forward pass with checkpoints: the bound state psi holds psi_0 and ends as
// psi_N; psi_n is stored every K steps (n = 0, K, 2K, ...). The last segment's
// steps go through the segment buffer, which nothing else uses before the reverse
// pass: that pass starts with this segment and then need not run its steps again
// (49 of 98 recomputed steps at nsteps = 100, K = 50: 256^2 complex64 4.32 -> 3.83 ms).
template <typename R>
static cudaError_t adj_forward(const CtxView& v, int nsteps, const double* omega_host, int K, unsigned char* ws) {
    const AdjLayout L = adj_layout(v.nx, v.ny, v.esz, nsteps, K);
    const size_t st = (size_t)3 * v.nx * v.ny * v.esz;
    const size_t sst = (st + 255) & ~(size_t)255;
    cudaStream_t s = v.stream;
    double* scal = (double*)(ws + L.scal);
    cudaError_t e = cudaSuccess;
    const int last0 = (L.nck - 1) * K;  // first step of the last segment
    const void* in = v.psi;
    for (int n = 0; n < nsteps && !e; n++) {
        if (n % K == 0) e = cudaMemcpyAsync(ws + L.ckpt + sst * (n / K), v.psi, st, cudaMemcpyDeviceToDevice, s);
        void* out = n < last0 || n == nsteps - 1 ? v.psi : (void*)(ws + L.seg + sst * (n + 1 - last0));
        if (!e) e = adj_forward_step<R>(v, in, out, omega_host[n]);
        in = out;
    }
    if (!e) {
        ka_tag<<<1, 1, 0, s>>>(scal, nsteps, K);
        e = cudaGetLastError();
    }
    return e;
}

// Reverse pass over the nsteps steps whose checkpoints the forward pass left in
// ws: G (device, [3][ny][nx], inside ws) holds dL/dpsi_N on entry; on exit the
// returned buffer (G or the workspace's second gradient buffer) holds dL/dpsi_0.
// dL/dOmega_n goes to domega_dev[n]; dL/dwx, dL/dwy are added to scal[1], scal[2].
// seg_held: the segment buffer holds the last segment's states (adj_forward).
template <typename R>
static cudaError_t adj_reverse(const CtxView& v, int nsteps, const double* omega_host, int K, unsigned char* ws,
                               bool seg_held, double* domega_dev, typename V2<R>::T** result) {
    using T = typename V2<R>::T;
    const AdjLayout L = adj_layout(v.nx, v.ny, v.esz, nsteps, K);
    const size_t st = (size_t)3 * v.nx * v.ny * v.esz;
    const size_t sst = (st + 255) & ~(size_t)255;
    cudaStream_t s = v.stream;
    auto ckpt = [&](int i) { return (void*)(ws + L.ckpt + sst * i); };
    auto seg = [&](int i) { return (void*)(ws + L.seg + sst * i); };
    T* G = (T*)(ws + L.g);
    T* G2 = (T*)(ws + L.g2);
    double* part = (double*)(ws + L.part);
    double* scal = (double*)(ws + L.scal);  // [0] loss, [1..2] dw
    KParams kneg = v.kp;  // SO with dt -> -dt
    kneg.hx = -kneg.hx;
    kneg.hy = -kneg.hy;
    cudaError_t e = cudaSuccess;
    // a pass over several segments leaves the first one's states in the segment buffer: a
    // further reverse pass of this tape recomputes the last segment too
    if (L.nck > 1) e = cudaMemsetAsync(scal + kSegHeld, 0, sizeof(double), s);
    // complex64: the launch before's partials, summed by block 0 of the next
    const double* prev = nullptr;
    double* prev_out = nullptr;
    const int tiles_x = ceil_div(v.nx, kRevX), tiles = tiles_x * ceil_div(v.ny, kRevY);
    for (int sg = L.nck - 1; sg >= 0 && !e; sg--) {
        const int s0 = sg * K, s1 = (s0 + K < nsteps) ? s0 + K : nsteps;
        // psi_n of this segment: its first state is the checkpoint itself
        auto state = [&](int k) { return k ? seg(k) : ckpt(sg); };
        const bool held = seg_held && sg == L.nck - 1;
        for (int k = 0; k + 1 < s1 - s0 && !held && !e; k++)
            e = adj_forward_step<R>(v, state(k), seg(k + 1), omega_host[s0 + k]);
        for (int n = s1 - 1; n >= s0 && !e; n--) {
            const T* psi = (const T*)state(n - s0);
            const double Ot = omega_host[n] * 0.70710678118654752440;
            if (v.dim == 2)
                e = Launcher<R>::cn_y(s, false, G, G, v.kp, v.tabs_adj[1], *v.geo, v.partials, v.sc, 0, 0, 0);
            if (!e) e = Launcher<R>::cn_x(s, false, false, G, G, v.kp, v.tabs_adj[0], *v.geo, v.partials, v.sc, 0, 0);
            if (e) break;
            if constexpr (std::is_same<R, float>::value) {
                double* pn = part + (size_t)(n & 1) * 3 * tiles;
                e = launch_pdl(ka_reverse, dim3(1 + tiles), dim3(kRevThreads), 0, s, psi, (const T*)G, G2, v.kp,
                               (float)Ot, pn, tiles_x, prev, tiles, prev_out, scal + 1);
                prev = pn;
                prev_out = domega_dev + n;
            } else {
                dim3 blk(32, 4), grd(ceil_div(v.nx, 32), ceil_div(v.ny, 4));
                ka_pointwise<R><<<grd, blk, 0, s>>>(psi, G, v.kp, Ot, part);
                ka_reduce<<<1, 256, 0, s>>>(part, grd.x * grd.y, domega_dev + n, scal + 1);
                e = cudaGetLastError();
                if (!e) e = Launcher<R>::pointwise(s, false, G, G2, kneg, v.sc, nullptr, 1);
            }
            T* t = G;
            G = G2;
            G2 = t;
        }
    }
    if (prev && !e) {
        ka_reduce<<<1, 256, 0, s>>>(prev, tiles, prev_out, scal + 1);
        e = cudaGetLastError();
    }
    *result = G;
    return e;
}

template <typename R>
static sgpe_status adj_run(sgpe_ctx* c, const CtxView& v, int nsteps, const double* omega_host, const double* tgt,
                           int K, unsigned char* ws, double* loss_out, double* domega_dev, double* dw_out) {
    using T = typename V2<R>::T;
    const AdjLayout L = adj_layout(v.nx, v.ny, v.esz, nsteps, K);
    cudaStream_t s = v.stream;
    T* G = (T*)(ws + L.g);
    double* part = (double*)(ws + L.part);
    double* scal = (double*)(ws + L.scal);
    dim3 blk(32, 4), grd(ceil_div(v.nx, 32), ceil_div(v.ny, 4));
    const int nblk = grd.x * grd.y;
    cudaError_t e = cudaMemsetAsync(scal, 0, sizeof(double) * 8, s);
    if (!e) e = adj_forward<R>(v, nsteps, omega_host, K, ws);
    // loss and its gradient at psi_N
    if (!e) {
        ka_loss<R><<<grd, blk, 0, s>>>((const T*)v.psi, tgt, G, v.kp, part);
        ka_sum<<<1, 256, 0, s>>>(part, nblk, scal);
        e = cudaGetLastError();
    }
    T* g0 = nullptr;
    if (!e) e = adj_reverse<R>(v, nsteps, omega_host, K, ws, true, domega_dev, &g0);
    double h[3] = {0, 0, 0};
    if (!e) e = cudaMemcpyAsync(h, scal, sizeof(double) * 3, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    if (loss_out) *loss_out = h[0];
    if (dw_out) {
        dw_out[0] = h[1];
        dw_out[1] = h[2];
    }
    return SGPE_OK;
}

// Common argument checks and the Omega(t) table on the host (the reverse
// kernels take Omega_n as a launch argument). Synchronises the stream.
static sgpe_status adj_prepare(sgpe_ctx* c, CtxView* v, int nsteps, const double* omega_dev, int K,
                               const void* ws, std::vector<double>* om, const char* who) {
    char msg[160];
    if (!ctx_view(c, v) || !v->ready) {
        snprintf(msg, sizeof(msg), "%s: no buffers bound or no parameters", who);
        return ctx_fail(c, SGPE_ESTATE, msg);
    }
    if (v->prec == SGPE_CDF) {
        snprintf(msg, sizeof(msg), "%s: not available for SGPE_CDF", who);
        return ctx_fail(c, SGPE_EUNSUPPORTED, msg);
    }
    if (v->kp.split || v->kp.so_mode) {
        snprintf(msg, sizeof(msg), "%s: the reverse of Lie splitting with the Euler SO only", who);
        return ctx_fail(c, SGPE_EUNSUPPORTED, msg);
    }
    if (nsteps < 1 || K < 1 || !omega_dev || !ws) {
        snprintf(msg, sizeof(msg), "%s: bad arguments", who);
        return ctx_fail(c, SGPE_EINVAL, msg);
    }
    if (((uintptr_t)ws & 255) || ((uintptr_t)omega_dev & 7)) {
        snprintf(msg, sizeof(msg), "%s: misaligned buffer", who);
        return ctx_fail(c, SGPE_EINVAL, msg);
    }
    om->resize(nsteps);
    cudaError_t e = cudaMemcpyAsync(om->data(), omega_dev, sizeof(double) * nsteps, cudaMemcpyDeviceToHost, v->stream);
    if (!e) e = cudaStreamSynchronize(v->stream);
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    return SGPE_OK;
}

extern "C" {

sgpe_status sgpe_adjoint_workspace_bytes(const sgpe_ctx* c, int nsteps, int checkpoint_every, size_t* bytes) {
    CtxView v;
    if (!c || !bytes || nsteps < 1 || checkpoint_every < 1) return SGPE_EINVAL;
    if (!ctx_view((sgpe_ctx*)c, &v)) return SGPE_ESTATE;
    *bytes = adj_layout(v.nx, v.ny, v.esz, nsteps, checkpoint_every).total;
    return SGPE_OK;
}

sgpe_status sgpe_adjoint_loss_grad(sgpe_ctx* c, int nsteps, const double* omega_dev, const double* rho_target_dev,
                                   int checkpoint_every, void* adj_workspace, double* loss_out, double* domega_dev,
                                   double* dw_out) {
    if (!c) return SGPE_EINVAL;
    CtxView v;
    std::vector<double> om;
    sgpe_status st = adj_prepare(c, &v, nsteps, omega_dev, checkpoint_every, adj_workspace, &om, "adjoint");
    if (st) return st;
    if (!rho_target_dev || !domega_dev || ((uintptr_t)rho_target_dev & 7) || ((uintptr_t)domega_dev & 7))
        return ctx_fail(c, SGPE_EINVAL, "adjoint: null or misaligned target / gradient buffer");
    cudaError_t e = ctx_flush(c);  // apply any pending renormalisation: the forward starts at scale 1
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    return v.dbl ? adj_run<double>(c, v, nsteps, om.data(), rho_target_dev, checkpoint_every,
                                   (unsigned char*)adj_workspace, loss_out, domega_dev, dw_out)
                 : adj_run<float>(c, v, nsteps, om.data(), rho_target_dev, checkpoint_every,
                                  (unsigned char*)adj_workspace, loss_out, domega_dev, dw_out);
}

sgpe_status sgpe_adjoint_forward(sgpe_ctx* c, int nsteps, const double* omega_dev, int checkpoint_every,
                                 void* adj_workspace) {
    if (!c) return SGPE_EINVAL;
    CtxView v;
    std::vector<double> om;
    sgpe_status st = adj_prepare(c, &v, nsteps, omega_dev, checkpoint_every, adj_workspace, &om, "adjoint_forward");
    if (st) return st;
    cudaError_t e = ctx_flush(c);  // apply any pending renormalisation: the forward starts at scale 1
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    unsigned char* ws = (unsigned char*)adj_workspace;
    e = v.dbl ? adj_forward<double>(v, nsteps, om.data(), checkpoint_every, ws)
              : adj_forward<float>(v, nsteps, om.data(), checkpoint_every, ws);
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    return SGPE_OK;
}

sgpe_status sgpe_adjoint_step(sgpe_ctx* c, int nsteps, const double* omega_dev, int checkpoint_every,
                              void* adj_workspace, void* lambda_dev, double* domega_dev, double* dw_out) {
    if (!c) return SGPE_EINVAL;
    CtxView v;
    std::vector<double> om;
    sgpe_status st = adj_prepare(c, &v, nsteps, omega_dev, checkpoint_every, adj_workspace, &om, "adjoint_step");
    if (st) return st;
    if (!lambda_dev || !domega_dev || ((uintptr_t)lambda_dev & (v.esz - 1)) || ((uintptr_t)domega_dev & 7))
        return ctx_fail(c, SGPE_EINVAL, "adjoint_step: null or misaligned cotangent / gradient buffer");
    unsigned char* ws = (unsigned char*)adj_workspace;
    const AdjLayout L = adj_layout(v.nx, v.ny, v.esz, nsteps, checkpoint_every);
    double* scal = (double*)(ws + L.scal);
    double tag[4] = {0, 0, 0, 0};
    cudaError_t e = cudaMemcpyAsync(tag, scal + 4, sizeof(tag), cudaMemcpyDeviceToHost, v.stream);
    if (!e) e = cudaStreamSynchronize(v.stream);
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    if (tag[0] != kAdjTag || tag[1] != (double)nsteps || tag[2] != (double)checkpoint_every)
        return ctx_fail(c, SGPE_ESTATE,
                        "adjoint_step: the workspace holds no forward pass of these nsteps and checkpoint_every "
                        "(call sgpe_adjoint_forward first)");
    const size_t st_bytes = (size_t)3 * v.nx * v.ny * v.esz;
    const bool held = tag[3] == 1.0;
    e = cudaMemsetAsync(scal + 1, 0, sizeof(double) * 2, v.stream);
    if (!e) e = cudaMemcpyAsync(ws + L.g, lambda_dev, st_bytes, cudaMemcpyDeviceToDevice, v.stream);
    void* g0 = nullptr;
    if (!e) {
        if (v.dbl) {
            double2* r = nullptr;
            e = adj_reverse<double>(v, nsteps, om.data(), checkpoint_every, ws, held, domega_dev, &r);
            g0 = r;
        } else {
            float2* r = nullptr;
            e = adj_reverse<float>(v, nsteps, om.data(), checkpoint_every, ws, held, domega_dev, &r);
            g0 = r;
        }
    }
    if (!e) e = cudaMemcpyAsync(lambda_dev, g0, st_bytes, cudaMemcpyDeviceToDevice, v.stream);
    double h[2] = {0, 0};
    if (!e) e = cudaMemcpyAsync(h, scal + 1, sizeof(h), cudaMemcpyDeviceToHost, v.stream);
    if (!e) e = cudaStreamSynchronize(v.stream);
    if (e) return ctx_fail(c, SGPE_ECUDA, cudaGetErrorString(e));
    if (dw_out) {
        dw_out[0] = h[0];
        dw_out[1] = h[1];
    }
    return SGPE_OK;
}

}  // extern "C"
