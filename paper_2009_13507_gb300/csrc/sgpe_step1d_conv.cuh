// sgpe_step1d_conv.cuh -- the whole 1D step loop of the complex64 form in one block with
// one thread per point and the Crank-Nicolson sweep as a short convolution.
//
// Why. A 1D grid lives in one SM's shared memory and a step is a chain of latencies. The
// lane-chunk sweep (k_step1d) gave a 1000-point line to three warps of 32 points a lane,
// two serial passes of 32 complex recurrences and ten scan levels, while 5 of 8 warps
// waited: 13.0 us a step in real time, nearly all of it that chain. With the constant
// factor g = bt/u (u the pivot limit, see Tabs) the sweep's increment is
//   x' = x + sum_k W_|k| r_(i+k),  r = L x,  W_k = 2 bt g^k / (u (1 - g^2)),
// r continued oddly past the line's ghost points, cut where |g|^k < 2^-34 (7 taps at bt =
// 0.02, the host allows 16: bt up to about 0.35): every thread sums its own point's taps
// from shared memory, three barriers a step. The differences in r are those of the
// increment form (exact for neighbouring values), each tap rounds to 2^-24 of an
// increment. Measured, us a step (imaginary /
// real time): 1000 points 11.6 / 13.1 -> 6.2 / 5.4, 500 6.8 -> 3.5, 256 3.0 / 3.0 -> 2.2 / 1.8,
// 40 2.0 / 1.9 -> 1.6 / 1.3.
//
// Under Eq. (DJ) lines of at most kConvDjMinN points keep the lane-chunk loop: the scale is a chain of seven
// FP64 square roots a step there too, but its sums are FP64 already and need no conversion (us a
// step, lane chunks / this: 64 points 5.2 / 6.0, 128 5.4 / 6.0, 256 6.3 / 6.4, 384 9.9 / 6.9, 1000 14.7 / 9.8).
//
// Norms (imaginary time): squares split exactly, summed in pairs by shuffles and across
// the warps by every warp for itself; one sum serves Eq. (DJ2), the components' are only
// formed where Eq. (DJ) or the end of the loop needs them.
#pragma once
#include "sgpe_cn.cuh"

namespace sgpe {

constexpr int kConvDjMinN = 256;

// W_k per time mode: (re, re, -im, im).
struct ConvTab {
    float4 w[kConvTaps];
    int kt;
};

__device__ __forceinline__ df sq_pair(cx<float> a) {  // |a|^2, the squares' rounding errors kept
    const float p = __fmul_rn(a.re, a.re), q = __fmul_rn(a.im, a.im);
    const df s = two_sum(p, q);
    return df(s.hi, __fadd_rn(s.lo, __fadd_rn(__fmaf_rn(a.re, a.re, -p), __fmaf_rn(a.im, a.im, -q))));
}

// nx + 2 kConvTaps entries of r per component, two buffers of the state.
inline size_t step1d_conv_smem(int nx) { return (size_t)3 * (3 * nx + 2 * kConvTaps) * sizeof(float2); }

template <bool IMAG>
__global__ void __launch_bounds__(1024, 1)
    k_step1d_conv(float2* __restrict__ A, KParams p, DevScalars* sc, const double* __restrict__ omega_tab, ConvTab t,
                  int nsteps, int renorm) {
    extern __shared__ __align__(16) unsigned char step1d_conv_smem_raw[];
    __shared__ df red[3][32];
    __shared__ float dsh[3];
    const int nx = p.nx, i = threadIdx.x, warp = i >> 5, lane = i & 31, nw = blockDim.x >> 5;
    float2* v0 = reinterpret_cast<float2*>(step1d_conv_smem_raw);  // [3][nx] the state
    float2* v1 = v0 + 3 * nx;                                       // [3][nx] after the pointwise substeps
    float2* rb = v1 + 3 * nx;                                       // [3][nx + 2 kConvTaps]
    const int rs = nx + 2 * kConvTaps;
    const bool in = i < nx;
    const cx<float> zero = {0.0f, 0.0f};
    cx<float> x[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        x[j] = in ? unpack(__ldcg(A + j * nx + i)) : zero;
        if (in) v0[j * nx + i] = pack(x[j]);
    }
    float ds[3] = {sc->scale_f[0], sc->scale_f[1], sc->scale_f[2]};
    const int step0 = sc->step_idx;
    __syncthreads();
    for (int s = 0; s < nsteps; s++) {
        const float Ot = omega_tab ? (float)(__ldg(omega_tab + step0 + s) * 0.70710678118654752440) : kc<float>(p, KC_OMEGA);
        cx<float> u[3] = {zero, zero, zero};
        if (in) {
            PointIn<float> pt;
#pragma unroll
            for (int j = 0; j < 3; j++) {
                pt.u[j] = x[j];
                const cx<float> xp = i + 1 < nx ? unpack(v0[j * nx + i + 1]) : zero;
                const cx<float> xm = i > 0 ? unpack(v0[j * nx + i - 1]) : zero;
                pt.X[j] = sub(xp, xm);
                pt.Y[j] = zero;
            }
            pointwise_apply<float, IMAG>(pt, p, ds, Ot, i, 0, 7, u);
#pragma unroll
            for (int j = 0; j < 3; j++) v1[j * nx + i] = pack(u[j]);
        }
        __syncthreads();
        if (in) {
#pragma unroll
            for (int j = 0; j < 3; j++) {
                const cx<float> um = i > 0 ? unpack(v1[j * nx + i - 1]) : zero;
                const cx<float> up = i + 1 < nx ? unpack(v1[j * nx + i + 1]) : zero;
                const cx<float> r = gadd(gsub(um, u[j]), gsub(up, u[j]));
                float2* R = rb + j * rs + kConvTaps;
                R[i] = pack(r);
                // r_(-1-k) = -r_(-1+k), r_(n+k) = -r_(n-k), zero at the ghost points
                const float2 nr = make_float2(-r.re, -r.im);
                if (i < kConvTaps - 1) R[-2 - i] = nr;
                if (nx - i < kConvTaps) R[2 * nx - i] = nr;
                if (i == 0) R[-1] = R[nx] = make_float2(0.0f, 0.0f);
            }
        }
        __syncthreads();
        const int kt = t.kt;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            if (in) {
                const float2* R = rb + j * rs + kConvTaps + i;
                float2 a = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int k = kConvTaps - 1; k >= 0; k--) {
                    if (k >= kt) continue;
                    const float2 d = k ? __fadd2_rn(R[k], R[-k]) : R[0];
                    a = __ffma2_rn(make_float2(t.w[k].x, t.w[k].y), d, a);
                    if constexpr (!IMAG) a = __ffma2_rn(make_float2(t.w[k].z, t.w[k].w), make_float2(d.y, d.x), a);
                }
                x[j] = fc(__fadd2_rn(f2(u[j]), a));
                v0[j * nx + i] = pack(x[j]);
            }
        }
        const bool last = s == nsteps - 1;
        const bool all = IMAG && renorm == 1 && !last;
        if (IMAG || last) {
            if (all) {
                const df q = warp_sum(sq_pair(x[0]) + sq_pair(x[1]) + sq_pair(x[2]));
                if (lane == 0) red[0][warp] = q;
            } else {
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const df q = warp_sum(sq_pair(x[j]));
                    if (lane == 0) red[j][warp] = q;
                }
            }
        }
        __syncthreads();
        if (IMAG && renorm && !last) {
            const df z = df(0.0f, 0.0f);
            if (all) {
                // the next pending scale, by every warp for itself (the same sums in the same order)
                const df N = warp_sum(lane < nw ? red[0][lane] : z) * df_from(p.cell);
                const bool ok = isfinite(N.hi) && N.hi > 0.0f;
                ds[0] = ds[1] = ds[2] = ok ? df_rsqrt(N).hi : 1.0f;
            } else if (warp == 0) {
                // Eq. (DJ): a chain of FP64 square roots and quotients, by one warp for the block (every warp
                // for itself, they shared the FP64 pipe: 131 points 6.95 us a step against 6.26)
                df S[3], f[3];
                double d[3], N[3];
                bool finite;
#pragma unroll
                for (int j = 0; j < 3; j++) S[j] = warp_sum(lane < nw ? red[j][lane] : z);
                scale_from_df_sums(S, p.cell, renorm, p.mag, f, d, N, finite);
#pragma unroll
                for (int j = 0; j < 3; j++)
                    if (lane == j) dsh[j] = f[j].hi;
            }
            __syncthreads();  // red is free for the next step's sums
            if (!all) {
#pragma unroll
                for (int j = 0; j < 3; j++) ds[j] = dsh[j];
            }
        } else if (!IMAG || !renorm) {
            ds[0] = ds[1] = ds[2] = 1.0f;
        }
    }
    if (in)
#pragma unroll
        for (int j = 0; j < 3; j++) A[j * nx + i] = pack(x[j]);
    if (i == 0) {
        double N[3], d[3];
        for (int j = 0; j < 3; j++) {
            double q = 0.0;
            for (int w = 0; w < nw; w++) q += df_to(red[j][w]);
            N[j] = q * p.cell;
        }
        const bool finite = isfinite(N[0]) && isfinite(N[1]) && isfinite(N[2]);
        renorm_factors(N, finite ? renorm : 0, p.mag, d);
        for (int j = 0; j < 3; j++) {
            sc->norms[j] = N[j];
            sc->scale[j] = d[j];
            sc->scale_f[j] = (float)d[j];
            sc->scale_l[j] = (float)(d[j] - (double)sc->scale_f[j]);
        }
        sc->scale_src = 0;
        if (!finite) sc->err |= 1;
        sc->step_idx = step0 + nsteps;
    }
}

}  // namespace sgpe
