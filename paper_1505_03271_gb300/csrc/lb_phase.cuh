// lb_phase.cuh -- arguments and one-cell collision of the two-launch FV step
// (k_fv_phase.cu).
#pragma once

#include "lb_internal.cuh"

namespace lbgb {

template <typename R>
struct PhaseArgs {
    StepArgs<R> s;
    R* h;            // [NQ][ny][pitch] advected field h^n (hg^n)
    R* hs;           // h* (hg*)
    R* b;            // f~ + Coll between steps, f~ + Coll - dt/2 A[h^n] within one
    const R* foldx;  // Axis::cell_weights of x and y
    const R* foldy;
    R k[2], kh[2];   // omh and omgh, and their halves
    R ctx;           // 3 hF a_x
    int early;       // let the next kernel's CTAs in while this one runs
};

// start: form h^n from the state; else one step (predictor and corrector)
cudaError_t launch_fv_phase(Prec p, bool thermal, const void* args, bool start, int sms, cudaStream_t s);

// The value a population has after it is stored and loaded again.
template <typename S> struct Round;
template <> struct Round<double> {
    __device__ static double of(double v) { return v; }
};
template <> struct Round<float> {
    __device__ static float of(float v) { return v; }
};
template <> struct Round<__half> {
    __device__ static float of(float v) { return __half2float(__float2half_rn(v * kF16Scale)) * (1.0f / kF16Scale); }
};
template <> struct Round<__nv_bfloat16> {
    __device__ static float of(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
};

// Moments of one cell and the changes t of its populations (h = d + t),
// with f_eq and F (Sec. II A, Eq. (F2)) regrouped into parts even and odd in
// c, as in PairMom (lb_pair.cuh), on base-state deviations:
//   f: t_a = k (w_a rp + 3 w_a c.(rho u) - d_a) + w_a rho (S + ct)
//   g: t_a = k (w_a Td + w_a T 3 c.u     - e_a) + w_a T S
// with ct = 3 hF c.a, S = 3 c.u (k/2 3 c.u + ct) - 1.5 k u.u - 3 hF u.a (no
// force in g's).
//
// A collision must not change mass, momentum (beyond the force) and heat, and
// a slow flow repeats the rounding that does so step after step.  So in FP32
// the linear part comes from the momentum rho u itself (rho (1 / rho) is off
// by 6e-8), its distance from d_a is formed first, by multiply-adds that leave
// one rounding of d_a's scale and none common to the populations, and the
// weights add up exactly: wsum to 1, wdir to 1/3 of c c (the nearest floats
// to 4/9, 1/9 and 1/36 add up to 1 + 7.5e-9).  Relative velocity error of 500
// FP32 steps of 64 x 64 decaying vortices: 1.2e-7, against 8.8e-6 for the
// paired tile; of 300 steps of a 100 x 90 box refined at its walls: 1.2e-7,
// against 3e-6 for the scalar tile.  FP64 takes the odd part with u.
template <typename R> __host__ __device__ constexpr R wsum(int a) { return wgt<R>(a); }
template <> __host__ __device__ constexpr float wsum<float>(int a) {
    return a == 0 ? 14913081.0f / 33554432.0f : (a <= 4 ? 14913081.0f / 134217728.0f : 3728270.0f / 134217728.0f);
}
static_assert(14913081LL + 14913081LL + 3728270LL == 33554432LL, "w_0 + 4 w_1 + 4 w_5 = 1");
// 3 w_a, with 2 wdir(1) + 4 wdir(5) = 1
template <typename R> __host__ __device__ constexpr R wdir(int a) { return R(3) * wgt<R>(a); }
template <> __host__ __device__ constexpr float wdir<float>(int a) {
    return a == 0 ? 0.0f : (a <= 4 ? 11184811.0f / 33554432.0f : 11184810.0f / 134217728.0f);
}
static_assert(2 * 11184811LL + 11184810LL == 33554432LL, "2 wdir(1) + 4 wdir(5) = 1");

template <typename R, bool TH>
struct CellMom {
    R rp, rho, ux3, uy3, mx, my, ay, uuneg, ua3neg, Td, T;  // mx = rho u_x

    __device__ __forceinline__ void build(const R* d, const R* e, const StepArgs<R>& A, R ro, R to) {
        const R e1 = d[1] - d[3], e2 = d[2] - d[4], e57 = d[5] - d[7], e68 = d[6] - d[8];
        rp = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])) + d[8];
        rho = rp + (R(1) + ro);
        const R ir = R(1) / rho;
        if constexpr (TH) {
            Td = ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7])) + e[8];
            const R dT0 = Td + to;
            T = dT0 + A.T0;
            ay = A.ay + A.bg * dT0;
        } else {
            ay = A.ay;
        }
        const R jx = (e1 + e57) - e68, jy = (e2 + e57) + e68;
        const R ux = jx * ir + A.hf * A.ax;
        const R uy = jy * ir + A.hf * ay;
        ux3 = R(3) * ux;
        uy3 = R(3) * uy;
        mx = my = 0;
        if constexpr (sizeof(R) == 4) {
            mx = jx + rho * (A.hf * A.ax);
            my = jy + rho * (A.hf * ay);
        }
        uuneg = R(-1.5) * (ux * ux + uy * uy);
        ua3neg = -(uy3 * ay + ux3 * A.ax);
    }

    __device__ __forceinline__ void change_f(const R* d, const PhaseArgs<R>& P, R* t) const {
        const R k = P.k[0], kh = P.kh[0], C0 = k * uuneg + P.s.hF * ua3neg, cty = R(3) * P.s.hF * ay;
        t[0] = k * (wsum<R>(0) * rp - d[0]) + (wgt<R>(0) * rho) * C0;
        const R w1 = wgt<R>(1) * rho, w5 = wgt<R>(5) * rho, m1 = wsum<R>(1) * rp, m5 = wsum<R>(5) * rp;
        pair(d, 1, ux3, wdir<R>(1), mx, k, kh, C0, P.ctx, m1, w1, t);
        pair(d, 2, uy3, wdir<R>(1), my, k, kh, C0, cty, m1, w1, t);
        pair(d, 5, ux3 + uy3, wdir<R>(5), mx + my, k, kh, C0, cty + P.ctx, m5, w5, t);
        pair(d, 6, uy3 - ux3, wdir<R>(5), my - mx, k, kh, C0, cty - P.ctx, m5, w5, t);
    }
    __device__ __forceinline__ void change_g(const R* e, const PhaseArgs<R>& P, R* t) const {
        const R k = P.k[1], kh = P.kh[1], C0 = k * uuneg;
        t[0] = k * (wsum<R>(0) * Td - e[0]) + (wgt<R>(0) * T) * C0;
        const R w1 = wgt<R>(1) * T, w5 = wgt<R>(5) * T, m1 = wsum<R>(1) * Td, m5 = wsum<R>(5) * Td;
        pair(e, 1, ux3, w1, ux3, k, kh, C0, R(0), m1, w1, t);
        pair(e, 2, uy3, w1, uy3, k, kh, C0, R(0), m1, w1, t);
        pair(e, 5, ux3 + uy3, w5, ux3 + uy3, k, kh, C0, R(0), m5, w5, t);
        pair(e, 6, uy3 - ux3, w5, uy3 - ux3, k, kh, C0, R(0), m5, w5, t);
    }
    // populations a and inv(a) = b, whose linear part is +- wl l
    static __device__ __forceinline__ void pair(const R* d, int a, R cu3, R wl, R l, R k, R kh, R C0, R ct, R m, R w,
                                                R* t) {
        const int b = inv(a);
        const R g = cu3 * kh + ct, S = cu3 * g + C0;
        if constexpr (sizeof(R) == 8) {  // one FP64 instruction less; its rounding does not show
            const R D = cu3 * kh + g;
            t[a] = k * (m - d[a]) + w * (S + D);
            t[b] = k * (m - d[b]) + w * (S - D);
            return;
        }
        t[a] = k * (wl * l + (m - d[a])) + w * (S + ct);
        t[b] = k * ((m - d[b]) - wl * l) + w * (S - ct);
    }
};

}  // namespace lbgb
