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

// Moments of one cell and the changes t of its populations in FP64 (h = d + t),
// with f_eq and F (Sec. II A, Eq. (F2)) regrouped into parts even and odd in
// c, as in PairMom (lb_pair.cuh, which states the algebra):
//   f: t_a = k (w_a rp - d_a) + w_a rho (S +- D)
//   g: the same with Td, T in place of rp, rho and no force.
template <bool TH>
struct CellMom {
    double rp, rho, ux3, uy3, ay, uuneg, ua3neg, Td, T;

    __device__ __forceinline__ void build(const double* d, const double* e, const StepArgs<double>& A, double ro,
                                          double to) {
        const double e1 = d[1] - d[3], e2 = d[2] - d[4], e57 = d[5] - d[7], e68 = d[6] - d[8];
        rp = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])) + d[8];
        rho = rp + (1.0 + ro);
        const double ir = 1.0 / rho;
        if constexpr (TH) {
            Td = ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7])) + e[8];
            const double dT0 = Td + to;
            T = dT0 + A.T0;
            ay = A.ay + A.bg * dT0;
        } else {
            ay = A.ay;
        }
        const double ux = ((e1 + e57) - e68) * ir + A.hf * A.ax;
        const double uy = ((e2 + e57) + e68) * ir + A.hf * ay;
        ux3 = 3.0 * ux;
        uy3 = 3.0 * uy;
        uuneg = -1.5 * (ux * ux + uy * uy);
        ua3neg = -(uy3 * ay + ux3 * A.ax);
    }

    __device__ __forceinline__ void change_f(const double* d, const PhaseArgs<double>& P, double* t) const {
        const double cty = 3.0 * P.s.hF * ay;
        change(d, P.k[0], P.kh[0], P.k[0] * uuneg + P.s.hF * ua3neg, P.ctx, cty, rp, rho, t);
    }
    __device__ __forceinline__ void change_g(const double* e, const PhaseArgs<double>& P, double* t) const {
        change(e, P.k[1], P.kh[1], P.k[1] * uuneg, 0.0, 0.0, Td, T, t);
    }

    __device__ __forceinline__ void change(const double* d, double k, double kh, double C0, double ctx, double cty,
                                           double m0, double m1, double* t) const {
        t[0] = (wgt<double>(0) * m1) * C0 + k * (wgt<double>(0) * m0 - d[0]);
        pair(d, 1, ux3, k, kh, C0, ctx, m0, m1, t);
        pair(d, 2, uy3, k, kh, C0, cty, m0, m1, t);
        pair(d, 5, ux3 + uy3, k, kh, C0, cty + ctx, m0, m1, t);
        pair(d, 6, uy3 - ux3, k, kh, C0, cty - ctx, m0, m1, t);
    }
    // populations a and inv(a) = b
    static __device__ __forceinline__ void pair(const double* d, int a, double cu3, double k, double kh, double C0,
                                                double ct, double m0, double m1, double* t) {
        const int b = inv(a);
        const double g = cu3 * kh + ct, S = cu3 * g + C0, D = cu3 * kh + g;
        const double w0 = wgt<double>(a) * m0, w1 = wgt<double>(a) * m1;
        t[a] = w1 * (S + D) + k * (w0 - d[a]);
        t[b] = w1 * (S - D) + k * (w0 - d[b]);
    }
};

}  // namespace lbgb
