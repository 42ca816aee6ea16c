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
// Every rounding is written out: a call forms h of its first state in another
// kernel than the steps before it did, and a run has the same bits however it
// is split into calls only if no compiler chooses which products are fused.
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
            ay = __fma_rn(A.bg, dT0, A.ay);
        } else {
            ay = A.ay;
        }
        const double ux = __fma_rn((e1 + e57) - e68, ir, __dmul_rn(A.hf, A.ax));
        const double uy = __fma_rn((e2 + e57) + e68, ir, __dmul_rn(A.hf, ay));
        ux3 = __dmul_rn(3.0, ux);
        uy3 = __dmul_rn(3.0, uy);
        uuneg = __dmul_rn(-1.5, __fma_rn(ux, ux, __dmul_rn(uy, uy)));
        ua3neg = -__fma_rn(uy3, ay, __dmul_rn(ux3, A.ax));
    }

    // the parts that the populations share: C0 of f and of g, and 3 hF a_y
    __device__ __forceinline__ double c0_f(const PhaseArgs<double>& P) const {
        return __fma_rn(P.k[0], uuneg, __dmul_rn(P.s.hF, ua3neg));
    }
    __device__ __forceinline__ double c0_g(const PhaseArgs<double>& P) const { return __dmul_rn(P.k[1], uuneg); }
    __device__ __forceinline__ double cty(const PhaseArgs<double>& P) const {
        return __dmul_rn(__dmul_rn(3.0, P.s.hF), ay);
    }

    // Even and odd part: cu3 = 3 c.u, ct = 3 hF c.a; for -c the odd one changes
    // sign.  t takes their sum.
    static __device__ __forceinline__ void parts(double cu3, double ct, double kh, double C0, double& S, double& D) {
        const double g = __fma_rn(cu3, kh, ct);
        S = __fma_rn(cu3, g, C0);
        D = __fma_rn(cu3, kh, g);
    }
    static __device__ __forceinline__ double change(double d, double sum, double k, double w, double m0, double m1) {
        return __fma_rn(__dmul_rn(w, m1), sum, __dmul_rn(k, __fma_rn(w, m0, -d)));
    }

    __device__ __forceinline__ void change_f(const double* d, const PhaseArgs<double>& P, double* t) const {
        changes(d, P.k[0], P.kh[0], c0_f(P), P.ctx, cty(P), rp, rho, t);
    }
    __device__ __forceinline__ void change_g(const double* e, const PhaseArgs<double>& P, double* t) const {
        changes(e, P.k[1], P.kh[1], c0_g(P), 0.0, 0.0, Td, T, t);
    }

    __device__ __forceinline__ void changes(const double* d, double k, double kh, double C0, double ctx, double cty,
                                            double m0, double m1, double* t) const {
        t[0] = change(d[0], C0, k, wgt<double>(0), m0, m1);
        pair(d, 1, ux3, k, kh, C0, ctx, m0, m1, t);
        pair(d, 2, uy3, k, kh, C0, cty, m0, m1, t);
        pair(d, 5, ux3 + uy3, k, kh, C0, cty + ctx, m0, m1, t);
        pair(d, 6, uy3 - ux3, k, kh, C0, cty - ctx, m0, m1, t);
    }
    // populations a and inv(a)
    static __device__ __forceinline__ void pair(const double* d, int a, double cu3, double k, double kh, double C0,
                                                double ct, double m0, double m1, double* t) {
        double S, D;
        parts(cu3, ct, kh, C0, S, D);
        t[a] = change(d[a], S + D, k, wgt<double>(a), m0, m1);
        t[inv(a)] = change(d[inv(a)], S - D, k, wgt<double>(a), m0, m1);
    }
};

}  // namespace lbgb
