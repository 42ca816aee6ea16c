// lb_lane.cuh -- the FV relaxation of one cell in FP32, with the roundings of
// the paired one (PairMom, lb_pair.cuh).
#pragma once

#include "lb_pair.cuh"

namespace lbgb {
namespace pairmath {

// One lane of PairMom: the same operations in the same order, so that a
// kernel that holds a cell's populations otherwise rounds as the paired ones
// do.
template <bool TH>
struct LaneMom {
    float rp, rho, ux3, uy3, ay, uuneg, ua3neg, Td, T;

    __device__ __forceinline__ void build(const float* d, const float* e, const StepArgs<float>& A, float ro,
                                          float to) {
        const float e1 = d[1] - d[3], e2 = d[2] - d[4], e57 = d[5] - d[7], e68 = d[6] - d[8];
        rp = ((d[0] + d[1]) + (d[2] + d[3])) + ((d[4] + d[5]) + (d[6] + d[7])) + d[8];
        const float jx = (e1 + e57) - e68, jy = (e2 + e57) + e68;
        rho = rp + (1.0f + ro);
        const float ir = __fdividef(1.0f, rho);
        if constexpr (TH) {
            Td = ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7])) + e[8];
            const float dT0 = Td + to;
            T = dT0 + A.T0;
            ay = __fmaf_rn(A.bg, dT0, A.ay);
        } else {
            ay = A.ay;
        }
        const float ux = __fmaf_rn(jx, ir, __fmul_rn(A.hf, A.ax));
        const float uy = __fmaf_rn(ay, A.hf, __fmul_rn(jy, ir));
        ux3 = __fmul_rn(ux, 3.0f);
        uy3 = __fmul_rn(uy, 3.0f);
        uuneg = __fmul_rn(__fmaf_rn(ux, ux, __fmul_rn(uy, uy)), -1.5f);
        ua3neg = -__fmaf_rn(uy3, ay, __fmul_rn(ux3, A.ax));
    }

    // The parts of a relaxation that its populations share.
    struct F {
        float k1h, k1c, C0, ctx, cty;
    };
    __device__ __forceinline__ F shared_f(const StepArgs<float>& A, float k1, float k2) const {
        return {0.5f * k1, 1.0f - k1, __fmaf_rn(k1, uuneg, __fmul_rn(k2, ua3neg)),
                __fmul_rn(__fmul_rn(3.0f, k2), A.ax), __fmul_rn(ay, __fmul_rn(3.0f, k2))};
    }
    // populations a (of 1, 2, 5, 6) and inv(a); w = w_a
    static __device__ __forceinline__ void pair_f(const F& f, float da, float db, float cu3, float ct, float wr,
                                                  float bb, float& oa, float& ob) {
        const float g = __fmaf_rn(cu3, f.k1h, ct);
        const float S = __fmaf_rn(cu3, g, f.C0), D = __fmaf_rn(cu3, f.k1h, g);
        oa = __fmaf_rn(wr, S + D, __fmaf_rn(f.k1c, da, bb));
        ob = __fmaf_rn(wr, S - D, __fmaf_rn(f.k1c, db, bb));
    }
    __device__ __forceinline__ void pair_g(float k, float ea, float eb, float cu3, float wT, float wTd, float& oa,
                                           float& ob) const {
        const float q = __fmaf_rn(__fmul_rn(cu3, 0.5f), cu3, uuneg);
        oa = __fmaf_rn(k, __fmaf_rn(wT, cu3 + q, wTd) - ea, ea);
        ob = __fmaf_rn(k, __fmaf_rn(wT, q - cu3, wTd) - eb, eb);
    }
    // one population: relax_f and relax_g of PairMom
    __device__ __forceinline__ float cu3_of(int a) const {
        return a == 1 || a == 3 ? ux3 : a == 2 || a == 4 ? uy3 : a == 5 || a == 7 ? ux3 + uy3 : uy3 - ux3;
    }
    __device__ __forceinline__ float one_f(int a, float d, const StepArgs<float>& A, float k1, float k2) const {
        const F f = shared_f(A, k1, k2);
        const float w = a == 0 ? wgt<float>(0) : a <= 4 ? wgt<float>(1) : wgt<float>(5);
        const float wr = __fmul_rn(rho, w), rest = __fmaf_rn(f.k1c, d, __fmul_rn(rp, __fmul_rn(k1, w)));
        if (a == 0) return __fmaf_rn(wr, f.C0, rest);
        const float ct = a == 1 || a == 3   ? f.ctx
                         : a == 2 || a == 4 ? f.cty
                         : a == 5 || a == 7 ? f.cty + f.ctx
                                            : f.cty - f.ctx;
        const float cu3 = cu3_of(a);
        const float g = __fmaf_rn(cu3, f.k1h, ct);
        const float S = __fmaf_rn(cu3, g, f.C0), D = __fmaf_rn(cu3, f.k1h, g);
        return __fmaf_rn(wr, a == 1 || a == 2 || a == 5 || a == 6 ? S + D : S - D, rest);
    }
    __device__ __forceinline__ float one_g(int a, float e, float k) const {
        const float w = a == 0 ? wgt<float>(0) : a <= 4 ? wgt<float>(1) : wgt<float>(5);
        const float wT = __fmul_rn(T, w), wTd = __fmul_rn(Td, w);
        if (a == 0) return __fmaf_rn(k, __fmaf_rn(wT, uuneg, wTd) - e, e);
        const float cu3 = cu3_of(a), q = __fmaf_rn(__fmul_rn(cu3, 0.5f), cu3, uuneg);
        return __fmaf_rn(k, __fmaf_rn(wT, a == 1 || a == 2 || a == 5 || a == 6 ? cu3 + q : q - cu3, wTd) - e, e);
    }
};

}  // namespace pairmath
}  // namespace lbgb
