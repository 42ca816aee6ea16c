// lb_block.cuh -- the FV tile step on packed FP32 pairs (k_fv_ptile and the
// server's k_fv_ptile_batched).
//
// A CTA owns TX x TY cells: stage A forms h^n on tile + 4 and f~ + Coll on
// tile + 2, stage B (the predictor) f~* and h* on tile + 2, stage C (the
// corrector) f~^(n+1) on the tile; the fields live in shared memory as units
// of two floats.  On a flow grid a unit is two adjacent columns; on a thermal
// grid it is f and g of one column, whose stencils have the same weights and
// whose relaxations are one formula with two sets of coefficients.
//
// What bounds it is instruction issue and the shared-memory pipe, so:
//   - a thread takes a column of R rows: the y stencil reads R + 3 rows for R
//     cells instead of 5 R, and a face between two of its rows is formed once;
//   - the wall's ghost rows are written by the threads that hold the rows they
//     mirror, so a step has two barriers, not four.
// Step times before and after: channel 256 x 512 FP32 9.0 -> 7.7 us (32 x 14),
// 512 x 512 16.3 -> 13.9; thermal 16-bit 256 x 256 9.2 -> 7.6 (32 x 14, 512
// threads), 512 x 512 32 -> 27 (where the march of k_fv_blocks.cu takes 23).
#pragma once

#include "lb_chain.cuh"
#include "lb_lane.cuh"

namespace lbgb {
namespace block {

using namespace pairmath;

__device__ __forceinline__ V2 swap_sign_g(V2 v) { return mk(v.v.x, -v.v.y); }

// h* of one column from f~*, g~* in (f, g) units, in place.
__device__ __forceinline__ void relax_fg(V2* d, const StepArgs<float>& A, float ro, float to) {
    float f[Q], g[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        f[a] = d[a].v.x;
        g[a] = d[a].v.y;
    }
    LaneMom<true> m;
    m.build(f, g, A, ro, to);
    const float k1 = A.omh, k = A.omgh;
    const auto s = m.shared_f(A, k1, A.hF);
    const float w0 = wgt<float>(0), wA = wgt<float>(1), wD = wgt<float>(5);
    d[0] = mk(__fmaf_rn(__fmul_rn(m.rho, w0), s.C0, __fmaf_rn(s.k1c, f[0], __fmul_rn(m.rp, __fmul_rn(k1, w0)))),
              __fmaf_rn(k, __fmaf_rn(__fmul_rn(m.T, w0), m.uuneg, __fmul_rn(m.Td, w0)) - g[0], g[0]));
    auto two = [&](int a, float cu3, float ct, float w) {
        const int b = inv(a);
        m.pair_f(s, f[a], f[b], cu3, ct, __fmul_rn(m.rho, w), __fmul_rn(m.rp, __fmul_rn(k1, w)), d[a].v.x, d[b].v.x);
        m.pair_g(k, g[a], g[b], cu3, __fmul_rn(m.T, w), __fmul_rn(m.Td, w), d[a].v.y, d[b].v.y);
    };
    two(1, m.ux3, s.ctx, wA);
    two(2, m.uy3, s.cty, wA);
    two(5, m.ux3 + m.uy3, s.cty + s.ctx, wD);
    two(6, m.uy3 - m.ux3, s.cty - s.ctx, wD);
}

// x weights of a unit, both upwind directions: faces W, M, E of a column
// pair, or W and E (in M) of one column; 1/dx.
struct XW {
    float wp[3], mp[3], ep[3], wm[3], mm[3], em[3];
    V2 inv;
    __device__ __forceinline__ void load(const float4* p) {
        const float4 a = p[0], b = p[1], c = p[2], d = p[3], e = p[4];
        wp[0] = a.x; wp[1] = a.y; wp[2] = a.z; mp[0] = a.w; mp[1] = b.x; mp[2] = b.y;
        ep[0] = b.z; ep[1] = b.w; ep[2] = c.x; wm[0] = c.y; wm[1] = c.z; wm[2] = c.w;
        mm[0] = d.x; mm[1] = d.y; mm[2] = d.z; em[0] = d.w; em[1] = e.x; em[2] = e.y;
        inv = mk(e.z, e.w);
    }
};

// An x face value.  The order of operations is that of the scalar form
// w0 a + w1 b + w2 c as the compiler contracts it, so that every paired
// kernel gives the same bits.
__device__ __forceinline__ float face(const float* w, float a, float b, float c) {
    return __fmaf_rn(w[2], c, __fmaf_rn(w[0], a, __fmul_rn(w[1], b)));
}
__device__ __forceinline__ V2 face(const float* w, V2 a, V2 b, V2 c) {
    return fma2(bc(w[2]), c, fma2(bc(w[0]), a, bc(w[1]) * b));
}

// c (Phi_e - Phi_w) / dx of population velocity a for the unit at p, whose
// own value is known.
template <bool TH, int a>
__device__ __forceinline__ V2 xflux(const V2* p, V2 own, const XW& X) {
    if constexpr (TH) {
        const float *w = cx(a) > 0 ? X.wp : X.wm, *e = cx(a) > 0 ? X.mp : X.mm;
        const V2 n0 = cx(a) > 0 ? p[-2] : p[-1], n1 = cx(a) > 0 ? p[-1] : own, n2 = cx(a) > 0 ? own : p[1],
                 n3 = cx(a) > 0 ? p[1] : p[2];
        const V2 fw = face(w, n0, n1, n2), fe = face(e, n1, n2, n3);
        return (cx(a) > 0 ? fe - fw : fw - fe) * bc(X.inv.v.x);
    } else {
        const float2 P0 = p[-1].v, P1 = own.v, P2 = p[1].v;  // columns x-2 .. x+3
        if constexpr (cx(a) > 0) {
            const float fw = face(X.wp, P0.x, P0.y, P1.x), fm = face(X.mp, P0.y, P1.x, P1.y),
                        fe = face(X.ep, P1.x, P1.y, P2.x);
            return (mk(fm, fe) - mk(fw, fm)) * X.inv;
        } else {
            const float fw = face(X.wm, P0.y, P1.x, P1.y), fm = face(X.mm, P1.x, P1.y, P2.x),
                        fe = face(X.em, P1.y, P2.x, P2.y);
            return (mk(fw, fm) - mk(fm, fe)) * X.inv;
        }
    }
}

// y weights of R consecutive rows: the south face of the first and the north
// face of each (a north face is the next row's south face), c > 0 and c < 0;
// 1/dy; on thermal grids the base state's flux divergences c_y w A[ref]
// (before the weight w) as (f, g) units.
template <bool TH, int R>
struct YW {
    float p[R + 1][3], m[R + 1][3], inv[R], ro[R], to[R];
    V2 rp[R], rm[R];
    __device__ __forceinline__ void load(const float4* t) {  // 5 float4 per row
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 a = t[5 * r], b = t[5 * r + 1], c = t[5 * r + 2], d = t[5 * r + 3];
            if (r == 0) {
                p[0][0] = a.x; p[0][1] = a.y; p[0][2] = a.z;
                m[0][0] = b.z; m[0][1] = b.w; m[0][2] = c.x;
            }
            p[r + 1][0] = a.w; p[r + 1][1] = b.x; p[r + 1][2] = b.y;
            m[r + 1][0] = c.y; m[r + 1][1] = c.z; m[r + 1][2] = c.w;
            inv[r] = d.x;
            ro[r] = d.y;
            to[r] = d.z;
            if constexpr (TH) {
                const float4 e = t[5 * r + 4];
                rp[r] = mk(d.w, e.y);
                rm[r] = mk(e.x, e.z);
            }
        }
    }
};

// A[h] of population velocity a at a column of R units.  P is the unit's
// column in the population's plane, o[i] the offset of row i - 2 from the
// first of the R rows (i = 0 .. R + 3).
template <bool TH, int R, int a>
__device__ __forceinline__ void column_flux(const V2* P, const int* o, const XW& X, const YW<TH, R>& Y, V2* v) {
    if constexpr (cy(a) != 0) {
        constexpr int i0 = cy(a) > 0 ? 0 : 1;  // first row of the stencil
        V2 c[R + 3];
#pragma unroll
        for (int i = 0; i < R + 3; ++i) c[i] = P[o[i0 + i]];
        V2 south;
#pragma unroll
        for (int f = 0; f <= R; ++f) {
            const float* w = cy(a) > 0 ? Y.p[f] : Y.m[f];
            const V2 face = fma2(bc(w[0]), c[f], fma2(bc(w[1]), c[f + 1], bc(w[2]) * c[f + 2]));
            if (f > 0) {
                V2 b = bc(0.0f);
                if constexpr (cx(a) != 0) b = xflux<TH, a>(P + o[f + 1], c[f + 1 - i0], X);
                b = cy(a) > 0 ? fma2(face - south, bc(Y.inv[f - 1]), b) : b - (face - south) * bc(Y.inv[f - 1]);
                if constexpr (TH) {
                    const V2 r = cy(a) > 0 ? Y.rp[f - 1] : Y.rm[f - 1];
                    constexpr float cw = float(cy(a)) * wgt<float>(a);
                    b = b + mk(__fmul_rn(cw, r.v.x), __fmul_rn(cw, r.v.y));
                }
                v[f - 1] = b;
            }
            south = face;
        }
    } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = xflux<TH, a>(P + o[r + 2], P[o[r + 2]], X);
    }
}

template <bool TH, int R, int a, typename F>
__device__ __forceinline__ void for_flux(const V2* P, int plane, const int* o, const XW& X, const YW<TH, R>& Y,
                                         F&& use) {
    V2 v[R];
    if constexpr (a == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = bc(0.0f);
    } else {
        column_flux<TH, R, a>(P + a * plane, o, X, Y, v);
    }
    use(a, v);
    if constexpr (a + 1 < Q) for_flux<TH, R, a + 1>(P, plane, o, X, Y, use);
}

template <bool TH, int TX, int TY>
struct Geo {
    static constexpr int UC = TH ? 1 : 2;  // columns per unit
    static constexpr int UW = TX / UC, EW = (TX + 8) / UC, BW = (TX + 4) / UC, EH = TY + 8, BH = TY + 4;
    static constexpr int NE = EW * EH, NB = BW * BH;
    static constexpr size_t smem = sizeof(V2) * Q * (NE + 2 * NB) + sizeof(float4) * 5 * (BH + BW);
};

// Ghost rows of a wall on y: row gy of a region (its first row is grid row
// gy0, H rows, row stride W) mirrors into -1 - gy and 2 ny - 1 - gy.  h'_a =
// h'_inv(a) for f and -h'_inv(a) for g.  put(a, row) writes value a's image.
template <typename F>
__device__ __forceinline__ void mirror_rows(int gy, int gy0, int H, const StepArgs<float>& A, F put) {
    if (A.bcy != LB_BC_WALLS) return;
    if (gy <= 1) {
        const int e = -1 - gy - gy0;
        if (e >= 0 && e < H) put(e);
    }
    if (gy >= A.ny - 2) {
        const int e = 2 * A.ny - 1 - gy - gy0;
        if (e >= 0 && e < H) put(e);
    }
}

template <typename S, bool TH, int TX, int TY, int NTH, int RC>
__device__ __forceinline__ void tile_step(const StepArgs<float>& A, const int x0, const int y0) {
    using G = Geo<TH, TX, TY>;
    constexpr int UC = G::UC, UW = G::UW, EW = G::EW, BW = G::BW, EH = G::EH, BH = G::BH, NE = G::NE, NB = G::NB;
    constexpr int RB = 2;
    static_assert(BH % RB == 0 && TY % RC == 0, "row blocks");
    static_assert(EW % 2 == 0 && NE % 2 == 0 && NB % 2 == 0, "16-byte stores of two units");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2* sH = reinterpret_cast<V2*>(smem_raw);  // [9][EH][EW] h^n
    V2* sFC = sH + Q * NE;                     // [9][BH][BW] f~ + Coll, then - dt/2 A[h^n] on the tile
    V2* sHs = sFC + Q * NB;                    // [9][BH][BW] h*
    float4* sRow = reinterpret_cast<float4*>(sHs + Q * NB);  // [BH][5] row entries of tile + 2
    float4* sCol = sRow + 5 * BH;                             // [BW][5] column entries of tile + 2
    const int nx = A.nx;
    const S* fin = static_cast<const S*>(A.fin);
    const S* gin = static_cast<const S*>(A.gin);

    for (int k = threadIdx.x; k < 5 * (BH + BW); k += NTH) {
        const int e = k / 5, part = k % 5;
        if (e < BH) {
            int gy;
            if (map_axis(y0 - 2 + e, A.ny, A.bcy, gy))
                sRow[k] = __ldg(reinterpret_cast<const float4*>(A.rowtab) + 5 * gy + part);
        } else {
            const int xu = x0 - 2 + UC * (e - BH);
            const int gxl = ((xu % nx) + nx) % nx;
            sCol[(e - BH) * 5 + part] = __ldg(reinterpret_cast<const float4*>(A.coltab) + 5 * gxl + part);
        }
    }

    chain_wait();

    // ---- A: time level n on tile + 4, two columns per thread ----
    constexpr int EP = (TX + 8) / 2;
    for (int k = threadIdx.x; k < EP * EH; k += NTH) {
        const int px = k % EP, ey = k / EP;
        int gy;
        if (!map_axis(y0 - 4 + ey, A.ny, A.bcy, gy)) continue;
        const int xu = x0 - 4 + 2 * px;
        const bool contiguous = xu >= 0 && xu + 1 < nx;
        const long long row = (long long)gy * A.pitch;
        V2 d[Q], e[Q];
        if (contiguous) {
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                d[a] = Chained<S>::two(fin + a * A.plane + row + xu);
                if constexpr (TH) e[a] = Chained<S>::two(gin + a * A.plane + row + xu);
            }
        } else {
            const int gxl = ((xu % nx) + nx) % nx, gxr = ((xu + 1) % nx + nx) % nx;
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                const S* b = fin + a * A.plane + row;
                d[a] = mk(Chained<S>::ld(b + gxl), Chained<S>::ld(b + gxr));
                if constexpr (TH) {
                    const S* bg = gin + a * A.plane + row;
                    e[a] = mk(Chained<S>::ld(bg + gxl), Chained<S>::ld(bg + gxr));
                }
            }
        }
        float ro = 0, to = 0;
        if constexpr (TH) {
            const float4 o = __ldg(reinterpret_cast<const float4*>(A.rowtab + 20 * gy) + 3);
            ro = o.y;
            to = o.z;
        }
        PairMom<TH> c;
        c.build(d, e, A, ro, to);
        const bool inB = px >= 1 && px < EP - 1 && ey >= 2 && ey < EH - 2;
        const int kh = ey * EW + px * (2 / UC), kb = (ey - 2) * BW + (px - 1) * (2 / UC);
        V2 h[Q], hg[Q];
        c.relax_f(d, A, A.omh, A.hF, h);
        if constexpr (TH) c.relax_g(e, A.omgh, hg);
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            if constexpr (!TH) sH[a * NE + kh] = h[a];
            else *reinterpret_cast<float4*>(sH + a * NE + kh) = make_float4(h[a].v.x, hg[a].v.x, h[a].v.y, hg[a].v.y);
        }
        mirror_rows(gy, y0 - 4, EH, A, [&](int er) {
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                if (cy(a) == 0) continue;
                V2* p = sH + inv(a) * NE + er * EW + kh % EW;
                if constexpr (!TH) *p = h[a];
                else *reinterpret_cast<float4*>(p) = make_float4(h[a].v.x, -hg[a].v.x, h[a].v.y, -hg[a].v.y);
            }
        });
        if (inB) {
            c.relax_f(d, A, A.om, A.cf, h);
            if constexpr (TH) c.relax_g(e, A.omg, hg);
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                if constexpr (!TH) sFC[a * NB + kb] = h[a];
                else *reinterpret_cast<float4*>(sFC + a * NB + kb) = make_float4(h[a].v.x, hg[a].v.x, h[a].v.y, hg[a].v.y);
            }
        }
    }
    __syncthreads();

    // ---- B: predictor on tile + 2, RB rows of a unit column per thread ----
    for (int k = threadIdx.x; k < BW * (BH / RB); k += NTH) {
        const int bx = k % BW, by = RB * (k / BW);
        XW X;
        X.load(sCol + 5 * bx);
        YW<TH, RB> Y;
        Y.load(sRow + 5 * by);
        const V2* P = sH + (by + 2) * EW + bx + 2 / UC;
        const int kb = by * BW + bx;
        const bool colt = bx >= 2 / UC && bx < BW - 2 / UC;
        V2 st[RB][Q];
        int o[RB + 4];
#pragma unroll
        for (int i = 0; i < RB + 4; ++i) o[i] = (i - 2) * EW;
        for_flux<TH, RB, 0>(P, NE, o, X, Y, [&](int a, const V2* v) {
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const V2 fc = sFC[a * NB + kb + r * BW];
                st[r][a] = fma2(bc(-A.dt), v[r], fc);
                if (colt && by + r >= 2 && by + r < BH - 2) sFC[a * NB + kb + r * BW] = fma2(bc(-A.hf), v[r], fc);
            }
        });
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            int gy;
            if (!map_axis(y0 - 2 + by + r, A.ny, A.bcy, gy)) continue;
            if constexpr (TH) {
                relax_fg(st[r], A, Y.ro[r], Y.to[r]);
            } else {
                PairMom<false> c;
                V2 h[Q];
                c.build(st[r], st[r], A, 0.0f, 0.0f);
                c.relax_f(st[r], A, A.omh, A.hF, h);
#pragma unroll
                for (int a = 0; a < Q; ++a) st[r][a] = h[a];
            }
#pragma unroll
            for (int a = 1; a < Q; ++a) sHs[a * NB + kb + r * BW] = st[r][a];
            mirror_rows(gy, y0 - 2, BH, A, [&](int er) {
#pragma unroll
                for (int a = 0; a < Q; ++a)
                    if (cy(a) != 0) sHs[inv(a) * NB + er * BW + bx] = TH ? swap_sign_g(st[r][a]) : st[r][a];
            });
        }
    }
    __syncthreads();

    // ---- C: corrector on the tile, RC rows of a unit column per thread ----
    S* fout = static_cast<S*>(A.fout);
    S* gout = static_cast<S*>(A.gout);
    for (int k = threadIdx.x; k < UW * (TY / RC); k += NTH) {
        const int tx = k % UW, ty = RC * (k / UW);
        const int gx = x0 + UC * tx, gy = y0 + ty;
        if (gx >= nx || gy >= A.ny) continue;
        XW X;
        X.load(sCol + 5 * (tx + 2 / UC));
        YW<TH, RC> Y;
        Y.load(sRow + 5 * (ty + 2));
        const int kb = (ty + 2) * BW + tx + 2 / UC;
        const long long at = (long long)gy * A.pitch + gx;
        const bool both = gx + 1 < nx;
        int o[RC + 4];
#pragma unroll
        for (int i = 0; i < RC + 4; ++i) o[i] = (i - 2) * BW;
        for_flux<TH, RC, 0>(sHs + kb, NB, o, X, Y, [&](int a, const V2* v) {
#pragma unroll
            for (int r = 0; r < RC; ++r) {
                if (r > 0 && gy + r >= A.ny) continue;
                const V2 o = fma2(bc(-A.hf), v[r], sFC[a * NB + kb + r * BW]);
                const long long q = a * A.plane + at + (long long)r * A.pitch;
                if constexpr (TH) {
                    Store<S>::st(fout + q, o.v.x);
                    Store<S>::st(gout + q, o.v.y);
                } else {
                    if (both) PairIO<S>::st(fout + q, o);
                    else Store<S>::st(fout + q, o.v.x);
                }
            }
        });
    }
}

}  // namespace block
}  // namespace lbgb
