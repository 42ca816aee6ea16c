// k_fv_pair.cu -- the FV time step (Sec. II B: Eqs. (semi), (semi-heun),
// QUICK faces of Sec. II B 3, double-reflection walls of Sec. II B 5) in
// tiles of packed FP32 pairs (Blackwell's f32x2 FMA, ADD and MUL):
//   k_fv_ptile            the tile step of lb_block.cuh;
//   k_fv_ptile_batched    the same over the server's request table;
//   k_fv_split_a / _c     a tile step in two launches.
// They serve x-periodic grids; grids with walls on x use the scalar kernels.
#include "lb_block.cuh"
#include "lb_launch.cuh"

namespace lbgb {

namespace {

using namespace pairmath;

// x metric of the thread's two columns: faces W (west of the left column),
// M (between them) and E (east of the right one), both upwind directions.
struct XPair {
    float wp[3], mp[3], ep[3];  // c > 0: nodes (k-2, k-1, k) of face k
    float wm[3], mm[3], em[3];  // c < 0: nodes (k-1, k, k+1)
    V2 inv;
};

// One row of the per-row table (20 floats, 80 bytes): QUICK weights of the
// row's south and north faces for both upwind directions, 1/dy, the base
// state offsets and the base state's y flux divergences.
struct YPair {
    V2 ps[3], pn[3], ms[3], mn[3], inv;
    float ro, to, dref[4];
};

__device__ __forceinline__ void load_row(const float* tab, int g, YPair& Y) {
    const float4* p = reinterpret_cast<const float4*>(tab + 20 * g);
    const float4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3), e = __ldg(p + 4);
    Y.ps[0] = bc(a.x); Y.ps[1] = bc(a.y); Y.ps[2] = bc(a.z);
    Y.pn[0] = bc(a.w); Y.pn[1] = bc(b.x); Y.pn[2] = bc(b.y);
    Y.ms[0] = bc(b.z); Y.ms[1] = bc(b.w); Y.ms[2] = bc(c.x);
    Y.mn[0] = bc(c.y); Y.mn[1] = bc(c.z); Y.mn[2] = bc(c.w);
    Y.inv = bc(d.x);
    Y.ro = d.y;
    Y.to = d.z;
    Y.dref[0] = d.w; Y.dref[1] = e.x; Y.dref[2] = e.y; Y.dref[3] = e.z;
}

// y flux divergence of the base state for population a (row data).
template <int a>
__device__ __forceinline__ float row_ref_flux(const YPair& Y, bool thermal) {
    if constexpr (cy(a) == 0) {
        return 0.0f;
    } else {
        return float(cy(a)) * wgt<float>(a) * Y.dref[(thermal ? 2 : 0) + (cy(a) > 0 ? 0 : 1)];
    }
}

}  // namespace

// x metric of the pair whose left column is g: from the per-column table
// (20 floats: wp at faces g, g+1, g_r+1; wm at the same faces; 1/dx of both).
__device__ __forceinline__ void load_col(const float* tab, int g, XPair& X) {
    const float4* p = reinterpret_cast<const float4*>(tab + 20 * g);
    const float4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2), d = __ldg(p + 3), e = __ldg(p + 4);
    X.wp[0] = a.x; X.wp[1] = a.y; X.wp[2] = a.z;
    X.mp[0] = a.w; X.mp[1] = b.x; X.mp[2] = b.y;
    X.ep[0] = b.z; X.ep[1] = b.w; X.ep[2] = c.x;
    X.wm[0] = c.y; X.wm[1] = c.z; X.wm[2] = c.w;
    X.mm[0] = d.x; X.mm[1] = d.y; X.mm[2] = d.z;
    X.em[0] = d.w; X.em[1] = e.x; X.em[2] = e.y;
    X.inv = mk(e.z, e.w);
}

// Flux divergence of population a at pair-cell (px, y) of a region plane
// with row stride W pairs.
template <int a>
__device__ __forceinline__ V2 advect_region(const V2* plane, int W, int px, int y, const XPair& X, const YPair& Y) {
    V2 v = bc(0.0f);
    if constexpr (cx(a) != 0) {
        const V2* row = plane + y * W;
        const float2 P0 = row[px - 1].v, P1 = row[px].v, P2 = row[px + 1].v;
        float fw, fm, fe;
        if constexpr (cx(a) > 0) {
            fw = X.wp[0] * P0.x + X.wp[1] * P0.y + X.wp[2] * P1.x;
            fm = X.mp[0] * P0.y + X.mp[1] * P1.x + X.mp[2] * P1.y;
            fe = X.ep[0] * P1.x + X.ep[1] * P1.y + X.ep[2] * P2.x;
        } else {
            fw = X.wm[0] * P0.y + X.wm[1] * P1.x + X.wm[2] * P1.y;
            fm = X.mm[0] * P1.x + X.mm[1] * P1.y + X.mm[2] * P2.x;
            fe = X.em[0] * P1.y + X.em[1] * P2.x + X.em[2] * P2.y;
        }
        const V2 dx = (mk(fm, fe) - mk(fw, fm)) * X.inv;
        v = cx(a) > 0 ? dx : v - dx;
    }
    if constexpr (cy(a) != 0) {
        V2 c[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) c[i] = plane[(y - 2 + i) * W + px];
        if constexpr (cy(a) > 0) {
            const V2 fn = fma2(Y.pn[0], c[1], fma2(Y.pn[1], c[2], Y.pn[2] * c[3]));
            const V2 fs = fma2(Y.ps[0], c[0], fma2(Y.ps[1], c[1], Y.ps[2] * c[2]));
            v = fma2(fn - fs, Y.inv, v);
        } else {
            const V2 fn = fma2(Y.mn[0], c[2], fma2(Y.mn[1], c[3], Y.mn[2] * c[4]));
            const V2 fs = fma2(Y.ms[0], c[1], fma2(Y.ms[1], c[2], Y.ms[2] * c[3]));
            v = v - (fn - fs) * Y.inv;
        }
    }
    return v;
}

template <bool TH, int NQ, int H, int W, int a>
__device__ __forceinline__ void advect_region_all(const V2* P, int px, int y, const XPair& X, const YPair& Y,
                                                  V2* out) {
    out[a] = advect_region<a>(P + a * H * W, W, px, y, X, Y) + bc(row_ref_flux<a>(Y, false));
    if constexpr (TH) out[Q + a] = advect_region<a>(P + (Q + a) * H * W, W, px, y, X, Y) + bc(row_ref_flux<a>(Y, true));
    if constexpr (a + 1 < Q) advect_region_all<TH, NQ, H, W, a + 1>(P, px, y, X, Y, out);
}

// Ghost rows of a region (walls on y), own pair-columns: h'_a = h'_inv(a)
// for f, -h'_inv(a) for g.
template <bool TH, int NQ, int H, int W>
__device__ __forceinline__ void ghost_rows_region(V2* P, int gy0, const StepArgs<float>& A) {
    if (A.bcy != LB_BC_WALLS) return;
    for (int k = threadIdx.x; k < W * 4; k += blockDim.x) {
        const int px = k % W, which = k / W;
        const int kk = (which & 1) + 1;
        const bool bot = which < 2;
        const int gy = bot ? -kk : A.ny - 1 + kk;
        const int gys = bot ? kk - 1 : A.ny - kk;
        const int ey = gy - gy0, eys = gys - gy0;
        if (ey < 0 || ey >= H) continue;
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            P[(a * H + ey) * W + px] = P[(inv(a) * H + eys) * W + px];
            if constexpr (TH) P[((Q + a) * H + ey) * W + px] = bc(0.0f) - P[((Q + inv(a)) * H + eys) * W + px];
        }
    }
}

template <typename S, bool TH, int TX, int TY, int NTH, int MINB, int RC>
__global__ void __launch_bounds__(NTH, MINB) k_fv_ptile(const StepArgs<float> A) {
    block::tile_step<S, TH, TX, TY, NTH, RC>(A, blockIdx.x * TX, blockIdx.y * TY);
}

// ---- split schedule: two kernels per step ----
// The fused tile recomputes the collision on tile + 4 and the predictor on
// tile + 2.  Here the first kernel computes the collision on tile + 2 and the
// predictor on the tile only, and hands h* and f~ + Coll - dt/2 A[h^n] to
// the second kernel through global memory (L2 on small grids); the second
// reads h* on tile + 2 and applies the corrector.  Halo work drops from
// 1.875x and 1.41x to 1.41x and 1x, and shared memory from three regions
// to one per kernel, at the price of a second launch and 72 B (144 B with
// g) per cell through L2.
template <typename S, bool TH, int TX, int TY, int NTH>
__global__ void __launch_bounds__(NTH) k_fv_split_a(const StepArgs<float> A) {
    constexpr int NQ = TH ? 2 * Q : Q;
    constexpr int BW = (TX + 4) / 2, BH = TY + 4, NB = BW * BH;
    constexpr int TW = TX / 2, NT = TW * TY;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2* sH = reinterpret_cast<V2*>(smem_raw);  // [NQ][BH][BW] h^n on tile + 2
    V2* sFC = sH + NQ * NB;                    // [NQ][TY][TW] f~ + Coll on the tile
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, nx = A.nx;
    const S* fin = static_cast<const S*>(A.fin);
    const S* gin = static_cast<const S*>(A.gin);
    for (int k = threadIdx.x; k < NB; k += NTH) {
        const int px = k % BW, ey = k / BW;
        int gy;
        if (!map_axis(y0 - 2 + ey, A.ny, A.bcy, gy)) continue;
        const int xu = x0 - 2 + 2 * px;
        const int gxl = ((xu % nx) + nx) % nx, gxr = ((xu + 1) % nx + nx) % nx;
        const bool contiguous = xu >= 0 && xu + 1 < nx;
        const long long row = (long long)gy * A.pitch;
        V2 d[Q], e[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            const S* b = fin + a * A.plane + row;
            d[a] = contiguous ? PairIO<S>::ld(b + xu) : mk(Store<S>::ld(b + gxl), Store<S>::ld(b + gxr));
            if constexpr (TH) {
                const S* bg = gin + a * A.plane + row;
                e[a] = contiguous ? PairIO<S>::ld(bg + xu) : mk(Store<S>::ld(bg + gxl), Store<S>::ld(bg + gxr));
            }
        }
        const float4 o = __ldg(reinterpret_cast<const float4*>(A.rowtab + 20 * gy) + 3);
        PairMom<TH> c;
        c.build(d, e, A, o.y, TH ? o.z : 0.0f);
        const bool inT = px >= 1 && px < BW - 1 && ey >= 2 && ey < BH - 2;
        const int kt = (ey - 2) * TW + (px - 1);
        V2 hv[Q], hg[Q];
        c.relax_f(d, A, A.omh, A.hF, hv);
        if constexpr (TH) c.relax_g(e, A.omgh, hg);
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            sH[a * NB + k] = hv[a];
            if constexpr (TH) sH[(Q + a) * NB + k] = hg[a];
        }
        if (inT) {
            V2 pv[Q], pg[Q];
            c.relax_f(d, A, A.om, A.cf, pv);
            if constexpr (TH) c.relax_g(e, A.omg, pg);
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                sFC[a * NT + kt] = pv[a];
                if constexpr (TH) sFC[(Q + a) * NT + kt] = pg[a];
            }
        }
    }
    __syncthreads();
    ghost_rows_region<TH, NQ, BH, BW>(sH, y0 - 2, A);
    __syncthreads();
    for (int k = threadIdx.x; k < NT; k += NTH) {
        const int tx = k % TW, ty = k / TW;
        const int gx = x0 + 2 * tx, gy = y0 + ty;
        if (gx >= nx || gy >= A.ny) continue;
        XPair X;
        load_col(A.coltab, gx, X);
        YPair Y;
        load_row(A.rowtab, gy, Y);
        V2 adv[NQ];
        advect_region_all<TH, NQ, BH, BW, 0>(sH, tx + 1, ty + 2, X, Y, adv);
        const long long at = (long long)gy * A.pitch + gx;
        const bool both = gx + 1 < nx;
        V2 fs[Q], es[Q];
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
            const V2 fc = sFC[a * NT + k];
            const V2 fcb = fma2(bc(-A.hf), adv[a], fc);
            float* p = A.xfc + a * A.plane + at;
            if (both) PairIO<float>::st(p, fcb);
            else *p = fcb.v.x;
            const V2 st = fma2(bc(-A.dt), adv[a], fc);
            if (a < Q) fs[a] = st;
            else if constexpr (TH) es[a - Q] = st;
        }
        PairMom<TH> c;
        c.build(fs, es, A, Y.ro, TH ? Y.to : 0.0f);
        V2 hv[Q], hgv[Q];
        c.relax_f(fs, A, A.omh, A.hF, hv);
        if constexpr (TH) c.relax_g(es, A.omgh, hgv);
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            float* p = A.xh + a * A.plane + at;
            if (both) PairIO<float>::st(p, hv[a]);
            else *p = hv[a].v.x;
            if constexpr (TH) {
                float* q = A.xh + (Q + a) * A.plane + at;
                if (both) PairIO<float>::st(q, hgv[a]);
                else *q = hgv[a].v.x;
            }
        }
    }
}

template <typename S, bool TH, int TX, int TY, int NTH>
__global__ void __launch_bounds__(NTH) k_fv_split_c(const StepArgs<float> A) {
    constexpr int NQ = TH ? 2 * Q : Q;
    constexpr int BW = (TX + 4) / 2, BH = TY + 4, NB = BW * BH;
    constexpr int TW = TX / 2, NT = TW * TY;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2* sHs = reinterpret_cast<V2*>(smem_raw);  // [NQ][BH][BW] h* on tile + 2
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, nx = A.nx;
    for (int k = threadIdx.x; k < NB; k += NTH) {
        const int px = k % BW, ey = k / BW;
        int gy;
        if (!map_axis(y0 - 2 + ey, A.ny, A.bcy, gy)) continue;
        const int xu = x0 - 2 + 2 * px;
        const int gxl = ((xu % nx) + nx) % nx, gxr = ((xu + 1) % nx + nx) % nx;
        const bool contiguous = xu >= 0 && xu + 1 < nx;
        const long long row = (long long)gy * A.pitch;
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
            const float* b = A.xh + a * A.plane + row;
            sHs[a * NB + k] = contiguous ? PairIO<float>::ld(b + xu) : mk(__ldg(b + gxl), __ldg(b + gxr));
        }
    }
    __syncthreads();
    ghost_rows_region<TH, NQ, BH, BW>(sHs, y0 - 2, A);
    __syncthreads();
    S* fout = static_cast<S*>(A.fout);
    S* gout = static_cast<S*>(A.gout);
    for (int k = threadIdx.x; k < NT; k += NTH) {
        const int tx = k % TW, ty = k / TW;
        const int gx = x0 + 2 * tx, gy = y0 + ty;
        if (gx >= nx || gy >= A.ny) continue;
        XPair X;
        load_col(A.coltab, gx, X);
        YPair Y;
        load_row(A.rowtab, gy, Y);
        V2 adv[NQ];
        advect_region_all<TH, NQ, BH, BW, 0>(sHs, tx + 1, ty + 2, X, Y, adv);
        const long long at = (long long)gy * A.pitch + gx;
        const bool both = gx + 1 < nx;
#pragma unroll
        for (int a = 0; a < NQ; ++a) {
            const float* p = A.xfc + a * A.plane + at;
            const V2 fcb = both ? PairIO<float>::ld(p) : mk(__ldg(p), 0.0f);
            const V2 o = fma2(bc(-A.hf), adv[a], fcb);
            S* base = (a < Q ? fout + a * A.plane : gout + (a - Q) * A.plane) + at;
            if (both) PairIO<S>::st(base, o);
            else Store<S>::st(base, o.v.x);
        }
    }
}

template <typename S, bool TH, int TX, int TY, int NTH>
static cudaError_t run_split(const void* vargs, cudaStream_t s) {
    const StepArgs<float>& A = *static_cast<const StepArgs<float>*>(vargs);
    constexpr int NQ = TH ? 2 * Q : Q;
    constexpr size_t smem_a = sizeof(V2) * NQ * (((TX + 4) / 2) * (TY + 4) + (TX / 2) * TY);
    constexpr size_t smem_c = sizeof(V2) * NQ * ((TX + 4) / 2) * (TY + 4);
    static_assert(smem_a <= 232448, "shared memory per CTA");
    {
        cudaError_t e = set_max_smem((const void*)k_fv_split_a<S, TH, TX, TY, NTH>, (int)smem_a);
        if (e == cudaSuccess) e = set_max_smem((const void*)k_fv_split_c<S, TH, TX, TY, NTH>, (int)smem_c);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((A.nx + TX - 1) / TX, (A.ny + TY - 1) / TY);
    k_fv_split_a<S, TH, TX, TY, NTH><<<grid, NTH, smem_a, s>>>(A);
    count_launch();
    k_fv_split_c<S, TH, TX, TY, NTH><<<grid, NTH, smem_c, s>>>(A);
    count_launch();
    return cudaGetLastError();
}

template <typename S, bool TH>
static cudaError_t run_split_shape(const void* args, int shape, cudaStream_t s) {
    if (shape == 16) return run_split<S, TH, 16, 16, 128>(args, s);
    return run_split<S, TH, 32, 16, 256>(args, s);
}

cudaError_t launch_fv_split(Prec p, bool th, const void* args, int shape, cudaStream_t s) {
    switch (p) {
        case Prec::F32:
            return th ? run_split_shape<float, true>(args, shape, s) : run_split_shape<float, false>(args, shape, s);
        case Prec::F16:
            return th ? run_split_shape<__half, true>(args, shape, s) : run_split_shape<__half, false>(args, shape, s);
        case Prec::BF16:
            return th ? run_split_shape<__nv_bfloat16, true>(args, shape, s)
                      : run_split_shape<__nv_bfloat16, false>(args, shape, s);
        default: return cudaErrorInvalidValue;
    }
}

// Many grids in one launch (the serving path): CTA b steps tile tiles[b] =
// (request, tile x, tile y) with that request's parameters, picking its
// input buffer from step k of the launch sequence; requests with fewer than
// k + 1 steps left are skipped.  Same tile code whatever else is batched.
template <typename S, bool TH, int TX, int TY, int NTH>
__global__ void __launch_bounds__(NTH)
k_fv_ptile_batched(const BatchReq<float>* reqs, const int4* tiles, const int* ntiles, const int k) {
    const bool listed = (int)blockIdx.x < *ntiles;
    const int4 t = tiles[listed ? blockIdx.x : 0];
    const BatchReq<float>& B = reqs[t.x];
    if (!listed || k >= B.remaining) {
        chain_wait();
        return;
    }
    StepArgs<float> A = B.args;
    const int p = (B.parity + k) & 1;
    A.fin = B.f[p];
    A.fout = B.f[p ^ 1];
    A.gin = B.g[p];
    A.gout = B.g[p ^ 1];
    block::tile_step<S, TH, TX, TY, NTH, TH ? 1 : 2>(A, t.y * TX, t.z * TY);
}

// Thermal tiles use 512 threads (one CTA per SM by shared memory, a thread
// takes f and g of a column as one unit), flow tiles 256.
template <typename S, bool TH>
static cudaError_t run_ptile_batched(const void* reqs, const int4* tiles, const int* ntiles, int capacity, int k,
                                     cudaStream_t s) {
    constexpr int NTH = TH ? 512 : 256;
    constexpr size_t smem = block::Geo<TH, 32, 16>::smem;
    {
        cudaError_t e = set_max_smem((const void*)k_fv_ptile_batched<S, TH, 32, 16, NTH>, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const cudaError_t e = launch_chained(k_fv_ptile_batched<S, TH, 32, 16, NTH>, dim3(capacity), NTH, smem, s,
                                         static_cast<const BatchReq<float>*>(reqs), tiles, ntiles, k);
    count_launch();
    return e;
}

cudaError_t launch_fv_ptile_batched(Prec p, bool th, const void* reqs, const int4* tiles, const int* ntiles,
                                    int capacity, int k, cudaStream_t s) {
    switch (p) {
        case Prec::F32:
            return th ? run_ptile_batched<float, true>(reqs, tiles, ntiles, capacity, k, s)
                      : run_ptile_batched<float, false>(reqs, tiles, ntiles, capacity, k, s);
        case Prec::F16:
            return th ? run_ptile_batched<__half, true>(reqs, tiles, ntiles, capacity, k, s)
                      : run_ptile_batched<__half, false>(reqs, tiles, ntiles, capacity, k, s);
        case Prec::BF16:
            return th ? run_ptile_batched<__nv_bfloat16, true>(reqs, tiles, ntiles, capacity, k, s)
                      : run_ptile_batched<__nv_bfloat16, false>(reqs, tiles, ntiles, capacity, k, s);
        default: return cudaErrorInvalidValue;
    }
}

template <typename S, bool TH, int TX, int TY, int NTH, int MINB, int RC>
static cudaError_t run_ptile(const void* vargs, cudaStream_t s) {
    const StepArgs<float>& A = *static_cast<const StepArgs<float>*>(vargs);
    constexpr size_t smem = block::Geo<TH, TX, TY>::smem;
    static_assert(smem <= 232448, "shared memory per CTA");
    {
        cudaError_t e = set_max_smem((const void*)k_fv_ptile<S, TH, TX, TY, NTH, MINB, RC>, (int)smem);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((A.nx + TX - 1) / TX, (A.ny + TY - 1) / TY);
    const cudaError_t e = launch_chained(k_fv_ptile<S, TH, TX, TY, NTH, MINB, RC>, grid, NTH, smem, s, A);
    count_launch();
    return e;
}

// shape: 0 = 32 x 16 tiles, 256 threads; 14 = 32 x 14, 256 threads;
// 16 = 16 x 16, 128 threads; 512 = 32 x 16, 512 threads; 526 = 32 x 14,
// 512 threads.  The 14-row tiles let a 512-row grid fill two CTAs on
// nearly every SM (296 tiles for 256 columns) instead of 256 tiles on 152.
template <typename S, bool TH>
static cudaError_t run_ptile_shape(const void* args, int shape, cudaStream_t s) {
    if (shape == 16) return run_ptile<S, TH, 16, 16, TH ? 256 : 128, 1, 2>(args, s);
    if (shape == 14) return run_ptile<S, TH, 32, 14, 256, 1, 2>(args, s);
    if (shape == 512) return run_ptile<S, TH, 32, 16, 512, TH ? 1 : 2, 1>(args, s);
    if (shape == 526) return run_ptile<S, TH, 32, 14, 512, TH ? 1 : 2, 1>(args, s);
    return run_ptile<S, TH, 32, 16, 256, 1, 2>(args, s);
}

cudaError_t launch_fv_ptile(Prec p, bool th, const void* args, int shape, cudaStream_t s) {
    switch (p) {
        case Prec::F32:
            return th ? run_ptile_shape<float, true>(args, shape, s) : run_ptile_shape<float, false>(args, shape, s);
        case Prec::F16:
            return th ? run_ptile_shape<__half, true>(args, shape, s) : run_ptile_shape<__half, false>(args, shape, s);
        case Prec::BF16:
            return th ? run_ptile_shape<__nv_bfloat16, true>(args, shape, s)
                      : run_ptile_shape<__nv_bfloat16, false>(args, shape, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbgb
