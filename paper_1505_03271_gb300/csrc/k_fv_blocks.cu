// k_fv_blocks.cu -- the FV time step (Sec. II B: Eqs. (semi), (semi-heun),
// QUICK faces of Sec. II B 3, double-reflection walls of Sec. II B 5) as a
// march up strips in blocks of four rows, every stage on warps of its own.
//
// A CTA owns a strip of UW units (lb_block.cuh: column pairs of a flow grid,
// f and g of one column of a thermal grid) and CH rows.  At iteration i
//   A warps form h^n and f~ + Coll of rows 4 i .. 4 i + 3 (from ys - 4),
//   B warps the predictor of the four rows that end six below them,
//   C warps the corrector of the four rows that end six below those,
// on shared-memory rings of 12 rows of h, 12 of h* and 16 of f~ + Coll, with
// one barrier an iteration: what a stage reads, the others finished an
// iteration ago, and no slot is written while it can be read.  A's
// populations are loaded an iteration before they are used.
//
// Why: the step is bound by instruction issue and the shared-memory pipe.  A
// tile (lb_block.cuh) evaluates 1.9x its cells in stage A and 1.4x in B, and
// its SM idles at each stage's end; the strip's halo is 8 columns of 60 units
// and 16 rows of a chunk, and a stage's stalls are filled by the others' work.
// Every schedule of the packed kernels forms the same values in the same
// order, so they agree bit for bit.  Step times, former two-column march (or
// tile) -> this:  FP32 1024 x 1024 72 -> 32 us, 2048 x 2048 199 -> 117, 4096 x
// 4096 585 -> 400 (42 GLUPS); thermal 16-bit 1024 x 1024 111 -> 68 us, FP32
// 1000 x 375 43 -> 30.  An iteration of four rows takes about 1.7 us of which
// instruction issue is busy for half and the FP32 pipe for 45 %; loading A's
// populations at the end of an iteration instead of its middle costs a fifth.
#include "lb_block.cuh"
#include "lb_launch.cuh"

namespace lbgb {

namespace {

using namespace block;

// A pair of columns as stored, loaded an iteration before it is converted.
template <typename S> struct RawPair;
template <> struct RawPair<float> {
    using T = float2;
    __device__ static T ld(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
    __device__ static T two(const float* l, const float* r) { return make_float2(__ldg(l), __ldg(r)); }
    __device__ static V2 cvt(T v) { return {v}; }
};
template <> struct RawPair<__half> {
    using T = __half2;
    __device__ static T ld(const __half* p) { return __ldg(reinterpret_cast<const __half2*>(p)); }
    __device__ static T two(const __half* l, const __half* r) { return __halves2half2(__ldg(l), __ldg(r)); }
    __device__ static V2 cvt(T v) { return V2{__half22float2(v)} * bc(1.0f / kF16Scale); }
};
template <> struct RawPair<__nv_bfloat16> {
    using T = __nv_bfloat162;
    __device__ static T ld(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const __nv_bfloat162*>(p)); }
    __device__ static T two(const __nv_bfloat16* l, const __nv_bfloat16* r) {
        return __halves2bfloat162(__ldg(l), __ldg(r));
    }
    __device__ static V2 cvt(T v) { return {__bfloat1622float2(v)}; }
};

template <bool TH, int UW>
struct Strip {
    // rows of a stage B or C thread's column (one row halves a stage's length but spills: thermal 1024 x 1024 68
    // -> 103 us)
    static constexpr int RB = 2, RC = 2;
    static constexpr int UC = TH ? 1 : 2;                // columns per unit
    static constexpr int W = UW * UC;                    // output columns
    static constexpr int EP = (W + 8) / 2;               // column pairs of stage A
    static constexpr int EW = (W + 8) / UC, BW = (W + 4) / UC;
    static constexpr int wpr(int n) { return (n + 31) / 32; }
    static constexpr int WA = 4 * wpr(EP), WB = 4 / RB * wpr(BW), WC = 4 / RC * wpr(UW);
    static constexpr int NTH = 32 * (WA + WB + WC);
    static constexpr int NH = 12 * EW, NF = 16 * BW, NS = 12 * BW;
    static constexpr size_t smem = sizeof(V2) * Q * (NH + NF + NS) + sizeof(float4) * 5 * 16;
    static_assert(EP % 32 == 0, "stage A: whole warps");
};

template <int n>
__device__ __forceinline__ int ring(int q) { return q >= n ? q - n : q; }

template <typename S, bool TH, int UW, int MINB>
__global__ void __launch_bounds__(Strip<TH, UW>::NTH, MINB)
    k_fv_blocks(const StepArgs<float> A, const int CH) {
    using G = Strip<TH, UW>;
    constexpr int RB = G::RB, RC = G::RC;
    constexpr int UC = G::UC, EP = G::EP, EW = G::EW, BW = G::BW, NH = G::NH, NF = G::NF, NS = G::NS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V2* sH = reinterpret_cast<V2*>(smem_raw);  // [9][12][EW] h^n
    V2* sFC = sH + Q * NH;                     // [9][16][BW] f~ + Coll, then - dt/2 A[h^n]
    V2* sHs = sFC + Q * NF;                    // [9][12][BW] h*
    float4* sRow = reinterpret_cast<float4*>(sHs + Q * NS);  // [16][5] row entries

    const int nx = A.nx, ny = A.ny;
    const int x0 = blockIdx.x * G::W, ys = blockIdx.y * CH, ye = min(ys + CH, ny);
    const int nit = (ye - ys + 3) / 4 + 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool wally = A.bcy == LB_BC_WALLS;
    auto sync = [] { asm volatile("barrier.cta.sync 1, %0;" ::"n"(G::NTH) : "memory"); };

    if (warp < G::WA) {
        // ---- stage A: row q = 4 it + r of the chunk (row ys - 4 + q), pair px ----
        constexpr int WPR = EP / 32;
        const int r = warp / WPR, px = (warp % WPR) * 32 + lane;
        const int xu = x0 - 4 + 2 * px;
        const int gxl = ((xu % nx) + nx) % nx, gxr = ((xu + 1) % nx + nx) % nx;
        const bool contiguous = xu >= 0 && xu + 1 < nx;
        const bool inB = px >= 1 && px < EP - 1;
        const int uh = px * (2 / UC), ub = (px - 1) * (2 / UC);
        const S* fin = static_cast<const S*>(A.fin);
        const S* gin = static_cast<const S*>(A.gin);
        typename RawPair<S>::T rd[Q], re[Q];
        float ro = 0, to = 0;
        auto fetch = [&](int row) {
            int gy;
            if (row >= ye + 4 || !map_axis(row, ny, A.bcy, gy)) return;
            // a plane has fewer than 2^32 elements: at most 2^31 cells in at most 65535
            // rows (the row is a grid's y in the kernels of lb_init)
            const unsigned at = (unsigned)gy * (unsigned)A.pitch;
            if (contiguous) {
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    rd[a] = RawPair<S>::ld(fin + a * A.plane + (at + xu));
                    if constexpr (TH) re[a] = RawPair<S>::ld(gin + a * A.plane + (at + xu));
                }
            } else {
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    const S* b = fin + a * A.plane + at;
                    rd[a] = RawPair<S>::two(b + gxl, b + gxr);
                    if constexpr (TH) {
                        const S* bg = gin + a * A.plane + at;
                        re[a] = RawPair<S>::two(bg + gxl, bg + gxr);
                    }
                }
            }
            if constexpr (TH) {
                const float4 o = __ldg(reinterpret_cast<const float4*>(A.rowtab + 20 * gy) + 3);
                ro = o.y;
                to = o.z;
            }
        };
        fetch(ys - 4 + r);
        int s12 = r, s16 = r;  // ring slots of the row
        for (int it = 0; it < nit; ++it) {
            const int row0 = ys - 4 + 4 * it, row = row0 + r;
            float4 tab;
            bool has_tab = false;
            if (warp == 0 && lane < 20) {
                int gt;
                const int rt = row0 + lane / 5;
                has_tab = rt < ye + 4 && map_axis(rt, ny, A.bcy, gt);
                if (has_tab) tab = __ldg(reinterpret_cast<const float4*>(A.rowtab) + 5 * gt + lane % 5);
            }
            int gy;
            if (row < ye + 4 && map_axis(row, ny, A.bcy, gy)) {
                V2 d[Q], e[Q];
#pragma unroll
                for (int a = 0; a < Q; ++a) {
                    d[a] = RawPair<S>::cvt(rd[a]);
                    if constexpr (TH) e[a] = RawPair<S>::cvt(re[a]);
                }
                PairMom<TH> c;
                c.build(d, e, A, ro, to);
                fetch(row + 4);
                const int kh = s12 * EW + uh, kb = s16 * BW + ub;
                V2 h[Q], hg[Q];
                c.relax_f(d, A, A.omh, A.hF, h);
                if constexpr (TH) c.relax_g(e, A.omgh, hg);
                auto put_h = [&](V2* p, int a, float sg) {
                    if constexpr (!TH) *p = h[a];
                    else *reinterpret_cast<float4*>(p) = make_float4(h[a].v.x, sg * hg[a].v.x, h[a].v.y, sg * hg[a].v.y);
                };
#pragma unroll
                for (int a = 1; a < Q; ++a) put_h(sH + a * NH + kh, a, 1.0f);
                // images in the ghost rows of this block, and of the block below the bottom wall
                if (wally && (gy <= 1 || gy >= ny - 2)) {
                    auto image = [&](int g) {
                        const int k = (g - (ys - 4)) % 12 * EW + uh;
#pragma unroll
                        for (int a = 0; a < Q; ++a)
                            if (cy(a) != 0) put_h(sH + inv(a) * NH + k, a, -1.0f);
                    };
                    if (gy <= 1 && ys == 0) image(-1 - gy);
                    if (gy >= ny - 2 && 2 * ny - 1 - gy <= row0 + 3) image(2 * ny - 1 - gy);
                }
                if (inB) {
                    c.relax_f(d, A, A.om, A.cf, h);
                    if constexpr (TH) c.relax_g(e, A.omg, hg);
#pragma unroll
                    for (int a = 0; a < Q; ++a) put_h(sFC + a * NF + kb, a, 1.0f);
                }
            } else {
                fetch(row + 4);
                // a ghost row whose mirrored row was formed an iteration ago
                const int src = 2 * ny - 1 - row;
                if (wally && (row == ny || row == ny + 1) && row < ye + 4 && src < row0) {
                    const int kd = s12 * EW + uh, ks = (src - (ys - 4)) % 12 * EW + uh;
#pragma unroll
                    for (int a = 0; a < Q; ++a) {
                        if (cy(a) == 0) continue;
#pragma unroll
                        for (int u = 0; u < 2 / UC; ++u) {
                            const V2 v = sH[a * NH + ks + u];
                            sH[inv(a) * NH + kd + u] = TH ? swap_sign_g(v) : v;
                        }
                    }
                }
            }
            if (has_tab) sRow[((4 * it + lane / 5) & 15) * 5 + lane % 5] = tab;
            s12 = ring<12>(s12 + 4);
            s16 = (s16 + 4) & 15;
            sync();
        }
    } else if (warp < G::WA + G::WB) {
        // ---- stage B: RB rows from r0 of the block from ys - 2 + 4 (it - 2), unit bx ----
        constexpr int WPR = G::wpr(BW);
        const int w = warp - G::WA, j = w / WPR, bx = (w % WPR) * 32 + lane;
        const bool in = bx < BW;
        XW X;
        {
            const int xu = x0 - 2 + UC * (in ? bx : 0);
            X.load(reinterpret_cast<const float4*>(A.coltab) + 5 * (((xu % nx) + nx) % nx));
        }
        sync();
        sync();
        int s12 = RB * j, s16 = RB * j + 2;
        for (int it = 2; it < nit; ++it) {
            const int blk = ys - 2 + 4 * (it - 2), r0 = blk + RB * j;
            if (in && r0 < ye + 2) {
                int o[RB + 4];
#pragma unroll
                for (int i = 0; i < RB + 4; ++i) o[i] = ring<12>(s12 + i) * EW;
                YW<TH, RB> Y;
                Y.load(sRow + 5 * s16);
                const int kb = s16 * BW + bx;
                V2 st[RB][Q];
                for_flux<TH, RB, 0>(sH + bx + 2 / UC, NH, o, X, Y, [&](int a, const V2* v) {
#pragma unroll
                    for (int r = 0; r < RB; ++r) {
                        const V2 fc = sFC[a * NF + kb + r * BW];
                        st[r][a] = fma2(bc(-A.dt), v[r], fc);
                        sFC[a * NF + kb + r * BW] = fma2(bc(-A.hf), v[r], fc);
                    }
                });
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const int row = r0 + r;
                    int gy;
                    if (map_axis(row, ny, A.bcy, gy)) {
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
                        const int ks = ring<12>(s12 + r) * BW + bx;
#pragma unroll
                        for (int a = 1; a < Q; ++a) sHs[a * NS + ks] = st[r][a];
                        if (wally && (gy <= 1 || gy >= ny - 2)) {
                            auto image = [&](int g) {
                                const int k = (g - (ys - 2)) % 12 * BW + bx;
#pragma unroll
                                for (int a = 0; a < Q; ++a)
                                    if (cy(a) != 0) sHs[inv(a) * NS + k] = TH ? swap_sign_g(st[r][a]) : st[r][a];
                            };
                            if (gy <= 1 && ys == 0) image(-1 - gy);
                            if (gy >= ny - 2 && 2 * ny - 1 - gy <= blk + 3) image(2 * ny - 1 - gy);
                        }
                    } else if (wally && (row == ny || row == ny + 1) && 2 * ny - 1 - row < blk) {
                        const int kd = ring<12>(s12 + r) * BW + bx, ks = (2 * ny - 1 - row - (ys - 2)) % 12 * BW + bx;
#pragma unroll
                        for (int a = 0; a < Q; ++a) {
                            if (cy(a) == 0) continue;
                            const V2 v = sHs[a * NS + ks];
                            sHs[inv(a) * NS + kd] = TH ? swap_sign_g(v) : v;
                        }
                    }
                }
            }
            s12 = ring<12>(s12 + 4);
            s16 = (s16 + 4) & 15;
            sync();
        }
    } else {
        // ---- stage C: RC rows from r0 of the block from ys + 4 (it - 4), unit tx ----
        constexpr int WPR = G::wpr(UW);
        const int w = warp - G::WA - G::WB, j = w / WPR, tx = (w % WPR) * 32 + lane;
        const int gx = x0 + UC * tx;
        const bool in = tx < UW && gx < nx, both = gx + 1 < nx;
        XW X;
        X.load(reinterpret_cast<const float4*>(A.coltab) + 5 * (in ? gx : 0));
        S* fout = static_cast<S*>(A.fout);
        S* gout = static_cast<S*>(A.gout);
        sync();
        sync();
        sync();
        sync();
        int s12 = RC * j, s16 = RC * j + 4;
        for (int it = 4; it < nit; ++it) {
            const int r0 = ys + 4 * (it - 4) + RC * j;
            if (in && r0 < ye) {
                int o[RC + 4];
#pragma unroll
                for (int i = 0; i < RC + 4; ++i) o[i] = ring<12>(s12 + i) * BW;
                YW<TH, RC> Y;
                Y.load(sRow + 5 * s16);
                const int kb = s16 * BW + tx + 2 / UC;
                const unsigned at = (unsigned)r0 * (unsigned)A.pitch + gx;
                for_flux<TH, RC, 0>(sHs + tx + 2 / UC, NS, o, X, Y, [&](int a, const V2* v) {
#pragma unroll
                    for (int r = 0; r < RC; ++r) {
                        if (r > 0 && r0 + r >= ye) continue;
                        const V2 u = fma2(bc(-A.hf), v[r], sFC[a * NF + kb + r * BW]);
                        const long long q = a * A.plane + (at + (unsigned)r * (unsigned)A.pitch);
                        if constexpr (TH) {
                            Store<S>::st(fout + q, u.v.x);
                            Store<S>::st(gout + q, u.v.y);
                        } else {
                            if (both) PairIO<S>::st(fout + q, u);
                            else Store<S>::st(fout + q, u.v.x);
                        }
                    }
                });
            }
            s12 = ring<12>(s12 + 4);
            s16 = (s16 + 4) & 15;
            sync();
        }
    }
}

template <typename S, bool TH, int UW, int MINB>
cudaError_t run_blocks(const StepArgs<float>& A, int ch, cudaStream_t s) {
    using G = Strip<TH, UW>;
    static_assert(G::smem * MINB <= 232448, "shared memory per SM");
    const auto kernel = k_fv_blocks<S, TH, UW, MINB>;
    const cudaError_t e = set_max_smem((const void*)kernel, (int)G::smem);
    if (e != cudaSuccess) return e;
    kernel<<<dim3((A.nx + G::W - 1) / G::W, (A.ny + ch - 1) / ch), G::NTH, G::smem, s>>>(A, ch);
    count_launch();
    return cudaGetLastError();
}

// Strip widths: stage A's pairs fill whole warps, B's and C's units nearly so.
template <typename S>
cudaError_t run_blocks(bool th, const StepArgs<float>& A, int ch, bool wide, cudaStream_t s) {
    if (th) return run_blocks<S, true, 56, 1>(A, ch, s);
    return wide ? run_blocks<S, false, 60, 1>(A, ch, s) : run_blocks<S, false, 28, 2>(A, ch, s);
}

}  // namespace

cudaError_t launch_fv_blocks(Prec p, bool th, const void* args, int chunk, bool wide, cudaStream_t s) {
    const StepArgs<float>& A = *static_cast<const StepArgs<float>*>(args);
    const int ch = chunk < 4 ? 4 : (chunk + 3) / 4 * 4;
    switch (p) {
        case Prec::F32: return run_blocks<float>(th, A, ch, wide, s);
        case Prec::F16: return run_blocks<__half>(th, A, ch, wide, s);
        case Prec::BF16: return run_blocks<__nv_bfloat16>(th, A, ch, wide, s);
        default: return cudaErrorInvalidValue;
    }
}

int blocks_width(bool th, bool wide) { return th || !wide ? 56 : 120; }

}  // namespace lbgb
