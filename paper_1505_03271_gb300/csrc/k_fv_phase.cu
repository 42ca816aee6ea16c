// k_fv_phase.cu -- the FV time step (Sec. II B: Eqs. (semi), (semi-heun),
// QUICK faces of Sec. II B 3, double-reflection walls of Sec. II B 5) in two
// launches per step that recompute nothing:
//   predictor  A[h^n] on each cell's cross of nodes -> f~*, its moments and
//              h*, and b = f~ + Coll - dt/2 A[h^n]
//   corrector  A[h*] -> f~^(n+1) = b - dt/2 A[h*], its moments and h^(n+1),
//              which the next step's predictor reads
// One launch before the first step of a call forms h^n and f~ + Coll.  FP64
// forms both from one relaxation: om = 2 omh and cf = 2 hF, so with the change
// t = h - f~, f~ + Coll = f~ + 2 t.  FP32 rounds as the paired kernels do,
// whose results it reproduces bit for bit, and takes two.
// b holds f~ + Coll between the steps, so the state is written but not read.
// h, h* and b are fields of the compute type in memory: a step streams eight
// values per population and cell instead of two.
//
// What it is for: arithmetic or latency that bounds a step, not bandwidth.
// An SM starts an FP64 warp instruction about every 16 clocks, so the fused
// tile of k_fv.cu, which evaluates the collision on tile + 4 cells and the
// predictor on tile + 2 (1.9x and 1.4x at 32 x 16) and puts a 64 x 64 grid on
// 8 of 152 SMs, is bound by the FP64 pipe of those few SMs.  Here nothing is
// evaluated twice, a warp is 32 cells (or 32 populations of a few cells), and
// each axis' QUICK divergence is four multiply-adds with folded weights.
// FP64 step, fused tile -> this: 1 x 64 132 -> 7.3 us, 64 x 64 132 -> 8.7 us,
// 1024 x 1024 2011 -> 654 us (0.52 -> 1.60 GLUPS).  FP32: 64 x 64 6.1 -> 3.7
// us, thermal 64 x 64 (16-bit) 9.0 -> 4.3 us.
#include "lb_chain.cuh"
#include "lb_lane.cuh"
#include "lb_phase.cuh"

namespace lbgb {

namespace {

// Nodes -2..2 of a cell's line on one axis: byte offset of the node in a
// plane, and an all-ones mask where it is a ghost of a wall (then the offset
// is the mirrored cell's).
struct Line {
    unsigned off[5];
    unsigned ghost[5];
};

__device__ __forceinline__ Line make_line(int pos, int n, int bc, unsigned own, unsigned stride) {
    Line L;
#pragma unroll
    for (int s = -2; s <= 2; ++s) {
        int q = pos + s;
        unsigned gh = 0;
        if (q < 0 || q >= n) {
            if (bc == LB_BC_PERIODIC) {
                q %= n;
                if (q < 0) q += n;
            } else {
                gh = ~0u;
                q = q < 0 ? -q - 1 : 2 * n - 1 - q;
            }
        }
        L.off[s + 2] = own + (unsigned)(q - pos) * stride;
        L.ghost[s + 2] = gh;
    }
    return L;
}

// A field value at a byte offset from a uniform base: 32-bit offsets keep
// the address arithmetic on the uniform datapath.
template <typename T>
__device__ __forceinline__ T at(const void* base, unsigned off) {
    return *reinterpret_cast<const T*>(static_cast<const char*>(base) + off);
}
template <typename T>
__device__ __forceinline__ T& ref(void* base, unsigned off) {
    return *reinterpret_cast<T*>(static_cast<char*>(base) + off);
}

__device__ __forceinline__ double flip(double v, unsigned mask) {
    return __hiloint2double(__double2hiint(v) ^ (int)(mask & 0x80000000u), __double2loint(v));
}
__device__ __forceinline__ float flip(float v, unsigned mask) {
    return __int_as_float(__float_as_int(v) ^ (int)(mask & 0x80000000u));
}

// Folded QUICK weights of a cell on one axis: K[s] of nodes -2..1 for
// c > 0, then of nodes -1..2 for c < 0 (c (Phi_e - Phi_w) / dx).
template <typename R>
struct Fold {
    R p[4], m[4];
    __device__ __forceinline__ void load(const R* t, int i) {
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            p[s] = __ldg(t + 8 * i + s);
            m[s] = __ldg(t + 8 * i + 4 + s);
        }
    }
};

// The cell a thread works on and its stencil geometry.
template <typename R>
struct Site {
    int y;
    unsigned c;  // cell index in a plane
    Line lx, ly;
    Fold<R> kx, ky;
    __device__ __forceinline__ bool set(const PhaseArgs<R>& P) {
        const StepArgs<R>& A = P.s;
        const unsigned id = blockIdx.x * blockDim.x + threadIdx.x;
        if (id >= (unsigned)A.nx * (unsigned)A.ny) return false;
        y = (int)(id / (unsigned)A.nx);
        const int x = (int)(id - (unsigned)y * (unsigned)A.nx);
        c = (unsigned)y * A.pitch + x;
        const unsigned own = c * (unsigned)sizeof(R);
        lx = make_line(x, A.nx, A.bcx, own, sizeof(R));
        ly = make_line(y, A.ny, A.bcy, own, A.pitch * (unsigned)sizeof(R));
        kx.load(P.foldx, x);
        ky.load(P.foldy, y);
        return true;
    }
};

// sum_k K_k h(node k0 + k) of population i (velocity a) on one line.  A
// ghost node reads the reflected population, two planes away (every pair of
// opposite moving velocities of D2Q9 is), negated for the thermal field.
template <typename R, int i, bool WALL>
__device__ __forceinline__ R line_sum(const R* H, const Line& L, const R* K, int k0, long long plane, R v) {
    constexpr int a = i % Q;
    static_assert(inv(a) == a + 2 || inv(a) == a - 2, "opposite populations are two planes apart");
    constexpr int lo = i - a + (inv(a) < a ? inv(a) : a);
    const R* base = H + lo * plane;
    const unsigned two = (unsigned)(2 * plane * (long long)sizeof(R));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        unsigned o = L.off[k0 + k];
        if constexpr (WALL) {
            const unsigned gh = L.ghost[k0 + k];
            o += (inv(a) < a ? ~gh : gh) & two;  // the upper plane of the pair
            R h = at<R>(base, o);
            if constexpr (i >= Q) h = flip(h, gh);
            v += K[k] * h;
        } else {
            v += K[k] * at<R>(H + i * plane, o);
        }
    }
    return v;
}

template <typename R, bool TH, bool WX, bool WY, int i = 0>
__device__ __forceinline__ void advect_sites(const R* H, const Site<R>& s, const StepArgs<R>& A, R* out) {
    constexpr int a = i % Q;
    R v = 0;
    if constexpr (cx(a) != 0)
        v = line_sum<R, i, WX>(H, s.lx, cx(a) > 0 ? s.kx.p : s.kx.m, cx(a) > 0 ? 0 : 1, A.plane, v);
    if constexpr (cy(a) != 0)
        v = line_sum<R, i, WY>(H, s.ly, cy(a) > 0 ? s.ky.p : s.ky.m, cy(a) > 0 ? 0 : 1, A.plane, v);
    if constexpr (TH && cy(a) != 0) v += ref_flux<R, a>(A, s.y, i >= Q);  // base state (thermal grids)
    out[i] = v;
    if constexpr (i + 1 < (TH ? 2 * Q : Q)) advect_sites<R, TH, WX, WY, i + 1>(H, s, A, out);
}

// h (and hg) of one cell from its populations, into H; and (FC) f~ + Coll, into b.
template <typename R, bool TH, bool FC>
__device__ __forceinline__ void store_h(const R* d, const R* e, const PhaseArgs<R>& P, int y, R* H, unsigned c) {
    const StepArgs<R>& A = P.s;
    const unsigned o = c * (unsigned)sizeof(R);
    if constexpr (sizeof(R) == 8) {
        CellMom<TH> m;
        m.build(d, e, A, TH ? A.roff[y] : R(0), TH ? A.toff[y] : R(0));
        R t[Q];
        m.change_f(d, P, t);
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            ref<R>(H + a * A.plane, o) = d[a] + t[a];
            if constexpr (FC) ref<R>(P.b + a * A.plane, o) = d[a] + R(2) * t[a];
        }
        if constexpr (TH) {
            m.change_g(e, P, t);
#pragma unroll
            for (int a = 0; a < Q; ++a) {
                ref<R>(H + (Q + a) * A.plane, o) = e[a] + t[a];
                if constexpr (FC) ref<R>(P.b + (Q + a) * A.plane, o) = e[a] + R(2) * t[a];
            }
        }
    } else {
        pairmath::LaneMom<TH> m;
        m.build(d, e, A, TH ? A.roff[y] : 0.0f, TH ? A.toff[y] : 0.0f);
#pragma unroll
        for (int a = 0; a < Q; ++a) {
            ref<R>(H + a * A.plane, o) = m.one_f(a, d[a], A, A.omh, A.hF);
            if constexpr (FC) ref<R>(P.b + a * A.plane, o) = m.one_f(a, d[a], A, A.om, A.cf);
            if constexpr (TH) {
                ref<R>(H + (Q + a) * A.plane, o) = m.one_g(a, e[a], A.omgh);
                if constexpr (FC) ref<R>(P.b + (Q + a) * A.plane, o) = m.one_g(a, e[a], A.omg);
            }
        }
    }
}

// Launches are chained by programmatic dependent launch: a kernel's CTAs may
// be resident, their indices and weights loaded, before the previous kernel
// has finished; every kernel waits here for its completion before it touches
// a field.  early lets the next kernel in at once, which hides its start-up
// where both fit (64 x 64, FP32: 1.0 us of a 4.4 us step); on grids that
// fill the SMs its waiting CTAs would unbalance the running kernel's
// (256 x 256, FP64: 72 us against 48), which then releases it as it ends.
__device__ __forceinline__ void dependency_wait(int early) {
    cudaGridDependencySynchronize();
    if (early) cudaTriggerProgrammaticLaunchCompletion();
}

template <typename R, typename S, bool TH>
__global__ void __launch_bounds__(128) k_phase_start(const PhaseArgs<R> P) {
    const StepArgs<R>& A = P.s;
    const unsigned id = blockIdx.x * blockDim.x + threadIdx.x;
    dependency_wait(P.early);
    if (id >= (unsigned)A.nx * (unsigned)A.ny) return;
    const int y = (int)(id / (unsigned)A.nx);
    const unsigned c = (unsigned)y * A.pitch + (id - (unsigned)y * (unsigned)A.nx);
    R d[Q], e[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        d[a] = Chained<S>::ld(static_cast<const S*>(A.fin) + a * A.plane + c);
        if constexpr (TH) e[a] = Chained<S>::ld(static_cast<const S*>(A.gin) + a * A.plane + c);
    }
    store_h<R, TH, true>(d, e, P, y, P.h, c);
}

template <typename R, bool TH, bool WX, bool WY>
__global__ void __launch_bounds__(128) k_phase_predict(const PhaseArgs<R> P) {
    const StepArgs<R>& A = P.s;
    Site<R> s;
    const bool in = s.set(P);
    dependency_wait(P.early);
    if (!in) return;
    constexpr int NQ = TH ? 2 * Q : Q;
    R adv[NQ];
    advect_sites<R, TH, WX, WY>(P.h, s, A, adv);
    R d[Q], e[Q];
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        const R fc = at<R>(P.b + i * A.plane, s.c * (unsigned)sizeof(R));
        ref<R>(P.b + i * A.plane, s.c * (unsigned)sizeof(R)) = fc - A.hf * adv[i];
        const R st = fc - A.dt * adv[i];
        if (i < Q) d[i] = st;
        else e[i - Q] = st;
    }
    store_h<R, TH, false>(d, e, P, s.y, P.hs, s.c);
}

template <typename R, typename S, bool TH, bool WX, bool WY>
__global__ void __launch_bounds__(128) k_phase_correct(const PhaseArgs<R> P) {
    const StepArgs<R>& A = P.s;
    Site<R> s;
    const bool in = s.set(P);
    dependency_wait(P.early);
    if (!in) return;
    constexpr int NQ = TH ? 2 * Q : Q;
    R adv[NQ];
    advect_sites<R, TH, WX, WY>(P.hs, s, A, adv);
    R d[Q], e[Q];
#pragma unroll
    for (int i = 0; i < NQ; ++i) {
        S* dst = (i < Q ? static_cast<S*>(A.fout) + i * A.plane : static_cast<S*>(A.gout) + (i - Q) * A.plane) + s.c;
        const R v = at<R>(P.b + i * A.plane, s.c * (unsigned)sizeof(R)) - A.hf * adv[i];
        Store<S>::st(dst, v);
        const R r = Round<S>::of(v);  // the next step starts from the stored value
        if (i < Q) d[i] = r;
        else e[i - Q] = r;
    }
    store_h<R, TH, true>(d, e, P, s.y, P.h, s.c);
}

// ---- the same two launches with one population per thread ----
// A CTA holds the 9 (18) populations of CELLS cells, one per thread; the
// moments pass through shared memory.  Each thread's instruction stream is
// short (one stencil, one relaxation), so a grid of a few thousand cells,
// whose warps run alone on their SM, is not bound by one long dependent
// stream.
//
// One axis of one population.  FP64 takes the folded weights: half the
// instructions of two face values.  FP32 forms the faces, in the order of
// operations of the paired kernels, whose results it then reproduces bit for
// bit (y: v + c (Phi_n - Phi_s) / dy; x: c (Phi_e - Phi_w) / dx).
template <typename R>
struct Quick {
    float4 p, q;  // west face's weights and the east face's first; its others and 1 / dx
    __device__ __forceinline__ void load(const float* t, int i, int v) {
        const float4* c = reinterpret_cast<const float4*>(t) + 4 * i + (v > 0 ? 0 : 2);
        p = __ldg(c);
        q = __ldg(c + 1);
    }
    __device__ __forceinline__ float x(const float* h, int v) const {
        const float w = __fmaf_rn(p.z, h[2], __fmaf_rn(p.x, h[0], __fmul_rn(p.y, h[1])));
        const float e = __fmaf_rn(q.y, h[3], __fmaf_rn(p.w, h[1], __fmul_rn(q.x, h[2])));
        const float d = __fmul_rn(e - w, q.z);
        return v > 0 ? d : -d;
    }
    __device__ __forceinline__ float y(const float* h, int v, float sum) const {
        const float s = __fmaf_rn(p.x, h[0], __fmaf_rn(p.y, h[1], __fmul_rn(p.z, h[2])));
        const float n = __fmaf_rn(p.w, h[1], __fmaf_rn(q.x, h[2], __fmul_rn(q.y, h[3])));
        return v > 0 ? __fmaf_rn(n - s, q.z, sum) : sum - __fmul_rn(n - s, q.z);
    }
};
template <>
struct Quick<double> {
    double k[4];
    __device__ __forceinline__ void load(const double* t, int i, int v) {
#pragma unroll
        for (int s = 0; s < 4; ++s) k[s] = __ldg(t + 8 * i + (v > 0 ? 0 : 4) + s);
    }
    __device__ __forceinline__ double x(const double* h, int) const {
        return k[0] * h[0] + k[1] * h[1] + k[2] * h[2] + k[3] * h[3];
    }
    __device__ __forceinline__ double y(const double* h, int v, double sum) const { return sum + x(h, v); }
};

__device__ __forceinline__ int vel(unsigned packed, int a) { return (int)((packed >> (2 * a)) & 3u) - 1; }
__host__ __device__ constexpr unsigned pack_vel(int axis, int a = 0) {
    return a == Q ? 0u : ((unsigned)((axis ? cy(a) : cx(a)) + 1) << (2 * a)) | pack_vel(axis, a + 1);
}

__device__ __forceinline__ double mad(double a, double b, double c) { return a * b + c; }
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
// the base state's flux divergence c_y w A[ref], as the paired kernels add it
__device__ __forceinline__ double add_base(double v, double w, double r) { return v + w * r; }
__device__ __forceinline__ float add_base(float v, float w, float r) { return v + __fmul_rn(w, r); }

template <typename R, bool TH> struct MomOf;
template <bool TH> struct MomOf<double, TH> { using T = CellMom<TH>; };
template <bool TH> struct MomOf<float, TH> { using T = pairmath::LaneMom<TH>; };

template <typename R, typename S, bool TH, bool CORR, int CELLS>
__global__ void __launch_bounds__((TH ? 18 : 9) * CELLS) k_phase_pop(const PhaseArgs<R> P) {
    constexpr int NQ = TH ? 2 * Q : Q;
    constexpr int NM = TH ? 9 : 7;
    __shared__ R sd[NQ][CELLS];
    // rp, rho, 3 ux, 3 uy; -1.5 u.u, -3 u.a, a_y (FP64: C0 of f and of g, 3 hF a_y); Td, T
    __shared__ R sm[NM][CELLS];
    const StepArgs<R>& A = P.s;
    const int lane = threadIdx.x % CELLS, i = threadIdx.x / CELLS;
    const bool G = TH && i >= Q;
    const int a = G ? i - Q : i;
    constexpr unsigned VX = pack_vel(0), VY = pack_vel(1);
    const int vx = vel(VX, a), vy = vel(VY, a);
    const int b = a == 0 ? 0 : (((a - 1) ^ 2) + 1);  // inv(a): 1<->3, 2<->4, 5<->7, 6<->8
    const unsigned id = blockIdx.x * CELLS + lane;
    const bool in = id < (unsigned)A.nx * (unsigned)A.ny;
    const unsigned cid = in ? id : 0;
    const int y = (int)(cid / (unsigned)A.nx), x = (int)(cid - (unsigned)y * (unsigned)A.nx);
    const unsigned c = (unsigned)y * A.pitch + x;
    // Elements: the lower plane of the pair a, inv(a) in 64 bits (18 planes can
    // pass 2^32), the rest in 32 (phase_applies bounds three planes).  A grid of
    // eight cells per CTA has at most 8 cells per SM, so all its planes fit 32 bits,
    // which shortens the kernel's one long chain (1 x 64, FP64: 7.15 -> 6.95 us
    // a step).
    constexpr bool kSmall = CELLS <= 8;
    const size_t lo = kSmall ? 0 : (size_t)(i - a + (b < a ? b : a)) * (size_t)A.plane;
    const unsigned pl = (unsigned)A.plane;
    const unsigned own = (kSmall ? (unsigned)i * pl : b < a ? 2u * pl : 0u) + c;
    const unsigned refl = (kSmall ? (unsigned)(i - a + b) * pl : b < a ? 0u : 2u * pl) + c;
    unsigned ox[4], oy[4], gx = 0, gy = 0;  // node offsets (elements); ghost flags of the four nodes
    Quick<R> kx, ky;
    auto line = [&](int pos, int n, int bc, unsigned stride, int v, unsigned* o, unsigned& g) {
        const int s0 = v > 0 ? -2 : -1;
#pragma unroll
        for (int s = 0; s < 4; ++s) o[s] = own + (unsigned)(s0 + s) * stride;
        if (pos >= 2 && pos + 2 < n) return;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            int q = pos + s0 + s;
            if (q >= 0 && q < n) continue;
            unsigned from = own;
            if (bc == LB_BC_PERIODIC) {
                q = ((q % n) + n) % n;
            } else {
                g |= 1u << s;
                from = refl;
                q = q < 0 ? -q - 1 : 2 * n - 1 - q;
            }
            o[s] = from + (unsigned)(q - pos) * stride;
        }
    };
    if (vx != 0) {
        kx.load(P.foldx, x, vx);
        line(x, A.nx, A.bcx, 1, vx, ox, gx);
    }
    if (vy != 0) {
        ky.load(P.foldy, y, vy);
        line(y, A.ny, A.bcy, A.pitch, vy, oy, gy);
    }
    R ro = 0, to = 0, base = 0;
    if constexpr (TH) {  // flow grids have the uniform base state
        ro = A.roff[y];
        to = A.toff[y];
        if (vy != 0) base = __ldg(A.dref + ((G ? 2 : 0) + (vy > 0 ? 0 : 1)) * A.ny + y);
    }
    dependency_wait(P.early);

    const R* H = (CORR ? P.hs : P.h) + lo;
    // formed here for the 64-bit planes (64 x 64, FP64: 8.7 -> 8.5 us a step), at
    // its use for the 32-bit ones
    R* const h64 = (CORR ? P.h : P.hs) + lo;
    R* const b64 = P.b + lo;
    auto h_out = [&]() -> R& { return (kSmall ? (CORR ? P.h : P.hs) : h64)[own]; };
    auto b_own = [&]() -> R& { return (kSmall ? P.b : b64)[own]; };
    R hx[4], hy[4];
    if (vx != 0) {
#pragma unroll
        for (int s = 0; s < 4; ++s) hx[s] = H[ox[s]];
    }
    if (vy != 0) {
#pragma unroll
        for (int s = 0; s < 4; ++s) hy[s] = H[oy[s]];
    }
    const R fc = b_own();
    R v = 0;
    if (vx != 0) v = kx.x(hx, vx);
    if (vy != 0) {
        if constexpr (TH) {
#pragma unroll
            for (int s = 0; s < 4; ++s) hy[s] = flip(hy[s], G && (gy >> s & 1u) ? ~0u : 0u);
        }
        v = ky.y(hy, vy, v);
        if constexpr (TH) v = add_base(v, R(vy) * wgt<R>(a <= 4 ? 1 : 5), base);
    }
    R d;
    if constexpr (CORR) {
        d = mad(-A.hf, v, fc);
        S* dst = static_cast<S*>(G ? A.gout : A.fout) + (kSmall ? (size_t)((unsigned)a * pl) : (size_t)a * A.plane) + c;
        if (in) Store<S>::st(dst, d);
        d = Round<S>::of(d);  // the next step starts from the stored value
    } else {
        if (in) b_own() = mad(-A.hf, v, fc);
        d = mad(-A.dt, v, fc);
    }
    sd[i][lane] = d;
    __syncthreads();
    if (i == 0) {
        R f[Q], e[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            f[q] = sd[q][lane];
            if constexpr (TH) e[q] = sd[Q + q][lane];
        }
        typename MomOf<R, TH>::T m;
        m.build(f, e, A, ro, to);
        sm[0][lane] = m.rp;
        sm[1][lane] = m.rho;
        sm[2][lane] = m.ux3;
        sm[3][lane] = m.uy3;
        if constexpr (sizeof(R) == 8) {  // formed once, not by every population's thread
            sm[4][lane] = m.c0_f(P);
            sm[5][lane] = m.c0_g(P);
            sm[6][lane] = m.cty(P);
        } else {
            sm[4][lane] = m.uuneg;
            sm[5][lane] = m.ua3neg;
            sm[6][lane] = m.ay;
        }
        if constexpr (TH) {
            sm[7][lane] = m.Td;
            sm[8][lane] = m.T;
        }
    }
    __syncthreads();
    if constexpr (sizeof(R) == 8) {
        // h = d + t of population a
        const R w = a == 0 ? wgt<R>(0) : (a <= 4 ? wgt<R>(1) : wgt<R>(5));
        R cu3 = 0;  // as in CellMom::changes: of velocities 1, 2, 5 and 6, or the negative
        if (vx != 0) cu3 = vx > 0 ? sm[2][lane] : -sm[2][lane];
        if (vy != 0) cu3 += vy > 0 ? sm[3][lane] : -sm[3][lane];
        R ct = 0;
        if (!G) {
            if (vx != 0) ct = vx > 0 ? P.ctx : -P.ctx;
            if (vy != 0) ct += vy > 0 ? sm[6][lane] : -sm[6][lane];
        }
        constexpr int kT = TH ? 7 : 0;  // first thermal moment
        R S, D;
        CellMom<TH>::parts(cu3, ct, P.kh[G], sm[G ? 5 : 4][lane], S, D);
        const R t = CellMom<TH>::change(d, S + D, P.k[G], w, sm[G ? kT : 0][lane], sm[G ? kT + 1 : 1][lane]);
        if (in) {
            h_out() = d + t;
            if constexpr (CORR) b_own() = d + R(2) * t;
        }
    } else {
        pairmath::LaneMom<TH> m;
        m.rp = sm[0][lane];
        m.rho = sm[1][lane];
        m.ux3 = sm[2][lane];
        m.uy3 = sm[3][lane];
        m.uuneg = sm[4][lane];
        m.ua3neg = sm[5][lane];
        m.ay = sm[6][lane];
        if constexpr (TH) {
            m.Td = sm[7][lane];
            m.T = sm[8][lane];
        }
        if (in) {
            h_out() = G ? m.one_g(a, d, A.omgh) : m.one_f(a, d, A, A.omh, A.hF);
            if constexpr (CORR) b_own() = G ? m.one_g(a, d, A.omg) : m.one_f(a, d, A, A.om, A.cf);
        }
    }
}

template <typename K, typename R>
cudaError_t launch_pdl(K kernel, const PhaseArgs<R>& P, int block, int cells, cudaStream_t s) {
    const long long n = (long long)P.s.nx * P.s.ny;
    const cudaError_t e = launch_chained(kernel, dim3((unsigned)((n + cells - 1) / cells)), block, 0, s, P);
    count_launch();
    return e;
}

template <typename R, typename S, bool TH, bool WX, bool WY>
cudaError_t run_step(const PhaseArgs<R>& P, int block, cudaStream_t s) {
    const cudaError_t e = launch_pdl(k_phase_predict<R, TH, WX, WY>, P, block, block, s);
    return e != cudaSuccess ? e : launch_pdl(k_phase_correct<R, S, TH, WX, WY>, P, block, block, s);
}

template <typename R, typename S, bool TH, int CELLS>
cudaError_t run_pop(PhaseArgs<R>& P, cudaStream_t s) {
    constexpr int T = CELLS * (TH ? 2 * Q : Q);
    P.early = 1;
    const cudaError_t e = launch_pdl(k_phase_pop<R, S, TH, false, CELLS>, P, T, CELLS, s);
    return e != cudaSuccess ? e : launch_pdl(k_phase_pop<R, S, TH, true, CELLS>, P, T, CELLS, s);
}

// Which form a size takes.  Cells per CTA of the one-population form: its
// moments are one warp's serial FP64 stream, so below eight cells per SM the
// grid is spread thinner (1 x 64, FP64: 7.4 us a step at 8 cells per CTA, 9.9
// at 32).  The one-cell form issues a quarter fewer FP64 instructions but one
// long stream per warp, and takes over where its warps fill the SMs: 64 x 64
// 8.7 us by population, 17 by cell; 128 x 128 20.7 and 20.0; thermal
// 128 x 128 50.9 and 32.0; 1024 x 1024 985 and 649, where the FP64 pipe is
// 90 % busy.  FP32 arithmetic takes only the one-population form, for the
// small grids phase_applies (lb_abi.cu) sends here.
template <typename R, typename S, bool TH>
cudaError_t run_phase(PhaseArgs<R> P, bool start, int sms, cudaStream_t s) {
    const long long cells = (long long)P.s.nx * P.s.ny;
    if (start) return launch_pdl(k_phase_start<R, S, TH>, P, 64, 64, s);
    if (cells <= 8LL * sms) return run_pop<R, S, TH, 8>(P, s);
    if constexpr (sizeof(R) == 8) {
        if ((TH ? 2 : 1) * cells > 96LL * sms) {
            const bool wx = P.s.bcx == LB_BC_WALLS, wy = P.s.bcy == LB_BC_WALLS;
            if constexpr (!TH)  // thermal grids are periodic in x
                if (wx) return wy ? run_step<R, S, TH, true, true>(P, 64, s) : run_step<R, S, TH, true, false>(P, 64, s);
            return wy ? run_step<R, S, TH, false, true>(P, 64, s) : run_step<R, S, TH, false, false>(P, 64, s);
        }
    }
    return run_pop<R, S, TH, 32>(P, s);
}

}  // namespace

cudaError_t launch_fv_phase(Prec p, bool th, const void* args, bool start, int sms, cudaStream_t s) {
    if (p == Prec::F64) {
        const PhaseArgs<double>& P = *static_cast<const PhaseArgs<double>*>(args);
        return th ? run_phase<double, double, true>(P, start, sms, s) : run_phase<double, double, false>(P, start, sms, s);
    }
    const PhaseArgs<float>& P = *static_cast<const PhaseArgs<float>*>(args);
    switch (p) {
        case Prec::F32:
            return th ? run_phase<float, float, true>(P, start, sms, s) : run_phase<float, float, false>(P, start, sms, s);
        case Prec::F16:
            return th ? run_phase<float, __half, true>(P, start, sms, s)
                      : run_phase<float, __half, false>(P, start, sms, s);
        default:
            return th ? run_phase<float, __nv_bfloat16, true>(P, start, sms, s)
                      : run_phase<float, __nv_bfloat16, false>(P, start, sms, s);
    }
}

}  // namespace lbgb
