// lb_abi.cu -- host side of the C ABI declared in include/lb.h: grid and
// metric construction, parameter checks, kernel dispatch and observables.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <optional>
#include <set>
#include <string>
#include <tuple>
#include <vector>

#include "lb_grid.cuh"
#include "lb_phase.cuh"
#include "lb_scratch.cuh"

using namespace lbgb;

namespace {

thread_local std::string g_err;
std::atomic<unsigned long long> g_launches{0};
// While this thread captures a step graph, launches are tallied here: they
// run (and count) only when the graph is replayed.
thread_local unsigned long long* t_captured = nullptr;

lb_status fail(lb_status s, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_err = buf;
    return s;
}

#define CK(call)                                                                             \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return fail(e_ == cudaErrorMemoryAllocation ? LB_ERR_OOM : LB_ERR_CUDA, "%s: %s", \
                        #call, cudaGetErrorString(e_));                                      \
    } while (0)

}  // namespace

namespace lbgb {
void count_launch() {
    if (t_captured) ++*t_captured;
    else g_launches.fetch_add(1, std::memory_order_relaxed);
}
cudaError_t set_max_smem(const void* fn, int bytes) {
    static std::mutex mu;
    static std::set<std::tuple<int, const void*, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({dev, fn, bytes})) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.insert({dev, fn, bytes});
    return e;
}
// 16-bit ST on flow grids periodic in x with nx % 4 == 0 (k_st16.cu).
bool st16_applies(Prec p, bool thermal, int nx, int bcx);
cudaError_t launch_st16(Prec p, const void* args, cudaStream_t s);
// FP32 ST on flow grids periodic in x with nx % 4 == 0 (k_st_quad.cu).
bool st_quad_applies(Prec p, bool thermal, int nx, int bcx);
cudaError_t launch_st_quad(const void* args, cudaStream_t s);
// Record a failure message for lb_last_error() from another translation unit.
lb_status set_last_error(lb_status s, const char* msg) { return fail(s, "%s", msg); }
}  // namespace lbgb

namespace {

void release(lb_grid* G) {
    void* ptrs[] = {G->arena, G->xh, G->xfc, G->phase};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (G->cap) cudaStreamDestroy(G->cap);
}

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// Host image of the tables from `first` up to `end` in a grid's arena, filled
// by the pointers they have on the device and sent by one copy.
class HostTables {
public:
    HostTables(void* first, const void* end)
        : first_(static_cast<unsigned char*>(first)), buf_(static_cast<const unsigned char*>(end) - first_) {}
    template <typename T>
    T* at(const void* p) {
        return reinterpret_cast<T*>(buf_.data() + (static_cast<const unsigned char*>(p) - first_));
    }
    void put(const void* p, const std::vector<double>& v, bool f32) {
        if (f32) std::copy(v.begin(), v.end(), at<float>(p));
        else std::copy(v.begin(), v.end(), at<double>(p));
    }
    cudaError_t upload() const { return cudaMemcpy(first_, buf_.data(), buf_.size(), cudaMemcpyHostToDevice); }

private:
    unsigned char* first_;
    std::vector<unsigned char> buf_;
};

AuxArgs aux_args(const lb_grid* G) {
    AuxArgs a{};
    a.f = G->f[G->cur];
    a.g = G->g[G->cur];
    a.nx = G->nx;
    a.ny = G->ny;
    a.pitch = G->pitch;
    a.plane = G->plane;
    a.dt = G->fv_scheme == LB_FV_EULER ? 0.0 : G->p.dt;  // dt/2 a shift of the tilded moments
    a.ax = G->p.ax;
    a.ay = G->p.ay;
    a.bg = G->p.beta * G->p.grav;
    a.T0 = G->p.T0;
    a.toff = G->toff;
    a.roff = G->roff;
    a.dxv = G->dxv;
    a.dyv = G->dyv;
    a.xc = G->xc;
    a.yc = G->yc;
    return a;
}

lb_status check_ready(lb_grid* G) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!G->has_params) return fail(LB_ERR_STATE, "grid has no parameters: call lb_init first");
    if (G->poisoned) return fail(LB_ERR_STATE, "grid diverged (LB_ERR_UNSTABLE); call lb_init again");
    return LB_OK;
}

bool pair_ok(const lb_grid* G) {
    return G->prec != Prec::F64 && G->d.bcx == LB_BC_PERIODIC && G->d.bcy != LB_BC_DENSITY;
}

bool has_density_axis(const lb_grid* G) { return G->d.bcx == LB_BC_DENSITY || G->d.bcy == LB_BC_DENSITY; }

// How many waves n CTAs take on `slots` places.
long long waves(long long n, long long slots) { return (n + slots - 1) / slots; }

// The block march (k_fv_blocks.cu): strip width and rows per CTA, and the
// time a step takes in microseconds.  A CTA that owns ch rows runs ch / 4 + 4
// iterations; measured, one takes 1.65 us on a wide flow strip (120 columns,
// one CTA per SM), 1.8 on two narrow ones (56 columns each, two CTAs per SM;
// one alone 1.5) and 1.75 on a thermal strip (56 columns).
struct March {
    bool wide;
    int chunk;
    double us;
};
March march_plan(const lb_grid* G, int chunk) {
    March best{true, 0, 1e300};
    const bool th = G->d.thermal != 0;
    for (int wide = th ? 1 : 0; wide < 2; ++wide) {
        const int width = blocks_width(th, wide != 0);
        const long long strips = (G->nx + width - 1) / width;
        auto cost = [&](long long ch) {
            const long long n = strips * ((G->ny + ch - 1) / ch);
            const double it = th ? 1.75 : wide ? 1.65 : n <= G->sms ? 1.5 : 1.8;
            return waves(n, (long long)G->sms * (wide ? 1 : 2)) * (ch / 4 + 4) * it + 1.5;
        };
        auto take = [&](long long ch) {
            ch = std::min((ch + 3) / 4 * 4, 1LL << 30);  // rows and CTA counts in 32 bits
            const double us = cost(ch);
            if (us < best.us) best = {wide != 0, (int)ch, us};
        };
        if (chunk > 0) take(chunk);
        else
            for (long long w = 1; w <= 8; ++w) {  // the tallest chunks that fill w waves
                const long long chunks = w * G->sms * (wide ? 1 : 2) / strips;
                take(chunks < 1 ? G->ny : (G->ny + chunks - 1) / chunks);
            }
    }
    return best;
}

// The paired tile (lb_block.cuh): shape and time.  A wave of tiles takes 6.5
// us at 16 rows and 6.2 at 14 (flow, two CTAs per SM), 6.7 and 6.55 on
// thermal grids (one per SM); 16 x 16 thermal tiles 5.7 in a single wave.
struct Tile {
    int shape;
    double us;
};
Tile tile_plan(const lb_grid* G) {
    const bool th = G->d.thermal != 0;
    const long long cols = (G->nx + 31) / 32, slots = (long long)G->sms * (th ? 1 : 2);
    Tile t{th ? 512 : 0, waves(cols * ((G->ny + 15) / 16), slots) * (th ? 6.7 : 6.5) + 1.5};
    const double us14 = waves(cols * ((G->ny + 13) / 14), slots) * (th ? 6.55 : 6.2) + 1.5;
    if (us14 < t.us) t = {th ? 526 : 14, us14};
    if (th && (long long)((G->nx + 15) / 16) * ((G->ny + 15) / 16) <= G->sms && t.us > 7.2) t = {16, 7.2};
    return t;
}

// Schedule actually used: AUTO takes the paired tile or the block march,
// whichever those figures put first (800 x 800 FP32: tile 29.4 us, march
// 21.5; 384 x 512: 11.5 and 11.1, taken as equal; thermal 16-bit 600 x 600:
// 38.7 and 29.4, 320 x 320: 13.6 and 13.7), and
// on grids they do not serve the scalar march once its strips fill the GPU,
// else the scalar tile.
int resolved_kernel(const lb_grid* G) {
    if (G->fv_kernel != LB_FV_AUTO) return G->fv_kernel;
    if (pair_ok(G)) return march_plan(G, 0).us < tile_plan(G).us ? LB_FV_PAIR : LB_FV_PTILE;
    return G->nx >= 480 && G->ny >= 256 && !G->d.thermal ? LB_FV_MARCH : LB_FV_TILE;
}

// Rows per CTA of the marching kernels.
int resolved_chunk(const lb_grid* G) {
    if (resolved_kernel(G) == LB_FV_PAIR) return march_plan(G, G->fv_chunk).chunk;
    if (G->fv_chunk > 0) return G->fv_chunk;
    const bool th = G->d.thermal != 0;
    const int width = march_width(G->prec, th);
    const int strips = (G->nx + width - 1) / width;
    int per_sm = (int)(227 * 1024 / march_smem(G->prec, th));
    if (per_sm < 1) per_sm = 1;
    if (per_sm > 4) per_sm = 4;
    // about four waves of resident CTAs: short marches balance better than
    // one wave with a ragged tail, at 12 halo rows per chunk
    const long long slots = (long long)G->sms * per_sm;
    long long chunks = (4 * slots + strips - 1) / strips;
    if (chunks < 1) chunks = 1;
    int ch = (int)((G->ny + chunks - 1) / chunks);
    return ch < 32 ? 32 : ch;
}

// Shape of the scalar tile: as asked for (32 x 16 where the two launches were,
// on a grid they do not serve), 32 x 16 for the single-stage schemes and density
// boundaries.  AUTO on FP32-math grids with walls on x: 16 x 8 while two of them
// per SM cover the grid (100 x 100: 6.2 us a step, 10.3 at 32 x 16), else
// 16 x 16, of which an SM holds three (333 x 257: 12.4, 13.3 at 32 x 16; 470 x
// 500 22.3 and 24.2; 300 x 5000 118 and 128), except where they just pass one
// wave and two of 32 x 16 per SM do not (460 x 300: 14.3 and 13.3), or nearly
// fill two waves (470 x 600: 25.4 and 24.6).
int scalar_shape(const lb_grid* G) {
    if (G->fv_kernel == LB_FV_TILE) return G->fv_chunk == 2 ? 0 : G->fv_chunk;
    if (G->fv_kernel != LB_FV_AUTO || G->prec == Prec::F64 || G->d.bcx != LB_BC_WALLS) return 0;
    if (G->fv_scheme != LB_FV_HEUN || has_density_axis(G)) return 0;
    auto tiles = [G](int tx, int ty) { return (long long)((G->nx + tx - 1) / tx) * ((G->ny + ty - 1) / ty); };
    const long long n8 = tiles(16, 8), n16 = tiles(16, 16), n32 = tiles(32, 16);
    if (n8 <= 2LL * G->sms) return 8;
    const bool one_wave = n32 <= 2LL * G->sms && n16 > 3LL * G->sms;
    const bool two_waves = n32 <= 4LL * G->sms && 2 * n32 > 7LL * G->sms;
    return one_wave || two_waves ? 0 : 16;
}

int resolved_shape(const lb_grid* G) { return G->fv_kernel == LB_FV_PTILE ? G->fv_chunk : tile_plan(G).shape; }

// The split schedule's two FP32 buffers (NQ planes each), allocated on
// first use.
cudaError_t ensure_split_buffers(lb_grid* G) {
    if (G->xh) return cudaSuccess;
    const size_t bytes = sizeof(float) * (G->d.thermal ? 18 : 9) * (size_t)G->plane;
    cudaError_t e = device_malloc((void**)&G->xh, bytes);
    if (e == cudaSuccess) e = device_malloc((void**)&G->xfc, bytes);
    if (e != cudaSuccess) {
        if (G->xh) cudaFree(G->xh);
        G->xh = G->xfc = nullptr;
    }
    return e;
}

template <typename R>
cudaError_t launch_fv_step(lb_grid* G) {
    StepArgs<R> A = step_args<R>(G, G->p.dt);
    const bool th = G->d.thermal != 0;
    if (A.stages == 1 || has_density_axis(G))  // single-stage schemes, density boundaries: scalar tile kernel
        return launch_fv(G->prec, th, &A, scalar_shape(G), G->stream);
    const int k = resolved_kernel(G);
    if (k == LB_FV_SPLIT) {
        cudaError_t e = ensure_split_buffers(G);
        if (e != cudaSuccess) return e;
        A.xh = G->xh;
        A.xfc = G->xfc;
        return launch_fv_split(G->prec, th, &A, G->fv_chunk, G->stream);
    }
    if (k == LB_FV_PAIR) {
        const March m = march_plan(G, G->fv_kernel == LB_FV_PAIR ? G->fv_chunk : 0);
        return launch_fv_blocks(G->prec, th, &A, m.chunk, m.wide, G->stream);
    }
    if (k == LB_FV_PTILE) return launch_fv_ptile(G->prec, th, &A, resolved_shape(G), G->stream);
    if (k == LB_FV_MARCH) return launch_fv_march(G->prec, th, &A, resolved_chunk(G), G->stream);
    return launch_fv(G->prec, th, &A, scalar_shape(G), G->stream);
}

// Whether lb_step_fv runs the two-launch step of k_fv_phase.cu: FP64 grids
// of every size (the fused kernels recompute on the scarce FP64 pipe), and
// x-periodic FP32-math grids up to 128 cells per SM (thermal: 64), where the fused tile
// leaves most SMs idle: 128 x 128 FP32 takes 5.0 us a step against 5.5,
// 150 x 150 7.0 against 5.4; thermal 96 x 96 5.4 against 7.0, 110 x 110 9.2
// against 7.1.  Its kernels address a pair of opposite planes, which lie two
// planes apart, with 32-bit byte offsets: three planes stay below 2^32 bytes.
bool phase_applies(const lb_grid* G) {
    if (G->fv_scheme != LB_FV_HEUN || has_density_axis(G)) return false;
    const bool f64 = G->prec == Prec::F64;
    if (3ULL * G->plane * (f64 ? 8 : 4) >= 1ULL << 32) return false;
    if (G->fv_kernel != LB_FV_AUTO) return G->fv_kernel == LB_FV_TILE && G->fv_chunk == 2;
    return f64 || (pair_ok(G) && (G->d.thermal ? 2LL : 1LL) * G->nx * G->ny <= 128LL * G->sms);
}

// Whether a call of n steps of such an FP32-math grid gains by the two
// launches.  They pay a third launch per call, for h of its first state, so a
// short call takes the paired tile (the same bits): 64 x 64 6.3 us for one
// step against 5.2, 10.0 for two against 10.5; 139 x 139 8.8 against 5.4;
// thermal 98 x 98 16-bit 11.2 against 6.9.  In microseconds, measured from 0.1
// to 128 cells per SM: a step of two launches (slower at up to 8 cells per SM,
// where a CTA has 8 cells), the start of a call, and a step of the tile.
bool phase_pays(const lb_grid* G, int n) {
    if (G->fv_kernel != LB_FV_AUTO || G->prec == Prec::F64) return true;
    const bool th = G->d.thermal != 0, f16 = G->prec != Prec::F32;
    const double c = (double)G->nx * G->ny / G->sms, over = c > 25 ? c - 25 : 0;
    const double step = (c <= 8 ? 4.4 : th ? 4.0 : 3.7) + over * (th ? 0.043 : 0.014);
    const double start = 2.6 + over * (th ? 0.058 : 0.005);
    const double tile = (th ? c <= 2 ? 5.0 : 6.0 : 5.2) + (f16 ? 0.8 : 0.0);
    return start + n * step < n * tile;
}

// The two-launch step's fields (216 bytes a cell on FP64 flow grids, 432 on
// thermal ones), borrowed for a call: a grid holds none between calls.  A call
// that is being captured into a graph gets memory of the grid's own, which
// the graph's launches may use until lb_destroy.  Empty where there is no
// memory: the step then takes the fused kernels.
class PhaseFields {
public:
    explicit PhaseFields(lb_grid* G) : G_(G) {
        if (G->phase) return;  // the grid's own
        const size_t rs = G->prec == Prec::F64 ? 8 : 4;
        const size_t bytes = 3 * rs * (G->d.thermal ? 18 : 9) * (size_t)G->plane;
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        cudaError_t e = cudaStreamIsCapturing(G->stream, &cs);
        if (e == cudaSuccess && cs == cudaStreamCaptureStatusActive) {
            cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // an allocation is not part of the graph
            cudaThreadExchangeStreamCaptureMode(&mode);
            e = cudaMalloc(&G->phase, bytes);
            cudaThreadExchangeStreamCaptureMode(&mode);
        } else if (e == cudaSuccess && cs == cudaStreamCaptureStatusNone) {
            if (!G->borrower) scratch_join(G->device);
            G->borrower = true;
            e = scratch_take(&G->phase, bytes, G->device, G->stream);
            borrowed_ = e == cudaSuccess;
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            G->phase = nullptr;
        }
    }
    ~PhaseFields() {
        if (!borrowed_) return;
        scratch_give(G_->phase, G_->stream);
        G_->phase = nullptr;
    }
    PhaseFields(const PhaseFields&) = delete;
    PhaseFields& operator=(const PhaseFields&) = delete;
    explicit operator bool() const { return G_->phase != nullptr; }

private:
    lb_grid* G_;
    bool borrowed_ = false;
};

// start: h of the present state (before the first step of a call); else one step
template <typename R>
cudaError_t launch_phase(lb_grid* G, bool start) {
    const size_t set = (G->d.thermal ? 18 : 9) * (size_t)G->plane;
    R* w = static_cast<R*>(G->phase);
    PhaseArgs<R> P{};
    P.s = step_args<R>(G, G->p.dt);
    P.h = w;
    P.hs = w + set;
    P.b = w + 2 * set;
    P.foldx = static_cast<const R*>(G->fold[0]);
    P.foldy = static_cast<const R*>(G->fold[1]);
    const double dt = G->p.dt;
    for (int q = 0; q < 2; ++q) {
        const double k = dt / (2.0 * (q ? G->p.tau_g : G->p.tau) + dt);  // omh, omgh
        P.k[q] = (R)k;
        P.kh[q] = (R)(0.5 * k);
    }
    P.ctx = (R)(3.0 * 0.5 * dt * (1.0 - dt / (2.0 * G->p.tau + dt)) * G->p.ax);

    return launch_fv_phase(G->prec, G->d.thermal != 0, &P, start, G->sms, G->stream);
}

cudaError_t launch_phase(lb_grid* G, bool start) {
    return G->prec == Prec::F64 ? launch_phase<double>(G, start) : launch_phase<float>(G, start);
}

lb_status reduce(lb_grid* G, double out[kRed]) {
    CK(launch_reduce(G->prec, G->d.thermal != 0, aux_args(G), G->partial, G->nred, G->red, G->stream));
    CK(cudaMemcpyAsync(out, G->red, sizeof(double) * kRed, cudaMemcpyDeviceToHost, G->stream));
    CK(cudaStreamSynchronize(G->stream));
    return LB_OK;
}

// LB_ERR_UNSTABLE (and the grid poisoned) where a conservation sum is not finite.
lb_status finite_sums(lb_grid* G, const double* v) {
    for (int q = 0; q < 4; ++q)
        if (!std::isfinite(v[q])) {
            G->poisoned = true;
            return fail(LB_ERR_UNSTABLE, "non-finite conservation sum: the run diverged (dt too large "
                                         "for tau or the grid)");
        }
    return LB_OK;
}

// Nusselt numbers from the reductions.
lb_status nusselt_of(lb_grid* G, const double (&v)[kRed], double* nu_vol, double* nu_bot, double* nu_top) {
    const lb_params& p = G->p;
    const double H = G->d.ly, dT = p.T_bot - p.T_top, kappa = p.tau_g / 3.0, Lx = G->d.lx;
    if (nu_vol) *nu_vol = 1.0 + H * (v[4] / v[5]) / (kappa * dT);
    // plate gradients: quadratic through the wall value and the first two
    // x-averaged nodes, differentiated at the wall
    const double t0 = v[6] / Lx, t1 = v[7] / Lx, tn2 = v[8] / Lx, tn1 = v[9] / Lx;
    const double y0 = G->ay.c[0], y1 = G->ay.c[1];
    const double gb = -(y0 + y1) / (y0 * y1) * p.T_bot + y1 / (y0 * (y1 - y0)) * t0 - y0 / (y1 * (y1 - y0)) * t1;
    const double s0 = H - G->ay.c[G->ny - 1], s1 = H - G->ay.c[G->ny - 2];
    const double gt = -(s0 + s1) / (s0 * s1) * p.T_top + s1 / (s0 * (s1 - s0)) * tn1 - s0 / (s1 * (s1 - s0)) * tn2;
    if (nu_bot) *nu_bot = -H * gb / dT;
    if (nu_top) *nu_top = H * gt / dT;
    for (double x : v)
        if (!std::isfinite(x)) {
            G->poisoned = true;
            return fail(LB_ERR_UNSTABLE, "non-finite reduction: the run diverged");
        }
    return LB_OK;
}

// Capture n steps of `one` on the grid's private stream into an executable
// graph.  The state flips buffers n times (n even), so it is back where it
// started and the captured buffer pointers hold for every replay.  False,
// with nothing launched, where capture is unavailable: the grid's stream is
// itself being captured, or a call inside the capture is refused.
template <typename F>
bool capture_steps(lb_grid* G, int n, F& one, cudaGraphExec_t* exec, unsigned long long* per) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(G->stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    if (!G->cap && cudaStreamCreateWithFlags(&G->cap, cudaStreamNonBlocking) != cudaSuccess) {
        G->cap = nullptr;
        cudaGetLastError();
        return false;
    }
    const cudaStream_t user = G->stream;
    const int cur0 = G->cur;
    unsigned long long count = 0;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(G->cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        G->stream = G->cap;
        t_captured = &count;
        for (int j = 0; j < n && e == cudaSuccess; ++j) {
            e = one();
            G->cur ^= 1;
        }
        t_captured = nullptr;
        G->stream = user;
        const cudaError_t e2 = cudaStreamEndCapture(G->cap, &graph);
        if (e == cudaSuccess) e = e2;
    }
    G->cur = cur0;
    *exec = nullptr;
    if (e == cudaSuccess) e = cudaGraphInstantiate(exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *exec = nullptr;
        return false;
    }
    *per = count;
    return true;
}

// nsteps steps, each one call of `one` on G->stream followed by a buffer
// flip.  A run of more than 2 graph_steps steps takes its first step
// directly (first-use function attributes and buffers are set outside any
// capture), then replays a graph of graph_steps captured steps on the
// grid's stream and launches the remainder one by one.  The replays run the
// same kernels with the same arguments as the direct launches; the graph
// only takes the per-launch host and front-end cost off each step.
template <typename F>
lb_status run_steps(lb_grid* G, int nsteps, F one) {
    int k = 0;
    const int n = G->graph_steps;
    if (n > 0 && nsteps > 2 * n) {
        CK(one());
        G->cur ^= 1;
        ++k;
        cudaGraphExec_t exec = nullptr;
        unsigned long long per = 0;
        if (capture_steps(G, n, one, &exec, &per)) {
            cudaError_t e = cudaSuccess;
            for (; k + n <= nsteps; k += n) {
                e = cudaGraphLaunch(exec, G->stream);
                if (e != cudaSuccess) break;
                g_launches.fetch_add(per, std::memory_order_relaxed);
                ++G->graph_replays;
            }
            cudaGraphExecDestroy(exec);  // released once its queued replays have run
            CK(e);
        }
    }
    for (; k < nsteps; ++k) {
        CK(one());
        G->cur ^= 1;
    }
    return LB_OK;
}

}  // namespace

namespace lbgb {
// A served request leaves the batched paired tiles for launches of its own
// where the block march is faster than the request's share of full tile
// waves: thermal grids from about 512 x 512 (600 x 600, 16-bit: 29.5 us a
// step against 31.8), flow grids from about 450 x 450 (600 x 600, FP32: 13.4
// against 15.4).  Both kernels give the same bits.  160 requests of 64 x 64 to
// 1024 x 1024 queued at once, 16-bit: 9.4 -> 12.4 GLUPS, p99 2.33 -> 1.77 s.
bool march_served(const lb_grid* G) {
    const double wave = G->d.thermal ? 6.7 : 6.5 / 2;
    const long long tiles = (long long)((G->nx + 31) / 32) * ((G->ny + 15) / 16);
    return pair_ok(G) && march_plan(G, 0).us * G->sms < wave * (double)tiles;
}

// Mass and (thermal grids) Nusselt numbers from one reduction: the figures
// lb_conservation and lb_nusselt would give, and their status.
lb_status final_figures(lb_grid* G, double* mass, double* nu_vol, double* nu_bot, double* nu_top) {
    if (!G->has_params) return fail(LB_ERR_STATE, "grid has no parameters: call lb_init first");
    DeviceGuard dg(G->device);
    double v[kRed];
    lb_status s = reduce(G, v);
    if (s != LB_OK) return s;
    *mass = v[0];
    s = finite_sums(G, v);
    return s == LB_OK && G->d.thermal ? nusselt_of(G, v, nu_vol, nu_bot, nu_top) : s;
}
}  // namespace lbgb

extern "C" {

const char* lb_last_error(void) { return g_err.c_str(); }

unsigned long long lb_kernel_launches(void) { return g_launches.load(); }

static lb_status create_grid(const lb_grid_desc* d, lb_grid** out) {
    if (!d || !out) return fail(LB_ERR_ARG, "NULL description or output");
    if (d->nx < 1 || d->ny < 1) return fail(LB_ERR_ARG, "nx, ny must be >= 1 (got %d, %d)", d->nx, d->ny);
    if ((long long)d->nx * d->ny > (1LL << 31))
        return fail(LB_ERR_ARG, "grid of %d x %d cells is larger than supported", d->nx, d->ny);
    if (d->bcx < LB_BC_PERIODIC || d->bcx > LB_BC_DENSITY) return fail(LB_ERR_ARG, "bad bcx");
    if (d->bcy < LB_BC_PERIODIC || d->bcy > LB_BC_DENSITY) return fail(LB_ERR_ARG, "bad bcy");
    if ((d->bcx != LB_BC_PERIODIC && d->nx < 2) || (d->bcy != LB_BC_PERIODIC && d->ny < 2))
        return fail(LB_ERR_ARG, "a wall or density axis needs at least 2 cells (two ghost layers)");
    if (d->thermal && d->bcx != LB_BC_PERIODIC)
        return fail(LB_ERR_ARG, "thermal grids have their isothermal plates on y; x must be periodic");
    if (d->thermal && d->bcy == LB_BC_DENSITY)
        return fail(LB_ERR_ARG, "thermal grids have isothermal plates on y, not a density boundary");
    if (d->store < LB_STORE_F64 || d->store > LB_STORE_BF16DEV) return fail(LB_ERR_ARG, "bad store");
    for (int k = 0; k < 2; ++k) {
        const int sp = k ? d->sy : d->sx, n = k ? d->ny : d->nx;
        const double L = k ? d->ly : d->lx, st = k ? d->stretch_y : d->stretch_x;
        if (sp < LB_AXIS_UNIFORM || sp > LB_AXIS_CHEB) return fail(LB_ERR_ARG, "bad spacing");
        if (!(L > 0)) return fail(LB_ERR_ARG, "domain length must be > 0");
        if ((sp == LB_AXIS_TANH || sp == LB_AXIS_SINH) && !(st > 0)) return fail(LB_ERR_ARG, "stretch must be > 0");
        if (sp == LB_AXIS_SINH && (n % 2)) return fail(LB_ERR_ARG, "sinh spacing needs an even cell count");
    }
    struct Drop {
        void operator()(lb_grid* g) const {
            release(g);
            delete g;
        }
    };
    std::unique_ptr<lb_grid, Drop> G(new lb_grid());
    set_sizes(*G, *d);
    G->stream = static_cast<cudaStream_t>(d->cuda_stream);
    G->ax = make_axis(d->nx, d->lx, d->sx, d->stretch_x, d->bcx);
    G->ay = make_axis(d->ny, d->ly, d->sy, d->stretch_y, d->bcy);
    G->dmin = 1e300;
    for (double v : G->ax.d) G->dmin = std::fmin(G->dmin, v);
    for (double v : G->ay.d) G->dmin = std::fmin(G->dmin, v);
    for (int k = 0; k < 2; ++k) {
        const Axis& a = k ? G->ay : G->ax;
        for (double v : a.d)
            if (!(v > 0)) return fail(LB_ERR_ARG, "degenerate cell width on axis %c", k ? 'y' : 'x');
    }
    cudaGetDevice(&G->device);
    cudaDeviceGetAttribute(&G->sms, cudaDevAttrMultiProcessorCount, G->device);
    if (G->sms <= 0) G->sms = 152;
    // one allocation for everything the grid owns: creating and destroying a
    // 128 x 128 thermal grid took 0.30 ms with an allocation and a copy apiece
    // and takes 0.20, which a server pays for every request.  It comes before
    // the host tables, so that a grid the device cannot hold fails here.
    const size_t total = grid_device_bytes(*d);
    cudaError_t e = device_malloc(&G->arena, total);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? LB_ERR_OOM : LB_ERR_CUDA, "cudaMalloc(%zu bytes): %s", total,
                    cudaGetErrorString(e));
    }
    unsigned char* at = static_cast<unsigned char*>(G->arena);
    grid_parts(*G, [&](void** p, size_t bytes) {
        *p = at;
        at += part_size(bytes);
    });
    const bool f32 = G->prec != Prec::F64;
    HostTables tables(G->arena, G->toff);
    const std::vector<double> mxv = G->ax.metric();
    tables.put(G->mx, mxv, f32);
    tables.put(G->my, G->ay.metric(), f32);
    tables.put(G->fold[0], G->ax.cell_weights(f32), f32);
    tables.put(G->fold[1], G->ay.cell_weights(f32), f32);
    tables.put(G->dxv, G->ax.d, false);
    tables.put(G->dyv, G->ay.d, false);
    tables.put(G->xc, G->ax.c, false);
    tables.put(G->yc, G->ay.c, false);
    if (f32) {
        // x data of the column pair starting at each column (the right column wraps)
        const int nx = G->nx;
        auto wpv = [&](int r, int k) { return (float)mxv[r * (size_t)(nx + 1) + k]; };
        auto wmv = [&](int r, int k) { return (float)mxv[(3 + r) * (size_t)(nx + 1) + k]; };
        for (int c = 0; c < nx; ++c) {
            const int cr = (c + 1) % nx;
            float* t = tables.at<float>(G->coltab) + 20 * (size_t)c;
            for (int r = 0; r < 3; ++r) {
                t[r] = wpv(r, c);
                t[3 + r] = wpv(r, c + 1);
                t[6 + r] = wpv(r, cr + 1);
                t[9 + r] = wmv(r, c);
                t[12 + r] = wmv(r, c + 1);
                t[15 + r] = wmv(r, cr + 1);
            }
            t[18] = (float)mxv[6 * (size_t)(nx + 1) + c];
            t[19] = (float)mxv[6 * (size_t)(nx + 1) + cr];
        }
    }
    e = tables.upload();
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, "table upload: %s", cudaGetErrorString(e));
    *out = G.release();
    return LB_OK;
}

lb_status lb_create_grid(const lb_grid_desc* d, lb_grid** out) {
    try {
        return create_grid(d, out);
    } catch (const std::bad_alloc&) {
        return fail(LB_ERR_OOM, "no host memory for the grid's tables");
    }
}

lb_status lb_destroy(lb_grid* G) {
    if (!G) return LB_OK;
    DeviceGuard dg(G->device);
    cudaStreamSynchronize(G->stream);
    if (G->borrower) scratch_leave(G->device);
    release(G);
    delete G;
    return LB_OK;
}

lb_status lb_sync(lb_grid* G) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    DeviceGuard dg(G->device);
    CK(cudaStreamSynchronize(G->stream));
    return LB_OK;
}

static lb_status init_grid(lb_grid* G, const lb_params* p, const lb_init_desc* in) {
    if (!G || !p || !in) return fail(LB_ERR_ARG, "NULL argument");
    if (!(p->tau > 0) || !(p->dt > 0)) return fail(LB_ERR_ARG, "tau and dt must be > 0");
    if (G->d.thermal && !(p->tau_g > 0)) return fail(LB_ERR_ARG, "tau_g must be > 0 on a thermal grid");
    if (in->kind < LB_INIT_TGV || in->kind > LB_INIT_FIELDS) return fail(LB_ERR_ARG, "bad init kind");
    if (in->kind == LB_INIT_RB && !G->d.thermal) return fail(LB_ERR_ARG, "RB preset needs a thermal grid");
    DeviceGuard dg(G->device);
    // Reference state of the storage: the barometric density and conductive
    // temperature of the RB base state on a grid with plates, else 1 and T0.
    double rho_norm = 1.0;
    const double dTp = p->T_bot - p->T_top, bgp = p->beta * p->grav, Hy = G->d.ly;
    auto baro = [&](double y) { return std::exp(3.0 * bgp * dTp * (0.5 * y - 0.5 * y * y / Hy)); };
    if (in->kind == LB_INIT_RB) {
        double s = 0.0;
        for (int j = 0; j < G->ny; ++j) s += G->ay.d[j] * baro(G->ay.c[j]);
        rho_norm = Hy / s;  // sum V rho = sum V
    }
    {
        std::vector<double> to(G->ny, 0.0), ro(G->ny, 0.0);
        const bool plates = G->d.thermal && G->d.bcy == LB_BC_WALLS;
        for (int j = 0; j < G->ny; ++j) {
            if (plates) to[j] = dTp * (0.5 - G->ay.c[j] / Hy) + 0.5 * (p->T_bot + p->T_top) - p->T0;
            if (in->kind == LB_INIT_RB) ro[j] = rho_norm * baro(G->ay.c[j]) - 1.0;
        }
        // y flux divergence of the base state per row and upwind sign, with
        // the same QUICK weights as the kernels; ghost rows extend rho_r
        // evenly and T_r oddly about the plate temperature.
        const int ny = G->ny;
        const bool wall = G->d.bcy == LB_BC_WALLS;
        auto ext = [&](const std::vector<double>& v, int i, double wall_lo, double wall_hi, bool odd) {
            if (i >= 0 && i < ny) return v[i];
            if (!wall) return v[((i % ny) + ny) % ny];
            if (i < 0) return odd ? 2.0 * wall_lo - v[-i - 1] : v[-i - 1];
            return odd ? 2.0 * wall_hi - v[2 * ny - 1 - i] : v[2 * ny - 1 - i];
        };
        std::vector<double> dref(4 * (size_t)ny, 0.0);
        for (int q = 0; q < 2; ++q) {
            const std::vector<double>& v = q ? to : ro;
            const double lo = q ? p->T_bot - p->T0 : 0.0, hi = q ? p->T_top - p->T0 : 0.0;
            bool any = false;
            for (double x : v) any = any || x != 0.0;
            if (!any) continue;
            for (int sgn = 0; sgn < 2; ++sgn) {
                auto face = [&](int kf) {
                    const int k0 = sgn == 0 ? kf - 2 : kf - 1;
                    double w[3];
                    G->ay.quick(k0, kf, w);
                    double phi = 0.0;
                    for (int m = 0; m < 3; ++m) phi += w[m] * ext(v, k0 + m, lo, hi, q == 1);
                    return phi;
                };
                for (int j = 0; j < ny; ++j) dref[(2 * q + sgn) * ny + j] = (face(j + 1) - face(j)) / G->ay.d[j];
            }
        }
        const bool f32 = G->prec != Prec::F64;
        HostTables tables(G->toff, G->partial);
        tables.put(G->toff, to, false);
        tables.put(G->roff, ro, false);
        tables.put(G->toff_r, to, f32);
        tables.put(G->roff_r, ro, f32);
        tables.put(G->dref_r, dref, f32);
        if (f32) {
            // per-row table of the paired kernels: one 80-byte entry per row
            const std::vector<double> my = G->ay.metric();
            for (int j = 0; j < ny; ++j) {
                float* t = tables.at<float>(G->rowtab) + 20 * (size_t)j;
                for (int q = 0; q < 3; ++q) {
                    t[q] = (float)my[q * (size_t)(ny + 1) + j];            // c > 0, south face j
                    t[3 + q] = (float)my[q * (size_t)(ny + 1) + j + 1];    // c > 0, north face j + 1
                    t[6 + q] = (float)my[(3 + q) * (size_t)(ny + 1) + j];  // c < 0, south
                    t[9 + q] = (float)my[(3 + q) * (size_t)(ny + 1) + j + 1];
                }
                t[12] = (float)my[6 * (size_t)(ny + 1) + j];
                t[13] = (float)ro[j];
                t[14] = (float)to[j];
                for (int q = 0; q < 4; ++q) t[15 + q] = (float)dref[q * (size_t)ny + j];
            }
        }
        CK(tables.upload());
    }
    InitArgs a{};
    a.f = G->f[0];
    a.g = G->g[0];
    a.nx = G->nx;
    a.ny = G->ny;
    a.pitch = G->pitch;
    a.plane = G->plane;
    a.kind = in->kind;
    a.mode = in->mode;
    a.u0 = in->u0;
    a.amp = in->amp;
    a.seed = in->seed;
    a.lx = G->d.lx;
    a.ly = G->d.ly;
    a.dt = G->fv_scheme == LB_FV_EULER ? 0.0 : p->dt;  // f~ = f_eq - dt/2 F; Euler starts at f_eq
    a.ax = p->ax;
    a.ay = p->ay;
    a.bg = p->beta * p->grav;
    a.T0 = p->T0;
    a.Tb = p->T_bot;
    a.Tt = p->T_top;
    a.xc = G->xc;
    a.yc = G->yc;
    a.toff = G->toff;
    a.roff = G->roff;
    a.fields = G->fields;
    a.rho_norm = rho_norm;
    if (in->kind == LB_INIT_FIELDS) {
        // each host field straight into the staging buffer (a DMA when the
        // caller's memory is pinned); absent fields filled on the device
        const long long n = (long long)G->nx * G->ny;
        const double* src[4] = {in->rho, in->ux, in->uy, in->T};
        const double fill[4] = {1.0, 0.0, 0.0, p->T0};
        for (int k = 0; k < 4; ++k) {
            if (src[k])
                CK(cudaMemcpyAsync(G->fields + k * n, src[k], sizeof(double) * n, cudaMemcpyHostToDevice, G->stream));
            else
                CK(launch_fill(G->fields + k * n, n, fill[k], G->stream));
        }
        // the density is checked before the populations are touched, so a
        // rejected call leaves the grid's state as it was
        unsigned long long* first = reinterpret_cast<unsigned long long*>(G->red);
        unsigned long long bad = ~0ULL;
        CK(launch_first_nonpositive(G->fields, n, first, G->stream));
        CK(cudaMemcpyAsync(&bad, first, sizeof(bad), cudaMemcpyDeviceToHost, G->stream));
        CK(cudaStreamSynchronize(G->stream));  // the host arrays are read before return
        if (bad != ~0ULL) return fail(LB_ERR_ARG, "density must be > 0 (cell %llu)", bad);
        CK(launch_init(G->prec, G->d.thermal != 0, a, G->stream));
    } else {
        CK(launch_init(G->prec, G->d.thermal != 0, a, G->stream));
    }
    G->p = *p;
    G->has_params = true;
    G->poisoned = false;
    G->cur = 0;
    return LB_OK;
}

lb_status lb_init(lb_grid* G, const lb_params* p, const lb_init_desc* in) {
    try {
        return init_grid(G, p, in);
    } catch (const std::bad_alloc&) {
        return fail(LB_ERR_OOM, "no host memory for the grid's tables");
    }
}

lb_status lb_step_fv(lb_grid* G, int nsteps) {
    lb_status s = check_ready(G);
    if (s != LB_OK) return s;
    if (nsteps < 0) return fail(LB_ERR_ARG, "nsteps must be >= 0");
    DeviceGuard dg(G->device);
    if (nsteps > 0 && phase_applies(G) && phase_pays(G, nsteps)) {
        const PhaseFields fields(G);
        if (fields) {
            CK(launch_phase(G, true));
            return run_steps(G, nsteps, [G] { return launch_phase(G, false); });
        }
    }
    return run_steps(G, nsteps,
                     [G] { return G->prec == Prec::F64 ? launch_fv_step<double>(G) : launch_fv_step<float>(G); });
}

lb_status lb_set_graph_steps(lb_grid* G, int n) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (n < 0 || n % 2 != 0 || n > 4096) return fail(LB_ERR_ARG, "graph length must be even, 0..4096 (got %d)", n);
    G->graph_steps = n;
    return LB_OK;
}

lb_status lb_get_graph_steps(lb_grid* G, int* n, unsigned long long* replays) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (n) *n = G->graph_steps;
    if (replays) *replays = G->graph_replays;
    return LB_OK;
}

lb_status lb_set_fv_schedule(lb_grid* G, int kernel, int chunk) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (kernel < LB_FV_AUTO || kernel > LB_FV_SPLIT) return fail(LB_ERR_ARG, "unknown FV kernel %d", kernel);
    if (chunk < 0) return fail(LB_ERR_ARG, "chunk must be >= 0");
    if (kernel == LB_FV_TILE && chunk != 0 && chunk != 8 && chunk != 16 && chunk != 2)
        return fail(LB_ERR_ARG, "tile shape must be 0 (32 x 16), 16 (16 x 16), 8 (16 x 8) or 2 (two launches, no tile)");
    if (kernel == LB_FV_PTILE && chunk != 0 && chunk != 14 && chunk != 16 && chunk != 512 && chunk != 526)
        return fail(LB_ERR_ARG, "paired tile shape must be 0 (32 x 16), 14 (32 x 14), 16 (16 x 16), 512 (32 x 16, "
                                "512 threads) or 526 (32 x 14, 512 threads)");
    if (kernel == LB_FV_SPLIT && chunk != 0 && chunk != 16)
        return fail(LB_ERR_ARG, "split tile shape must be 0 (32 x 16) or 16 (16 x 16)");
    if ((kernel == LB_FV_PAIR || kernel == LB_FV_PTILE || kernel == LB_FV_SPLIT) && !pair_ok(G))
        return fail(LB_ERR_ARG, "the paired FV kernel needs FP32/FP16/BF16 storage and a periodic x axis");
    G->fv_kernel = kernel;
    G->fv_chunk = chunk;
    return LB_OK;
}

lb_status lb_set_fv_scheme(lb_grid* G, int scheme) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (scheme < LB_FV_HEUN || scheme > LB_FV_EULER) return fail(LB_ERR_ARG, "unknown FV scheme %d", scheme);
    if (scheme != G->fv_scheme) {
        G->fv_scheme = scheme;
        G->has_params = false;  // the state's meaning changed: lb_init again
    }
    return LB_OK;
}

lb_status lb_set_boundary_density(lb_grid* G, double rho_x0, double rho_x1, double rho_y0, double rho_y1) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!(rho_x0 > 0) || !(rho_x1 > 0) || !(rho_y0 > 0) || !(rho_y1 > 0))
        return fail(LB_ERR_ARG, "boundary densities must be > 0");
    G->rho_bc[0] = rho_x0;
    G->rho_bc[1] = rho_x1;
    G->rho_bc[2] = rho_y0;
    G->rho_bc[3] = rho_y1;
    return LB_OK;
}

lb_status lb_get_fv_scheme(lb_grid* G, int* scheme) {
    if (!G || !scheme) return fail(LB_ERR_ARG, "NULL argument");
    *scheme = G->fv_scheme;
    return LB_OK;
}

lb_status lb_get_fv_schedule(lb_grid* G, int* kernel, int* chunk) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (phase_applies(G)) {
        if (kernel) *kernel = LB_FV_TILE;
        if (chunk) *chunk = 2;
        return LB_OK;
    }
    if (kernel) *kernel = resolved_kernel(G);
    if (chunk) {
        const int k = resolved_kernel(G);
        *chunk = k == LB_FV_PTILE                        ? resolved_shape(G)
                 : k == LB_FV_TILE                       ? scalar_shape(G)
                 : k == LB_FV_SPLIT                      ? G->fv_chunk
                                                       : resolved_chunk(G);
    }
    return LB_OK;
}

lb_status lb_autotune_fv(lb_grid* G, int steps) {
    lb_status s = check_ready(G);
    if (s != LB_OK) return s;
    if (steps < 1) return fail(LB_ERR_ARG, "steps must be >= 1");
    DeviceGuard dg(G->device);
    const size_t bytes = (size_t)Q * G->plane * elem_size(G->d.store);
    void *sf = nullptr, *sg = nullptr;
    CK(device_malloc(&sf, bytes));
    if (G->d.thermal && device_malloc(&sg, bytes) != cudaSuccess) {
        cudaFree(sf);
        return fail(LB_ERR_OOM, "autotune: no memory for the state copy");
    }
    const int cur0 = G->cur;
    cudaMemcpyAsync(sf, G->f[cur0], bytes, cudaMemcpyDeviceToDevice, G->stream);
    if (sg) cudaMemcpyAsync(sg, G->g[cur0], bytes, cudaMemcpyDeviceToDevice, G->stream);
    const int k0 = G->fv_kernel, c0 = G->fv_chunk;
    std::vector<std::pair<int, int>> cands = {{LB_FV_TILE, 0}, {LB_FV_TILE, 16}, {LB_FV_TILE, 8}};
    if (pair_ok(G)) {
        cands.push_back({LB_FV_PTILE, 0});
        cands.push_back({LB_FV_PTILE, 16});
        cands.push_back({LB_FV_PTILE, 512});
        cands.push_back({LB_FV_PTILE, 14});
        cands.push_back({LB_FV_PTILE, 526});
        if (ensure_split_buffers(G) == cudaSuccess) {
            cands.push_back({LB_FV_SPLIT, 0});
            cands.push_back({LB_FV_SPLIT, 16});
        }
    }
    cands.push_back({LB_FV_TILE, 2});
    for (int kern : {(int)LB_FV_MARCH, (int)LB_FV_PAIR}) {
        if (kern == LB_FV_PAIR && !pair_ok(G)) continue;
        G->fv_kernel = kern;
        G->fv_chunk = 0;
        const int base = resolved_chunk(G);
        for (int ch : {base / 2, base, base * 2, 32, 64, 128})
            if (ch >= 16 && ch <= 4 * G->ny) cands.push_back({kern, ch});
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    std::pair<int, int> pick = {LB_FV_TILE, 0};
    lb_status st = LB_OK;
    for (auto& c : cands) {
        G->fv_kernel = c.first;
        G->fv_chunk = c.second;
        G->cur = cur0;
        const bool phase = c == std::make_pair((int)LB_FV_TILE, 2);
        if (phase && !phase_applies(G)) continue;
        std::optional<PhaseFields> fields;
        if (phase) {
            fields.emplace(G);
            if (!*fields) continue;
        }
        auto one = [&] {
            return phase ? launch_phase(G, false)
                         : G->prec == Prec::F64 ? launch_fv_step<double>(G) : launch_fv_step<float>(G);
        };
        // warm-up step, then the timed ones as one call of lb_step_fv takes them
        auto start = [&] { return phase ? launch_phase(G, true) : cudaSuccess; };
        cudaError_t e = start();
        if (e == cudaSuccess) e = one();
        G->cur ^= 1;
        cudaEventRecord(e0, G->stream);
        if (e == cudaSuccess) e = start();
        for (int k = 0; k < steps && e == cudaSuccess; ++k) {
            e = one();
            G->cur ^= 1;
        }
        cudaEventRecord(e1, G->stream);
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        if (e != cudaSuccess) {
            st = fail(LB_ERR_CUDA, "autotune: %s", cudaGetErrorString(e));
            break;
        }
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        if (ms < best) {
            best = ms;
            pick = c;
        }
    }
    // restore the state into the buffer it started in
    G->cur = cur0;
    cudaMemcpyAsync(G->f[cur0], sf, bytes, cudaMemcpyDeviceToDevice, G->stream);
    if (sg) cudaMemcpyAsync(G->g[cur0], sg, bytes, cudaMemcpyDeviceToDevice, G->stream);
    cudaStreamSynchronize(G->stream);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(sf);
    if (sg) cudaFree(sg);
    if (st != LB_OK) {
        G->fv_kernel = k0;
        G->fv_chunk = c0;
        return st;
    }
    G->fv_kernel = pick.first;
    G->fv_chunk = pick.second;
    return LB_OK;
}

lb_status lb_step_st(lb_grid* G, int nsteps) {
    lb_status s = check_ready(G);
    if (s != LB_OK) return s;
    if (nsteps < 0) return fail(LB_ERR_ARG, "nsteps must be >= 0");
    if (G->fv_scheme == LB_FV_EULER) return fail(LB_ERR_STATE, "ST steps tilded populations, not an Euler grid");
    if (has_density_axis(G)) return fail(LB_ERR_ARG, "the fixed-density boundary is an FV boundary (no ST form)");
    for (int k = 0; k < 2; ++k) {
        const int sp = k ? G->d.sy : G->d.sx, n = k ? G->ny : G->nx;
        const double L = k ? G->d.ly : G->d.lx;
        if (sp != LB_AXIS_UNIFORM || std::fabs(L / n - 1.0) > 1e-12)
            return fail(LB_ERR_ARG, "ST needs uniform axes with unit spacing (axis %c: L/n = %g)",
                        k ? 'y' : 'x', L / n);
    }
    if (std::fabs(G->p.dt - 1.0) > 1e-12) return fail(LB_ERR_ARG, "ST needs dt = 1 (got %g)", G->p.dt);
    DeviceGuard dg(G->device);
    const bool th = G->d.thermal != 0;
    return run_steps(G, nsteps, [G, th] {
        if (G->prec == Prec::F64) {
            StepArgs<double> A = step_args<double>(G, 1.0);
            return launch_st(G->prec, th, &A, G->stream);
        }
        StepArgs<float> A = step_args<float>(G, 1.0);
        if (st16_applies(G->prec, th, G->nx, G->d.bcx)) return launch_st16(G->prec, &A, G->stream);
        if (st_quad_applies(G->prec, th, G->nx, G->d.bcx)) return launch_st_quad(&A, G->stream);
        return launch_st(G->prec, th, &A, G->stream);
    });
}

lb_status lb_moments(lb_grid* G, double* rho, double* ux, double* uy, double* T) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!G->has_params) return fail(LB_ERR_STATE, "grid has no parameters: call lb_init first");
    DeviceGuard dg(G->device);
    CK(launch_moments(G->prec, G->d.thermal != 0, aux_args(G), G->fields, G->stream));
    const size_t n = (size_t)G->nx * G->ny;
    double* outs[4] = {rho, ux, uy, T};
    for (int k = 0; k < 4; ++k)
        if (outs[k])
            CK(cudaMemcpyAsync(outs[k], G->fields + k * n, sizeof(double) * n, cudaMemcpyDeviceToHost,
                               G->stream));
    CK(cudaStreamSynchronize(G->stream));
    return LB_OK;
}

lb_status lb_conservation(lb_grid* G, double* mass, double* momx, double* momy, double* heat) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!G->has_params) return fail(LB_ERR_STATE, "grid has no parameters: call lb_init first");
    DeviceGuard dg(G->device);
    double v[kRed];
    lb_status s = reduce(G, v);
    if (s != LB_OK) return s;
    if (mass) *mass = v[0];
    if (momx) *momx = v[1];
    if (momy) *momy = v[2];
    if (heat) *heat = v[3];
    return finite_sums(G, v);
}

lb_status lb_nusselt(lb_grid* G, double* nu_vol, double* nu_bot, double* nu_top) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!G->d.thermal) return fail(LB_ERR_STATE, "Nusselt numbers need a thermal grid");
    if (!G->has_params) return fail(LB_ERR_STATE, "grid has no parameters: call lb_init first");
    DeviceGuard dg(G->device);
    double v[kRed];
    lb_status s = reduce(G, v);
    if (s != LB_OK) return s;
    return nusselt_of(G, v, nu_vol, nu_bot, nu_top);
}

lb_status lb_set_populations(lb_grid* G, const double* f, const double* g) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!G->has_params) return fail(LB_ERR_STATE, "set parameters with lb_init before setting populations");
    if (g && !G->d.thermal) return fail(LB_ERR_STATE, "thermal populations on a flow-only grid");
    DeviceGuard dg(G->device);
    const size_t n = (size_t)Q * G->nx * G->ny;
    double* tmp = nullptr;
    CK(device_malloc((void**)&tmp, sizeof(double) * n));
    lb_status st = LB_OK;
    const double* srcs[2] = {f, g};
    void* dsts[2] = {G->f[G->cur], G->g[G->cur]};
    const double offs[2] = {1.0, G->p.T0};
    const double* rowoffs[2] = {G->roff, G->toff};
    for (int k = 0; k < 2 && st == LB_OK; ++k) {
        if (!srcs[k]) continue;
        cudaError_t e = cudaMemcpy(tmp, srcs[k], sizeof(double) * n, cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = launch_pack(G->prec, tmp, dsts[k], G->nx, G->ny, G->pitch, G->plane, offs[k], rowoffs[k],
                            G->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(G->stream);
        if (e != cudaSuccess) st = fail(LB_ERR_CUDA, "set_populations: %s", cudaGetErrorString(e));
    }
    cudaFree(tmp);
    return st;
}

lb_status lb_get_window(lb_grid* G, int x0, int y0, int w, int h, double* f, double* g) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    if (!G->has_params) return fail(LB_ERR_STATE, "grid has no parameters: call lb_init first");
    if (g && !G->d.thermal) return fail(LB_ERR_STATE, "thermal populations on a flow-only grid");
    if (w < 1 || h < 1 || w > G->nx || h > G->ny)
        return fail(LB_ERR_ARG, "window %d x %d does not fit a %d x %d grid", w, h, G->nx, G->ny);
    DeviceGuard dg(G->device);
    x0 = ((x0 % G->nx) + G->nx) % G->nx;
    y0 = ((y0 % G->ny) + G->ny) % G->ny;
    const size_t n = (size_t)Q * w * h;
    double* tmp = nullptr;
    CK(device_malloc((void**)&tmp, sizeof(double) * n));
    lb_status st = LB_OK;
    double* dsts[2] = {f, g};
    const void* srcs[2] = {G->f[G->cur], G->g[G->cur]};
    const double offs[2] = {1.0, G->p.T0};
    const double* rowoffs[2] = {G->roff, G->toff};
    for (int k = 0; k < 2 && st == LB_OK; ++k) {
        if (!dsts[k]) continue;
        cudaError_t e = launch_unpack(G->prec, srcs[k], tmp, G->nx, G->ny, G->pitch, G->plane, offs[k],
                                      rowoffs[k], x0, y0, w, h, G->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dsts[k], tmp, sizeof(double) * n, cudaMemcpyDeviceToHost, G->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(G->stream);
        if (e != cudaSuccess) st = fail(LB_ERR_CUDA, "get_window: %s", cudaGetErrorString(e));
    }
    cudaFree(tmp);
    return st;
}

lb_status lb_get_populations(lb_grid* G, double* f, double* g) {
    if (!G) return fail(LB_ERR_ARG, "grid is NULL");
    return lb_get_window(G, 0, 0, G->nx, G->ny, f, g);
}

}  // extern "C"
