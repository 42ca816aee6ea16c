// lb_launch.cuh -- launchers of the 2-D kernels, implemented in the kernel
// translation units and called by the host side.
#pragma once

#include "lb_internal.cuh"

namespace lbgb {

cudaError_t launch_st(Prec p, bool thermal, const void* args, cudaStream_t s);
cudaError_t launch_fv(Prec p, bool thermal, const void* args, int shape, cudaStream_t s);
// One request of a batched FV launch: its step parameters, both buffers
// of each population set, the parity of its current state at step 0 of the
// launch sequence and how many steps it still has to take.
template <typename R>
struct BatchReq {
    StepArgs<R> args;
    void* f[2];
    void* g[2];
    int parity;
    int remaining;
};
// tiles[b] = (request, tile x, tile y, 0); CTAs beyond *ntiles exit
cudaError_t launch_fv_batched(Prec p, bool thermal, const void* reqs, const int4* tiles, const int* ntiles,
                              int capacity, int k, cudaStream_t s);
void tile_shape(Prec p, bool thermal, int* tx, int* ty);
// y-marching FV kernel: strips of march_width() output columns, `chunk` rows per CTA
cudaError_t launch_fv_march(Prec p, bool thermal, const void* args, int chunk, cudaStream_t s);
int march_width(Prec p, bool thermal);
size_t march_smem(Prec p, bool thermal);
// march in blocks of four rows, packed FP32 pairs (x-periodic grids only): strips of
// blocks_width() columns, `chunk` rows per CTA (rounded up to a multiple of 4);
// wide: one CTA per SM, else (flow grids) two of half the strip
cudaError_t launch_fv_blocks(Prec p, bool thermal, const void* args, int chunk, bool wide, cudaStream_t s);
int blocks_width(bool thermal, bool wide);
// paired tile kernel: shape 0 = 32 x 16, 16 = 16 x 16 (x-periodic, FP32 arithmetic)
cudaError_t launch_fv_ptile(Prec p, bool thermal, const void* args, int shape, cudaStream_t s);
// split paired schedule: two launches per step (collision + predictor, corrector),
// h* and f~ + Coll - dt/2 A[h^n] through the xh / xfc buffers
cudaError_t launch_fv_split(Prec p, bool thermal, const void* args, int shape, cudaStream_t s);
// batched paired tile (32 x 16) over a request table, as launch_fv_batched
cudaError_t launch_fv_ptile_batched(Prec p, bool thermal, const void* reqs, const int4* tiles, const int* ntiles,
                                    int capacity, int k, cudaStream_t s);

struct AuxArgs {
    const void* f;  // state buffers (deviation storage)
    const void* g;
    int nx, ny, pitch;
    long long plane;
    double dt, ax, ay, bg, T0;
    const double* toff; // per-row storage offset of g (thermal grids)
    const double* roff; // per-row storage offset of f
    const double* dxv;  // cell widths x (nx), FP64
    const double* dyv;  // cell widths y (ny)
    const double* xc;   // centres x
    const double* yc;   // centres y
};

// Moments of every cell into out[4][ny][nx] (rho, ux, uy, T), FP64.
cudaError_t launch_moments(Prec p, bool thermal, const AuxArgs& a, double* out, cudaStream_t s);
// Block partial sums of the reduction quantities (kRed values) then a final
// fixed-order sum into out[kRed].
constexpr int kRed = 10;
cudaError_t launch_reduce(Prec p, bool thermal, const AuxArgs& a, double* partial, int nblocks,
                          double* out, cudaStream_t s);
int reduce_blocks(int nx, int ny);

// Populations FP64 host layout [9][ny][nx] (device copy) -> storage, and back.
// Stored value = value - w (off + rowoff[y]); rowoff may be NULL.
cudaError_t launch_pack(Prec p, const double* src, void* dst, int nx, int ny, int pitch,
                        long long plane, double off, const double* rowoff, cudaStream_t s);
// Window [9][h][w] starting at (x0, y0), indices wrapping modulo nx, ny.
cudaError_t launch_unpack(Prec p, const void* src, double* dst, int nx, int ny, int pitch,
                          long long plane, double off, const double* rowoff, int x0, int y0, int w,
                          int h, cudaStream_t s);

struct InitArgs {
    void* f;
    void* g;
    int nx, ny, pitch;
    long long plane;
    int kind, mode;
    double u0, amp;
    unsigned long long seed;
    double lx, ly;
    double dt, ax, ay, bg, T0, Tb, Tt;
    double rho_norm;
    const double* toff;
    const double* roff;
    const double* xc;
    const double* yc;
    const double* fields;  // LB_INIT_FIELDS: [4][ny][nx] rho, ux, uy, T on device
};
cudaError_t launch_init(Prec p, bool thermal, const InitArgs& a, cudaStream_t s);
// n doubles at p set to v; and the smallest index i with !(rho[i] > 0) into
// *first (all ones when there is none)
cudaError_t launch_fill(double* p, long long n, double v, cudaStream_t s);
cudaError_t launch_first_nonpositive(const double* rho, long long n, unsigned long long* first, cudaStream_t s);

}  // namespace lbgb
