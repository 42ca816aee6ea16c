// lb_scratch.cu -- device memory borrowed for the length of a call.
//
// One memory pool per device.  A loan is taken and given back in stream order
// (2 us of host time the pair), so it costs no synchronisation and grids on
// several streams and threads hold only what their running calls need.  The
// pool keeps kKeep of what was given back; the rest returns to the device at
// the next synchronisation, and all of it when the last borrower leaves or an
// allocation of the library fails.  A loan beyond kKeep maps its memory anew
// after each synchronisation: 2 ms per GiB, against the tens of ms that a
// call of a grid of that size takes.
#include "lb_scratch.cuh"

#include <cstdint>
#include <map>
#include <mutex>

namespace lbgb {

namespace {

constexpr uint64_t kKeep = 1ULL << 30;

struct Pool {
    cudaMemPool_t pool = nullptr;
    int borrowers = 0;
};
std::mutex g_mu;
std::map<int, Pool>& pools() {
    static std::map<int, Pool>* p = new std::map<int, Pool>;  // lives until the process ends
    return *p;
}

// Another thread's stream capture does not forbid what happens here.
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

cudaError_t open_pool(Pool& P, int device) {
    if (P.pool) return cudaSuccess;
    RelaxedCapture relaxed;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    uint64_t keep = kKeep;
    // a loan never waits for another stream's work: two grids on two streams stay independent
    int wait = 0;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &wait);
    if (e != cudaSuccess) {
        cudaMemPoolDestroy(pool);
        return e;
    }
    P.pool = pool;
    return cudaSuccess;
}

}  // namespace

cudaError_t scratch_take(void** p, size_t bytes, int device, cudaStream_t s) {
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        Pool& P = pools()[device];
        const cudaError_t e = open_pool(P, device);
        if (e != cudaSuccess) return e;
        pool = P.pool;
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

void scratch_give(void* p, cudaStream_t s) { cudaFreeAsync(p, s); }

void scratch_join(int device) {
    std::lock_guard<std::mutex> lock(g_mu);
    ++pools()[device].borrowers;
}

void scratch_leave(int device) {
    std::lock_guard<std::mutex> lock(g_mu);
    Pool& P = pools()[device];
    if (--P.borrowers == 0 && P.pool) cudaMemPoolTrimTo(P.pool, 0);
}

bool scratch_reclaim(int device) {
    std::lock_guard<std::mutex> lock(g_mu);
    const auto it = pools().find(device);
    uint64_t held = 0;
    if (it == pools().end() || !it->second.pool ||
        cudaMemPoolGetAttribute(it->second.pool, cudaMemPoolAttrReservedMemCurrent, &held) != cudaSuccess || held == 0)
        return false;
    return cudaDeviceSynchronize() == cudaSuccess && cudaMemPoolTrimTo(it->second.pool, 0) == cudaSuccess;
}

cudaError_t device_malloc(void** p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    int device = 0;
    if (e == cudaErrorMemoryAllocation && cudaGetDevice(&device) == cudaSuccess && scratch_reclaim(device)) {
        cudaGetLastError();
        e = cudaMalloc(p, bytes);
    }
    return e;
}

}  // namespace lbgb
