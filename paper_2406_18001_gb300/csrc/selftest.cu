// selftest.cu -- failure-path hooks of libdcd_gb300.so, for testing how the
// library reports failures without faulting, trapping or hanging a GPU.
//
// dcd_selftest_bounded_wait: every wait on an mbarrier in the library's
// kernels is bounded; when the bound runs out the kernel records DEV_TIMEOUT
// in the device error word, stops waiting and returns, and the host turns the
// word into DCD_ETIMEOUT.  The self-test runs that path for real: one thread
// waits, with the library's bounded wait, on an mbarrier whose arrival count
// (2) is never reached (one arrival).
//
// dcd_inject_alloc_failures: the next `count` device allocations the library
// makes fail as if the device were out of memory (DCD_ENOMEM), a fake of the
// failing call made on the host.
#include "dcd_internal.cuh"
#include "ptx.cuh"

#include <cuda.h>

#include <atomic>
#include <mutex>

namespace dcd {
namespace {

std::atomic<int> g_fail_allocs{0};

// The number of the current context (one is made where none is current, or the one that was has been
// reset), never used twice in a process; 0: it cannot be had.
unsigned long long context_id(int dev)
{
    typedef CUresult(CUDAAPI * GetId)(CUcontext, unsigned long long *);
    static const GetId get = [] {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        return cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                       q == cudaDriverEntryPointSuccess
                   ? (GetId)p
                   : nullptr;
    }();
    unsigned long long id = 0;
    if (!get) return 0;
    if (get(nullptr, &id) == CUDA_SUCCESS) return id;
    if (cudaSetDevice(dev) != cudaSuccess || get(nullptr, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// The library's own memory pool in the current context (nullptr: none could be made; a stream-ordered
// pool, so safe from several threads and streams).  It keeps at most POOL_KEEP of freed memory mapped:
// the default pool returns all of it to the driver at every synchronisation, and mapping it again took
// 50 to 170 us of an allocation after one (a sweep of 32 plans: 19.7 -> 15.9 ms on one host, 22.0 -> 19.0
// on another).  What it keeps goes
// back when an allocation of the library's fails, and with the process.  A pool dies with its context
// (cudaDeviceReset), so pools go by the context's number.
constexpr size_t POOL_CONTEXTS = 64;
constexpr uint64_t POOL_KEEP = 512ull << 20;

cudaMemPool_t context_pool()
{
    struct Entry {
        unsigned long long id;
        cudaMemPool_t pool;
    };
    static std::mutex mu;
    static Entry pools[POOL_CONTEXTS];
    static size_t count = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    const unsigned long long id = context_id(dev);
    if (!id) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    for (size_t i = 0; i < count; ++i)
        if (pools[i].id == id) return pools[i].pool;
    if (count == POOL_CONTEXTS) return nullptr;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    uint64_t keep = POOL_KEEP;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();
        pool = nullptr;
    } else if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();  // it keeps nothing, as the default pool
    }
    pools[count++] = {id, pool};
    return pool;
}

__global__ void bounded_wait_selftest_kernel(unsigned long long limit_ns, int *err, int *waited)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    ptx::mbar_init(&bar, 2);
    ptx::mbar_init_fence();
    ptx::mbar_arrive(&bar);  // one of the two arrivals the phase needs
    const bool done = ptx::mbar_wait_bounded(&bar, 0, limit_ns);
    *waited = 1;
    if (!done) set_error(err, DEV_TIMEOUT);
}

}  // namespace

cudaError_t malloc_async(void **p, size_t bytes, cudaStream_t st)
{
    int n = g_fail_allocs.load();
    while (n > 0) {
        if (g_fail_allocs.compare_exchange_weak(n, n - 1)) {
            *p = nullptr;
            return cudaErrorMemoryAllocation;
        }
    }
    const cudaMemPool_t pool = context_pool();
    if (!pool) return cudaMallocAsync(p, bytes, st);
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    if (e == cudaErrorMemoryAllocation) {  // what the pool keeps may be in the way
        cudaGetLastError();
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    }
    return e;
}

}  // namespace dcd

using namespace dcd;

extern "C" dcd_status dcd_inject_alloc_failures(int32_t count)
{
    if (count < 0) return DCD_EINVAL;
    g_fail_allocs.store(count);
    return DCD_OK;
}

extern "C" dcd_status dcd_selftest_bounded_wait(int64_t limit_ns, void *stream)
{
    if (limit_ns < 1000 || limit_ns > 1000000000) return DCD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int *d = nullptr;
    cudaError_t e = malloc_async((void **)&d, 2 * sizeof(int), st);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? DCD_ENOMEM : DCD_ECUDA;
    int h[2] = {0, 0};
    e = cudaMemsetAsync(d, 0, 2 * sizeof(int), st);
    if (e == cudaSuccess) {
        bounded_wait_selftest_kernel<<<1, 32, 0, st>>>((unsigned long long)limit_ns, d, d + 1);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(d, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return DCD_ECUDA;
    if (!h[1]) return DCD_EINTERNAL;  // the kernel did not reach its wait
    return h[0] == DEV_TIMEOUT ? DCD_ETIMEOUT : h[0] ? DCD_EINTERNAL : DCD_OK;
}
