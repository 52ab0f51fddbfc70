// Error reporting, device memory and copy helpers shared by the liblds sources.
#include <cstdarg>
#include <mutex>

#include "common.cuh"

namespace lds {

namespace {
thread_local std::string t_last_error;
}

void set_error(const char* fmt, ...) {
    char buf[1024];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    t_last_error = buf;
}

const char* last_error() { return t_last_error.c_str(); }

int g_fail_alloc_countdown = 0;
std::atomic<long long> g_launches{0};

// Device memory comes from a pool of this library's own, one per device.  The default
// pool hands what a call frees back to the driver at the next synchronisation, and a
// query synchronises hundreds of times: mapping its memory again took 4 of the 16 ms of
// ingest and core numbers of an R-MAT scale-20 graph and 35 of the 300 ms of an R-MAT
// scale-18 triangle query (GB300).  The pool keeps at most 1/16 of the device's memory
// while a handle is alive and 1/32 once none is, and gives everything unused back when
// an allocation fails.  Allocation and release are stream-ordered as before, so
// threads and streams share it as they shared the default pool.
namespace {
constexpr int kMaxDevices = 64;
struct DevPool {
    std::once_flag once;
    cudaMemPool_t pool = nullptr;
    size_t total = 0;
};
DevPool g_pools[kMaxDevices];
std::atomic<int64_t> g_handles{0};

// the current device's pool, or null (the default pool then serves)
DevPool* dev_pool() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return nullptr;
    }
    DevPool& d = g_pools[dev];
    std::call_once(d.once, [&] {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        size_t free_b = 0, total = 0;
        cudaMemPool_t p = nullptr;
        if (cudaMemGetInfo(&free_b, &total) != cudaSuccess || cudaMemPoolCreate(&p, &props) != cudaSuccess) {
            cudaGetLastError();
            return;
        }
        uint64_t keep = total / 16;
        if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaGetLastError();
            cudaMemPoolDestroy(p);
            return;
        }
        d.total = total;
        d.pool = p;
    });
    return d.pool ? &d : nullptr;
}
}  // namespace

void handle_created() { g_handles.fetch_add(1, std::memory_order_relaxed); }

void handle_freed() {
    if (g_handles.fetch_sub(1, std::memory_order_relaxed) == 1)
        if (DevPool* d = dev_pool())
            if (cudaMemPoolTrimTo(d->pool, d->total / 32) != cudaSuccess) cudaGetLastError();
}

void* dev_alloc(size_t bytes, cudaStream_t s) {
    if (g_fail_alloc_countdown > 0) {
        if (--g_fail_alloc_countdown == 0) {
            set_error("device allocation of %zu bytes failed (injected)", bytes);
            throw Error{LDS_ENOMEM};
        }
    }
    void* p = nullptr;
    DevPool* d = dev_pool();
    cudaError_t e = d ? cudaMallocFromPoolAsync(&p, bytes, d->pool, s) : cudaMallocAsync(&p, bytes, s);
    if (e == cudaErrorMemoryAllocation && d) {
        // frees that are still pending on this stream, and whatever the pool keeps unused
        cudaGetLastError();
        cudaStreamSynchronize(s);
        cudaMemPoolTrimTo(d->pool, 0);
        e = cudaMallocFromPoolAsync(&p, bytes, d->pool, s);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("device allocation of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
        throw Error{e == cudaErrorMemoryAllocation ? LDS_ENOMEM : LDS_ECUDA};
    }
    return p;
}

void dev_free(void* p, cudaStream_t s) {
    if (p) cudaFreeAsync(p, s);
}

int num_sms() {
    static int sms = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        cudaGetDevice(&dev);
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 132;
        sms = v;
    });
    return sms;
}

void copy_out(void* dst, lds_mem where, const void* src_dev, size_t bytes, cudaStream_t s) {
    if (!bytes || !dst) return;
    LDS_CUDA(cudaMemcpyAsync(dst, src_dev, bytes,
                             where == LDS_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, s));
}

void copy_in(void* dst_dev, const void* src, lds_mem where, size_t bytes, cudaStream_t s) {
    if (!bytes) return;
    LDS_CUDA(cudaMemcpyAsync(dst_dev, src, bytes,
                             where == LDS_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, s));
}

}  // namespace lds

extern "C" {

const char* lds_version(void) { return "liblds 0.1 (sm_103a)"; }

const char* lds_last_error(void) { return lds::last_error(); }

int32_t lds_device_count(void) {
    int c = 0;
    if (cudaGetDeviceCount(&c) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return c;
}

int64_t lds_launch_count(void) { return (int64_t)lds::g_launches.load(); }

void lds_debug_fail_alloc_after(int32_t k) { lds::g_fail_alloc_countdown = k > 0 ? k : 0; }

}  // extern "C"
