// Error reporting, device memory and copy helpers shared by the liblds sources.
#include <cuda.h>

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
// while a handle made on the device is alive and 1/32 once none is, and nothing after
// lds_release_memory.  When an allocation fails, the frees queued on its own stream are
// waited for, the pool's unused memory is given back, and it is tried once more.
// Allocation and release are stream-ordered as before, so threads and streams share it
// as they shared the default pool.
//
// A pool dies with its context (cudaDeviceReset), so it is known by the context's id,
// which is never used again, and a context that has none yet gets one of its own.  The
// look-up is made once per entry point and thread, at its first allocation (at every
// allocation it cost about 1 % of a query of 6 ms).
namespace {
constexpr int kMaxDevices = 64;
constexpr int kMaxContexts = 16;         // per device, over the process's life; then the default pool serves
struct DevPool {
    unsigned long long context = 0;
    cudaMemPool_t pool = nullptr;        // null: could not be made
    size_t total = 0;
};
struct DevPools {
    std::mutex mu;
    std::atomic<int> count{0};           // pools[0 .. count) are whole
    DevPool pools[kMaxContexts];
    std::atomic<int64_t> handles{0};
};
DevPools g_pools[kMaxDevices];

// the id of the current context, made current first if there is none; 0 on failure
unsigned long long context_id() {
    using GetId = CUresult (*)(CUcontext, unsigned long long*);
    using GetState = CUresult (*)(CUdevice, unsigned int*, int*);
    static GetId get_id = nullptr;
    static GetState get_state = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *f = nullptr, *h = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPointByVersion("cuDevicePrimaryCtxGetState", &h, 7000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess) {
            get_state = reinterpret_cast<GetState>(h);
            get_id = reinterpret_cast<GetId>(f);
        } else {
            cudaGetLastError();
        }
    });
    if (!get_id) return 0;
    int dev = 0, active = 0;
    unsigned int flags = 0;
    unsigned long long id = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    // a reset context is begun again by the runtime's next call, which this makes
    if ((get_state(dev, &flags, &active) != CUDA_SUCCESS || !active || get_id(nullptr, &id) != CUDA_SUCCESS) &&
        (cudaFree(nullptr) != cudaSuccess || get_id(nullptr, &id) != CUDA_SUCCESS)) {
        cudaGetLastError();
        return 0;
    }
    return id;
}

DevPools* dev_pools() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return nullptr;
    }
    return g_pools + dev;
}

// the current context's pool, or null (the default pool then serves)
DevPool* dev_pool(bool make) {
    DevPools* d = dev_pools();
    const unsigned long long id = d ? context_id() : 0;
    if (!id) return nullptr;
    auto find = [&]() -> DevPool* {
        for (int i = 0, n = d->count.load(std::memory_order_acquire); i < n; ++i)
            if (d->pools[i].context == id) return d->pools + i;
        return nullptr;
    };
    DevPool* e = find();
    if (!e && make) {
        std::lock_guard<std::mutex> lk(d->mu);
        e = find();
        const int n = d->count.load(std::memory_order_relaxed);
        if (!e && n < kMaxContexts) {
            e = d->pools + n;
            e->context = id;
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = (int)(d - g_pools);
            size_t free_b = 0;
            if (cudaMemGetInfo(&free_b, &e->total) == cudaSuccess && cudaMemPoolCreate(&e->pool, &props) == cudaSuccess) {
                uint64_t keep = e->total / 16;
                if (cudaMemPoolSetAttribute(e->pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
                    cudaMemPoolDestroy(e->pool);
                    e->pool = nullptr;
                }
            } else {
                e->pool = nullptr;
            }
            if (!e->pool) cudaGetLastError();
            d->count.store(n + 1, std::memory_order_release);
        }
    }
    return e && e->pool ? e : nullptr;
}

// runs f with device dev current
template <class F>
void on_device(int dev, F&& f) {
    int old = 0;
    if (cudaGetDevice(&old) != cudaSuccess || (old != dev && cudaSetDevice(dev) != cudaSuccess)) {
        cudaGetLastError();
        return;
    }
    f();
    if (old != dev) cudaSetDevice(old);
}
}  // namespace

int handle_created() {
    DevPools* d = dev_pools();
    if (!d) return -1;
    d->handles.fetch_add(1, std::memory_order_relaxed);
    return (int)(d - g_pools);
}

void handle_freed(int dev) {
    if (dev < 0 || g_pools[dev].handles.fetch_sub(1, std::memory_order_relaxed) != 1) return;
    on_device(dev, [] {
        if (DevPool* e = dev_pool(false))
            if (cudaMemPoolTrimTo(e->pool, e->total / 32) != cudaSuccess) cudaGetLastError();
    });
}

static thread_local bool t_pool_known = false;
static thread_local DevPool* t_pool = nullptr;

void pool_forget() { t_pool_known = false; }

void* dev_alloc(size_t bytes, cudaStream_t s) {
    if (g_fail_alloc_countdown > 0) {
        if (--g_fail_alloc_countdown == 0) {
            set_error("device allocation of %zu bytes failed (injected)", bytes);
            throw Error{LDS_ENOMEM};
        }
    }
    void* p = nullptr;
    if (!t_pool_known) {
        t_pool = dev_pool(true);
        t_pool_known = true;
    }
    DevPool* d = t_pool;
    cudaError_t e = d ? cudaMallocFromPoolAsync(&p, bytes, d->pool, s) : cudaMallocAsync(&p, bytes, s);
    if (e == cudaErrorMemoryAllocation && d) {
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

lds_status lds_release_memory(void) {
    return lds::guard([] {
        for (int dev = 0; dev < lds::kMaxDevices; ++dev) {
            if (lds::g_pools[dev].count.load() == 0) continue;
            lds::on_device(dev, [] {
                if (lds::DevPool* e = lds::dev_pool(false)) {
                    LDS_CUDA(cudaDeviceSynchronize());
                    LDS_CUDA(cudaMemPoolTrimTo(e->pool, 0));
                }
            });
        }
    });
}

lds_status lds_memory_info(int64_t* held, int64_t* in_use, int64_t* peak) {
    return lds::guard([&] {
        uint64_t h = 0, u = 0, p = 0, zero = 0;
        LDS_REQUIRE(lds_device_count() > 0, LDS_ECUDA, "lds_memory_info: no CUDA device");
        if (lds::DevPool* e = lds::dev_pool(false)) {
            LDS_CUDA(cudaMemPoolGetAttribute(e->pool, cudaMemPoolAttrReservedMemCurrent, &h));
            LDS_CUDA(cudaMemPoolGetAttribute(e->pool, cudaMemPoolAttrUsedMemCurrent, &u));
            LDS_CUDA(cudaMemPoolGetAttribute(e->pool, cudaMemPoolAttrUsedMemHigh, &p));
            if (peak) LDS_CUDA(cudaMemPoolSetAttribute(e->pool, cudaMemPoolAttrUsedMemHigh, &zero));
        }
        if (held) *held = (int64_t)h;
        if (in_use) *in_use = (int64_t)u;
        if (peak) *peak = (int64_t)p;
    });
}

void lds_debug_fail_alloc_after(int32_t k) { lds::g_fail_alloc_countdown = k > 0 ? k : 0; }

}  // extern "C"
