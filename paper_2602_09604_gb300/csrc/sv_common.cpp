// Error reporting and small shared helpers.
#include <algorithm>
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <future>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>

#include "sv_internal.h"

namespace svg {

namespace {
struct DevBuf {
    void *p;
    size_t bytes;
};
std::mutex g_buf_mu;
std::vector<DevBuf> g_buf_cache[64];
constexpr size_t kBufCacheCount = 8;
constexpr size_t kBufCacheBytes = size_t(256) << 20;
SharedBuffer *g_dropped = nullptr;   // shared buffers without an owner, not yet back in the cache

// A graph that held a buffer has been destroyed, or never took it over: called by the driver on a
// thread of its own, where no CUDA call is allowed.
void release_from_graph(void *b) { shared_buffer_release(static_cast<SharedBuffer *>(b)); }
}  // namespace

int shared_buffer_get(int device, size_t bytes, SharedBuffer **out)
{
    *out = nullptr;
    SharedBuffer *b = new (std::nothrow) SharedBuffer;
    if (!b) { set_error("out of host memory"); return SV_ENOMEM; }
    b->device = device;
    const int rc = dev_buffer_get(device, bytes, &b->p, &b->bytes);
    if (rc != SV_OK) {
        delete b;
        return rc;
    }
    *out = b;
    return SV_OK;
}

void shared_buffer_release(SharedBuffer *b)
{
    if (!b || b->owners.fetch_sub(1) != 1) return;
    std::lock_guard<std::mutex> lk(g_buf_mu);
    b->next = g_dropped;
    g_dropped = b;
}

int shared_buffer_retain_in_capture(SharedBuffer *b, cudaStream_t stream)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    SV_CUDA_TRY(cudaStreamGetCaptureInfo(stream, &st, nullptr, &graph, nullptr, nullptr, nullptr));
    if (st != cudaStreamCaptureStatusActive || !graph) { set_error("stream is not being captured"); return SV_ESTATE; }
    cudaUserObject_t obj = nullptr;
    SV_CUDA_TRY(cudaUserObjectCreate(&obj, b, release_from_graph, 1, cudaUserObjectNoDestructorSync));
    b->owners.fetch_add(1);   // the object's; its end releases it
    const cudaError_t e = cudaGraphRetainUserObject(graph, obj, 1, cudaGraphUserObjectMove);
    if (e != cudaSuccess) {
        cudaUserObjectRelease(obj, 1);
        set_error("keeping a buffer with a captured graph: %s", cudaGetErrorString(e));
        return SV_ECUDA;
    }
    return SV_OK;
}

int dev_buffer_get(int device, size_t bytes, void **out, size_t *got_bytes)
{
    *out = nullptr;
    *got_bytes = 0;
    shared_buffers_collect(false);
    if (device >= 0 && device < 64) {
        std::lock_guard<std::mutex> lk(g_buf_mu);
        std::vector<DevBuf> &c = g_buf_cache[device];
        size_t best = c.size();
        for (size_t i = 0; i < c.size(); ++i)
            if (c[i].bytes >= bytes && c[i].bytes <= 4 * bytes && (best == c.size() || c[i].bytes < c[best].bytes)) best = i;
        if (best < c.size()) {
            *out = c[best].p;
            *got_bytes = c[best].bytes;
            c.erase(c.begin() + (long)best);
            return SV_OK;
        }
    }
    SV_CUDA_TRY(cudaMalloc(out, bytes));
    *got_bytes = bytes;
    return SV_OK;
}

namespace {
// whether the cache took the buffer
bool cache_buffer(int device, void *p, size_t bytes)
{
    if (device < 0 || device >= 64) return false;
    std::lock_guard<std::mutex> lk(g_buf_mu);
    std::vector<DevBuf> &c = g_buf_cache[device];
    size_t held = 0;
    for (const DevBuf &b : c) held += b.bytes;
    if (c.size() >= kBufCacheCount || held + bytes > kBufCacheBytes) return false;
    c.push_back(DevBuf{p, bytes});
    return true;
}
}  // namespace

void dev_buffer_put(int device, void *p, size_t bytes)
{
    if (!p || cache_buffer(device, p, bytes)) return;
    int cur = -1;
    cudaGetDevice(&cur);
    if (device >= 0 && cur != device) cudaSetDevice(device);
    cudaFree(p);
    if (device >= 0 && cur >= 0 && cur != device) cudaSetDevice(cur);
}

void shared_buffers_collect(bool may_free)
{
    SharedBuffer *b = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_buf_mu);
        std::swap(b, g_dropped);
    }
    while (b) {
        SharedBuffer *next = b->next;
        if (may_free) dev_buffer_put(b->device, b->p, b->bytes);
        if (may_free || cache_buffer(b->device, b->p, b->bytes)) {
            delete b;
        } else {
            std::lock_guard<std::mutex> lk(g_buf_mu);
            b->next = g_dropped;
            g_dropped = b;
        }
        b = next;
    }
}

int upload_now(int device, void *dst, const void *pinned, size_t bytes)
{
    static std::mutex mu;
    static cudaStream_t streams[64] = {};
    if (device < 0 || device >= 64) { set_error("upload: device %d out of range", device); return SV_EINVAL; }
    std::lock_guard<std::mutex> lk(mu);
    cudaStream_t &s = streams[device];
    if (!s) SV_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    SV_CUDA_TRY(cudaMemcpyAsync(dst, pinned, bytes, cudaMemcpyHostToDevice, s));
    SV_CUDA_TRY(cudaStreamSynchronize(s));
    return SV_OK;
}

namespace {
std::mutex g_pin_mu;
unsigned char *g_pin = nullptr;
size_t g_pin_bytes = 0;
}  // namespace

int pinned_staging(size_t bytes, unsigned char **out, std::unique_lock<std::mutex> &lock)
{
    lock = std::unique_lock<std::mutex>(g_pin_mu);
    if (g_pin_bytes < bytes) {
        if (g_pin) cudaFreeHost(g_pin);
        g_pin = nullptr;
        g_pin_bytes = 0;
        const size_t want = std::max(bytes, size_t(4) << 20);
        const cudaError_t e = cudaMallocHost(reinterpret_cast<void **>(&g_pin), want);
        if (e != cudaSuccess) {
            g_pin = nullptr;
            set_error("pinned staging buffer: %s", cudaGetErrorString(e));
            return SV_ECUDA;
        }
        g_pin_bytes = want;
    }
    *out = g_pin;
    return SV_OK;
}

void host_parallel_for(size_t n, size_t threads, const std::function<void(size_t)> &fn)
{
    std::atomic<size_t> next{0};
    auto work = [&]() {
        for (size_t i = next++; i < n; i = next++) fn(i);
    };
    const size_t hw = std::max(1u, std::thread::hardware_concurrency());
    const size_t nt = std::min(std::min(threads, n), hw);
    std::vector<std::future<void>> jobs;
    try {
        for (size_t t = 1; t < nt; ++t) jobs.push_back(std::async(std::launch::async, work));
    } catch (const std::system_error &) {   // no more threads: the ones started and this one finish
    }
    work();
    for (auto &j : jobs) j.get();   // rethrows a worker's exception (e.g. std::bad_alloc)
}

static thread_local char g_err[512] = "";

void set_error(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    std::vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

void clear_error() { g_err[0] = '\0'; }

int device_sm_count(int device)
{
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
    return v;
}

}  // namespace svg

extern "C" const char *sv_last_error(void) { return svg::g_err; }

extern "C" const char *sv_version(void) { return "svgb300 0.1 (sm_103a)"; }
