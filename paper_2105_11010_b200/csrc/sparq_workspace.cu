// Scratch memory of the entry points that run as transform + plain contraction: a memory pool of
// the library's own per device, allocated from and freed to in stream order, so that concurrent
// calls on other threads and streams get memory of their own without any bookkeeping here.  The
// pool keeps up to kKeepBytes between synchronizations (allocating from the driver costs about a
// millisecond) and gives back the rest; sparq_shutdown releases it.  A stream that is being
// captured gets none: the allocation would become nodes of the user's graph, which then cannot be
// cloned, be a child graph or be instantiated twice, and whose memory neither bound covers.
#include <mutex>

#include "sparq_common.cuh"

namespace sparq {

namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kKeepBytes = 256ull << 20;

std::mutex g_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaMemPool_t pool_of_current_device()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) return nullptr;
        unsigned long long keep = kKeepBytes;
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        g_pool[dev] = pool;
    }
    return g_pool[dev];
}

}  // namespace

bool workspace_possible(size_t bytes, cudaStream_t st)
{
    if (bytes > kWorkspaceMaxBytes) return false;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &capture) == cudaSuccess) return capture == cudaStreamCaptureStatusNone;
    cudaGetLastError();
    return false;
}

void *workspace_alloc(size_t bytes, cudaStream_t st)
{
    if (!workspace_possible(bytes, st)) return nullptr;
    cudaMemPool_t pool = pool_of_current_device();
    void *p = nullptr;
    if (!pool || cudaMallocFromPoolAsync(&p, bytes, pool, st) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return p;
}

void workspace_free(void *p, cudaStream_t st)
{
    if (p) cudaFreeAsync(p, st);
}

void release_workspace()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return;
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_pool[dev]) cudaMemPoolDestroy(g_pool[dev]);
    g_pool[dev] = nullptr;
}

}  // namespace sparq
