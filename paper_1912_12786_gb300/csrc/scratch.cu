// Scratch from a stream-ordered pool of the library's own, one per device.
//
// The device's default pool gives its memory back to the system at every
// synchronisation, so a program that waits for each frame pays for mapping the
// scratch again on each call (a persistent trace's 8-byte counter: 200 us).
// This pool keeps up to kKeepBytes across synchronisations.  It exists while
// scenes do: the last scene's destruction on a device returns what it holds.
// Allocation and freeing are ordered on the caller's stream, as with the
// default pool, so calls on several streams and threads do not share memory
// that is in use.
#include <mutex>

#include "vsr_internal.h"

namespace vsr {

namespace {

constexpr unsigned long long kKeepBytes = 512ull << 20;
constexpr int kDevices = 64;

struct Pool {
    cudaMemPool_t pool = nullptr;
    unsigned long long ctx = 0;  // id of the context it belongs to
    unsigned long long scenes = 0;
};
std::mutex g_mutex;
Pool g_pools[kDevices];

// The current device's pool, made on first use; null where there is none (the
// default pool serves then).  `make`: not on a stream under capture.
cudaMemPool_t current_pool(int* device, bool make) {
    unsigned long long ctx = 0;
    if (cudaGetDevice(device) != cudaSuccess || *device < 0 || *device >= kDevices ||
        !current_context_id(&ctx))
        return nullptr;
    Pool& p = g_pools[*device];
    if (p.pool && p.ctx == ctx) return p.pool;
    p.pool = nullptr;  // its context is gone, and it with it
    if (!make) return nullptr;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = *device;
    cudaMemPool_t made = nullptr;
    unsigned long long keep = kKeepBytes;
    if (cudaMemPoolCreate(&made, &props) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        cudaMemPoolDestroy(made);
        return nullptr;
    }
    p.pool = made;
    p.ctx = ctx;
    return made;
}

}  // namespace

cudaError_t scratch_alloc(void** ptr, size_t bytes, cudaStream_t stream) {
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        int device = 0;
        pool = current_pool(&device, false);
    }
    return pool ? cudaMallocFromPoolAsync(ptr, bytes, pool, stream)
                : cudaMallocAsync(ptr, bytes, stream);
}

void scratch_scene_created() {
    std::lock_guard<std::mutex> lock(g_mutex);
    int device = 0;
    current_pool(&device, true);
    if (device >= 0 && device < kDevices) ++g_pools[device].scenes;
}

void scratch_scene_destroyed() {
    std::lock_guard<std::mutex> lock(g_mutex);
    int device = 0;
    cudaMemPool_t pool = current_pool(&device, false);
    if (device < 0 || device >= kDevices || g_pools[device].scenes == 0) return;
    if (--g_pools[device].scenes == 0 && pool) cudaMemPoolTrimTo(pool, 0);
}

}  // namespace vsr
