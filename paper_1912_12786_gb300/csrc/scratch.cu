// Scratch from a stream-ordered pool of the library's own, one per context.
//
// The device's default pool gives its memory back to the system at every
// synchronisation, so a program that waits for each frame pays for mapping the
// scratch again on each call (a persistent trace's 8-byte counter: 200 us).
// This pool keeps up to kKeepBytes across synchronisations.  It exists while
// scenes do: the last scene's destruction in a context returns what it holds.
// Allocation and freeing are ordered on the caller's stream, as with the
// default pool, so calls on several streams and threads do not share memory
// that is in use.
#include <mutex>
#include <vector>

#include "vsr_internal.h"

namespace vsr {

namespace {

constexpr unsigned long long kKeepBytes = 512ull << 20;

// A context is on one device, and its id is not used again: the entry of one
// that has ended, with scenes alive or not, is never looked at again.
struct Pool {
    unsigned long long ctx;
    cudaMemPool_t pool;  // null: none could be made, the default pool serves
    unsigned long long scenes;
};
std::mutex g_mutex;
std::vector<Pool> g_pools;

Pool* pool_of(unsigned long long ctx) {
    for (Pool& p : g_pools)
        if (p.ctx == ctx) return &p;
    return nullptr;
}

cudaMemPool_t make_pool() {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    if (cudaGetDevice(&props.location.id) != cudaSuccess) return nullptr;
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
    return made;
}

}  // namespace

cudaError_t scratch_alloc(void** ptr, size_t bytes, cudaStream_t stream) {
    cudaMemPool_t pool = nullptr;
    unsigned long long ctx = 0;
    if (current_context_id(&ctx)) {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (const Pool* p = pool_of(ctx)) pool = p->pool;
    }
    return pool ? cudaMallocFromPoolAsync(ptr, bytes, pool, stream)
                : cudaMallocAsync(ptr, bytes, stream);
}

unsigned long long scratch_scene_created() {
    unsigned long long ctx = 0;
    if (!current_context_id(&ctx)) return 0;
    std::lock_guard<std::mutex> lock(g_mutex);
    Pool* p = pool_of(ctx);
    if (!p) {
        g_pools.push_back(Pool{ctx, nullptr, 0});
        p = &g_pools.back();
    }
    if (!p->pool) p->pool = make_pool();
    ++p->scenes;
    return ctx + 1;
}

void scratch_scene_destroyed(unsigned long long noted) {
    unsigned long long ctx = 0;
    if (!noted || !current_context_id(&ctx) || ctx + 1 != noted) return;
    std::lock_guard<std::mutex> lock(g_mutex);
    Pool* p = pool_of(ctx);
    if (p && p->scenes && --p->scenes == 0 && p->pool) cudaMemPoolTrimTo(p->pool, 0);
}

}  // namespace vsr
