// Dispatch of the statically injected trace kernels (trace_static.cuh) over
// the register-stack depths, and the persistent grid size.  The kernels of
// each depth K are instantiated in trace_k<K>.cu.
#include "vsr_internal.h"

#include <atomic>

namespace vsr {

cudaError_t launch_static_k0(const LaunchArgs& a, int kind, bool stats);
cudaError_t launch_static_k1(const LaunchArgs& a, int kind, bool stats);
cudaError_t launch_static_k2(const LaunchArgs& a, int kind, bool stats);
cudaError_t launch_static_k4(const LaunchArgs& a, int kind, bool stats);
cudaError_t launch_static_k8(const LaunchArgs& a, int kind, bool stats);

bool stack_regs_supported(uint32_t k) { return k == 0 || k == 1 || k == 2 || k == 4 || k == 8; }

cudaError_t launch_static(const LaunchArgs& a, int kind, bool stats) {
    // the measurement variant keeps the stack in shared memory: the depth
    // changes neither the visiting order nor the counts
    if (stats) return launch_static_k0(a, kind, true);
    if (a.reg_cap >= 3) return launch_static_capped(a, kind, a.reg_cap);
    if (walks_records(a, kind)) return launch_wide(a, kind);
    // a shape that leaves the traversal's form open (records_limit, api.cu)
    if (!a.persistent && !a.lockstep && !a.octant && a.reg_cap == 0 && a.stack_regs == 0 &&
        kind <= 3 && a.n <= a.records_up_to) {
        LaunchArgs b = a;
        b.lockstep = 1u;
        return walks_records(b, kind) ? launch_wide(b, kind) : launch_static_k0(b, kind, false);
    }
    // The octant-dispatching kernel also runs launches that do not ask for it: on
    // pixel tiles, with few rays, which it spreads, and every closest hit (mixed
    // warps are no slower in it: 1,000,003 diffuse rays, default 985 us against
    // 1,038, alpha mask 1,396 / 1,398; camera rays in rows gain 4 to 18%).  Any hit
    // in buffer order keeps the generic kernel, where rays that point anywhere are
    // 1 to 3% faster (default 927 / 955, alpha mask 1,322 / 1,344), and so does the
    // clip box's closest hit there (518,400 diffuse rays, 100,000 quads 588 / 617 us,
    // 4,000 quads 310 / 322; the forest's 1,440,000 3,354 / 3,477).
    // reg_cap 1 asks for a kernel without a register budget, which the octant
    // kernels have: it gets the generic one, unless octant is asked for too.
    if (a.octant || (!a.persistent && !a.lockstep && a.stack_regs == 0 && a.reg_cap == 0 &&
                     ((a.query == kClosest && kind != 5) || a.map.width > 0 ||
                      spreads_rays(a.map, kSpreadWarps))))
        return launch_static_octant(a, kind);
    switch (a.stack_regs) {
        case 0: return launch_static_k0(a, kind, false);
        case 1: return launch_static_k1(a, kind, false);
        case 2: return launch_static_k2(a, kind, false);
        case 4: return launch_static_k4(a, kind, false);
        case 8: return launch_static_k8(a, kind, false);
        default: return cudaErrorInvalidValue;
    }
}

int sm_count() {
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < kDevices && (sms = known[dev].load(std::memory_order_relaxed)) > 0)
        return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < kDevices) known[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

int persistent_grid(uint32_t block, uint32_t blocks_per_sm, const void* kernel, size_t smem) {
    int per_sm = 0;
    const int sms = sm_count();
    if (sms <= 0) return 0;
    if (blocks_per_sm) {
        per_sm = (int)blocks_per_sm;
    } else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, (int)block, smem) !=
               cudaSuccess) {
        return 0;
    }
    if (per_sm < 1) per_sm = 1;
    return sms * per_sm;
}

}  // namespace vsr
