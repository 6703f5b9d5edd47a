// Lock-step trace kernels over the two-level node records (wide.cuh), one
// scene: one ray per thread, or persistent warps.
#include "wide.cuh"

namespace vsr {

namespace {

template <int Q, class H>
__global__ void __launch_bounds__(256, 4) k_trace_wide(DevScene sc, IsectParams ip,
                                                    const float4* __restrict__ rays, RayMap map,
                                                    float4* __restrict__ hits) {
    extern __shared__ float4 s_lane[];
    const unsigned long long g = slot_of_thread(map);
    const unsigned long long i = g < map.threads ? ray_of_thread(g, map) : map.n;
    const LaneStore m(s_lane);
    WideLane<Q, H> w;
    bool busy = i < map.n;
    if (busy && !w.start(sc, ip, __ldg(rays + 2 * i), __ldg(rays + 2 * i + 1), m)) {
        hits[i] = m.hit();
        busy = false;
    }
    while (__any_sync(kFullMask, busy)) {
        if (wide_step(sc, ip, w, m, busy)) {
            hits[i] = m.hit();
            busy = false;
        }
    }
}

template <int Q, class H>
__global__ void __launch_bounds__(256, 4) k_trace_wide_persistent(
    DevScene sc, IsectParams ip, const float4* __restrict__ rays, RayMap map,
    float4* __restrict__ hits, unsigned long long* __restrict__ work, uint32_t refill,
    Watchdog wd) {
    extern __shared__ float4 s_lane[];
    const LaneStore m(s_lane);
    WideLane<Q, H> w;
    persistent_rays<true>(
        map, work, refill, wd, sc.err,
        [&](unsigned long long ri) {
            m.index() = ri;
            return w.start(sc, ip, __ldg(rays + 2 * ri), __ldg(rays + 2 * ri + 1), m);
        },
        [&](bool busy) { return wide_step(sc, ip, w, m, busy); },
        [&](unsigned long long) { hits[m.index()] = m.hit(); }, [&]() { w.fail(m); });
}

template <class Kern>
cudaError_t allow_smem(Kern kernel, size_t smem) {
    if (smem <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <int Q, class H>
cudaError_t wide_one(const LaunchArgs& a) {
    const size_t smem = wide_smem(a.block, a.sc.stack_depth);
    if (!a.persistent) {
        auto k = k_trace_wide<Q, H>;
        cudaError_t e = allow_smem(k, smem);
        if (e != cudaSuccess) return e;
        RayMap map = a.map;
        const unsigned long long grid = (spread_rays(map, kSpreadWarpsLarge) + a.block - 1) / a.block;
        k<<<(unsigned)grid, a.block, smem, a.stream>>>(a.sc, a.ip, a.rays, map, a.hits);
        return cudaGetLastError();
    }
    auto k = k_trace_wide_persistent<Q, H>;
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    const int grid = persistent_grid(a, reinterpret_cast<const void*>(k), smem);
    if (grid <= 0) return cudaErrorInvalidConfiguration;
    return with_ray_counter(a.work, a.stream, [&](unsigned long long* work) {
        k<<<grid, a.block, smem, a.stream>>>(a.sc, a.ip, a.rays, a.map, a.hits, work, a.refill,
                                             a.wd);
        return cudaGetLastError();
    });
}

template <int Q>
cudaError_t wide_kind(const LaunchArgs& a, int kind) {
    switch (kind) {
        case 0:
        case 1: return wide_one<Q, IsectDefault>(a);
        case 2: return wide_one<Q, IsectAlphaTex>(a);
        case 3: return wide_one<Q, IsectProcAlpha>(a);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Lock step walks the records on trees with long descents (records_limit), for
// rays in buffer order; on other trees, whose nodes stay in L1, and on pixel tiles
// a record costs more instructions than it saves round trips.  Persistent, L2
// flushed, alpha texture, us records / binary nodes:
//   500,000 diffuse rays, closest and any hit: quads 1,000 141/131 129/129, 5,000
//   301/283 272/267, 50,000 391/394 365/380, 500,000 579/593 546/582; occlusion
//   rays on 50,000 134/144 127/142; forest 200,002 1,622/1,421 463/449
//   400,000 camera rays on tiles: quads 50,000 169/166 164/156, 400,000 264/251
//   249/241; forest 1,000,002 at 1080p 866/684 551/474
bool walks_records(const LaunchArgs& a, int kind) {
    return a.sc.wide && a.records_up_to > 0 && a.map.width == 0 && !a.binary_nodes &&
           kind >= 0 && kind <= 3 && a.lockstep && a.stack_regs == 0;
}

cudaError_t launch_wide(const LaunchArgs& a, int kind) {
    return a.query == kClosest ? wide_kind<kClosest>(a, kind) : wide_kind<kAny>(a, kind);
}

}  // namespace vsr
