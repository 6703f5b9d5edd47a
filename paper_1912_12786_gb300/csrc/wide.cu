// The two-level node records (wide.cuh): built from the binary nodes at load
// and after a refit.
#include "wide_build.cuh"

namespace vsr {

namespace {

// A plane's cell, rounded toward the box's outside.
// (`per`: 1 / cell, a power of two).
__device__ __forceinline__ uint32_t cell_below(float x, float origin, float per) {
    return (uint32_t)fminf(fmaxf(floorf(__fmul_rd(__fsub_rd(x, origin), per)), 0.0f), 65535.0f);
}
__device__ __forceinline__ uint32_t cell_above(float x, float origin, float per) {
    return (uint32_t)fminf(fmaxf(ceilf(__fmul_ru(__fsub_ru(x, origin), per)), 0.0f), 65535.0f);
}

// One thread per slot.  Every inner node gets a record; the traversal visits
// those an even number of levels below the root.
__global__ void __launch_bounds__(256) k_build_wide(const float4* __restrict__ nodes,
                                                    uint32_t pairs, uint32_t* __restrict__ wide) {
    const unsigned long long t = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned long long k = t >> 2;
    if (k == 0 || k >= pairs) return;  // record 0 is the header
    const float4 g = reinterpret_cast<const float4*>(wide)[0];
    const float4 c = reinterpret_cast<const float4*>(wide)[1];
    const uint32_t half = (uint32_t)(t >> 1) & 1u, s = (uint32_t)t & 1u;
    float4 lo = nodes[4 * k + 2 * half], hi = nodes[4 * k + 2 * half + 1];
    uint32_t ref = __float_as_uint(lo.w);
    bool empty = false;
    if (ref & kLeafBit) {
        empty = s;
    } else {
        const uint64_t n = 2ull * (ref >> 2) + s;
        lo = nodes[2 * n];
        hi = nodes[2 * n + 1];
        ref = __float_as_uint(lo.w);
        if (!(ref & kLeafBit)) ref = record_ref(nodes, ref);
    }
    uint32_t* o = wide + 16 * k + 2u * half + s;
    o[0] = empty ? 0xFFFFu : cell_below(lo.x, g.x, 1.0f / c.x) | cell_above(hi.x, g.x, 1.0f / c.x) << 16;
    o[4] = empty ? 0xFFFFu : cell_below(lo.y, g.y, 1.0f / c.y) | cell_above(hi.y, g.y, 1.0f / c.y) << 16;
    o[8] = empty ? 0xFFFFu : cell_below(lo.z, g.z, 1.0f / c.z) | cell_above(hi.z, g.z, 1.0f / c.z) << 16;
    o[12] = ref;
}

// The header, and each leaf's node id into the spare word of its triangles'
// second vector (the refit writes both itself).
__global__ void __launch_bounds__(256) k_wide_ids(const float4* __restrict__ nodes,
                                                  uint32_t num_nodes, float4* __restrict__ tris,
                                                  uint32_t* __restrict__ wide) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= num_nodes || i == 1u) return;
    if (i == 0u) write_wide_header(nodes, nodes[0], nodes[1], true, wide);
    const uint32_t ref = __float_as_uint(nodes[2ull * i].w);
    if (!(ref & kLeafBit)) return;
    const uint64_t first = (ref >> 3) & 0x0FFFFFFFu;
    for (uint32_t s = 0; s <= (ref & 7u); ++s)
        tris[3 * (first + s) + 1].w = __uint_as_float(i);
}

}  // namespace

bool wide_fits(uint32_t num_nodes) {
    return num_nodes > 2u && num_nodes / 2u <= (kRecField >> 6);
}

cudaError_t launch_wide_tables(const float4* nodes, uint32_t num_nodes, float4* tris,
                               uint32_t* wide, cudaStream_t stream) {
    k_wide_ids<<<(num_nodes + 255u) / 256u, 256, 0, stream>>>(nodes, num_nodes, tris, wide);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_build_wide(nodes, num_nodes, wide, stream);
}

cudaError_t launch_build_wide(const float4* nodes, uint32_t num_nodes, uint32_t* wide,
                              cudaStream_t stream) {
    const uint32_t pairs = num_nodes / 2u;
    k_build_wide<<<(unsigned)((4ull * pairs + 255u) / 256u), 256, 0, stream>>>(nodes, pairs, wide);
    return cudaGetLastError();
}

}  // namespace vsr
