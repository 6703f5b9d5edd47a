// BVH refit after a vertex update: triangle layout and node boxes in one
// launch.
//
// One thread per leaf writes its triangles and its box, then climbs: at each
// pair the first of the two threads to arrive stops and the second takes the
// union of both boxes to the parent, so every box is written once both children
// are there, and no thread waits.  A box is a union of its children's, which
// does not depend on the order, so the result is that of a launch per level.
// That form spent its time on launches (20 levels for 65,000 triangles, 3 to 8
// us each, most of them with one block); the climb costs a fence and an atomic
// per level, about 0.7 us.
#include "wide_build.cuh"

namespace vsr {

namespace {

constexpr uint32_t kNoParent = 0xFFFFFFFFu;

__global__ void __launch_bounds__(256) k_parents(const float4* __restrict__ nodes,
                                                 uint32_t num_nodes,
                                                 uint32_t* __restrict__ parent,
                                                 uint32_t* __restrict__ arrived) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= num_nodes) return;
    if (i < num_nodes / 2u) arrived[i] = 0u;
    if (i == 0u) parent[0] = kNoParent;
    if (i == 1u) return;  // padding beside the root
    const uint32_t ref = __float_as_uint(nodes[2ull * i].w);
    if (!(ref & kLeafBit)) parent[ref >> 2] = i;
}

__global__ void __launch_bounds__(256) k_refit(RefitArgs a) {
    uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= a.num_nodes || id == 1u) return;
    const uint32_t ref = __float_as_uint(a.nodes[2ull * id].w);
    if (!(ref & kLeafBit)) return;
    // the leaf's triangles (as k_build_tris) and the bounds of their vertices
    float lo[3] = {__int_as_float(0x7f800000), __int_as_float(0x7f800000),
                   __int_as_float(0x7f800000)};
    float hi[3] = {-lo[0], -lo[1], -lo[2]};
    const uint64_t first = (ref >> 3) & 0x0FFFFFFFu;
    for (uint64_t s = first; s <= first + (ref & 7u); ++s) {
        const uint32_t p = a.order[s];
        float v[3][3];
        for (int k = 0; k < 3; ++k) {
            const float* q = a.verts + 3ull * a.idx[3ull * p + k];
            for (int c = 0; c < 3; ++c) {
                v[k][c] = q[c];
                lo[c] = fminf(lo[c], v[k][c]);
                hi[c] = fmaxf(hi[c], v[k][c]);
            }
        }
        float4* t = a.tris + 3ull * s;
        t[0] = make_float4(v[0][0], v[0][1], v[0][2], __uint_as_float(p));
        t[1] = make_float4(__fsub_rn(v[1][0], v[0][0]), __fsub_rn(v[1][1], v[0][1]),
                           __fsub_rn(v[1][2], v[0][2]), __uint_as_float(id));
        t[2] = make_float4(__fsub_rn(v[2][0], v[0][0]), __fsub_rn(v[2][1], v[0][1]),
                           __fsub_rn(v[2][2], v[0][2]), 0.0f);
    }
    float w = __uint_as_float(ref);
    for (;;) {
        a.nodes[2ull * id] = make_float4(lo[0], lo[1], lo[2], w);
        a.nodes[2ull * id + 1] = make_float4(hi[0], hi[1], hi[2], 0.0f);
        // the octant-specialised box test needs finite boxes with lo <= hi
        bool ordered = true;
        for (int c = 0; c < 3; ++c)
            ordered = ordered && isfinite(lo[c]) && isfinite(hi[c]) && lo[c] <= hi[c];
        if (!ordered) atomicOr(a.unordered, 1u);
        const uint32_t pair = id >> 1;
        const uint32_t up = a.parent[pair];
        if (up == kNoParent) break;
        // each pair is counted twice per refit, so the counts need no reset
        __threadfence();
        if ((atomicAdd(a.arrived + pair, 1u) & 1u) == 0u) return;
        __threadfence();
        // both children, past this SM's L1 (the other may have been written
        // elsewhere)
        lo[0] = lo[1] = lo[2] = __int_as_float(0x7f800000);
        hi[0] = hi[1] = hi[2] = -lo[0];
        for (uint64_t c = 2ull * pair; c <= 2ull * pair + 1; ++c) {
            const float4 ca = __ldcg(a.nodes + 2 * c), cb = __ldcg(a.nodes + 2 * c + 1);
            lo[0] = fminf(lo[0], ca.x);
            lo[1] = fminf(lo[1], ca.y);
            lo[2] = fminf(lo[2], ca.z);
            hi[0] = fmaxf(hi[0], cb.x);
            hi[1] = fmaxf(hi[1], cb.y);
            hi[2] = fmaxf(hi[2], cb.z);
        }
        id = up;
        w = __ldcg(&a.nodes[2ull * id].w);
    }
    // the root: every box is written, and every report in *unordered
    const uint32_t bad = atomicOr(a.unordered, 0u);
    const float4 ra = make_float4(lo[0], lo[1], lo[2], 0.0f),
                 rb = make_float4(hi[0], hi[1], hi[2], __uint_as_float(bad));
    if (a.wide)
        write_wide_header(a.nodes, make_float4(lo[0], lo[1], lo[2], w), rb, !bad, a.wide);
    a.state[0] = ra;
    a.state[1] = rb;
    a.user->root_a = ra;
    a.user->root_b = make_float4(hi[0], hi[1], hi[2], 0.0f);
    a.user->boxes_ordered = bad ? 0u : 1u;
}

}  // namespace

cudaError_t launch_parents(const float4* nodes, uint32_t num_nodes, uint32_t* parent,
                           uint32_t* arrived, cudaStream_t stream) {
    k_parents<<<(num_nodes + 255) / 256, 256, 0, stream>>>(nodes, num_nodes, parent, arrived);
    return cudaGetLastError();
}

cudaError_t launch_refit(const RefitArgs& a, cudaStream_t stream) {
    k_refit<<<(a.num_nodes + 255) / 256, 256, 0, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace vsr
