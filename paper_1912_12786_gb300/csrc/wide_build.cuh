// What the kernels that build the two-level node records share (wide.cuh has
// the format).
#pragma once

#include "wide.cuh"

namespace vsr {

// Reference of the inner node with binary reference `ref`.
__device__ __forceinline__ uint32_t record_ref(const float4* nodes, uint32_t ref) {
    const uint64_t k = ref >> 2;
    const uint32_t a = __float_as_uint(nodes[4 * k].w), b = __float_as_uint(nodes[4 * k + 2].w);
    const uint32_t xa = (a & kLeafBit) ? 3u : a & 3u, xb = (b & kLeafBit) ? 3u : b & 3u;
    return kLeft | kRight | (uint32_t)(k << 6) | xb << 4 | xa << 2 | (ref & 3u);
}

// Cell size on one axis: the least power of two with which 65535 cells cover
// [lo, hi], at least 2^-40 (WideLane::start's limit on the inverse direction
// keeps 2^-40 times it normal).
__device__ __forceinline__ float cell_of(float lo, float hi) {
    const float need = __fdiv_ru(__fsub_ru(hi, lo), 65535.0f);
    const float c = ldexpf(1.0f, ilogbf(fmaxf(need, 0x1p-40f)));
    return c >= need ? c : 2.0f * c;
}

// The header for a root with box (ra, rb) and its reference in ra.w; usable:
// the tree's boxes are finite and ordered.  Cells go up to 2^20 (S * 2^23 then
// stays finite).
__device__ __forceinline__ void write_wide_header(const float4* nodes, float4 ra, float4 rb,
                                                  bool usable, uint32_t* wide) {
    constexpr float kExtent = 0x1p35f;
    const bool fits = usable && rb.x - ra.x <= kExtent && rb.y - ra.y <= kExtent &&
                      rb.z - ra.z <= kExtent;
    const uint32_t root = __float_as_uint(ra.w);
    float4* o = reinterpret_cast<float4*>(wide);
    o[0] = make_float4(ra.x, ra.y, ra.z, __uint_as_float(fits ? 1u : 0u));
    o[1] = fits ? make_float4(cell_of(ra.x, rb.x), cell_of(ra.y, rb.y), cell_of(ra.z, rb.z),
                              __uint_as_float((root & kLeafBit) ? root : record_ref(nodes, root)))
                : make_float4(1.0f, 1.0f, 1.0f, ra.w);
}

}  // namespace vsr
