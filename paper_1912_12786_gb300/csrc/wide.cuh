// Lock-step traversal over two-level node records with 16-bit boxes.
//
// A record stands for one inner node N of the binary tree and holds the boxes
// and references of its four grandchildren in 64 bytes, where the two levels
// of binary nodes take up to 192: half the dependent fetches per ray and half
// the 32-byte sectors and L1 wavefronts per box, which is what the traversal
// of incoherent rays is bound by (L1 data pipe 78% busy, 12% L1 hits, long
// scoreboard 7.8 of 14.5 cycles between issues with the binary nodes).
//
//   words 0..3, 4..7, 8..11   x, y and z planes of slots 0..3: the lower in the
//                             low, the upper in the high 16 bits, as cells of
//                             the scene's grid
//   words 12..15              references
// Slots 0 and 1 are the children of N's left child, 2 and 3 of its right; a
// child that is a leaf itself fills the first slot of its half, and the second
// gets an inverted box and the same reference.
// Reference: a leaf as in the binary nodes; an inner node as
// record << 6 | axis of its right child << 4 | of its left << 2 | its own
// (axis 3: that child is a leaf), with kLeft and kRight for the halves meant.
// A record's index is its children's pair index.
// Record 0 (no node has it) is the header: the grid's origin in words 0..2,
// its cell sizes in words 4..6, the root's reference in word 7; word 3 is 0
// where the last refit left boxes that the records cannot stand for.
//
// Boxes are rounded outward to the grid, and the plane distances are formed so
// that a slot is hit whenever the exact test of its box is.  With S = ix * cell
// (exact: cells are powers of two) and the cell number n placed in a float as
// 2^23 + n, the distance is fma(2^23 + n, S, C).  In real numbers
// (2^23 + n) S + origin ix + nox - 2^23 S is the distance of the rounded plane;
// C is that constant part rounded down for the entry plane and up for the
// exit, so, rounding being monotone, the entry distance is never above
// box_hit's for the exact plane and the exit distance never below.  Rays whose
// inverse direction could make S underflow walk the binary nodes.
//
// Results are those of traverse_body bit for bit:
//  - a box lies in its parent's and FMA rounding is monotone in the plane
//    coordinate, so along a path entry distances never fall and exit distances
//    never rise: traverse_body reaches a leaf iff the leaf's own exact box test
//    passes at the far limit at which its parent was visited;
//  - the near half's slots are tested where traverse_body tests these boxes (no
//    leaf lies between); the far half waits on the stack and is tested when
//    popped, at the far limit of that moment, as there.  So every leaf
//    traverse_body tests is tested here, in the same order;
//  - a leaf more than those must not change the result: before a candidate is
//    taken, its leaf's exact box is tested (WideLane::test).  If it is missed at
//    the ray's own limits, traverse_body never tests the leaf.  If it is hit at
//    the far limit held when the leaf was reached here, traverse_body's limit
//    was no smaller and it tests the leaf.  Between the two (the candidate lies
//    in front of its leaf's box by rounding) the ray starts over on the binary
//    nodes.
// The stack holds at most one entry per level of the binary tree, as there;
// its column has kWideSlack words more, so that the check on its height is made
// once per record.
//
// Registers: a lane keeps what every record needs (slab constants, limits,
// position).  The ray itself and the running result, needed at leaves only, are
// in shared memory beside the stack (LaneStore), which takes the kernels from
// 78-80 registers, 24 resident warps per SM, to 64 and 32 (closest hit 816 ->
// 785 us below; at 48 registers they spill and lose a quarter).  At 64 the way
// back to the binary nodes, inlined twice, still spills: 44 to 108 bytes in the
// closest-hit kernels of one ray per thread, 46 in the persistent and 98 to 118 in
// the batched ones, 8 to 40 with any hit.
//
// Measured against warp_step on the binary nodes (persistent, refill 24):
// 1,000,003 diffuse rays on 200,000 triangles, alpha texture, closest 838 ->
// 782 us, any 812 -> 707 us; 1.2 M occlusion rays on 2 M triangles, procedural
// alpha, 505 -> 424 us; batch of 40 scenes, any, 1,245 -> 1,142 us.  Issue and
// divergence bound it now (15-17 of 32 lanes active, issue 52%, L1 data pipe
// 56%).  Coherent camera rays stay on the binary nodes: there all lanes fetch
// the same few nodes and the extra instructions per box cost more than the
// fetches save (forest frame 472 us with k_trace_oct, 807 here).
#pragma once

#include "vsr_internal.h"

namespace vsr {

constexpr uint32_t kLeft = 0x20000000u, kRight = 0x40000000u;
constexpr uint32_t kRecField = 0x1FFFFFC0u;  // record << 6
constexpr uint32_t kWideSlack = 2u;
// As kLeafWait for wide_step, whose passes make two levels (2 to 5 differ by
// 1%).
constexpr uint32_t kWideWait = 4u;

typedef unsigned long long f32x2;  // two floats, the first in the low word

__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
// Both components rounded as __fmaf_rn.
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

struct WideRec {
    uint32_t w[16];
};
__device__ __forceinline__ WideRec load_rec(const uint32_t* p) {
    WideRec r;
#ifdef VSR_CHECKED_LOADS
    for (int k = 0; k < 4; ++k) {
        const uint4 v = VSR_LDG(reinterpret_cast<const uint4*>(p) + k);
        r.w[4 * k] = v.x;
        r.w[4 * k + 1] = v.y;
        r.w[4 * k + 2] = v.z;
        r.w[4 * k + 3] = v.w;
    }
#else
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3]), "=r"(r.w[4]), "=r"(r.w[5]),
          "=r"(r.w[6]), "=r"(r.w[7])
        : "l"(p));
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(r.w[8]), "=r"(r.w[9]), "=r"(r.w[10]), "=r"(r.w[11]), "=r"(r.w[12]), "=r"(r.w[13]),
          "=r"(r.w[14]), "=r"(r.w[15])
        : "l"(p + 8));
#endif
    return r;
}

// What a thread keeps in shared memory: the ray as loaded, the running result
// as a hit record, the ray's index, the leaves it has tested, and its column of
// the traversal stack.
struct LaneStore {
    float4* rec;  // [0] origin and tmin, [stride] direction and tmax, [2 stride] result
    uint32_t stride;
    // s: the block's dynamic shared memory (wide_smem bytes)
    __device__ __forceinline__ explicit LaneStore(float4* s)
        : rec(s + threadIdx.x), stride(blockDim.x) {}
    __device__ __forceinline__ float4& org() const { return rec[0]; }
    __device__ __forceinline__ float4& dir() const { return rec[stride]; }
    __device__ __forceinline__ float4& hit() const { return rec[2u * stride]; }
    __device__ __forceinline__ Ray ray() const { return make_ray(org(), dir()); }
    // words after the block's float4s: index (two words), leaves, stack
    __device__ __forceinline__ uint32_t* words() const {
        return reinterpret_cast<uint32_t*>(rec - threadIdx.x + 3u * stride);
    }
    __device__ __forceinline__ unsigned long long& index() const {
        return reinterpret_cast<unsigned long long*>(words())[threadIdx.x];
    }
    __device__ __forceinline__ uint32_t& leaves() const {
        return words()[2u * stride + threadIdx.x];
    }
    __device__ __forceinline__ uint32_t* col() const {
        return words() + 3u * stride + threadIdx.x;
    }
    __device__ __forceinline__ uint32_t& entry(uint32_t k) const { return col()[k * stride]; }
};
inline size_t wide_smem(uint32_t block, uint32_t depth) {
    return (size_t)block * (3u * sizeof(float4) + (3u + depth + kWideSlack) * sizeof(uint32_t));
}

// A ray's constants on one axis: S twice, C of the entry and of the exit
// plane, and the byte selector that puts the entry plane's cell into the
// mantissa of 2^23 (the exit plane's is the other half word).
struct WideAxis {
    f32x2 s, c;
    uint32_t in;
    __device__ __forceinline__ void set(float inv, float no, float origin, float cell) {
        const float sc = __fmul_rn(inv, cell), base = __fmul_rn(sc, 0x1p23f);
        s = pack2(sc, sc);
        c = pack2(__fadd_rd(__fmaf_rd(origin, inv, no), -base),
                  __fadd_ru(__fmaf_ru(origin, inv, no), -base));
        in = signbit(inv) ? 0x7432u : 0x7410u;
    }
    __device__ __forceinline__ void planes(uint32_t w, float& entry, float& exit) const {
        const f32x2 q = pack2(__uint_as_float(__byte_perm(w, 0x4B000000u, in)),
                              __uint_as_float(__byte_perm(w, 0x4B000000u, in ^ 0x22u)));
        unpack2(fma2(q, s, c), entry, exit);
    }
};

// One lane's traversal.
template <int Q, class H>
struct WideLane {
    WideAxis x, y, z;
    float tmin, far;  // far: closest hit, the best t so far; any hit, tmax
    uint32_t neg, ref, n;

    __device__ __forceinline__ bool hit(const WideRec& d, int slot) const {
        float nx, fx, ny, fy, nz, fz;
        x.planes(d.w[slot], nx, fx);
        y.planes(d.w[4 + slot], ny, fy);
        z.planes(d.w[8 + slot], nz, fz);
        return fmax3(nx, ny, fmaxf(nz, tmin)) <= fmin3(fx, fy, fminf(fz, far));
    }
    __device__ __forceinline__ void fail(const LaneStore& m) const {
        m.hit() = make_float4(__int_as_float(0x7f800000), 0.0f, 0.0f, __uint_as_float(kMiss));
    }
    // The whole ray on the binary nodes (rare).  The lane's state is reset so
    // that none of it is live across that traversal, whose registers would add
    // to it.
    __device__ __forceinline__ void start_over(const DevScene& sc, const IsectParams& ip,
                                               const LaneStore& m) {
        H h;
        Best best;
        Stats st;
        ShortStack<0> stk;
        stk.init(m.col(), m.stride);
        traverse<Q, H, false>(sc, ip, m.ray(), h, best, st, stk);
        m.hit() = hit_record(best);
        x.s = x.c = y.s = y.c = z.s = z.c = 0ull;
        x.in = y.in = z.in = 0u;
        tmin = far = 0.0f;
        neg = n = 0u;
        ref = kLeafBit;
    }

    // Begin a ray; false when it needs no steps (the result is there).
    __device__ __forceinline__ bool start(const DevScene& sc, const IsectParams& ip, float4 a,
                                          float4 b, const LaneStore& m) {
        m.org() = a;
        m.dir() = b;
        m.leaves() = 0u;
        fail(m);
        const Ray r = make_ray(a, b);
        if (sc.nprims == 0 || !box_hit(r, sc.root_a, sc.root_b, r.tmax)) return false;
        uint4 ha = make_uint4(0u, 0u, 0u, 0u), hb = ha;
        if (sc.wide) {
            ha = VSR_LDG(reinterpret_cast<const uint4*>(sc.wide));
            hb = VSR_LDG(reinterpret_cast<const uint4*>(sc.wide) + 1);
        }
        if (!ha.w || !(fabsf(r.ix) >= 0x1p-80f) || !(fabsf(r.iy) >= 0x1p-80f) ||
            !(fabsf(r.iz) >= 0x1p-80f)) {
            start_over(sc, ip, m);
            return false;
        }
        x.set(r.ix, r.nox, __uint_as_float(ha.x), __uint_as_float(hb.x));
        y.set(r.iy, r.noy, __uint_as_float(ha.y), __uint_as_float(hb.y));
        z.set(r.iz, r.noz, __uint_as_float(ha.z), __uint_as_float(hb.z));
        tmin = r.tmin;
        far = r.tmax;
        neg = r.negmask * 0x11111111u;
        ref = hb.w;
        n = 0;
        return true;
    }

    // Visit the record of `ref` and move on; false when no node is left.
    __device__ __forceinline__ bool visit(const DevScene& sc, const LaneStore& m) {
        const WideRec d = load_rec(reinterpret_cast<const uint32_t*>(
            reinterpret_cast<const char*>(sc.wide) + (ref & kRecField)));
        const bool left_on = ref & kLeft, right_on = ref & kRight;
        const bool h0 = hit(d, 0) && left_on, h1 = hit(d, 1) && left_on;
        const bool h2 = hit(d, 2) && right_on, h3 = hit(d, 3) && right_on;
        const bool any_l = h0 || h1, any_r = h2 || h3;
        if (!any_l && !any_r) return pop(m);
        if (n > sc.stack_depth) {  // unreachable for a validated blob
            atomicOr(sc.err, kErrStack);
            fail(m);
            return false;
        }
        // the half on the side of the direction's sign first (`neg` repeats
        // every four bits, so the wrapping shift needs no mask)
        const bool right =
            any_r && (!any_l || (__funnelshift_r(neg, neg, ref) & 1u));
        const uint32_t axes = ref >> (right ? 4 : 2);
        if (any_l && any_r) {  // the other half waits
            const uint32_t other = ref >> (right ? 2 : 4);
            m.entry(n++) = (other & 3u) == 3u ? (right ? d.w[12] : d.w[14])
                                              : (ref & ~(right ? kRight : kLeft));
        }
        const bool a = right ? h2 : h0, b = right ? h3 : h1;
        const uint32_t r0 = right ? d.w[14] : d.w[12], r1 = right ? d.w[15] : d.w[13];
        const bool second = b && (!a || (__funnelshift_r(neg, neg, axes) & 1u));
        if (a && b && (axes & 3u) != 3u) m.entry(n++) = second ? r0 : r1;
        ref = second ? r1 : r0;
        return true;
    }
    __device__ __forceinline__ bool pop(const LaneStore& m) {
        if (n == 0u) return false;
        ref = m.entry(--n);
        return true;
    }

    // Primitive k of the leaf `ref`; `checked`: its box was tested.  Returns
    // 0 to go on, 1 to leave the leaf, 2 when the ray has its result.
    __device__ __forceinline__ int test(const DevScene& sc, const IsectParams& ip,
                                        const LaneStore& m, uint32_t k, float limit,
                                        bool& checked) {
        const float4* tp = sc.tris + 3ull * (((ref >> 3) & 0x0FFFFFFFu) + k);
        const float4 a = VSR_LDG(tp), e1 = VSR_LDG(tp + 1), e2 = VSR_LDG(tp + 2);
        const float4 o = m.org(), dd = m.dir();
        Ray r;
        r.ox = o.x; r.oy = o.y; r.oz = o.z;
        r.dx = dd.x; r.dy = dd.y; r.dz = dd.z;
        float t, u, v;
        if (!tri_test(r, a, e1, e2, t, u, v)) return 0;
        const bool geo = u >= 0.0f && v >= 0.0f && __fadd_rn(u, v) <= 1.0f;
        if (!geo || !(t > tmin) || !(t < dd.w)) return 0;
        const uint32_t prim = __float_as_uint(a.w);
        if (Q == kClosest && !hit_before(t, prim, far, __float_as_uint(m.hit().w))) return 0;
        H h;
        if (!h.accept(sc, ip, prim, u, v, t)) return 0;
        if (!checked) {
            // whether traverse_body tests this leaf
            const uint32_t leaf = __float_as_uint(e1.w);
            const float4 lo = VSR_LDG(sc.nodes + 2ull * leaf),
                         hi = VSR_LDG(sc.nodes + 2ull * leaf + 1);
            const Ray e = m.ray();
            if (!box_hit(e, lo, hi, limit)) {
                if (Q == kAny || !box_hit(e, lo, hi, e.tmax)) return 1;
                start_over(sc, ip, m);
                return 2;
            }
            checked = true;
        }
        m.hit() = make_float4(t, u, v, __uint_as_float(prim));
        if (Q == kAny) return 2;
        far = t;
        return 0;
    }
};

// warp_step (vsr_device.cuh) over the records: called by all 32 lanes, those
// without a ray with busy = false; true on busy lanes whose ray has finished.
template <int Q, class H>
__device__ __forceinline__ bool wide_step(const DevScene& sc, const IsectParams& ip,
                                          WideLane<Q, H>& w, const LaneStore& m, bool busy) {
    bool live = busy;
    const uint32_t held = (uint32_t)__popc(__ballot_sync(kFullMask, busy));
    uint32_t waited = 0;
    for (;;) {
        const bool inner = live && !(w.ref & kLeafBit);
        const uint32_t descending = (uint32_t)__popc(__ballot_sync(kFullMask, inner));
        waited += held - descending;
        if (waited >= kWideWait * descending) break;
        if (inner) live = w.visit(sc, m);
    }
    // test the leaves reached, one primitive of every lane per pass
    const bool leaf = live && (w.ref & kLeafBit);
    uint32_t cnt = leaf ? (w.ref & 7u) + 1u : 0u;
    if (leaf && ++m.leaves() > sc.max_steps) {
        atomicOr(sc.err, kErrSteps);
        w.fail(m);
        live = false;
        cnt = 0;
    }
    const float limit = w.far;
    bool checked = false;
    for (uint32_t k = 0; __any_sync(kFullMask, k < cnt); ++k) {
        if (k < cnt) {
            const int s = w.test(sc, ip, m, k, limit, checked);
            if (s) cnt = 0;
            if (s == 2) live = false;
        }
    }
    if (leaf && live) live = w.pop(m);
    return busy && !live;
}

}  // namespace vsr
