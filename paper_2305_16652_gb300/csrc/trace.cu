// Closest-hit / any-hit tracing: stack-based traversal of the BVH2 (Sec. 3.1)
// with the Moller-Trumbore ray/triangle test (1997).  GB300 has no
// ray-tracing cores, so traversal is software: one thread per ray, each
// internal node holding its children's boxes (32-byte 8-bit quantised
// layout or 64-byte exact FP32 layout of the BVH2, or 128-byte 4-ary nodes
// collapsed from it), a per-thread stack of (node, entry distance) pairs.
// Every layout's traces walk the compact 64-byte 4-ary nodes instead where the
// scene and the stack allow it (launch_layout); the layout's own nodes serve the
// other scenes and the counting diagnostic.
//
// Robustness: decoded child boxes are rounded outward (they contain the exact
// boxes), the far slab distance is widened by 1 + 2*gamma(3) to cover the
// rounding of the distances (Ize 2013, "Robust BVH Ray Traversal"; the wide
// nodes' directed-rounding distances leave only the reciprocal's rounding
// to cover, the compact nodes' bounds hold a margin for it), and a subtree is dropped only when its entry
// distance exceeds the best hit by more than 2^-16 relative, so traversal
// reaches every triangle that a ray meets.  (One that only the rounding of the
// triangle test lets it meet, past an edge or from 10^5 scene sizes away, may
// lie outside the boxes on the way to it.)
// Triangle arithmetic is the canonical Moller-Trumbore sequence with explicit
// round-to-nearest intrinsics (built with --fmad=false), so the (t, u, v) of
// a triangle are the same bit patterns on every run and in every ray order.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "hcc_internal.cuh"

namespace hcc {
namespace {

constexpr int TRACE_BLOCK = 128;
constexpr int STACK = HCC_TRACE_STACK;
// What slab distances are widened by, and the best hit before it prunes, as fractions
// of their magnitudes (distances may be negative): 2 * gamma(3), gamma(n) = n u / (1 - n u),
// u = 2^-24; and 2^-16.
constexpr float ROBUST_FAR = 0x3p-23f;
constexpr float PRUNE_SLACK = 0x1p-16f;
// idle lanes that make a warp take new rays: in input order, and in sorted
// order (rays fetched through a permutation), where waiting longer keeps the
// warp's neighbouring rays together (measured faster for each)
constexpr uint32_t REFILL_MIN = 12;
constexpr uint32_t REFILL_MIN_SORTED = 24;
// ... and over compact nodes in either order: there a round is run by the whole
// warp and costs little, so lanes need not wait as long (room's 16.6M rays in HCC
// order, whole bounce: 3.74 ms at 8, 3.75 at 6, 3.73 at 10; with a heavier step 4.20
// against 3.97 at 24)
constexpr uint32_t REFILL_MIN_COMPACT = 8;
// resident threads per SM the persistent kernel is built for; the register cap
// follows from threads x registers <= 64K: exact and quantised binary nodes
// (48 registers at 128-thread blocks), wide nodes or a batch of scenes (56), and
// compact nodes (64; at 56 or 48 registers the loop spills and more warps share
// the L1: 3.77 against 3.67 ms for the bounce above at 56; 72 registers 4.11 against 3.97)
constexpr int pool_threads(int layout, bool multi) { return layout == 3 ? 1024 : layout == 2 || multi ? 1152 : 1280; }

__device__ __forceinline__ float byte_to_float(uint32_t w, uint32_t sel) {
    // 0x4B0000bb as float is 2^23 + bb exactly
    return __fsub_rn(__uint_as_float(__byte_perm(w, 0x4B000000u, sel)), 8388608.0f);
}
// selectors for byte 0..3 of w combined with bytes of 0x4B000000
constexpr uint32_t SEL0 = 0x7540u, SEL1 = 0x7541u, SEL2 = 0x7542u, SEL3 = 0x7543u;

// The origin is kept negated and paired, (-ox, -oy) and (-oz, -oz), with the
// reciprocal direction paired alike, so one packed add and one packed
// multiply give two slab distances (lo - o) * inv.
struct Ray {
    float2 nxy, nzz, ixy, izz;
    float tmin, dx, dy, dz, tmax;
    float lx, ly, lz, ux, uy, uz;  // o * (1/d) rounded down and up, per axis
};

__device__ __forceinline__ float safe_inv(float d) {
    // a zero (or denormal) direction component is replaced by +-1e-30 for the
    // slab test only; this keeps every slab distance a number (no 0 * inf)
    return __frcp_rn(fabsf(d) > 1e-30f ? d : copysignf(1e-30f, d));
}

// A child box as pairs: (lo.x, lo.y), (hi.x, hi.y), (lo.z, hi.z).
struct Box2 {
    float2 lxy, hxy, zz;
};

// Entry / exit distance of the ray through one decoded child box of a
// binary node: t = (bound - o) * inv with round-to-nearest, two axes per
// packed add and multiply ((bound + (-o)) * inv, the same results as one at
// a time), near and far by min/max per axis.  Its three roundings make it a
// relative-error estimate, which the far distance widened by 1 + 2*gamma(3)
// covers.
__device__ __forceinline__ void slab(const Ray &r, const Box2 &b, float tcap, float &tn, float &tf) {
    const float2 a = __fmul2_rn(__fadd2_rn(b.lxy, r.nxy), r.ixy);
    const float2 c = __fmul2_rn(__fadd2_rn(b.hxy, r.nxy), r.ixy);
    const float2 z = __fmul2_rn(__fadd2_rn(b.zz, r.nzz), r.izz);
    tn = fmax3(fminf(a.x, c.x), fminf(a.y, c.y), fmaxf(fminf(z.x, z.y), r.tmin));
    const float f = fmin3(fmaxf(a.x, c.x), fmaxf(a.y, c.y), fmaxf(z.x, z.y));
    tf = fminf(__fmaf_rn(fabsf(f), ROBUST_FAR, f), tcap);
}

// A ray with a zero direction component may lie in the plane of a box's face, where the
// reciprocal that stands in for infinity gives an entry or exit at t = 0.  For
// such rays a distance of zero is taken as beyond either end.  (The check costs
// the walk of exact and quantised nodes 0.3 to 1.6 %; applied to every ray it cost
// 5 to 30 %, as rays that start on a wall then test the wall.)
__device__ __forceinline__ bool flat_ray(const Ray &r) {
    return fmax3(fabsf(r.ixy.x), fabsf(r.ixy.y), fabsf(r.izz.x)) > 0.9e30f;  // safe_inv's stand-in is 1e30
}
__device__ __forceinline__ float flat_near(float t) { return t == 0.0f ? -__int_as_float(0x7F800000) : t; }
__device__ __forceinline__ float flat_far(float t) { return t == 0.0f ? __int_as_float(0x7F800000) : t; }

__device__ __forceinline__ void slab_flat(const Ray &r, const Box2 &b, float tcap, float &tn, float &tf) {
    const float2 a = __fmul2_rn(__fadd2_rn(b.lxy, r.nxy), r.ixy);
    const float2 c = __fmul2_rn(__fadd2_rn(b.hxy, r.nxy), r.ixy);
    const float2 z = __fmul2_rn(__fadd2_rn(b.zz, r.nzz), r.izz);
    tn = fmax3(flat_near(fminf(a.x, c.x)), flat_near(fminf(a.y, c.y)), fmaxf(flat_near(fminf(z.x, z.y)), r.tmin));
    const float f = fmin3(flat_far(fmaxf(a.x, c.x)), flat_far(fmaxf(a.y, c.y)), flat_far(fmaxf(z.x, z.y)));
    tf = fminf(__fmaf_rn(fabsf(f), ROBUST_FAR, f), tcap);
}

// Moller-Trumbore; returns true with (t, u, v) if the ray's line meets the
// triangle (the caller checks t against the ray's interval).  Same operation sequence as the definition: p = d x e2,
// det = e1 . p, s = o - v0, u = (s . p) / det, q = s x e1, v = (d . q) / det,
// t = (e2 . q) / det; dot(a, b) = fma(az, bz, fma(ay, by, ax * bx)),
// cross(a, b).x = fma(ay, bz, -(az * by)) and cyclically.
__device__ __forceinline__ bool intersect(float ox, float oy, float oz, float dx, float dy, float dz, const float4 &A,
                                          const float4 &E1, const float4 &E2, float &t, float &u, float &v) {
    const float px = __fmaf_rn(dy, E2.z, -__fmul_rn(dz, E2.y));
    const float py = __fmaf_rn(dz, E2.x, -__fmul_rn(dx, E2.z));
    const float pz = __fmaf_rn(dx, E2.y, -__fmul_rn(dy, E2.x));
    const float det = __fmaf_rn(E1.z, pz, __fmaf_rn(E1.y, py, __fmul_rn(E1.x, px)));
    const float inv = __frcp_rn(det);
    const float sx = __fsub_rn(ox, A.x), sy = __fsub_rn(oy, A.y), sz = __fsub_rn(oz, A.z);
    u = __fmul_rn(__fmaf_rn(sz, pz, __fmaf_rn(sy, py, __fmul_rn(sx, px))), inv);
    const float qx = __fmaf_rn(sy, E1.z, -__fmul_rn(sz, E1.y));
    const float qy = __fmaf_rn(sz, E1.x, -__fmul_rn(sx, E1.z));
    const float qz = __fmaf_rn(sx, E1.y, -__fmul_rn(sy, E1.x));
    v = __fmul_rn(__fmaf_rn(dz, qz, __fmaf_rn(dy, qy, __fmul_rn(dx, qx))), inv);
    t = __fmul_rn(__fmaf_rn(E2.z, qz, __fmaf_rn(E2.y, qy, __fmul_rn(E2.x, qx))), inv);
    // as !(x < 0): a NaN is not rejected here, and t is then NaN as well
    return det != 0.0f && !(u < 0.0f) && !(u > 1.0f) && !(v < 0.0f) && !(__fadd_rn(u, v) > 1.0f);
}

constexpr int COMPACT = 3;  // kernel layout number of the compact nodes (0-2: hcc_bvh_layout)
constexpr uint32_t REF_NONE = 0xFFFFFFFFu;  // no node (empty stack, no postponed leaf)

// Both children's boxes of an internal node, decoded for the slab test.
struct ChildBoxes {
    Box2 b0, b1;
    uint32_t ref0, ref1;
};

// One 32-byte read-only load (sm_100+ 256-bit vector load); p must be 32-byte aligned.
__device__ __forceinline__ void ldg256(const void *p, uint4 &a, uint4 &b) {
    asm("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
        : "l"(p));
}

__device__ __forceinline__ float2 f2(uint32_t a, uint32_t b) { return make_float2(__uint_as_float(a), __uint_as_float(b)); }

// 32-byte quantised node: bounds are origin + q * 2^E rounded outward.
__device__ __forceinline__ void fetch_quant8(const uint4 *nodes, uint32_t ref, ChildBoxes &c) {
    uint4 A, B;
    ldg256(nodes + 2 * (size_t)ref, A, B);
    const float ox = __uint_as_float(A.x & 0xFFFFFF00u);
    const float oy = __uint_as_float(A.y & 0xFFFFFF00u);
    const float oz = __uint_as_float(A.z & 0xFFFFFF00u);
    const float sx = __uint_as_float((A.x & 0xFFu) << 23);
    const float sy = __uint_as_float((A.y & 0xFFu) << 23);
    const float sz = __uint_as_float((A.z & 0xFFu) << 23);
    c.b0.lxy = make_float2(__fmaf_rd(byte_to_float(A.w, SEL0), sx, ox), __fmaf_rd(byte_to_float(A.w, SEL1), sy, oy));
    c.b0.zz.x = __fmaf_rd(byte_to_float(A.w, SEL2), sz, oz);
    c.b0.hxy = make_float2(__fmaf_ru(byte_to_float(A.w, SEL3), sx, ox), __fmaf_ru(byte_to_float(B.x, SEL0), sy, oy));
    c.b0.zz.y = __fmaf_ru(byte_to_float(B.x, SEL1), sz, oz);
    c.b1.lxy = make_float2(__fmaf_rd(byte_to_float(B.x, SEL2), sx, ox), __fmaf_rd(byte_to_float(B.x, SEL3), sy, oy));
    c.b1.zz.x = __fmaf_rd(byte_to_float(B.y, SEL0), sz, oz);
    c.b1.hxy = make_float2(__fmaf_ru(byte_to_float(B.y, SEL1), sx, ox), __fmaf_ru(byte_to_float(B.y, SEL2), sy, oy));
    c.b1.zz.y = __fmaf_ru(byte_to_float(B.y, SEL3), sz, oz);
    c.ref0 = B.z;
    c.ref1 = B.w;
}

// 64-byte exact node: per child (lo.x, lo.y), (hi.x, hi.y), (lo.z, hi.z) as
// stored in the input BVH, then the two references.
__device__ __forceinline__ void fetch_exact(const uint4 *nodes, uint32_t ref, ChildBoxes &c) {
    uint4 w0, w1, w2, n3;
    ldg256(nodes + 4 * (size_t)ref, w0, w1);
    ldg256(nodes + 4 * (size_t)ref + 2, w2, n3);
    c.b0.lxy = f2(w0.x, w0.y);
    c.b0.hxy = f2(w0.z, w0.w);
    c.b0.zz = f2(w1.x, w1.y);
    c.b1.lxy = f2(w1.z, w1.w);
    c.b1.hxy = f2(w2.x, w2.y);
    c.b1.zz = f2(w2.z, w2.w);
    c.ref0 = n3.x;
    c.ref1 = n3.y;
}

// Child c of a 128-byte wide node (rows of four floats: lo.x hi.x lo.y
// hi.y lo.z hi.z, then the four references) given the ray's near and far
// rows (boxes are stored with lo <= hi, so the near plane of an axis is lo
// for a positive reciprocal direction and hi for a negative one).  Directed
// slab test: the near distance (near - o) * inv is bounded from below by one
// fma rounded down against o * inv rounded up, the far one from above by
// one fma rounded up against o * inv rounded down, so the only error left
// is the relative one of the rounded reciprocal, which the widened far
// distance covers.  t is the child's entry distance if the ray meets it
// (clamped to the largest float, so +inf marks only unused and missed
// slots), else +inf.
__device__ __forceinline__ float wide_child(const Ray &r, float nx, float ny, float nz, float fx, float fy, float fz,
                                            uint32_t ref, float tcap) {
    const float ix = r.ixy.x, iy = r.ixy.y, iz = r.izz.x;
    const float tn = fmax3(__fmaf_rd(nx, ix, -r.ux), __fmaf_rd(ny, iy, -r.uy), fmaxf(__fmaf_rd(nz, iz, -r.uz), r.tmin));
    const float f = fmin3(__fmaf_ru(fx, ix, -r.lx), __fmaf_ru(fy, iy, -r.ly), __fmaf_ru(fz, iz, -r.lz));
    const float tf = fminf(__fmaf_rn(fabsf(f), ROBUST_FAR, f), tcap);
    return (tn <= tf && ref != 0xFFFFFFFFu) ? fminf(tn, 3.40282347e38f) : __int_as_float(0x7F800000);
}

// Orders two (distance, reference) pairs by distance.
__device__ __forceinline__ void order2(float &ta, uint32_t &ra, float &tb, uint32_t &rb) {
    const bool sw = tb < ta;
    const float t = ta;
    const uint32_t x = ra;
    ta = sw ? tb : ta;
    ra = sw ? rb : ra;
    tb = sw ? t : tb;
    rb = sw ? x : rb;
}

// Diagnostic counters of one ray (the COUNT variants only).
struct Counters {
    uint32_t nodes = 0, tris = 0, warp_nodes = 0, warp_leaves = 0;
};

// Traversal state of one ray: the ray, the best hit so far, the node being
// descended and the parked leaf.  The stack lives beside it in the kernel.
struct RayState {
    Ray r;
    float best_t, best_u, best_v, tcap;  // tcap: best_t widened by the prune slack
    int32_t best_prim;
    int sp;
    uint32_t node, leaf;
    bool overflow;
};

// o * inv rounded down and up, for wide nodes.  For a zero direction component they
// are moved apart by 1e20 or four places, so that a ray in the plane of a
// box's face lies within the box (as slab_flat does for binary nodes).
__device__ __forceinline__ void scaled_origin(float o, float d, float inv, float &down, float &up) {
    down = __fmul_rd(o, inv);
    up = __fmul_ru(o, inv);
    if (!(fabsf(d) > 1e-30f)) {
        const float apart = fmaxf(fabsf(up) * 0x1p-22f, 1e20f);
        down = __fsub_rd(down, apart);
        up = __fadd_ru(up, apart);
    }
}

__device__ __forceinline__ void ray_init(RayState &s, const float4 o4, const float4 d4, uint32_t root_ref) {
    s.r.nxy = make_float2(-o4.x, -o4.y);
    s.r.nzz = make_float2(-o4.z, -o4.z);
    s.r.tmin = o4.w;
    s.r.dx = d4.x;
    s.r.dy = d4.y;
    s.r.dz = d4.z;
    s.r.tmax = d4.w;
    const float ix = safe_inv(d4.x), iy = safe_inv(d4.y), iz = safe_inv(d4.z);
    s.r.ixy = make_float2(ix, iy);
    s.r.izz = make_float2(iz, iz);
    scaled_origin(o4.x, d4.x, ix, s.r.lx, s.r.ux);
    scaled_origin(o4.y, d4.y, iy, s.r.ly, s.r.uy);
    scaled_origin(o4.z, d4.z, iz, s.r.lz, s.r.uz);
    s.best_t = s.r.tmax;
    s.best_u = s.best_v = 0.0f;
    s.best_prim = -1;
    s.tcap = s.r.tmax;
    s.sp = 0;
    s.overflow = false;
    s.node = root_ref;
    s.leaf = REF_NONE;
    if (s.node & REF_LEAF) {
        s.leaf = s.node;
        s.node = REF_NONE;
    }
}

__device__ __forceinline__ bool ray_done(const RayState &s) { return s.node == REF_NONE && s.leaf == REF_NONE; }

// Pending subtrees are (node reference, entry distance) entries of a
// STACKN-entry array in local memory, one 8-byte access each.
template <int STACKN>
__device__ __forceinline__ bool ray_push(RayState &s, uint2 *stack, uint2 e) {  // false: no room
    if (s.sp >= STACKN) return false;
    stack[s.sp++] = e;
    return true;
}

// Next pending subtree that can still hold a closer hit, or REF_NONE.
__device__ __forceinline__ uint32_t ray_pop(RayState &s, const uint2 *stack) {
    while (s.sp > 0) {
        const uint2 e = stack[--s.sp];
        if (__uint_as_float(e.y) <= s.tcap) return e.x;
    }
    return REF_NONE;
}

// The node loop of a closest-hit round ends once all but LEAF_SLACK of the
// warp's lanes still descending hold a parked leaf.  Waiting for every lane
// (the plain postponed-leaf rule) kept the others idle behind the last few
// descents: on the room's 16.6M rays a slack of 3 or 4 traced 4.6 %
// (unsorted) and 2 % (HCC order) faster than 0, 6 and 8 slower than 3.
// The leaf loop of a closest-hit round goes on to the next leaf on the stack
// while at least LEAF_MIN lanes have one (4 measured best of 0, 4, 8 and 12:
// 0.6 % faster than chaining leaves while any lane has one).  Any-hit traces
// keep the plain rules (every lane; chain while any lane has a leaf), which
// measured 1-2 % faster for them.
constexpr int LEAF_SLACK = 3;
constexpr int LEAF_MIN = 4;
template <bool ANY>
__device__ __forceinline__ bool leaves_ready(uint32_t leaf) {
    if (ANY) return __all_sync(__activemask(), leaf != REF_NONE);
    const uint32_t active = __activemask();
    const uint32_t parked = __ballot_sync(active, leaf != REF_NONE);
    return __popc(parked) + LEAF_SLACK >= __popc(active);
}

// One round of the traversal loop ("while-while" with postponed leaves,
// Aila & Laine 2009): descend internal nodes until (nearly) every lane of
// the warp holds a leaf (a lane that reaches a leaf parks it and keeps
// descending), then test the parked leaf and any leaf that is next on the
// stack; a lane without a leaf yet resumes its descent in the next round.  The
// nearer child is visited first and the farther one is pushed with its
// entry distance, which lets a pop skip subtrees beyond the best hit.
template <bool ANY, bool COUNT, int LAYOUT, int STACKN>
__device__ __forceinline__ void ray_round(RayState &s, uint2 *stack, const uint4 *__restrict__ nodes,
                                          const float4 *__restrict__ tris, Counters &cn) {
    const uint32_t lane = threadIdx.x & 31;
    // wide nodes: the met children sorted by entry distance (a five-exchange
    // network on four pairs), the nearest descended, the others pushed
    // farthest first
    while (LAYOUT == 2 && s.node != REF_NONE && !(s.node & REF_LEAF)) {
        const float4 *nd = reinterpret_cast<const float4 *>(nodes) + 8 * (size_t)s.node;
        if (COUNT) {
            ++cn.nodes;
            if (lane == (uint32_t)(__ffs(__activemask()) - 1)) ++cn.warp_nodes;
        }
        // the near row of an axis is lo for a positive reciprocal direction
        const uint32_t sx = s.r.ixy.x < 0.0f, sy = s.r.ixy.y < 0.0f, sz = s.r.izz.x < 0.0f;
        const float4 nx = __ldg(nd + sx), fx = __ldg(nd + 1 - sx);
        const float4 ny = __ldg(nd + 2 + sy), fy = __ldg(nd + 3 - sy);
        const float4 nz = __ldg(nd + 4 + sz), fz = __ldg(nd + 5 - sz);
        const uint4 rf = __ldg(reinterpret_cast<const uint4 *>(nd + 6));
        uint32_t r0 = rf.x, r1 = rf.y, r2 = rf.z, r3 = rf.w;
        float t0 = wide_child(s.r, nx.x, ny.x, nz.x, fx.x, fy.x, fz.x, r0, s.tcap);
        float t1 = wide_child(s.r, nx.y, ny.y, nz.y, fx.y, fy.y, fz.y, r1, s.tcap);
        float t2 = wide_child(s.r, nx.z, ny.z, nz.z, fx.z, fy.z, fz.z, r2, s.tcap);
        float t3 = wide_child(s.r, nx.w, ny.w, nz.w, fx.w, fy.w, fz.w, r3, s.tcap);
        order2(t0, r0, t1, r1);
        order2(t2, r2, t3, r3);
        order2(t0, r0, t2, r2);
        order2(t1, r1, t3, r3);
        order2(t1, r1, t2, r2);
        const float INF = __int_as_float(0x7F800000);
        const int met = (t0 < INF) + (t1 < INF) + (t2 < INF) + (t3 < INF);
        if (met == 0) {
            s.node = ray_pop(s, stack);
        } else {
            if (s.sp + met - 1 > STACKN) {
                s.overflow = true;
                s.node = s.leaf = REF_NONE;
                break;
            }
            if (met > 3) ray_push<STACKN>(s, stack, make_uint2(r3, __float_as_uint(t3)));
            if (met > 2) ray_push<STACKN>(s, stack, make_uint2(r2, __float_as_uint(t2)));
            if (met > 1) ray_push<STACKN>(s, stack, make_uint2(r1, __float_as_uint(t1)));
            s.node = r0;
        }
        if (s.node != REF_NONE && (s.node & REF_LEAF) && s.leaf == REF_NONE) {
            s.leaf = s.node;
            s.node = ray_pop(s, stack);
        }
        if (leaves_ready<ANY>(s.leaf)) break;
    }
    // internal nodes: descend until (nearly) every lane has a leaf parked
    while (LAYOUT != 2 && s.node != REF_NONE && !(s.node & REF_LEAF)) {
        ChildBoxes c;
        if (LAYOUT == 0)
            fetch_quant8(nodes, s.node, c);
        else
            fetch_exact(nodes, s.node, c);
        if (COUNT) {
            ++cn.nodes;  // this lane's node visit; the lowest active lane counts the warp's step
            if (lane == (uint32_t)(__ffs(__activemask()) - 1)) ++cn.warp_nodes;
        }
        float tn0, tf0, tn1, tf1;
        slab(s.r, c.b0, s.tcap, tn0, tf0);
        slab(s.r, c.b1, s.tcap, tn1, tf1);
        if (flat_ray(s.r)) {
            slab_flat(s.r, c.b0, s.tcap, tn0, tf0);
            slab_flat(s.r, c.b1, s.tcap, tn1, tf1);
        }
        const bool h0 = tn0 <= tf0, h1 = tn1 <= tf1;
        if (h0 && h1) {
            const bool first0 = tn0 <= tn1;
            if (!ray_push<STACKN>(s, stack, make_uint2(first0 ? c.ref1 : c.ref0, __float_as_uint(first0 ? tn1 : tn0)))) {
                s.overflow = true;
                s.node = s.leaf = REF_NONE;
                break;
            }
            s.node = first0 ? c.ref0 : c.ref1;
        } else if (h0) {
            s.node = c.ref0;
        } else if (h1) {
            s.node = c.ref1;
        } else {
            s.node = ray_pop(s, stack);
        }
        if (s.node != REF_NONE && (s.node & REF_LEAF) && s.leaf == REF_NONE) {
            s.leaf = s.node;
            s.node = ray_pop(s, stack);
        }
        if (leaves_ready<ANY>(s.leaf)) break;
    }
    // leaves: the parked one, then any leaf that is next on the stack
    while (s.leaf != REF_NONE) {
        if (COUNT && lane == (uint32_t)(__ffs(__activemask()) - 1)) ++cn.warp_leaves;
        const uint32_t first = s.leaf & REF_TRI_MASK, cnt = ((s.leaf >> 29) & 3u) + 1u;
        bool hit_any = false;
        for (uint32_t k = 0; k < cnt; ++k) {
            const float4 *rec = tris + 3 * (size_t)(first + k);
            const float4 A = __ldg(rec), E1 = __ldg(rec + 1), E2 = __ldg(rec + 2);
            if (COUNT) ++cn.tris;
            float t, u, v;
            if (!intersect(-s.r.nxy.x, -s.r.nxy.y, -s.r.nzz.x, s.r.dx, s.r.dy, s.r.dz, A, E1, E2, t, u, v)) continue;
            if (!(t > s.r.tmin && t < s.r.tmax)) continue;
            const int32_t prim = __float_as_int(A.w);
            if (s.best_prim < 0 || t < s.best_t || (t == s.best_t && prim < s.best_prim)) {
                s.best_t = t;
                s.best_u = u;
                s.best_v = v;
                s.best_prim = prim;
                s.tcap = __fmaf_rn(fabsf(t), PRUNE_SLACK, t);
            }
            hit_any = true;
            if (ANY) break;
        }
        if (ANY && hit_any) {
            s.node = s.leaf = REF_NONE;
            break;
        }
        s.leaf = REF_NONE;
        if (s.node != REF_NONE && (s.node & REF_LEAF)) {
            s.leaf = s.node;
            s.node = ray_pop(s, stack);
        }
        // fewer than LEAF_MIN lanes with a next leaf: keep it parked for
        // the next round rather than hold the warp here for them
        if (!ANY && __popc(__ballot_sync(__activemask(), s.leaf != REF_NONE)) < LEAF_MIN) break;
    }
}

// ---------------------------------------------------------------- compact nodes
//
// Why these nodes: a trace over the exact binary nodes kept the L1 data pipe 72 %
// busy (two 32-byte loads per lane and visit, each lane its own line; the wide
// nodes, seven 16-byte loads, 85 %) and waited for loads in 7.6 of 16 cycles per
// instruction.  A compact node is read with two 32-byte loads for four children, so a
// ray needs 16 visits and 33 loads where the binary nodes take 36 and 72, and the room's
// nodes shrink from 32 to 13 MB.  What bounds the walk now (ncu, 1.0M rays in
// HCC order): the ALU pipe 64 %, issue 62 %, L1 data pipe 60 % busy at 21 lanes an
// instruction, waits for loads 4.3 of 12.2 cycles per instruction; for 16.6M rays
// 2.45 billion warp instructions against 3.41.

// Traversal state over compact 4-ary nodes.  The slab test works in the
// scene's grid: per axis tau = b * inv + c with b a decoded bound, inv the
// reciprocal of the grid-space direction and c = -(origin * inv), one fma per
// bound.  Its rounding, and that of the ray's grid coordinates, is below the
// margin by which the stored bounds were widened, so no factor on the far
// distance is needed.  tau is the ray's parameter t measured from `from` (tmin, or
// the entry into the scene for an origin or a tmin far outside it) and scaled by a power
// of two that brings the scene's far side below 1: a saturating fma then
// clamps the entry distance to the ray's start.
struct CompactState {
    float2 ixy, cxy, far_cxy;  // far_c: c + widen, rounded up
    float iz, cz, far_cz;
    uint32_t sx, sy, sz;  // byte selectors of each axis's near bound (lo or hi by the direction's sign)
    float tcap;           // tau of the best hit widened by the prune slack
    float widen;          // added to a box's exit distance (0 unless the origin is far outside the scene)
    float ox, oy, oz, dx, dy, dz;
    float best_t, best_u, best_v;
    int32_t best_prim;
    uint32_t sp;          // local address of the next free stack entry
    uint32_t node, leaf;  // subtree to descend and parked leaf, or REF_NONE
    uint32_t top_ref;     // copy of the topmost stack entry
    float top_t;
    static constexpr bool overflow = false;  // launch_trace walks compact nodes only where the stack suffices
};

// Stack slots below the pending subtrees: (tmin, scale) and (from, -), read only when a triangle is met.
constexpr int COMPACT_SLOTS = 2;
// What the triangle test's own rounding may move a ray by, of its distance from its origin
// (it grows with that distance; the other layouts' slab tests round alike).
constexpr double FAR_NOISE = 0x1p-20;
// Least component of a direction that counts, of the longest one.
constexpr float LEAST_COMPONENT = 0x1p-60f;
constexpr uint32_t GRID_HI_LO = 0x0220u;  // turns the selector of one bound of a word into the other's

// A 16-bit bound of word w as a grid coordinate in [2, 8): bytes (0, low, high, 0x40).
__device__ __forceinline__ float grid_bound(uint32_t w, uint32_t sel) {
    return __uint_as_float(__byte_perm(w, 0x40u, sel));
}

// A ray as the slab test sees it: point p at t = `from` (to within its rounding), grid-space
// direction d times 1 / unit, and what its distances may be off by (in t * unit).
struct GridRay {
    float3 p, d;
    float from, unit, noise;
};

// Sets up, in double, a ray whose origin is more than GRID_REACH from the grid's zero, whose
// interval starts further than that behind its origin, or whose direction is of extreme
// length: measures t from the point where it enters the scene's neighbourhood (one
// unit and the noise around the grid's box), so that the grid coordinates of the slab test
// and the distances it takes from them stay small, and brings the direction's length near 1.
// Returns 0 if the ray never comes near, 2 if the noise is larger than the scene on every
// axis (then no box can be told from any other), else 1.
__device__ __noinline__ int enter_grid(const float4 o4, const float4 d4, const Grid &g, GridRay &r) {
    const float o[3] = {o4.x, o4.y, o4.z}, d[3] = {d4.x, d4.y, d4.z};
    double op[3], dp[3];
    for (int k = 0; k < 3; ++k) {
        op[k] = ((double)o[k] - (double)g.lo[k]) * (double)g.scale[k] + (double)GRID_ORIGIN;
        dp[k] = (double)d[k] * (double)g.scale[k];
        if (!isfinite(op[k]) || !isfinite(dp[k])) return 0;  // not a ray
    }
    const double longest = fmax(fmax(fabs(dp[0]), fabs(dp[1])), fabs(dp[2]));
    if (longest == 0.0) return 0;
    const int e = min(max(ilogb(longest), -120), 120);
    double tin = (double)o4.w - fabs((double)o4.w) * FAR_NOISE, tout = (double)d4.w + fabs((double)d4.w) * FAR_NOISE;
    for (int k = 0; k < 3; ++k) {
        const double lo = 1.0 - fabs(op[k]) * FAR_NOISE, hi = 9.0 + fabs(op[k]) * FAR_NOISE;
        if (dp[k] == 0.0) {
            if (!(op[k] >= lo && op[k] <= hi)) return 0;
        } else {
            const double a = (lo - op[k]) / dp[k], b = (hi - op[k]) / dp[k];
            tin = fmax(tin, fmin(a, b));
            tout = fmin(tout, fmax(a, b));
        }
    }
    if (!(tin <= tout)) return 0;
    r.from = __double2float_rd(tin);
    r.unit = (float)scalbn(1.0, e);
    r.p = make_float3((float)(op[0] + tin * dp[0]), (float)(op[1] + tin * dp[1]), (float)(op[2] + tin * dp[2]));
    r.d = make_float3((float)scalbn(dp[0], -e), (float)scalbn(dp[1], -e), (float)scalbn(dp[2], -e));
    r.noise = __double2float_ru(scalbn(fabs(tin) * FAR_NOISE, e));
    // below the gap between the bounds of an unused child (5.99 units), which must never be met
    const float least = LEAST_COMPONENT * fmax3(fabsf(r.d.x), fabsf(r.d.y), fabsf(r.d.z));
    const float slowest = fmaxf(fminf(fminf(fabsf(r.d.x), fabsf(r.d.y)), fabsf(r.d.z)), least);
    return r.noise * slowest < 5.9f ? 1 : 2;
}

__device__ __forceinline__ uint32_t local_address(const void *p) {
    uint64_t a;
    asm("cvta.to.local.u64 %0, %1;" : "=l"(a) : "l"(p));
    return (uint32_t)a;
}

// As safe_inv, for a grid-space direction; one ulp of error, which the bounds' margin covers.
// A component of less than `least` counts as that much: at 2^-60 of the longest one it moves
// a ray by nothing, and what comes of its reciprocal stays finite at any scale.
// (A constant least value, of 1e-36, took c to infinity for rays that soon leave the scene.)
__device__ __forceinline__ float grid_inv(float d, float least) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(fabsf(d) > least ? d : copysignf(least, d)));
    return r;
}

// A lane without a ray.
__device__ __forceinline__ void ray_none(CompactState &s, uint32_t stack_base) {
    s.node = s.leaf = REF_NONE;
    s.sp = stack_base;
}

__device__ __forceinline__ bool ray_done(const CompactState &s, uint32_t stack_base) {
    return s.node == REF_NONE && s.leaf == REF_NONE && s.sp == stack_base;
}

__device__ __forceinline__ void ray_init(CompactState &s, uint2 *stack, const float4 o4, const float4 d4,
                                         const Grid &g, uint32_t root) {
    s.ox = o4.x;
    s.oy = o4.y;
    s.oz = o4.z;
    s.dx = d4.x;
    s.dy = d4.y;
    s.dz = d4.z;
    float3 p = make_float3(__fmaf_rn(__fsub_rn(o4.x, g.lo[0]), g.scale[0], GRID_ORIGIN),
                           __fmaf_rn(__fsub_rn(o4.y, g.lo[1]), g.scale[1], GRID_ORIGIN),
                           __fmaf_rn(__fsub_rn(o4.z, g.lo[2]), g.scale[2], GRID_ORIGIN));
    const float gx = __fmul_rn(d4.x, g.scale[0]), gy = __fmul_rn(d4.y, g.scale[1]), gz = __fmul_rn(d4.z, g.scale[2]);
    const float longest = fmax3(fabsf(gx), fabsf(gy), fabsf(gz));
    float from = o4.w, tau_scale;
    int meets = 1;
    // the rest for a ray whose tmin is `start` as seen from p and whose distances are off by up to noise
    auto set_up = [&](float3 dir, float length, float start, float unit, float noise) {
        const float least = __fmul_rn(length, LEAST_COMPONENT);
        const float ix = grid_inv(dir.x, least), iy = grid_inv(dir.y, least), iz = grid_inv(dir.z, least);
        // the far side of the scene, in t from `from` (times unit)
        const float cx = __fmaf_rn(-p.x, ix, -start), cy = __fmaf_rn(-p.y, iy, -start), cz = __fmaf_rn(-p.z, iz, -start);
        const float leave = __fadd_rn(fmin3(__fmaf_rn(ix < 0.0f ? 2.0f : 8.0f, ix, cx), __fmaf_rn(iy < 0.0f ? 2.0f : 8.0f, iy, cy),
                                            __fmaf_rn(iz < 0.0f ? 2.0f : 8.0f, iz, cz)), noise);
        const float tmax = __fmaf_ru(__fsub_ru(d4.w, from), unit, noise);
        // 2^-(e + 2) for a far side in [2^e, 2^(e+1)); a far side at or before the start is a miss
        const uint32_t e = __float_as_uint(fmaxf(leave, 2e-38f)) >> 23;
        const float scale = __uint_as_float((252u - (e < 251u ? e : 251u)) << 23);
        if (!(leave > 0.0f && tmax > 0.0f)) meets = 0;
        s.ixy = make_float2(__fmul_rn(ix, scale), __fmul_rn(iy, scale));
        s.iz = __fmul_rn(iz, scale);
        s.cxy = make_float2(__fmul_rn(cx, scale), __fmul_rn(cy, scale));
        s.cz = __fmul_rn(cz, scale);
        s.sx = ix < 0.0f ? 0x4325u : 0x4105u;
        s.sy = iy < 0.0f ? 0x4325u : 0x4105u;
        s.sz = iz < 0.0f ? 0x4325u : 0x4105u;
        s.tcap = __fmul_ru(tmax, scale);
        s.widen = __fmul_rn(noise, scale);
        tau_scale = __fmul_rn(scale, unit);
    };
    // a far origin or a direction longer than 2^120, a far tmin behind the origin (one that far
    // ahead is beyond the scene, and the ray a miss above), or a direction shorter than 2^-60
    if (fmax3(__fmaf_rn(longest, 0x1p-115f, fmax3(fabsf(p.x), fabsf(p.y), fabsf(p.z))), __fmul_rn(-from, longest),
              __fmaf_rn(longest, -0x1p70f, 0x1p10f)) > GRID_REACH) {
        GridRay r = {};
        meets = enter_grid(o4, d4, g, r);
        p = r.p;
        from = r.from;
        set_up(r.d, fmax3(fabsf(r.d.x), fabsf(r.d.y), fabsf(r.d.z)), 0.0f, r.unit, r.noise);
        if (meets == 2) {
            // every box is met and none is pruned: one axis takes them to entries of at most 3
            // and exits of at least 2.4 steps, an unused child to 3 and 2.4, the others to 0 and 5.4
            constexpr float STEP = 1.0f / 16.0f;
            s.ixy = make_float2(STEP, 0.0f);
            s.cxy = make_float2(-5.0f * STEP, 0.0f);
            s.iz = s.cz = 0.0f;
            s.sx = s.sy = s.sz = 0x4105u;
            s.widen = 5.4f * STEP;
            s.tcap = __int_as_float(0x7F800000);
            from = -__int_as_float(0x7F800000);  // compact_cap: infinite
            tau_scale = 1.0f;
        }
    } else {
        set_up(make_float3(gx, gy, gz), longest, from, 1.0f, 0.0f);
    }
    s.far_cxy = make_float2(__fadd_ru(s.cxy.x, s.widen), __fadd_ru(s.cxy.y, s.widen));
    s.far_cz = __fadd_ru(s.cz, s.widen);
    s.best_t = d4.w;
    s.best_u = s.best_v = 0.0f;
    s.best_prim = -1;
    stack[0] = make_uint2(__float_as_uint(o4.w), __float_as_uint(tau_scale));
    stack[1] = make_uint2(__float_as_uint(from), 0u);
    s.node = meets ? root : REF_NONE;
    s.leaf = REF_NONE;
}

// tau of a hit at t, widened by the prune slack.
__device__ __forceinline__ float compact_cap(float t, float from, float scale) {
    const float tau = __fsub_ru(t, from);
    return __fmul_ru(__fmaf_ru(__fadd_ru(fabsf(t), tau), PRUNE_SLACK, tau), scale);
}

// A leaf that is next becomes the lane's parked leaf if it has none (a node of
// REF_NONE changes nothing).  Predicated moves: no branch, and off the ALU pipe.
__device__ __forceinline__ void park_leaf(CompactState &s) {
    asm("{\n\t.reg .pred p;\n\t"
        "setp.eq.u32 p, %1, 0xffffffff;\n\t"
        "setp.lt.and.s32 p, %0, 0, p;\n\t"
        "@p mov.b32 %1, %0;\n\t"
        "@p mov.b32 %0, 0xffffffff;\n\t}"
        : "+r"(s.node), "+r"(s.leaf));
}

// Takes the next pending subtree if the lane has none to descend; one beyond
// the best hit is dropped (the lane tries again in the next step).  The topmost
// entry is kept in registers and its successor is loaded when it is taken, so a
// pop does not wait for local memory.  (Any hit: the best hit never moves, so
// entries are references only.)
template <bool ANY>
__device__ __forceinline__ void pop_node(CompactState &s, uint32_t stack_base) {
    if (ANY) {
        asm volatile("{\n\t.reg .pred p;\n\t"
            "setp.eq.u32 p, %0, 0xffffffff;\n\t"
            "setp.ne.and.u32 p, %1, %2, p;\n\t"
            "@p add.u32 %1, %1, -4;\n\t"
            "@p ld.local.b32 %0, [%1];\n\t}"
            : "+r"(s.node), "+r"(s.sp) : "r"(stack_base) : "memory");
        return;
    }
    asm volatile("{\n\t.reg .pred p, q;\n\t"
        "setp.eq.u32 p, %0, 0xffffffff;\n\t"
        "setp.ne.and.u32 p, %1, %5, p;\n\t"
        "setp.le.and.f32 q, %3, %4, p;\n\t"
        "@q mov.b32 %0, %2;\n\t"
        "@p add.u32 %1, %1, -8;\n\t"
        "@p ld.local.v2.b32 {%2, %3}, [%1+-8];\n\t}"
        : "+r"(s.node), "+r"(s.sp), "+r"(s.top_ref), "+f"(s.top_t) : "f"(s.tcap), "r"(stack_base) : "memory");
}

// Entry and exit distance of a child (slab words wx, wy, wz); CAP: the exit no later
// than the best hit; FAR_C: the exit widened by its own constants.  The near and far
// bound of an axis come out of its word by byte permutes whose selectors hold the
// direction's sign, so decoding costs no more than sorting the two distances by
// min and max would.
template <bool CAP, bool FAR_C>
__device__ __forceinline__ void compact_child(const CompactState &s, uint32_t wx, uint32_t wy, uint32_t wz, float &tn,
                                              float &tf) {
    const float2 n = __ffma2_rn(make_float2(grid_bound(wx, s.sx), grid_bound(wy, s.sy)), s.ixy, s.cxy);
    const float2 f = __ffma2_rn(make_float2(grid_bound(wx, s.sx ^ GRID_HI_LO), grid_bound(wy, s.sy ^ GRID_HI_LO)),
                                s.ixy, FAR_C ? s.far_cxy : s.cxy);
    const float nz = __saturatef(__fmaf_rn(grid_bound(wz, s.sz), s.iz, s.cz));
    const float fz = __fmaf_rn(grid_bound(wz, s.sz ^ GRID_HI_LO), s.iz, FAR_C ? s.far_cz : s.cz);
    tn = fmax3(n.x, n.y, nz);
    tf = fmin3(f.x, f.y, fz);
    if (!FAR_C) tf = __fadd_rn(tf, s.widen);
    if (CAP) tf = fminf(tf, s.tcap);
}

// Entry distance of a child for the order of a step: its own if the ray meets it,
// beyond any cap if it does not, by two multiply-adds where a compare and a
// select would take the ALU pipe.  (A box missed by less than 1e-37 of the scene
// may count as met, which costs a visit.)  With the best hit capping the pushes
// alone, 12 of the step's ALU instructions less: 16.6M rays in HCC order, whole
// bounce, 3.87 -> 3.77 ms, 2.1M unsorted 427 -> 414 us.
constexpr float CAP_MAX = 8.0f;  // no box of the scene is met beyond 1
__device__ __forceinline__ float met_distance(float tn, float tf) {
    return __fmaf_rn(__saturatef(__fsub_rn(tn, tf)), 1e38f, tn);
}

// Pushes a subtree met at distance t before the best hit.  TOP: the last push of a
// step, which leaves the topmost entry.
template <bool TOP>
__device__ __forceinline__ void push_node(CompactState &s, uint32_t ref, float t) {
    if (TOP)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %4, %5;\n\t"
            "@p st.local.v2.b32 [%0], {%3, %4};\n\t@p add.u32 %0, %0, 8;\n\t@p mov.b32 %1, %3;\n\t@p mov.b32 %2, %4;\n\t}"
            : "+r"(s.sp), "+r"(s.top_ref), "+f"(s.top_t) : "r"(ref), "f"(t), "f"(s.tcap) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %2, %3;\n\t"
            "@p st.local.v2.b32 [%0], {%1, %2};\n\t@p add.u32 %0, %0, 8;\n\t}"
            : "+r"(s.sp) : "r"(ref), "f"(t), "f"(s.tcap) : "memory");
}

// One node step: tests the four children, descends into the nearest one met
// and pushes the others, farthest first.  (Pushing them unsorted saved 10
// instructions of 185 a step but took 13 % more steps; multiply-adds in place of
// the selects of the exchanges, to relieve the ALU pipe, changed nothing.)
// FAR_C pays where three registers are left for it: an addition per child less
// for single wavefronts' closest hits (1080p bounce 3736 -> 3674 us, 2.1M unsorted 409 ->
// 400), but any hit (559 -> 566 us for 4.1M shadow rays) and a batch (1188 -> 1230)
// run out of registers.
template <bool ANY, bool FAR_C>
__device__ __forceinline__ void node_step(CompactState &s, const uint4 *__restrict__ nodes) {
    uint4 w0, w1, w2, rf;
    ldg256(nodes + 4 * (size_t)s.node, w0, w1);
    ldg256(nodes + 4 * (size_t)s.node + 2, w2, rf);
    float n0, n1, n2, n3, f0, f1, f2, f3;
    compact_child<ANY, FAR_C>(s, w0.x, w0.y, w0.z, n0, f0);
    compact_child<ANY, FAR_C>(s, w0.w, w1.x, w1.y, n1, f1);
    compact_child<ANY, FAR_C>(s, w1.z, w1.w, w2.x, n2, f2);
    compact_child<ANY, FAR_C>(s, w2.y, w2.z, w2.w, n3, f3);
    if (ANY) {
        // no order and no distance: every met child is pushed, the last taken back
        asm volatile("{\n\t.reg .pred h0, h1, h2, h3, p;\n\t"
            "setp.lt.f32 h0, %2, %6;\n\tsetp.lt.f32 h1, %3, %7;\n\tsetp.lt.f32 h2, %4, %8;\n\tsetp.lt.f32 h3, %5, %9;\n\t"
            "mov.b32 %0, 0xffffffff;\n\t"
            "@h0 st.local.b32 [%1], %10;\n\t@h0 add.u32 %1, %1, 4;\n\t@h0 mov.b32 %0, %10;\n\t"
            "@h1 st.local.b32 [%1], %11;\n\t@h1 add.u32 %1, %1, 4;\n\t@h1 mov.b32 %0, %11;\n\t"
            "@h2 st.local.b32 [%1], %12;\n\t@h2 add.u32 %1, %1, 4;\n\t@h2 mov.b32 %0, %12;\n\t"
            "@h3 st.local.b32 [%1], %13;\n\t@h3 add.u32 %1, %1, 4;\n\t@h3 mov.b32 %0, %13;\n\t"
            "setp.ne.u32 p, %0, 0xffffffff;\n\t@p add.u32 %1, %1, -4;\n\t}"
            : "=&r"(s.node), "+r"(s.sp)
            : "f"(n0), "f"(n1), "f"(n2), "f"(n3), "f"(f0), "f"(f1), "f"(f2), "f"(f3), "r"(rf.x), "r"(rf.y), "r"(rf.z), "r"(rf.w)
            : "memory");
        return;
    }
    n0 = met_distance(n0, f0);
    n1 = met_distance(n1, f1);
    n2 = met_distance(n2, f2);
    n3 = met_distance(n3, f3);
    uint32_t r0 = rf.x, r1 = rf.y, r2 = rf.z, r3 = rf.w;
    order2(n0, r0, n1, r1);
    order2(n2, r2, n3, r3);
    order2(n0, r0, n2, r2);
    order2(n1, r1, n3, r3);
    order2(n1, r1, n2, r2);
    s.node = n0 < s.tcap ? r0 : REF_NONE;
    push_node<false>(s, r3, n3);
    push_node<false>(s, r2, n2);
    push_node<true>(s, r1, n1);
}

// A read-only 16-byte load that L1 evicts first: triangles are met by few rays
// each and would push out nodes and stacks (16.6M rays in HCC order, whole
// bounce: 3.92 -> 3.87 ms, 2.1M unsorted 434 -> 426 us; not cached in L1 at all: 4.65 ms and
// 604 us; nodes evicted last on top: no change).
__device__ __forceinline__ float4 ldg_first(const float4 *p) {
    float4 r;
    asm("ld.global.nc.L1::evict_first.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
        : "l"(p));
    return r;
}

// One round over compact nodes, run by the whole warp together (a lane without
// a ray takes part in the votes only): node steps until all but COMPACT_SLACK of
// the lanes that could go on hold a parked leaf, then triangle tests, one triangle
// per lane and step, while at least COMPACT_TRI_MIN lanes have one; a leaf that
// is not finished stays parked for the next round.  A step keeps its branches
// few (predicated pushes, pops and moves, all of the triangle test computed at
// once): with a branch around each, a warp spent 30 of 206 instructions per node
// step on branching, and pops alone in loops at 10 % of its lanes.  (The plain
// rules for any hit, as for the other layouts: 592 us for 4.1M shadow rays and
// their order against 596 with a slack of 4 lanes.)
constexpr int COMPACT_SLACK = 6;    // 4: equal in HCC order, 1.8 % slower unsorted; 8: 0.3 % slower, 0.8 % faster
constexpr int COMPACT_TRI_MIN = 6;  // 4 and 8 within 0.5 %
template <bool ANY, bool FAR_C>
__device__ __forceinline__ void ray_round(CompactState &s, const uint2 *stack, uint32_t stack_base,
                                          const uint4 *__restrict__ nodes, const float4 *__restrict__ tris) {
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    bool more;
    do {
        pop_node<ANY>(s, stack_base);
        if ((int)s.node >= 0) node_step<ANY, FAR_C>(s, nodes);
        park_leaf(s);
        more = s.leaf == REF_NONE && (s.node != REF_NONE || s.sp != stack_base);
    } while (__popc(__ballot_sync(FULL, more)) > (ANY ? 0 : COMPACT_SLACK));
    while (__any_sync(FULL, s.leaf != REF_NONE)) {
        if (s.leaf != REF_NONE) {
            const float4 *rec = tris + 3 * (size_t)(s.leaf & REF_TRI_MASK);
            const float4 A = ldg_first(rec), E1 = ldg_first(rec + 1), E2 = ldg_first(rec + 2);
            // the next triangle of the leaf, or the next leaf
            if (s.leaf & ~(REF_LEAF | REF_TRI_MASK)) {
                s.leaf -= REF_TRI_MASK;
            } else {
                s.leaf = REF_NONE;
                park_leaf(s);
            }
            float t, u, v;
            const bool met = intersect(s.ox, s.oy, s.oz, s.dx, s.dy, s.dz, A, E1, E2, t, u, v);
            const int32_t prim = __float_as_int(A.w);
            if (met && (t < s.best_t || (t == s.best_t && prim < s.best_prim))) {
                const uint2 e0 = stack[0], e1 = stack[1];
                if (t > __uint_as_float(e0.x)) {
                    s.best_t = t;
                    s.best_u = u;
                    s.best_v = v;
                    s.best_prim = prim;
                    s.tcap = compact_cap(t, __uint_as_float(e1.x), __uint_as_float(e0.y));
                    if (ANY) ray_none(s, stack_base);
                }
            }
        }
        if (__popc(__ballot_sync(FULL, s.leaf != REF_NONE)) < (ANY ? 1 : COMPACT_TRI_MIN)) break;
    }
}

// The hit record {prim, t, u, v} (prim -1 and t = +inf on a miss or a
// stack overflow).
template <typename State>
__device__ __forceinline__ int4 ray_result(const State &s) {
    const bool miss = s.overflow || s.best_prim < 0;
    int4 out;
    out.x = miss ? -1 : s.best_prim;
    out.y = __float_as_int(miss ? __int_as_float(0x7F800000) : s.best_t);
    out.z = __float_as_int(miss ? 0.0f : s.best_u);
    out.w = __float_as_int(miss ? 0.0f : s.best_v);
    return out;
}

template <bool COUNT>
__device__ __forceinline__ void add_counts(const TraceArgs &a, const Counters &cn) {
    if (COUNT) {
        if (cn.nodes) atomicAdd(a.counts, (unsigned long long)cn.nodes);
        if (cn.tris) atomicAdd(a.counts + 1, (unsigned long long)cn.tris);
        if (cn.warp_nodes) atomicAdd(a.counts + 2, (unsigned long long)cn.warp_nodes);
        if (cn.warp_leaves) atomicAdd(a.counts + 3, (unsigned long long)cn.warp_leaves);
    }
}

// Reads ray slot i (the ray is org/dir[gather[i]], or i) and sets up its
// traversal.  Returns false (and reports) for an out-of-range permutation entry.
template <bool ANY, bool MULTI, int LAYOUT, typename State>
__device__ __forceinline__ bool start_ray(const TraceArgs &a, uint64_t i, State &s, uint2 *stack,
                                          const uint4 *&nodes, const float4 *&tris) {
    float4 o4, d4;
    uint64_t src = i;
    if (a.gather) {
        src = a.gather[i];
        if (src >= a.n) {  // invalid permutation entry: report, never read out of bounds
            atomicOr(a.err, ERR_INDEX);
            return false;
        }
    }
    if (a.rec) {  // one 32-byte record: a single access per ray
        asm volatile("ld.global.cs.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(o4.x), "=f"(o4.y), "=f"(o4.z), "=f"(o4.w), "=f"(d4.x), "=f"(d4.y), "=f"(d4.z), "=f"(d4.w)
                     : "l"(a.org + 2 * src));
    } else {
        o4 = __ldcs(a.org + src * a.rs);
        d4 = __ldcs(a.dir + src * a.rs);
    }
    const SceneDesc *sc = MULTI ? a.scenes + scene_of(a.offsets, a.num_scenes, src) : nullptr;
    if (MULTI) {
        tris = sc->tris;
        nodes = LAYOUT == COMPACT ? sc->cnodes : sc->nodes;
    }
    if constexpr (LAYOUT == COMPACT) {
        ray_init(s, stack, o4, d4, MULTI ? sc->grid : a.grid, MULTI ? sc->croot : a.croot);
        if (!ANY) s.tcap = fminf(s.tcap, CAP_MAX);
    } else {
        ray_init(s, o4, d4, MULTI ? sc->root_ref : a.root_ref);
    }
    return true;
}

template <int LAYOUT>
using StateOf = std::conditional_t<LAYOUT == COMPACT, CompactState, RayState>;
// Stack entries of a kernel with STACKN entries for pending subtrees.
template <int LAYOUT, int STACKN>
constexpr int STACK_SIZE = STACKN + (LAYOUT == COMPACT ? COMPACT_SLOTS : 0);

// Writes the record of ray slot i to hits[scatter[i]] (or i).
template <typename State>
__device__ __forceinline__ void store_hit(const TraceArgs &a, uint64_t i, const State &s) {
    if (i >= a.n) {  // not a ray slot: report, never index the permutation out of bounds
        atomicOr(a.err, ERR_INDEX);
        return;
    }
    if (s.overflow) atomicOr(a.err, ERR_STACK);
    const uint64_t dst = a.scatter ? (uint64_t)a.scatter[i] : i;
    if (dst < a.n)
        __stcs(a.hits + dst, ray_result(s));
    else  // invalid scatter entry: report, never write out of bounds
        atomicOr(a.err, ERR_INDEX);
}

// One thread per ray slot.  MULTI: the ray's BVH is that of its scene in a
// batch (a.scenes, ray ranges a.offsets).  COUNT = true is a diagnostic
// variant that also adds up work counters into a.counts (never timed).
// (Compact nodes: nine blocks per SM, 56 registers, 583 us for 4.1M shadow rays and
// their order against 595 at seven or eight and 590 at ten.)
template <bool ANY, bool COUNT, int LAYOUT, bool MULTI>
__global__ void __launch_bounds__(TRACE_BLOCK, LAYOUT == COMPACT ? 9 : 1) k_trace(TraceArgs a) {
    uint64_t i = (uint64_t)blockIdx.x * TRACE_BLOCK + threadIdx.x;
    const uint4 *nodes = MULTI ? nullptr : LAYOUT == COMPACT ? a.cnodes : a.nodes;
    const float4 *tris = MULTI ? nullptr : a.tris;
    StateOf<LAYOUT> s;
    uint2 stack[STACK_SIZE<LAYOUT, STACK>];
    Counters cn;
    bool have = i < a.n;
    if (have) {
        if (a.gather || a.scatter) i = a.n - 1 - i;  // sorted order from its end (blocks start in index order)
        have = start_ray<ANY, MULTI, LAYOUT>(a, i, s, stack, nodes, tris);
    }
    if constexpr (LAYOUT == COMPACT) {
        const uint32_t base = local_address(stack + COMPACT_SLOTS);
        s.sp = base;
        if (!have) ray_none(s, base);
        while (__any_sync(0xFFFFFFFFu, !ray_done(s, base))) ray_round<ANY, false>(s, stack, base, nodes, tris);
        if (!have) return;
    } else {
        if (!have) return;
        while (!ray_done(s)) ray_round<ANY, COUNT, LAYOUT, STACK>(s, stack, nodes, tris, cn);
    }
    store_hit(a, i, s);
    add_counts<COUNT>(a, cn);
}

// ------------------------------------------------- four lanes per ray
//
// For wavefronts too small to fill the GPU a trace lasts as long as its longest
// ray, and that ray as long as its chain of dependent steps.  Here four lanes
// share a ray: each tests one child of a compact node and keeps the pending
// children that it met on a stack of its own, and each tests one
// triangle of a leaf, so that a step is a third of the instructions of
// node_step and a leaf a single test.  All four hold the ray; minima over the quad
// (two shuffles) pick the next subtree: the nearest child met, else the topmost
// entry of the deepest level, ordered by one 32-bit key:
//   63 - level, then 22 bits of the entry distance (rounded down), then the lane
// The deepest level first makes it a depth-first walk, so a lane's stack holds at
// most one entry per level.  Bound by the latency of that chain (a load from L2, two
// shuffles and about 80 instructions a step); as throughput it is worse (0.96M
// rays: 563 against 321 us), so launch_layout keeps it to small wavefronts.
// (Prefetching the met children's nodes: no change at 4,096 rays, 4 % slower at 65,536.)
constexpr int QUAD_SLACK = 8;  // lanes that may still descend when the triangles are tested (0: 5 % slower, 16: 1 %)
constexpr uint64_t QUAD_MAX_N = 70000, QUAD_MAX_N_ANY = 50000;
constexpr uint32_t QUAD_MAX_LEVEL = 60;
constexpr uint32_t QUAD_NONE = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t quad_min(uint32_t v) {
    v = min(v, __shfl_xor_sync(0xFFFFFFFFu, v, 1));
    return min(v, __shfl_xor_sync(0xFFFFFFFFu, v, 2));
}

// Lower bound of the entry distance in a key.
__device__ __forceinline__ float quad_distance(uint32_t key) { return __uint_as_float((key & 0x00FFFFFCu) << 6); }

template <bool ANY>
__global__ void __launch_bounds__(TRACE_BLOCK) k_trace_quad(TraceArgs a) {
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const uint32_t lane = threadIdx.x & 31, child = lane & 3;
    uint64_t i = (uint64_t)blockIdx.x * (TRACE_BLOCK / 4) + threadIdx.x / 4;
    wait_for_previous();
    CompactState s;
    uint2 aux[COMPACT_SLOTS], stack[STACK];
    s.node = s.leaf = REF_NONE;
    s.best_prim = -1;
    const uint4 *nodes = a.cnodes;
    const float4 *tris = a.tris;
    bool have = i < a.n;
    if (have) {
        if (a.gather || a.scatter) i = a.n - 1 - i;  // sorted order from its end, as the other traces
        have = start_ray<ANY, false, COMPACT>(a, i, s, aux, nodes, tris);
    }
    const float tmin = __uint_as_float(aux[0].x), scale = __uint_as_float(aux[0].y), from = __uint_as_float(aux[1].x);
    uint32_t level = 1;  // of the current node's children
    uint32_t top_ref = REF_NONE, top_key = QUAD_NONE;
    int sp = 0;
    bool owner = false;  // this lane found the quad's best hit
    // drops the topmost entry, and those below it beyond the best hit
    auto pop = [&]() {
        do {
            --sp;
            const uint2 e = sp > 0 ? stack[sp - 1] : make_uint2(REF_NONE, QUAD_NONE);
            top_ref = e.x;
            top_key = e.y;
        } while (sp > 0 && quad_distance(top_key) > s.tcap);
    };
    bool live = have && (s.node != REF_NONE || s.leaf != REF_NONE);
    while (__any_sync(FULL, live)) {
        bool more;
        do {
            if (s.leaf == REF_NONE && s.node != REF_NONE && (s.node & REF_LEAF)) {  // park
                s.leaf = s.node;
                s.node = REF_NONE;
            }
            const bool internal = !(s.node & REF_LEAF);
            uint32_t key = QUAD_NONE, ref = REF_NONE;
            if (internal) {
                const uint32_t *w = reinterpret_cast<const uint32_t *>(a.cnodes) + 16 * (size_t)s.node;
                const uint32_t wx = __ldg(w + 3 * child), wy = __ldg(w + 3 * child + 1), wz = __ldg(w + 3 * child + 2);
                ref = __ldg(w + 12 + child);
                float tn, tf;
                compact_child<true, false>(s, wx, wy, wz, tn, tf);
                if (tn < tf) key = ((63u - level) << 24) | ((__float_as_uint(tn) >> 6) & 0x00FFFFFCu) | child;
            }
            const bool met = key != QUAD_NONE;
            const bool wants = internal || s.node == REF_NONE;  // not held up by a second leaf
            if (!met) {
                key = wants ? top_key : QUAD_NONE;
                ref = top_ref;
            }
            const uint32_t best = quad_min(key);
            const uint32_t next = __shfl_sync(FULL, ref, (lane & ~3u) | (best & 3u));
            if (met && key != best) {  // another child is nearer: pending
                stack[sp++] = make_uint2(ref, key);
                top_ref = ref;
                top_key = key;
            } else if (!met && key == best && key != QUAD_NONE) {
                pop();
            }
            if (wants) {
                s.node = best != QUAD_NONE ? next : REF_NONE;
                level = 64u - (best >> 24);
            }
            if (s.leaf == REF_NONE && s.node != REF_NONE && (s.node & REF_LEAF)) {
                s.leaf = s.node;
                s.node = REF_NONE;
            }
            more = s.leaf == REF_NONE && (s.node != REF_NONE);
        } while (__popc(__ballot_sync(FULL, more)) > (ANY ? 0 : QUAD_SLACK));
        // every lane one triangle of its quad's parked leaf
        const bool at_leaf = s.leaf != REF_NONE;
        float t = 0.0f, u = 0.0f, v = 0.0f;
        int32_t prim = 0x7FFFFFFF;
        bool hit = false;
        if (at_leaf && child <= ((s.leaf >> 29) & 3u)) {
            const float4 *rec = tris + 3 * (size_t)((s.leaf & REF_TRI_MASK) + child);
            const float4 A = __ldg(rec), E1 = __ldg(rec + 1), E2 = __ldg(rec + 2);
            const int32_t id = __float_as_int(A.w);
            if (intersect(s.ox, s.oy, s.oz, s.dx, s.dy, s.dz, A, E1, E2, t, u, v) && t > tmin &&
                (t < s.best_t || (t == s.best_t && id < s.best_prim))) {
                hit = true;
                prim = id;
            }
        }
        if (at_leaf) s.leaf = REF_NONE;
        if (__any_sync(FULL, hit)) {
            // the quad's smallest (t, triangle id)
            float bt = hit ? t : __int_as_float(0x7F800000);
            bt = fminf(bt, __shfl_xor_sync(FULL, bt, 1));
            bt = fminf(bt, __shfl_xor_sync(FULL, bt, 2));
            const bool tied = hit && t == bt;
            int32_t bp = tied ? prim : 0x7FFFFFFF;
            bp = min(bp, __shfl_xor_sync(FULL, bp, 1));
            bp = min(bp, __shfl_xor_sync(FULL, bp, 2));
            if (bp != 0x7FFFFFFF) {
                s.best_t = bt;
                s.best_prim = bp;
                owner = tied && prim == bp;
                if (owner) {
                    s.best_u = u;
                    s.best_v = v;
                }
                s.tcap = compact_cap(bt, from, scale);
                if (ANY) {
                    s.node = REF_NONE;
                    sp = 0;
                    top_key = QUAD_NONE;
                } else if (sp > 0 && quad_distance(top_key) > s.tcap) {
                    pop();
                }
            }
        }
        // a quad lives while it has a node, a leaf or a pending entry
        const uint32_t pending = __ballot_sync(FULL, sp > 0);
        live = s.node != REF_NONE || s.leaf != REF_NONE || ((pending >> (lane & ~3u)) & 15u);
    }
    if (!have) return;
    if (s.best_prim >= 0 ? owner : child == 0) store_hit(a, i, s);
}

// Persistent variant with ray replacement (Aila & Laine 2009, "replacing
// terminated rays"): each warp takes ray slots from a global counter, runs
// traversal rounds, and after each round the lanes whose ray has finished
// take new slots (all at once, one atomic per warp) as soon as refill_min of
// them are idle or none is busy.  Slots are handed out in counter order,
// so lanes of a warp trace neighbouring slots -- in sorted order, rays with
// equal keys.  Every ray's record is the same as in k_trace: a ray's own
// traversal does not depend on which rays share its warp, except for which
// of several hits an any-hit query returns first.  A trace in sorted order
// (rays fetched through a permutation, or already gathered and their hits
// written back through one) hands out its slots from the end of
// the order, largest keys first: in HCC order those are the rays whose keys
// set the most cut nodes and the longest traversals (the room's 16.6M rays:
// 54.8 node visits per ray in the last tenth of the order, 15.8 in the
// first), and starting them first leaves short rays for the end of the
// launch, where warps run out of work (its HCC trace: 4.08 ms against 4.19
// in ascending order).
// BLOCK threads per block and STACKN stack entries per ray are a shape the
// autotuner may pick.
template <bool ANY, bool COUNT, int LAYOUT, bool MULTI, int BLOCK, int STACKN>
__global__ void __launch_bounds__(BLOCK, pool_threads(LAYOUT, MULTI) / BLOCK)
    k_trace_pool(TraceArgs a) {
    wait_for_previous();
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lt;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt));
    StateOf<LAYOUT> s;
    uint2 stack[STACK_SIZE<LAYOUT, STACKN>];
    Counters cn;
    const uint4 *nodes = MULTI ? nullptr : LAYOUT == COMPACT ? a.cnodes : a.nodes;
    const float4 *tris = MULTI ? nullptr : a.tris;
    uint32_t slot = 0;  // below n, which fits 32 bits
    bool have = false, exhausted = false;
    const uint32_t stack_base = LAYOUT == COMPACT ? local_address(stack + COMPACT_SLOTS) : 0u;
    if constexpr (LAYOUT == COMPACT) ray_none(s, stack_base);
    const uint32_t refill_min = LAYOUT == COMPACT ? REFILL_MIN_COMPACT : a.gather ? REFILL_MIN_SORTED : REFILL_MIN;
    for (;;) {
        const bool want = !have && !exhausted;
        const uint32_t need = __ballot_sync(FULL, want);
        const uint32_t busy = __ballot_sync(FULL, have);
        if (need && (busy == 0 || (uint32_t)__popc(need) >= refill_min)) {
            const int leader = __ffs(need) - 1;
            unsigned long long base = 0;
            if ((int)lane == leader) base = atomicAdd(&a.work->next, (unsigned long long)__popc(need));
            base = __shfl_sync(FULL, base, leader);
            if (want) {
                const uint64_t at = base + __popc(need & lt);
                if (at < a.n) {
                    slot = (uint32_t)((a.gather || a.scatter) ? a.n - 1 - at : at);  // sorted order from its end
                    have = start_ray<ANY, MULTI, LAYOUT>(a, slot, s, stack, nodes, tris);
                } else {
                    exhausted = true;
                }
            }
        }
        if (!__any_sync(FULL, have)) {
            if (__any_sync(FULL, exhausted)) break;
            continue;
        }
        bool done;
        if constexpr (LAYOUT == COMPACT) {
            ray_round<ANY, !ANY && !MULTI>(s, stack, stack_base, nodes, tris);
            done = ray_done(s, stack_base);
        }
        if (have) {
            if constexpr (LAYOUT != COMPACT) {
                ray_round<ANY, COUNT, LAYOUT, STACKN>(s, stack, nodes, tris, cn);
                done = ray_done(s);
            }
            if (done) {
                store_hit(a, slot, s);
                have = false;
            }
        }
    }
    add_counts<COUNT>(a, cn);
    // the last block to finish clears the counters for the next trace
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&a.work->done, 1u) == gridDim.x - 1) {
            a.work->next = 0;
            a.work->done = 0;
        }
    }
}

}  // namespace

namespace {

// Resident blocks per SM of one persistent kernel on the current device
// (queried once per device and kernel).
int resident_blocks(const void *kernel, int block) {
    static std::mutex mu;
    static std::vector<std::pair<std::pair<int, const void *>, int>> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    for (const auto &e : cache)
        if (e.first.first == dev && e.first.second == kernel) return e.second;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0) != cudaSuccess || per_sm <= 0) {
        cudaGetLastError();
        per_sm = 1;
    }
    cache.push_back({{dev, kernel}, per_sm});
    return per_sm;
}

// Persistent grid: every block resident at once.
template <bool ANY, bool CNT, int LAYOUT, bool MULTI, int BLOCK, int STACKN>
cudaError_t launch_pool(cudaStream_t s, const TraceArgs &a) {
    const auto kernel = k_trace_pool<ANY, CNT, LAYOUT, MULTI, BLOCK, STACKN>;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const unsigned cap = (unsigned)std::max(1, sms) * (unsigned)resident_blocks((const void *)kernel, BLOCK);
    const unsigned blocks = (unsigned)std::min<uint64_t>((a.n + BLOCK - 1) / BLOCK, cap);
    return launch_early(kernel, blocks, BLOCK, 0, s, a);
}

// The closest-hit persistent trace in the shape the context asks for; the
// any-hit and counting variants keep the default shape.
template <bool ANY, bool CNT, int LAYOUT, bool MULTI>
cudaError_t launch_pool_shaped(cudaStream_t s, const TraceArgs &a) {
    if constexpr (ANY || CNT) {
        return launch_pool<ANY, CNT, LAYOUT, MULTI, TRACE_BLOCK, STACK>(s, a);
    } else {
        switch (a.block * 1000 + a.stack) {
            case 64032: return launch_pool<ANY, CNT, LAYOUT, MULTI, 64, 32>(s, a);
            case 64048: return launch_pool<ANY, CNT, LAYOUT, MULTI, 64, 48>(s, a);
            case 64064: return launch_pool<ANY, CNT, LAYOUT, MULTI, 64, 64>(s, a);
            case 128032: return launch_pool<ANY, CNT, LAYOUT, MULTI, 128, 32>(s, a);
            case 128048: return launch_pool<ANY, CNT, LAYOUT, MULTI, 128, 48>(s, a);
            case 256032: return launch_pool<ANY, CNT, LAYOUT, MULTI, 256, 32>(s, a);
            case 256048: return launch_pool<ANY, CNT, LAYOUT, MULTI, 256, 48>(s, a);
            case 256064: return launch_pool<ANY, CNT, LAYOUT, MULTI, 256, 64>(s, a);
            default: return launch_pool<ANY, CNT, LAYOUT, MULTI, TRACE_BLOCK, STACK>(s, a);
        }
    }
}

template <bool ANY, bool CNT, bool MULTI>
cudaError_t launch_layout(cudaStream_t s, const TraceArgs &a, bool pool) {
    // Compact nodes wherever they exist and their deepest stack fits the trace's.
    // They replaced each layout's own nodes by measurement (the trace alone, exact nodes
    // against compact: the room's 16.6M rays unsorted 4.79 -> 3.00 ms, in HCC order
    // 3.97 -> 2.92, 33.2M shadow rays 3.82 -> 3.18 and 2.90 -> 2.49).  Rays so alike
    // that the binary nodes stay in L1 gain least, as a step over four children is
    // bound by its arithmetic: 16.6M rays off one patch of floor 3.75 -> 3.20 ms
    // unsorted, but 3.04 -> 3.06 in HCC order and 2.67 -> 2.95 by origin and direction
    // (a context may ask for its layout's nodes: a.cstack is then beyond any stack).
    if constexpr (!CNT) {
        const int depth = pool && !ANY ? a.stack : STACK;
        if (a.cstack <= (uint32_t)depth) {
            if constexpr (!MULTI) {
                // Four lanes per ray where the rays do not fill the GPU (whole call, one
                // lane against four: sorted 4,096 rays 76 / 55 us, 20,000 83 / 67, 65,536 96 /
                // 86, 80,000 106 / 100; unsorted 40,000 60 / 45, 65,536 65 / 66, 80,000 69 /
                // 71; shadow rays 40,000 51 / 48, 65,536 52 / 53, 80,000 60 / 65); a walk's
                // levels are at most its stack entries.
                if (a.quads && a.n <= (ANY ? QUAD_MAX_N_ANY : QUAD_MAX_N) && a.cstack <= QUAD_MAX_LEVEL) {
                    return launch_early(k_trace_quad<ANY>, (unsigned)((a.n + TRACE_BLOCK / 4 - 1) / (TRACE_BLOCK / 4)),
                                        TRACE_BLOCK, 0, s, a);
                }
            }
            if (pool) return launch_pool_shaped<ANY, CNT, COMPACT, MULTI>(s, a);
            k_trace<ANY, CNT, COMPACT, MULTI><<<(unsigned)((a.n + TRACE_BLOCK - 1) / TRACE_BLOCK), TRACE_BLOCK, 0, s>>>(a);
            return cudaGetLastError();
        }
    }
    if (pool) {
        if (a.layout == 0) return launch_pool_shaped<ANY, CNT, 0, MULTI>(s, a);
        if (a.layout == 1) return launch_pool_shaped<ANY, CNT, 1, MULTI>(s, a);
        return launch_pool_shaped<ANY, CNT, 2, MULTI>(s, a);
    }
    const unsigned blocks = (unsigned)((a.n + TRACE_BLOCK - 1) / TRACE_BLOCK);
    if (a.layout == 0)
        k_trace<ANY, CNT, 0, MULTI><<<blocks, TRACE_BLOCK, 0, s>>>(a);
    else if (a.layout == 1)
        k_trace<ANY, CNT, 1, MULTI><<<blocks, TRACE_BLOCK, 0, s>>>(a);
    else
        k_trace<ANY, CNT, 2, MULTI><<<blocks, TRACE_BLOCK, 0, s>>>(a);
    return cudaGetLastError();
}

template <bool ANY, bool CNT>
cudaError_t launch_multi(cudaStream_t s, const TraceArgs &a, bool pool) {
    return a.scenes ? launch_layout<ANY, CNT, true>(s, a, pool) : launch_layout<ANY, CNT, false>(s, a, pool);
}

}  // namespace

bool trace_shape_supported(uint32_t block, uint32_t stack) {
    const uint32_t shapes[][2] = {{64, 32}, {64, 48}, {64, 64}, {128, 32}, {128, 48}, {128, 64},
                                  {256, 32}, {256, 48}, {256, 64}};
    for (const auto &sh : shapes)
        if (sh[0] == block && sh[1] == stack) return true;
    return false;
}

cudaError_t launch_trace(cudaStream_t s, const TraceArgs &a, int any_hit) {
    if (a.n == 0) return cudaSuccess;
    const bool count = a.counts != nullptr, pool = a.work != nullptr;
    if (any_hit && count) return launch_multi<true, true>(s, a, pool);
    if (any_hit) return launch_multi<true, false>(s, a, pool);
    if (count) return launch_multi<false, true>(s, a, pool);
    return launch_multi<false, false>(s, a, pool);
}

}  // namespace hcc
