// Key encoding kernels: hierarchy cut code (Algorithm 1, Sec. 4.2.1), its
// multi-level form (Sec. 4.3), the prefix path code (Sec. 4.1) and the
// TwoPoint, Origin and Origin-Direction baselines (Sec. 3.2, Sec. 5).
//
// Floating point: every rounding step is an explicit round-to-nearest
// intrinsic (scalar, or Blackwell's packed FP32x2 add and multiply, which
// round each half the same way) and the library is built with
// --fmad=false, so each key is the same bit pattern the arithmetic defines,
// whatever the compiler schedules.
#include "hcc_internal.cuh"

namespace hcc {
namespace {

constexpr int ENC_BLOCK = 256;
constexpr int ENC_BLOCKS = 8;  // blocks per SM of the encode grids
constexpr uint32_t MAX_CUT_BITS = 64;

int encode_grid(uint64_t n, int block, int per_sm) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
    uint64_t want = (n + block - 1) / block;
    uint64_t cap = (uint64_t)sms * per_sm;
    return (int)(want < cap ? (want ? want : 1) : cap);
}

// Slab test of one ray against one box: t = (bound - o) * (1/d) per axis,
// tnear = max over axes and tmin, tfar = min over axes and tmax, met when
// tnear <= tfar (fminf/fmaxf ignore the NaN of 0 * inf).
__device__ __forceinline__ bool meets(const float4 &o, const float4 &d, float ix, float iy, float iz, const float4 &lo,
                                      const float4 &hi) {
    const float ax = __fmul_rn(__fsub_rn(lo.x, o.x), ix), bx = __fmul_rn(__fsub_rn(hi.x, o.x), ix);
    const float ay = __fmul_rn(__fsub_rn(lo.y, o.y), iy), by = __fmul_rn(__fsub_rn(hi.y, o.y), iy);
    const float az = __fmul_rn(__fsub_rn(lo.z, o.z), iz), bz = __fmul_rn(__fsub_rn(hi.z, o.z), iz);
    const float tnear = fmax3(fminf(ax, bx), fminf(ay, by), fmaxf(fminf(az, bz), o.w));
    const float tfar = fmin3(fmaxf(ax, bx), fmaxf(ay, by), fminf(fmaxf(az, bz), d.w));
    return tnear <= tfar;
}

// Cut boxes staged in shared memory for the slab test: per box and axis the two
// orders of its bounds, entry 2 * axis holding (lo, hi) and entry 2 * axis + 1 (hi,
// lo), so that a ray reads the (near, far) bounds of an axis with one 64-bit
// load indexed by its direction's sign.  Returns whether the box is finite with lo <= hi.
constexpr uint32_t BOX = 6;  // entries of a box
__device__ __forceinline__ bool stage_box(float2 *b, const float4 *__restrict__ box) {
    const float4 lo = __ldg(box), hi = __ldg(box + 1);
    b[0] = make_float2(lo.x, hi.x);
    b[1] = make_float2(hi.x, lo.x);
    b[2] = make_float2(lo.y, hi.y);
    b[3] = make_float2(hi.y, lo.y);
    b[4] = make_float2(lo.z, hi.z);
    b[5] = make_float2(hi.z, lo.z);
    const float inf = __int_as_float(0x7F800000);
    auto ordered = [&](float l, float u) { return -inf < l && l <= u && u < inf; };
    return ordered(lo.x, hi.x) && ordered(lo.y, hi.y) && ordered(lo.z, hi.z);
}

__device__ __forceinline__ bool stage_boxes(float2 *staged, const float4 *__restrict__ boxes, uint32_t n) {
    bool ordered = true;
    for (uint32_t q = threadIdx.x; q < n; q += blockDim.x) ordered = stage_box(staged + BOX * q, boxes + 2 * q) && ordered;
    return ordered;
}

// A ray set up for the slab test of staged boxes.
struct SlabRay {
    float4 o, d;
    float ix, iy, iz;
    bool fast;
};

__device__ __forceinline__ SlabRay slab_ray(const float4 &o, const float4 &d, bool ordered) {
    SlabRay r;
    r.o = o;
    r.d = d;
    r.ix = __frcp_rn(d.x);
    r.iy = __frcp_rn(d.y);
    r.iz = __frcp_rn(d.z);
    r.fast = ordered && isfinite(r.ix) && isfinite(r.iy) && isfinite(r.iz);
    return r;
}

// Bits of n staged boxes, box 0 in the highest of the n low bits: 1 = the ray
// meets it.  Every ray may call it.
//
// With finite reciprocals and finite boxes with lo <= hi the near and far bound of
// an axis are known from the reciprocal's sign (rounding is monotonic; a NaN, from
// a zero reciprocal or a NaN origin, is both or neither), so no distance is sorted: (bound + (-o)) * inv of both bounds is one packed add and
// one packed multiply, the same round-to-nearest results as (bound - o) * inv one at a
// time.
//
// Bound by the shared-memory data pipe, which returns the 24 bytes per ray and
// box in six cycles a warp (90 % of the time of 16.6M rays against 32 boxes,
// 0.36 ms).  Two boxes per 128-bit load with the result taken from the sign of a
// difference, 13 instructions per ray and box instead of 20, left that time as it is
// (0.365 ms), and cost two-level keys 5 to 15 % (16 bits: 0.289 against 0.270 ms).
template <typename K>
__device__ __forceinline__ K met_boxes(const SlabRay &r, const float2 *boxes, uint32_t n) {
    K bits = 0;
    if (r.fast) {
        const float2 *px = boxes + (r.ix < 0.0f), *py = boxes + 2 + (r.iy < 0.0f), *pz = boxes + 4 + (r.iz < 0.0f);
        const float2 nox = make_float2(-r.o.x, -r.o.x), noy = make_float2(-r.o.y, -r.o.y),
                     noz = make_float2(-r.o.z, -r.o.z);
        const float2 ixx = make_float2(r.ix, r.ix), iyy = make_float2(r.iy, r.iy), izz = make_float2(r.iz, r.iz);
#pragma unroll 8
        for (uint32_t q = 0; q < n; ++q) {
            const float2 tx = __fmul2_rn(__fadd2_rn(px[BOX * q], nox), ixx);
            const float2 ty = __fmul2_rn(__fadd2_rn(py[BOX * q], noy), iyy);
            const float2 tz = __fmul2_rn(__fadd2_rn(pz[BOX * q], noz), izz);
            const float tnear = fmax3(tx.x, ty.x, fmaxf(tz.x, r.o.w));
            const float tfar = fmin3(tx.y, ty.y, fminf(tz.y, r.d.w));
            bits = (bits << 1) | (K)(tnear <= tfar);
        }
    } else {
        for (uint32_t q = 0; q < n; ++q) {
            const float2 x = boxes[BOX * q], y = boxes[BOX * q + 2], z = boxes[BOX * q + 4];
            bits = (bits << 1) | (K)meets(r.o, r.d, r.ix, r.iy, r.iz, make_float4(x.x, y.x, z.x, 0.f),
                                          make_float4(x.y, y.y, z.y, 0.f));
        }
    }
    return bits;
}

// HCC key of one ray against `used` staged boxes: node r drives bit key_bits - 1 - r.
template <typename K>
__device__ __forceinline__ K hcc_key(const SlabRay &r, const float2 *boxes, uint32_t used, uint32_t key_bits) {
    const K key = met_boxes<K>(r, boxes, used);
    return used ? key << (key_bits - used) : key;
}

// Algorithm 1: the cut nodes are staged in shared memory once per block
// (line 1); every ray is tested against every cut node and each result is
// one key bit.
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_hcc(const float4 *__restrict__ org,
                                                          const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                          const float4 *__restrict__ cut, uint32_t used,
                                                          uint32_t key_bits, K *__restrict__ keys) {
    __shared__ float2 s_boxes[MAX_CUT_BITS * BOX];
    const bool ordered = __syncthreads_and(stage_boxes(s_boxes, cut, used));  // a cut is not written after its creation
    wait_for_previous();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const SlabRay r = slab_ray(__ldcs(org + i * rs), __ldcs(dir + i * rs), ordered);
        __stcs(keys + i, hcc_key<K>(r, s_boxes, used, key_bits));
    }
}

// Normalise p to the box [lo, lo + ext], clamp to [0, 1], quantise to b bits.
__device__ __forceinline__ uint32_t quantise(float p, float lo, float ext, uint32_t b) {
    if (b == 0) return 0u;
    float u = (ext == 0.0f) ? 0.0f : __fdiv_rn(__fsub_rn(p, lo), ext);
    u = fminf(fmaxf(u, 0.0f), 1.0f);
    const uint32_t q = __float2uint_rz(__fmul_rn(u, (float)(1u << b)));
    const uint32_t qmax = (1u << b) - 1u;
    return q < qmax ? q : qmax;
}

// The bits of x (below 2^5 for M = 6, 2^10 for M = 3 and 2) M apart.  M = 6: copies
// of the five bits five apart do not overlap, so one multiplication puts bit j
// of copy j at 6 j; otherwise the bits are moved apart in halving groups.
template <int M>
__device__ __forceinline__ uint32_t spread(uint32_t x) {
    if (M == 6) return (x * 0x00108421u) & 0x01041041u;
    if (M == 3) {
        x = (x | (x << 16)) & 0x030000FFu;
        x = (x | (x << 8)) & 0x0300F00Fu;
        x = (x | (x << 4)) & 0x030C30C3u;
        return (x | (x << 2)) & 0x09249249u;
    }
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}

// Morton interleave, most significant level first, coordinates in order: the
// bits of all coordinates 30 key bits at a time.  (One key bit at a time took 51
// us for 4M 48-bit TwoPoint keys.)
template <typename K, int M>
__device__ __forceinline__ K interleave(const uint32_t (&q)[M], uint32_t b) {
    constexpr uint32_t GROUP = M == 6 ? 5 : 10;  // bits of a coordinate per group
    K key = 0;
#pragma unroll
    for (uint32_t g = 0; g < (sizeof(K) == 8 ? 3u : 1u); ++g) {
        if (g * GROUP >= b) break;
        uint32_t part = 0;
#pragma unroll
        for (int c = 0; c < M; ++c) part |= spread<M>((q[c] >> (g * GROUP)) & ((1u << GROUP) - 1u)) << (M - 1 - c);
        key |= (K)part << (g * GROUP * M);
    }
    return key;
}

// TwoPoint: o and t = o + L d (one fused multiply-add per axis) normalised
// to the scene box, quantised to b bits, Morton-interleaved most significant
// level first in the order o.x o.y o.z t.x t.y t.z, left-justified in k bits.
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_twopoint(const float4 *__restrict__ org,
                                                               const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                               float lox, float loy, float loz, float ex, float ey,
                                                               float ez, float L, uint32_t key_bits,
                                                               K *__restrict__ keys) {
    const uint32_t b = key_bits / 6, pad = key_bits - 6 * b;
    wait_for_previous();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float4 o = __ldcs(org + i * rs);
        const float4 d = __ldcs(dir + i * rs);
        const float p[6] = {o.x, o.y, o.z, __fmaf_rn(L, d.x, o.x), __fmaf_rn(L, d.y, o.y), __fmaf_rn(L, d.z, o.z)};
        const float lo[3] = {lox, loy, loz}, ext[3] = {ex, ey, ez};
        uint32_t q[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) q[c] = quantise(p[c], lo[c % 3], ext[c % 3], b);
        K key = interleave<K, 6>(q, b);
        if (pad) key <<= pad;
        __stcs(keys + i, key);
    }
}

// Octahedral map of a direction: L1-normalise, fold the lower hemisphere
// (z < 0) over the diagonals, map [-1, 1]^2 to [0, 1]^2; zero -> centre.
__device__ __forceinline__ void octahedral(const float4 &d, float &u, float &v) {
    u = 0.5f;
    v = 0.5f;
    const float s = __fadd_rn(__fadd_rn(fabsf(d.x), fabsf(d.y)), fabsf(d.z));
    if (s > 0.0f) {
        const float nx = __fdiv_rn(d.x, s), ny = __fdiv_rn(d.y, s), nz = __fdiv_rn(d.z, s);
        float x = nx, y = ny;
        if (nz < 0.0f) {
            x = __fmul_rn(__fsub_rn(1.0f, fabsf(ny)), nx >= 0.0f ? 1.0f : -1.0f);
            y = __fmul_rn(__fsub_rn(1.0f, fabsf(nx)), ny >= 0.0f ? 1.0f : -1.0f);
        }
        u = __fadd_rn(__fmul_rn(x, 0.5f), 0.5f);
        v = __fadd_rn(__fmul_rn(y, 0.5f), 0.5f);
    }
}

// Origin key: 3D Morton code of the origin, floor(k/3) bits per axis,
// left-justified in k bits.
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_origin(const float4 *__restrict__ org, uint64_t n, uint32_t rs, float lox,
                                                             float loy, float loz, float ex, float ey, float ez,
                                                             uint32_t key_bits, K *__restrict__ keys) {
    const uint32_t b = key_bits / 3, pad = key_bits - 3 * b;
    wait_for_previous();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float4 o = __ldcs(org + i * rs);
        const uint32_t q[3] = {quantise(o.x, lox, ex, b), quantise(o.y, loy, ey, b), quantise(o.z, loz, ez, b)};
        K key = interleave<K, 3>(q, b);
        if (pad) key <<= pad;
        __stcs(keys + i, key);
    }
}

// Origin-Direction key: origin Morton code (bo bits per axis) above a Morton
// code of the octahedral map of the direction (bd bits per coordinate),
// bd = floor(k/6), bo = floor((k - 2 bd)/3), left-justified in k bits.
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_origin_dir(const float4 *__restrict__ org,
                                                                 const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                                 float lox, float loy, float loz, float ex,
                                                                 float ey, float ez, uint32_t key_bits,
                                                                 K *__restrict__ keys) {
    const uint32_t bd = key_bits / 6, bo = (key_bits - 2 * bd) / 3;
    const uint32_t pad = key_bits - (3 * bo + 2 * bd);
    wait_for_previous();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float4 o = __ldcs(org + i * rs);
        const float4 d = __ldcs(dir + i * rs);
        float u, v;
        octahedral(d, u, v);
        const uint32_t qo[3] = {quantise(o.x, lox, ex, bo), quantise(o.y, loy, ey, bo), quantise(o.z, loz, ez, bo)};
        const uint32_t qd[2] = {quantise(u, 0.0f, 1.0f, bd), quantise(v, 0.0f, 1.0f, bd)};
        K key = (interleave<K, 3>(qo, bo) << (2 * bd)) | interleave<K, 2>(qd, bd);
        if (pad) key <<= pad;
        __stcs(keys + i, key);
    }
}

// Key statistics over keys in sorted order (keys[perm[j]] ascending):
// cnt[0] += changes of key between consecutive positions, cnt[1] += changes
// inside groups of 32 consecutive positions.
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_key_stats(const K *__restrict__ keys, const uint32_t *__restrict__ perm,
                                                         uint64_t n, K mask, unsigned long long *cnt) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    unsigned long long all = 0, inner = 0;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x + 1; j < n; j += stride) {
        const uint32_t a = perm[j - 1], b = perm[j];
        if (a < n && b < n && ((keys[a] & mask) != (keys[b] & mask))) {
            ++all;
            if (j % 32 != 0) ++inner;
        }
    }
    if (all) atomicAdd(cnt, all);
    if (inner) atomicAdd(cnt + 1, inner);
}

// TwoPoint / Origin / Origin-Direction keys of one ray (the formulas of the
// single-scene kernels above, as functions of the scene box).
template <typename K>
__device__ __forceinline__ K twopoint_key(const float4 &o, const float4 &d, const SceneDesc &sc, uint32_t key_bits) {
    const uint32_t b = key_bits / 6, pad = key_bits - 6 * b;
    const float p[6] = {o.x, o.y, o.z, __fmaf_rn(sc.L, d.x, o.x), __fmaf_rn(sc.L, d.y, o.y),
                        __fmaf_rn(sc.L, d.z, o.z)};
    uint32_t q[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) q[c] = quantise(p[c], sc.lo[c % 3], sc.ext[c % 3], b);
    K key = interleave<K, 6>(q, b);
    return pad ? (K)(key << pad) : key;
}

template <typename K>
__device__ __forceinline__ K origin_key(const float4 &o, const SceneDesc &sc, uint32_t key_bits) {
    const uint32_t b = key_bits / 3, pad = key_bits - 3 * b;
    const uint32_t q[3] = {quantise(o.x, sc.lo[0], sc.ext[0], b), quantise(o.y, sc.lo[1], sc.ext[1], b),
                           quantise(o.z, sc.lo[2], sc.ext[2], b)};
    K key = interleave<K, 3>(q, b);
    return pad ? (K)(key << pad) : key;
}

template <typename K>
__device__ __forceinline__ K origin_dir_key(const float4 &o, const float4 &d, const SceneDesc &sc, uint32_t key_bits) {
    const uint32_t bd = key_bits / 6, bo = (key_bits - 2 * bd) / 3, pad = key_bits - (3 * bo + 2 * bd);
    float u, v;
    octahedral(d, u, v);
    const uint32_t qo[3] = {quantise(o.x, sc.lo[0], sc.ext[0], bo), quantise(o.y, sc.lo[1], sc.ext[1], bo),
                            quantise(o.z, sc.lo[2], sc.ext[2], bo)};
    const uint32_t qd[2] = {quantise(u, 0.0f, 1.0f, bd), quantise(v, 0.0f, 1.0f, bd)};
    K key = (interleave<K, 3>(qo, bo) << (2 * bd)) | interleave<K, 2>(qd, bd);
    return pad ? (K)(key << pad) : key;
}

// Batch of wavefronts: one launch encodes the rays of every scene against
// that scene's box; the scene index sits above the key so that one sort groups
// rays by scene, then by key.
template <typename K, int METHOD>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_multi(const float4 *__restrict__ org,
                                                            const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                            const SceneDesc *__restrict__ scenes,
                                                            const uint64_t *__restrict__ offsets, uint32_t num_scenes,
                                                            uint32_t key_bits, K *__restrict__ keys) {
    wait_for_previous();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const uint32_t s = scene_of(offsets, num_scenes, i);
        const SceneDesc &sc = scenes[s];
        const float4 o = __ldcs(org + i * rs);
        const float4 d = __ldcs(dir + i * rs);
        K key;
        if (METHOD == HCC_METHOD_TWOPOINT)
            key = twopoint_key<K>(o, d, sc, key_bits);
        else if (METHOD == HCC_METHOD_ORIGIN)
            key = origin_key<K>(o, sc, key_bits);
        else
            key = origin_dir_key<K>(o, d, sc, key_bits);
        if (key_bits < 8 * sizeof(K)) key |= (K)s << key_bits;
        __stcs(keys + i, key);
    }
}

// The same for HCC keys: a block takes a run of consecutive rays and stages the
// cut of each scene that the run touches (nearly always one), then encodes as
// k_encode_hcc does.  (Reading the boxes from each ray's own scene and ordering
// their bounds per ray took 83 us for 2.6M rays of six scenes and 24-bit keys.)
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_multi_hcc(const float4 *__restrict__ org,
                                                                const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                                const SceneDesc *__restrict__ scenes,
                                                                const uint64_t *__restrict__ offsets,
                                                                uint32_t num_scenes, uint32_t key_bits,
                                                                K *__restrict__ keys) {
    __shared__ float2 s_boxes[MAX_CUT_BITS * BOX];
    wait_for_previous();
    const uint64_t run = (n + gridDim.x - 1) / gridDim.x;
    uint64_t i0 = run * blockIdx.x;
    const uint64_t end = i0 + run < n ? i0 + run : n;
    if (i0 >= end) return;
    for (uint32_t s = scene_of(offsets, num_scenes, i0); i0 < end; ++s) {  // scene s owns ray i0, or is empty
        const uint64_t i1 = offsets[s + 1] < end ? offsets[s + 1] : end;
        if (i1 <= i0) continue;
        const uint32_t used = min(scenes[s].used, min(key_bits, MAX_CUT_BITS));
        __syncthreads();  // the previous scene's boxes are no longer read
        const bool ordered = __syncthreads_and(stage_boxes(s_boxes, scenes[s].cut, used));
        for (uint64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            const SlabRay r = slab_ray(__ldcs(org + i * rs), __ldcs(dir + i * rs), ordered);
            K key = hcc_key<K>(r, s_boxes, used, key_bits);
            if (key_bits < 8 * sizeof(K)) key |= (K)s << key_bits;
            __stcs(keys + i, key);
        }
        i0 = i1;
    }
}

}  // namespace

cudaError_t launch_encode_multi(cudaStream_t s, int method, const float4 *org, const float4 *dir, uint64_t n, uint32_t rs,
                                const SceneDesc *scenes, const uint64_t *offsets, uint32_t num_scenes,
                                uint32_t key_bits, uint32_t total_bits, void *keys) {
    if (n == 0) return cudaSuccess;
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
#define HCC_ENC_MULTI(K, KERNEL)                                                                                    \
    return launch_early(KERNEL, grid, ENC_BLOCK, 0, s, org, dir, n, rs, scenes, offsets, num_scenes, key_bits, (K *)keys)
#define HCC_ENC_MULTI_K(K)                                            \
    do {                                                              \
        if (method == HCC_METHOD_HCC)                                 \
            HCC_ENC_MULTI(K, k_encode_multi_hcc<K>);                  \
        else if (method == HCC_METHOD_TWOPOINT)                       \
            HCC_ENC_MULTI(K, (k_encode_multi<K, HCC_METHOD_TWOPOINT>)); \
        else if (method == HCC_METHOD_ORIGIN)                         \
            HCC_ENC_MULTI(K, (k_encode_multi<K, HCC_METHOD_ORIGIN>)); \
        else                                                          \
            HCC_ENC_MULTI(K, (k_encode_multi<K, HCC_METHOD_ORIGIN_DIR>)); \
    } while (0)
    if (total_bits <= 32)
        HCC_ENC_MULTI_K(uint32_t);
    else
        HCC_ENC_MULTI_K(uint64_t);
#undef HCC_ENC_MULTI_K
#undef HCC_ENC_MULTI
}

cudaError_t launch_key_stats(cudaStream_t s, const void *keys, uint32_t key_bits, const uint32_t *perm, uint64_t n,
                             unsigned long long *cnt) {
    if (n < 2) return cudaSuccess;
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32) {
        const uint32_t mask = key_bits == 32 ? 0xFFFFFFFFu : ((1u << key_bits) - 1u);
        k_key_stats<uint32_t><<<grid, ENC_BLOCK, 0, s>>>((const uint32_t *)keys, perm, n, mask, cnt);
    } else {
        const uint64_t mask = key_bits == 64 ? ~0ull : ((1ull << key_bits) - 1ull);
        k_key_stats<uint64_t><<<grid, ENC_BLOCK, 0, s>>>((const uint64_t *)keys, perm, n, mask, cnt);
    }
    return cudaGetLastError();
}

cudaError_t launch_encode_origin(cudaStream_t s, const float4 *org, uint64_t n, uint32_t rs, const float lo[3], const float ext[3],
                                 uint32_t key_bits, void *keys) {
    if (n == 0) return cudaSuccess;
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32)
        return launch_early(k_encode_origin<uint32_t>, grid, ENC_BLOCK, 0, s, org, n, rs, lo[0], lo[1], lo[2], ext[0],
                            ext[1], ext[2], key_bits, (uint32_t *)keys);
    return launch_early(k_encode_origin<uint64_t>, grid, ENC_BLOCK, 0, s, org, n, rs, lo[0], lo[1], lo[2], ext[0],
                        ext[1], ext[2], key_bits, (uint64_t *)keys);
}

cudaError_t launch_encode_origin_dir(cudaStream_t s, const float4 *org, const float4 *dir, uint64_t n, uint32_t rs,
                                     const float lo[3], const float ext[3], uint32_t key_bits, void *keys) {
    if (n == 0) return cudaSuccess;
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32)
        return launch_early(k_encode_origin_dir<uint32_t>, grid, ENC_BLOCK, 0, s, org, dir, n, rs, lo[0], lo[1], lo[2],
                            ext[0], ext[1], ext[2], key_bits, (uint32_t *)keys);
    return launch_early(k_encode_origin_dir<uint64_t>, grid, ENC_BLOCK, 0, s, org, dir, n, rs, lo[0], lo[1], lo[2],
                        ext[0], ext[1], ext[2], key_bits, (uint64_t *)keys);
}

namespace {

// Multi-level HCC (Sec. 4.3): the top field as in Algorithm 1; the first met
// top node (HAD order) is the representative, and its low-level cut fills the
// next low_field bits.  All boxes of both levels are staged in shared memory:
// top boxes first, then the low boxes row by row, the rows an odd number of
// entries apart: lanes read the rows of their own representatives, which would
// otherwise lie in the same banks.
__host__ __device__ constexpr uint32_t ml_row(uint32_t low_field) { return BOX * low_field + 1; }

template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_mlhcc(const float4 *__restrict__ org,
                                                            const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                            const float4 *__restrict__ top, uint32_t ntop,
                                                            uint32_t top_field, const float4 *__restrict__ low,
                                                            uint32_t low_field, uint32_t key_bits,
                                                            K *__restrict__ keys) {
    extern __shared__ float2 s_ml[];
    const uint32_t row_len = ml_row(low_field);
    bool ordered = true;
    for (uint32_t q = threadIdx.x; q < ntop + ntop * low_field; q += blockDim.x) {
        const uint32_t row = q < ntop ? 0 : (q - ntop) / low_field;
        float2 *b = q < ntop ? s_ml + BOX * q : s_ml + BOX * ntop + row * row_len + BOX * (q - ntop - row * low_field);
        ordered = stage_box(b, q < ntop ? top + 2 * q : low + 2 * (q - ntop)) && ordered;
    }
    ordered = __syncthreads_and(ordered);
    wait_for_previous();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const SlabRay r = slab_ray(__ldcs(org + i * rs), __ldcs(dir + i * rs), ordered);
        // top bits first (node t at bit ntop - 1 - t), then the low row of
        // the first met top node (the highest set bit)
        const uint64_t tb = met_boxes<uint64_t>(r, s_ml, ntop);
        K key = ntop ? (K)(tb << (key_bits - ntop)) : (K)0;
        if (tb) {
            const uint32_t rep = ntop - 64u + (uint32_t)__clzll((long long)tb);
            const uint64_t lb = met_boxes<uint64_t>(r, s_ml + BOX * ntop + rep * row_len, low_field);
            if (low_field) key |= (K)(lb << (key_bits - top_field - low_field));
        }
        __stcs(keys + i, key);
    }
}

// Prefix path code (Sec. 4.1): a depth-first, left-child-first walk that
// every ray takes in the same order; each visited node's box test is one key
// bit, a met internal node is entered, a missed subtree skipped, and the walk
// stops after key_bits tests.  The children's exact boxes come from the
// parent's 64-byte node; a parent whose right child is still due waits on a
// stack of node indices (each entry follows a test, so key_bits entries
// suffice).
template <typename K>
__global__ void __launch_bounds__(ENC_BLOCK) k_encode_ppc(const float4 *__restrict__ org,
                                                          const float4 *__restrict__ dir, uint64_t n, uint32_t rs,
                                                          const float4 *__restrict__ nodes, uint32_t root_ref,
                                                          float4 root_lo, float4 root_hi, uint32_t key_bits,
                                                          K *__restrict__ keys) {
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float4 o = __ldcs(org + i * rs);
        const float4 d = __ldcs(dir + i * rs);
        const float ix = __frcp_rn(d.x), iy = __frcp_rn(d.y), iz = __frcp_rn(d.z);
        K key = 0;
        uint32_t m = 0;  // tests made
        const bool root_met = meets(o, d, ix, iy, iz, root_lo, root_hi);
        if (root_met) key |= (K)1 << (key_bits - 1);
        m = 1;
        uint32_t stack[64];
        uint32_t sp = 0;
        uint32_t cur = root_ref;
        bool right = false;  // which child of cur is visited next
        bool go = root_met && !(root_ref & REF_LEAF);
        while (go && m < key_bits) {
            const float4 *f = nodes + 4 * (size_t)cur;
            const float4 n0 = __ldg(f), n1 = __ldg(f + 1), n2 = __ldg(f + 2);
            const uint4 n3 = __ldg(reinterpret_cast<const uint4 *>(f + 3));
            float4 lo, hi;
            uint32_t child;
            if (!right) {  // exact node: per child (lo.x, lo.y), (hi.x, hi.y), (lo.z, hi.z)
                lo = make_float4(n0.x, n0.y, n1.x, 0.f);
                hi = make_float4(n0.z, n0.w, n1.y, 0.f);
                child = n3.x;
                stack[sp++] = cur;  // its right child follows the left subtree
            } else {
                lo = make_float4(n1.z, n1.w, n2.z, 0.f);
                hi = make_float4(n2.x, n2.y, n2.w, 0.f);
                child = n3.y;
            }
            const bool met = meets(o, d, ix, iy, iz, lo, hi);
            if (met) key |= (K)1 << (key_bits - 1 - m);
            ++m;
            if (met && !(child & REF_LEAF)) {
                cur = child;
                right = false;
            } else if (sp > 0) {
                cur = stack[--sp];
                right = true;
            } else {
                go = false;
            }
        }
        __stcs(keys + i, key);
    }
}

}  // namespace

cudaError_t launch_encode_mlhcc(cudaStream_t s, const float4 *org, const float4 *dir, uint64_t n, uint32_t rs,
                                const float4 *top, uint32_t ntop, uint32_t top_field, const float4 *low,
                                uint32_t low_field, uint32_t key_bits, void *keys) {
    if (n == 0) return cudaSuccess;
    if (ntop > top_field || top_field + low_field > MAX_CUT_BITS || top_field + low_field > key_bits)
        return cudaErrorInvalidValue;
    // at most 33 rows of 31 boxes: 50,952 bytes
    const size_t smem = sizeof(float2) * ntop * ((size_t)BOX + ml_row(low_field));
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32) {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(k_encode_mlhcc<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return launch_early(k_encode_mlhcc<uint32_t>, grid, ENC_BLOCK, smem, s, org, dir, n, rs, top, ntop, top_field, low,
                            low_field, key_bits, (uint32_t *)keys);
    }
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_encode_mlhcc<uint64_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return launch_early(k_encode_mlhcc<uint64_t>, grid, ENC_BLOCK, smem, s, org, dir, n, rs, top, ntop, top_field, low,
                        low_field, key_bits, (uint64_t *)keys);
}

cudaError_t launch_encode_ppc(cudaStream_t s, const float4 *org, const float4 *dir, uint64_t n, uint32_t rs, const uint4 *nodes,
                              uint32_t root_ref, const float root_lo[3], const float root_hi[3], uint32_t key_bits,
                              void *keys) {
    if (n == 0) return cudaSuccess;
    if (key_bits < 1 || key_bits > MAX_CUT_BITS) return cudaErrorInvalidValue;
    const float4 lo = make_float4(root_lo[0], root_lo[1], root_lo[2], 0.f);
    const float4 hi = make_float4(root_hi[0], root_hi[1], root_hi[2], 0.f);
    const float4 *f = reinterpret_cast<const float4 *>(nodes);
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32)
        k_encode_ppc<uint32_t><<<grid, ENC_BLOCK, 0, s>>>(org, dir, n, rs, f, root_ref, lo, hi, key_bits,
                                                          (uint32_t *)keys);
    else
        k_encode_ppc<uint64_t><<<grid, ENC_BLOCK, 0, s>>>(org, dir, n, rs, f, root_ref, lo, hi, key_bits,
                                                          (uint64_t *)keys);
    return cudaGetLastError();
}

cudaError_t launch_encode_hcc(cudaStream_t s, const float4 *org, const float4 *dir, uint64_t n, uint32_t rs,
                              const float4 *cut_boxes, uint32_t used, uint32_t key_bits, void *keys) {
    if (n == 0) return cudaSuccess;
    if (used > MAX_CUT_BITS) used = MAX_CUT_BITS;
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32)
        return launch_early(k_encode_hcc<uint32_t>, grid, ENC_BLOCK, 0, s, org, dir, n, rs, cut_boxes, used, key_bits,
                            (uint32_t *)keys);
    return launch_early(k_encode_hcc<uint64_t>, grid, ENC_BLOCK, 0, s, org, dir, n, rs, cut_boxes, used, key_bits,
                        (uint64_t *)keys);
}

cudaError_t launch_encode_twopoint(cudaStream_t s, const float4 *org, const float4 *dir, uint64_t n, uint32_t rs,
                                   const float lo[3], const float ext[3], float L, uint32_t key_bits, void *keys) {
    if (n == 0) return cudaSuccess;
    const int grid = encode_grid(n, ENC_BLOCK, ENC_BLOCKS);
    if (key_bits <= 32)
        return launch_early(k_encode_twopoint<uint32_t>, grid, ENC_BLOCK, 0, s, org, dir, n, rs, lo[0], lo[1], lo[2],
                            ext[0], ext[1], ext[2], L, key_bits, (uint32_t *)keys);
    return launch_early(k_encode_twopoint<uint64_t>, grid, ENC_BLOCK, 0, s, org, dir, n, rs, lo[0], lo[1], lo[2],
                        ext[0], ext[1], ext[2], L, key_bits, (uint64_t *)keys);
}

}  // namespace hcc
