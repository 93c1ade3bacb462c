// Stable LSD radix sort of ray ids by key (Sec. 4.2.3 "Sorting": keys are
// sorted as natural numbers; Sec. 5: the sort orders ray indices).
//
// Design (one pass per 8-bit digit, "onesweep" structure; up to 65,536 32-bit
// or 4,096 64-bit keys k_sort_small does all passes in one launch, in a cluster's or a
// block's shared memory):
//   k_hist   one read of every key builds the digit histograms of all passes
//            (each warp counts its most common digit in a register, the rest
//            with shared-memory atomics); the last block to finish scans them
//            and plans the
//            passes: a pass whose digit is the same for every key is marked
//            inactive (skipping it cannot change a stable result), and the
//            ping-pong buffers are chosen so that the first active pass reads
//            the caller's keys and synthesises ids, and the last one writes
//            only the permutation
//   k_pass   one block per tile of keys: warp-level stable ranking
//            (match.any, or a ballot split when a warp's digits are spread),
//            per-digit tile counts published to a decoupled look-back chain
//            (bounded waits), keys reordered in shared memory and written out
//            in runs of equal digits (coalesced); the last launch writes the
//            identity permutation when no pass is active
// Blocks take their tile from an atomic counter when they start, so a tile
// only ever waits for tiles that are already running.  The passes are launched
// early (launch_early): their launch and first steps overlap the end of the
// previous one (100,000-ray bounce 112 -> 100 us, 0.96M 316 -> 312; letting a
// pass's blocks start as soon as all of the previous one's had gave half of that
// back, as they take room from blocks at work).
#include <algorithm>
#include <atomic>
#include <type_traits>
#include <utility>

#include "hcc_internal.cuh"

namespace hcc {
namespace {

constexpr int RADIX = 256;
constexpr int MAX_PASSES = 8;
constexpr int SORT_BLOCK = 256;  // one thread per digit in the scan / look-back
constexpr int SORT_WARPS = SORT_BLOCK / 32;
// 14 keys per thread (3584-key tiles) and four resident blocks per SM
// measured fastest among 8-16 keys and 3-6 blocks on 16.6M ray keys; up to
// SORT_MID_N keys, where larger tiles leave SMs idle and a pass is one tile's
// latency, 7 (uniform / skewed 32-bit keys, 14 against 7, measured before the passes'
// launches overlapped: 100,000 keys 55 / 47 against 47 / 46 us, 250,000 56 / 54 against
// 55 / 47, 1M 76 / 65 against 84 / 73; with them 35 / 33, 41 / 37 and, at 14, 65 / 55)
constexpr int SORT_ITEMS = 14;
constexpr int SORT_ITEMS_MID = 7;
constexpr uint64_t SORT_MID_N = 450000;
constexpr int SORT_MIN_BLOCKS = 4;
constexpr int WIDE_MIN_BLOCKS = 2;  // passes that carry 64-bit keys (3: 3 % slower at 1M keys, 3 % faster at 16M)
constexpr uint32_t ST_AGG = 1u << 30;  // tile count of this digit available
constexpr uint32_t ST_INC = 2u << 30;  // inclusive prefix of this digit available
constexpr uint32_t ST_VALUE = (1u << 30) - 1u;
constexpr int LOOKBACK = 4;                // predecessors read per look-back round
constexpr int MATCH_MAX_DISTINCT = 16;     // distinct digits per warp item below which match.any ranks
constexpr int HIST_BLOCK = 256;

enum : int { BUF_USER = 0, BUF_A = 1, BUF_B = 2, BUF_PERM = 3 };

// Where a digit pass reads and writes its items: the caller's keys (ids are
// the positions), one of two buffers, or the permutation (ids only).
struct PassPlan {
    int active, src, dst;
    int narrow;  // a wide pass: writes the pairs of the narrow passes
};

// Passes of `passes` over 64-bit keys that carry whole keys: once four digits are left, 32 bits are
// enough.
__host__ __device__ constexpr int wide_passes(int passes) { return passes > 4 ? passes - 4 : 0; }

// Scratch header, followed by the status words [passes][tiles][RADIX] and
// the ping-pong buffers.
struct SortHeader {
    uint32_t hist[MAX_PASSES][RADIX];
    uint32_t start[MAX_PASSES][RADIX];
    PassPlan plan[MAX_PASSES];
    uint32_t tile_counter[MAX_PASSES];
    uint32_t identity;
    uint32_t abort;
    uint32_t hist_done;  // blocks of k_hist that have added their counts
    uint32_t pad[13];
};

// Keys per tile of a sort of n keys.
inline uint32_t tile_keys(uint64_t n) { return SORT_BLOCK * (n <= SORT_MID_N ? SORT_ITEMS_MID : SORT_ITEMS); }

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Layout {
    size_t header, status, pa, pb, va, total;
};

// Buffers between passes: two ping-pong arrays of (key word, id) pairs; the wide
// passes of 64-bit keys keep whole keys there, and their ids in an array of their
// own beside the first and in the permutation beside the second.
Layout layout(uint64_t n, uint32_t key_bits) {
    const uint32_t passes = (key_bits + 7) / 8;
    const uint64_t tiles = (n + tile_keys(n) - 1) / tile_keys(n);
    Layout L;
    L.header = 0;
    L.status = align256(sizeof(SortHeader));
    L.pa = L.status + align256((size_t)passes * tiles * RADIX * sizeof(uint32_t));
    L.pb = L.pa + align256(n * 8);
    L.va = L.pb + align256(n * 8);
    L.total = L.va + (passes > 4 ? align256(n * sizeof(uint32_t)) : 0);
    return L;
}

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t *p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
// Highest set lane of a non-zero mask.
__device__ __forceinline__ int top_lane(uint32_t m) { return 31 - __clz(m); }

// Digit `byte` (0..7) of a key: one byte permute of the key word holding it.
__device__ __forceinline__ uint32_t digit_of(uint32_t k, uint32_t byte) { return __byte_perm(k, 0u, 0x4440u | byte); }
__device__ __forceinline__ uint32_t digit_of(uint64_t k, uint32_t byte) {
    const uint32_t w = byte >= 4 ? (uint32_t)(k >> 32) : (uint32_t)k;
    return __byte_perm(w, 0u, 0x4440u | (byte & 3u));
}

// Lanes of the warp whose digit equals this lane's, found with one ballot per
// digit bit (data-independent cost, unlike match.any whose cost grows with
// the number of distinct values); bits above a short digit are zero in every
// lane and change nothing.  valid_mask: lanes holding a real item.
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, uint32_t valid_mask) {
    uint32_t peers = valid_mask;
#pragma unroll
    for (uint32_t b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, bit);
        peers &= bit ? bal : ~bal;
    }
    return peers;
}

template <typename K>
__device__ __forceinline__ K key_mask(uint32_t key_bits) {
    return key_bits >= 8 * sizeof(K) ? (K)~(K)0 : (K)(((K)1 << key_bits) - 1);
}

// Exclusive scan of each pass's histogram, pass activity and the buffer plan
// (run by one block of RADIX threads, the last k_hist block, while nothing else
// runs: all P scans go together, one barrier for all warps' sums).
template <int P>
__device__ void plan_passes(SortHeader *h, uint64_t n) {
    __shared__ uint32_t s_sum[P][RADIX / 32];
    __shared__ int s_trivial[P];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t c[P], incl[P];
#pragma unroll
    for (int p = 0; p < P; ++p) incl[p] = c[p] = ld_relaxed(&h->hist[p][t]);
    if (t < P) s_trivial[t] = 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl[p], off);
            if (lane >= off) incl[p] += v;
        }
    }
#pragma unroll
    for (int p = 0; p < P; ++p)
        if (lane == 31) s_sum[p][warp] = incl[p];
    __syncthreads();
#pragma unroll
    for (int p = 0; p < P; ++p) {
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += s_sum[p][w];
        h->start[p][t] = before + incl[p] - c[p];
        if ((uint64_t)c[p] == n) s_trivial[p] = 1;
    }
    __syncthreads();
    // thread p plans pass p from the set of active passes
    const uint32_t active = __ballot_sync(0xFFFFFFFFu, lane < P && !s_trivial[lane < P ? lane : 0]);
    if (t < P) {
        const int m = __popc(active), idx = __popc(active & ((1u << t) - 1u));
        // wide passes alternate so that the last one reads the first buffer (its
        // ids are not in the permutation) and writes pairs to the second
        const int lw = __popc(active & ((1u << wide_passes(P)) - 1u)) - 1;  // last active wide pass
        auto target = [&](int i) {  // where active pass i writes
            if (i == m - 1) return (int)BUF_PERM;
            if (i < lw) return (lw - 1 - i) % 2 == 0 ? (int)BUF_A : (int)BUF_B;
            return (i - lw) % 2 == 0 ? (int)BUF_B : (int)BUF_A;
        };
        PassPlan pl;
        pl.active = (active >> t) & 1u;
        pl.src = idx == 0 ? (int)BUF_USER : target(idx - 1);
        pl.dst = target(idx);
        pl.narrow = idx == lw && idx < m - 1;
        h->plan[t] = pl;
        if (t == 0) h->identity = m == 0;
    }
}

// One read of all keys: the digit histograms of every pass.  Keys of ray
// batches are heavily skewed (one digit value often holds most keys), so
// each warp first picks the most common digit of its first 32 keys for each
// pass and counts that value in a register; every other digit goes to a
// shared-memory add (predicated, not branched around).  Threads read 16
// bytes of keys at a time (VEC keys) where the keys are 16-byte aligned; the
// last n % VEC keys are read one at a time.  The block's counts then go to the
// global histograms, and the last block to finish plans the passes.
template <typename K, int P>
__device__ __forceinline__ void hist_key(K k, const uint32_t (&dom)[P], uint32_t (&cnt)[P], uint32_t sh) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const uint32_t d = digit_of(k, (uint32_t)p);
        cnt[p] += d == dom[p] ? 1u : 0u;
        // a predicated shared-memory add for the other digits, no branch
        asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, %1;\n\t@q red.shared.add.u32 [%2], 1;\n\t}" ::"r"(d),
                     "r"(dom[p]), "r"(sh + (uint32_t)(p * RADIX + d) * 4u)
                     : "memory");
    }
}

// P: the number of digit passes (a template argument, so that the per-key
// loop has no pass test).
template <typename K, int VEC, int P>
__global__ void __launch_bounds__(HIST_BLOCK) k_hist(const K *__restrict__ keys, uint64_t n, uint32_t key_bits,
                                                     SortHeader *h) {
    __shared__ uint32_t sh[MAX_PASSES * RADIX];
    __shared__ bool s_last;
    for (int i = threadIdx.x; i < P * RADIX; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    const K mask = key_mask<K>(key_bits);
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t first = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // dominant digit per pass among the warp's first keys
    const K k0 = first < n ? (keys[first] & mask) : (K)0;
    uint32_t dom[P], cnt[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        cnt[p] = 0;
        const uint32_t d = digit_of(k0, (uint32_t)p);
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, first < n ? d : 256u + lane);
        uint32_t best = ((uint32_t)__popc(peers) << 9) | d;
        best = __reduce_max_sync(0xFFFFFFFFu, best);
        dom[p] = best & 511u;
    }
    constexpr int UNROLL = 4;  // independent 16-byte loads in flight per thread
    using V = typename std::conditional<VEC == 1, K, uint4>::type;
    const V *kv = reinterpret_cast<const V *>(keys);
    const uint32_t shb = (uint32_t)__cvta_generic_to_shared(sh);
    const uint64_t nv = n / VEC;  // whole vectors; the last n % VEC keys follow one at a time
    for (uint64_t base = first; base < nv; base += UNROLL * stride) {
        V x[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const uint64_t v = base + (uint64_t)u * stride;
            x[u] = v < nv ? kv[v] : V{};
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            if (base + (uint64_t)u * stride >= nv) break;
            if constexpr (VEC == 1) {
                hist_key<K, P>(x[u] & mask, dom, cnt, shb);
            } else if constexpr (sizeof(K) == 4) {
                hist_key<K, P>((K)x[u].x & mask, dom, cnt, shb);
                hist_key<K, P>((K)x[u].y & mask, dom, cnt, shb);
                hist_key<K, P>((K)x[u].z & mask, dom, cnt, shb);
                hist_key<K, P>((K)x[u].w & mask, dom, cnt, shb);
            } else {
                hist_key<K, P>((((K)x[u].y << 32) | x[u].x) & mask, dom, cnt, shb);
                hist_key<K, P>((((K)x[u].w << 32) | x[u].z) & mask, dom, cnt, shb);
            }
        }
    }
    for (uint64_t i = nv * VEC + first; i < n; i += stride) hist_key<K, P>(keys[i] & mask, dom, cnt, shb);
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, cnt[p]);
        if (lane == 0 && c && dom[p] < 256u) atomicAdd(&sh[p * RADIX + dom[p]], c);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < P * RADIX; i += blockDim.x)
        if (sh[i]) atomicAdd(&h->hist[0][0] + i, sh[i]);
    // the last block to finish plans the passes
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&h->hist_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (s_last) {
        __threadfence();
        plan_passes<P>(h, n);
    }
}

// The histogram kernel for `passes` digit passes (1-4 for 32-bit keys, 5-8
// for 64-bit keys) and the keys' alignment.
template <typename K, int VEC>
void launch_hist(cudaStream_t s, unsigned blocks, const K *keys, uint64_t n, uint32_t key_bits, int passes,
                 SortHeader *h) {
    constexpr int LO = sizeof(K) == 4 ? 1 : 5;
    switch (passes - LO) {
        case 0: k_hist<K, VEC, LO><<<blocks, HIST_BLOCK, 0, s>>>(keys, n, key_bits, h); break;
        case 1: k_hist<K, VEC, LO + 1><<<blocks, HIST_BLOCK, 0, s>>>(keys, n, key_bits, h); break;
        case 2: k_hist<K, VEC, LO + 2><<<blocks, HIST_BLOCK, 0, s>>>(keys, n, key_bits, h); break;
        default: k_hist<K, VEC, LO + 3><<<blocks, HIST_BLOCK, 0, s>>>(keys, n, key_bits, h); break;
    }
}

template <typename K>
struct PassArgs {
    const K *user_keys;
    void *buf_a, *buf_b;  // between passes: (key word, id) pairs, or whole keys ...
    uint32_t *va;         // ... with their ids here (buf_a) or in perm (buf_b)
    uint32_t *perm;
    uint32_t *status;
    SortHeader *h;
    uint64_t n;
    uint32_t key_bits, num_tiles;
    uint32_t *err;
    uint32_t wait_limit;     // status reads a tile may wait in the look-back
    uint32_t withhold_tile;  // test hook: this tile never publishes its counts
    int last_launch;         // the last pass launch writes the identity permutation if no pass is active
};

// Decoupled look-back for digit d of tile `tile`: the sum of the digit's
// counts in all earlier tiles, read from their status words newest first
// (LOOKBACK per round) until an inclusive prefix is found.  Each wait is
// bounded: after wait_limit status reads without progress (or once another
// tile has given up) it records a timeout and returns.
template <typename K>
__device__ __forceinline__ uint32_t look_back(const PassArgs<K> &a, int pass, uint32_t tile, uint32_t d,
                                              bool &timed_out) {
    uint32_t excl = 0;
    int64_t j = (int64_t)tile - 1;
    uint32_t spins = 0;
    bool done = false;
    const uint32_t wait_rounds = a.wait_limit / LOOKBACK;
    const uint32_t *col = a.status + (size_t)pass * a.num_tiles * RADIX + d;
    while (!done) {
        uint32_t sv[LOOKBACK];
#pragma unroll
        for (int w = 0; w < LOOKBACK; ++w) sv[w] = (j - w >= 0) ? ld_relaxed(col + (size_t)(j - w) * RADIX) : ST_INC;
        int used = 0;
        bool stalled = false;
#pragma unroll
        for (int w = 0; w < LOOKBACK; ++w) {
            if (done || stalled) continue;
            const uint32_t flag = sv[w] & ~ST_VALUE;
            if (flag == 0) {
                stalled = true;
                continue;
            }
            if (j - w >= 0) excl += sv[w] & ST_VALUE;
            ++used;
            if (flag == ST_INC) done = true;
        }
        j -= used;
        if (done) break;
        if (stalled) {
            if (++spins > wait_rounds || ((spins & 63u) == 0 && ld_relaxed(&a.h->abort))) {
                timed_out = true;
                atomicOr(a.err, ERR_TIMEOUT);
                atomicExch(&a.h->abort, 1u);
                break;
            }
            __nanosleep(spins < 8 ? 32u * spins : 256u);
        }
    }
    return excl;
}

// Stable rank of this thread's items within their digit in the warp's
// running count: lanes with equal digits found by a ballot split or by match.any,
// the group reads the warp's counter and its highest lane adds the group's size (the
// counters `wh` belong to this warp alone).  FULL: every item of the tile is
// valid.  MATCH: match.any takes over after the first item if that one shows few
// distinct digits: match.any takes about 100 cycles for 32 distinct
// values, the split about 55 instructions whatever they are (so the first item,
// and sorts whose few items do not pay for the choice, are split).
template <bool FULL, bool MATCH, int ITEMS, typename K, typename R>
__device__ __forceinline__ void rank_items(const K (&kreg)[ITEMS], R (&rank)[ITEMS], uint32_t *wh, uint32_t byte,
                                           uint32_t wfirst, uint32_t tile_n) {
    const int lane = threadIdx.x & 31;
    const uint32_t lt = lanemask_lt();
    bool use_match = false;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t d = digit_of(kreg[i], byte);
        uint32_t peers;
        bool valid = true;
        if (FULL) {
            peers = MATCH && use_match ? __match_any_sync(0xFFFFFFFFu, d) : digit_peers(d, 0xFFFFFFFFu);
        } else {
            valid = wfirst + (uint32_t)i * 32 < tile_n;
            const uint32_t vmask = __ballot_sync(0xFFFFFFFFu, valid);
            peers = MATCH && use_match ? (__match_any_sync(0xFFFFFFFFu, valid ? d : 256u + lane) & vmask)
                                       : digit_peers(d, vmask);
        }
        const bool leader = valid && lane == top_lane(peers);
        if (MATCH && i == 0)  // the first item's number of distinct digits picks the method for the rest
            use_match = __popc(__ballot_sync(0xFFFFFFFFu, leader)) <= MATCH_MAX_DISTINCT;
        const uint32_t prior = wh[d];
        __syncwarp();
        if (leader) wh[d] = prior + (uint32_t)__popc(peers);
        __syncwarp();
        rank[i] = (R)(prior + __popc(peers & lt));
    }
}

// One digit pass, one block per tile of SORT_BLOCK x ITEMS keys.  A block takes its tile
// from an atomic counter when it starts, so tiles are worked on in the order
// blocks start and a tile's predecessors are already running when it looks
// back.  Per tile: each thread loads its items (a warp reads 32
// consecutive elements per item), the warp-level stable ranking, the tile's
// digit counts published at once to the decoupled look-back chain, the tile
// reordered by digit in shared memory, the look-back for the global offsets
// (bounded waits with back-off), and runs of equal digits written out
// coalesced.  Items travel between passes as (key word, id) pairs, so an
// element moves with one 8-byte access.  WIDE: the passes of 64-bit keys while
// more than 32 bits are still to be sorted by; they carry keys and ids apart (12
// bytes; 47 us a pass for 4M keys against 33), and the last of them leaves
// pairs of the bits that remain.  (Sorting by the low words first and fetching
// the high words by id moves 8 bytes in every pass, but the random fetch
// costs 45 us at 4M keys and 100 at 8M, more than it saves.)
template <typename K, int ITEMS, bool WIDE>
__global__ void __launch_bounds__(SORT_BLOCK, WIDE ? WIDE_MIN_BLOCKS : SORT_MIN_BLOCKS) k_pass(PassArgs<K> a, int pass) {
    constexpr uint32_t TILE = SORT_BLOCK * ITEMS;
    using Word = typename std::conditional<WIDE, uint64_t, uint32_t>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];     // the tile, reordered:
    uint2 *tp = reinterpret_cast<uint2 *>(smem_raw);              // pairs, and ...
    uint32_t *tvs = reinterpret_cast<uint32_t *>(tp + TILE);       // ... their ids in input order; or
    uint64_t *tk = reinterpret_cast<uint64_t *>(smem_raw);        // keys ...
    uint32_t *tv = reinterpret_cast<uint32_t *>(tk + TILE);        // ... and their ids
    // per-warp digit counts of the tile, then each warp's first reorder slot per digit
    __shared__ uint32_t s_wofs[SORT_WARPS][RADIX];
    __shared__ uint32_t s_gofs[RADIX];  // global position of digit d's run minus its first tile slot
    __shared__ uint32_t s_wsum[SORT_WARPS];
    __shared__ uint32_t s_tile, s_abort;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // before the previous pass is done: its tile, and cleared counts
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) s_wofs[w][tid] = 0;
    if (tid == 0) {
        s_tile = atomicAdd(&a.h->tile_counter[pass], 1u);
        s_abort = 0;
    }
    wait_for_previous();
    const PassPlan pl = a.h->plan[pass];
    if (!pl.active) {
        if (a.last_launch && a.h->identity) {  // no active pass: the permutation is the identity
            const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
            for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride)
                a.perm[i] = (uint32_t)i;
        }
        return;
    }
    // bits sorted by the wide passes, which the pairs no longer hold
    const uint32_t gone = sizeof(K) == 8 ? 8u * (uint32_t)wide_passes((int)(a.key_bits + 7) / 8) : 0u;
    const uint32_t byte = WIDE || sizeof(K) == 4 ? (uint32_t)pass : (uint32_t)pass - gone / 8;
    const bool from_user = pl.src == BUF_USER;
    const K mask = key_mask<K>(a.key_bits);
    const void *in = pl.src == BUF_A ? a.buf_a : a.buf_b;
    void *out = pl.dst == BUF_A ? a.buf_a : (pl.dst == BUF_B ? a.buf_b : nullptr);
    const uint32_t wfirst = (uint32_t)warp * (ITEMS * 32) + lane;  // tile position of this lane's item 0

    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= a.num_tiles) return;  // uniform; the grid has one block per tile, so this never happens
    const uint64_t base = (uint64_t)tile * TILE;
    const uint32_t tile_n = (uint32_t)((a.n - base) < (uint64_t)TILE ? (a.n - base) : TILE);
    const bool full = tile_n == TILE;

    Word kreg[ITEMS];
    uint32_t vreg[ITEMS], rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t pos = wfirst + (uint32_t)i * 32;
        const bool ok = full || pos < tile_n;
        const uint64_t g = base + pos;
        if (from_user) {
            kreg[i] = ok ? (Word)((a.user_keys[g] & mask) >> (WIDE || sizeof(K) == 4 ? 0u : gone)) : (Word)0;
            if (WIDE) vreg[i] = (uint32_t)g;
        } else if (WIDE) {
            kreg[i] = ok ? static_cast<const Word *>(in)[g] : (Word)0;
            vreg[i] = ok ? (pl.src == BUF_A ? a.va : a.perm)[g] : 0u;
        } else {  // the id waits in shared memory, not in a register, until the reorder
            const uint2 e = ok ? static_cast<const uint2 *>(in)[g] : make_uint2(0u, 0u);
            kreg[i] = (Word)e.x;
            if (ok) tvs[pos] = e.y;
        }
    }
    uint32_t *wh = s_wofs[warp];
    if (full)
        rank_items<true, true>(kreg, rank, wh, byte, wfirst, tile_n);
    else
        rank_items<false, true>(kreg, rank, wh, byte, wfirst, tile_n);
    __syncthreads();  // (1) warp counts complete
    // thread tid owns digit tid: warp offsets, tile count, publication
    uint32_t total = 0;  // the counts become each warp's offset within the digit, in place
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) {
        const uint32_t c = s_wofs[w][tid];
        s_wofs[w][tid] = total;
        total += c;
    }
    uint32_t *st = a.status + ((size_t)pass * a.num_tiles + tile) * RADIX;
    const bool publish = tile != a.withhold_tile;
    if (publish) {
        if (tile == 0)
            st_relaxed(st + tid, ST_INC | ((a.h->start[pass][tid] + total) & ST_VALUE));
        else
            st_relaxed(st + tid, ST_AGG | total);
    }
    uint32_t incl = total;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += v;
    }
    if (lane == 31) s_wsum[warp] = incl;
    __syncthreads();  // (2) per-warp sums of the digit totals
    uint32_t local = incl - total;
    for (int w = 0; w < warp; ++w) local += s_wsum[w];
#pragma unroll
    for (int w = 0; w < SORT_WARPS; ++w) s_wofs[w][tid] += local;
    __syncthreads();  // (3) reorder slots ready
    // reorder the tile by digit (stable)
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const uint32_t pos = wfirst + (uint32_t)i * 32;
        if (full || pos < tile_n) {
            const uint32_t o = wh[digit_of(kreg[i], byte)] + rank[i];
            if (WIDE) {
                tk[o] = kreg[i];
                tv[o] = vreg[i];
            } else {
                tp[o] = make_uint2((uint32_t)kreg[i], from_user ? (uint32_t)(base + pos) : tvs[pos]);
            }
        }
    }
    // decoupled look-back for digit tid
    uint32_t excl;
    if (tile == 0) {
        excl = a.h->start[pass][tid];
    } else {
        bool timed_out = false;
        excl = look_back(a, pass, tile, tid, timed_out);
        if (timed_out) s_abort = 1;
        if (publish) st_relaxed(st + tid, ST_INC | ((excl + total) & ST_VALUE));
    }
    s_gofs[tid] = excl - local;
    __syncthreads();  // (4) the tile reordered, global offsets ready
    if (s_abort) return;
    // runs of equal digits to their global positions
    if (WIDE) {
        uint32_t *vout = pl.dst == BUF_A ? a.va : a.perm;
#pragma unroll 4
        for (uint32_t p = tid; p < tile_n; p += SORT_BLOCK) {
            const uint64_t k = tk[p];
            const uint32_t g = s_gofs[digit_of(k, byte)] + p;
            if (pl.narrow) {
                static_cast<uint2 *>(out)[g] = make_uint2((uint32_t)(k >> gone), tv[p]);
            } else {
                if (out) static_cast<uint64_t *>(out)[g] = k;
                vout[g] = tv[p];
            }
        }
    } else if (out) {
#pragma unroll 4
        for (uint32_t p = tid; p < tile_n; p += SORT_BLOCK) {
            const uint2 e = tp[p];
            static_cast<uint2 *>(out)[s_gofs[digit_of(e.x, byte)] + p] = e;
        }
    } else {
#pragma unroll 4
        for (uint32_t p = tid; p < tile_n; p += SORT_BLOCK) {
            const uint2 e = tp[p];
            a.perm[s_gofs[digit_of(e.x, byte)] + p] = e.y;
        }
    }
}

// ------------------------------------------------------------ small sorts
//
// Up to 65,536 32-bit keys in one launch: a cluster of up to sixteen blocks of 1024
// threads holds all (key, id) pairs in its shared memory.  Per digit pass
// every thread takes its items into registers and ranks them within its warp
// (rank_items), the block orders them by digit in shared memory while the
// cluster exchanges the blocks' digit counts, and runs of equal digits go to
// their places, which may lie in another block's shared memory (items stored
// one by one there instead took 1.2 cycles each, more than the rest of a pass).
// The last pass's ids leave in whole lines.  Two cluster barriers a pass
// replace the launches, the look-back and the round trips through L2 of the
// general path, whose launches take 27 us for 32-bit keys at any size below.
// 64-bit keys sort here if they fit one block.
constexpr int SMALL_BLOCK = 1024;
constexpr int SMALL_WARPS = SMALL_BLOCK / 32;
constexpr int SMALL_ITEMS = 4;  // keys per thread (8 on half as many blocks: 47 against 35 us for 65,536 uniform keys)
constexpr uint32_t SMALL_CAP = SMALL_ITEMS * SMALL_BLOCK;  // keys per block
constexpr int SMALL_CLUSTER = 16;  // more than 8 needs a kernel's consent, and a processing cluster that large

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Barrier of all threads of the cluster's blocks in two halves; what was
// written before an arrival, in any block's shared memory, is visible after the wait.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Shared-memory address `a` of this block in block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_address(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// Items of one block: (key, id) pairs for 32-bit keys, keys and ids apart for 64-bit ones.
template <typename K>
struct SmallItems {
    uint64_t key[SMALL_CAP];
    uint32_t id[sizeof(K) == 4 ? 1 : SMALL_CAP];
};

template <typename K>
struct SmallShared {
    SmallItems<K> buf[2];               // the block's positions, written by the whole cluster, and its staged items
    uint32_t wofs[SMALL_WARPS][RADIX];  // per-warp digit counts, then first staged slots
    uint32_t part[4][RADIX];            // digit counts of eight warps each
    uint32_t count[2][RADIX];           // ... and of the block, read by the others (by pass parity)
    uint32_t start[RADIX];              // first staged slot of a digit, then its global position minus that slot
    uint32_t wsum[2][RADIX / 32];
};

// Exclusive prefix sum over the threads tid < RADIX (all of the block call it); wsum: one word per warp.
__device__ __forceinline__ uint32_t digit_scan(uint32_t v, uint32_t *wsum) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
    if (threadIdx.x < RADIX) {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (lane >= (uint32_t)off) incl += u;
        }
        if (lane == 31) wsum[warp] = incl;
    }
    __syncthreads();
    if (threadIdx.x < RADIX)
        for (uint32_t w = 0; w < warp; ++w) incl += wsum[w];
    return incl - v;
}

template <typename K>
__global__ void __launch_bounds__(SMALL_BLOCK, 1) k_sort_small(const K *__restrict__ keys, uint32_t n, uint32_t key_bits,
                                                               uint32_t *__restrict__ perm) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallShared<K> &sh = *reinterpret_cast<SmallShared<K> *>(smem_raw);
    constexpr bool PAIRS = sizeof(K) == 4;
    constexpr int QUARTER = SMALL_WARPS / 4;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank_in = PAIRS ? cluster_rank() : 0u, blocks = PAIRS ? cluster_size() : 1u;
    const uint32_t first = rank_in * SMALL_CAP;  // this block's positions
    const uint32_t tile_n = n > first ? min(n - first, SMALL_CAP) : 0u;
    const uint32_t wfirst = warp * (SMALL_ITEMS * 32) + lane;
    const K mask = key_mask<K>(key_bits);
    const uint32_t d = tid & (RADIX - 1), quarter = tid >> 8;
    wait_for_previous();
    uint32_t cur = 0;  // the buffer that holds the block's positions; a block alone alternates
    for (uint32_t pass = 0; 8 * pass < key_bits; ++pass) {
        K kreg[SMALL_ITEMS];
        uint32_t vreg[SMALL_ITEMS];
        uint16_t rank[SMALL_ITEMS];
#pragma unroll
        for (int w = 0; w < QUARTER; ++w) sh.wofs[quarter * QUARTER + w][d] = 0;
#pragma unroll
        for (int i = 0; i < SMALL_ITEMS; ++i) {
            const uint32_t pos = wfirst + (uint32_t)i * 32;
            const bool ok = pos < tile_n;
            if (pass == 0) {
                kreg[i] = ok ? (K)(keys[first + pos] & mask) : (K)0;
                vreg[i] = first + pos;
            } else {
                const uint64_t e = ok ? sh.buf[cur].key[pos] : 0ull;
                kreg[i] = (K)e;
                vreg[i] = PAIRS ? (uint32_t)(e >> 32) : ok ? sh.buf[cur].id[pos] : 0u;
            }
        }
        __syncthreads();  // counts cleared
        if (warp * (SMALL_ITEMS * 32) < tile_n)  // a warp with items
            rank_items<false, true>(kreg, rank, sh.wofs[warp], pass, wfirst, tile_n);
        __syncthreads();  // warp counts complete
        uint32_t sum = 0;
#pragma unroll
        for (int w = 0; w < QUARTER; ++w) {
            uint32_t &c = sh.wofs[quarter * QUARTER + w][d];
            const uint32_t v = c;
            c = sum;
            sum += v;
        }
        sh.part[quarter][d] = sum;
        __syncthreads();
        uint32_t total = 0;
        if (tid < RADIX) {
            total = sh.part[0][d] + sh.part[1][d] + sh.part[2][d] + sh.part[3][d];
            sh.count[pass & 1][d] = total;
        }
        if (blocks > 1) cluster_arrive();  // this block's counts are written, and its items in registers
        const uint32_t local = digit_scan(total, sh.wsum[0]);
        if (tid < RADIX) sh.start[d] = local;
        __syncthreads();
        uint32_t add = sh.start[d];
        for (uint32_t q = 0; q < quarter; ++q) add += sh.part[q][d];
#pragma unroll
        for (int w = 0; w < QUARTER; ++w) sh.wofs[quarter * QUARTER + w][d] += add;
        __syncthreads();  // staged slots ready
#pragma unroll
        for (int i = 0; i < SMALL_ITEMS; ++i) {
            if (wfirst + (uint32_t)i * 32 < tile_n) {
                const uint32_t slot = sh.wofs[warp][digit_of(kreg[i], pass)] + rank[i];
                sh.buf[cur ^ 1].key[slot] = PAIRS ? (uint64_t)vreg[i] << 32 | (uint32_t)kreg[i] : (uint64_t)kreg[i];
                if (!PAIRS) sh.buf[cur ^ 1].id[slot] = vreg[i];
            }
        }
        if (!PAIRS || blocks == 1) {  // staged is sorted: no exchange, and the next pass reads it there
            cur ^= 1;
            __syncthreads();
            continue;
        }
        if constexpr (PAIRS) {
            const uint32_t in_key = (uint32_t)__cvta_generic_to_shared(sh.buf[0].key);
            cluster_wait();  // every block's counts
            uint32_t all = 0, before = 0;
            if (tid < RADIX) {
                const uint32_t at = (uint32_t)__cvta_generic_to_shared(&sh.count[pass & 1][d]);
                for (uint32_t r = 0; r < blocks; ++r) {
                    uint32_t v;
                    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_address(at, r)) : "memory");
                    all += v;
                    before += r < rank_in ? v : 0u;
                }
            }
            const uint32_t global = digit_scan(all, sh.wsum[1]);
            if (tid < RADIX) sh.start[d] = global + before - local;
            __syncthreads();  // the block's items staged, their global positions ready
#pragma unroll
            for (int i = 0; i < SMALL_ITEMS; ++i) {
                const uint32_t p = tid + (uint32_t)i * SMALL_BLOCK;
                if (p < tile_n) {
                    const uint64_t e = sh.buf[1].key[p];
                    const uint32_t pos = sh.start[digit_of((K)e, pass)] + p;
                    const uint32_t to = pos / SMALL_CAP, slot = pos % SMALL_CAP;
                    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_address(in_key + slot * 8u, to)), "l"(e) : "memory");
                }
            }
            cluster_arrive();
            cluster_wait();  // every item at its place; no block leaves while others may write to it
        }
    }
    for (uint32_t p = tid; p < tile_n; p += SMALL_BLOCK)
        perm[first + p] = PAIRS ? (uint32_t)(sh.buf[cur].key[p] >> 32) : sh.buf[cur].id[p];
}

template <typename K>
cudaLaunchConfig_t small_config(unsigned blocks, cudaStream_t s, cudaLaunchAttribute (&attr)[2]) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(SMALL_BLOCK);
    cfg.dynamicSmemBytes = sizeof(SmallShared<K>);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// Blocks that a cluster of k_sort_small may have on device dev: 16 where the
// device can place such a cluster, else the 8 that every device can; a block alone
// for 64-bit keys (looked up, with the kernel's shared-memory opt-in, once per device).
template <typename K>
cudaError_t small_blocks(int dev, unsigned *blocks) {
    static std::atomic<unsigned> known[64];
    const bool cached = dev >= 0 && dev < 64;
    *blocks = cached ? known[dev].load() : 0u;
    if (*blocks) return cudaSuccess;
    const auto kernel = k_sort_small<K>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallShared<K>));
    if (e != cudaSuccess) return e;
    *blocks = sizeof(K) == 8 ? 1 : 8;
    if (sizeof(K) == 4 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = small_config<K>(SMALL_CLUSTER, nullptr, attr);
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0) *blocks = SMALL_CLUSTER;
    }
    cudaGetLastError();
    if (cached) known[dev].store(*blocks);
    return cudaSuccess;
}

template <typename K>
cudaError_t run_sort(cudaStream_t s, const K *keys, uint32_t key_bits, uint64_t n, uint32_t *perm,
                     unsigned char *scratch, uint32_t *err, const SortOptions &opt) {
    // One launch where 32-bit keys fit a cluster or 64-bit keys a block (measured
    // against the general path, uniform / skewed keys: 4,096 32-bit keys 17 / 13 against
    // 29 / 27 us, 16,384 26 / 21 against 31 / 28, 65,536 32 / 26 against 33 / 31; 4,096
    // 64-bit keys 35 / 26 against 48 / 46, but in a cluster 8,192 55 / 44 against 50 / 44
    // and 65,536 82 / 62 against 61 / 55: eight exchanges cost more than eight
    // launches that overlap).  The withheld-tile test hook is about the general path's tiles.
    int dev = 0;
    cudaGetDevice(&dev);
    if (n <= (sizeof(K) == 4 ? SMALL_CLUSTER * SMALL_CAP : SMALL_CAP) && opt.withhold_tile == SortOptions().withhold_tile) {
        unsigned most = 0, blocks = 1;
        const cudaError_t e = small_blocks<K>(dev, &most);
        if (e != cudaSuccess) return e;
        while (blocks * SMALL_CAP < n) blocks *= 2;
        if (blocks <= most) {
            cudaLaunchAttribute attr[2];
            const cudaLaunchConfig_t cfg = small_config<K>(blocks, s, attr);
            return cudaLaunchKernelEx(&cfg, k_sort_small<K>, keys, (uint32_t)n, key_bits, perm);
        }
    }
    const Layout L = layout(n, key_bits);
    const int passes = (int)((key_bits + 7) / 8);
    // (the test hook counts tiles of the large size)
    const bool mid = n <= SORT_MID_N && opt.withhold_tile == SortOptions().withhold_tile;
    const uint32_t tile = SORT_BLOCK * (mid ? SORT_ITEMS_MID : SORT_ITEMS);
    const uint32_t tiles = (uint32_t)((n + tile - 1) / tile);
    SortHeader *h = reinterpret_cast<SortHeader *>(scratch + L.header);
    cudaError_t e = cudaMemsetAsync(scratch, 0, L.pa, s);  // header + status words
    if (e != cudaSuccess) return e;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    uint64_t hblocks = (n + HIST_BLOCK * 8 - 1) / (HIST_BLOCK * 8);
    const uint64_t hcap = (uint64_t)(sms > 0 ? sms : 1) * 4;
    if (hblocks > hcap) hblocks = hcap;
    if (hblocks == 0) hblocks = 1;
    const size_t dyn = (sizeof(uint2) + sizeof(uint32_t)) * tile;
    const auto pass = mid ? k_pass<K, SORT_ITEMS_MID, false> : k_pass<K, SORT_ITEMS, false>;
    const auto wide = mid ? k_pass<uint64_t, SORT_ITEMS_MID, true> : k_pass<uint64_t, SORT_ITEMS, true>;
    // the shared-memory opt-in is set once per device (so that a sort can be
    // captured in a CUDA graph without any non-stream call)
    static std::atomic<uint64_t> opted{0};
    if (dev >= 0 && dev < 64 && !(opted.load() & (1ull << dev))) {
        constexpr int per_item = (int)(sizeof(uint2) + sizeof(uint32_t)) * SORT_BLOCK;
        const std::pair<const void *, int> all[] = {{(const void *)k_pass<K, SORT_ITEMS, false>, SORT_ITEMS},
                                                    {(const void *)k_pass<K, SORT_ITEMS_MID, false>, SORT_ITEMS_MID},
                                                    {(const void *)k_pass<uint64_t, SORT_ITEMS, true>, SORT_ITEMS},
                                                    {(const void *)k_pass<uint64_t, SORT_ITEMS_MID, true>, SORT_ITEMS_MID}};
        for (const auto &f : all) {
            e = cudaFuncSetAttribute(f.first, cudaFuncAttributeMaxDynamicSharedMemorySize, per_item * f.second);
            if (e != cudaSuccess) return e;
        }
        opted.fetch_or(1ull << dev);
    }
    if ((reinterpret_cast<uintptr_t>(keys) & 15u) == 0)
        launch_hist<K, 16 / sizeof(K)>(s, (unsigned)hblocks, keys, n, key_bits, passes, h);
    else
        launch_hist<K, 1>(s, (unsigned)hblocks, keys, n, key_bits, passes, h);
    PassArgs<K> a;
    a.user_keys = keys;
    a.buf_a = scratch + L.pa;
    a.buf_b = scratch + L.pb;
    a.va = reinterpret_cast<uint32_t *>(scratch + L.va);
    a.perm = perm;
    a.status = reinterpret_cast<uint32_t *>(scratch + L.status);
    a.h = h;
    a.n = n;
    a.key_bits = key_bits;
    a.num_tiles = tiles;
    a.err = err;
    a.wait_limit = opt.wait_limit;
    a.withhold_tile = opt.withhold_tile;
    for (int p = 0; p < passes; ++p) {
        a.last_launch = p == passes - 1;
        if constexpr (sizeof(K) == 8) {
            if (p < wide_passes(passes)) {
                if ((e = launch_early(wide, tiles, SORT_BLOCK, dyn, s, a, p)) != cudaSuccess) return e;
                continue;
            }
        }
        if ((e = launch_early(pass, tiles, SORT_BLOCK, dyn, s, a, p)) != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

}  // namespace

size_t sort_scratch_bytes(uint64_t n, uint32_t key_bits) { return layout(n, key_bits).total; }

// The small tiles of up to SORT_MID_N keys take more status words than the large tiles
// of somewhat more keys (32-bit keys: 8.25 MB at 450,000, 7.73 at 450,001).
size_t sort_scratch_bytes_upto(uint64_t max_n, uint32_t key_bits) {
    return std::max(sort_scratch_bytes(max_n, key_bits), sort_scratch_bytes(std::min(max_n, SORT_MID_N), key_bits));
}

cudaError_t launch_sort(cudaStream_t s, const void *keys, uint32_t key_bits, uint64_t n, uint32_t *perm,
                        void *scratch, uint32_t *err_word, const SortOptions &opt) {
    if (n == 0) return cudaSuccess;
    unsigned char *sc = static_cast<unsigned char *>(scratch);
    if (key_bits <= 32) return run_sort<uint32_t>(s, (const uint32_t *)keys, key_bits, n, perm, sc, err_word, opt);
    return run_sort<uint64_t>(s, (const uint64_t *)keys, key_bits, n, perm, sc, err_word, opt);
}

}  // namespace hcc
