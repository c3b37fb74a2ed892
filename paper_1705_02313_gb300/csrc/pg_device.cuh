// Device helpers shared by the valuation translation units (pg_iter.cu,
// pg_deep.cu): launch shapes, warp and block reductions, the compact
// nearest-greater word, the software grid barrier of the cooperative kernels.
#pragma once

#include "pg_internal.cuh"

namespace pg {
namespace {

constexpr unsigned kFull = 0xffffffffu;

inline unsigned ilp_grid(int64_t n) {
    int64_t tiles = (n + 32 * 4 - 1) / (32 * 4);
    int64_t b = (tiles + kBlock / 32 - 1) / (kBlock / 32);
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 64));
}

inline unsigned grid_for(int64_t n) {
    int64_t b = (n + kBlock - 1) / kBlock;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 64));
}

// All 32 lanes must call this (uniform control flow).
__device__ inline int32_t warp_append(bool pred, int32_t* counter) {
    unsigned m = __ballot_sync(kFull, pred);
    if (!m) return -1;
    int lane = threadIdx.x & 31;
    int leader = __ffs(m) - 1;
    int32_t base = 0;
    if (lane == leader) base = atomicAdd(counter, __popc(m));
    base = __shfl_sync(kFull, base, leader);
    return pred ? base + __popc(m & ((1u << lane) - 1u)) : -1;
}

__device__ inline void block_add(int32_t v, int32_t* counter) {
    __shared__ int32_t acc;
    if (threadIdx.x == 0) acc = 0;
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&acc, v);
    __syncthreads();
    if (threadIdx.x == 0 && acc) atomicAdd(counter, acc);
}

__device__ inline uint64_t ld_cg(const uint64_t* p) { return __ldcg((const unsigned long long*)p); }
__device__ inline void st_cg(uint64_t* p, uint64_t v) { __stcg((unsigned long long*)p, (unsigned long long)v); }

// Compact g-word read by every chain pass: bit 31 = "none" (v is above its
// whole infinite future; the low bits then name the cycle maximum), bit 30 =
// g(v) is the game's sink, low 30 bits = g(v) (ids < 2^30).
constexpr uint32_t kG32None = 0x80000000u;
constexpr uint32_t kG32Sink = 0x40000000u;
__device__ inline uint32_t g32_of(uint64_t w) {
    return (gd_none(w) ? kG32None : 0u) | (gd_sink(w) ? kG32Sink : 0u) | (uint32_t)gd_ptr(w);
}
__device__ inline bool g32_none(uint32_t w) { return (w & kG32None) != 0; }
__device__ inline bool g32_sink(uint32_t w) { return (w & kG32Sink) != 0; }
__device__ inline int32_t g32_ptr(uint32_t w) { return (int32_t)(w & 0x3fffffffu); }

// Words of the iterations that compare valuations (k_walk_cmp, k_jump32_coop,
// k_inc). A word with both the none and the sink
// bit set is pending: its low bits are a jump pointer (every vertex strictly
// between v and it on the play is below v, and so is the pointer). A word
// with only the sink bit (g(v) is the game's sink slot, which the word does
// not repeat) carries v's priority parity in bit 0, so that the vertex that
// ends a chain gives its top's parity with no further read.
constexpr uint32_t kG32Pend = kG32None | kG32Sink;
__device__ inline bool g32_pending(uint32_t w) { return (w & kG32Pend) == kG32Pend; }
__device__ inline uint32_t g32_sink_word(uint8_t fl) { return kG32Sink | ((fl & kPriOdd) ? 1u : 0u); }

// After k_classify, bit 31 of a g-word marks a TOP vertex (its play ends in
// a cycle); finite words are unchanged (bit 30: g(v) is the game's sink slot).
constexpr uint32_t kG32Top = 0x80000000u;
// k_classify also writes one "top word" per vertex: bit 31 = TOP; for a finite
// vertex bits 0..29 = its top, the last vertex of its g-chain below the sink
// slot (a child of the sink in the g-forest), and bit 30 = that top's priority
// is odd.
constexpr uint32_t kTopOdd = 0x40000000u;
__device__ inline int32_t top_id(uint32_t t) { return (int32_t)(t & 0x3fffffffu); }

template <bool CG>
__device__ inline uint32_t ld_word(const uint32_t* p) {
    return CG ? __ldcg(p) : *p;
}

// Compares the valuations of two finite vertices u and w of one game with the
// same top: walk both g-chains (words wu, ww) upwards, always advancing the
// smaller id, until they meet (at the top at the latest). The larger of the
// last two vertices passed below the meeting point is the largest vertex of
// the symmetric difference of the two plays; its side is better for Even
// when its priority is even. Returns > 0 if Val(u) is better for Even, < 0 if
// worse, 0 if u == w. g(x) > x for every vertex below the top, so each step
// raises a or b. CG: the words change during the kernel (k_inc) and are read
// from L2.
template <bool CG = false>
__device__ inline int cmp_walk(int32_t u, int32_t w, const uint32_t* __restrict__ gd32,
                               const uint8_t* __restrict__ flags) {
    int32_t a = u, b = w, pa = -1, pb = -1;
    uint32_t wa = 0, wb = 0;
    if (a != b) {
        wa = ld_word<CG>(gd32 + a);
        wb = ld_word<CG>(gd32 + b);
    }
    while (a != b) {
        if (a < b) {
            pa = a;
            a = g32_ptr(wa);
            if (a <= pa) return 0;  // g-chains rise (a guard that keeps every walk finite; never taken)
            wa = ld_word<CG>(gd32 + a);
        } else {
            pb = b;
            b = g32_ptr(wb);
            if (b <= pb) return 0;
            wb = ld_word<CG>(gd32 + b);
        }
    }
    if (pa == pb) return 0;  // u == w
    const bool u_side = pa > pb;
    const bool even = !(flags[u_side ? pa : pb] & kPriOdd);
    return u_side == even ? 1 : -1;
}

// Order of the valuations of u and w (vertices of one game, with their top
// words tu, tw): > 0 if Val(u) is better for Even than Val(w), < 0 if worse,
// 0 if equal. TOP is above every finite valuation and equal to TOP. Finite
// plays with different tops differ above everything else at the larger top,
// which decides by its parity; with the same top the chains are walked.
template <bool CG = false>
__device__ inline int cmp_val(int32_t u, uint32_t tu, int32_t w, uint32_t tw, const uint32_t* __restrict__ gd32,
                              const uint8_t* __restrict__ flags) {
    const int xu = (tu & kG32Top) ? 1 : 0, xw = (tw & kG32Top) ? 1 : 0;
    if (xu | xw) return xu - xw;
    const int32_t hu = top_id(tu), hw = top_id(tw);
    if (hu != hw) {
        const bool u_side = hu > hw;
        const bool even = !((u_side ? tu : tw) & kTopOdd);
        return u_side == even ? 1 : -1;
    }
    return cmp_walk<CG>(u, w, gd32, flags);
}

// Against the sink's empty valuation: the top of a finite play is its largest
// vertex, so Val(u) is better for Even exactly when that top is even.
__device__ inline int cmp_sink(uint32_t tu) {
    if (tu & kG32Top) return 1;
    return (tu & kTopOdd) ? -1 : 1;
}

// Count-vector keys (pg_cv.cu): the top key, the level of an id, and the key
// weight of one vertex.
using i128 = __int128;

__device__ inline i128 top_key() { return (i128)(~(unsigned __int128)0 >> 1); }

__device__ inline int level_of(const Levels& L, int32_t v) {
    int l = 0;
#pragma unroll
    for (int i = 1; i < kMaxLevels; ++i) l += (i < L.n && v >= L.start[i]) ? 1 : 0;
    return l;
}

__device__ inline i128 weight_of(const Levels& L, int32_t v) {
    const int l = level_of(L, v);
    const i128 w = (i128)1 << L.shift[l];
    return ((L.odd_mask >> l) & 1u) ? -w : w;
}

// The vertices that a switching pass switched, for k_inc: each warp gathers
// its own in shared memory and appends kSwBuf - 31 or more of them at a time
// (one counter step per switched vertex, or per warp round, would serialise a
// pass that switches millions). Entries beyond cap are only counted.
constexpr int kSwBuf = 128;
__device__ inline void list_flush(const int32_t* buf, int32_t have, int32_t* list, int32_t* counter, int32_t cap) {
    if (!have) return;
    const int lane = threadIdx.x & 31;
    int32_t base = 0;
    if (lane == 0) base = atomicAdd(counter, have);
    base = __shfl_sync(kFull, base, 0);
    for (int32_t j = lane; j < have; j += 32)
        if (base + j < cap) list[base + j] = buf[j];
    __syncwarp();
}

// All 32 lanes call this; have (the entries held) stays uniform over the warp.
__device__ inline void list_push(bool sw, int32_t v, int32_t* buf, int32_t* have, int32_t* list, int32_t* counter,
                                 int32_t cap) {
    const unsigned m = __ballot_sync(kFull, sw);
    if (!m) return;
    if (sw) buf[*have + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = v;
    *have += __popc(m);
    __syncwarp();
    if (*have > kSwBuf - 32) {
        list_flush(buf, *have, list, counter, cap);
        *have = 0;
    }
}

// The sink slot of v's game.
__device__ inline int32_t sink_of(int32_t v, const int32_t* vgame, const int32_t* gsink, int32_t sink0) {
    return vgame ? gsink[vgame[v]] : sink0;
}

// kind[v], written by k_chain1
constexpr uint8_t kKFin = 1;        // finite valuation
constexpr uint8_t kKSinkChild = 2;  // g(v) is the sink
constexpr uint8_t kKOdd = 4;        // odd priority
constexpr uint8_t kKSinkSlot = 8;   // the id is a sink slot

// Software grid barrier for cooperative launches (all blocks co-resident).
// Gives up after a bounded number of spins, records kErrBarrier and returns
// false; the caller then returns.
__device__ bool grid_sync(Counters* c) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        volatile uint32_t* genp = &c->bar_gen;
        uint32_t gen = *genp;
        __threadfence();
        uint32_t arrived = atomicAdd(&c->bar_count, 1u);
        if (arrived == gridDim.x - 1) {
            atomicExch(&c->bar_count, 0u);
            __threadfence();
            atomicAdd(&c->bar_gen, 1u);
        } else {
            int64_t spins = 0;
            while (*genp == gen) {
                if (++spins > (1ll << 24)) {
                    atomicOr(&c->err, kErrBarrier);
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// Exclusive scan of one 64-bit value per thread of a 1024-thread block; *total:
// the block's sum.
__device__ inline uint64_t block_scan_1024(uint64_t v, uint64_t* total) {
    __shared__ uint64_t wsum[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint64_t w = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(kFull, w, o);
            if (lane >= o) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    const uint64_t before = (wid ? wsum[wid - 1] : 0) + x - v;
    *total = wsum[32 - 1];
    __syncthreads();
    return before;
}

// ---------------------------------------------------------------------------
// Pointer-chasing passes give each thread kIlp vertices, v + 32 j for
// j < kIlp within a warp tile of 32 kIlp vertices: per-vertex reads and writes
// stay coalesced for every j, and the walks of one thread issue their gathers
// together, so each thread keeps kIlp loads in flight.
constexpr int kIlp = 4;

__device__ inline int64_t warp_tile_base(int64_t tile) { return tile * 32 * kIlp; }

}  // namespace
}  // namespace pg
