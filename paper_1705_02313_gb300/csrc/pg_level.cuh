// Forests with few roots (single games of more than kSmallIds ids).
//
// k_chain1 and k_chain2 walk every vertex's g-chain, so they cost a chain's length
// per vertex: little on random games, whose forests have a root for every few
// vertices, but 1,620 and 548 us on a play through 10M vertices in random order
// (16 roots, chains of 16 vertices on average). There the walks stop at the first
// vertex whose own walk has ended: it left what the rest of the chain holds in its
// word. Larger ids are nearer to the roots and go first, so on that play a walk
// ends after a step or two, and both passes are bound by their gathers of 32-byte
// sectors, one or two per vertex: 360 and 227 us. Sizes go up the forest without
// levels or barriers (k_lv_sizes, 339 us; sorting by level and one grid barrier per
// level took 993 with the classification, 842 for the ranks).
//
// k_walk counts the roots; these bodies run when there is one for fewer than
// kLvShare ids. Valuations of 10M vertices in random order by plays of 16, 64, 256,
// 1,024 and 4,096 vertices, a root for 6, 15, 46, 148 and 492: by walks 1,311,
// 1,596, 1,866, 2,136 and 2,506 us, by words 1,544, 1,663, 1,730, 1,766 and 1,798.
#pragma once
#include "pg_device.cuh"

namespace pg {
namespace {

constexpr int32_t kLvShare = 32;
constexpr int32_t kLvMaxCut = 1 << 16;  // the chain lengths in the words

// Whether this valuation's forest has few roots.
__device__ inline bool lv_applies(const Counters* c, int32_t n) {
    return c->leveled && (int64_t)c->n_roots * kLvShare < n;
}

// A vertex's word in k_chain1: 0 unknown, else kLvDone and the number of its g-ancestors in bits 32..47, with kLvTop and
// the cycle maximum in the low half above a cycle.
constexpr uint64_t kLvDone = 1ull << 63, kLvTop = 1ull << 62;
__device__ inline int32_t lv_len(uint64_t w) { return (int32_t)((w >> 32) & 0xffff); }

// k_chain1's classification and slots; the sizes follow in k_lv_sizes.
template <int ILP>
__device__ inline void lv_classify(int32_t n, const uint32_t* __restrict__ gd32, const uint8_t* __restrict__ flags,
                                   const int32_t* __restrict__ pri, int32_t* ccnt, int32_t* __restrict__ slot,
                                   uint8_t* __restrict__ kind, uint8_t* __restrict__ cls, int32_t* __restrict__ dom,
                                   int want_dom, uint64_t* word, GameState* gst, Counters* cnt, int32_t deep_cut) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t nfin = 0, nodd = 0;
    for (int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; tile * 32 * ILP < n; tile += nwarps) {
        int32_t v[ILP], x[ILP], len[ILP], cyc[ILP], par[ILP];
        bool act[ILP];
#pragma unroll
        for (int j = 0; j < ILP; ++j) {
            const int64_t i = tile * 32 * ILP + lane + 32 * j;
            v[j] = i < n ? (int32_t)(n - 1 - i) : -1;
            const uint32_t w = v[j] >= 0 ? gd32[v[j]] : kG32Sink;
            x[j] = g32_ptr(w);
            cyc[j] = g32_none(w) ? x[j] : -1;
            act[j] = !g32_none(w) && !g32_sink(w);
            par[j] = act[j] ? x[j] : -1;
            len[j] = act[j] ? 1 : 0;  // the g-ancestors up to x
        }
        for (;;) {
            bool any = false;
            uint64_t wx[ILP];
            uint32_t gx[ILP];
#pragma unroll
            for (int j = 0; j < ILP; ++j) {
                wx[j] = act[j] ? ld_cg(word + x[j]) : 0;
                gx[j] = act[j] ? gd32[x[j]] : 0u;
            }
#pragma unroll
            for (int j = 0; j < ILP; ++j) {
                if (!act[j]) continue;
                if (wx[j] & kLvDone) {
                    if (wx[j] & kLvTop) cyc[j] = (int32_t)(uint32_t)wx[j];
                    len[j] += lv_len(wx[j]);
                    act[j] = false;
                } else if (g32_none(gx[j])) {
                    cyc[j] = g32_ptr(gx[j]);
                    act[j] = false;
                } else if (g32_sink(gx[j])) {
                    act[j] = false;
                } else {
                    x[j] = g32_ptr(gx[j]);
                    ++len[j];
                    act[j] = len[j] <= deep_cut;
                }
                any |= act[j];
            }
            if (!any) break;
        }
#pragma unroll
        for (int j = 0; j < ILP; ++j) {
            const uint8_t f = v[j] >= 0 ? flags[v[j]] : 0;
            const bool sink = (f & kSinkSlot) != 0, cut = len[j] > deep_cut;
            const bool fin = v[j] >= 0 && !sink && cyc[j] < 0 && !cut;
            // children of one parent in a warp take their slots with one addition
            const int32_t p = fin ? par[j] : -1;
            const unsigned peers = __match_any_sync(kFull, p);
            const int lead = __ffs(peers) - 1;
            int32_t at = 0;
            if (p >= 0 && lane == lead) at = atomicAdd(ccnt + p, __popc(peers));
            at = __shfl_sync(peers, at, lead) + __popc(peers & ((1u << lane) - 1));
            if (v[j] < 0) continue;
            slot[v[j]] = p >= 0 ? at : -1;
            int32_t d = -1;
            if (fin) {
                st_cg(word + v[j], kLvDone | (uint64_t)len[j] << 32);
                kind[v[j]] = kKFin | (par[j] < 0 ? kKSinkChild : 0) | ((f & kPriOdd) ? kKOdd : 0);
                cls[v[j]] = kFin;
                ++nfin;
            } else if (sink) {
                kind[v[j]] = kKSinkSlot;
                cls[v[j]] = kFin;
            } else if (cut) {  // the ruling-set path takes over
                cnt->deep = 1;
            } else {
                const bool odd = (flags[cyc[j]] & kPriOdd) != 0;
                st_cg(word + v[j], kLvDone | kLvTop | (uint64_t)len[j] << 32 | (uint32_t)cyc[j]);
                kind[v[j]] = 0;
                cls[v[j]] = odd ? kOddCycle : kTop;
                d = want_dom ? pri[cyc[j]] : -1;
                nodd += odd;
            }
            if (want_dom) dom[v[j]] = d;
        }
    }
    block_add(nfin, &cnt->n_fin);
    block_add(nodd, &cnt->n_odd);
    block_add(nodd, &gst[0].nodd);
}

// Subtree sizes: every leaf adds itself to its parent's word (its children so far in the low half, their sizes above);
// who completes a parent's count goes on up with the parent's size. One atomic per vertex, no order and no barrier.
__global__ void __launch_bounds__(kBlock) k_lv_sizes(int32_t n, const uint32_t* __restrict__ gd32,
                                                     const uint8_t* __restrict__ kind,
                                                     const int32_t* __restrict__ ccnt, int32_t* __restrict__ sz,
                                                     uint64_t* sum, const Counters* cnt) {
    if (cnt->err || cnt->deep || !lv_applies(cnt, n)) return;
    const int lane = threadIdx.x & 31;
    const int64_t T = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i - lane < n; i += T) {
        const uint8_t kd = i < n ? kind[i] : 0;
        const bool leaf = (kd & kKFin) && !(kd & kKSinkChild) && ccnt[i] == 0;
        int32_t p = leaf ? g32_ptr(gd32[i]) : -1;
        const unsigned peers = __match_any_sync(kFull, p);  // a warp's leaves below one parent add once
        if (p < 0 || lane != __ffs(peers) - 1) continue;
        uint32_t s = __popc(peers), c = s;
        for (;;) {
            const uint32_t w = gd32[p];
            const uint32_t all = (uint32_t)ccnt[p];
            const uint64_t old = atomicAdd((unsigned long long*)sum + p, (unsigned long long)s << 32 | c);
            if ((uint32_t)old + c != all) break;
            s += (uint32_t)(old >> 32);
            sz[p] = (int32_t)s;
            if (g32_sink(w)) break;
            p = g32_ptr(w);
            ++s;
            c = 1;
        }
    }
}

// k_chain2's sums; a vertex's word holds the weights on its chain, itself included (high half), kLvKnown and its depth.
constexpr uint32_t kLvKnown = 1u << 31;

template <bool DEPTH, int ILP>
__device__ inline void lv_ranks(int32_t n, const uint32_t* __restrict__ gd32, const uint64_t* __restrict__ gd,
                                const uint8_t* __restrict__ kind, const int32_t* __restrict__ wgt,
                                const int32_t* __restrict__ oddsz, int32_t* __restrict__ key,
                                int32_t* __restrict__ depth, uint64_t* word) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; tile * 32 * ILP < n; tile += nwarps) {
        int32_t v[ILP], x[ILP], acc[ILP], dep[ILP];
        uint8_t kd[ILP];
        bool act[ILP];
#pragma unroll
        for (int j = 0; j < ILP; ++j) {
            const int64_t i = tile * 32 * ILP + lane + 32 * j;
            v[j] = i < n ? (int32_t)(n - 1 - i) : -1;
            kd[j] = v[j] >= 0 ? kind[v[j]] : 0;
            const bool fin = (kd[j] & kKFin) != 0;
            const uint64_t w = fin && DEPTH ? gd[v[j]] : 0;
            const uint32_t w32 = !fin ? kG32Sink : DEPTH ? g32_of(w) : gd32[v[j]];
            acc[j] = fin ? wgt[v[j]] : 0;
            dep[j] = (int32_t)gd_dist(w);
            x[j] = g32_ptr(w32);
            act[j] = !g32_sink(w32);
        }
        for (;;) {
            bool any = false;
            uint64_t wx[ILP], gx[ILP];
            int32_t wg[ILP];
#pragma unroll
            for (int j = 0; j < ILP; ++j) wx[j] = act[j] ? ld_cg(word + x[j]) : 0;
#pragma unroll
            for (int j = 0; j < ILP; ++j) {
                const bool step = act[j] && !(wx[j] & kLvKnown);
                gx[j] = !step ? 0 : DEPTH ? gd[x[j]] : (uint64_t)gd32[x[j]];
                wg[j] = step ? wgt[x[j]] : 0;
            }
#pragma unroll
            for (int j = 0; j < ILP; ++j) {
                if (!act[j]) continue;
                if (wx[j] & kLvKnown) {
                    acc[j] += (int32_t)(wx[j] >> 32);
                    dep[j] += (int32_t)((uint32_t)wx[j] & ~kLvKnown);
                    act[j] = false;
                } else {
                    const uint32_t w32 = DEPTH ? g32_of(gx[j]) : (uint32_t)gx[j];
                    acc[j] += wg[j];
                    if (DEPTH) dep[j] += (int32_t)gd_dist(gx[j]);
                    x[j] = g32_ptr(w32);
                    act[j] = !g32_sink(w32);
                }
                any |= act[j];
            }
            if (!any) break;
        }
#pragma unroll
        for (int j = 0; j < ILP; ++j) {
            if (v[j] < 0) continue;
            const bool fin = (kd[j] & kKFin) != 0;
            if (fin) st_cg(word + v[j], (uint64_t)(uint32_t)acc[j] << 32 | kLvKnown | (uint32_t)dep[j]);
            if (!(kd[j] & kKSinkSlot)) key[v[j]] = fin ? oddsz[v[j]] + acc[j] : INT32_MAX;
            if (DEPTH) depth[v[j]] = fin ? dep[j] : -1;
        }
    }
}

}  // namespace
}  // namespace pg
