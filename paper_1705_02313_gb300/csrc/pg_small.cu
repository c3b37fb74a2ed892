// The full valuation of a small game (K1 and K2 of pg_iter.cu, distinct
// priorities) in one launch.
//
// Below about 10^5 vertices the dozen launches and memsets of
// enqueue_valuation are latency only: each pass takes 2 to 10 us for reads that
// take one, plus the gap to the next. k_val_small runs them all in one launch:
// of a cluster of up to 16 blocks with the cluster barrier (about 0.4 us)
// between the passes or, beyond kSmallGrid ids, of one or two blocks per SM with
// the software barrier (about 1.3 us). The ranks and depths are those of the
// separate kernels. pg_valuate_static of 100k vertices: 158 -> 76 us.
#include <cooperative_groups.h>

#include "pg_device.cuh"

namespace cg = cooperative_groups;

namespace pg {
namespace {

// Up to the sibling weights, cluster against grid: 10k ids 22 / 33 us, 40k 40 /
// 35 us, 100k 76 / 36 us, 262k 170 / 47 us. The cluster takes what its threads hold
// at once: beyond, a second round of chains doubles the time of deep forests (20k
// vertices in runs of 50: 202 / 161 us). For the same reason the grid has two
// blocks per SM beyond 155,648 ids (260k: 276 / 172 us).
constexpr int kSmallThreads = 1024;
constexpr int kSmallCluster = 16;
constexpr int32_t kSmallGrid = kSmallCluster * kSmallThreads;
// A warp orders up to this many children of one parent, a block more (that many,
// in blocks: 260k vertices, 100 to a parent, 497 us, 407 with warps).
constexpr int kSmallWarpKids = 128;
constexpr int kSmallHot = 2048;  // the block's table of additions near the roots (as in k_chain1)
constexpr int kSmallHotBits = 11;
constexpr int kSmallTop = 8;     // takes the last this many g-ancestors of a chain
// With two blocks per SM the lanes of a warp add to the table in step, or else
// several chains wait for each other's: plays through 160k, 200k and 260k vertices
// 304, 372 and 390 us, in step 259, 292 and 351 (by the separate kernels 312, 344
// and 341); runs of 50 rising vertices 206, 220 and 218, in step 211, 214 and 220
// (100k, one block: 191, in step 262).
constexpr int kSmallSteps = 128;   // steps of one resolution round

// Three sums in one word: children of vertices, sizes of the sink's even and of its odd children. Each is at
// most kSmallIds < 2^21.
constexpr int kSumBits = 21;
static_assert(kSmallIds < (1 << kSumBits), "the packed sums must hold every id");
constexpr uint64_t kSumMask = (1ull << kSumBits) - 1;

struct SmallArgs {
    int32_t n, sink0;
    int32_t* strat;
    uint8_t* flags;
    const int32_t* pri;
    uint64_t* gd;
    uint32_t* gd32;
    int32_t *biglist, *hugelist, *sz, *oddsz, *ccnt, *coff, *slot, *wgt, *key, *depth, *dom;
    uint8_t *kind, *cls;
    int2* cl_ks;
    int64_t* tiles;  // [kSmallBlocks] block sums
    GameState* gst;
    Counters* cnt;
    int32_t want_dom, deep_cut, deep_fallback, jump_cap;
    // pg_valuate_static: the caller's successor function and parities, copied and checked first (null otherwise)
    const int32_t* succ;
    const uint8_t* odd;
    int8_t* val_class;  // its outputs (each nullable)
    int32_t *val_depth, *val_rank;
};

__device__ inline void small_hot_add(int32_t x, int32_t* tkey, int32_t* tcnt, int32_t* sz) {
    const uint32_t h = ((uint32_t)x * 2654435761u) >> (32 - kSmallHotBits);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t i = (h + p) & (kSmallHot - 1);
        int32_t k = *(volatile int32_t*)&tkey[i];
        if (k == -1) k = atomicCAS(&tkey[i], -1, x);
        if (k == -1 || k == x) {
            atomicAdd(&tcnt[i], 1);
            return;
        }
    }
    atomicAdd(sz + x, 1);
}

// What id v adds to the packed sums, once sizes and children counts are final.
__device__ inline uint64_t small_sums(const SmallArgs& a, int32_t v, uint8_t kd) {
    uint64_t s = (uint64_t)__ldcg(a.ccnt + v);
    if ((kd & (kKFin | kKSinkChild)) == (kKFin | kKSinkChild)) {
        const uint64_t size = 1 + (uint64_t)__ldcg(a.sz + v);
        s += size << ((kd & kKOdd) ? 2 * kSumBits : kSumBits);
    }
    return s;
}

// PER_SM > 0: the launch is cooperative, of up to that many blocks per SM, and its
// blocks meet at the software barrier (which gives up after a bounded wait: every
// block then returns); otherwise it is one cluster. Reads of what the kernel itself
// writes go to L2 (__ldcg): the barrier makes them visible there.
template <int PER_SM>
__global__ void __launch_bounds__(kSmallThreads, PER_SM == 2 ? 2 : 1) k_val_small(SmallArgs a) {
    constexpr bool kInStep = PER_SM == 2;
    const int32_t tid = threadIdx.x, CL = (int32_t)gridDim.x, rank = (int32_t)blockIdx.x;
    const int32_t T = CL * kSmallThreads, t0 = rank * kSmallThreads + tid;
    auto sync = [&] {
        if constexpr (PER_SM > 0) return grid_sync(a.cnt);
        cg::this_cluster().sync();
        return true;
    };
    const int32_t n = a.n;
    const int lane = tid & 31;
    // the table of additions near the roots, then the segments of parents with many children
    __shared__ int2 sk[kHugeChildren];
    int32_t *tkey = (int32_t*)sk, *tcnt = tkey + kSmallHot;
    static_assert(sizeof(sk) >= 2 * sizeof(int32_t) * kSmallHot, "the table fits");
    Counters* cnt = a.cnt;
    for (int i = tid; i < kSmallHot; i += kSmallThreads) {
        tkey[i] = -1;
        tcnt[i] = 0;
    }
    // every vertex's word starts as a jump pointer of one step
    for (int32_t v = t0; v < n; v += T) {
        int32_t s;
        if (!a.succ) {
            s = __ldcg(a.strat + v);
        } else if (v == a.sink0) {
            s = v;
            a.flags[v] = kSinkSlot;
        } else {
            s = a.succ[v];
            if (s < 0 || s > a.sink0) {
                atomicAdd(&cnt->bad, 1);
                s = a.sink0;
            }
            a.flags[v] = a.odd[v] ? kPriOdd : 0;
        }
        const uint64_t w = v == a.sink0 ? gd_pack(true, false, 0, v, true)
                           : s > v ? gd_pack(true, false, 1, s, s == a.sink0)
                           : s == v ? gd_pack(true, true, 1, v)
                                    : gd_pack(false, false, 1, s);
        st_cg(a.gd + v, w);
        __stcg(a.gd32 + v, g32_of(w));
        __stcg(a.sz + v, 0);
        __stcg(a.oddsz + v, 0);
        __stcg(a.ccnt + v, 0);
    }
    if (t0 == 0 && a.succ) a.gst->nodd = 0;
    if (!sync()) return;
    // nearest greater vertices: words turn from jump pointers into g-words, in rounds. Any word is valid whenever
    // it is read (every vertex between v and a pending word's pointer is below v), so a walk uses the progress of
    // the others and takes a few steps where one along the play takes dozens.
    for (int32_t r = 0;; ++r) {
        if (t0 == 0) cnt->left[(r + 1) % 3] = 0;
        int32_t left = 0;
        for (int32_t v = t0; v < n; v += T) {
            uint64_t w = ld_cg(a.gd + v);
            if (gd_resolved(w)) continue;
            int32_t x = gd_ptr(w);
            uint64_t d = gd_dist(w);
            bool none = false;
            for (int k = 0; k < kSmallSteps && x < v; ++k) {
                const uint64_t wx = ld_cg(a.gd + x);
                if (gd_resolved(wx) && gd_none(wx)) {  // v is above its whole future too (same cycle)
                    none = true;
                    x = gd_ptr(wx);
                    break;
                }
                d += gd_dist(wx);
                x = gd_ptr(wx);
            }
            if (d > kDistMax) d = kDistMax;  // only reachable around cycles, where dist is unused
            if (none) w = gd_pack(true, true, 0, x);
            else if (x > v) w = gd_pack(true, false, (uint32_t)d, x, x == a.sink0);
            else if (x == v) w = gd_pack(true, true, (uint32_t)d, v);
            else {
                w = gd_pack(false, false, (uint32_t)d, x);
                left = 1;
            }
            st_cg(a.gd + v, w);
            if (gd_resolved(w)) __stcg(a.gd32 + v, g32_of(w));
        }
        left = __reduce_add_sync(kFull, left);
        if (lane == 0 && left) atomicAdd(&cnt->left[r % 3], left);
        if (!sync()) return;
        if (__ldcg(&cnt->left[r % 3]) == 0) {
            if (t0 == 0) cnt->jump_rounds = r;
            break;
        }
        if (r + 1 >= a.jump_cap) {  // the ruling-set path retries with a larger cap, or the call fails
            if (t0 == 0) {
                if (a.deep_fallback) cnt->deep = 1;
                else atomicOr(&cnt->err, kErrJumpRounds);
            }
            for (int32_t v = t0; v <= n; v += T) a.ccnt[v] = 0;
            return;
        }
    }
    // classification, g-subtree sizes, children counts (as k_chain1)
    int32_t nfin = 0, nodd = 0;
    for (int32_t b = t0 - lane; b < n; b += T) {
        const int32_t v = b + lane;
        const uint32_t w = v < n ? __ldcg(a.gd32 + v) : kG32Sink;
        const uint8_t f = v < n ? a.flags[v] : kSinkSlot;
        const bool slot = (f & kSinkSlot) != 0;
        int32_t x = g32_ptr(w), cyc = !slot && g32_none(w) ? x : -1, len = 0;
        bool cut = false;
        for (bool act = !slot && !g32_none(w) && !g32_sink(w); act;) {
            if (len >= a.deep_cut) {
                cut = true;
                cnt->deep = 1;
                break;
            }
            const uint32_t wx = __ldcg(a.gd32 + x);
            ++len;
            if (g32_none(wx)) {
                cyc = g32_ptr(wx);
                act = false;
            } else {
                x = g32_ptr(wx);
                act = !g32_sink(wx);
            }
        }
        // one more for each of the len g-ancestors of a finite vertex, the last ones of a long chain in the block's
        // table (in step: with all lanes at the same distance from their roots)
        int32_t sl = -1;
        const bool child = !slot && cyc < 0 && !g32_sink(w) && !cut, table = child && len >= 4;
        x = g32_ptr(w);
        if (child) {
            sl = atomicAdd(a.ccnt + x, 1);
            for (;; --len) {
                if (table && len <= kSmallTop) {
                    if (kInStep) break;
                    small_hot_add(x, tkey, tcnt, a.sz);
                } else {
                    atomicAdd(a.sz + x, 1);
                }
                const uint32_t wx = __ldcg(a.gd32 + x);
                if (g32_sink(wx)) break;
                x = g32_ptr(wx);
            }
        }
        if (kInStep && __any_sync(kFull, table)) {
            for (int32_t l = kSmallTop; l > 0; --l) {
                if (table && len >= l) {
                    small_hot_add(x, tkey, tcnt, a.sz);
                    if (l > 1) x = g32_ptr(__ldcg(a.gd32 + x));
                }
                __syncwarp();
            }
        }
        if (v >= n) continue;
        a.slot[v] = sl;
        if (slot) {
            a.kind[v] = kKSinkSlot;
            a.cls[v] = kFin;
            if (a.want_dom) a.dom[v] = -1;
        } else if (cyc < 0) {
            a.kind[v] = kKFin | (g32_sink(w) ? kKSinkChild : 0) | ((f & kPriOdd) ? kKOdd : 0);
            a.cls[v] = kFin;
            if (a.want_dom) a.dom[v] = -1;
            ++nfin;
        } else {
            const bool odd = (a.flags[cyc] & kPriOdd) != 0;
            a.kind[v] = 0;
            a.cls[v] = odd ? kOddCycle : kTop;
            if (a.want_dom) a.dom[v] = a.pri[cyc];
            nodd += odd;
        }
    }
    __syncthreads();
    for (int i = tid; i < kSmallHot; i += kSmallThreads)
        if (tcnt[i]) atomicAdd(a.sz + tkey[i], tcnt[i]);
    nfin = __reduce_add_sync(kFull, nfin);
    nodd = __reduce_add_sync(kFull, nodd);
    if (lane == 0 && nfin) atomicAdd(&cnt->n_fin, nfin);
    if (lane == 0 && nodd) {
        atomicAdd(&cnt->n_odd, nodd);
        atomicAdd(&a.gst->nodd, nodd);
    }
    if (!sync()) return;
    if (__ldcg(&cnt->deep)) {  // the ruling-set path takes over (it expects no children counts)
        for (int32_t v = t0; v <= n; v += T) a.ccnt[v] = 0;
        return;
    }
    // children segments and the id-ordered sums over the sink's children: each block scans a range of ids
    const int32_t per = ((n + CL - 1) / CL + kSmallThreads - 1) / kSmallThreads * kSmallThreads;
    const int32_t lo = min(n, rank * per), hi = min(n, lo + per);
    uint64_t sum = 0, total;
    for (int32_t v = lo + tid; v < hi; v += kSmallThreads) sum += small_sums(a, v, __ldcg(a.kind + v));
    block_scan_1024(sum, &total);
    if (tid == 0) __stcg((unsigned long long*)a.tiles + rank, (unsigned long long)total);
    if (!sync()) return;
    __shared__ uint64_t s_run;
    uint64_t all;
    {
        const uint64_t x = tid < CL ? __ldcg((unsigned long long*)a.tiles + tid) : 0;
        const uint64_t before = block_scan_1024(x, &all);
        if (tid == rank) s_run = before;
        __syncthreads();
    }
    uint64_t run = s_run;
    const int32_t tot_o = (int32_t)(all >> (2 * kSumBits));
    if (t0 == 0) {
        __stcg(a.coff + n, (int32_t)(all & kSumMask));
        a.key[a.sink0] = tot_o;
        cnt->sink_rank = tot_o;
        a.ccnt[n] = 0;
    }
    for (int32_t b = lo; b < hi; b += kSmallThreads) {
        const int32_t v = b + tid;
        const uint8_t kd = v < hi ? __ldcg(a.kind + v) : 0;
        const uint64_t own = v < hi ? small_sums(a, v, kd) : 0;
        const uint64_t at = run + block_scan_1024(own, &total);
        run += total;
        if (v >= hi) continue;
        __stcg(a.coff + v, (int32_t)(at & kSumMask));
        a.ccnt[v] = 0;
        const int32_t se = (int32_t)((own >> kSumBits) & kSumMask), so = (int32_t)(own >> (2 * kSumBits));
        if (se) a.wgt[v] = 1 + tot_o + (int32_t)((at >> kSumBits) & kSumMask);
        else if (so) a.wgt[v] = tot_o - ((int32_t)(at >> (2 * kSumBits)) + so);
    }
    if (!sync()) return;
    // children into their segments (as k_scatter)
    for (int32_t v = t0; v < n; v += T) {
        const uint8_t kd = __ldcg(a.kind + v);
        if (!(kd & kKFin) || (kd & kKSinkChild)) continue;
        const int32_t p = __ldcg(a.coff + g32_ptr(__ldcg(a.gd32 + v))) + __ldcg(a.slot + v);
        __stcg(a.cl_ks + p, make_int2((kd & kKOdd) ? -(v + 1) : v, 1 + __ldcg(a.sz + v)));
    }
    if (!sync()) return;
    // sibling weights (as k_siblings)
    for (int32_t b = t0 - lane; b < n; b += T) {
        const int32_t p = b + lane;
        int32_t s0 = 0, k = 0;
        if (p < n) {
            s0 = __ldcg(a.coff + p);
            k = __ldcg(a.coff + p + 1) - s0;
        }
        if (k > kHugeChildren) __stcg(a.hugelist + atomicAdd(&cnt->n_huge, 1), p);
        else if (k > 32) __stcg(a.biglist + atomicAdd(&cnt->n_big, 1), p);
        else if (k > 0 && k <= 4) {
            int2 c[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) c[i] = i < k ? __ldcg(a.cl_ks + s0 + i) : make_int2(INT32_MAX, 0);
            int32_t os = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i >= k) continue;
                int32_t pre = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (c[j].x < c[i].x) pre += c[j].y;
                a.wgt[c[i].x >= 0 ? c[i].x : -c[i].x - 1] = pre + (c[i].x >= 0 ? 1 : 0);
                if (c[i].x < 0) os += c[i].y;
            }
            a.oddsz[p] = os;
        }
        unsigned mid = __ballot_sync(kFull, k > 4 && k <= 32);
        while (mid) {
            const int src = __ffs(mid) - 1;
            mid &= mid - 1;
            const int32_t pp = __shfl_sync(kFull, p, src), ps = __shfl_sync(kFull, s0, src),
                          pk = __shfl_sync(kFull, k, src);
            const int2 mine = lane < pk ? __ldcg(a.cl_ks + ps + lane) : make_int2(INT32_MAX, 0);
            int32_t pre = 0;
            for (int j = 0; j < pk; ++j) {
                const int32_t kx = __shfl_sync(kFull, mine.x, j), ky = __shfl_sync(kFull, mine.y, j);
                if (kx < mine.x) pre += ky;
            }
            const int32_t os = __reduce_add_sync(kFull, lane < pk && mine.x < 0 ? mine.y : 0);
            if (lane < pk) a.wgt[mine.x >= 0 ? mine.x : -mine.x - 1] = pre + (mine.x >= 0 ? 1 : 0);
            if (lane == 0) a.oddsz[pp] = os;
        }
    }
    if (!sync()) return;
    const int32_t nb = __ldcg(&cnt->n_big), nh = __ldcg(&cnt->n_huge);
    // parents with up to kSmallWarpKids children: a warp each, four children to a lane
    for (int32_t b = t0 >> 5; b < nb; b += T >> 5) {
        const int32_t p = __ldcg(a.biglist + b), s0 = __ldcg(a.coff + p), k = __ldcg(a.coff + p + 1) - s0;
        if (k > kSmallWarpKids) continue;
        int2 c[4];
        int32_t pre[4] = {0, 0, 0, 0}, os = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            c[i] = lane + 32 * i < k ? __ldcg(a.cl_ks + s0 + lane + 32 * i) : make_int2(INT32_MAX, 0);
            if (c[i].x < 0) os += c[i].y;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int kn = min(32, k - 32 * i);
            for (int j = 0; j < kn; ++j) {
                const int32_t kx = __shfl_sync(kFull, c[i].x, j), ky = __shfl_sync(kFull, c[i].y, j);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (kx < c[q].x) pre[q] += ky;
            }
        }
        os = __reduce_add_sync(kFull, os);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (lane + 32 * i < k) a.wgt[c[i].x >= 0 ? c[i].x : -c[i].x - 1] = pre[i] + (c[i].x >= 0 ? 1 : 0);
        if (lane == 0) a.oddsz[p] = os;
    }
    // parents with up to kHugeChildren children: a block each sorts the segment and scans it
    for (int32_t b = rank; b < nb; b += CL) {
        const int32_t p = __ldcg(a.biglist + b), s0 = __ldcg(a.coff + p), k = __ldcg(a.coff + p + 1) - s0;
        if (k <= kSmallWarpKids) continue;
        int p2 = 64;
        while (p2 < k) p2 <<= 1;
        for (int i = tid; i < p2; i += kSmallThreads) sk[i] = i < k ? __ldcg(a.cl_ks + s0 + i) : make_int2(INT32_MAX, 0);
        __syncthreads();
        for (int kk = 2; kk <= p2; kk <<= 1) {
            for (int j = kk >> 1; j > 0; j >>= 1) {
                for (int i = tid; i < p2; i += kSmallThreads) {
                    const int o = i ^ j;
                    if (o <= i) continue;
                    const int2 x = sk[i], y = sk[o];
                    if ((x.x > y.x) == ((i & kk) == 0)) {
                        sk[i] = y;
                        sk[o] = x;
                    }
                }
                __syncthreads();
            }
        }
        uint64_t before = 0, odd_all = 0, part;
        for (int base = 0; base < k; base += kSmallThreads) {
            const int i = base + tid;
            const int2 e = i < k ? sk[i] : make_int2(0, 0);
            const uint64_t at = before + block_scan_1024(i < k ? (uint64_t)e.y : 0, &part);
            before += part;
            if (i < k) a.wgt[e.x >= 0 ? e.x : -e.x - 1] = (int32_t)at + (e.x >= 0 ? 1 : 0);
            block_scan_1024(i < k && e.x < 0 ? (uint64_t)e.y : 0, &part);
            odd_all += part;
        }
        if (tid == 0) a.oddsz[p] = (int32_t)odd_all;
        __syncthreads();
    }
    // parents with more: the id-ordered scan over every vertex, as for the sink's children
    for (int32_t h = 0; h < nh; ++h) {
        const int32_t p = __ldcg(a.hugelist + h);
        auto size_of = [&](int32_t v) {
            const uint8_t kd = __ldcg(a.kind + v);
            if (!(kd & kKFin) || (kd & kKSinkChild) || g32_ptr(__ldcg(a.gd32 + v)) != p) return (uint64_t)0;
            return (1 + (uint64_t)__ldcg(a.sz + v)) << ((kd & kKOdd) ? 2 * kSumBits : kSumBits);
        };
        sum = 0;
        for (int32_t v = lo + tid; v < hi; v += kSmallThreads) sum += size_of(v);
        block_scan_1024(sum, &total);
        if (tid == 0) __stcg((unsigned long long*)a.tiles + rank, (unsigned long long)total);
        if (!sync()) return;
        const uint64_t bx = block_scan_1024(tid < CL ? __ldcg((unsigned long long*)a.tiles + tid) : 0, &all);
        if (tid == rank) s_run = bx;
        __syncthreads();
        run = s_run;
        const int32_t podd = (int32_t)(all >> (2 * kSumBits));
        for (int32_t b = lo; b < hi; b += kSmallThreads) {
            const int32_t v = b + tid;
            const uint64_t own = v < hi ? size_of(v) : 0;
            const uint64_t at = run + block_scan_1024(own, &total);
            run += total;
            const int32_t se = (int32_t)((own >> kSumBits) & kSumMask), so = (int32_t)(own >> (2 * kSumBits));
            if (se) a.wgt[v] = 1 + podd + (int32_t)((at >> kSumBits) & kSumMask);
            else if (so) a.wgt[v] = podd - ((int32_t)(at >> (2 * kSumBits)) + so);
        }
        if (t0 == 0) a.oddsz[p] = podd;
        if (!sync()) return;  // the block sums are reused
    }
    if (nb && !sync()) return;
    // ranks and depths (as k_chain2)
    for (int32_t v = t0; v < n; v += T) {
        const uint8_t kd = __ldcg(a.kind + v);
        if (kd & kKSinkSlot) continue;
        const bool fin = (kd & kKFin) != 0;
        int32_t rnk = INT32_MAX, dep = -1;
        if (fin) {
            uint64_t w = ld_cg(a.gd + v);
            rnk = __ldcg(a.oddsz + v) + __ldcg(a.wgt + v);
            dep = (int32_t)gd_dist(w);
            while (!gd_sink(w)) {
                const int32_t x = gd_ptr(w);
                w = ld_cg(a.gd + x);
                rnk += __ldcg(a.wgt + x);
                dep += (int32_t)gd_dist(w);
            }
        }
        a.key[v] = rnk;
        a.depth[v] = dep;
        if (a.val_class) a.val_class[v] = fin ? 0 : 1;
        if (a.val_depth) a.val_depth[v] = dep;
        if (a.val_rank) a.val_rank[v] = rnk;
    }
}

}  // namespace

int cluster_blocks(const void* kern, int threads, size_t shared, int want, int device, std::atomic<int>* cache) {
    const bool cached = device >= 0 && device < kClusterDevices;
    if (int c = cached ? cache[device].load() : 0) return c;
    cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);  // (refused: smaller clusters)
    bool ready = !shared || cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared) ==
                                cudaSuccess;
    for (int c = want; ready && c >= 1; c >>= 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = shared;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = c;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int k = 0;
        if (cudaOccupancyMaxActiveClusters(&k, kern, &cfg) == cudaSuccess && k > 0) {
            cudaGetLastError();
            if (cached) cache[device].store(c);
            return c;
        }
    }
    cudaGetLastError();
    return 1;  // (asked again next time: the launch says what is wrong)
}

namespace {
std::atomic<int> g_small_cluster[kClusterDevices];
}

pg_status enqueue_val_small(pg_game* g, bool want_dom) {
    pg_ctx* ctx = g->ctx;
    SmallArgs a = {};
    a.n = g->n;
    a.sink0 = g->sink0;
    a.strat = g->strat;
    a.flags = g->flags;
    a.pri = g->pri;
    a.gd = g->gd;
    a.gd32 = g->gd32;
    a.biglist = g->plist;
    a.hugelist = g->hugelist;
    a.sz = g->sz;
    a.oddsz = g->oddsz;
    a.ccnt = g->ccnt;
    a.coff = g->coff;
    a.slot = g->slot;
    a.wgt = g->wgt;
    a.key = g->key;
    a.depth = g->depth;
    a.dom = g->dom;
    a.kind = g->kind;
    a.cls = g->cls;
    a.cl_ks = g->cl_ks;
    a.tiles = g->tiles;
    a.gst = g->gst;
    a.cnt = g->cnt;
    a.want_dom = want_dom ? 1 : 0;
    a.deep_cut = g->tune.deep_cut;
    a.deep_fallback = ctx->deep_fallback ? 1 : 0;
    a.jump_cap = 64;
    for (int64_t x = g->n; x > 1; x >>= 1) a.jump_cap += 2;
    a.succ = g->in_succ;
    a.odd = g->in_odd;
    a.val_class = g->out_class;
    a.val_depth = g->out_depth;
    a.val_rank = g->out_rank;
    if (g->n > kSmallGrid) {
        int sms = 0;
        PG_CUDA_TRY(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device));
        const int per = g->n > sms * kSmallThreads ? 2 : 1;
        const int blocks = std::max(1, std::min({per * sms, kSmallBlocks, (g->n + kSmallThreads - 1) / kSmallThreads}));
        void* args[] = {(void*)&a};
        PG_CUDA_TRY(ctx, cudaLaunchCooperativeKernel(per == 2 ? (void*)k_val_small<2> : (void*)k_val_small<1>, blocks,
                                                     kSmallThreads, args, 0, ctx->stream));
        return PG_OK;
    }
    int c = kSmallCluster;
    while (c > 1 && (int64_t)c * kSmallThreads / 2 >= g->n) c >>= 1;
    c = std::min(c, cluster_blocks((const void*)k_val_small<0>, kSmallThreads, 0, kSmallCluster, g->device,
                                   g_small_cluster));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(kSmallThreads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    PG_CUDA_TRY(ctx, cudaLaunchKernelEx(&cfg, k_val_small<0>, a));
    return PG_OK;
}

}  // namespace pg
