// Loading a small game in one launch: the validation, the admissibility
// preprocessing of Section 3 and the relabelling of load_game_pass (pg_load.cu).
//
// That path is about 45 kernels and memsets, 35 temporary allocations and four
// host waits, 340 us for a game of 1,000 vertices and 390 us for one of 30,000,
// of which the GPU works for a third. Here one kernel runs its passes with a
// barrier between them (a cluster, or one block per SM, as k_val_small): 170 and
// 215 us; at 1M vertices 660 -> 465 us, at 3M 1,150 -> 990, at 6M 2,010 -> 2,130
// (ladders, whose traps unravel in long cascades: 100k 820 -> 490 us, 3M 1,670 ->
// 1,240). Nothing it writes is sized by a count the host has to read first (a game has at most
// as many dummies as vertices), so the host waits once, at the end. A game that
// this kernel does not take (refused inputs, repeated or sparse priorities) is
// loaded again by the general path, which decides what becomes of it.
#include <cooperative_groups.h>

#include "pg_device.cuh"

namespace cg = cooperative_groups;

namespace pg {
namespace {

constexpr int kLsThreads = 1024;
constexpr int kLsCluster = 16;
constexpr int kLsBlocks = 256;      // at most this many blocks (the array of their sums)
// A thread peels this many vertices depth first, of this many it may hold, before
// it hands over to the next round: 4 / 8 / 16 / 32 / 64 / 256 load the ladder of
// 100k vertices, whose cascades are long, in 481 / 561 / 668 / 834 / 1,140 /
// 1,672 us and the random game of 1M in 472 / 464 / 456 / 444 / 445 / 447 us.
constexpr int kLsStack = 4, kLsBudget = 4;
constexpr int kLsRounds = 2048;     // peeling rounds before the general path takes over

struct LoadStatus {
    Counters c;         // the software barrier, c.err
    int32_t general;    // the general path must load this game
    int32_t maxpri;
    int32_t k;          // dummies
    int32_t front[3];   // peeling frontiers, in turn
};

struct LoadArgs {
    int32_t n, words;  // words: what bits holds
    int64_t m;
    // the caller's arrays
    const int32_t *off, *tgt, *pri;
    const uint8_t* own;
    // temporaries
    int32_t *indeg, *roff, *radj, *left, *fa, *fb, *widx, *gid, *wprefix, *nidu;
    uint8_t *inU, *isW;
    uint32_t* bits;
    int64_t* tiles;  // [kLsBlocks]
    LoadStatus* st;
    // the game's arrays (2 n + 2 ids, m + n edges at most)
    int32_t *goff, *gtgt, *gpri, *nid0, *orig_of, *dnid, *dummy_of, *strat, *gsink;
    uint8_t* gflags;
};

// Words of the priority bitmap: 64 priorities for each vertex or, as long as that
// is 16 MB with the prefix, 2,048. One block takes 1 us per 1,024 of them, so a
// game of 1,000 vertices loads in 190 us at the most, against 370 the general
// way. Sparser games are left to that, whose first priorities tell: the copies
// and the passes up to the maximum were wasted on them (1M vertices from host
// arrays, 300 per vertex: 1,052 us with them, 855 without).
constexpr int64_t kLsWords = 1 << 21;
inline int32_t ls_words(int64_t n) { return (int32_t)std::max(2 * n + 2048, std::min(kLsWords, 64 * n)); }
__host__ __device__ inline bool ls_sparse(int32_t p, int32_t n, int32_t words) {
    return (int64_t)p + 2 * (int64_t)n >= 32 * (int64_t)words;
}

template <bool GRID>
__global__ void __launch_bounds__(kLsThreads, 1) k_load_small(LoadArgs a) {
    const int32_t tid = threadIdx.x, CL = (int32_t)gridDim.x, rank = (int32_t)blockIdx.x;
    const int32_t T = CL * kLsThreads, t0 = rank * kLsThreads + tid;
    LoadStatus* st = a.st;
    auto sync = [&] {
        if constexpr (GRID) return grid_sync(&st->c);
        cg::this_cluster().sync();
        return true;
    };
    const int32_t n = a.n;
    const int lane = tid & 31;
    __shared__ uint64_t s_run;
    // exclusive scan of value(i), i < count, each block over a range of its own; store(i, prefix, value). Returns
    // false if the barrier gave up; *total: the sum.
    auto scan = [&](int32_t count, auto&& value, auto&& store, int64_t* total) {
        const int32_t per = ((count + CL - 1) / CL + kLsThreads - 1) / kLsThreads * kLsThreads;
        const int32_t lo = min(count, rank * per), hi = min(count, lo + per);
        uint64_t sum = 0, part;
        for (int32_t i = lo + tid; i < hi; i += kLsThreads) sum += (uint64_t)value(i);
        block_scan_1024(sum, &part);
        if (tid == 0) __stcg((unsigned long long*)a.tiles + rank, (unsigned long long)part);
        if (!sync()) return false;
        const uint64_t before = block_scan_1024(tid < CL ? __ldcg((unsigned long long*)a.tiles + tid) : 0, &sum);
        if (tid == rank) s_run = before;
        __syncthreads();
        uint64_t run = s_run;
        for (int32_t b = lo; b < hi; b += kLsThreads) {
            const int32_t i = b + tid;
            const int32_t x = i < hi ? value(i) : 0;
            const uint64_t at = run + block_scan_1024((uint64_t)x, &part);
            run += part;
            if (i < hi) store(i, (int32_t)at, x);
        }
        *total = (int64_t)sum;
        return true;
    };
    {  // few distinct priorities repeat among the first vertices, very sparse ones show there: the general path
        const int32_t p = lane < n ? a.pri[lane] : -1 - lane;
        if (__any_sync(kFull, __popc(__match_any_sync(kFull, p)) > 1 || ls_sparse(p, n, a.words))) {
            if (t0 == 0) st->general = 1;
            return;
        }
    }
    // validation (as k_validate), and the arrays that start at zero
    int32_t bad = 0, mx = -1;
    for (int32_t v = t0; v < n; v += T) {
        const int32_t x = a.off[v], y = a.off[v + 1], p = a.pri[v];
        if (x < 0 || y <= x || (int64_t)y > a.m || (v == 0 && x != 0) || (v == n - 1 && (int64_t)y != a.m) ||
            a.own[v] > 1 || p < 0)
            bad = 1;
        mx = max(mx, p);
        __stcg(a.indeg + v, 0);
        a.isW[v] = 0;
    }
    for (int64_t e = t0; e < a.m; e += T) bad |= a.tgt[e] < 0 || a.tgt[e] >= n;
    bad = __reduce_or_sync(kFull, (unsigned)bad);
    mx = __reduce_max_sync(kFull, mx);
    if (lane == 0 && bad) st->general = 1;
    if (lane == 0) atomicMax(&st->maxpri, mx);
    if (!sync()) return;
    const int64_t top = (int64_t)__ldcg(&st->maxpri) + 2 * (int64_t)n;  // no G' priority is larger
    if (__ldcg(&st->general) || top >= 32ll * a.words) {  // (ls_sparse of the largest)
        if (t0 == 0) st->general = 1;
        return;
    }
    for (int32_t w = t0; w <= (int32_t)(top >> 5); w += T) __stcg(a.bits + w, 0u);
    // U starts as the Odd vertices with an edge to one (as k_indegree, k_trap_init)
    for (int32_t v = t0; v < n; v += T) {
        int32_t c = 0;
        if (a.own[v]) {
            for (int32_t e = a.off[v]; e < a.off[v + 1]; ++e) {
                const int32_t t = a.tgt[e];
                if (!a.own[t]) continue;
                ++c;
                atomicAdd(a.indeg + t, 1);
            }
            __stcg(a.left + v, c);
            if (c == 0) __stcg(a.fa + atomicAdd(&st->front[0], 1), v);
        }
        a.inU[v] = c > 0;
    }
    if (!sync()) return;
    int64_t total;
    auto at_indeg = [&](int32_t v) { return __ldcg(a.indeg + v); };
    if (!scan(n, at_indeg, [&](int32_t v, int32_t at, int32_t) { __stcg(a.roff + v, at); }, &total)) return;
    if (t0 == 0) __stcg(a.roff + n, (int32_t)total);
    if (!sync()) return;
    for (int32_t v = t0; v < n; v += T) {  // indeg counts down: the free slots of each list
        if (!a.own[v]) continue;
        for (int32_t e = a.off[v]; e < a.off[v + 1]; ++e) {
            const int32_t t = a.tgt[e];
            if (a.own[t]) __stcg(a.radj + __ldcg(a.roff + t) + atomicSub(a.indeg + t, 1) - 1, v);
        }
    }
    if (!sync()) return;
    // peeling: a vertex that leaves U takes one from the counts of its Odd predecessors; one whose count reaches
    // zero leaves too. Depth first per thread within a budget, the rest in the next round.
    for (int32_t r = 0;; ++r) {
        const int32_t nf = __ldcg(&st->front[r % 3]);
        if (nf == 0) break;
        if (r >= kLsRounds) {
            if (t0 == 0) st->general = 1;
            return;
        }
        if (t0 == 0) st->front[(r + 2) % 3] = 0;
        const int32_t* cur = (r & 1) ? a.fb : a.fa;
        int32_t* nxt = (r & 1) ? a.fa : a.fb;
        for (int32_t i = t0; i < nf; i += T) {
            int32_t stack[kLsStack], depth = 0, budget = kLsBudget;
            stack[depth++] = __ldcg(cur + i);
            while (depth > 0) {
                const int32_t x = stack[--depth];
                const int32_t e1 = __ldcg(a.roff + x + 1);
                for (int32_t e = __ldcg(a.roff + x); e < e1; ++e) {
                    const int32_t y = __ldcg(a.radj + e);
                    if (atomicSub(a.left + y, 1) != 1) continue;
                    a.inU[y] = 0;
                    if (depth < kLsStack && budget > 0) {
                        stack[depth++] = y;
                        --budget;
                    } else {
                        __stcg(nxt + atomicAdd(&st->front[(r + 1) % 3], 1), y);
                    }
                }
            }
        }
        if (!sync()) return;
    }
    // W: the vertices of U entered by an edge from U; dummies in their order
    for (int32_t v = t0; v < n; v += T) {
        if (!__ldcg(a.inU + v)) continue;
        for (int32_t e = a.off[v]; e < a.off[v + 1]; ++e)
            if (__ldcg(a.inU + a.tgt[e])) a.isW[a.tgt[e]] = 1;
    }
    if (!sync()) return;
    int64_t total_w;
    if (!scan(n, [&](int32_t v) { return (int32_t)__ldcg(a.isW + v); },
              [&](int32_t v, int32_t at, int32_t w) {
                  __stcg(a.widx + v, at);
                  if (w) __stcg(a.dummy_of + at, v);
              },
              &total_w))
        return;
    const int32_t k = (int32_t)total_w, np = n + k;
    if (t0 == 0) st->k = k;
    if (!sync()) return;
    // ids: ranks of the G' priorities (originals raised by 2k, dummy j has 2j)
    auto prio = [&](int32_t x) { return x < n ? a.pri[x] + 2 * k : 2 * (x - n); };
    int32_t dup = 0;
    for (int32_t x = t0; x < np; x += T) {
        const int32_t p = prio(x);
        dup |= (atomicOr(a.bits + (p >> 5), 1u << (p & 31)) >> (p & 31)) & 1u;
    }
    dup = __reduce_or_sync(kFull, (unsigned)dup);
    if (lane == 0 && dup) st->general = 1;
    if (!sync()) return;
    if (__ldcg(&st->general)) return;
    const int32_t words = (int32_t)(((int64_t)__ldcg(&st->maxpri) + 2 * (int64_t)k) >> 5) + 1;
    if (!scan(words, [&](int32_t w) { return __popc(__ldcg(a.bits + w)); },
              [&](int32_t w, int32_t at, int32_t) { __stcg(a.wprefix + w, at); }, &total))
        return;
    if (!sync()) return;
    for (int32_t x = t0; x < np; x += T) {
        const int32_t p = prio(x);
        const int32_t id = __ldcg(a.wprefix + (p >> 5)) + __popc(__ldcg(a.bits + (p >> 5)) & ((1u << (p & 31)) - 1u));
        __stcg((x < n ? a.nid0 + x : a.dnid + (x - n)), id);
        __stcg(a.gid + id, x);
    }
    if (!sync()) return;
    // each vertex's id as the target of an edge from U; edge offsets in relabelled order
    for (int32_t v = t0; v < n; v += T)
        __stcg(a.nidu + v, __ldcg(a.isW + v) ? __ldcg(a.dnid + __ldcg(a.widx + v)) : __ldcg(a.nid0 + v));
    auto degree = [&](int32_t i) {
        const int32_t x = __ldcg(a.gid + i);
        return x < n ? a.off[x + 1] - a.off[x] : 1;
    };
    if (!scan(np, degree, [&](int32_t i, int32_t at, int32_t) { __stcg(a.goff + i, at); }, &total)) return;
    if (!sync()) return;
    for (int32_t i = t0; i <= np; i += T) {
        if (i == np) {  // the sink slot: no edges
            a.goff[np] = a.goff[np + 1] = (int32_t)total;
            a.gflags[np] = kSinkSlot;
            a.gpri[np] = a.orig_of[np] = -1;
            a.strat[np] = *a.gsink = np;
            continue;
        }
        const int32_t x = __ldcg(a.gid + i), p = prio(x);
        int32_t* row = a.gtgt + __ldcg(a.goff + i);
        uint8_t f = (p & 1) ? kPriOdd : 0;
        if (x < n) {
            const int32_t* map = __ldcg(a.inU + x) ? a.nidu : a.nid0;
            const int32_t e0 = a.off[x], deg = a.off[x + 1] - e0;
            for (int32_t j = 0; j < deg; ++j) row[j] = __ldcg(map + a.tgt[e0 + j]);
            if (a.own[x]) f |= kOwnerOdd;
            a.orig_of[i] = x;
        } else {
            const int32_t w = __ldcg(a.dummy_of + (x - n));
            row[0] = __ldcg(a.nid0 + w);
            a.orig_of[i] = w;
        }
        a.gflags[i] = f;
        a.gpri[i] = p;
    }
}

std::atomic<int> g_ls_cluster[kClusterDevices];

// Parts of one allocation, each 256-byte aligned.
struct Parts {
    size_t bytes = 0;
    size_t add(size_t b) {
        const size_t at = bytes;
        bytes = (bytes + b + 255) & ~(size_t)255;
        return at;
    }
};

}  // namespace

pg_status load_small(pg_ctx* ctx, int32_t n, int64_t m, const int32_t* off, const int32_t* tgt, const uint8_t* own,
                     const int32_t* pri, int32_t mem_kind, pg_game** out, bool* general) {
    *out = nullptr;
    *general = true;
    const int32_t words = ls_words(n);
    if (mem_kind == PG_MEM_HOST)  // repeated or sparse priorities, before the arrays are copied
        for (int32_t v = 0; v < std::min(n, 32); ++v) {
            if (ls_sparse(pri[v], n, words)) return PG_OK;
            for (int32_t u = 0; u < v; ++u)
                if (pri[u] == pri[v]) return PG_OK;
        }
    cudaStream_t s = ctx->stream;
    const size_t N = (size_t)n, M = (size_t)m;
    LoadArgs a = {};
    a.n = n;
    a.m = m;
    a.words = words;
    // the temporaries, one allocation
    Parts tp;
    const bool host = mem_kind == PG_MEM_HOST;
    const size_t o_st = tp.add(sizeof(LoadStatus)), o_off = host ? tp.add(4 * (N + 1)) : 0,
                 o_tgt = host ? tp.add(4 * M) : 0, o_pri = host ? tp.add(4 * N) : 0, o_own = host ? tp.add(N) : 0,
                 o_ind = tp.add(4 * N), o_roff = tp.add(4 * (N + 1)), o_radj = tp.add(4 * M), o_left = tp.add(4 * N),
                 o_fa = tp.add(4 * N), o_fb = tp.add(4 * N), o_widx = tp.add(4 * N), o_gid = tp.add(8 * N),
                 o_wp = tp.add(4 * (size_t)a.words), o_nidu = tp.add(4 * N), o_inU = tp.add(N), o_isW = tp.add(N),
                 o_bits = tp.add(4 * (size_t)a.words), o_tiles = tp.add(8 * kLsBlocks);
    char* t = nullptr;
    PG_CUDA_TRY(ctx, dev_alloc(ctx, (void**)&t, tp.bytes, s));
    struct Free {
        void* p;
        cudaStream_t s;
        ~Free() { cudaFreeAsync(p, s); }
    } guard{t, s};
    pg_game* g = new pg_game();
    g->ctx = ctx;
    g->device = ctx->device;
    auto bail = [&](cudaError_t e, const char* where) {
        free_game(g);
        return cuda_fail(ctx, e, where);
    };
#define LS_TRY(expr)                                   \
    do {                                               \
        cudaError_t _e = (expr);                       \
        if (_e != cudaSuccess) return bail(_e, #expr); \
    } while (0)
    auto A = [&](auto** p, size_t count) { return dev_alloc(ctx, (void**)p, sizeof(**p) * count, s); };
    LS_TRY(A(&g->off, 2 * N + 2));
    LS_TRY(A(&g->tgt, M + N));
    LS_TRY(A(&g->flags, 2 * N + 1));
    LS_TRY(A(&g->pri, 2 * N + 1));
    LS_TRY(A(&g->nid0, N));
    LS_TRY(A(&g->orig_of, 2 * N + 1));
    LS_TRY(A(&g->dnid, N));
    LS_TRY(A(&g->dummy_of, N));
    LS_TRY(A(&g->strat, 2 * N + 1));
    LS_TRY(A(&g->gsink, 1));
    LS_TRY(cudaMemsetAsync(t + o_st, 0, sizeof(LoadStatus), s));
    a.off = off;
    a.tgt = tgt;
    a.pri = pri;
    a.own = own;
    if (host) {
        LS_TRY(cudaMemcpyAsync(t + o_off, off, 4 * (N + 1), cudaMemcpyHostToDevice, s));
        LS_TRY(cudaMemcpyAsync(t + o_tgt, tgt, 4 * M, cudaMemcpyHostToDevice, s));
        LS_TRY(cudaMemcpyAsync(t + o_pri, pri, 4 * N, cudaMemcpyHostToDevice, s));
        LS_TRY(cudaMemcpyAsync(t + o_own, own, N, cudaMemcpyHostToDevice, s));
        a.off = (int32_t*)(t + o_off);
        a.tgt = (int32_t*)(t + o_tgt);
        a.pri = (int32_t*)(t + o_pri);
        a.own = (uint8_t*)(t + o_own);
    }
    a.st = (LoadStatus*)(t + o_st);
    a.indeg = (int32_t*)(t + o_ind);
    a.roff = (int32_t*)(t + o_roff);
    a.radj = (int32_t*)(t + o_radj);
    a.left = (int32_t*)(t + o_left);
    a.fa = (int32_t*)(t + o_fa);
    a.fb = (int32_t*)(t + o_fb);
    a.widx = (int32_t*)(t + o_widx);
    a.gid = (int32_t*)(t + o_gid);
    a.wprefix = (int32_t*)(t + o_wp);
    a.nidu = (int32_t*)(t + o_nidu);
    a.inU = (uint8_t*)(t + o_inU);
    a.isW = (uint8_t*)(t + o_isW);
    a.bits = (uint32_t*)(t + o_bits);
    a.tiles = (int64_t*)(t + o_tiles);
    a.goff = g->off;
    a.gtgt = g->tgt;
    a.gpri = g->pri;
    a.nid0 = g->nid0;
    a.orig_of = g->orig_of;
    a.dnid = g->dnid;
    a.dummy_of = g->dummy_of;
    a.strat = g->strat;
    a.gsink = g->gsink;
    a.gflags = g->flags;
    if (n > kLoadCluster) {
        int sms = 0;
        LS_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
        const int blocks = std::max(1, std::min({sms, kLsBlocks, (n + kLsThreads - 1) / kLsThreads}));
        void* args[] = {(void*)&a};
        LS_TRY(cudaLaunchCooperativeKernel((void*)k_load_small<true>, blocks, kLsThreads, args, 0, s));
    } else {
        int c = kLsCluster;
        while (c > 1 && (int64_t)c * kLsThreads / 2 >= n) c >>= 1;
        c = std::min(c, cluster_blocks((const void*)k_load_small<false>, kLsThreads, 0, kLsCluster, ctx->device,
                                       g_ls_cluster));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kLsThreads);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = c;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        LS_TRY(cudaLaunchKernelEx(&cfg, k_load_small<false>, a));
    }
    ctx->launches += 1;
    LoadStatus h;
    LS_TRY(cudaMemcpyAsync(&h, a.st, sizeof(h), cudaMemcpyDeviceToHost, s));
    LS_TRY(cudaStreamSynchronize(s));
#undef LS_TRY
    if (h.c.err) {
        free_game(g);
        return fail(ctx, PG_ECUDA, "pg_load_csr: a grid barrier timed out");
    }
    if (h.general) {
        free_game(g);
        return PG_OK;
    }
    g->n0 = n;
    g->m0 = m;
    g->k = h.k;
    g->n = n + h.k + 1;  // G' vertices and the sink slot
    g->m = m + h.k;
    g->sink0 = n + h.k;
    g->ngames = 1;
    g->h_base0 = {0, (int64_t)n};
    g->h_dbase = {0, h.k};
    *general = false;
    *out = g;
    return PG_OK;
}

}  // namespace pg
