// Incremental iterations of the compare-mode loop: for one game, and for all games of a small batch at once.
//
// After a switching pass only vertices whose play passes a switched vertex
// can change their valuation (Section 3: a valuation is a function of the
// play). Past the first iterations of a best response these are few: on the
// 10M-vertex random game (G': 13.3M vertices) 23% and 3% of the vertices in
// the first two iterations, under 0.1% from the fourth on, and after an Even
// switch 50%, 27%, 5%, 1%, 0.2%, ... k_inc therefore runs whole iterations of
// Algorithm 1 on that set alone:
//   closure   A = the switched vertices and everything upstream of them in the
//             strategy graph, found through the reverse adjacency of G' (a
//             predecessor y of x belongs to x's tree when strat[y] = x); the
//             g-word of each becomes a one-step jump pointer
//   resolve   nearest greater vertices of A by walking jump pointers inside A
//             and g-chains outside it, in rounds
//   classify  class and top of A from the g-chains; predecessors of a vertex
//             whose top changed, and predecessors whose last decision compared
//             chains (their tie mark), are queued for their player
//   switch    Odd's queue, or Even's when Odd had nothing to switch, with the
//             rules of k_switch_cmp_pl
// so that the decisions, and with them the trajectory, are those of full
// iterations. One thread-block cluster runs all of them in one launch: an
// iteration is a chain of dependent reads whatever its size, so what counts is
// the number of dependent reads and barriers, not throughput. Every block keeps
// its share of A, of the queues and of the switched vertices in its shared
// memory (a vertex stays with the block that found it; a closure level costs a
// block barrier, and its two dependent reads are the predecessors and, issued
// together, their strategies, words and own list bounds); the blocks meet at
// the hardware cluster barrier (about 0.3 us) after each step and pass their
// counts through distributed shared memory. Random games, load and solve,
// before and after (full iterations only; then these): 1k vertices 2.26 -> 1.11
// ms, 30k 2.94 -> 1.76, 1M 5.05 -> 4.23, 10M 29.5 -> 23.1; the 10M ladder 43.0
// -> 29.4 ms.
#include <cooperative_groups.h>

#include "pg_device.cuh"

namespace cg = cooperative_groups;

namespace pg {
namespace {

constexpr int kIncThreads = 1024;
constexpr int kIncCluster = 16;      // blocks of the cluster (non-portable size; fewer when the device refuses it)
constexpr int kIncSet = 10240;       // vertices of A a block holds
constexpr int kIncQueue = 8192;      // Odd's queue of a block (the rest spills to global memory)
constexpr int kIncEven = 16384;      // Even's queue of a block (beyond it Even's next pass is full)
constexpr int kIncFanIn = 1024;      // a vertex of A with more predecessors ends the incremental iteration
constexpr int kIncRounds = 128;      // rounds of the resolution
constexpr int kIncWalk = 256;        // count-vector mode: steps of a play inside A
constexpr int kIncSteps = 128;       // steps of one resolution round
// A block has kIncThreads / div threads and that share of the lists.
constexpr size_t inc_shared(int div) { return sizeof(int32_t) * (3 * kIncSet + kIncQueue + kIncEven) / div; }
constexpr size_t kIncShared = inc_shared(1);
constexpr int32_t kIncBig = 1 << 24;  // (16 blocks' counts sum below 2^31)
// A full iteration follows a pass that switched more vertices than this. Large
// games: against 270 us for a full iteration of the 10M random game, an
// incremental one took 102 us from 7.4k switched vertices, 425 us from 11.8k
// and 1,025 us from 27.9k; against 62 us on the 1M game, 48 us from 1.3k and
// 125 us from 4.7k.
constexpr int kIncSeedShare = 1024, kIncSeeds = 8192;
// Count-vector games, against 310 us for a full iteration of the 3M-vertex game
// with 4 priorities: 72 us from 5.8k switched vertices, 126 us from 12.6k
// (350 us and more from 8-15k when their trees are deep).
constexpr int kIncSeedShareCv = 256, kIncSeedsCv = 16384;
// Small count-vector games gain least: their full iterations take 40 us, best
// responses end after a few, and the ones below bring that down. Even's pass over
// all ids is run in k_inc (5 us; as the next body of the graph 20 us), the cluster
// has no more blocks than the game has use for, the classes of the outputs come
// from the keys unless a full valuation has them (40 us), and best responses have
// a third of the budget. Solves and best responses of 45 games of 1k to 30k
// vertices, 4 priorities, against full iterations alone: before these 0.67 to 1.35
// and 0.82 to 1.33 of the time, now 0.61 to 1.19 and 0.73 to 1.17.
// In a launch that runs the whole loop (41k ids): an iteration over all ids
// takes 17-32 us, an incremental one 13 us (a few switched vertices) to 35 us
// (a hundred, for the levels of the closure).
constexpr int kIncWholeShare = 512;

// Packed games (GAMES): a cluster for each game runs the game's whole loop over
// its range of ids, all games at once. Against the lockstep loop, whose
// iterations take 50 us at least, as many as the slowest game needs: 608 games
// of 500 vertices 2.6 -> 0.8 ms, of 2,000 vertices 3.9 -> 2.4; 100 of 9,000
// (12k ids) 3.9 -> 2.7; 19 and 9 of 20,000 (several blocks each) 3.5 -> 2.0 and
// 3.1 -> 1.6. An SM moves a sector or two per clock and the loop reads its words
// at random, so this holds while an SM has few ids: 150 games of 12,000 (16k
// ids) take 5.8 ms against 5.7, 152 of 100,000 44 against 30. The route is taken
// when every game can run at once with at most kIncBlockIds ids for an SM.
constexpr int kIncSmallDiv = 4;              // blocks of a quarter of the threads, four to an SM
constexpr int32_t kIncBlockIds = 12800;      // (a block of 1,024 threads; a quarter for the small ones)
// A full iteration follows a pass that switched more than this part of a packed
// game: a 32nd, 64th, 200th: 2.3, 2.5, 2.7 ms (608 games of 2,000), 2.5, 2.3,
// 2.3 ms (9 games of 20,000).
constexpr int kIncGameShare = 64;

// A closure that takes too long is abandoned, and a full iteration follows. The
// budget counts vertices that a block has found (45 ns each) and levels, which
// take as long as 44 of them (2 us). It is about two full iterations of a game
// whose plays are short: these take 45 us and 17 us per million ids, 45 and 62
// with keys; over all ids in one launch it is one, 16 us and 1 us per 128 ids of a
// block. (A third less: 300k vertices 5.97 ms, so 5.89; 400k ladder 5.41 and 5.27;
// 663k with 4 priorities 14.5 and 14.0.) Where plays are long (a torus, a ring with
// chords) half of the attempts went on to 256 levels, or to as many vertices as a
// block holds, 260 us (200k vertices) to 600 us (4M), for nothing. Solving a torus
// of 4M vertices by full iterations, by these attempts, and with the budget and
// the waits: 1,324, 2,254 and 1,298 ms; a ring of 4M 5,299, 8,735 and 5,510; a
// torus of 200k 180, 185 and 156; a random game of 1M 6.7, 5.1 and 5.1.
constexpr int32_t kIncLevelCost = 44;
// An abandoned attempt is followed by 1 full iteration; by 2, 4, ... 32 while they keep failing.
constexpr int32_t kIncFails = 5;

struct IncArgs {
    int32_t n;       // ids, the sink slot included
    int32_t sink0;
    const int32_t* off;
    const int32_t* tgt;
    const uint8_t* flags;
    const int2* rv;
    const int32_t* rv_src;
    int32_t* strat;
    uint32_t* gd32;
    uint32_t* topw;
    uint8_t* omark;
    uint8_t* emark;
    const int32_t* alist;  // the switched vertices of the last full pass (cnt->n_list of them)
    int32_t* qlist;        // [n] Odd's queue beyond the blocks' own
    GameState* gst;
    Counters* cnt;
    IncState* st;
    int32_t* n_q;          // its length (GAMES: one per game)
    const int2* games;     // GAMES: first id and index of each cluster's game,
    const int32_t* gsink;  //    and the games' sinks
    int32_t* gactive;
    int64_t* loop_iters;
    i128* key;   // count-vector mode: the keys, and the levels they count
    Levels lev;
    int64_t cap;
    int32_t max_seeds;  // more switched vertices than this take a full iteration
    int32_t budget;     // of a block's closure (kIncLevelCost)
    int32_t whole;      // 1: the launch runs the whole loop, full iterations included (over all ids)
    int32_t even_here;  // 1: Even's passes over all ids are run here too
    int32_t even;       // 0: best response (the inner loop only)
    int32_t reset;      // SI-Reset
    int32_t deep_cut;
    int32_t deep_fallback;
};

// (a launch that runs the whole loop, by its ids and blocks; inc_budget: a launch after a full iteration)
__host__ __device__ inline int32_t inc_budget_whole(int32_t ids, int32_t blocks) {
    return kIncLevelCost * (16 + ids / (128 * blocks));
}

// Sets bit b of byte p (in a 4-byte aligned array); returns whether it was clear.
__device__ inline bool claim_byte(uint8_t* base, int32_t i, uint32_t b) {
    const uint32_t sh = 8u * (uint32_t)(i & 3);
    return !((atomicOr((uint32_t*)base + (i >> 2), b << sh) >> sh) & b);
}

// Decision of one vertex (the rules of k_switch_cmp): returns whether it
// switched; *tie_out: the decision compared the chains of two finite
// successors.
template <int PLAYER>
__device__ inline bool inc_switch(const IncArgs& a, int32_t v, bool* tie_out) {
    const int32_t* tgt = a.tgt + a.off[v];
    const int32_t deg = a.off[v + 1] - a.off[v];
    const int32_t cur = __ldcg(a.strat + v);
    int32_t best = PLAYER == 0 ? a.sink0 : -1;
    uint32_t tbest = 0;
    bool cur_top = false, tie = false;
    for (int32_t e = 0; e < deg; e += 4) {
        int32_t t[4];
        uint32_t tt[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = e + j < deg ? tgt[e + j] : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) tt[j] = t[j] >= 0 ? __ldcg(a.topw + t[j]) : 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (t[j] < 0) continue;
            const bool first = PLAYER == 0 ? best == a.sink0 : best < 0;
            if (PLAYER == 0 && t[j] == cur) cur_top = (tt[j] & kG32Top) != 0;
            tie |= !first && !((tt[j] | tbest) & kG32Top) && top_id(tt[j]) == top_id(tbest);
            bool take;
            if (PLAYER == 1) take = first || cmp_val<true>(t[j], tt[j], best, tbest, a.gd32, a.flags) < 0;
            else take = (first ? cmp_sink(tt[j]) : cmp_val<true>(t[j], tt[j], best, tbest, a.gd32, a.flags)) > 0;
            if (take) {
                best = t[j];
                tbest = tt[j];
            }
        }
    }
    *tie_out = tie;
    const bool sw = best != cur && (PLAYER == 0 ? !cur_top : !(tbest & kG32Top));
    if (sw) __stcg(a.strat + v, best);
    return sw;
}

__device__ inline i128 ld_key(const i128* p) {
    const longlong2 w = __ldcg(reinterpret_cast<const longlong2*>(p));
    return (i128)w.y << 64 | (unsigned long long)w.x;
}
__device__ inline void st_key(i128* p, i128 k) {
    __stcg(reinterpret_cast<longlong2*>(p), make_longlong2((long long)k, (long long)(k >> 64)));
}

// Decision of one vertex on keys (the rules of k_switch_cv).
template <int PLAYER>
__device__ inline bool inc_switch_cv(const IncArgs& a, int32_t v) {
    const int32_t* tgt = a.tgt + a.off[v];
    const int32_t deg = a.off[v + 1] - a.off[v];
    const int32_t cur = __ldcg(a.strat + v);
    const i128 curkey = ld_key(a.key + cur);
    int32_t best = PLAYER == 0 ? a.sink0 : -1;
    i128 bk = 0;  // (the sink's key: the empty count vector)
    for (int32_t e = 0; e < deg; e += 4) {
        int32_t t[4];
        i128 k[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = e + j < deg ? tgt[e + j] : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j) k[j] = t[j] >= 0 ? ld_key(a.key + t[j]) : (i128)0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (t[j] < 0 || !(PLAYER == 0 ? k[j] > bk : (best < 0 || k[j] < bk))) continue;
            best = t[j];
            bk = k[j];
        }
    }
    const bool sw = PLAYER == 0 ? bk > curkey : bk < curkey;
    if (sw) __stcg(a.strat + v, best);
    return sw;
}

// Key of a vertex of A (its word is pending): the weights along its play as far
// as the play stays in A, plus the key of the first vertex outside. A play that
// stays in A forever ends in a cycle (Brent's method finds it): TOP, and *odd
// when the cycle's largest vertex is. *cut: the play is longer than kIncWalk.
__device__ inline i128 inc_key(const IncArgs& a, int32_t v, bool* odd, bool* cut) {
    i128 acc = weight_of(a.lev, v);
    int32_t x = g32_ptr(__ldcg(a.gd32 + v)), mark = v;
    for (int32_t steps = 1, power = 1, lam = 0;; ++steps) {
        const uint32_t w = __ldcg(a.gd32 + x);
        if (!g32_pending(w)) {
            const i128 k = ld_key(a.key + x);
            return k == top_key() ? k : acc + k;
        }
        if (x == mark) break;
        if (steps >= kIncWalk) {
            *cut = true;
            return 0;
        }
        if (++lam == power) {
            mark = x;
            power *= 2;
            lam = 0;
        }
        acc += weight_of(a.lev, x);
        x = g32_ptr(w);
    }
    int32_t big = x;
    for (int32_t y = g32_ptr(__ldcg(a.gd32 + x)); y != x; y = g32_ptr(__ldcg(a.gd32 + y))) big = max(big, y);
    if (a.flags[big] & kPriOdd) *odd = true;
    return top_key();
}

// Queues the predecessors of la[i] that want it (all of them if changed, else
// those with a tie mark) for their player.
template <int DIV>
__device__ inline void inc_queue(const IncArgs& a, int32_t e0, int32_t nodd, int32_t deg, bool changed, int32_t* lq,
                                 int32_t* c_q, int32_t* le, int32_t* c_e) {
    const int32_t* src = a.rv_src + e0;
    for (int32_t e = 0; e < deg; e += 4) {
        int32_t y[4];
        bool want[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = e + j < deg ? src[e + j] : -1;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            want[j] = y[j] >= 0 && (changed || (__ldcg((e + j < nodd ? a.omark : a.emark) + y[j]) & kMarkTie));
#pragma unroll
        for (int j = 0; j < 4; ++j)
            want[j] = want[j] && claim_byte(e + j < nodd ? a.omark : a.emark, y[j], kMarkQueued);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (!want[j]) continue;
            if (e + j < nodd) {
                const int32_t p = atomicAdd(c_q, 1);
                if (p < kIncQueue / DIV) lq[p] = y[j];
                else __stcg(a.qlist + atomicAdd(a.n_q, 1), y[j]);
            } else {
                const int32_t p = atomicAdd(c_e, 1);
                if (p < kIncEven / DIV) le[p] = y[j];
            }
        }
    }
}

// CV: count-vector mode (repeated priorities). A valuation is a key summed along
// the play, so the g-words only tell who is in A, and decisions compare keys
// (no tie marks); full iterations are not run here. 3M vertices, 4 priorities, load and solve: 30.5 -> 15.0 ms.
template <bool CV, int DIV, bool GAMES>
__global__ void __launch_bounds__(kIncThreads / DIV, DIV) k_inc(IncArgs a) {
    constexpr int TH = kIncThreads / DIV, SET = kIncSet / DIV, QUEUE = kIncQueue / DIV, EVEN = kIncEven / DIV;
    cg::cluster_group cl = cg::this_cluster();
    const int32_t CL = (int32_t)cl.num_blocks(), rank = (int32_t)cl.block_rank(), tid = threadIdx.x;
    const int32_t T = CL * TH, t0 = rank * TH + tid;
    int32_t lo0 = 0;  // the first id
    if constexpr (GAMES) {
        const int2 game = a.games[blockIdx.x / CL];
        lo0 = game.x;
        a.sink0 = a.gsink[game.y];
        a.n = a.sink0 + 1;
        a.max_seeds = min(max(1, (a.n - lo0) / kIncGameShare), CL * (SET / 2));
        a.budget = inc_budget_whole(a.n - lo0, CL);
        a.gst += game.y;
        a.n_q += game.y;
        a.qlist += lo0;
    }
    const auto whole = [&] { return GAMES || a.whole; };
    extern __shared__ int32_t dyn[];
    int32_t* la = dyn;             // this block's part of A: vertex,
    int32_t* ls = la + SET;    //    start of its predecessors,
    int32_t* lc = ls + SET;    //    their number << 16 | Odd's among them
    int32_t* lq = lc + SET;    // its part of Odd's queue
    int32_t* le = lq + QUEUE;  //    and of Even's
    __shared__ int2 xb[2][kIncCluster];
    __shared__ int32_t lvl[3], c_bad, c_left, c_q, c_odd, c_s, c_e, c_zero;
    // incremental iterations: none for the next p_wait iterations, p_fails abandoned in a row, p_since done since
    __shared__ int32_t p_wait, p_fails, p_since;
    int par = 0;
    // The sums over the cluster of two counts, final in each block when all its threads call: every block stores
    // its pair in every block's shared memory and sums after the barrier. Two buffers in turn: a block that is
    // ahead writes the other one.
    auto exchange = [&](const int32_t* pa, const int32_t* pb) {
        __syncthreads();
        if (tid < CL) cl.map_shared_rank(&xb[par][0], tid)[rank] = make_int2(*pa, *pb);
        cl.sync();
        int2 sum = make_int2(0, 0);
        for (int i = 0; i < CL; ++i) {
            const int2 x = xb[par][i];
            sum.x += x.x;
            sum.y += x.y;
        }
        par ^= 1;
        return sum;
    };
    // every decision below is taken by all threads from sums that they share, so the cluster stays uniform
    GameState gs;
    gs.phase = __ldcg(&a.gst->phase);
    gs.inner = __ldcg(&a.gst->inner);
    gs.major = __ldcg(&a.gst->major);
    const bool dead = (!GAMES && (__ldcg(&a.cnt->err) || __ldcg(&a.cnt->deep))) || gs.phase != kPhaseActive;
    // every Odd vertex is evaluated (the first iteration, or after an SI-Reset: gactive[1], set by k_bookkeep)
    bool fresh = whole() || __ldcg(a.gactive + 1);
    bool even_full = whole() || __ldcg(&a.st->even_full);
    int32_t ns = fresh ? 0 : __ldcg(&a.cnt->n_list);  // switched vertices, all blocks
    const int32_t wait = whole() ? 0 : __ldcg(&a.st->wait), fails = whole() ? 0 : __ldcg(&a.st->fails);
    // nothing to do here (the state stays as k_bookkeep left it: a full iteration is next)
    if (dead || (!whole() && (fresh || ns > a.max_seeds || wait > 0))) return;
    int32_t nsl = ns > rank ? (ns - rank + CL - 1) / CL : 0;  // this block's, in la
    for (int32_t i = tid; i < nsl; i += TH) la[i] = __ldcg(a.alist + rank + i * CL);
    if (tid == 0) {
        c_e = c_zero = p_wait = p_since = 0;
        p_fails = fails;
    }
    int32_t mode = kIncFull, iters = 0;
    bool done = false;
    auto abandoned = [&] {  // (by one thread of each block, where a barrier follows)
        if (p_since > 1) p_fails = 0;
        p_wait = 1 << p_fails;
        p_fails = min(p_fails + 1, kIncFails);
        p_since = 0;
    };
    cl.sync();
    while (!done) {
        bool all = fresh || ns > a.max_seeds;
        if (all && !whole()) break;
        all |= p_wait > 0;
        if (tid == 0) {
            c_bad = c_left = c_q = c_odd = 0;
            lvl[1] = 0;
        }
        if (t0 == 0) *a.n_q = 0;
        __syncthreads();
        int32_t na = nsl;
        if (!all) {
            for (int32_t i = tid; i < nsl; i += TH) {
                const int32_t v = la[i];
                const int2 r = a.rv[v];
                const int32_t k = a.rv[v + 1].x - r.x;
                __stcg(a.gd32 + v, kG32Pend | (uint32_t)__ldcg(a.strat + v));
                ls[i] = r.x;
                lc[i] = k << 16 | ((r.y - r.x) & 0xffff);
                if (k > kIncFanIn) c_bad = 1;
            }
            cl.sync();
            // level r expands la[lo .. na) into la[na ..]; lvl[] rotates, so a count is stable while it is read. A
            // level that cannot be held (kIncBig) or that passes the budget ends the closure.
            bool bad = c_bad != 0;
            int32_t lo = 0;
            for (int32_t r = 0; !bad && lo < na; ++r) {
                int32_t* next = &lvl[(r + 1) % 3];
                if (tid == 0) lvl[(r + 2) % 3] = 0;
                for (int32_t i = lo + tid; i < na; i += TH) {
                    const int32_t x = la[i], deg = lc[i] >> 16;
                    const int32_t* src = a.rv_src + ls[i];
                    for (int32_t e = 0; e < deg; e += 4) {
                        int32_t y[4], s[4], r1[4];
                        uint32_t w[4];
                        int2 r0[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) y[j] = e + j < deg ? src[e + j] : x;  // (x: not below itself)
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            s[j] = __ldcg(a.strat + y[j]);
                            w[j] = __ldcg(a.gd32 + y[j]);
                            r0[j] = a.rv[y[j]];
                            r1[j] = a.rv[y[j] + 1].x;
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            // one thread reads all of x's predecessors: a repeated edge shows in its own earlier
                            // write, or inside this group of four
                            bool in = s[j] == x && !g32_pending(w[j]);
#pragma unroll
                            for (int q = 0; q < j; ++q) in = in && y[q] != y[j];
                            if (!in) continue;
                            __stcg(a.gd32 + y[j], kG32Pend | (uint32_t)x);
                            const int32_t p = na + atomicAdd(next, 1), k = r1[j] - r0[j].x;
                            if (p >= SET || k > kIncFanIn) {
                                atomicOr(next, kIncBig);
                                continue;
                            }
                            la[p] = y[j];
                            ls[p] = r0[j].x;
                            lc[p] = k << 16 | (r0[j].y - r0[j].x);
                        }
                    }
                }
                __syncthreads();
                const int32_t found = *next;
                bad = found >= kIncBig || (r + 1) * kIncLevelCost + na + found > a.budget;
                lo = na;
                if (!bad) na += found;
            }
            if (bad && tid == 0) c_bad = 1;
            all = exchange(&c_bad, &c_zero).x != 0;
            if (all && tid == 0) abandoned();
            if (all && !whole()) break;
        }
        if (all) {
            even_full = true;
            if (tid == 0) c_bad = 0;
            for (int32_t v = lo0 + t0; v < a.n; v += T)
                __stcg(a.gd32 + v, v == a.sink0 ? kG32Sink : kG32Pend | (uint32_t)__ldcg(a.strat + v));
            cl.sync();
        }
        // ids [i0, i1) in steps of st are this thread's, or la[i] of them
        const int32_t i0 = all ? lo0 + t0 : tid, i1 = all ? a.n : na, step = all ? T : TH;
        bool unresolved = false;
        if constexpr (CV) {
            for (int32_t i = tid; i < na; i += TH) {
                const int32_t v = la[i];
                const i128 old = ld_key(a.key + v);
                bool odd = false, cut = false;
                const i128 k = inc_key(a, v, &odd, &cut);
                if (odd) c_odd = 1;
                if (cut) {
                    c_left = 1;
                    continue;
                }
                const int32_t nodd = lc[i] & 0xffff;
                if (k == old) continue;
                // (a key outside A is never this one: it may change while other plays are walked)
                st_key(a.key + v, k);
                inc_queue<DIV>(a, ls[i], nodd, even_full ? nodd : lc[i] >> 16, true, lq, &c_q, le, &c_e);
            }
            unresolved = exchange(&c_left, &c_zero).x != 0;
            for (int32_t i = tid; i < na; i += TH) __stcg(a.gd32 + la[i], kG32None);  // no longer in A
            if (unresolved) {  // Odd's queue is dropped (Even's: its next pass is full)
                const int32_t nq = min(c_q, QUEUE), spill = __ldcg(a.n_q);
                for (int32_t i = tid; i < nq; i += TH) a.omark[lq[i]] = 0;
                for (int32_t i = t0; i < spill; i += T) a.omark[__ldcg(a.qlist + i)] = 0;
            }
        } else {
            // resolve: words of A turn from jump pointers into g-words; any word read is valid whenever it is read
            for (int32_t r = 0;; ++r) {
                int32_t left = 0;
                for (int32_t i = i0; i < i1; i += step) {
                    const int32_t v = all ? i : la[i];
                    const uint32_t w = __ldcg(a.gd32 + v);
                    if (!g32_pending(w)) continue;
                    int32_t x = g32_ptr(w);
                    bool top = false;
                    for (int k = 0; k < kIncSteps && x < v; ++k) {
                        const uint32_t wx = __ldcg(a.gd32 + x);
                        if (g32_none(wx) && !g32_pending(wx)) {  // TOP: v's play ends in the same cycle
                            top = true;
                            break;
                        }
                        x = g32_sink(wx) && !g32_pending(wx) ? a.sink0 : g32_ptr(wx);
                    }
                    uint32_t nw;
                    if (top) nw = kG32None | (uint32_t)a.sink0;  // (a pointer that no cycle maximum has)
                    else if (x > v) nw = x == a.sink0 ? g32_sink_word(a.flags[v]) : (uint32_t)x;
                    else if (x == v) nw = kG32None | (uint32_t)v;
                    else {
                        nw = kG32Pend | (uint32_t)x;
                        left = 1;
                    }
                    __stcg(a.gd32 + v, nw);
                }
                if (left) c_left = 1;
                const int32_t rem = exchange(&c_left, &c_zero).x;
                if (rem == 0) break;
                if (r + 1 >= kIncRounds) {
                    unresolved = true;
                    break;
                }
                if (tid == 0) c_left = 0;
                __syncthreads();
            }
        }
        if (unresolved) {
            if (!all && tid == 0) abandoned();
            if (!whole()) break;  // the full iteration decides
            if (!all) {  // over all ids once
                ns = a.n;
                __syncthreads();
                continue;
            }
            if (!GAMES && t0 == 0) {  // (a packed game stays active)
                if (a.deep_fallback) a.cnt->deep = 1;
                else atomicOr(&a.cnt->err, kErrJumpRounds);
            }
            ++iters;
            break;
        }
        if constexpr (!CV) {
            // classify (as k_classify)
            for (int32_t i = i0; i < i1; i += step) {
                const int32_t v = all ? i : la[i];
                const uint32_t w0 = __ldcg(a.gd32 + v), old = all ? 0u : __ldcg(a.topw + v);
                int32_t x = g32_sink(w0) ? v : g32_ptr(w0);
                bool top = g32_none(w0), odd = g32_sink(w0) && (w0 & 1u);
                if (top && x == v && (a.flags[v] & kPriOdd)) c_odd = 1;
                if (!top && !g32_sink(w0)) {
                    for (int32_t len = 1;; ++len) {
                        if (len > a.deep_cut) {  // a deep forest: the iteration is abandoned
                            c_bad = 1;
                            break;
                        }
                        const uint32_t wx = __ldcg(a.gd32 + x);
                        if (wx & kG32Top) {
                            top = true;
                            break;
                        }
                        if (g32_sink(wx)) {
                            odd = wx & 1u;
                            break;
                        }
                        const int32_t nx = g32_ptr(wx);
                        if (nx <= x) break;  // g-chains rise (a guard, never taken)
                        x = nx;
                    }
                    if (top) __stcg(a.gd32 + v, w0 | kG32Top);
                }
                const uint32_t tw = top ? kG32Top : (odd ? kTopOdd : 0u) | (uint32_t)x;
                if (all) {  // everyone is evaluated: no queues
                    __stcg(a.topw + v, tw);
                    continue;
                }
                const bool changed = tw != old;
                if (changed) __stcg(a.topw + v, tw);
                const int32_t nodd = lc[i] & 0xffff;
                inc_queue<DIV>(a, ls[i], nodd, even_full ? nodd : lc[i] >> 16, changed, lq, &c_q, le, &c_e);
            }
        }
        if (tid == 0) {
            c_s = 0;
            if (all) p_wait -= p_wait > 0;
            else ++p_since;
        }
        const int2 bad_odd = exchange(&c_bad, &c_odd);
        if (bad_odd.x) {  // the iteration is abandoned
            if (!GAMES && t0 == 0) a.cnt->deep = 1;
            ++iters;
            break;
        }
        // Odd's pass; the switched vertices are the next iteration's seeds
        auto odd_vertex = [&](int32_t v) {
            bool tie = false;
            const bool sw = CV ? inc_switch_cv<1>(a, v) : inc_switch<1>(a, v, &tie);
            a.omark[v] = tie ? kMarkTie : 0;
            if (!sw) return;
            const int32_t p = atomicAdd(&c_s, 1);
            if (p < SET) la[p] = v;
        };
        if (all) {
            for (int32_t v = lo0 + t0; v < a.n; v += T)
                if ((a.flags[v] & (kOwnerOdd | kSinkSlot)) == kOwnerOdd) odd_vertex(v);
        } else {
            const int32_t nq = min(c_q, QUEUE), spill = __ldcg(a.n_q);
            for (int32_t i = tid; i < nq; i += TH) odd_vertex(lq[i]);
            for (int32_t i = t0; i < spill; i += T) odd_vertex(__ldcg(a.qlist + i));
        }
        // (a block that switched more than it can hold makes the next iteration a full one)
        __syncthreads();
        if (tid == 0 && c_s > SET) c_s = kIncBig;
        if (tid == 0) c_bad = c_e > EVEN;
        const int2 odd_sum = exchange(&c_s, &c_bad);
        ns = odd_sum.x;
        nsl = c_s;
        even_full |= odd_sum.y != 0;
        int32_t nse = 0;
        if (ns == 0 && a.even) {
            if (!whole() && ((even_full && !a.even_here) || a.reset)) {  // Even's pass over its view counts this one
                mode = kIncEvenOnly;
                if (t0 == 0 && bad_odd.y) a.gst->nodd = 1;
                break;
            }
            auto even_vertex = [&](int32_t v) {
                bool tie = false;
                const bool sw = CV ? inc_switch_cv<0>(a, v) : inc_switch<0>(a, v, &tie);
                a.emark[v] = tie ? kMarkTie : 0;
                if (!sw) return;
                const int32_t p = atomicAdd(&c_s, 1);
                if (p < SET) la[p] = v;
            };
            if (even_full) {
                for (int32_t v = lo0 + t0; v < a.n; v += T)
                    if (!(a.flags[v] & (kOwnerOdd | kSinkSlot))) even_vertex(v);
            } else {
                for (int32_t i = tid; i < c_e; i += TH) even_vertex(le[i]);
            }
            __syncthreads();
            if (tid == 0 && c_s > SET) c_s = kIncBig;
            nse = exchange(&c_s, &c_zero).x;
            nsl = c_s;
            even_full = false;
            __syncthreads();
            if (tid == 0) c_e = 0;
        }
        // bookkeeping (as k_bookkeep)
        fresh = false;
        ++iters;
        ++gs.inner;
        if (bad_odd.y) gs.phase = kPhaseOddCycle;
        else if (ns == 0) {
            if (nse == 0) gs.phase = kPhaseDone;
            else {
                ++gs.major;
                ns = nse;
                if (a.reset) {  // Odd restarts from its first edges
                    for (int32_t v = lo0 + t0; v < a.n; v += T)
                        if ((a.flags[v] & (kOwnerOdd | kSinkSlot)) == kOwnerOdd) __stcg(a.strat + v, a.tgt[a.off[v]]);
                    fresh = true;
                    cl.sync();
                }
            }
        }
        if (gs.phase == kPhaseActive && gs.inner >= a.cap) gs.phase = kPhaseTimeout;
        done = gs.phase != kPhaseActive;
    }
    cl.sync();  // no block writes this one's shared memory, or reads the state below, any more
    if (t0 == 0) {
        a.gst->phase = gs.phase;
        a.gst->inner = gs.inner;
        a.gst->major = gs.major;
        a.gst->sw_odd = a.gst->sw_even = a.gst->reset = 0;
        if (GAMES) return;
        a.gactive[0] = gs.phase == kPhaseActive;
        a.st->mode = mode;
        a.st->even_full = even_full;
        a.st->wait = p_wait;
        a.st->fails = p_since > 1 ? 0 : p_fails;
        if (p_since) a.st->stale = 1;
        *a.loop_iters += iters;
    }
}

// Both passes over the edges below take the targets in [lo, hi) only. Their
// counters and lists are written at random, a whole sector moved for 4 bytes
// when they miss the L2 cache, so a large game takes several passes, each over a
// range of targets whose counters and lists fit (build_reverse), and reads its
// edges in order once per pass. 10M ladder (82 MB of counters, 162 MB of
// counters and lists), count and fill: one pass 196 + 887 us, ranges of 16 MB
// 329 + 739, 32 MB 205 + 407, 48 MB 151 + 337, 64 MB 197 + 371.
constexpr size_t kRvBytes = 48 << 20;
// Every pass reads all edges, while one pass moves a sector per edge each way:
// random games of 20M and 40M vertices (11 and 21 ranges), load and solve, 44.6
// and 117.0 ms in ranges, 47.0 and 118.2 in one pass; more ranges are not worth
// it.
constexpr size_t kRvPasses = 24;

// In-degree of every id: all edges in the low half, Odd's in the high half.
__global__ void __launch_bounds__(kBlock) k_rv_count(int32_t n, const int32_t* __restrict__ off,
                                                     const int32_t* __restrict__ tgt,
                                                     const uint8_t* __restrict__ flags, int32_t lo, int32_t hi,
                                                     unsigned long long* __restrict__ deg) {
    for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const unsigned long long one = (flags[v] & kOwnerOdd) ? (1ull << 32) + 1ull : 1ull;
        const int32_t e1 = off[v + 1];
        for (int32_t e = off[v]; e < e1; ++e) {
            const int32_t t = tgt[e];
            if (t >= lo && t < hi) atomicAdd(deg + t, one);
        }
    }
}

// List bounds from the scanned in-degrees (start in rv[].x), and the fill
// cursors (Odd's, Even's) in place of the degrees.
__global__ void __launch_bounds__(kBlock) k_rv_bounds(int32_t n, const int32_t* __restrict__ start, uint64_t* deg,
                                                      int2* __restrict__ rv) {
    for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += gridDim.x * blockDim.x) {
        const int32_t s = start[v];
        const int2 r = make_int2(s, v < n ? s + (int32_t)(deg[v] >> 32) : s);
        rv[v] = r;
        if (v < n) reinterpret_cast<int2*>(deg)[v] = r;
    }
}

__global__ void __launch_bounds__(kBlock) k_rv_fill(int32_t n, const int32_t* __restrict__ off,
                                                    const int32_t* __restrict__ tgt,
                                                    const uint8_t* __restrict__ flags, int32_t lo, int32_t hi,
                                                    int2* __restrict__ cur, int32_t* __restrict__ rv_src) {
    for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const bool odd = (flags[v] & kOwnerOdd) != 0;
        const int64_t e1 = off[v + 1];
        for (int64_t e = off[v]; e < e1; e += 4) {  // four cursor steps in flight
            int32_t t[4], p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) t[j] = e + j < e1 ? tgt[e + j] : -1;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (t[j] >= lo && t[j] < hi) p[j] = atomicAdd(odd ? &cur[t[j]].x : &cur[t[j]].y, 1);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (t[j] >= lo && t[j] < hi) rv_src[p[j]] = v;
        }
    }
}

// Odd's edges alone (the marks of k_classify), from Odd's view, whose edges lie
// together: a server makes these lists again for every layout. Counting over all
// vertices instead, in 8-byte counters, made a round of a stream of 200 games/s
// 3% longer.
__global__ void __launch_bounds__(kBlock) k_rv_count_odd(int32_t m, const int32_t* __restrict__ ptgt,
                                                         int32_t* __restrict__ deg) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(deg + ptgt[e], 1);
}

__global__ void __launch_bounds__(kBlock) k_rv_bounds_odd(int32_t n, const int32_t* __restrict__ start,
                                                          int32_t* __restrict__ cur, int2* __restrict__ rv) {
    for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += gridDim.x * blockDim.x) {
        const int32_t s = start[v];
        rv[v] = make_int2(s, v < n ? start[v + 1] : s);
        if (v < n) cur[v] = s;
    }
}

__global__ void __launch_bounds__(kBlock) k_rv_fill_odd(int32_t np, const int32_t* __restrict__ vid,
                                                        const int32_t* __restrict__ poff,
                                                        const int32_t* __restrict__ ptgt, int32_t* __restrict__ cur,
                                                        int32_t* __restrict__ rv_src) {
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
        const int32_t e1 = poff[i + 1], v = vid[i];
        for (int32_t e = poff[i]; e < e1; ++e) rv_src[atomicAdd(cur + ptgt[e], 1)] = v;
    }
}

}  // namespace

bool inc_applies(const pg_game* g) { return !g->vgame && g->ngames == 1 && g->off != nullptr && !g->no_inc; }

void drop_reverse(pg_game* g) {
    g->rv_ok = false;
    for (void** q : {(void**)&g->rv, (void**)&g->rv_src, (void**)&g->omark, (void**)&g->emark}) {
        if (*q) cudaFreeAsync(*q, g->ctx->stream);
        *q = nullptr;
    }
}

static pg_status make_reverse(pg_game* g, int64_t odd_edges);

pg_status build_reverse(pg_game* g, int64_t odd_edges) {
    if (g->rv_ok) return PG_OK;
    drop_reverse(g);
    pg_status st = make_reverse(g, odd_edges);
    if (!st) {
        g->rv_ok = true;
        return PG_OK;
    }
    drop_reverse(g);
    if (st == PG_ENOMEM) cudaGetLastError();
    return st;
}

static pg_status make_reverse(pg_game* g, int64_t odd_edges) {
    pg_ctx* ctx = g->ctx;
    cudaStream_t s = ctx->stream;
    const int32_t n = g->n;
    // packed games take no incremental iterations: their lists hold Odd's edges only (odd_edges of them; Odd's view
    // is complete then)
    const int odd_only = inc_applies(g) || g->by_game ? 0 : 1;
    const size_t edges = (size_t)(odd_only ? odd_edges : g->m), mark_bytes = ((size_t)n + 16) & ~(size_t)15;
    PG_CUDA_TRY(ctx, dev_alloc(ctx, (void**)&g->rv, sizeof(int2) * ((size_t)n + 1), s));
    PG_CUDA_TRY(ctx, dev_alloc(ctx, (void**)&g->rv_src, sizeof(int32_t) * std::max<size_t>(edges, 1), s));
    PG_CUDA_TRY(ctx, dev_alloc(ctx, (void**)&g->omark, mark_bytes, s));
    PG_CUDA_TRY(ctx, cudaMemsetAsync(g->omark, 0, mark_bytes, s));
    if (!odd_only) {
        PG_CUDA_TRY(ctx, dev_alloc(ctx, (void**)&g->emark, mark_bytes, s));
        PG_CUDA_TRY(ctx, cudaMemsetAsync(g->emark, 0, mark_bytes, s));
        if (!g->inc && !g->by_game) PG_CUDA_TRY(ctx, dev_alloc(ctx, (void**)&g->inc, sizeof(IncState), s));
    }
    // the valuation's scratch is free before a loop: degrees and cursors in gd, the scan's output in coff
    unsigned long long* deg = (unsigned long long*)g->gd;
    const unsigned grid = grid_for(n);
    if (odd_only) {
        int32_t* cur = (int32_t*)g->gd;
        const int32_t np = (int32_t)g->pl_n[1], mp = (int32_t)odd_edges;
        PG_CUDA_TRY(ctx, cudaMemsetAsync(cur, 0, sizeof(int32_t) * (size_t)n, s));
        k_rv_count_odd<<<grid_for(std::max(mp, 1)), kBlock, 0, s>>>(mp, g->pl_tgt[1], cur);
        PG_CUDA_TRY(ctx, exclusive_scan_i32(cur, g->coff, n, nullptr, g->scan_tmp, g->scan_tmp_bytes, s));
        k_rv_bounds_odd<<<grid, kBlock, 0, s>>>(n, g->coff, cur, g->rv);
        k_rv_fill_odd<<<grid_for(std::max(np, 1)), kBlock, 0, s>>>(np, g->pl_vid[1], g->pl_off[1], g->pl_tgt[1], cur,
                                                                   g->rv_src);
        PG_CUDA_TRY(ctx, cudaGetLastError());
        ctx->launches += 6;
        return PG_OK;
    }
    PG_CUDA_TRY(ctx, cudaMemsetAsync(deg, 0, sizeof(uint64_t) * (size_t)n, s));
    auto ranges = [&](size_t bytes, auto&& pass) {
        const size_t want = (bytes + kRvBytes / 2) / kRvBytes;
        const int32_t np = want > kRvPasses || want < 1 ? 1 : (int32_t)want;
        for (int32_t i = 0; i < np; ++i)
            pass((int32_t)((int64_t)n * i / np), (int32_t)((int64_t)n * (i + 1) / np));
        ctx->launches += np;
    };
    ranges(sizeof(uint64_t) * (size_t)n, [&](int32_t lo, int32_t hi) {
        k_rv_count<<<grid, kBlock, 0, s>>>(n, g->off, g->tgt, g->flags, lo, hi, deg);
    });
    PG_CUDA_TRY(ctx, exclusive_scan_low32(g->gd, g->coff, n, g->scan_tmp, g->scan_tmp_bytes, s));
    k_rv_bounds<<<grid, kBlock, 0, s>>>(n, g->coff, g->gd, g->rv);
    ranges(sizeof(int2) * (size_t)n + sizeof(int32_t) * edges, [&](int32_t lo, int32_t hi) {
        k_rv_fill<<<grid, kBlock, 0, s>>>(n, g->off, g->tgt, g->flags, lo, hi, (int2*)g->gd, g->rv_src);
    });
    PG_CUDA_TRY(ctx, cudaGetLastError());
    ctx->launches += 4;
    return PG_OK;
}

static int32_t inc_budget(const pg_game* g, bool even) {
    const int64_t base = !g->cv ? 50 : even ? 66 : 12, per = !g->cv ? 20 : even ? 62 : 12;
    return kIncLevelCost * (int32_t)(base + g->n * per / 1000000);
}

int32_t inc_max_seeds(const pg_game* g) {
    return g->cv ? std::max(1, std::min(g->n / kIncSeedShareCv, kIncSeedsCv))
                 : std::max(1, std::min(g->n / kIncSeedShare, kIncSeeds));
}

static std::atomic<int> g_inc_cluster[2][kClusterDevices];

static IncArgs inc_args(const pg_game* g, int64_t cap, bool even) {
    IncArgs a = {};
    a.n = g->n;
    a.sink0 = g->sink0;
    a.off = g->off;
    a.tgt = g->tgt;
    a.flags = g->flags;
    a.rv = g->rv;
    a.rv_src = g->rv_src;
    a.strat = g->strat;
    a.gd32 = g->gd32;
    a.topw = (uint32_t*)g->wgt;
    a.omark = g->omark;
    a.emark = g->emark;
    // lists in the valuation's scratch, free during a loop
    a.alist = g->plist;
    a.qlist = g->hugelist;
    a.gst = g->gst;
    a.cnt = g->cnt;
    a.st = g->inc;
    a.n_q = g->inc ? &g->inc->n_q : nullptr;
    a.gactive = g->gactive;
    a.loop_iters = g->loop_iters;
    a.key = g->key128;
    a.lev = g->lev;
    a.cap = cap;
    a.even = even ? 1 : 0;
    a.reset = even && g->reset_tau ? 1 : 0;
    a.deep_cut = g->tune.deep_cut;
    a.deep_fallback = g->ctx->deep_fallback ? 1 : 0;
    return a;
}

struct IncLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    IncLaunch(int clusters, int c, int div, cudaStream_t s) {
        cfg.gridDim = dim3((unsigned)clusters * c);
        cfg.blockDim = dim3(kIncThreads / div);
        cfg.dynamicSmemBytes = inc_shared(div);
        cfg.stream = s;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = c;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};

pg_status enqueue_inc(pg_game* g, int64_t cap, bool even, bool whole) {
    pg_ctx* ctx = g->ctx;
    IncArgs a = inc_args(g, cap, even);
    a.whole = whole ? 1 : 0;
    a.even_here = g->n <= kIncWhole;
    int want = kIncCluster;
    if (whole || g->n <= kIncWhole)
        while (want > 1 && (int64_t)want * kIncThreads / 2 >= g->n) want >>= 1;  // (a small cluster starts sooner)
    auto kern = g->cv ? k_inc<true, 1, false> : k_inc<false, 1, false>;
    const int c = std::min(want, cluster_blocks((const void*)kern, kIncThreads, kIncShared, kIncCluster, g->device,
                                                g_inc_cluster[g->cv ? 1 : 0]));
    a.max_seeds = std::min(whole ? std::max(1, g->n / kIncWholeShare) : inc_max_seeds(g), c * (kIncSet / 2));
    a.budget = whole ? inc_budget_whole(g->n, c) : inc_budget(g, even);
    IncLaunch l(1, c, 1, ctx->stream);
    PG_CUDA_TRY(ctx, cudaLaunchKernelEx(&l.cfg, kern, a));
    ctx->launches += 1;
    return PG_OK;
}

static std::atomic<int> g_game_cluster[2][kClusterDevices];

bool games_apply(const pg_game* g, int* div, int* blocks) {
    const int64_t ng = g->ngames;
    if (!g->vgame || g->cv || !g->off || g->tune.loop_ranks || g->deep_mode || (int64_t)g->h_base0.size() != ng + 1 ||
        (int64_t)g->h_dbase.size() != ng + 1)
        return false;
    int64_t most = 0;  // ids of the largest game
    for (int32_t i = 0; i < ng; ++i)
        most = std::max<int64_t>(most, g->h_base0[i + 1] - g->h_base0[i] + g->h_dbase[i + 1] - g->h_dbase[i] + 1);
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device) != cudaSuccess) return false;
    *blocks = 0;
    for (int d : {1, kIncSmallDiv}) {
        if (ng > (int64_t)sms * d) continue;
        auto kern = d == 1 ? k_inc<false, 1, true> : k_inc<false, kIncSmallDiv, true>;
        const int largest = cluster_blocks((const void*)kern, kIncThreads / d, inc_shared(d), kIncCluster, g->device,
                                           g_game_cluster[d == 1 ? 0 : 1]);
        // as many blocks for each game as the device has room for and the game has use for
        int c = 1;
        while (2 * c <= largest && 2 * c * ng <= (int64_t)sms * d && c * (kIncThreads / d) < most) c *= 2;
        for (int fit = 0; c > 1; c /= 2) {  // (a cluster's blocks share a part of the device: fewer of them may fit)
            IncLaunch l((int)ng, c, d, nullptr);
            if (cudaOccupancyMaxActiveClusters(&fit, kern, &l.cfg) == cudaSuccess && fit >= ng) break;
            cudaGetLastError();
        }
        if (most > (int64_t)c * (kIncBlockIds / d) || (*blocks && c * *div <= *blocks * d)) continue;
        *div = d;
        *blocks = c;
    }
    return *blocks > 0;
}

pg_status run_games(pg_game* g, int64_t cap, int div, int blocks, bool* done) {
    pg_ctx* ctx = g->ctx;
    cudaStream_t s = ctx->stream;
    *done = false;
    g->by_game = true;
    g->rv_ok = false;
    pg_status st = build_reverse(g, 0);
    g->by_game = false;
    if (st) return st == PG_ENOMEM ? PG_OK : st;
    g->rv_ok = false;  // (the lockstep loop keeps Odd's lists only)
    const int32_t ng = g->ngames;
    std::vector<int2> games(ng);
    for (int32_t i = 0; i < ng; ++i) games[i] = make_int2((int32_t)(g->h_base0[i] + g->h_dbase[i] + i), i);
    int2* list = (int2*)g->slot;  // (scratch that is free during a loop; a game has two ids at least)
    PG_CUDA_TRY(ctx, cudaMemcpyAsync(list, games.data(), sizeof(int2) * ng, cudaMemcpyHostToDevice, s));
    IncArgs a = inc_args(g, cap, true);
    a.n_q = (int32_t*)g->cl_ks;
    a.gsink = g->gsink;
    a.games = list;
    IncLaunch l(ng, blocks, div, s);
    PG_CUDA_TRY(ctx, cudaLaunchKernelEx(&l.cfg, div == 1 ? k_inc<false, 1, true> : k_inc<false, kIncSmallDiv, true>, a));
    ctx->launches += 1;
    std::vector<GameState> gs(ng);
    PG_CUDA_TRY(ctx, cudaMemcpyAsync(gs.data(), g->gst, sizeof(GameState) * ng, cudaMemcpyDeviceToHost, s));
    PG_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    *done = true;
    for (const GameState& x : gs) *done = *done && x.phase != kPhaseActive;
    return PG_OK;
}

}  // namespace pg
