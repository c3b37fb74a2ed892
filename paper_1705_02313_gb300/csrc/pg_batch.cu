// Batches: many games solved together in one id space (pg_solve_batch).
//
// The packed layout: game i's relabelled vertices occupy ids [B_i, B_i + n_i'),
// its sink slot is B_i + n_i', and its edges [E_i, E_i + m_i'). The games are
// loaded (validation, the admissibility preprocessing of Section 3, relabelling)
// as one union straight into that layout (load_union; in chunks, copied
// together, beyond the sizes of one). Loading them one by one, about 45 kernels,
// 35 allocations and 4 host waits per game, took three quarters of a batch of
// 256 games of 1k-100k vertices even on 8 threads (71.5 -> 15.2 ms in all); the
// general path still does
// so for batches that load_union hands back (a game that is refused, or with
// very sparse priorities). Each pass of Algorithm 1 then runs once over all
// games; each game keeps its own state on the device and follows exactly the
// trajectory it would follow alone.
#include <string.h>

#include <atomic>
#include <chrono>
#include <thread>

#include "pg_internal.cuh"

// Loader threads of a batch (each with its own stream).
#ifndef PG_LOADERS
#define PG_LOADERS 8
#endif

namespace pg {
namespace {

template <typename OffT>
__global__ void k_pack(int32_t np, int64_t mp, int32_t B, int64_t E, int32_t gi, int64_t o0, int32_t n0, int32_t k,
                       int32_t d0, const int32_t* __restrict__ off_i, const int32_t* __restrict__ tgt_i,
                       const uint8_t* __restrict__ flags_i, const int32_t* __restrict__ pri_i,
                       const int32_t* __restrict__ orig_i, const int32_t* __restrict__ nid0_i,
                       const int32_t* __restrict__ dnid_i, const int32_t* __restrict__ dummy_i, OffT* off, int32_t* tgt,
                       uint8_t* flags, int32_t* pri, int32_t* orig, int32_t* nid0, int32_t* dnid, int32_t* dummy,
                       int32_t* vgame, int32_t* strat) {
    int64_t span = (int64_t)np + 1;
    if (mp > span) span = mp;
    if (n0 > span) span = n0;
    if (k > span) span = k;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < span; t += (int64_t)gridDim.x * blockDim.x) {
        if (t <= np) {
            off[B + t] = (OffT)(E + off_i[t]);
            flags[B + t] = flags_i[t];
            pri[B + t] = pri_i[t];
            orig[B + t] = orig_i[t];
            vgame[B + t] = gi;
            if (t == np) strat[B + t] = B + np;  // the sink slot points at itself (never read)
        }
        if (t < mp) tgt[E + t] = B + tgt_i[t];
        if (t < n0) nid0[o0 + t] = B + nid0_i[t];
        if (t < k) {
            dnid[d0 + t] = B + dnid_i[t];
            dummy[d0 + t] = dummy_i[t];
        }
    }
}

// A chunk of a batch (loaded by load_union) into the whole batch's layout.
template <typename OffT>
__global__ void k_pack_chunk(int32_t n, int64_t m, int32_t B, int64_t E, int32_t gi, int64_t o0, int32_t n0, int32_t k,
                             int32_t d0, int32_t ng, const int32_t* __restrict__ off_i,
                             const int32_t* __restrict__ tgt_i, const uint8_t* __restrict__ flags_i,
                             const int32_t* __restrict__ pri_i, const int32_t* __restrict__ orig_i,
                             const int32_t* __restrict__ vgame_i, const int32_t* __restrict__ nid0_i,
                             const int32_t* __restrict__ dnid_i, const int32_t* __restrict__ dummy_i,
                             const int32_t* __restrict__ gsink_i, OffT* off, int32_t* tgt, uint8_t* flags,
                             int32_t* pri, int32_t* orig, int32_t* vgame, int32_t* nid0, int32_t* dnid,
                             int32_t* dummy, int32_t* gsink, int32_t* strat) {
    const int64_t span = m > n ? m : n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < span; t += (int64_t)gridDim.x * blockDim.x) {
        if (t < n) {
            off[B + t] = (OffT)(E + off_i[t]);
            flags[B + t] = flags_i[t];
            pri[B + t] = pri_i[t];
            orig[B + t] = orig_i[t];
            vgame[B + t] = gi + vgame_i[t];
            strat[B + t] = (int32_t)(B + t);  // (the sink slots'; the others' are set by the initial profile)
        }
        if (t < m) tgt[E + t] = B + tgt_i[t];
        if (t < n0) nid0[o0 + t] = B + nid0_i[t];
        if (t < k) {
            dnid[d0 + t] = B + dnid_i[t];
            dummy[d0 + t] = dummy_i[t];
        }
        if (t < ng) gsink[gi + t] = B + gsink_i[t];
    }
}

template <typename OffT>
__global__ void k_pack_last(OffT* off, int64_t N, int64_t M) {
    off[N] = (OffT)M;
}

inline unsigned grid_of(int64_t n) {
    int64_t b = (n + kBlock - 1) / kBlock;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 32));
}

// Allocates the packed layout of g (its counts are set).
pg_status alloc_packed(pg_game* g, bool wide) {
    pg_ctx* ctx = g->ctx;
    auto A = [&](void** p, size_t bytes) { return dev_alloc(ctx, p, bytes, ctx->stream); };
    const size_t N = g->n, M = g->m, n0 = g->n0, K = g->k;
    if (wide) PG_CUDA_TRY(ctx, A((void**)&g->off64, sizeof(int64_t) * (N + 1)));
    else PG_CUDA_TRY(ctx, A((void**)&g->off, sizeof(int32_t) * (N + 1)));
    PG_CUDA_TRY(ctx, A((void**)&g->tgt, sizeof(int32_t) * M));
    PG_CUDA_TRY(ctx, A((void**)&g->flags, N));
    PG_CUDA_TRY(ctx, A((void**)&g->pri, sizeof(int32_t) * N));
    PG_CUDA_TRY(ctx, A((void**)&g->orig_of, sizeof(int32_t) * N));
    PG_CUDA_TRY(ctx, A((void**)&g->nid0, sizeof(int32_t) * n0));
    PG_CUDA_TRY(ctx, A((void**)&g->dnid, sizeof(int32_t) * K));
    PG_CUDA_TRY(ctx, A((void**)&g->dummy_of, sizeof(int32_t) * K));
    PG_CUDA_TRY(ctx, A((void**)&g->vgame, sizeof(int32_t) * N));
    PG_CUDA_TRY(ctx, A((void**)&g->strat, sizeof(int32_t) * N));
    PG_CUDA_TRY(ctx, A((void**)&g->gsink, sizeof(int32_t) * g->ngames));
    return PG_OK;
}

// A chunk holds at most this many edges and vertices: its ids and offsets are
// int32, and its temporaries (about 70 bytes per vertex, 12 per edge) are to stay
// a few GB. Larger games are chunks of their own.
constexpr int64_t kChunkEdges = 1ll << 28, kChunkVertices = 1ll << 26;

template <typename OffT>
void pack_chunk(pg_game* g, const pg_game* c, int64_t B, int64_t E, int32_t gi, int64_t o0, int32_t d0, OffT* off) {
    k_pack_chunk<OffT><<<grid_of(std::max<int64_t>(c->n, c->m)), kBlock, 0, g->ctx->stream>>>(
        c->n, c->m, (int32_t)B, E, gi, o0, (int32_t)c->n0, c->k, d0, c->ngames, c->off, c->tgt, c->flags, c->pri,
        c->orig_of, c->vgame, c->nid0, c->dnid, c->dummy_of, c->gsink, off, g->tgt, g->flags, g->pri, g->orig_of,
        g->vgame, g->nid0, g->dnid, g->dummy_of, g->gsink, g->strat);
    g->ctx->launches += 1;
}

// Loads the games of a batch as unions. *general: some chunk needs the general path (nothing is returned).
pg_status load_batch(pg_ctx* ctx, int32_t ngames, const int64_t* vb, const int64_t* eb, const int32_t* off,
                     const int32_t* tgt, const uint8_t* own, const int32_t* pri, int32_t mem_kind, pg_game** out,
                     bool* general) {
    *out = nullptr;
    *general = false;
    std::vector<pg_game*> chunks;
    auto drop = [&] {
        for (pg_game* c : chunks) free_game(c);
        chunks.clear();
    };
    for (int32_t i = 0; i < ngames;) {
        int32_t j = i + 1;
        while (j < ngames && eb[j + 1] - eb[i] <= kChunkEdges && vb[j + 1] - vb[i] <= kChunkVertices) ++j;
        pg_game* c = nullptr;
        // (a game's offsets start one further per game before it)
        pg_status st = load_union(ctx, j - i, vb + i, eb + i, off + i, tgt, own, pri, mem_kind, &c, general);
        if (st == PG_ENOMEM) {  // one game at a time takes less
            cudaGetLastError();
            *general = true;
            st = PG_OK;
        }
        if (st || *general) {
            drop();
            return st;
        }
        chunks.push_back(c);
        i = j;
    }
    int64_t N = 0, M = 0, n0 = 0, m0 = 0, K = 0;
    for (const pg_game* c : chunks) {
        N += c->n;
        M += c->m;
        n0 += c->n0;
        m0 += c->m0;
        K += c->k;
    }
    if (N >= (1ll << 30) - 1 || K > INT32_MAX) {
        drop();
        return fail(ctx, PG_EUNSUPPORTED, K > INT32_MAX ? "pg_solve_batch: too many dummy vertices"
                                                         : "pg_solve_batch: more than 2^30 vertices in the batch");
    }
    const bool wide = ctx->wide_offsets || M > INT32_MAX - 1;
    pg_game* g = chunks[0];
    if (chunks.size() > 1 || wide) {
        g = new pg_game();
        g->ctx = ctx;
        g->device = ctx->device;
        g->ngames = ngames;
        g->n = (int32_t)N;
        g->m = M;
        g->n0 = n0;
        g->m0 = m0;
        g->k = (int32_t)K;
        pg_status st = alloc_packed(g, wide);
        g->h_base0.assign(1, 0);
        g->h_dbase.assign(1, 0);
        int64_t B = 0, E = 0, o0 = 0;
        int32_t d0 = 0, gi = 0;
        for (const pg_game* c : chunks) {
            if (st) break;
            if (wide) pack_chunk<int64_t>(g, c, B, E, gi, o0, d0, g->off64);
            else pack_chunk<int32_t>(g, c, B, E, gi, o0, d0, g->off);
            for (int32_t i = 1; i <= c->ngames; ++i) {
                g->h_base0.push_back(o0 + c->h_base0[i]);
                g->h_dbase.push_back(d0 + c->h_dbase[i]);
            }
            B += c->n;
            E += c->m;
            o0 += c->n0;
            d0 += c->k;
            gi += c->ngames;
        }
        g->sink0 = chunks[0]->sink0;
        if (!st) {
            if (wide) k_pack_last<int64_t><<<1, 1, 0, ctx->stream>>>(g->off64, N, M);
            else k_pack_last<int32_t><<<1, 1, 0, ctx->stream>>>(g->off, N, M);
            ctx->launches += 1;
            cudaError_t e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
            if (e != cudaSuccess) st = cuda_fail(ctx, e, "pack_chunk");
        }
        drop();
        if (st) {
            free_game(g);
            return st;
        }
    }
    pg_status st = alloc_scratch(g);
    if (st) {
        free_game(g);
        return st;
    }
    *out = g;
    return PG_OK;
}

}  // namespace

pg_status pack_games(pg_ctx* ctx, pg_game** games, int32_t ngames, pg_game** out) {
    *out = nullptr;
    cudaStream_t s = ctx->stream;
    int64_t N = 0, M = 0, n0 = 0;
    int64_t K = 0;
    for (int32_t i = 0; i < ngames; ++i) {
        N += games[i]->n;  // G' vertices plus the sink slot
        M += games[i]->m;
        n0 += games[i]->n0;
        K += games[i]->k;
    }
    if (N >= (1ll << 30) - 1) return fail(ctx, PG_EUNSUPPORTED, "pg_solve_batch: more than 2^30 vertices in the batch");
    if (K > INT32_MAX) return fail(ctx, PG_EUNSUPPORTED, "pg_solve_batch: too many dummy vertices");
    pg_game* g = new pg_game();
    g->ctx = ctx;
    g->device = ctx->device;
    g->ngames = ngames;
    g->n = (int32_t)N;
    g->m = M;
    g->n0 = n0;
    g->k = (int32_t)K;
    for (int32_t i = 0; i < ngames; ++i) g->m0 += games[i]->m0;
    const bool wide = ctx->wide_offsets || M > INT32_MAX - 1;
#define PK_TRY(expr)                                                 \
    do {                                                             \
        cudaError_t _e = (expr);                                     \
        if (_e != cudaSuccess) {                                     \
            free_game(g);                                            \
            return cuda_fail(ctx, _e, #expr);                        \
        }                                                            \
    } while (0)
    if (pg_status st = alloc_packed(g, wide)) {
        free_game(g);
        return st;
    }
    std::vector<int32_t> hsink(ngames);
    g->h_base0.assign(ngames + 1, 0);
    g->h_dbase.assign(ngames + 1, 0);
    int64_t B = 0, E = 0, o0 = 0;
    int32_t d0 = 0;
    for (int32_t i = 0; i < ngames; ++i) {
        pg_game* gi = games[i];
        const int32_t np = gi->n - 1;  // G' vertices of game i
        if (wide)
            k_pack<int64_t><<<grid_of(std::max<int64_t>(std::max<int64_t>(gi->n, gi->m), gi->n0)), kBlock, 0, s>>>(
                np, gi->m, (int32_t)B, E, i, o0, (int32_t)gi->n0, gi->k, d0, gi->off, gi->tgt, gi->flags, gi->pri,
                gi->orig_of, gi->nid0, gi->dnid, gi->dummy_of, g->off64, g->tgt, g->flags, g->pri, g->orig_of, g->nid0,
                g->dnid, g->dummy_of, g->vgame, g->strat);
        else
            k_pack<int32_t><<<grid_of(std::max<int64_t>(std::max<int64_t>(gi->n, gi->m), gi->n0)), kBlock, 0, s>>>(
                np, gi->m, (int32_t)B, E, i, o0, (int32_t)gi->n0, gi->k, d0, gi->off, gi->tgt, gi->flags, gi->pri,
                gi->orig_of, gi->nid0, gi->dnid, gi->dummy_of, g->off, g->tgt, g->flags, g->pri, g->orig_of, g->nid0,
                g->dnid, g->dummy_of, g->vgame, g->strat);
        ctx->launches += 1;
        PK_TRY(cudaGetLastError());
        hsink[i] = (int32_t)(B + np);
        B += gi->n;
        E += gi->m;
        o0 += gi->n0;
        d0 += gi->k;
        g->h_base0[i + 1] = o0;
        g->h_dbase[i + 1] = d0;
    }
    if (wide) k_pack_last<int64_t><<<1, 1, 0, s>>>(g->off64, N, M);
    else k_pack_last<int32_t><<<1, 1, 0, s>>>(g->off, N, M);
    ctx->launches += 1;
    PK_TRY(cudaMemcpyAsync(g->gsink, hsink.data(), sizeof(int32_t) * ngames, cudaMemcpyHostToDevice, s));
    PK_TRY(cudaStreamSynchronize(s));
    g->sink0 = hsink[0];
#undef PK_TRY
    for (int32_t i = 0; i < ngames; ++i) {
        free_game(games[i]);
        games[i] = nullptr;
    }
    pg_status st = alloc_scratch(g);
    if (st) {
        free_game(g);
        return st;
    }
    *out = g;
    return PG_OK;
}

}  // namespace pg

using namespace pg;

namespace {

double wall() {
    return std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

// The general path: every game loaded by itself, then packed. *loaded: the time when all were loaded.
pg_status load_general(pg_ctx* ctx, int32_t ngames, const int64_t* vb, const int64_t* eb, const int32_t* offsets,
                       const int32_t* targets, const uint8_t* owner, const int32_t* pri, int32_t mem_kind,
                       pg_game** out, double* loaded) {
    std::vector<pg_game*> games(ngames, nullptr);
    auto cleanup = [&]() {
        for (pg_game* gi : games)
            if (gi) free_game(gi);
    };
    // Loading (validation, preprocessing, relabelling) is a chain of small
    // kernels and host synchronisations per game: up to kLoaders threads,
    // each with its own stream, load games concurrently so that their work
    // overlaps on the device. The first failing game (in index order) decides
    // the status.
    constexpr int kLoaders = PG_LOADERS;
    const int nload = std::max(1, std::min<int>(kLoaders, ngames));
    std::vector<pg_ctx*> lctx(nload, nullptr);
    std::vector<pg_status> gst_load(ngames, PG_OK);
    std::vector<std::string> gerr(ngames);
    for (int t = 0; t < nload; ++t) {
        pg_status st = pg_ctx_create(&lctx[t], ctx->device);
        if (st == PG_OK && cudaStreamCreateWithFlags(&lctx[t]->stream, cudaStreamNonBlocking) != cudaSuccess)
            st = PG_ECUDA;
        if (st) {
            for (pg_ctx* c : lctx)
                if (c) {
                    if (c->stream) cudaStreamDestroy(c->stream);
                    pg_ctx_destroy(c);
                }
            return fail(ctx, st, "pg_solve_batch: could not create loader streams");
        }
    }
    std::atomic<int32_t> next(0);
    auto loader = [&](int t) {
        cudaSetDevice(ctx->device);
        for (;;) {
            const int32_t i = next.fetch_add(1);
            if (i >= ngames) break;
            const int64_t ni = vb[i + 1] - vb[i], mi = eb[i + 1] - eb[i];
            pg_status st = load_game(lctx[t], (int32_t)ni, mi, offsets + vb[i] + i, targets + eb[i], owner + vb[i],
                                     pri + vb[i], mem_kind, &games[i], false);
            if (st == PG_OK && games[i]->cv) {
                st = fail(lctx[t], PG_EUNSUPPORTED,
                          "pg_solve_batch: games with repeated priorities are solved one at a time");
            }
            if (st) {
                gst_load[i] = st;
                gerr[i] = lctx[t]->err;
                next.store(ngames);  // stop the other loaders early
            }
        }
    };
    std::vector<std::thread> th;
    for (int t = 1; t < nload; ++t) th.emplace_back(loader, t);
    loader(0);
    for (auto& x : th) x.join();
    for (pg_ctx* c : lctx) {
        cudaStreamDestroy(c->stream);
        pg_ctx_destroy(c);
    }
    for (int32_t i = 0; i < ngames; ++i) {
        if (gst_load[i] != PG_OK) {
            cleanup();
            ctx->err = gerr[i];
            return gst_load[i];
        }
        if (!games[i]) {  // not reached because another game failed first
            cleanup();
            return fail(ctx, PG_ECUDA, "pg_solve_batch: a game was not loaded");
        }
    }
    *loaded = wall();
    pg_status st = pack_games(ctx, games.data(), ngames, out);
    if (st) cleanup();
    return st;
}

pg_status batch_solve(pg_ctx* ctx, int32_t ngames, const int64_t* vb, const int64_t* eb, const int32_t* offsets,
                      const int32_t* targets, const uint8_t* owner, const int32_t* pri, int32_t mem_kind,
                      int64_t max_inner, pg_result_batch* out) {
    const double t0 = wall();
    pg_game* g = nullptr;
    bool general = false;
    pg_status st = load_batch(ctx, ngames, vb, eb, offsets, targets, owner, pri, mem_kind, &g, &general);
    double t1 = wall();
    if (!st && general) st = load_general(ctx, ngames, vb, eb, offsets, targets, owner, pri, mem_kind, &g, &t1);
    if (st) return st;
    int64_t nmax = 0;  // G' vertices and the sink slot of the largest game
    for (int32_t i = 0; i < ngames; ++i)
        nmax = std::max<int64_t>(nmax, g->h_base0[i + 1] - g->h_base0[i] + g->h_dbase[i + 1] - g->h_dbase[i] + 1);
    struct Guard {
        pg_game* g;
        ~Guard() { free_game(g); }
    } guard{g};
    const int64_t cap = max_inner > 0 ? max_inner : 64 * (nmax + 64);
    st = apply_profile(g, nullptr, nullptr, nullptr, PG_MEM_HOST);
    if (!st) st = reset_scratch(g);
    if (st) return st;
    Timer tm(g);
    tm.mark(3);
    const double t2 = wall();
    st = run_loop(g, cap, true, tm);
    if (st) return st;
    out->load_ms = t1 - t0;
    out->pack_ms = t2 - t1;
    out->loop_ms = wall() - t2;
    std::vector<GameState> gs(ngames);
    PG_CUDA_TRY(ctx, cudaMemcpy(gs.data(), g->gst, sizeof(GameState) * ngames, cudaMemcpyDeviceToHost));
    bool any_timeout = false, any_odd = false;
    for (const GameState& x : gs) {
        any_timeout |= x.phase == kPhaseTimeout;
        any_odd |= x.phase == kPhaseOddCycle;
    }
    if (any_timeout || g->last_cmp) {  // the full valuation of the profiles being returned
        st = full_valuation(g, false);
        if (st) return st;
        g->last_cmp = false;
    }
    tm.mark(2);
    g->t_total = tm.since(3, 2);
    for (int32_t i = 0; i < ngames; ++i) {
        if (out->major) out->major[i] = gs[i].major;
        if (out->inner) out->inner[i] = gs[i].inner;
        if (out->status)
            out->status[i] = gs[i].phase == kPhaseDone ? PG_OK
                             : gs[i].phase == kPhaseTimeout ? PG_ETIMEOUT
                                                            : PG_ENOTADMISSIBLE;
    }
    if (out->dummy_base)
        for (int32_t i = 0; i <= ngames; ++i) out->dummy_base[i] = g->h_dbase[i];
    out->iterations = 0;  // (the games' loops need not run in step)
    for (const GameState& q : gs) out->iterations = std::max<int64_t>(out->iterations, q.inner);
    st = write_outputs(g, out->mem_kind, out->win, out->sigma, out->tau, out->val_class, out->val_depth,
                       out->val_rank, nullptr, out->dummy_sigma);
    if (st) return st;
    if (any_odd) return fail(ctx, PG_ENOTADMISSIBLE, "pg_solve_batch: a game reached an odd cycle");
    if (any_timeout) return fail(ctx, PG_ETIMEOUT, "pg_solve_batch: iteration cap reached");
    return PG_OK;
}

}  // namespace

extern "C" pg_status pg_solve_batch(pg_ctx* ctx, int32_t ngames, const int64_t* vtx_base, const int64_t* edge_base,
                                    const int32_t* offsets, const int32_t* targets, const uint8_t* owner,
                                    const int32_t* pri, int32_t mem_kind, int64_t max_inner, pg_result_batch* out) {
    if (!ctx) return PG_EINVAL;
    if (ngames < 1 || !vtx_base || !edge_base || !offsets || !targets || !owner || !pri || !out)
        return fail(ctx, PG_EINVAL, "pg_solve_batch: bad arguments");
    if (mem_kind != PG_MEM_HOST && mem_kind != PG_MEM_DEVICE) return fail(ctx, PG_EINVAL, "pg_solve_batch: bad mem_kind");
    if (vtx_base[0] != 0 || edge_base[0] != 0) return fail(ctx, PG_EINVAL, "pg_solve_batch: bases must start at 0");
    for (int32_t i = 0; i < ngames; ++i) {
        if (vtx_base[i + 1] <= vtx_base[i] || edge_base[i + 1] < edge_base[i])
            return fail(ctx, PG_EINVAL, "pg_solve_batch: every game needs at least one vertex");
        if (vtx_base[i + 1] - vtx_base[i] >= (1 << 29))
            return fail(ctx, PG_EINVAL, "pg_solve_batch: a game has more than 2^29 vertices");
    }
    if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, PG_ECUDA, "cudaSetDevice failed");
    return batch_solve(ctx, ngames, vtx_base, edge_base, offsets, targets, owner, pri, mem_kind, max_inner, out);
}
