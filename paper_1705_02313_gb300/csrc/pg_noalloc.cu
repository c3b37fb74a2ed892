// pg_valuate_static: the valuation of one successor function with every
// piece of working memory taken from a fixed array compiled into the library,
// for callers that cannot allocate device memory (see include/pg.h).
//
// The working memory is one file-scope device array of kStaticBytes bytes,
// sized for kStaticMaxN vertices. Host code cannot use the array's name as a
// device address, so every call looks the address up with
// cudaGetSymbolAddress (with the call's device current; the lookup allocates
// nothing, and a context made after a device reset gets the new address). The call
// then lays out the valuation's arrays inside the static buffer, copies the
// successor function into it (a successor outside [0, n] is recorded and
// replaced by the sink, so no kernel reads out of bounds), runs the same
// kernels as pg_valuate on the copy, writes class, depth and rank into the
// caller's arrays and waits for its stream once, at the end, to read the
// error words. No device or host memory is allocated on any path; error
// messages are not recorded (only the status is returned).
#include <algorithm>

#include "pg_internal.cuh"

namespace pg {
namespace {

constexpr int32_t kStaticMaxN = 1 << 18;
static_assert(kStaticMaxN + 1 <= kSmallIds, "every call takes the small games' path, whose arrays are laid out here");

constexpr size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Byte offsets of the arrays inside the static buffer, for kStaticMaxN vertices.
struct Layout {
    size_t succ, gd, gd32, plist, slot, ccnt, coff, cl_ks, sz, wgt, oddsz, key, cls, kind, depth, hugelist,
        flags, tiles, gst, cnt, bytes;
};

constexpr Layout make_layout() {
    const size_t N = kStaticMaxN + 1;  // the vertices and the sink slot
    const size_t ntiles = (N + kCoopTile - 1) / kCoopTile;
    Layout L{};
    size_t p = 0;
    L.succ = p;     p = al256(p + 4 * N);
    L.gd = p;       p = al256(p + 8 * N);
    L.gd32 = p;     p = al256(p + 4 * N);
    L.plist = p;    p = al256(p + 4 * N);
    L.slot = p;     p = al256(p + 4 * N);
    L.ccnt = p;     p = al256(p + 4 * (N + 1));
    L.coff = p;     p = al256(p + 4 * (N + 2));
    L.cl_ks = p;    p = al256(p + 8 * N);
    L.sz = p;       p = al256(p + 4 * N);
    L.wgt = p;      p = al256(p + 4 * N);
    L.oddsz = p;    p = al256(p + 4 * N);
    L.key = p;      p = al256(p + 4 * (N + 1));
    L.cls = p;      p = al256(p + N);
    L.kind = p;     p = al256(p + N);
    L.depth = p;    p = al256(p + 4 * N);
    L.hugelist = p; p = al256(p + 4 * N);
    L.flags = p;    p = al256(p + N);
    L.tiles = p;    p = al256(p + 8 * std::max<size_t>(2 * ntiles + 2, kSmallBlocks));
    L.gst = p;      p = al256(p + sizeof(GameState));
    L.cnt = p;      p = al256(p + sizeof(Counters));
    L.bytes = p;
    return L;
}

constexpr Layout kLayout = make_layout();
constexpr size_t kStaticBytes = kLayout.bytes;

// Every call shares this buffer; it keeps the last call's contents.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

Counters g_static_hcnt;  // host copy of the counters (pageable, fixed)

}  // namespace
}  // namespace pg

using namespace pg;

extern "C" pg_status pg_valuate_static(int32_t n, const int32_t* succ, const uint8_t* odd, int8_t* val_class,
                                       int32_t* val_depth, int32_t* val_rank, void* stream) {
    if (n < 1 || !succ || !odd) return PG_EINVAL;
    if (n > kStaticMaxN) return PG_EUNSUPPORTED;
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return PG_ECUDA;

    pg_ctx ctx;  // on the stack; quiet: no message strings are built
    ctx.device = device;
    ctx.stream = (cudaStream_t)stream;
    ctx.quiet = true;
    ctx.tune.deep_cut = INT32_MAX;  // no ruling-set path here (its scratch is not in the fixed array)
    ctx.deep_fallback = false;
    // the array's address on the current device, looked up on every call
    void* found = nullptr;
    if (cudaGetSymbolAddress(&found, g_static_scratch) != cudaSuccess || !found) return PG_ECUDA;
    unsigned char* base = (unsigned char*)found;

    // a game view over the static buffer: only the fields the valuation reads
    pg_game g;
    g.ctx = &ctx;
    g.device = device;
    g.n = n + 1;  // the vertices and the sink slot
    g.sink0 = n;
    g.ngames = 1;
    g.strat = (int32_t*)(base + kLayout.succ);  // the checked copy of succ
    g.gd = (uint64_t*)(base + kLayout.gd);
    g.gd32 = (uint32_t*)(base + kLayout.gd32);
    g.plist = (int32_t*)(base + kLayout.plist);
    g.slot = (int32_t*)(base + kLayout.slot);
    g.ccnt = (int32_t*)(base + kLayout.ccnt);
    g.coff = (int32_t*)(base + kLayout.coff);
    g.cl_ks = (int2*)(base + kLayout.cl_ks);
    g.sz = (int32_t*)(base + kLayout.sz);
    g.wgt = (int32_t*)(base + kLayout.wgt);
    g.oddsz = (int32_t*)(base + kLayout.oddsz);
    g.key = (int32_t*)(base + kLayout.key);
    g.cls = (uint8_t*)(base + kLayout.cls);
    g.kind = (uint8_t*)(base + kLayout.kind);
    g.depth = (int32_t*)(base + kLayout.depth);
    g.hugelist = (int32_t*)(base + kLayout.hugelist);
    g.flags = (uint8_t*)(base + kLayout.flags);
    g.tiles = (int64_t*)(base + kLayout.tiles);
    g.ntiles = std::max<int64_t>(1, ((int64_t)n + 1 + kCoopTile - 1) / kCoopTile);
    g.gst = (GameState*)(base + kLayout.gst);
    g.cnt = (Counters*)(base + kLayout.cnt);
    g.hcnt = &g_static_hcnt;

    g.in_succ = succ;  // copied and checked by the valuation
    g.in_odd = odd;
    g.out_class = val_class;
    g.out_depth = val_depth;
    g.out_rank = val_rank;
    g.tune = ctx.tune;
    pg_status st = enqueue_valuation(&g, false, true);
    if (st != PG_OK) return st;
    // the one wait of the call: the counters, the range check's among them
    st = sync_counters(&g);
    if (st != PG_OK) return st;
    if (g_static_hcnt.bad) return PG_EINVAL;
    return g_static_hcnt.n_odd > 0 ? PG_ENOTADMISSIBLE : PG_OK;
}
