// Stands in for the library's device allocator (pg::dev_alloc, which every
// translation unit of libpg.so calls by its dynamic symbol) in a process that
// loads this before libpg.so: chosen allocations fail as if the device had no
// memory left. No GPU state is touched.
#include <dlfcn.h>
#include <stddef.h>
#include <stdlib.h>

#include <atomic>

struct pg_ctx;
struct CUstream_st;

namespace {
std::atomic<long> calls{0}, from{-1}, count{0};
using Alloc = int (*)(pg_ctx*, void**, size_t, CUstream_st*);
}  // namespace

extern "C" void shim_fail(long first, long n) {  // the next allocations are numbered from 0: [first, first + n) fail
    calls = 0;
    from = first;
    count = n;
}
extern "C" long shim_calls() { return calls; }

namespace pg {
int dev_alloc(pg_ctx* ctx, void** p, size_t bytes, CUstream_st* s) {
    static Alloc real = (Alloc)dlsym(dlopen(getenv("SHIM_LIBPG"), RTLD_NOLOAD | RTLD_NOW),
                                     "_ZN2pg9dev_allocEP6pg_ctxPPvmP11CUstream_st");
    const long i = calls++;
    if (from >= 0 && i >= from && i < from + count) return 2;  // cudaErrorMemoryAllocation
    return real(ctx, p, bytes, s);
}
}  // namespace pg
