// Host check of the device buffer's bookkeeping (DBuf in osrc_internal.cuh)
// with an allocator that fails on demand: after a failed alloc the buffer is
// empty (no pointer, size 0), so that a later size test allocates again
// instead of passing a null pointer to a kernel, and the accounted bytes match.
// Prints "ok <cases>" and exits 0, or reports the first violation and exits 1.
#include <cstdio>
#include <cstdlib>
#include <map>

#include "../paper_2104_04609_gb300/csrc/osrc_internal.cuh"

static std::map<void *, size_t> g_live;
void osrc_set_error(const std::string &) {}

int ctx_alloc(osrc_ctx *ctx, void **p, size_t bytes) {
    *p = nullptr;
    if (ctx->used.load() + bytes > ctx->budget) return OSRC_OUT_OF_MEMORY;
    ctx->used += bytes;
    *p = std::malloc(bytes);
    g_live[*p] = bytes;
    return OSRC_OK;
}

void ctx_free(osrc_ctx *ctx, void *p, size_t bytes) {
    if (!g_live.count(p) || g_live[p] != bytes) {
        std::printf("FAIL freed %zu bytes of a block of another size\n", bytes);
        std::exit(1);
    }
    g_live.erase(p);
    std::free(p);
    ctx->used -= bytes;
}

#define CHECK(c)                                    \
    do {                                            \
        if (!(c)) {                                 \
            std::printf("FAIL line %d: %s\n", __LINE__, #c); \
            return 1;                               \
        }                                           \
        ++cases;                                    \
    } while (0)

int main() {
    int cases = 0;
    osrc_ctx ctx;
    ctx.budget = 1000;
    {
        DBuf<double> b, c;
        CHECK(b.alloc(&ctx, 1000) == OSRC_OUT_OF_MEMORY);
        CHECK(b.p == nullptr && b.n == 0);  // a test "b.n < needed" allocates again
        CHECK(b.alloc(&ctx, 100) == OSRC_OK);
        CHECK(b.p != nullptr && b.n == 100 && ctx.used.load() == 800);
        CHECK(b.alloc(&ctx, 126) == OSRC_OUT_OF_MEMORY);  // growing releases, then fails
        CHECK(b.p == nullptr && b.n == 0 && ctx.used.load() == 0);
        CHECK(b.alloc(&ctx, 0) == OSRC_OK);
        CHECK(b.p == nullptr && b.n == 0);
        CHECK(b.alloc(&ctx, 10) == OSRC_OK);
        c.borrow(b);
        CHECK(c.p == b.p && c.n == 10);
        CHECK(c.alloc(&ctx, 1000) == OSRC_OUT_OF_MEMORY);  // a borrowed buffer frees nothing
        CHECK(c.p == nullptr && c.n == 0 && b.p != nullptr && ctx.used.load() == 80);
    }
    CHECK(ctx.used.load() == 0 && g_live.empty());
    std::printf("ok %d\n", cases);
    return 0;
}
