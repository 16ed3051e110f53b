// Test driver for devmem.h over a runtime of its own (no GPU): an allocator with a
// fixed amount of memory and, as CUDA has it, a last error that stays until it is
// asked for.  Exits 0 if every check holds, else with the failed check's line.
#include "devmem.h"

#include <cstdio>
#include <cstdlib>

namespace {

size_t g_left = 0;
bool g_error = false;
std::map<void*, size_t> g_live;

struct Fake {
    static bool alloc(void** p, size_t bytes) {
        if (bytes > g_left) { g_error = true; *p = (void*)1; return false; }
        *p = std::malloc(1);
        g_left -= bytes;
        g_live[*p] = bytes;
        return true;
    }
    static void free(void* p) {
        g_left += g_live.at(p);
        g_live.erase(p);
        std::free(p);
    }
    static void clear() { g_error = false; }
};

}  // namespace

#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
    using Pool = mantra::MemoryPool<Fake>;
    void* p = nullptr;
    g_left = 1000;
    // a failed allocation: no pointer, no error left behind
    CHECK(!mantra::take_memory<Fake>(&p, 2000) && p == nullptr && !g_error);
    CHECK(mantra::take_memory<Fake>(&p, 1000) && p && g_left == 0);
    Fake::free(p);

    // a get that only succeeds once the cached blocks are given back
    g_left = 4096;
    Pool pool(1 << 20);
    void* a = pool.get(2048);
    pool.put(a, 2048);
    CHECK(pool.cached == 2048 && g_left == 2048);
    void* b = pool.get(4096);
    CHECK(b && !g_error && pool.cached == 0 && g_left == 0);
    // one that fails all the same
    CHECK(pool.get(256) == nullptr && !g_error);
    pool.put(b, 4096);
    CHECK(pool.get(3900) == b);                 // by rounded size
    pool.put(b, 3900);
    pool.put(nullptr, 77);
    pool.release_all();
    CHECK(g_left == 4096 && g_live.empty());

    // the limit on what stays cached
    Pool small(1024);
    a = small.get(512);
    b = small.get(700);
    small.put(a, 512);
    small.put(b, 700);                          // 512 + 768 exceeds it: the older block goes
    CHECK(small.cached == 768 && g_left == 4096 - 768 && small.get(768) == b);
    small.put(b, 768);
    a = small.get(2048);
    small.put(a, 2048);                         // larger than the cache may be
    CHECK(small.cached == 768 && g_left == 4096 - 768);
    a = small.get(256);
    small.put(a, 256);                          // both fit
    CHECK(small.cached == 1024 && small.get(768) == b && small.get(256) == a);
    small.put(b, 768);
    small.put(a, 256);
    small.release_all();
    CHECK(g_left == 4096 && g_live.empty());
    return 0;
}
