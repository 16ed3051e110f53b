// Device memory as the engine takes it, over a runtime Rt (CUDA's, or a test's):
// Rt::alloc(void**, size_t) returns whether it succeeded, Rt::free(void*), and
// Rt::clear() forgets the runtime's last error.  A failed allocation is a normal
// outcome (the caller does with less, or answers "out of memory"), so it never
// stays behind as the last error, which the next launch would report as its own.
#pragma once

#include <algorithm>
#include <cstddef>
#include <map>

namespace mantra {

template <class Rt>
bool take_memory(void** p, size_t bytes) {
    *p = nullptr;
    if (Rt::alloc(p, bytes)) return true;
    *p = nullptr;
    Rt::clear();
    return false;
}

// Blocks kept by exact (256-rounded) size and reused by later problems and
// graphs; at most `limit` bytes stay cached (the oldest blocks go first), and all
// of them are given back before a get fails.
template <class Rt>
struct MemoryPool {
    struct Block { void* p; unsigned long long age; };
    size_t limit;
    std::multimap<size_t, Block> free_blocks;
    size_t cached = 0;
    unsigned long long puts = 0;
    explicit MemoryPool(size_t limit_bytes) : limit(limit_bytes) {}
    static size_t rounded(size_t bytes) { return (std::max<size_t>(bytes, 256) + 255) & ~(size_t)255; }
    void* get(size_t bytes) {
        bytes = rounded(bytes);
        auto it = free_blocks.find(bytes);
        if (it != free_blocks.end()) {
            void* p = it->second.p;
            free_blocks.erase(it);
            cached -= bytes;
            return p;
        }
        void* p = nullptr;
        if (!take_memory<Rt>(&p, bytes)) {
            release_all();
            take_memory<Rt>(&p, bytes);
        }
        return p;
    }
    void put(void* p, size_t bytes) {
        if (!p) return;
        bytes = rounded(bytes);
        if (bytes > limit) { Rt::free(p); return; }
        while (cached + bytes > limit) {
            auto old = std::min_element(free_blocks.begin(), free_blocks.end(),
                                        [](const auto& x, const auto& y) { return x.second.age < y.second.age; });
            Rt::free(old->second.p);
            cached -= old->first;
            free_blocks.erase(old);
        }
        free_blocks.emplace(bytes, Block{p, puts++});
        cached += bytes;
    }
    void release_all() {
        for (auto& kv : free_blocks) Rt::free(kv.second.p);
        free_blocks.clear();
        cached = 0;
    }
};

}  // namespace mantra
