// Test driver for the cut of the edge stream into waves (waves.h), run without a
// GPU.  Reads uint64 m, then t[m] and dep[m] as uint32; runs every part of the
// cut, the last part first, and writes as uint32: 1 if all steps fit, the largest
// number of marks on one edge, the number of waves, then their first edges and
// their step flags.  With --indexable N it prints whether N waves can be swept.
#include "waves.h"

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    if (!std::strcmp(argv[1], "--indexable")) {
        std::printf("%d\n", mantra::waves_indexable(std::strtoull(argv[2], nullptr, 10)) ? 1 : 0);
        return 0;
    }
    FILE* f = std::fopen(argv[1], "rb");
    if (!f) return 2;
    uint64_t m = 0;
    if (std::fread(&m, 8, 1, f) != 1) return 2;
    std::vector<uint32_t> t(m), dep(m), marks(m, 0u), out;
    if (std::fread(t.data(), 4, m, f) != m || std::fread(dep.data(), 4, m, f) != m) return 2;
    std::fclose(f);
    bool fit = true;
    for (uint64_t x = (m + mantra::WAVE_CUT - 1) / mantra::WAVE_CUT; x-- > 0;)
        fit &= mantra::wave_cut_part(t.data(), dep.data(), (uint32_t)m, (uint32_t)x, [&](uint32_t i) { ++marks[i]; });
    std::vector<uint32_t> first;
    for (uint32_t i = 0; i < m; ++i)
        if (marks[i]) first.push_back(i);
    out.push_back(fit ? 1u : 0u);
    out.push_back(m ? *std::max_element(marks.begin(), marks.end()) : 0u);
    out.push_back((uint32_t)first.size());
    out.insert(out.end(), first.begin(), first.end());
    first.push_back((uint32_t)m);
    for (size_t w = 0; w + 1 < first.size(); ++w)
        out.push_back(mantra::wave_step_flags(t.data(), (uint32_t)m, first[w], first[w + 1]));
    FILE* o = std::fopen(argv[2], "wb");
    if (!o) return 2;
    std::fwrite(out.data(), 4, out.size(), o);
    std::fclose(o);
    return 0;
}
