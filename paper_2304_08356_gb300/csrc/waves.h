// The cut of the time-sorted edge stream into waves (k_sweep.cu), as functions
// that the device kernels and a host program both run.
#pragma once

#include <cstdint>

namespace mantra {

// Stream edges per part of the wave cut (a thread each: 512 made a load of 125,000
// edges 0.25 ms longer, 128 a sweep 2 % longer); waves of one time step at most; waves
// per batch.  Flags of a wave: part of a time step of several waves, the last of
// them; an edge's head slot has several in-edges.
constexpr uint32_t WAVE_CUT = 128, WAVE_STEP = 512, WAVE_BATCH = 8;
constexpr uint32_t WAVE_BIG = 1u, WAVE_LAST = 2u, WAVE_SEVERAL = 4u;

// Part x of the cut of a stream with times t (ascending, m of them): takes the
// time steps that begin in [x WAVE_CUT, (x + 1) WAVE_CUT) and extends a wave by
// whole steps while it has at most 32 edges and none depends on an edge of the
// wave (dep[i]: one past the last earlier edge, of another time, into an end of
// edge i); a step of more edges gets waves of its own.  mark(i): edge i is a
// wave's first.  The edges of a step belong to the part in which the step
// begins, so no two parts mark the same edge, and every edge is in the wave of
// the last mark up to it.  False: a step has more than WAVE_STEP waves.
template <class Mark>
__host__ __device__ inline bool wave_cut_part(const uint32_t* t, const uint32_t* dep, uint32_t m, uint32_t x, Mark mark) {
    const uint64_t lo = (uint64_t)x * WAVE_CUT;
    if (lo >= m) return true;
    const uint32_t hi = lo + WAVE_CUT < m ? (uint32_t)lo + WAVE_CUT : m;
    uint32_t i = (uint32_t)lo;
    while (i > 0 && i < hi && t[i] == t[i - 1]) ++i;                  // a step that began earlier
    uint32_t s = i;
    bool open = false;
    while (i < hi) {
        uint32_t e = i, d = 0;                                        // the step [i, e)
        while (e < m && t[e] == t[i] && e - i <= 32u * WAVE_STEP) {
            if (dep[e] > d) d = dep[e];
            ++e;
        }
        if (e - i > 32u) {                                            // several waves for the step
            if (e - i > 32u * WAVE_STEP) return false;
            for (uint32_t y = i; y < e; y += 32u) mark(y);
            open = false;
        } else if (!open || d > s || e - s > 32u) {
            s = i;
            open = true;
            mark(s);
        }
        i = e;
    }
    return true;
}

// WAVE_BIG and WAVE_LAST of the wave of edges [i0, i1): a wave that shares its
// time with a neighbour is part of a step of several waves.
__host__ __device__ inline uint32_t wave_step_flags(const uint32_t* t, uint32_t m, uint32_t i0, uint32_t i1) {
    if (i0 >= i1) return 0u;
    const uint32_t tm = t[i1 - 1];
    const bool more = i1 < m && t[i1] == tm;
    return more ? WAVE_BIG : (i0 > 0 && t[i0 - 1] == tm ? WAVE_BIG | WAVE_LAST : 0u);
}

// Whether a stream of that many waves can be swept: a record of the log names
// its edge by its place in the waves (32 a wave, whole batches) in 32 bits.
__host__ __device__ inline bool waves_indexable(uint64_t waves) {
    return (waves + WAVE_BATCH - 1) / WAVE_BATCH * WAVE_BATCH * 32u <= (uint64_t)1 << 32;
}

}  // namespace mantra
