// Hop-level temporal search for the shortest (sh) and shortest-foremost (sfm)
// optimalities (paper Sec. 3 Def. 1; running-time theorem of Sec. 4.4), the
// backward path draw of the temporal Riondato-Kornaropoulos estimator
// (App. C), the ob estimator (Sec. 4.1), the Update step of Algorithm 1, and
// Algorithm 2's searches for sh / sfm.
//
// One CTA owns one sample at a time.  States are arrival appearances (v, t)
// ("slots"); level k holds the states at hop distance k from (s, -inf).  The
// search keeps no per-state data.  It rests on two facts:
//
//   * A vertex u on level k pushes its out-edges later than its earliest
//     level-k time.  Edges later than u's earliest time on an older level were
//     pushed then, and their heads are visited.  So only the edges between the
//     two times can find anything: every out-edge is walked at most once per
//     search, and a slot with a single in-edge is new whenever its edge is
//     walked -- no visited bitmap (slots with several in-edges carry a stamp).
//     A level is therefore a list of vertices with their earliest arrival (an
//     "event"), kept as the first out-edge later than it: an edge carries that
//     index for its head (out_vn), so a level needs no times.  The other edges
//     and states are counted by index arithmetic.
//   * Path counts are needed only for states on optimal s-z paths.  On the
//     bursty 20,000-node graph a search discovers 16,000 states and about 30
//     of them lie on such a path.  So the search finds levels only; when z is
//     reached, the states that lead to it are collected backward level by
//     level (whether a slot is on level k follows from its tail's events), and
//     path counts are summed over those states alone.
//
// What bounds it: latency and instruction issue.  A level is a chain of dependent
// L2 accesses (list entry, arrival and row directory, a few probes of the row,
// the edge window, the heads' arrivals) with five block barriers; about 170,000
// warp instructions per sample on the bursty 20,000-node graph, 0.3 issued per
// scheduler and cycle, DRAM at 18 % and L2 at 33 % of their peaks (with the arrivals
// in shared memory 131,000 instructions, DRAM 14 %, L2 24 %, 8.7 of 23 cycles
// per instruction at barriers).  The loads of
// four edge windows and two vertices per thread are issued together (one at a
// time: 40 against 10 ms with the arrivals in global memory).  22,000 sh samples
// on that graph take 7.2 ms; the search with per-state path counts and a visited
// bitmap (k_bfs) took 23.6 ms.
#include "mantra_dev.cuh"

#include <algorithm>
#include <mutex>

namespace mantra {

namespace {

constexpr int WALK_K = 4;            // edge windows with loads in flight per warp
constexpr int CONE_K = 4;            // the same for the slot windows of the backward collection
constexpr int EVB = 2;               // vertices of a level with loads in flight per thread
constexpr uint32_t HOP_PMAX = 256;   // states of the path sets kept in shared memory (512: 10 KB more per CTA,
                                     // less L1, 9.9 against 9.5 ms)
constexpr uint32_t HOP_DMAX = 30;    // its levels (a lane each when the path is written out)
constexpr uint32_t BLOOM_W = 128;    // words of the vertex filter (4,096 bits)

__device__ __forceinline__ uint32_t bloom_hash(uint32_t v) { return (v * 0x9E3779B1u) >> 20; }

// Shared memory of a CTA (dynamic; the next level's arrivals follow in the SM variant).
template <int NT>
struct __align__(16) HopSh {
    Task task;
    uint64_t i;                                      // sample index
    uint64_t unit;                                   // the next work unit
    u64 sigma;
    u64* ctr;                                        // counters of the current task
    u64 tot[4];                                      // its work counters (flushed when the task changes)
    u64 esc[NT / 32], walk;                          // the sample's counted edges (per warp), walked edges
    int t, cur_t;                                    // task of the sample (-1: no sample left), task loaded
    uint32_t s, z, ok;
    uint32_t scan[2][64];                            // block scans in turn
    uint32_t off[NT * EVB + 33], base[NT * EVB + 1]; // range table (see lbs_walk_warp)
    uint32_t bloom[BLOOM_W];
    uint32_t nq[2];                                  // vertices of the next level
    uint32_t nw, nh, nt;                             // list lengths
    uint32_t ovf, err, len;
    uint32_t e_lo, e_hi, tz, b;                      // z's in-edges, its latest in-edge time and that time's bucket
    uint32_t f, old, dup;                            // vertices; walked edges to older states, to no new state
    uint32_t rade[4];
    // small path sets (hop_small): per state its slot and, when it has one in-edge, the
    // first slot of the in-edge's tail and the end of the tail's usable slots
    uint32_t pa[HOP_PMAX], pw[HOP_PMAX], pl[HOP_PMAX];
    u64 ps[HOP_PMAX];                                // path counts summed over the level up to the state
    uint32_t hit[HOP_PMAX];
    uint32_t plev[HOP_DMAX + 2], pick[HOP_DMAX + 1];
};

// Region arrays of a CTA.
struct HopReg {
    uint2* fb;           // per vertex, as ~(first out-edge later than the arrival), 0: none: x the earliest
                         // arrival on the next level, y on any level so far (both 0 between samples)
    uint32_t* want;      // end of the slots wanted (0 between uses)
    uint32_t* grp;       // vertex -> event or group of a level (checked on use)
    uint32_t* grp2;      // the same, the next level's
    u64* acc;            // ob sums (0 between uses)
    uint32_t* Q;         // event -> vertex, level by level
    uint32_t* ea;        // event -> the first out-edge later than the vertex's arrival on the level
    uint32_t* eb;        // event -> the same for its older levels (NONE: none): [ea, eb) was walked from it
    uint2* rng;          // walk ranges of a level of several tiles
    uint32_t* list;      // wanted events / ob vertices (n entries; shares rng)
    uint32_t* lev;       // first event of each level
    uint32_t* clev;      // first path state of level lv (levels are stored from d down)
    uint32_t* glev;      // first group of level lv
    uint32_t* mst;       // level stamp of a slot with several in-edges
    uint32_t* Ca;        // path states: slot, time, path count (then the running sum over the group)
    uint32_t* Ct;
    u64* Cs;
    u64* Cb;             // ob: continuation counts
    uint32_t* Gw;        // group: one vertex's path states of a level, ascending in time; and its start
    uint32_t* Gs;
    uint32_t* path;
    uint32_t* pathe;
    uint32_t* stamp;     // last level stamp used
    __device__ __forceinline__ explicit HopReg(const HopWs& ws) {
        char* r = ws.base + (size_t)blockIdx.x * ws.stride;
        fb = reinterpret_cast<uint2*>(r + ws.o_fb);
        want = reinterpret_cast<uint32_t*>(r + ws.o_want);
        grp = reinterpret_cast<uint32_t*>(r + ws.o_grp);
        grp2 = reinterpret_cast<uint32_t*>(r + ws.o_grp2);
        acc = reinterpret_cast<u64*>(r + ws.o_acc);
        Q = reinterpret_cast<uint32_t*>(r + ws.o_q);
        ea = reinterpret_cast<uint32_t*>(r + ws.o_ea);
        eb = reinterpret_cast<uint32_t*>(r + ws.o_eb);
        rng = reinterpret_cast<uint2*>(r + ws.o_rng);
        list = reinterpret_cast<uint32_t*>(r + ws.o_rng);
        lev = reinterpret_cast<uint32_t*>(r + ws.o_lev);
        clev = lev + (ws.n_cap + 4);
        glev = clev + (ws.n_cap + 4);
        mst = reinterpret_cast<uint32_t*>(r + ws.o_mst);
        Ca = reinterpret_cast<uint32_t*>(r + ws.o_ca);
        Ct = reinterpret_cast<uint32_t*>(r + ws.o_ct);
        Cs = reinterpret_cast<u64*>(r + ws.o_cs);
        Cb = reinterpret_cast<u64*>(r + ws.o_cb);
        Gw = reinterpret_cast<uint32_t*>(r + ws.o_gw);
        Gs = reinterpret_cast<uint32_t*>(r + ws.o_gs);
        path = reinterpret_cast<uint32_t*>(r + ws.o_path);
        pathe = reinterpret_cast<uint32_t*>(r + ws.o_pathe);
        stamp = reinterpret_cast<uint32_t*>(r + ws.o_stamp);
    }
};

// The states on optimal paths, their counts and the draw when the sets are
// small (the usual case): everything but the graph and the events in shared
// memory, five barriers a level, counts and draw by warp 0.  All threads of
// the CTA; k: the level that reached z (events [q0, q1)).  False when a set is
// too large (nothing has been drawn or changed then); a count past 64 bits
// sets S.ovf.
template <int NT>
__device__ __forceinline__ bool hop_small(const HopWs& ws, uint32_t k, uint32_t q0, uint32_t q1, uint32_t E0) {
    constexpr int NW = NT / 32;
    constexpr uint32_t HMAX = NT < (int)HOP_PMAX ? NT : HOP_PMAX;      // states of a level
    extern __shared__ __align__(16) unsigned char hop_dyn[];
    HopSh<NT>& S = *reinterpret_cast<HopSh<NT>*>(hop_dyn);
    const HopReg R(ws);
    const DevGraph& g = S.task.g;
    const Job& job = S.task.job;
    const uint32_t s = S.s, z = S.z, d = k + 1u;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t FULL = 0xFFFFFFFFu;
    // events by vertex: two maps in turn, so that one level's is filled while the other is read
    auto put = [&](uint32_t l0, uint32_t l1, uint32_t* map) {
        for (uint32_t p = l0 + tid; p < l1; p += NT) map[R.Q[p]] = p;
    };
    auto event_of = [&](uint32_t u, uint32_t l0, uint32_t l1, const uint32_t* map) -> uint32_t {
        const uint32_t p = map[u];
        return p >= l0 && p < l1 && R.Q[p] == u ? p : NONE;
    };
    uint32_t* map = R.grp;
    uint32_t* map2 = R.grp2;
    if (d > 1) put(q0, q1, map);
    __syncthreads();
    // z's endpoints, ascending (sfm: the earliest)
    const uint32_t zs = g.slot_ptr[z], ze = g.slot_ptr[z + 1];
    int sp = 0;
    uint32_t nP = 0;
    for (uint32_t a0 = zs; a0 < ze; a0 += NT) {
        const uint32_t a = a0 + (uint32_t)tid;
        bool f = false;
        if (a < ze) {
            const uint32_t e1 = g.slot_in[a + 1];
            for (uint32_t e = g.slot_in[a]; e < e1 && !f; ++e) {
                const uint32_t w = g.in_u[e];
                if (d == 1) { f = w == s; continue; }
                const uint32_t o = g.in_out[e], p = event_of(w, q0, q1, map);
                f = p != NONE && R.ea[p] <= o;
            }
        }
        uint32_t x = f ? 1u : 0u, y = 0, tx, ty;
        block_exclusive_scan2<NT>(x, y, &tx, &ty, S.scan[sp]);
        sp ^= 1;
        if (f && nP + x < HMAX) S.pa[nP + x] = a;
        nP += tx;
        if (nP > HMAX) return false;
        if (job.opt == 1 && nP) { nP = 1; break; }
    }
    if (tid == 0) { S.plev[d] = 0; S.plev[d - 1] = nP; }
    uint32_t cb = 0;                     // states of level lv: [cb, nP)
    for (uint32_t lv = d; lv >= 2; --lv) {
        const uint32_t l0 = R.lev[lv - 1], l1 = R.lev[lv], m0 = R.lev[lv - 2], C = nP - cb;
        if (tid < (int)BLOOM_W) S.bloom[tid] = 0u;
        if (tid == 0) S.nh = 0;
        __syncthreads();                 // the states of level lv; the cleared filter
        // every state's in-edge: the tail's slots [a0, lim) may hold level lv - 1 states
        uint32_t a0 = NONE, w0 = NONE, lim = 0;
        bool several = false;
        if ((uint32_t)tid < C) {
            const uint32_t b = S.pa[cb + tid], e = g.slot_in[b], e1 = g.slot_in[b + 1];
            several = e1 - e > 1u;
            const uint32_t w = g.in_u[e], o = g.in_out[e];
            const uint32_t p = event_of(w, l0, l1, map);
            w0 = g.slot_ptr[w];
            lim = g.out_pend[o];
            const uint32_t r0 = g.out_ptr[w];
            if (p != NONE) {
                const uint32_t x = R.ea[p];
                if (x <= o) a0 = x > r0 ? g.out_pend[x - 1] : w0;
            }
            S.pw[cb + tid] = w0; S.pl[cb + tid] = lim;
            S.base[tid] = a0;
        }
        const bool filter = lv > 2 && l0 - m0 <= 2048u;       // level lv - 2's vertices
        if (lv > 2)
            for (uint32_t p = m0 + tid; p < l0; p += NT) {
                const uint32_t u = R.Q[p], h = bloom_hash(u);
                map2[u] = p;
                if (filter) atomicOr(S.bloom + (h >> 5), 1u << (h & 31));
            }
        if (__syncthreads_or(several)) return false;
        // one range per tail: the widest (its states share the start)
        uint32_t cnt = 0;
        if (a0 != NONE) {
            cnt = lim - a0;
            for (uint32_t y = 0; y < C; ++y)
                if (S.pw[cb + y] == w0 && S.base[y] != NONE &&
                    (S.pl[cb + y] > lim || (S.pl[cb + y] == lim && y < (uint32_t)tid))) { cnt = 0; break; }
        }
        uint32_t gx = cnt ? 1u : 0u, ex = cnt, Gc, E;
        block_exclusive_scan2<NT>(gx, ex, &Gc, &E, S.scan[sp]);
        sp ^= 1;
        if (cnt) { S.base[gx] = a0 - ex; S.off[gx] = ex; }
        if (tid < 33) S.off[Gc + tid] = tid ? NONE : E;
        __syncthreads();
        const uint32_t per = ((E + NW * 32u - 1u) / (NW * 32u)) * 32u;
        const uint32_t w_lo = min((uint32_t)wid * per, E), w_hi = min(w_lo + per, E);
        lbs_walk_warp<CONE_K>(S.off, Gc, S.base, w_lo, w_hi, [&](const uint32_t (&a)[CONE_K]) {
            uint32_t s0[CONE_K], s1[CONE_K], uu[CONE_K];
#pragma unroll
            for (int x = 0; x < CONE_K; ++x) {
                s0[x] = s1[x] = 0u;
                if (a[x] != NONE) { s0[x] = __ldg(g.slot_in + a[x]); s1[x] = __ldg(g.slot_in + a[x] + 1); }
            }
#pragma unroll
            for (int x = 0; x < CONE_K; ++x) uu[x] = s1[x] > s0[x] ? __ldg(g.in_u + s0[x]) : NONE;
#pragma unroll
            for (int x = 0; x < CONE_K; ++x) {
                if (a[x] == NONE) continue;
                bool f;
                if (s1[x] - s0[x] > 1u) {
                    f = __ldcg(R.mst + a[x]) == E0 + lv - 1u;
                } else if (lv == 2) {
                    f = uu[x] == s;
                } else {
                    const uint32_t h = bloom_hash(uu[x]);
                    f = !filter || ((S.bloom[h >> 5] >> (h & 31u)) & 1u);
                    if (f) {
                        const uint32_t o = g.in_out[s0[x]], p = event_of(uu[x], m0, l0, map2);
                        f = p != NONE && R.ea[p] <= o && o < R.eb[p];
                    }
                }
                if (f) {
                    const uint32_t p = atomicAdd(&S.nh, 1u);
                    if (p < HMAX) S.hit[p] = a[x];
                }
            }
        });
        __syncthreads();
        const uint32_t H = S.nh;
        if (H > HMAX || nP + H > HOP_PMAX) return false;
        if ((uint32_t)tid < H) {         // in slot order, i.e. by vertex and time
            const uint32_t a = S.hit[tid];
            uint32_t r = 0;
            for (uint32_t y = 0; y < H; ++y) r += S.hit[y] < a ? 1u : 0u;
            S.pa[nP + r] = a;
        }
        cb = nP;
        nP += H;
        if (tid == 0) S.plev[lv - 2] = nP;
        uint32_t* const t = map; map = map2; map2 = t;
    }
    __syncthreads();
    if (wid == 0) {
        // path counts summed over each level: a state's count is the sum over its tail's
        // states [pw, pl) of the level below, a difference of two of that level's sums
        bool bad = false;
        for (uint32_t lv = 1; lv <= d; ++lv) {
            const uint32_t p0 = S.plev[lv], p1 = S.plev[lv - 1];
            const uint32_t b0 = p1, b1 = lv > 1 ? S.plev[lv - 2] : p1;
            u64 carry = 0;
            for (uint32_t c = p0; c < p1; c += 32) {
                const uint32_t p = c + lane;
                u64 v = 0;
                if (p < p1) {
                    if (lv == 1) {
                        v = 1;
                    } else {
                        const uint32_t x0 = lower_bound_u32(S.pa, b0, b1, S.pw[p]), x1 = lower_bound_u32(S.pa, x0, b1, S.pl[p]);
                        if (x1 > x0) v = S.ps[x1 - 1] - (x0 > b0 ? S.ps[x0 - 1] : 0ull);
                    }
                }
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u64 y = shfl_up_w(v, o);
                    if (lane >= o) { const u64 sm = v + y; bad |= sm < v; v = sm; }
                }
                const u64 sm = v + carry;
                bad |= sm < v;
                if (p < p1) S.ps[p] = sm;
                carry = shfl_idx_w(sm, 31);
            }
            __syncwarp();
        }
        if (__any_sync(FULL, bad)) {     // the level's sum, perhaps not a path count, passed 64 bits
            if (lane == 0) S.ovf = 1u;
        } else {
            const u64 tot = S.ps[S.plev[d - 1] - 1];
            u128 x = 0;
            uint32_t ok = 1;
            if (lane == 0) ok = draw_below128((u128)tot, job.seed, S.i, job.dom_path, &x) ? 1u : 0u;
            ok = __shfl_sync(FULL, ok, 0);
            u64 xs = shfl_idx_w((u64)x, 0);
            bool err = !ok;
            if (err && lane == 0) set_status(job.status, ST_RNG);
            uint32_t lo = 0, hi = S.plev[d - 1];
            for (uint32_t lv = d; lv >= 1 && !err; --lv) {
                // the first state of [lo, hi) whose sum, counted from lo, exceeds xs
                const u64 before = lo > S.plev[lv] ? S.ps[lo - 1] : 0ull;
                uint32_t p = NONE;
                for (uint32_t c = lo; c < hi && p == NONE; c += 32) {
                    const uint32_t y = c + lane;
                    const unsigned msk = __ballot_sync(FULL, y < hi && xs < S.ps[y] - before);
                    if (msk) p = c + (uint32_t)(__ffs(msk) - 1);
                }
                if (p == NONE) { err = true; break; }
                if (p > lo) xs -= S.ps[p - 1] - before;
                if (lane == 0) S.pick[lv] = S.pa[p];
                if (lv > 1) {
                    const uint32_t b0 = S.plev[lv - 1], b1 = S.plev[lv - 2];
                    lo = lower_bound_u32(S.pa, b0, b1, S.pw[p]);
                    hi = lower_bound_u32(S.pa, lo, b1, S.pl[p]);
                }
            }
            __syncwarp();
            bool bade = false;
            if (!err && lane >= 1 && lane <= (int)d) {       // a lane per level: its vertex and edge
                const uint32_t b = S.pick[lane], e0 = g.slot_in[b], e1 = g.slot_in[b + 1];
                R.path[lane] = g.slot_v[b];
                uint32_t e = e0;
                if (lane == 1) {
                    e = lower_bound_u32(g.in_u, e0, e1, s);  // the edge from s
                    bade = e >= e1 || g.in_u[e] != s;
                }
                R.pathe[lane - 1] = e;
            }
            err |= __any_sync(FULL, bade);
            if (lane == 0) {
                R.path[0] = s;
                if (err) { S.err = 1; set_status(job.status, ST_CHECK); }
                S.len = d + 1u;
                S.sigma = tot;
                uint32_t w4[4];
                philox_block(job.seed, S.i, DOM_RADE, 0, w4);
                S.rade[0] = w4[0]; S.rade[1] = w4[1]; S.rade[2] = w4[2]; S.rade[3] = w4[3];
            }
        }
    }
    __syncthreads();
    return true;
}

// After the levels of a sample, all threads of the CTA: with z found from level
// k (events [q0, q1)), the states on optimal paths, their counts, the draw (or
// the ob values), then the sample's hits, Rademacher sums and record.  E0: the
// sample's first level stamp.  Sets S.ovf to 1 when the sample needs the 128-bit
// kernel, to 2 when it exceeds a cap.  Out of line, so that the levels' loop does not
// carry its registers.
template <int NT>
__device__ __noinline__ void hop_finish(const HopWs* wsp, bool found, uint32_t k, uint32_t q0, uint32_t q1,
                                        uint32_t E0) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char hop_dyn[];
    HopSh<NT>& S = *reinterpret_cast<HopSh<NT>*>(hop_dyn);
    const HopWs& ws = *wsp;
    const HopReg R(ws);
    const DevGraph& g = S.task.g;
    const Job& job = S.task.job;
    const uint32_t s = S.s, z = S.z;
    const uint64_t i = S.i;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t FULL = 0xFFFFFFFFu;
    const uint32_t* const slot_t = g.slot_t;
    uint32_t* const Ca = R.Ca;
    uint32_t* const Ct = R.Ct;
    u64* const Cs = R.Cs;
    uint32_t* const Gw = R.Gw;
    uint32_t* const Gs = R.Gs;
    uint32_t* const clev = R.clev;
    uint32_t* const glev = R.glev;
    int sp = 0;
    const uint32_t d = k + 1u;               // z's level when found
    uint32_t nC = 0, ng = 1;
    // u's event on the level with events [l0, l1) (whose vertices are in grp), or NONE
    auto event_of = [&](uint32_t u, uint32_t l0, uint32_t l1) -> uint32_t {
        const uint32_t p = R.grp[u];
        return p >= l0 && p < l1 && R.Q[p] == u ? p : NONE;
    };
    // the first of w's slots from which out-edge o is the first later one
    auto first_slot = [&](uint32_t w, uint32_t o) -> uint32_t {
        return o > g.out_ptr[w] ? g.out_pend[o - 1] : g.slot_ptr[w];
    };
    const bool small = found && !job.ob && d <= HOP_DMAX && hop_small<NT>(ws, k, q0, q1, E0);
    if (found && !small) {
        __syncthreads();
        const uint32_t zs = g.slot_ptr[z], ze = g.slot_ptr[z + 1];
        const bool one = job.opt == 1;       // sfm: z's earliest endpoint only
        if (d > 1)
            for (uint32_t p = q0 + tid; p < q1; p += NT) R.grp[R.Q[p]] = p;
        __syncthreads();
        // level d: z's slots with an in-edge from an earlier level-(d-1) state
        for (uint32_t a0 = zs; a0 < ze; a0 += NT) {
            const uint32_t a = a0 + (uint32_t)tid;
            bool f = false;
            uint32_t ta = 0;
            if (a < ze) {
                ta = slot_t[a];
                const uint32_t e1 = g.slot_in[a + 1];
                for (uint32_t e = g.slot_in[a]; e < e1 && !f; ++e) {
                    const uint32_t w = g.in_u[e];
                    if (d == 1) { f = w == s; continue; }
                    const uint32_t p = event_of(w, q0, q1);
                    f = p != NONE && R.ea[p] <= g.in_out[e];
                }
            }
            uint32_t x = f ? 1u : 0u, y = 0, tx, ty;
            block_exclusive_scan2<NT>(x, y, &tx, &ty, S.scan[sp]);
            sp ^= 1;
            if (f && nC + x < ws.c_cap && (!one || nC + x == 0)) { Ca[nC + x] = a; Ct[nC + x] = ta; }
            nC += tx;
            if (one && nC) { nC = 1; break; }
        }
        if (tid == 0) {
            Gw[0] = z; Gs[0] = 0; Gs[1] = nC;
            clev[d] = 0; clev[d - 1] = nC; glev[d] = 0; glev[d - 1] = 1;
        }
        if (nC > ws.c_cap) S.ovf = 2u;
        // level lv - 1 from level lv
        uint32_t cb = 0;                     // first state of level lv
        for (uint32_t lv = d; lv >= 2 && nC <= ws.c_cap; --lv) {
            if (tid == 0) { S.nw = 0; S.nh = 0; }
            if (tid < (int)BLOOM_W) S.bloom[tid] = 0u;
            __syncthreads();
            const uint32_t l0 = R.lev[lv - 1], l1 = R.lev[lv], m0 = R.lev[lv - 2];
            // the tails that matter, each with the end of the slots that a child asks for
            for (uint32_t p = cb + tid; p < nC; p += NT) {
                const uint32_t b = Ca[p];
                const uint32_t e1 = g.slot_in[b + 1];
                for (uint32_t e = g.slot_in[b]; e < e1; ++e) {
                    const uint32_t w = g.in_u[e];
                    const uint32_t x = event_of(w, l0, l1);
                    if (x == NONE || R.ea[x] > g.in_out[e]) continue;
                    if (atomicMax(R.want + w, g.out_pend[g.in_out[e]]) == 0u) R.list[atomicAdd(&S.nw, 1u)] = x;
                }
            }
            __syncthreads();
            const uint32_t nW = S.nw;
            cb = nC;
            // level lv - 2's vertices (read after the next scan's barrier)
            const bool filter = lv > 2 && l0 - m0 <= 2048u;
            if (lv > 2)
                for (uint32_t p = m0 + tid; p < l0; p += NT) {
                    const uint32_t u = R.Q[p], h = bloom_hash(u);
                    R.grp[u] = p;
                    if (filter) atomicOr(S.bloom + (h >> 5), 1u << (h & 31));
                }
            // whether slot a (in-edges from s0 to s1, the first from u) is on level lv - 1
            auto on_level = [&](uint32_t a, uint32_t s0, uint32_t s1, uint32_t u) -> bool {
                if (s1 - s0 > 1u) return __ldcg(R.mst + a) == E0 + lv - 1u;
                if (lv == 2) return u == s;
                const uint32_t h = bloom_hash(u);
                if (filter && !((S.bloom[h >> 5] >> (h & 31u)) & 1u)) return false;
                const uint32_t p = event_of(u, m0, l0);
                if (p == NONE) return false;
                const uint32_t o = g.in_out[s0];
                return R.ea[p] <= o && o < R.eb[p];
            };
            bool done = false;
            for (uint32_t g0 = 0; g0 < nW && !done; g0 += NT) {
                const uint32_t gi = g0 + (uint32_t)tid;
                uint32_t a0 = 0, cnt = 0;
                if (gi < nW) {
                    const uint32_t x = R.list[gi], w = R.Q[x];
                    a0 = first_slot(w, R.ea[x]);
                    cnt = __ldcg(R.want + w) - a0;
                    R.want[w] = 0u;
                }
                uint32_t gx = cnt ? 1u : 0u, ex = cnt, Gc, E;
                block_exclusive_scan2<NT>(gx, ex, &Gc, &E, S.scan[sp]);
                sp ^= 1;
                if (cnt) { S.base[gx] = a0 - ex; S.off[gx] = ex; }
                if (tid < 33) S.off[Gc + tid] = tid ? NONE : E;
                __syncthreads();
                // w's slots from its level-(lv - 1) arrival to the latest time.
                // Few of them are on the level: every warp collects its finds, and up
                // to NT of them are put in slot order (by vertex, then time) by rank
                if (nW <= NT) {
                    const uint32_t per = ((E + NW * 32u - 1u) / (NW * 32u)) * 32u;
                    const uint32_t w_lo = min((uint32_t)wid * per, E), w_hi = min(w_lo + per, E);
                    lbs_walk_warp<CONE_K>(S.off, Gc, S.base, w_lo, w_hi, [&](const uint32_t (&a)[CONE_K]) {
                        uint32_t s0[CONE_K], s1[CONE_K], uu[CONE_K];
#pragma unroll
                        for (int x = 0; x < CONE_K; ++x) {
                            s0[x] = s1[x] = 0u;
                            if (a[x] != NONE) { s0[x] = __ldg(g.slot_in + a[x]); s1[x] = __ldg(g.slot_in + a[x] + 1); }
                        }
#pragma unroll
                        for (int x = 0; x < CONE_K; ++x) uu[x] = s1[x] > s0[x] ? __ldg(g.in_u + s0[x]) : NONE;
#pragma unroll
                        for (int x = 0; x < CONE_K; ++x)
                            if (a[x] != NONE && on_level(a[x], s0[x], s1[x], uu[x])) {
                                const uint32_t p = atomicAdd(&S.nh, 1u);
                                if (p < NT) Ca[nC + p] = a[x];   // nC <= c_cap; the array has NT spare entries
                            }
                    });
                    __syncthreads();
                    const uint32_t H = S.nh;
                    if (H <= NT) {
                        uint32_t a = NONE;
                        if ((uint32_t)tid < H) { a = Ca[nC + tid]; S.base[tid] = a; }
                        __syncthreads();
                        if ((uint32_t)tid < H) {
                            uint32_t r = 0;
                            for (uint32_t y = 0; y < H; ++y) r += S.base[y] < a ? 1u : 0u;
                            S.off[r] = a;
                        }
                        __syncthreads();
                        uint32_t hd = 0, y = 0, tx, ty, v = 0;
                        if ((uint32_t)tid < H) {
                            a = S.off[tid];
                            v = g.slot_v[a];
                            hd = (tid == 0 || g.slot_v[S.off[tid - 1]] != v) ? 1u : 0u;
                        }
                        const uint32_t head = hd;
                        block_exclusive_scan2<NT>(hd, y, &tx, &ty, S.scan[sp]);
                        sp ^= 1;
                        if ((uint32_t)tid < H) {
                            if (nC + tid < ws.c_cap) { Ca[nC + tid] = a; Ct[nC + tid] = slot_t[a]; }
                            if (head) { Gw[ng + hd] = v; Gs[ng + hd] = nC + tid; }
                        }
                        nC += H;
                        done = true;
                        continue;
                    }
                }
                for (uint32_t j0 = 0; j0 < E; j0 += NT) {
                    const uint32_t j = j0 + (uint32_t)tid;
                    bool f = false;
                    uint32_t gg = 0, a = 0;
                    if (j < E) {
                        uint32_t hi = Gc;
                        while (hi - gg > 1) {
                            const uint32_t mid = (gg + hi) >> 1;
                            if (S.off[mid] <= j) gg = mid; else hi = mid;
                        }
                        a = S.base[gg] + j;
                        const uint32_t e = g.slot_in[a], e1 = g.slot_in[a + 1];
                        f = on_level(a, e, e1, g.in_u[e]);
                    }
                    uint32_t x = f ? 1u : 0u, y = 0, tx, ty;
                    block_exclusive_scan2<NT>(x, y, &tx, &ty, S.scan[sp]);
                    sp ^= 1;
                    if (f && nC + x < ws.c_cap) { Ca[nC + x] = a; Ct[nC + x] = slot_t[a]; }
                    nC += tx;
                    if (tx && nC > ws.c_cap) nC = ws.c_cap + 1u;
                }
            }
            if (!done && nC <= ws.c_cap) {       // groups of the ordered list
                __syncthreads();
                uint32_t gc = 0;
                for (uint32_t p0 = cb; p0 < nC; p0 += NT) {
                    const uint32_t p = p0 + (uint32_t)tid;
                    const uint32_t v = p < nC ? g.slot_v[Ca[p]] : NONE;
                    uint32_t x = p < nC && (p == cb || g.slot_v[Ca[p - 1]] != v) ? 1u : 0u, y = 0, tx, ty;
                    const bool head = x != 0u;
                    block_exclusive_scan2<NT>(x, y, &tx, &ty, S.scan[sp]);
                    sp ^= 1;
                    if (head) { Gw[ng + gc + x] = v; Gs[ng + gc + x] = p; }
                    gc += tx;
                }
            }
            ng += nW;
            if (tid == 0) {
                Gs[ng] = nC;
                clev[lv - 2] = nC;
                glev[lv - 2] = ng;
                if (nC > ws.c_cap) S.ovf = 2u;
            }
        }
        __syncthreads();
    }
    // group of w on the level with groups [g0, g1): its states before time tb are [*lo, result)
    auto before = [&](uint32_t w, uint32_t g0, uint32_t g1, uint32_t tb, uint32_t* lo) -> uint32_t {
        const uint32_t x = R.grp[w];
        *lo = 0;
        if (x < g0 || x >= g1 || Gw[x] != w) return 0u;
        *lo = Gs[x];
        return lower_bound_u32(Ct, *lo, Gs[x + 1], tb);
    };
    const bool count = found && !small && !S.ovf;      // block-uniform: S.ovf was set before the last barrier
    if (count) {
        // ---------------- path counts, level by level ----------------
        bool bad = false;
        for (uint32_t lv = 1; lv <= d; ++lv) {
            const uint32_t p0 = clev[lv], p1 = clev[lv - 1], g0 = glev[lv], g1 = glev[lv - 1];
            const uint32_t h0 = g1, h1 = lv > 1 ? glev[lv - 2] : g1;   // groups of level lv - 1
            for (uint32_t p = p0 + tid; p < p1; p += NT) {
                u64 sum = 1ull;               // level 1: the edge from s
                if (lv > 1) {
                    sum = 0ull;
                    const uint32_t b = Ca[p], tb = Ct[p], e1 = g.slot_in[b + 1];
                    for (uint32_t e = g.slot_in[b]; e < e1; ++e) {
                        uint32_t lo;
                        const uint32_t x = before(g.in_u[e], h0, h1, tb, &lo);
                        if (x <= lo) continue;
                        const u64 y = sum + Cs[x - 1];
                        bad |= y < sum;
                        sum = y;
                    }
                }
                Cs[p] = sum;
            }
            __syncthreads();
            // running sums per group (a warp each); this level's groups by vertex
            for (uint32_t x = g0 + (uint32_t)wid; x < g1; x += NW) {
                const uint32_t a0 = Gs[x], a1 = Gs[x + 1];
                if (lane == 0) R.grp[Gw[x]] = x;
                u64 carry = 0;
                if (a1 - a0 > 1u)
                    for (uint32_t b0 = a0; b0 < a1; b0 += 32) {
                        const uint32_t p = b0 + lane;
                        u64 v = p < a1 ? Cs[p] : 0ull;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const u64 y = shfl_up_w(v, o);
                            if (lane >= o) { const u64 sm = v + y; bad |= sm < v; v = sm; }
                        }
                        const u64 sm = v + carry;
                        bad |= sm < v;
                        if (p < a1) Cs[p] = sm;
                        carry = shfl_idx_w(sm, 31);
                    }
            }
            if (bad) S.ovf = 1u;
            __syncthreads();
            if (S.ovf) break;
        }
    }
    const bool drawn = (count || small) && !S.ovf;
    if (drawn && !small && wid == 0) {
        // ---------------- backward draw (warp 0); ob: sigma_sz and the Rademacher bits only ----------------
        const u64 tot = Cs[Gs[1] - 1];
        bool err = false;
        if (!job.ob) {
            u128 x = 0;
            uint32_t rng_ok = 1;
            if (lane == 0) rng_ok = draw_below128((u128)tot, job.seed, i, job.dom_path, &x) ? 1u : 0u;
            rng_ok = __shfl_sync(FULL, rng_ok, 0);
            u64 xs = shfl_idx_w((u64)x, 0);
            if (!rng_ok) { err = true; if (lane == 0) set_status(job.status, ST_RNG); }
            // the first of [lo, hi) whose running sum exceeds xs
            auto pick = [&](uint32_t lo, uint32_t hi) -> uint32_t {
                for (uint32_t b0 = lo; b0 < hi; b0 += 32) {
                    const uint32_t p = b0 + lane;
                    const unsigned msk = __ballot_sync(FULL, p < hi && xs < Cs[p]);
                    if (msk) {
                        const uint32_t r = b0 + (uint32_t)(__ffs(msk) - 1);
                        if (r > lo) xs -= Cs[r - 1];
                        return r;
                    }
                }
                return NONE;
            };
            uint32_t p = err ? NONE : pick(0, Gs[1]);
            err |= p == NONE;
            if (lane == 0) R.path[d] = z;
            for (uint32_t lv = d; !err && lv > 1; --lv) {
                const uint32_t h0 = glev[lv - 1], h1 = glev[lv - 2];
                for (uint32_t x = h0 + lane; x < h1; x += 32) R.grp[Gw[x]] = x;
                __syncwarp();
                const uint32_t b = Ca[p], tb = Ct[p];
                const uint32_t e_hi2 = g.slot_in[b + 1];
                uint32_t nxt = NONE;
                for (uint32_t e0 = g.slot_in[b]; e0 < e_hi2; e0 += 32) {
                    const uint32_t e = e0 + lane;
                    u64 wt = 0;
                    uint32_t w = 0, lo = 0, x = 0;
                    if (e < e_hi2) {
                        w = g.in_u[e];
                        x = before(w, h0, h1, tb, &lo);
                        if (x > lo) wt = Cs[x - 1];
                    }
                    const u64 incl = warp_inclusive_sum(wt);
                    const unsigned msk = __ballot_sync(FULL, xs < incl);
                    if (msk) {
                        const int l = __ffs(msk) - 1;
                        xs -= shfl_idx_w(incl - wt, l);
                        const uint32_t plo = __shfl_sync(FULL, lo, l), phi = __shfl_sync(FULL, x, l);
                        w = __shfl_sync(FULL, w, l);
                        nxt = pick(plo, phi);
                        if (lane == 0) { R.pathe[lv - 1] = e0 + l; R.path[lv - 1] = w; }
                        break;
                    }
                    xs -= shfl_idx_w(incl, 31);
                }
                if (nxt == NONE) { err = true; break; }
                p = nxt;
            }
            if (lane == 0 && !err) {   // the first edge: s's in-edge of the level-1 slot
                const uint32_t b = Ca[p];
                const uint32_t e = lower_bound_u32(g.in_u, g.slot_in[b], g.slot_in[b + 1], s);
                R.path[0] = s;
                if (e < g.slot_in[b + 1] && g.in_u[e] == s) R.pathe[0] = e;
                else err = true;
            }
        }
        if (lane == 0) {
            if (err) { S.err = 1; set_status(job.status, ST_CHECK); }
            S.len = job.ob ? 0u : d + 1u;
            S.sigma = tot;
            uint32_t w4[4];
            philox_block(job.seed, i, DOM_RADE, 0, w4);
            S.rade[0] = w4[0]; S.rade[1] = w4[1]; S.rade[2] = w4[2]; S.rade[3] = w4[3];
        }
    }
    __syncthreads();

    if (S.ovf) {
        // another kernel takes (and counts) the sample
        if (tid == 0) {
            if (S.ovf == 2u) push_capped(job, i); else push_overflow(job, i);
        }
    } else {
        if (!S.err && !job.stats) {
            const uint32_t nint = family_count(job, S.len);
            if (job.hits && nint > 0) {
                const uint32_t rows = 1 + (job.S ? job.c : 0);
                for (uint32_t it = tid; it < nint * rows; it += NT) {
                    const uint32_t p = it % nint, j = it / nint;
                    const uint32_t x = family_item(job, g, R.path, R.pathe, p);
                    if (j == 0) atomicAdd(job.hits + x, 1ull);
                    else {
                        const uint32_t jj = j - 1;
                        const int lam = ((S.rade[jj >> 5] >> (jj & 31)) & 1u) ? 1 : -1;
                        atomicAdd(job.S + (size_t)jj * job.fam + x, lam);
                    }
                }
                if (tid == 0) atomicAdd(job.ctr + C_SUMINT, (u64)nint);
            }
            if (job.rec_len) {
                const uint64_t r = i - job.i0;
                const uint32_t len = S.len;
                if (tid == 0) {
                    job.rec_s[r] = s; job.rec_z[r] = z;
                    job.rec_sig[2 * r] = S.sigma; job.rec_sig[2 * r + 1] = 0ull;
                    job.rec_len[r] = len;
                }
                for (uint32_t p = tid; p < len && p < job.rec_cap; p += NT)
                    job.rec_nodes[r * job.rec_cap + p] = R.path[p];
                if (job.rec_edges)
                    for (uint32_t p = tid; p + 1 < len && p < job.rec_cap; p += NT)
                        job.rec_edges[r * job.rec_cap + p] = R.pathe[p];
            }
        }
        // ---------------- ob (Sec. 4.1; block-uniform condition) ----------------
        if (drawn && job.ob && job.hits && d >= 2) {
            // continuation counts: a child adds its count to the tail's states before
            // its time, a prefix of the tail's group: added to the prefix's last state,
            // then summed from the group's end
            for (uint32_t p = clev[d] + tid; p < clev[0]; p += NT) R.Cb[p] = p < clev[d - 1] ? 1ull : 0ull;
            if (tid == 0) S.nt = 0;
            for (uint32_t lv = d; lv >= 2; --lv) {
                const uint32_t h0 = glev[lv - 1], h1 = glev[lv - 2];
                for (uint32_t x = h0 + tid; x < h1; x += NT) R.grp[Gw[x]] = x;
                __syncthreads();
                for (uint32_t p = clev[lv] + tid; p < clev[lv - 1]; p += NT) {
                    const uint32_t b = Ca[p], tb = Ct[p], e1 = g.slot_in[b + 1];
                    const u64 y = __ldcg(R.Cb + p);
                    for (uint32_t e = g.slot_in[b]; e < e1; ++e) {
                        uint32_t lo;
                        const uint32_t x = before(g.in_u[e], h0, h1, tb, &lo);
                        if (x > lo) atomicAdd(R.Cb + x - 1, y);
                    }
                }
                __syncthreads();
                for (uint32_t x = h0 + (uint32_t)wid; x < h1; x += NW) {
                    const uint32_t a0 = Gs[x], a1 = Gs[x + 1];
                    u64 carry = 0;
                    for (uint32_t b1 = a1; b1 > a0; b1 -= min(32u, b1 - a0)) {
                        const bool in = b1 - a0 > (uint32_t)lane;
                        u64 v = in ? __ldcg(R.Cb + b1 - 1 - lane) : 0ull;
                        v = warp_inclusive_sum(v) + carry;
                        if (in) R.Cb[b1 - 1 - lane] = v;
                        carry = shfl_idx_w(v, 31);
                    }
                }
            }
            __syncthreads();
            // sigma_sz(v) = sum over v's states of sigma * continuations (a path visits v once)
            for (uint32_t x = glev[d - 1] + (uint32_t)wid; x < glev[0]; x += NW) {
                const uint32_t a0 = Gs[x], a1 = Gs[x + 1];
                u64 v = 0;
                for (uint32_t p = a0 + lane; p < a1; p += 32)
                    v += (Cs[p] - (p > a0 ? Cs[p - 1] : 0ull)) * __ldcg(R.Cb + p);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += shfl_xor_w(v, o);
                if (lane == 0 && v && atomicAdd(R.acc + Gw[x], v) == 0ull) R.list[atomicAdd(&S.nt, 1u)] = Gw[x];
            }
            __syncthreads();
            const uint32_t T = S.nt, rows = 2 + (job.S64 ? job.c : 0);
            u64 my_sum = 0;
            for (uint32_t p = tid; p < T; p += NT) {
                const uint32_t v = R.list[p];
                const uint64_t x = ob_q((u128)__ldcg(R.acc + v), (u128)S.sigma);
                R.acc[v] = x;
                my_sum += x;
            }
            __syncthreads();
            for (uint32_t it = tid; it < T * rows; it += NT) {
                const uint32_t v = R.list[it % T];
                const uint64_t x = R.acc[v];
                if (x) ob_term(job, v, x, it / T, S.rade);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) my_sum += __shfl_xor_sync(FULL, my_sum, o);
            if (lane == 0 && my_sum) atomicAdd(job.ctr + C_SUMINT, my_sum);
            __syncthreads();
            for (uint32_t p = tid; p < T; p += NT) R.acc[R.list[p]] = 0ull;
        }
    }
}

}  // namespace

// NT threads per CTA, 64 registers (48 and 40, for more CTAs per SM, spill and
// measured 4 to 25 % slower).  SM: the next level's arrivals in shared memory,
// else in the region.
template <int NT, bool SM>
__global__ void __launch_bounds__(NT, 1024 / NT) k_hop(const Task* tasks, const uint64_t* unit_start,
                                                       const uint32_t* ntasks_p, u64* work,
                                                       const __grid_constant__ HopWs ws) {
    constexpr int NW = NT / 32;
    extern __shared__ __align__(16) unsigned char hop_dyn[];
    HopSh<NT>& S = *reinterpret_cast<HopSh<NT>*>(hop_dyn);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t FULL = 0xFFFFFFFFu;
    const HopReg R(ws);
    uint32_t* const first_sm = reinterpret_cast<uint32_t*>(hop_dyn + sizeof(HopSh<NT>));
    // the next level's earliest arrival of v (see HopReg::fb)
    auto first = [&](uint32_t v) -> uint32_t* { return SM ? first_sm + v : &R.fb[v].x; };

    if constexpr (SM)
        for (uint32_t v = tid; v < ws.n_smem; v += NT) *first(v) = 0u;
    uint32_t lst = *R.stamp;                       // last level stamp used (the same in every thread)
    int sp = 0;                                    // scan scratch in turn
    // thread 0: the finished task's counters
    auto flush = [&]() {
        const int slot[4] = {C_ESCAN, C_EADD, C_SNEW, C_FSEG};
        for (int j = 0; j < 4; ++j) {
            if (S.ctr && S.tot[j]) atomicAdd(S.ctr + slot[j], S.tot[j]);
            S.tot[j] = 0ull;
        }
    };
    // thread 0: the sample's index and vertices (Algorithm 2 draws a source only)
    auto draw = [&](uint64_t q) {
        const Job& job = S.task.job;
        const uint64_t i = job.idx_list ? job.idx_list[q] : job.i0 + q;
        uint32_t s = 0, z = NONE;
        bool ok;
        if (job.stats) {
            uint64_t x = 0;
            ok = draw_below64(S.task.g.n, job.seed, i, DOM_STATS, &x);
            s = (uint32_t)x;
        } else {
            ok = draw_pair(S.task.g.n, job.seed, i, job.dom_pair, &s, &z);
        }
        if (!ok) { set_status(job.status, ST_RNG); s = 0; z = NONE; }
        S.i = i; S.s = s; S.z = z;
        S.ok = ok ? 1u : 0u;
    };
    if (tid == 0) { S.unit = atomicAdd(work, 1ull); S.cur_t = -1; S.ctr = nullptr; S.tot[0] = S.tot[1] = S.tot[2] = S.tot[3] = 0ull; }
    __syncthreads();

    for (;;) {
        uint64_t q = 0;
        if (tid == 0) {
            const uint32_t ntasks = *ntasks_p;
            const uint64_t unit = S.unit;
            int t = -1;
            if (ntasks && unit < unit_start[ntasks]) {
                t = task_of_unit(unit_start, ntasks, unit);
                q = unit - unit_start[t];
                S.unit = atomicAdd(work, 1ull);
            }
            S.t = t;
            if (t >= 0 && t == S.cur_t) draw(q);
            S.nq[0] = S.nq[1] = 0;
            S.ovf = 0; S.err = 0; S.len = 0; S.sigma = 0;
            S.f = S.old = S.dup = 0; S.walk = 0ull;
        }
        if (tid < (int)BLOOM_W) S.bloom[tid] = 0u;
        if (lane == 0) S.esc[wid] = 0ull;
        __syncthreads();
        if (S.t < 0) break;
        if (S.t != S.cur_t) {
            if (wid == 0) {
                const u64* src = reinterpret_cast<const u64*>(tasks + S.t);
                u64* dst = reinterpret_cast<u64*>(&S.task);
                for (uint32_t w = lane; w < sizeof(Task) / 8; w += 32) dst[w] = src[w];
                __syncwarp();
                if (lane == 0) {
                    flush();
                    S.ctr = S.task.job.ctr;
                    draw(q);
                }
            }
            __syncthreads();
            if (tid == 0) S.cur_t = S.t;
        }
        const DevGraph& g = S.task.g;
        const Job& job = S.task.job;
        const bool full = job.stats != 0;     // Algorithm 2: a source only, every vertex searched
        const uint32_t s = S.s;
        bool live = S.ok && (g.out_ptr[s + 1] > g.out_ptr[s]);
        if (live && !full) {
            const uint32_t z = S.z, zs = g.slot_ptr[z], ze = g.slot_ptr[z + 1];
            if (ze == zs) {
                live = false;                 // z has no in-edges
            } else {
                const uint32_t e_lo = g.slot_in[zs], e_hi = g.slot_in[ze];
                const uint32_t tz = g.tmax_in[z];
                if (wid == 0) {
                    const unsigned b = __ballot_sync(FULL, (uint32_t)lane < g.dir_n && g.dir_t[lane] <= tz);
                    if (lane == 0) { S.e_lo = e_lo; S.e_hi = e_hi; S.tz = tz; S.b = (uint32_t)__popc(b) - 1u; }
                }
                // z's in-neighbours, so that a level that touches none of them needs no pull test
                for (uint32_t e = e_lo + tid; e < e_hi; e += NT) {
                    const uint32_t h = bloom_hash(g.in_u[e]);
                    atomicOr(S.bloom + (h >> 5), 1u << (h & 31));
                }
            }
        }
        // slots with several in-edges found on level k hold E0 + k
        if (lst > NONE - (g.n + 16u)) {
            for (uint32_t a = tid; a < ws.A_cap; a += NT) R.mst[a] = 0u;
            lst = 0u;
            __syncthreads();
        }
        const uint32_t E0 = lst + 1u;
        const bool multi = !full && g.max_slot_in > 1u;

        uint32_t k = 0, q0 = 0, q1 = 1, L = 1;      // level k: events [q0, q1), L = q1 - q0
        bool found = false;
        if (tid == 0) { R.lev[0] = 0; R.lev[1] = 1; R.Q[0] = s; }
        __syncthreads();
        // ---------------- levels ----------------
        while (live) {
            if (tid == 0) { S.f += L; if (!full) S.esc[0] += S.e_hi - S.e_lo; }
            const uint32_t* const Qc = full ? R.Q + (size_t)(k & 1u) * ws.n_cap : R.Q + q0;
            uint32_t* const Qn = full ? R.Q + (size_t)((k + 1u) & 1u) * ws.n_cap : R.Q + q1;
            // pull: does level k reach z?  (only if one of its vertices may be an in-neighbour)
            if (!full) {
                bool hit = k == 0;
                if (k > 0)
                    for (uint32_t x = tid; x < L; x += NT) {
                        const uint32_t h = bloom_hash(Qc[x]);
                        hit |= (S.bloom[h >> 5] >> (h & 31u)) & 1u;
                    }
                if (__syncthreads_or(hit)) {
                    hit = false;
                    for (uint32_t e = S.e_lo + tid, e_hi = S.e_hi; e < e_hi; e += NT) {
                        const uint32_t w = g.in_u[e];
                        if (k == 0) {
                            hit |= w == s;
                        } else {
                            const uint32_t f = SM ? *first(w) : __ldcg(first(w));
                            if (f && ~f <= g.in_out[e]) hit = true;
                        }
                    }
                    found = __syncthreads_or(hit) != 0;
                }
            }
            const uint2* const dir = g.dir + (size_t)(full ? g.dir_n - 1u : S.b) * g.n;
            // events of the level: every vertex's arrival, and the out-edges to walk
            uint32_t wl[EVB], wh[EVB], newv = 0;
            for (uint32_t c0 = 0; c0 < L; c0 += NT * EVB) {
                if (k == 0) {
#pragma unroll
                    for (int j = 0; j < EVB; ++j) wl[j] = wh[j] = 0u;
                    if (tid == 0) {
                        uint32_t lo[1] = {g.out_ptr[s]}, hi[1] = {g.out_ptr[s + 1]};
                        wl[0] = lo[0];
                        if (full) lo[0] = hi[0];
                        else if (S.tz > 0u) upper_bounds_5<1>(g.out_t, lo, hi, S.tz - 1u);
                        wh[0] = found ? wl[0] : lo[0];
                        S.esc[0] += wh[0] - wl[0];
                    }
                } else {
                    // EVB vertices per thread, each stage's loads issued for all of them first
                    uint32_t u[EVB], lo[EVB], hi[EVB];
                    uint2 fb[EVB];
#pragma unroll
                    for (int j = 0; j < EVB; ++j) {
                        const uint32_t x = c0 + (uint32_t)tid + (uint32_t)j * NT;
                        u[j] = x < L ? Qc[x] : NONE;
                    }
#pragma unroll
                    for (int j = 0; j < EVB; ++j) {
                        fb[j] = make_uint2(0u, 0u);
                        lo[j] = hi[j] = 0u;
                        if (u[j] != NONE) {
                            if (SM) fb[j] = make_uint2(*first(u[j]), R.fb[u[j]].y);
                            else fb[j] = __ldcg(R.fb + u[j]);
                            if (!found) { const uint2 r = __ldg(dir + u[j]); lo[j] = r.x; hi[j] = r.y; }
                        }
                    }
                    // [wl, wh): from the first edge later than the arrival to the first that an older
                    // level walked (s: every edge) or at tz; the bucket of tz holds the latter, and
                    // it is not below wl (states are earlier than tz)
#pragma unroll
                    for (int j = 0; j < EVB; ++j) {
                        wl[j] = u[j] != NONE ? ~fb[j].x : 0u;
                        lo[j] = full ? hi[j] : min(max(lo[j], wl[j]), hi[j]);
                    }
                    if (!full) upper_bounds_5<EVB>(g.out_t, lo, hi, S.tz - 1u);
                    uint32_t esc = 0;     // at most the graph's edges: the vertices are distinct
#pragma unroll
                    for (int j = 0; j < EVB; ++j) {
                        wh[j] = wl[j];
                        if (u[j] != NONE) {
                            const uint32_t p = q0 + c0 + (uint32_t)tid + (uint32_t)j * NT;
                            const uint32_t lold = u[j] == s ? 0u : ~fb[j].y;      // ~0: not walked before
                            if (!full) {
                                R.ea[p] = wl[j];
                                R.eb[p] = lold;
                            } else if (!fb[j].y && u[j] != s) {
                                ++newv;
                                if (job.clos) atomicAdd(job.clos + u[j], recip32(k));
                            }
                            const uint32_t best = u[j] == s ? 0u : max(fb[j].x, fb[j].y);
                            if (SM) { *first(u[j]) = 0u; R.fb[u[j]].y = best; }
                            else R.fb[u[j]] = make_uint2(0u, best);
                            if (!found) {
                                if (lo[j] > wl[j]) esc += lo[j] - wl[j];
                                wh[j] = min(lo[j], lold);
                            }
                        }
                    }
                    esc = __reduce_add_sync(FULL, esc);
                    if (lane == 0) S.esc[wid] += esc;
                }
                if (L > NT * EVB && !found)
#pragma unroll
                    for (int j = 0; j < EVB; ++j) {
                        const uint32_t x = c0 + (uint32_t)tid + (uint32_t)j * NT;
                        if (x < L) R.rng[x] = make_uint2(wl[j], wh[j]);
                    }
            }
            if (full && k > 0) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) newv += __shfl_xor_sync(FULL, newv, o);
                if (lane == 0 && newv) {
                    atomicAdd(job.cnt + k, (u64)newv);
                    atomicMax(job.dmax, (u64)k);
                }
            }
            if (found) break;
            // walk the ranges
            const uint32_t nx = (k + 1u) & 1u, cur = E0 + k + 1u, cap = full ? NONE : ws.ev_cap - q1;
            for (uint32_t c0 = 0; c0 < L; c0 += NT * EVB) {
                if (L > NT * EVB)
#pragma unroll
                    for (int j = 0; j < EVB; ++j) {
                        const uint32_t x = c0 + (uint32_t)tid + (uint32_t)j * NT;
                        const uint2 r = x < L ? R.rng[x] : make_uint2(0u, 0u);
                        wl[j] = r.x; wh[j] = r.y;
                    }
                uint32_t cand[EVB], gx = 0, ex = 0, Gc, E;
#pragma unroll
                for (int j = 0; j < EVB; ++j) {
                    cand[j] = wh[j] > wl[j] ? wh[j] - wl[j] : 0u;
                    gx += cand[j] > 0u ? 1u : 0u;
                    ex += cand[j];
                }
                block_exclusive_scan2<NT>(gx, ex, &Gc, &E, S.scan[sp]);
                sp ^= 1;
                if (c0 == 0 && tid == 0) S.nq[k & 1u] = 0;
                if (tid == 0) S.walk += E;
                if (!E) continue;
#pragma unroll
                for (int j = 0; j < EVB; ++j)
                    if (cand[j]) { S.base[gx] = wl[j] - ex; S.off[gx] = ex; ++gx; ex += cand[j]; }
                if (tid < 33) S.off[Gc + tid] = tid ? NONE : E;
                __syncthreads();
                const uint32_t per = ((E + NW * 32u - 1u) / (NW * 32u)) * 32u;
                const uint32_t w_lo = min((uint32_t)wid * per, E), w_hi = min(w_lo + per, E);
                lbs_walk_warp<WALK_K>(S.off, Gc, S.base, w_lo, w_hi, [&](const uint32_t (&e)[WALK_K]) {
                    uint32_t v[WALK_K], key[WALK_K], was[WALK_K];
#pragma unroll
                    for (int x = 0; x < WALK_K; ++x) {
                        const uint2 vn = e[x] != NONE ? __ldg(g.out_vn + e[x]) : make_uint2(0u, NONE);
                        v[x] = vn.x; key[x] = ~vn.y;         // key 0: no edge, or nothing new
                    }
#pragma unroll
                    for (int x = 0; x < WALK_K; ++x) {
                        if (v[x] & 0x80000000u) {
                            v[x] &= 0x7FFFFFFFu;
                            if (multi) {
                                const uint32_t a = __ldg(g.out_slot + e[x]), y = __ldcg(R.mst + a);
                                if (y >= E0 && y < cur) { key[x] = 0u; atomicAdd(&S.old, 1u); atomicAdd(&S.dup, 1u); }   // older level
                                else if (atomicMax(R.mst + a, cur) >= E0) { key[x] = 0u; atomicAdd(&S.dup, 1u); }        // another edge
                            }
                        }
                        was[x] = SM ? *first(v[x]) : __ldcg(first(v[x]));
                    }
                    // most edges do not improve their head's arrival: only an improvement is an atomic
#pragma unroll
                    for (int x = 0; x < WALK_K; ++x) was[x] = was[x] < key[x] ? atomicMax(first(v[x]), key[x]) : 1u;
#pragma unroll
                    for (int x = 0; x < WALK_K; ++x)
                        if (was[x] == 0u) {                  // a first touch
                            const uint32_t p = atomicAdd(S.nq + nx, 1u);
                            if (p < cap) Qn[p] = v[x]; else S.ovf = 2u;
                        }
                });
                __syncthreads();
            }
            L = S.nq[nx];
            if (L == 0 || S.ovf) break;
            q0 = q1; q1 += L; ++k;
            if (!full && tid == 0) R.lev[k + 1] = q1;
        }
        lst = E0 + k + 1u;
        hop_finish<NT>(&ws, found, k, q0, q1, E0);
        if (S.ovf) {
            // pending arrivals are dropped
            for (uint32_t v = tid; v < g.n; v += NT) { *first(v) = 0u; R.fb[v].y = 0u; }
        } else if (full) {
            for (uint32_t v = tid; v < g.n; v += NT) R.fb[v].y = 0u;
        } else {
            for (uint32_t p = 1u + (uint32_t)tid; p < q1; p += NT) R.fb[R.Q[p]].y = 0u;
        }
        if (!S.ovf && tid == 0) {
            for (int w = 0; w < NW; ++w) S.tot[0] += S.esc[w];
            S.tot[1] += S.walk - S.old;
            S.tot[2] += S.walk - S.dup;
            S.tot[3] += S.f;
        }
        __syncthreads();
    }
    if (tid == 0) {
        flush();
        *R.stamp = lst;
    }
}

// Host-side launch helpers -------------------------------------------------

// Region of one CTA.  Above 2^18 slots (where a region would grow from 10 to 19
// bytes a slot) the events of a sample are capped at A / 4 + 2 n + 4096 (a
// search of the bursty graphs makes one event per five states), and the states
// on optimal paths at A / 8 + 65536 (they are a few hundred at most there);
// a sample that needs more goes to k_bfs, which has no such cap.
size_t hop_region_bytes(uint32_t n, uint32_t A, HopWs* ws) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const uint64_t all = (uint64_t)A + 1;
    ws->n_cap = n;
    ws->A_cap = A;
    ws->ev_cap = (uint32_t)(A <= 1u << 18 ? all : std::min<uint64_t>(all, (uint64_t)A / 4 + 2ull * n + 4096));
    ws->c_cap = (uint32_t)std::min<uint64_t>(all, (uint64_t)A / 8 + 65536);
    const size_t nq = std::max<size_t>(ws->ev_cap, 2 * (size_t)n), ng = (size_t)ws->c_cap + n + 4;
    size_t o = 0;
    ws->o_fb = o;     o = al(o + (size_t)n * 8);
    ws->o_want = o;   o = al(o + (size_t)n * 4);
    ws->o_grp = o;    o = al(o + (size_t)n * 4);
    ws->o_grp2 = o;   o = al(o + (size_t)n * 4);
    ws->o_acc = o;    o = al(o + (size_t)n * 8);
    ws->o_q = o;      o = al(o + (nq + 1) * 4);
    ws->o_ea = o;     o = al(o + ((size_t)ws->ev_cap + 1) * 4);
    ws->o_eb = o;     o = al(o + ((size_t)ws->ev_cap + 1) * 4);
    ws->o_rng = o;    o = al(o + (size_t)n * 8);
    ws->o_lev = o;    o = al(o + 3 * ((size_t)n + 4) * 4);
    ws->o_mst = o;    o = al(o + (size_t)A * 4);
    ws->o_ca = o;     o = al(o + ((size_t)ws->c_cap + 1024) * 4);
    ws->o_ct = o;     o = al(o + (size_t)ws->c_cap * 4);
    ws->o_cs = o;     o = al(o + (size_t)ws->c_cap * 8);
    ws->o_cb = o;     o = al(o + (size_t)ws->c_cap * 8);
    ws->o_gw = o;     o = al(o + ng * 4);
    ws->o_gs = o;     o = al(o + ng * 4);
    ws->o_path = o;   o = al(o + (size_t)(n + 2) * 4);
    ws->o_pathe = o;  o = al(o + (size_t)(n + 2) * 4);
    ws->o_stamp = o;  o = al(o + 4);
    return o;
}

// Dynamic shared memory of the nt-thread kernel; n: nodes whose arrivals are in
// shared memory.
size_t hop_smem_bytes(int nt, uint32_t n) {
    const size_t s = nt == 1024 ? sizeof(HopSh<1024>) : (nt == 512 ? sizeof(HopSh<512>) : sizeof(HopSh<256>));
    return s + (size_t)n * 4;
}

namespace {

const void* hop_kernel(int nt, bool sm) {
    if (nt == 1024) return sm ? (const void*)k_hop<1024, true> : (const void*)k_hop<1024, false>;
    if (nt == 512) return sm ? (const void*)k_hop<512, true> : (const void*)k_hop<512, false>;
    return sm ? (const void*)k_hop<256, true> : (const void*)k_hop<256, false>;
}

}  // namespace

// Raises (never lowers) the dynamic shared-memory limit of the kernels on the
// current device.
cudaError_t hop_configure(size_t smem) {
    static std::mutex mu;
    static size_t configured[64] = {};
    int dev = 0;
    const cudaError_t ed = cudaGetDevice(&dev);
    if (ed != cudaSuccess) return ed;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= configured[dev]) return cudaSuccess;
    for (int nt : {256, 512, 1024})
        for (bool sm : {false, true}) {
            const cudaError_t e = cudaFuncSetAttribute(hop_kernel(nt, sm), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)smem);
            if (e != cudaSuccess) return e;
        }
    configured[dev] = smem;
    return cudaSuccess;
}

cudaError_t hop_blocks_per_sm(int nt, bool first_in_smem, size_t smem, int* out) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, hop_kernel(nt, first_in_smem), nt, smem);
}

cudaError_t launch_hop(const Task* tasks, const uint64_t* unit_start, const uint32_t* ntasks, u64* work,
                       const HopWs& ws, int grid, cudaStream_t st) {
    HopWs w = ws;
    const size_t smem = hop_smem_bytes(ws.nt, ws.n_smem);
    void* args[] = {(void*)&tasks, (void*)&unit_start, (void*)&ntasks, (void*)&work, (void*)&w};
    return cudaLaunchKernel(hop_kernel(ws.nt, ws.n_smem != 0), dim3(grid), dim3(ws.nt), args, smem, st);
}

// Per out-edge e = (u, v, t): its head and the head's first later out-edge
// (out_vn), e's place in the in-CSR (in_out: in-edge -> out-edge), and one
// past u's last slot earlier than t (out_pend).
__global__ void k_edge_maps(DevGraph g, uint2* out_vn, uint32_t* in_out, uint32_t* out_pend) {
    const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= g.m) return;
    uint32_t u = 0, hi = g.n;                        // the row of e: out_ptr[u] <= e < out_ptr[hi]
    while (hi - u > 1) {
        const uint32_t mid = u + ((hi - u) >> 1);
        if (g.out_ptr[mid] <= e) u = mid; else hi = mid;
    }
    const uint32_t a = g.out_slot[e], s0 = g.slot_in[a], s1 = g.slot_in[a + 1];
    out_vn[e] = make_uint2(g.out_v[e] | (s1 - s0 > 1u ? 0x80000000u : 0u), g.slot_nout[a]);
    in_out[lower_bound_u32(g.in_u, s0, s1, u)] = e;
    out_pend[e] = lower_bound_u32(g.slot_t, g.slot_ptr[u], g.slot_ptr[u + 1], g.out_t[e]);
}

// dir[b n + v]: the edges of v's out-row that bucket b of the times spans.
__global__ void k_edge_dir(DevGraph g, DirTimes dt, uint2* dir, uint32_t* dir_t) {
    const uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x < 32) dir_t[x] = dt.t[x];
    if (x >= (uint64_t)g.n * g.dir_n) return;
    const uint32_t b = (uint32_t)(x / g.n), v = (uint32_t)(x - (uint64_t)b * g.n);
    const uint32_t r0 = g.out_ptr[v], r1 = g.out_ptr[v + 1];
    const uint32_t lo = lower_bound_u32(g.out_t, r0, r1, dt.t[b]);
    dir[x] = make_uint2(lo, b + 1 < g.dir_n ? lower_bound_u32(g.out_t, lo, r1, dt.t[b + 1]) : r1);
}

// Fills out_vn, in_out, out_pend, dir and dir_t of g (whose other arrays are in place).
cudaError_t launch_edge_maps(const DevGraph& g, const DirTimes& dt, uint2* out_vn, uint32_t* in_out, uint32_t* out_pend,
                             uint2* dir, uint32_t* dir_t, cudaStream_t st) {
    if (g.m) k_edge_maps<<<(g.m + 255) / 256, 256, 0, st>>>(g, out_vn, in_out, out_pend);
    const uint64_t d = (uint64_t)g.n * g.dir_n;
    k_edge_dir<<<(unsigned)((d + 255) / 256), 256, 0, st>>>(g, dt, dir, dir_t);
    return cudaGetLastError();
}

}  // namespace mantra
