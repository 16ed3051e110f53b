// Prefix-foremost (pfm) samples 32 at a time by one sweep over the time-sorted
// edges (paper Sec. 3 Def. 1(3), the stream scan of Sec. 4.4), the backward
// path draw (App. C) and the Update step of Algorithm 1.
//
// R[v] holds a bit per sample: v is reached.  An edge (u, v, t) carries the bits
// R[u] & ~R[v] to v, with arrival t: one and-not serves 32 samples where a
// search per sample walks every edge 32 times.  Edges must be applied in time
// order, but an edge only depends on earlier edges into its own ends.  The
// store keeps the stream cut into waves: at most 32 consecutive edges, whole
// time steps, in which no edge's tail or head is the head of an earlier edge
// of another time (k_wave_cut).  A wave's edges read R as it stood before the
// wave and may then be applied together, one lane each; edges of one time step
// never depend on each other (times strictly increase along a path).
// A time step of more than 32 edges takes several waves, read first and then
// applied.  On the bursty 20,000-node graph a wave has 18 edges (hubs cut them).
//
// A sample ends at the arrival of its z, or at z's latest in-edge time: the
// wave in which that happens is applied time step by time step.  Arrivals are
// logged as they happen: one record (head, bits, slot) per edge that brought
// any.  Reading the log backward once then resolves all 32 paths: nearly every
// arrival slot has one in-edge, so a path's current vertex and its record give
// the vertex before it, whose record lies further back.  A path that meets a
// slot with several in-edges may have a choice; its sample's arrivals are
// copied out of the log, and the vertices that lead to z are counted and drawn
// from by the whole warp (draw_choice).  Samples with more than 1,024 of them, or
// with a path of more than 2,048 vertices, go to k_pfm_cta.
//
// What bounds it: the chain of a wave (a shared-memory read, the and-not, the
// store back), 72 ns; the edges are prefetched, the usual batch of eight waves
// has no branch and no vote on that chain (with a vote per wave 200 ns); 0.16
// instructions issued per scheduler and cycle, L2 at 3 %, DRAM at 2 %.  So a
// CTA is one warp, and the samples in flight are set by the shared memory of R,
// 4 n bytes a warp.  42,000 samples of the bursty 20,000-node graph take 9.1
// ms; a search per sample (k_pfm_cta) takes 33.4 ms.
#include "mantra_dev.cuh"
#include "waves.h"

#include <algorithm>
#include <mutex>

namespace mantra {

namespace {

constexpr uint32_t WB = WAVE_BATCH;    // waves per batch
constexpr uint32_t PF = 4;             // batches in the prefetch ring
constexpr uint32_t FULL = 0xFFFFFFFFu;

__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

}  // namespace

// Dynamic shared memory: R[n + 1] | waiting bits | mark bits (of n_smem nodes).
__global__ void __launch_bounds__(32) k_sweep(const Task* tasks, const uint64_t* unit_start, const uint32_t* ntasks_p,
                                              u64* work, const __grid_constant__ SweepWs ws) {
    extern __shared__ __align__(16) uint32_t sweep_dyn[];
    __shared__ __align__(16) Task sh_task;
    __shared__ uint32_t sh_cnt;
    __shared__ __align__(16) uint2 ring[PF][WB][32];       // batches, copied ahead; a lane reads its own edges only
    const uint32_t lane = threadIdx.x;
    const uint32_t bw = (ws.n_smem + 32) / 32;
    uint32_t* const R = sweep_dyn;
    uint32_t* const WM = sweep_dyn + ws.n_smem + 1;          // vertices that some path waits at
    uint32_t* const MK = WM + bw;
    char* const region = ws.base + (size_t)blockIdx.x * ws.stride;
    uint4* const log = reinterpret_cast<uint4*>(region + ws.o_log);           // arrivals: head, samples, place in the waves
    uint32_t* const arr = reinterpret_cast<uint32_t*>(region + ws.o_arr);     // one sample's arrival slots
    uint32_t* const stp = reinterpret_cast<uint32_t*>(region + ws.o_stp);     // bits of a step of several waves
    uint32_t* const path = reinterpret_cast<uint32_t*>(region + ws.o_path);   // [sample][path_cap], from z
    uint32_t* const pathe = reinterpret_cast<uint32_t*>(region + ws.o_pathe); // in-CSR index of the edge into path[k]
    uint32_t* const cv = reinterpret_cast<uint32_t*>(region + ws.o_cv);       // vertices that lead to z
    uint32_t* const co = reinterpret_cast<uint32_t*>(region + ws.o_co);       // the same by arrival time
    u64* const ck = reinterpret_cast<u64*>(region + ws.o_ck);                 // their sort keys
    u64* const sig = reinterpret_cast<u64*>(region + ws.o_sig);               // their path counts, by vertex

    for (uint32_t v = lane; v < bw; v += 32) { WM[v] = 0u; MK[v] = 0u; }
    const uint32_t ntasks = *ntasks_p;
    const uint64_t total = ntasks ? unit_start[ntasks] : 0ull;
    int cur_t = -1;
    for (;;) {
        uint64_t unit = 0;
        if (lane == 0) unit = atomicAdd(work, 1ull);
        unit = __shfl_sync(FULL, unit, 0);
        if (unit >= total) break;
        const int t = task_of_unit(unit_start, ntasks, unit);
        if (t != cur_t) {
            cur_t = t;
            __syncwarp();
            const u64* src = reinterpret_cast<const u64*>(tasks + t);
            u64* dst = reinterpret_cast<u64*>(&sh_task);
            for (uint32_t w = lane; w < sizeof(Task) / 8; w += 32) dst[w] = src[w];
            __syncwarp();
        }
        const DevGraph& g = sh_task.g;
        const Job& job = sh_task.job;
        const uint32_t n = g.n;
        // ---- lane j: sample j of the unit ----
        uint64_t q = (unit - unit_start[t]) * 32ull + lane;
        const bool have = q < job.count;
        if (have && ws.order) q = ws.order[unit * 32ull + lane];
        const uint64_t i = have ? (job.idx_list ? job.idx_list[q] : job.i0 + q) : 0ull;
        uint32_t s = n, z = n;
        bool live = have;
        if (have && !draw_pair(n, job.seed, i, job.dom_pair, &s, &z)) {
            set_status(job.status, ST_RNG);
            live = false;
            s = z = n;
        }
        live = live && g.out_ptr[s + 1] > g.out_ptr[s] && g.slot_ptr[z + 1] > g.slot_ptr[z];
        const uint32_t ts = live ? g.tmin_out[s] : NONE, tz = live ? g.tmax_in[z] : 0u;
        const uint32_t bit = 1u << lane;
        for (uint32_t v = lane; v <= n; v += 32) R[v] = 0u;
        __syncwarp();
        if (live) atomicOr(R + s, bit);
        __syncwarp();
        // a sample whose window is empty has nothing to reach (ts > tz)
        uint32_t act = __ballot_sync(FULL, live && ts <= tz);
        uint32_t te = tz;                                   // the sample's last time
        bool reached = false;
        const uint32_t ts0 = __reduce_min_sync(FULL, ts);
        uint32_t next_end = __reduce_min_sync(FULL, (act & bit) ? te : NONE);
        u64 c_add = 0;
        // ---- the waves from the first that holds a time >= ts0 ----
        uint32_t w0 = 0;
        {
            uint32_t hi = g.n_waves;
            while (w0 < hi) {
                const uint32_t mid = w0 + ((hi - w0) >> 1);
                if (g.wave_t[mid] < ts0) w0 = mid + 1; else hi = mid;   // wave_t: the wave's last time
            }
        }
        const uint2* const uv = g.wave_uv;
        const uint2* const at = g.wave_at;
        const uint32_t nb_all = act ? g.n_waves / WB : 0u;  // (n_waves is a multiple of WB)
        auto fetch = [&](uint32_t b) {                      // batch b's edges of the lane, into the ring
            if (b < nb_all)
#pragma unroll
                for (uint32_t x = 0; x < WB; ++x) cp_async8(&ring[b % PF][x][lane], uv + ((size_t)b * WB + x) * 32u + lane);
            cp_async_commit();
        };
        uint32_t nlog = 0;
        // the warp's edges bring the samples nb to the heads v
        auto apply = [&](uint32_t v, uint32_t pos, uint32_t nb) {
            const unsigned on = __ballot_sync(FULL, nb != 0u);
            if (nb) {
                atomicOr(R + v, nb);
                log[nlog + __popc(on & (bit - 1u))] = make_uint4(v, nb, pos, 0u);
            }
            c_add += __popc(nb);
            nlog += __popc(on);
        };
        // samples that reached z since the log had log0 records: their last time, from those
        // records; what they gained at later times is not counted
        auto settle = [&](uint32_t log0) {
            const unsigned hit = __ballot_sync(FULL, (act & bit) && (R[z] & bit));
            if (!hit) return;
            __syncwarp();                                   // (a vote does not order the lanes' log records)
            for (uint32_t p0 = log0; p0 < nlog; p0 += 32) {
                const uint32_t p = p0 + lane;
                const uint4 r = p < nlog ? log[p] : make_uint4(n, 0u, 0u, 0u);
                for (unsigned d = hit; d; d &= d - 1) {
                    const int j = __ffs(d) - 1;
                    const uint32_t zj = __shfl_sync(FULL, z, j);
                    const unsigned f = __ballot_sync(FULL, r.x == zj && ((r.y >> j) & 1u));
                    if (f) {
                        const uint32_t pos = __shfl_sync(FULL, r.z, __ffs(f) - 1);
                        if ((int)lane == j) { reached = true; te = __ldg(at + pos).y; }
                    }
                }
            }
            for (uint32_t p0 = log0; p0 < nlog; p0 += 32) {
                const uint32_t p = p0 + lane;
                const uint4 r = p < nlog ? log[p] : make_uint4(n, 0u, 0u, 0u);
                const uint32_t tp = r.y ? __ldg(at + r.z).y : 0u;
                for (unsigned d = hit; d; d &= d - 1) {
                    const int j = __ffs(d) - 1;
                    const uint32_t tj = __shfl_sync(FULL, te, j);
                    if (((r.y >> j) & 1u) && tp > tj) c_add -= 1;
                }
            }
            act &= ~hit;
            next_end = __reduce_min_sync(FULL, (act & bit) ? te : NONE);
        };
        uint32_t nstp = 0;                                  // waves read of a step of several
        const uint32_t b0 = w0 / WB;
        for (uint32_t x = 0; x + 1 < PF; ++x) fetch(b0 + x);
        uint2 info_next = b0 < nb_all ? __ldg(g.wave_info + b0) : make_uint2(0u, 0u);
        for (uint32_t b = b0; b < nb_all && act; ++b) {
            fetch(b + PF - 1);
            const uint2 info = info_next;                   // the batch's last time; not 0: has a special wave
            if (b + 1 < nb_all) info_next = __ldg(g.wave_info + b + 1);
            cp_async_wait<PF - 1>();
            if (info.y == 0u && info.x <= next_end) {
                // no vote and no branch: heads are distinct within a wave, so the head's bits
                // are stored back; the log entry is off the chain
                uint2 e[WB];
#pragma unroll
                for (uint32_t x = 0; x < WB; ++x) e[x] = ring[b % PF][x][lane];
                const uint32_t log0 = nlog;
#pragma unroll
                for (uint32_t x = 0; x < WB; ++x) {
                    const uint32_t rv = R[e[x].y], nb = R[e[x].x] & ~rv & act;
                    __syncwarp();
                    R[e[x].y] = rv | nb;
                    __syncwarp();
                    const unsigned on = __ballot_sync(FULL, nb != 0u);
                    if (nb) log[nlog + __popc(on & (bit - 1u))] = make_uint4(e[x].y, nb, (b * WB + x) * 32u + lane, 0u);
                    nlog += __popc(on);
                    c_add += __popc(nb);
                }
                settle(log0);
            } else {
                // a wave at a time; time step by time step where a sample may end by its z's
                // latest in-edge time, or where a step spans waves
                const uint32_t wx = b * WB + (lane % WB);
                const uint32_t flx = __ldg(g.wave_fl + wx), tlx = __ldg(g.wave_t + wx);
                for (uint32_t x = 0; x < WB && act; ++x) {
                    const uint2 e = ring[b % PF][x][lane];
                    const uint32_t pos = (b * WB + x) * 32u + lane, u = e.x;
                    const uint32_t fl = __shfl_sync(FULL, flx, x), tl = __shfl_sync(FULL, tlx, x);
                    if (!(fl & WAVE_BIG) && tl <= next_end) {
                        const uint32_t log0 = nlog, m = R[u] & ~R[e.y] & act;
                        __syncwarp();
                        apply(e.y, pos, m);
                        __syncwarp();
                        settle(log0);
                        continue;
                    }
                    const uint32_t te_e = __ldg(at + pos).y;
                    unsigned todo = __ballot_sync(FULL, u != n);
                    while (todo && act) {
                        const int l = __ffs(todo) - 1;
                        const uint32_t tm = __shfl_sync(FULL, te_e, l);               // in time order
                        const bool mine = u != n && te_e == tm;
                        act &= ~__ballot_sync(FULL, (act & bit) && te < tm);          // z's latest in-edge is past
                        const uint32_t m = mine ? R[u] & ~R[e.y] & act : 0u;
                        __syncwarp();
                        todo &= ~__ballot_sync(FULL, mine);
                        if (!(fl & WAVE_BIG)) {
                            apply(e.y, pos, m);
                        } else {
                            // a step of several waves: all are read before any is applied
                            stp[nstp * 32u + lane] = m;
                            ++nstp;
                            if (!(fl & WAVE_LAST)) break;
                            __syncwarp();
                            for (uint32_t y = 0; y < nstp; ++y) {
                                const uint32_t ps = (b * WB + x + 1u - nstp + y) * 32u + lane;
                                apply(__ldg(uv + ps).y, ps, stp[y * 32u + lane]);
                            }
                            nstp = 0;
                        }
                        __syncwarp();
                        if ((act & bit) && (R[z] & bit)) { reached = true; te = tm; }
                        act &= ~__ballot_sync(FULL, reached);
                    }
                }
                next_end = __reduce_min_sync(FULL, (act & bit) ? te : NONE);
            }
        }
        cp_async_wait<0>();
        // (a sample's own step te was applied whole: the step that reached z, or all steps up to tz)

        // ---- edges of the scan window: tmin_out(s) <= t <= te, not into s ----
        u64 c_scan = 0;
        if (live && ts <= te) {
            const uint32_t a = lower_bound_u32(g.st_t, 0, g.m, ts), b = lower_bound_u32(g.st_t, a, g.m, te + 1u);
            const uint32_t s0 = g.slot_ptr[s], s1 = g.slot_ptr[s + 1];
            const uint32_t sa = lower_bound_u32(g.slot_t, s0, s1, ts), sb = lower_bound_u32(g.slot_t, sa, s1, te + 1u);
            c_scan = (u64)(b - a) - (u64)(g.slot_in[sb] - g.slot_in[sa]);
        }
        // ---- backward from z through the log, all samples together ----
        uint32_t len = 0;                                    // path vertices
        bool choice = false, ovf = false, capped = false, err = false;
        u64 sigma = 0;
        {
            uint32_t cur = reached ? z : NONE;               // the path's vertex whose record is wanted
            if (cur != NONE) atomicOr(WM + (cur >> 5), 1u << (cur & 31u));
            __syncwarp();
            unsigned open = __ballot_sync(FULL, cur != NONE);
            uint32_t* const pv = path + (size_t)lane * ws.path_cap;
            uint32_t* const pe = pathe + (size_t)lane * ws.path_cap;
            constexpr int LK = 4;                            // chunks of the log with loads in flight
            uint4 nx[LK];
            const uint32_t nh = (nlog + 31u) / 32u;
            auto chunk = [&](uint32_t y) -> uint4 {          // the y-th chunk from the end
                const uint32_t p = (nh - 1u - y) * 32u + lane;
                return y < nh && p < nlog ? log[p] : make_uint4(0u, 0u, 0u, 0u);
            };
#pragma unroll
            for (int y = 0; y < LK; ++y) nx[y] = chunk(y);
            for (uint32_t y0 = 0; y0 < nh && open; y0 += LK)
#pragma unroll
            for (int yy = 0; yy < LK; ++yy) {
                const uint4 r = nx[yy];
                nx[yy] = chunk(y0 + yy + LK);
                // (the mark of a vertex may be stale: the exact test is below)
                unsigned hit = __ballot_sync(FULL, (r.y & open) && ((WM[r.x >> 5] >> (r.x & 31u)) & 1u));
                while (hit) {                                // the latest record first
                    const int l = 31 - __clz(hit);
                    hit &= ~(1u << l);
                    const uint32_t v = __shfl_sync(FULL, r.x, l), nb = __shfl_sync(FULL, r.y, l), pos = __shfl_sync(FULL, r.z, l);
                    const bool at = cur == v && (nb & bit);
                    if (!__any_sync(FULL, at)) continue;
                    if (at) {
                        const uint32_t a = __ldg(g.wave_at + pos).x, e0 = g.slot_in[a];
                        if (g.slot_in[a + 1] - e0 > 1u) { choice = true; cur = NONE; }
                        else if (len + 2 > ws.path_cap) { capped = true; cur = NONE; }
                        else {
                            pv[len] = v; pe[len] = e0;
                            ++len;
                            cur = g.in_u[e0];
                            if (cur == s) { pv[len] = s; ++len; sigma = 1; cur = NONE; }   // the only path: nothing to draw
                            else atomicOr(WM + (cur >> 5), 1u << (cur & 31u));
                        }
                    }
                    open = __ballot_sync(FULL, cur != NONE);
                    __syncwarp();
                    // earlier records of this chunk that the paths now wait for
                    hit = __ballot_sync(FULL, (int)lane < l && (r.y & open) && ((WM[r.x >> 5] >> (r.x & 31u)) & 1u));
                }
            }
            if (cur != NONE) err = true;                     // every reached vertex has a record
            for (uint32_t x = lane; x < bw; x += 32) WM[x] = 0u;
            __syncwarp();
        }
        if (choice || capped) len = 0;
        // fa(w) < tv for the sample whose arrivals are in arr, with source src
        auto fa_before = [&](uint32_t w, uint32_t src, uint32_t j, uint32_t tv) -> bool {
            if (w == src) return true;
            return ((R[w] >> j) & 1u) && g.slot_t[arr[w]] < tv;
        };
        auto copy_arrivals = [&](uint32_t j) {
            __syncwarp();
            for (uint32_t p = lane; p < nlog; p += 32) {
                const uint4 r = log[p];
                if ((r.y >> j) & 1u) arr[r.x] = __ldg(g.wave_at + r.z).x;
            }
            __syncwarp();
        };
        // ---- samples with a choice: counts over the vertices that lead to z, by the warp ----
        for (unsigned todo = __ballot_sync(FULL, choice); todo; todo &= todo - 1) {
            const uint32_t j = __ffs(todo) - 1;
            const uint32_t sj = __shfl_sync(FULL, s, j), zj = __shfl_sync(FULL, z, j);
            const uint64_t ij = __shfl_sync(FULL, i, j);
            copy_arrivals(j);
            uint32_t plen = 0;
            u64 tot = 0;
            const int got = draw_choice(g, job, ij, sj, zj, arr, [&](uint32_t w, uint32_t tv) { return fa_before(w, sj, j, tv); },
                                        ChoiceWs{cv, co, ck, sig, MK, ws.cone_cap, ws.path_cap}, &sh_cnt,
                                        path + (size_t)j * ws.path_cap, pathe + (size_t)j * ws.path_cap, &plen, &tot);
            if (lane == j) {
                choice = false;
                ovf = got == CHOICE_OVF;
                capped = got == CHOICE_CAPPED;
                err = got == CHOICE_ERR;
                if (got == CHOICE_DRAWN) { len = plen; sigma = tot; }
            }
            __syncwarp();
        }
        if (err) set_status(job.status, ST_CHECK);
        if (ovf) push_overflow(job, i);
        if (capped) push_capped(job, i);
        // ---- hits, Rademacher sums and records, a sample at a time ----
        uint32_t rade[4] = {0, 0, 0, 0};
        if (len > 0) philox_block(job.seed, i, DOM_RADE, 0, rade);
        u64 c_int = 0;
        __syncwarp();
        for (unsigned todo = __ballot_sync(FULL, have && !ovf && !capped && !err && (len > 0 || job.rec_len)); todo; todo &= todo - 1) {
            const uint32_t j = __ffs(todo) - 1;
            const uint32_t lj = __shfl_sync(FULL, len, j);
            const uint32_t nint = job.target == 0 ? (lj < 2 ? 0u : lj - 2u) : (lj < 2 ? 0u : lj - 1u);
            uint32_t rj[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) rj[x] = __shfl_sync(FULL, rade[x], j);
            const uint32_t* const pv = path + (size_t)j * ws.path_cap;     // pv[lj - 1 - k]: vertex k from s
            const uint32_t* const pe = pathe + (size_t)j * ws.path_cap;    // pe[lj - 2 - k]: edge k from s
            if (job.hits && nint > 0) {
                const uint32_t rows = 1 + (job.S ? job.c : 0);
                for (uint32_t it = lane; it < nint * rows; it += 32) {
                    const uint32_t p = it % nint, jr = it / nint;
                    const uint32_t x = job.target == 0 ? pv[lj - 2 - p]
                                       : (job.target == 2 ? pe[lj - 2 - p] : g.in_uedge[pe[lj - 2 - p]]);
                    if (jr == 0) {
                        atomicAdd(job.hits + x, 1ull);
                    } else {
                        const uint32_t jj = jr - 1;
                        const int lam = ((rj[jj >> 5] >> (jj & 31)) & 1u) ? 1 : -1;
                        atomicAdd(job.S + (size_t)jj * job.fam + x, lam);
                    }
                }
                c_int += nint;
            }
            if (job.rec_len) {
                const uint32_t sj = __shfl_sync(FULL, s, j), zj = __shfl_sync(FULL, z, j);
                const u64 sgj = __shfl_sync(FULL, sigma, j);
                const uint64_t r = __shfl_sync(FULL, i, j) - job.i0;
                if (lane == 0) {
                    job.rec_s[r] = sj; job.rec_z[r] = zj;
                    job.rec_sig[2 * r] = sgj; job.rec_sig[2 * r + 1] = 0ull;
                    job.rec_len[r] = lj;
                }
                for (uint32_t p = lane; p < lj && p < job.rec_cap; p += 32) job.rec_nodes[r * job.rec_cap + p] = pv[lj - 1 - p];
                if (job.rec_edges)
                    for (uint32_t p = lane; p + 1 < lj && p < job.rec_cap; p += 32)
                        job.rec_edges[r * job.rec_cap + p] = pe[lj - 2 - p];
            }
        }
        // ---- counters; a sample that another kernel re-runs is counted there ----
        for (unsigned todo = __ballot_sync(FULL, ovf || capped); todo; todo &= todo - 1) {
            const uint32_t j = __ffs(todo) - 1, sj = __shfl_sync(FULL, s, j), tej = __shfl_sync(FULL, te, j);
            copy_arrivals(j);
            if (lane == j) c_scan = 0;
            for (uint32_t v = lane; v < n; v += 32) {
                if (v == sj || !((R[v] >> j) & 1u)) continue;
                const uint32_t a = arr[v], e0 = g.slot_in[a], e1 = g.slot_in[a + 1], tv = g.slot_t[a];
                if (tv > tej) continue;
                for (uint32_t e = e0; e < e1; ++e)
                    if (e1 - e0 == 1u || fa_before(g.in_u[e], sj, j, tv)) c_add -= 1;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            c_scan += shfl_xor_w(c_scan, o);
            c_add += shfl_xor_w(c_add, o);
        }
        if (lane == 0) {
            if (c_scan) atomicAdd(job.ctr + C_ESCAN, c_scan);
            if (c_add) atomicAdd(job.ctr + C_EADD, c_add);
            if (c_int) atomicAdd(job.ctr + C_SUMINT, c_int);
        }
        __syncwarp();
    }
}

// The samples of a task ordered by the parts of the time range in which they
// run (from s's first out-edge to z's last in-edge), so that a warp's 32 samples
// need about the same part of the stream; the longest first.  One CTA per task,
// a counting sort by the two times' buckets; order: 32 places per unit.  On the
// bursty 20,000-node graph 42,000 samples take 9.1 ms so (this kernel included),
// 14.9 as they come; 8,000 of the uniform 50,000-node graph 12.3 and 17.9.
__global__ void __launch_bounds__(1024) k_sweep_order(const Task* tasks, const uint64_t* unit_start,
                                                      const uint32_t* ntasks_p, uint32_t* order) {
    __shared__ uint32_t hist[1024], sm[32];
    const uint32_t ntasks = *ntasks_p, tid = threadIdx.x;
    for (uint32_t t = blockIdx.x; t < ntasks; t += gridDim.x) {
        const Task& T = tasks[t];
        const DevGraph& g = T.g;
        const Job& job = T.job;
        hist[tid] = 0u;
        __syncthreads();
        auto bucket = [&](uint32_t time) -> uint32_t {       // dir_t: ascending, the first 0
            uint32_t lo = 0, hi = g.dir_n;
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (g.dir_t[mid] <= time) lo = mid; else hi = mid;
            }
            return lo;
        };
        auto key_of = [&](uint64_t q) -> uint32_t {
            const uint64_t i = job.idx_list ? job.idx_list[q] : job.i0 + q;
            uint32_t s, z;
            if (!draw_pair(g.n, job.seed, i, job.dom_pair, &s, &z)) return 1023u;
            if (g.out_ptr[s + 1] == g.out_ptr[s] || g.slot_ptr[z + 1] == g.slot_ptr[z]) return 1023u;
            return bucket(g.tmin_out[s]) * 32u + (31u - bucket(g.tmax_in[z]));
        };
        for (uint64_t q = tid; q < job.count; q += 1024) atomicAdd(hist + key_of(q), 1u);
        __syncthreads();
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<1024>(hist[tid], &tot, sm);
        hist[tid] = ex;
        __syncthreads();
        uint32_t* const o = order + unit_start[t] * 32ull;
        for (uint64_t q = tid; q < job.count; q += 1024) o[atomicAdd(hist + key_of(q), 1u)] = (uint32_t)q;
        __syncthreads();
    }
}

// ---- host side ----

// Region of one CTA: the log holds a record per edge at most (edges of one slot
// may bring the same samples).
size_t sweep_region_bytes(uint32_t n, uint64_t m, SweepWs* ws) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    ws->path_cap = std::min<uint32_t>(n + 2, 2048);
    ws->cone_cap = std::min<uint32_t>(n + 1, 1024);
    size_t o = 0;
    ws->o_log = o;   o = al(o + ((size_t)m + 32) * sizeof(uint4));
    ws->o_arr = o;   o = al(o + (size_t)n * 4);
    ws->o_stp = o;   o = al(o + (size_t)WAVE_STEP * 32 * 4);
    ws->o_path = o;  o = al(o + (size_t)ws->path_cap * 32 * 4);
    ws->o_pathe = o; o = al(o + (size_t)ws->path_cap * 32 * 4);
    ws->o_cv = o;    o = al(o + (size_t)ws->cone_cap * 4);
    ws->o_co = o;    o = al(o + (size_t)ws->cone_cap * 4);
    ws->o_ck = o;    o = al(o + (size_t)ws->cone_cap * 8);
    ws->o_sig = o;   o = al(o + (size_t)n * 8);
    return o;
}

size_t sweep_smem_bytes(uint32_t n) { return ((size_t)n + 1 + 2 * ((size_t)(n + 32) / 32)) * 4; }

cudaError_t sweep_configure(size_t smem) {
    static std::mutex mu;
    static size_t configured[64] = {};
    int dev = 0;
    const cudaError_t ed = cudaGetDevice(&dev);
    if (ed != cudaSuccess) return ed;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= configured[dev]) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(k_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) configured[dev] = smem;
    return e;
}

size_t sweep_static_smem() {
    cudaFuncAttributes a{};
    return cudaFuncGetAttributes(&a, k_sweep) == cudaSuccess ? a.sharedSizeBytes : 1024;
}

cudaError_t sweep_blocks_per_sm(size_t smem, int* out) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_sweep, 32, smem);
}

cudaError_t launch_sweep(const Task* tasks, const uint64_t* unit_start, const uint32_t* ntasks, u64* work,
                         const SweepWs& ws, int grid, cudaStream_t st) {
    if (ws.order) k_sweep_order<<<64, 1024, 0, st>>>(tasks, unit_start, ntasks, ws.order);
    k_sweep<<<grid, 32, sweep_smem_bytes(ws.n_smem), st>>>(tasks, unit_start, ntasks, work, ws);
    return cudaGetLastError();
}

// ---- the waves of a graph ----

// Per stream edge: its head's slot; per slot: its last stream edge.
__global__ void k_wave_slots(DevGraph g, uint32_t* slot, uint32_t* slot_last) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.m) return;
    const uint32_t v = g.st_v[i];
    const uint32_t a = lower_bound_u32(g.slot_t, g.slot_ptr[v], g.slot_ptr[v + 1], g.st_t[i]);
    slot[i] = a;
    atomicMax(slot_last + a, i);
}

// Per stream edge: one past the last earlier stream edge, of another time, into
// its tail or its head (0: none).
__global__ void k_wave_deps(DevGraph g, const uint32_t* slot, const uint32_t* slot_last, uint32_t* dep) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.m) return;
    const uint32_t u = g.st_u[i], v = g.st_v[i], a = slot[i];
    const uint32_t u0 = g.slot_ptr[u], b = lower_bound_u32(g.slot_t, u0, g.slot_ptr[u + 1], g.st_t[i]);
    uint32_t d = 0;
    if (b > u0) d = slot_last[b - 1] + 1u;
    if (a > g.slot_ptr[v]) d = max(d, slot_last[a - 1] + 1u);
    dep[i] = d;
}

// Cuts the stream into waves (wave_cut_part), a thread per part.  A wave is noted
// at its own first edge: marks[i] = 1 (zeroed before), which no other thread
// writes.  *big: a step has more than WAVE_STEP waves.
__global__ void k_wave_cut(DevGraph g, const uint32_t* dep, unsigned char* marks, uint32_t* big) {
    const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (!wave_cut_part(g.st_t, dep, g.m, x, [&](uint32_t i) { marks[i] = 1; })) atomicMax(big, 1u);
}

// The marks of a part: four edges per lane of a warp; the lane's number of marks
// and, in *before, those of the lanes before it.
__device__ __forceinline__ uint32_t wave_marks(const unsigned char* marks, uint32_t x, uint32_t* word, uint32_t* before) {
    static_assert(WAVE_CUT == 128, "a warp takes a part, four edges a lane");
    const uint32_t lane = threadIdx.x & 31;
    *word = reinterpret_cast<const uint32_t*>(marks)[(size_t)x * 32u + lane];
    const uint32_t c = __popc(*word);
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
    }
    *before = incl - c;
    return c;
}

// count[x]: marks of part x.
__global__ void k_wave_count(const unsigned char* marks, uint32_t nb, uint32_t* count) {
    const uint32_t x = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (x >= nb) return;
    uint32_t word, before;
    const uint32_t c = wave_marks(marks, x, &word, &before);
    if ((threadIdx.x & 31) == 31) count[x] = before + c;
}

// first[w]: the first edge of wave w (base: the exclusive sums of count).
__global__ void k_wave_first(const unsigned char* marks, uint32_t nb, const uint32_t* base, uint32_t* first) {
    const uint32_t x = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (x >= nb) return;
    uint32_t word, before;
    wave_marks(marks, x, &word, &before);
    uint32_t* f = first + base[x] + before;
#pragma unroll
    for (uint32_t y = 0; y < 4; ++y)
        if ((word >> (8u * y)) & 1u) *f++ = x * WAVE_CUT + (threadIdx.x & 31) * 4u + y;
}

// Exclusive sums of count (one CTA); *total.
__global__ void __launch_bounds__(1024) k_wave_sum(uint32_t* count, uint32_t nb, uint32_t* total) {
    __shared__ uint32_t sm[32];
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t b = 0; b < nb; b += 1024) {
        const uint32_t x = b + threadIdx.x;
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<1024>(x < nb ? count[x] : 0u, &tot, sm);
        if (x < nb) count[x] = carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

// The waves' edges, 32 places each (padding: u = v = n), up to a multiple of
// WAVE_BATCH waves; a wave ends where the next begins.
__global__ void k_wave_fill(DevGraph g, const uint32_t* slot, const uint32_t* first, uint32_t total, WaveArrays wa) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t w = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (w >= wa.n_waves) return;
    const uint32_t i0 = w < total ? first[w] : g.m, i1 = w + 1 < total ? first[w + 1] : g.m, i = i0 + lane;
    uint2 uv = make_uint2(g.n, g.n), at = make_uint2(0u, 0u);
    uint32_t fl = 0;
    if (i < i1) {
        const uint32_t a = slot[i], tm = g.st_t[i];
        uv = make_uint2(g.st_u[i], g.st_v[i]);
        at = make_uint2(a, tm);
        if (g.slot_in[a + 1] - g.slot_in[a] > 1u) fl = WAVE_SEVERAL;
    }
    wa.uv[(size_t)w * 32u + lane] = uv;
    wa.at[(size_t)w * 32u + lane] = at;
    fl = __reduce_or_sync(0xFFFFFFFFu, fl) | wave_step_flags(g.st_t, g.m, i0, i1);
    if (lane == 0) {
        wa.fl[w] = fl;
        wa.t[w] = g.st_t[(i1 ? i1 : 1u) - 1u];
        if (fl) atomicOr(&wa.info[w / WAVE_BATCH].y, 1u);             // (zeroed before)
        if (w % WAVE_BATCH == WAVE_BATCH - 1) wa.info[w / WAVE_BATCH].x = g.st_t[(i1 ? i1 : 1u) - 1u];
    }
}

// Waves of g, first part: the cut.  tmp (wave_tmp_bytes(m, A)): the number of waves
// and the oversize flag in its first two words | marks | slot | dep, then first |
// last | count.
size_t wave_tmp_bytes(uint32_t m, uint32_t A) {
    const size_t nb = ((size_t)m + WAVE_CUT - 1) / WAVE_CUT;
    return 256 + nb * WAVE_CUT + ((size_t)m * 2 + A + nb + 64) * 4;
}

cudaError_t launch_wave_cut(const DevGraph& g, char* tmp, cudaStream_t st) {
    const uint32_t nb = (g.m + WAVE_CUT - 1) / WAVE_CUT;
    uint32_t* head = reinterpret_cast<uint32_t*>(tmp);
    unsigned char* marks = reinterpret_cast<unsigned char*>(tmp + 256);
    uint32_t* slot = reinterpret_cast<uint32_t*>(tmp + 256 + (size_t)nb * WAVE_CUT);
    uint32_t *dep = slot + g.m, *last = dep + g.m, *count = last + g.A;
    cudaError_t e = cudaMemsetAsync(tmp, 0, 256 + (size_t)nb * WAVE_CUT, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(last, 0, (size_t)g.A * 4, st);
    if (e != cudaSuccess) return e;
    k_wave_slots<<<(g.m + 255) / 256, 256, 0, st>>>(g, slot, last);
    k_wave_deps<<<(g.m + 255) / 256, 256, 0, st>>>(g, slot, last, dep);
    k_wave_cut<<<(nb + 31) / 32, 32, 0, st>>>(g, dep, marks, head + 1);
    k_wave_count<<<(nb + 7) / 8, 256, 0, st>>>(marks, nb, count);
    k_wave_sum<<<1, 1024, 0, st>>>(count, nb, head);
    k_wave_first<<<(nb + 7) / 8, 256, 0, st>>>(marks, nb, count, dep);
    return cudaGetLastError();
}

size_t wave_bytes(uint32_t total) {
    const size_t nw = ((size_t)total + WAVE_BATCH - 1) / WAVE_BATCH * WAVE_BATCH;
    return nw * 32 * 16 + nw * 8 + nw / WAVE_BATCH * 8 + 256;
}

// Second part: the waves' arrays, laid out in mem (wave_bytes(total)), filled.
cudaError_t launch_wave_fill(DevGraph* g, char* tmp, uint32_t total, char* mem, cudaStream_t st) {
    const size_t nb = ((size_t)g->m + WAVE_CUT - 1) / WAVE_CUT;
    const uint32_t* slot = reinterpret_cast<const uint32_t*>(tmp + 256 + nb * WAVE_CUT);
    WaveArrays wa;
    wa.n_waves = (total + WAVE_BATCH - 1) / WAVE_BATCH * WAVE_BATCH;
    wa.uv = reinterpret_cast<uint2*>(mem);
    wa.at = wa.uv + (size_t)wa.n_waves * 32;
    wa.info = wa.at + (size_t)wa.n_waves * 32;
    wa.t = reinterpret_cast<uint32_t*>(wa.info + wa.n_waves / WAVE_BATCH);
    wa.fl = wa.t + wa.n_waves;
    cudaError_t e = cudaMemsetAsync(wa.info, 0, wa.n_waves / WAVE_BATCH * sizeof(uint2), st);
    if (e != cudaSuccess) return e;
    k_wave_fill<<<(wa.n_waves + 7) / 8, 256, 0, st>>>(*g, slot, slot + g->m, total, wa);
    g->n_waves = wa.n_waves;
    g->wave_uv = wa.uv; g->wave_at = wa.at; g->wave_info = wa.info; g->wave_t = wa.t; g->wave_fl = wa.fl;
    return cudaGetLastError();
}

}  // namespace mantra
