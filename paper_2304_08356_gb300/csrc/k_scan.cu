// Prefix-foremost (pfm) samples, a CTA each, by one pass over the part of the
// time-sorted edges in which the sample runs (paper Sec. 3 Def. 1(3), the stream
// scan of Sec. 4.4), the backward path draw (App. C) and the Update step of
// Algorithm 1.  The label-correcting search (k_pfm_cta) tests every out-edge
// against the head's arrival at a random place of a per-sample array, twice as
// many edges as the scan window has on large graphs; here an edge costs two
// bits of shared memory.
//
// The stream comes in chunks of whole time steps.  Vertices reached in earlier
// chunks are final, one bit each.  Within a chunk an edge whose head is final is
// dead, one whose tail is final brings an arrival at once, and the others wait:
// the chunk's arrivals (head, earliest time so far) are in a small hash table,
// and the waiting edges are tested against it until no arrival changes (a few
// passes; times strictly increase along a path).  Then every edge that brings
// the arrival's time is a prefix-foremost in-edge and counts; the arrival slots
// go to an array for the way back from z.  A path that meets a vertex with
// several prefix-foremost in-edges is counted and drawn over the vertices that
// lead to z (warp 0, draw_choice; a sample with more than 2,048 of them goes to
// k_pfm_cta).
//
// What bounds it: the block barriers of a chunk (four and one per pass over the
// waiting edges) and, between them, the instructions of its edges (on 304 samples of
// a graph of 200,000 vertices 0.48 issued per scheduler and cycle, 3.3 of 16
// cycles per instruction at barriers, DRAM at 4 % of its peak); the edges stream
// from L2 and the final bits are in shared memory, so a sample's time grows with the
// length of its window and not with the spread of its search.  Measured against
// k_pfm_cta, ms: n = 10^6, m = 2*10^7 uniform times, 1,000 samples 55.2 for 264 (32
// samples 15.2 for 47.2); n = 200,000, 1,000 samples 10.5 for 38.6; n = 1,000
// bursty, 2,000 samples 0.293 for 0.379.  1,536 edges per stored chunk leave room
// in a CTA's 2,048 (or two chunks in its 4,096) for the whole steps at the ends.
#include "mantra_dev.cuh"

#include <algorithm>
#include <mutex>

namespace mantra {

namespace {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr int EPT = 4;                 // edges of a chunk per thread
constexpr uint32_t CNW = 256;          // words of the chunk's head filter

// Shared memory of a CTA; the final bits (n_smem of them) follow.
template <int NT>
struct __align__(16) ScanSh {
    Task task;
    uint64_t i;
    u64 sigma;
    u64 esc;
    int t, cur_t;
    uint32_t s, z, ok, len, ovf, err, cnt, first;
    uint32_t rade[4];
    uint32_t cn[CNW];
    uint32_t key[2 * EPT * NT], val[2 * EPT * NT];    // heads of the chunk's arrivals, their earliest times
};

}  // namespace

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_scan(const Task* tasks, const uint64_t* unit_start,
                                                        const uint32_t* ntasks_p, u64* work,
                                                        const __grid_constant__ ScanWs ws) {
    constexpr uint32_t TM = 2 * EPT * NT - 1;          // table mask
    constexpr uint32_t CPC = NT / 512;                 // store chunks per chunk
    extern __shared__ __align__(16) unsigned char scan_dyn[];
    ScanSh<NT>& S = *reinterpret_cast<ScanSh<NT>*>(scan_dyn);
    uint32_t* const FB = reinterpret_cast<uint32_t*>(scan_dyn + sizeof(ScanSh<NT>));
    const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    char* const region = ws.base + (size_t)blockIdx.x * ws.stride;
    uint32_t* const arr = reinterpret_cast<uint32_t*>(region + ws.o_arr);     // arrival slots of final vertices
    uint32_t* const path = reinterpret_cast<uint32_t*>(region + ws.o_path);   // from z
    uint32_t* const pathe = reinterpret_cast<uint32_t*>(region + ws.o_pathe);
    uint32_t* const cv = reinterpret_cast<uint32_t*>(region + ws.o_cv);       // vertices that lead to z
    uint32_t* const co = reinterpret_cast<uint32_t*>(region + ws.o_co);       // the same by arrival time
    u64* const ck = reinterpret_cast<u64*>(region + ws.o_ck);
    u64* const sig = reinterpret_cast<u64*>(region + ws.o_sig);
    uint32_t* const MK = reinterpret_cast<uint32_t*>(region + ws.o_mk);       // marks (0 between uses)
    for (uint32_t x = tid; x <= TM; x += NT) { S.key[x] = NONE; S.val[x] = NONE; }
    for (uint32_t x = tid; x < CNW; x += NT) S.cn[x] = 0u;
    if (tid == 0) S.cur_t = -1;
    const uint32_t ntasks = *ntasks_p;
    const uint64_t total = ntasks ? unit_start[ntasks] : 0ull;
    auto draw = [&](uint64_t q) {
        const Job& job = S.task.job;
        const uint64_t i = job.idx_list ? job.idx_list[q] : job.i0 + q;
        uint32_t s = 0, z = 1;
        const bool ok = draw_pair(S.task.g.n, job.seed, i, job.dom_pair, &s, &z);
        if (!ok) { set_status(job.status, ST_RNG); s = 0; z = 1; }
        S.i = i; S.s = s; S.z = z; S.ok = ok ? 1u : 0u;
    };
    u64 my_eadd = 0, my_scan = 0;
    u64* flush_ctr = nullptr;
    auto flush = [&]() {
        if (!flush_ctr) return;
        if (my_scan) atomicAdd(flush_ctr + C_ESCAN, my_scan);
        if (my_eadd) atomicAdd(flush_ctr + C_EADD, my_eadd);
        my_scan = my_eadd = 0;
    };
    uint64_t unit = 0;
    if (tid == 0) unit = atomicAdd(work, 1ull);
    __syncthreads();

    for (;;) {
        uint64_t q = 0;
        if (tid == 0) {
            int t = -1;
            if (unit < total) {
                t = task_of_unit(unit_start, ntasks, unit);
                q = unit - unit_start[t];
                unit = atomicAdd(work, 1ull);
            }
            S.t = t;
            if (t >= 0 && t == S.cur_t) draw(q);
            S.len = S.ovf = S.err = 0; S.sigma = 0;
        }
        __syncthreads();
        if (S.t < 0) break;
        if (S.t != S.cur_t) {
            if (wid == 0) {
                const u64* src = reinterpret_cast<const u64*>(tasks + S.t);
                u64* dst = reinterpret_cast<u64*>(&S.task);
                for (uint32_t w = lane; w < sizeof(Task) / 8; w += 32) dst[w] = src[w];
                __syncwarp();
                if (lane == 0) draw(q);
            }
            __syncthreads();
            if (tid == 0) S.cur_t = S.t;
        }
        const DevGraph& g = S.task.g;
        const Job& job = S.task.job;
        if (job.ctr != flush_ctr) { flush(); flush_ctr = job.ctr; }
        const uint32_t n = g.n, s = S.s, z = S.z;
        const uint64_t i = S.i;
        const bool live = S.ok && g.out_ptr[s + 1] > g.out_ptr[s] && g.slot_ptr[z + 1] > g.slot_ptr[z];
        const uint32_t ts = live ? g.tmin_out[s] : NONE, tz = live ? g.tmax_in[z] : 0u;
        for (uint32_t x = tid; x < (n + 31u) / 32u; x += NT) FB[x] = 0u;
        if (wid == 0 && live && ts <= tz) {
            const uint32_t a = warp_lower_bound(g.st_t, 0, g.m, ts);
            if (lane == 0) S.first = a;
        }
        __syncthreads();
        if (tid == 0) FB[s >> 5] |= 1u << (s & 31u);
        __syncthreads();
        uint32_t te = tz;
        bool reached = false;
        if (live && ts <= tz) {
            const uint32_t* const cp = g.scan_ptr;
            const uint32_t nc = g.n_scan;
            uint32_t c = S.first / SCAN_CHUNK;               // the chunk that holds edge S.first
            while (cp[c + 1] <= S.first) ++c;                // (a long step leaves empty chunks)
            uint32_t p0 = cp[c], p1 = cp[min(c + CPC, nc)];
            uint32_t eu[EPT], ev[EPT], et[EPT], fu[EPT], fv[EPT], ft[EPT];
            auto load = [&](uint32_t (&u)[EPT], uint32_t (&v)[EPT], uint32_t (&t)[EPT], uint32_t b0, uint32_t b1) {
#pragma unroll
                for (int j = 0; j < EPT; ++j) {
                    const uint32_t p = b0 + tid + (uint32_t)j * NT;
                    u[j] = v[j] = 0u; t[j] = NONE;
                    if (p < b1) { u[j] = __ldg(g.st_u + p); v[j] = __ldg(g.st_v + p); t[j] = __ldg(g.st_t + p); }
                }
            };
            // the table's place of v, entered with time t; *lower: its time was later (or none)
            auto enter = [&](uint32_t v, uint32_t t, bool* lower) -> uint32_t {
                uint32_t h = (v * 0x9E3779B1u) >> 7 & TM;
                for (;;) {
                    uint32_t k = S.key[h];
                    if (k == NONE) k = atomicCAS(&S.key[h], NONE, v);
                    if (k == NONE || k == v) break;
                    h = (h + 1u) & TM;
                }
                const uint32_t old = atomicMin(&S.val[h], t);
                if (old == NONE) atomicOr(&S.cn[(v >> 5) & (CNW - 1u)], 1u << (v & 31u));
                *lower = t < old;
                return h;
            };
            auto time_of = [&](uint32_t v) -> uint32_t {     // arrival of v in this chunk so far, or NONE
                if (!((S.cn[(v >> 5) & (CNW - 1u)] >> (v & 31u)) & 1u)) return NONE;
                uint32_t h = (v * 0x9E3779B1u) >> 7 & TM;
                for (;;) {
                    const uint32_t k = S.key[h];
                    if (k == v) return S.val[h];
                    if (k == NONE) return NONE;
                    h = (h + 1u) & TM;
                }
            };
            load(eu, ev, et, p0, p1);
            for (;;) {
                // the next chunk's edges load while this one is worked on
                const uint32_t c2 = min(c + CPC, nc), q0 = p1, q1 = cp[min(c2 + CPC, nc)];
                const uint32_t tl = p1 > p0 ? __ldg(g.st_t + p1 - 1u) : 0u;
                load(fu, fv, ft, q0, q1);
                uint32_t valid = 0, wait = 0, h[EPT];
#pragma unroll
                for (int j = 0; j < EPT; ++j) {
                    h[j] = 0u;
                    if (et[j] > tz) continue;                // (no edge: NONE)
                    if ((FB[ev[j] >> 5] >> (ev[j] & 31u)) & 1u) continue;
                    if ((FB[eu[j] >> 5] >> (eu[j] & 31u)) & 1u) {
                        bool lower;
                        h[j] = enter(ev[j], et[j], &lower);
                        valid |= 1u << j;
                    } else {
                        wait |= 1u << j;
                    }
                }
                if (__syncthreads_or(valid)) {
                    for (;;) {
                        bool changed = false;
#pragma unroll
                        for (int j = 0; j < EPT; ++j)
                            if (((wait >> j) & 1u) && time_of(eu[j]) < et[j]) {
                                bool lower;
                                h[j] = enter(ev[j], et[j], &lower);
                                valid |= 1u << j;
                                wait &= ~(1u << j);
                                changed |= lower;
                            }
                        if (!__syncthreads_or(changed)) break;
                    }
                    const uint32_t zt = time_of(z);
                    if (zt != NONE) { reached = true; te = zt; }
#pragma unroll
                    for (int j = 0; j < EPT; ++j)
                        if (((valid >> j) & 1u) && S.val[h[j]] == et[j]) {
                            if (et[j] <= te) ++my_eadd;
                            arr[ev[j]] = __ldg(g.st_slot + p0 + tid + (uint32_t)j * NT);
                            atomicOr(FB + (ev[j] >> 5), 1u << (ev[j] & 31u));
                        }
                    __syncthreads();
#pragma unroll
                    for (int j = 0; j < EPT; ++j)
                        if ((valid >> j) & 1u) { S.key[h[j]] = NONE; S.val[h[j]] = NONE; }
                    for (uint32_t x = tid; x < CNW; x += NT) S.cn[x] = 0u;
                    __syncthreads();
                }
                if (reached || tl >= tz || c2 >= nc) break;
                c = c2; p0 = q0; p1 = q1;
#pragma unroll
                for (int j = 0; j < EPT; ++j) { eu[j] = fu[j]; ev[j] = fv[j]; et[j] = ft[j]; }
            }
        }
        // fa(w) < tv
        auto before = [&](uint32_t w, uint32_t tv) -> bool {
            if (w == s) return true;
            return ((FB[w >> 5] >> (w & 31u)) & 1u) && g.slot_t[arr[w]] < tv;
        };
        if (wid == 0) {
            if (live && ts <= te) {
                // edges of the scan window: tmin_out(s) <= t <= te, not into s
                const uint32_t a = S.first, b = warp_lower_bound(g.st_t, a, g.m, te + 1u);
                const uint32_t s0 = g.slot_ptr[s], s1 = g.slot_ptr[s + 1];
                const uint32_t sa = warp_lower_bound(g.slot_t, s0, s1, ts), sb = warp_lower_bound(g.slot_t, sa, s1, te + 1u);
                if (lane == 0) S.esc = (u64)(b - a) - (u64)(g.slot_in[sb] - g.slot_in[sa]);
            } else if (lane == 0) {
                S.esc = 0;
            }
            __syncwarp();
            if (reached) {
                // the way back: path[k], edge into it pathe[k]
                uint32_t v = z, plen = 0;
                bool choice = false, perr = false;
                uint32_t away = 0;                           // CHOICE_OVF or CHOICE_CAPPED
                u64 tot = 1;                                 // the only path: nothing to draw
                while (v != s) {
                    const uint32_t a = arr[v], e0 = g.slot_in[a], e1 = g.slot_in[a + 1];
                    uint32_t e = e0;
                    if (e1 - e0 > 1u) {
                        const uint32_t tv = g.slot_t[a];
                        uint32_t found = 0;
                        for (uint32_t x0 = e0; x0 < e1 && found < 2u; x0 += 32) {
                            const uint32_t x = x0 + lane;
                            const unsigned msk = __ballot_sync(FULL, x < e1 && before(g.in_u[min(x, e1 - 1u)], tv));
                            if (msk) e = x0 + __ffs(msk) - 1;
                            found += __popc(msk);
                        }
                        if (found > 1u) { choice = true; break; }
                        if (found == 0u) { perr = true; break; }
                    }
                    if (plen > n) { perr = true; break; }
                    if (lane == 0) { path[plen] = v; pathe[plen] = e; }
                    ++plen;
                    v = g.in_u[e];
                }
                if (!choice && !perr) {
                    if (lane == 0) path[plen] = s;
                    ++plen;
                }
                __syncwarp();
                if (choice) {
                    const int got = draw_choice(g, job, i, s, z, arr, before,
                                                ChoiceWs{cv, co, ck, sig, MK, ws.cone_cap, n + 2u}, &S.cnt, path, pathe,
                                                &plen, &tot);
                    perr = got == CHOICE_ERR;
                    away = got == CHOICE_OVF || got == CHOICE_CAPPED ? (uint32_t)got : 0u;
                }
                if (lane == 0) {
                    if (perr) { S.err = 1; set_status(job.status, ST_CHECK); }
                    else if (away) S.ovf = away;
                    else {
                        S.len = plen;
                        S.sigma = tot;
                        uint32_t w4[4];
                        philox_block(job.seed, i, DOM_RADE, 0, w4);
                        S.rade[0] = w4[0]; S.rade[1] = w4[1]; S.rade[2] = w4[2]; S.rade[3] = w4[3];
                    }
                }
            }
        }
        __syncthreads();
        if (S.ovf) {
            // another kernel takes (and counts) the sample
            if (tid == 0) {
                if (S.ovf == CHOICE_CAPPED) push_capped(job, i); else push_overflow(job, i);
            }
            for (uint32_t v = tid; v < n; v += NT) {
                if (v == s || !((FB[v >> 5] >> (v & 31u)) & 1u)) continue;
                const uint32_t a = arr[v], tv = g.slot_t[a];
                if (tv > te) continue;
                for (uint32_t e = g.slot_in[a]; e < g.slot_in[a + 1]; ++e)
                    if (before(g.in_u[e], tv)) my_eadd -= 1;
            }
        } else {
            if (tid == 0) my_scan += S.esc;
            if (!S.err) {
                const uint32_t len = S.len, nint = family_count(job, len);
                if (job.hits && nint > 0) {
                    const uint32_t rows = 1 + (job.S ? job.c : 0);
                    for (uint32_t it = tid; it < nint * rows; it += NT) {
                        const uint32_t p = it % nint, jr = it / nint;
                        const uint32_t x = job.target == 0 ? path[len - 2 - p]
                                           : (job.target == 2 ? pathe[len - 2 - p] : g.in_uedge[pathe[len - 2 - p]]);
                        if (jr == 0) {
                            atomicAdd(job.hits + x, 1ull);
                        } else {
                            const uint32_t jj = jr - 1;
                            const int lam = ((S.rade[jj >> 5] >> (jj & 31)) & 1u) ? 1 : -1;
                            atomicAdd(job.S + (size_t)jj * job.fam + x, lam);
                        }
                    }
                    if (tid == 0) atomicAdd(job.ctr + C_SUMINT, (u64)nint);
                }
                if (job.rec_len) {
                    const uint64_t r = i - job.i0;
                    if (tid == 0) {
                        job.rec_s[r] = s; job.rec_z[r] = z;
                        job.rec_sig[2 * r] = S.sigma; job.rec_sig[2 * r + 1] = 0ull;
                        job.rec_len[r] = len;
                    }
                    for (uint32_t p = tid; p < len && p < job.rec_cap; p += NT)
                        job.rec_nodes[r * job.rec_cap + p] = path[len - 1 - p];
                    if (job.rec_edges)
                        for (uint32_t p = tid; p + 1 < len && p < job.rec_cap; p += NT)
                            job.rec_edges[r * job.rec_cap + p] = pathe[len - 2 - p];
                }
            }
        }
        __syncthreads();
    }
    flush();
}

// ---- host side ----

size_t scan_region_bytes(uint32_t n, ScanWs* ws) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    ws->cone_cap = std::min<uint32_t>(n + 1, 2048);
    size_t o = 0;
    ws->o_arr = o;   o = al(o + (size_t)n * 4);
    ws->o_path = o;  o = al(o + (size_t)(n + 2) * 4);
    ws->o_pathe = o; o = al(o + (size_t)(n + 2) * 4);
    ws->o_cv = o;    o = al(o + (size_t)ws->cone_cap * 4);
    ws->o_co = o;    o = al(o + (size_t)ws->cone_cap * 4);
    ws->o_ck = o;    o = al(o + (size_t)ws->cone_cap * 8);
    ws->o_sig = o;   o = al(o + (size_t)n * 8);
    ws->o_mk = o;    o = al(o + (size_t)((n + 31) / 32) * 4);
    return o;
}

size_t scan_smem_bytes(int nt, uint32_t n) {
    return (nt == 1024 ? sizeof(ScanSh<1024>) : sizeof(ScanSh<512>)) + (size_t)((n + 31) / 32) * 4;
}

cudaError_t scan_configure(size_t smem) {
    static std::mutex mu;
    static size_t configured[64] = {};
    int dev = 0;
    const cudaError_t ed = cudaGetDevice(&dev);
    if (ed != cudaSuccess) return ed;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (smem <= configured[dev]) return cudaSuccess;
    for (const void* k : {(const void*)k_scan<512>, (const void*)k_scan<1024>}) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    configured[dev] = smem;
    return cudaSuccess;
}

cudaError_t scan_blocks_per_sm(int nt, size_t smem, int* out) {
    if (nt == 1024) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_scan<1024>, 1024, smem);
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_scan<512>, 512, smem);
}

cudaError_t launch_scan(const Task* tasks, const uint64_t* unit_start, const uint32_t* ntasks, u64* work,
                        const ScanWs& ws, int grid, cudaStream_t st) {
    const size_t smem = scan_smem_bytes(ws.nt, ws.n_smem);
    if (ws.nt == 1024) k_scan<1024><<<grid, 1024, smem, st>>>(tasks, unit_start, ntasks, work, ws);
    else k_scan<512><<<grid, 512, smem, st>>>(tasks, unit_start, ntasks, work, ws);
    return cudaGetLastError();
}

// Per stream edge its head's slot; the chunks' first edges (the start of the
// time step that edge k SCAN_CHUNK is in); *big: a step does not fit a chunk.
__global__ void k_scan_maps(DevGraph g, uint32_t nc, uint32_t* st_slot, uint32_t* ptr, uint32_t* big) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < g.m) {
        const uint32_t v = g.st_v[i];
        st_slot[i] = lower_bound_u32(g.slot_t, g.slot_ptr[v], g.slot_ptr[v + 1], g.st_t[i]);
    }
    if (i <= nc) {
        auto cut = [&](uint64_t k) -> uint32_t {
            const uint64_t x = k * SCAN_CHUNK;
            return x >= g.m ? g.m : lower_bound_u32(g.st_t, 0, (uint32_t)x + 1u, g.st_t[x]);
        };
        const uint32_t p = cut(i);
        ptr[i] = p;
        if (i < nc && cut((uint64_t)i + 1) - p > 2048u) atomicMax(big, 1u);
    }
}

cudaError_t launch_scan_maps(const DevGraph& g, uint32_t* st_slot, uint32_t* ptr, uint32_t* big, cudaStream_t st) {
    const uint32_t nc = (g.m + SCAN_CHUNK - 1) / SCAN_CHUNK;
    const cudaError_t e = cudaMemsetAsync(big, 0, 4, st);
    if (e != cudaSuccess) return e;
    k_scan_maps<<<(g.m + 256) / 256, 256, 0, st>>>(g, nc, st_slot, ptr, big);
    return cudaGetLastError();
}

}  // namespace mantra
