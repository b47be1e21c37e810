// bfs_multi.cu -- batched multi-source BFS over 64-bit per-vertex lane masks.
//
// Up to 64 searches advance together.  Lane i of vertex v is bit i of three
// masks: seen[v] (lane i has reached v), front[v] (v is in lane i's current
// frontier), next[v] (v joins lane i's next frontier).  One level of all
// lanes at once, in either direction of "Parallel Direction-Optimizing BFS":
//   top-down  (push, the per-lane Algorithm 1 step): for v with front[v] != 0,
//             for u in adj(v): next[u] |= front[v] & ~seen[u]  (64-bit atomicOr)
//   bottom-up (pull, the per-lane Algorithm 2 step): for u with lanes missing
//             (miss = active & ~seen[u]): OR front[v] over adj(u) in order and
//             stop once every missing lane is covered; next[u] = acc & miss
//   apply:    seen |= next, front = next, next = 0; for each new lane bit i of
//             v: level_i[v] = iteration + 1 - start_i.
// A batch keeps the levels bit-sliced while it runs (64 lanes x 4 bits = one
// 32-byte sector per vertex) and writes the 64 level rows once, at the end, in
// whole lines; a search that finds vertices deeper than four bits hold writes the
// rows it has then and goes on writing them directly.  The same sectors give the minimum-id
// parents: one read of a neighbour's sector compares all 64 lanes at once.
// Direction per iteration from the union frontier with the same rule as the
// single-source search (m_f * alpha > m_u; n_f * beta < n).  Levels do not
// depend on it.
//
// Two drivers share these phases:
//  * bfs_multi_kernel: one persistent cooperative launch for a batch of <= 64
//    roots (bfs_run_multi), bounded grid barriers between phases;
//  * bfs_serve_kernel: one persistent launch per server step that runs levels
//    until a lane finishes (or an iteration cap), so that new lanes can join
//    at a level boundary (continuous batching).
#include <algorithm>
#include <cstring>

#include "bfs_common.cuh"
#include "bfs_internal.h"
#include "bfs_multi.h"

namespace bfsk {

constexpr int kMBlock = 512;
constexpr int kMChunk = 512;      // edges per top-down chunk task
constexpr int kMBigDeg = 256;     // rows above this become chunk tasks (the task lists are sized for it)
constexpr int kPullChunk = 512;   // ids per chunk task of a long row (pulls, parents)
constexpr int kPullSteps = 4;     // 16-id steps a 4-lane group pulls before the rest of the row becomes tasks
constexpr int kPullEnd = 8;       // ... and of a row that is read to its end in so many
constexpr int kPlaneMax = 15;     // largest level + 1 that the four planes hold
// a batch of levels of up to so many roots writes its rows as it goes: the planes are 32
// bytes a vertex whatever the lanes (R-MAT 22: 8 roots 1140 us without, 1196 with planes,
// 40 roots 1785 and 1470; Erdos-Renyi of 4 M vertices, 20 roots: 1372 and 1277)
constexpr int kDirectLanes = 8;
constexpr unsigned kMFull = 0xffffffffu;

__device__ __forceinline__ long long m_gtid() { return (long long)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ long long m_gthreads() { return (long long)gridDim.x * blockDim.x; }

__device__ __forceinline__ unsigned long long ldcg64(const unsigned long long* p) { return __ldcg(p); }

__device__ __forceinline__ unsigned long long warp_or64(unsigned long long x) {
    unsigned lo = __reduce_or_sync(kMFull, (unsigned)x);
    unsigned hi = __reduce_or_sync(kMFull, (unsigned)(x >> 32));
    return ((unsigned long long)hi << 32) | lo;
}

// Lane table cached in shared memory by each CTA.
struct LaneSmem {
    int* rows[64];
    int start[64];
};

__device__ __forceinline__ void load_lanes(const MultiParams& p, LaneSmem& L) {
    for (int i = threadIdx.x; i < 64; i += blockDim.x) {
        L.rows[i] = p.rows[i];
        L.start[i] = p.start[i];
    }
    __syncthreads();
}

// ---------------------------------------------------------------- phases
//
// The union frontier is kept twice: as masks (front[v] != 0) and as a queue of
// its vertices (fq); the vertices that gain lane bits during a level are
// listed once each in the touched queue (tq), which becomes the next fq.  So a
// top-down level and the apply step cost O(frontier + touched), not O(n); only
// bottom-up levels sweep all vertices (they are chosen when the frontier is
// large).  The two queues alternate: qsel picks fq.

// Per-warp staging of queue appends in shared memory, flushed in batches so a
// queue counter sees one atomicAdd per batch rather than one per warp step.
constexpr int kMStage = 256;
struct MStage {
    int* buf;
    int cnt;   // warp-uniform
};

__device__ __forceinline__ MStage m_stage() {
    __shared__ int s_mstage[kMBlock / 32][kMStage];
    MStage st;
    st.buf = s_mstage[threadIdx.x >> 5];
    st.cnt = 0;
    return st;
}

__device__ __forceinline__ void m_flush(MStage& st, int* q, unsigned long long* len) {
    if (st.cnt == 0) return;
    __syncwarp();
    unsigned long long b = 0;
    if (lane_id() == 0) b = atomicAdd(len, (unsigned long long)st.cnt);
    b = __shfl_sync(kMFull, b, 0);
    for (int i = lane_id(); i < st.cnt; i += 32) q[b + i] = st.buf[i];
    __syncwarp();
    st.cnt = 0;
}

// Final flush of a phase, every thread of the CTA calls it: the warps'
// remaining entries go out with one atomicAdd per CTA (block scan of counts).
__device__ void m_block_flush(MStage& st, int* q, unsigned long long* len) {
    __shared__ int s_wcnt[kMBlock / 32];
    __shared__ unsigned long long s_base;
    const int lane = lane_id(), wib = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    if (lane == 0) s_wcnt[wib] = st.cnt;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int c = lane < nwb ? s_wcnt[lane] : 0;
        const int incl = warp_inclusive_scan(c);
        const int total = __shfl_sync(kMFull, incl, 31);
        unsigned long long b = 0;
        if (lane == 0 && total) b = atomicAdd(len, (unsigned long long)total);
        if (lane < nwb) s_wcnt[lane] = incl - c;
        if (lane == 0) s_base = b;
    }
    __syncthreads();
    const unsigned long long b = s_base + (unsigned long long)s_wcnt[wib];
    for (int i = lane; i < st.cnt; i += 32) q[b + i] = st.buf[i];
    __syncwarp();
    st.cnt = 0;
}

// Stage `v` (where `want`) for queue q; all lanes call.
__device__ __forceinline__ void m_append(MStage& st, int* q, unsigned long long* len, bool want, int v) {
    const unsigned m = __ballot_sync(kMFull, want);
    if (m) {
        if (want) st.buf[st.cnt + __popc(m & lanemask_lt())] = v;
        st.cnt += __popc(m);
        if (st.cnt > kMStage - 32) m_flush(st, q, len);
    }
}

// Push the lane bits nb[q] to u[q] (-1: none), four edges per lane: the seen masks
// in flight together, then the atomics; u is recorded the first time its next mask
// becomes nonzero.  All lanes call.
__device__ __forceinline__ void ms_push4(const MultiParams& p, unsigned long long (&nb)[4], const int (&u)[4],
                                         MStage& st, int* tq, unsigned long long* tlen) {
#pragma unroll
    for (int q = 0; q < 4; q++) nb[q] = u[q] >= 0 ? nb[q] & ~ldcg64(p.seen + u[q]) : 0ull;
    unsigned long long old[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        old[q] = 1ull;
        if (nb[q]) old[q] = atomicOr(p.next + u[q], nb[q]);
    }
#pragma unroll
    for (int q = 0; q < 4; q++) m_append(st, tq, tlen, old[q] == 0ull, u[q]);
}

// Top-down push over the frontier queue (warp-balanced gather; heavy rows
// become chunk tasks processed by ms_tasks_phase after a barrier).
__device__ void ms_td_phase(const MultiParams& p, MCtrl* c, int slot, const int* fq, long long flen, int* tq,
                            unsigned long long* tlen) {
    const int lane = lane_id();
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    MStage st = m_stage();
    // a small frontier is spread over every warp (one gather round each)
    const long long per = flen >= nw * 32 ? 32 : max(1LL, (flen + nw - 1) / nw);
    for (long long base = gw * per; base < flen; base += nw * per) {
        const long long i = base + lane;
        int v = 0;
        unsigned long long f = 0;
        long long s = 0, e = 0;
        if (lane < per && i < flen) {
            v = __ldcg(fq + i);
            f = ldcg64(p.front + v);
            if (f) {
                // v leaves the frontier here (its mask travels in registers, or
                // with its chunk tasks); nothing else reads front[v] this phase
                p.front[v] = 0ull;
                s = __ldg(p.off + v);
                e = __ldg(p.off + v + 1);
            }
        }
        const long long deg = e - s;
        const bool big = deg > p.big_deg;
        const int mydeg = big ? 0 : (int)deg;
        unsigned bm = __ballot_sync(kMFull, big);
        while (bm) {
            const int L = __ffs(bm) - 1;
            bm &= bm - 1;
            const long long bs = __shfl_sync(kMFull, s, L), be = __shfl_sync(kMFull, e, L);
            const unsigned long long bf = __shfl_sync(kMFull, f, L);
            const long long nch = (be - bs + kMChunk - 1) / kMChunk;
            unsigned long long t0 = 0;
            if (lane == 0) t0 = atomicAdd(&c->ntask[slot], (unsigned long long)nch);
            t0 = __shfl_sync(kMFull, t0, 0);
            // the row's lane mask is kept at the slot of its first chunk
            if (lane == 0 && (long long)t0 < p.task_cap) p.hubmask[t0] = bf;
            for (long long k = lane; k < nch; k += 32) {
                const long long ti = (long long)t0 + k;
                if (ti < p.task_cap) {
                    MTask t;
                    t.start = bs + k * kMChunk;
                    t.len = (int)min((long long)kMChunk, be - t.start);
                    t.v = (int)t0;
                    p.tasks[ti] = t;
                } else {
                    raise_status(&c->b, kDevOverflow);
                }
            }
        }
        const int incl = warp_inclusive_scan(mydeg);
        const int total = __shfl_sync(kMFull, incl, 31);
        const int excl = incl - mydeg;
        // four edges per lane per step: the ids, the seen masks, the pushes
        for (int k0 = 0; k0 < total; k0 += 128) {
            int u[4];
            unsigned long long nb[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                u[q] = -1;
                nb[q] = 0;
                if (k0 + q * 32 >= total) continue;   // (the same in every lane)
                const int k = k0 + q * 32 + lane;
                int j = 0;
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1) {
                    const int cc = __shfl_sync(kMFull, incl, j + step - 1);
                    if (cc <= k) j += step;
                }
                const long long sj = __shfl_sync(kMFull, s, j);
                const int exj = __shfl_sync(kMFull, excl, j);
                nb[q] = __shfl_sync(kMFull, f, j);
                u[q] = k < total ? __ldg(p.cols + sj + (k - exj)) : -1;
            }
            ms_push4(p, nb, u, st, tq, tlen);
        }
    }
    m_block_flush(st, tq, tlen);
}

__device__ void ms_tasks_phase(const MultiParams& p, MCtrl* c, int slot, int* tq, unsigned long long* tlen) {
    const int lane = lane_id();
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    MStage st = m_stage();
    const long long nt = min((long long)ld_relaxed64(&c->ntask[slot]), p.task_cap);
    for (long long t = gw; t < nt; t += nw) {
        const int4 raw = __ldcg(reinterpret_cast<const int4*>(p.tasks + t));
        const long long start = (long long)(unsigned)raw.x | ((long long)raw.y << 32);
        const int len = raw.z, h = raw.w;
        const unsigned long long f = ldcg64(p.hubmask + h);
        // four edges per lane per step: the ids, then the seen masks in flight together
        for (int k0 = 0; k0 < len; k0 += 128) {
            int u[4];
            unsigned long long nb[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int k = k0 + q * 32 + lane;
                u[q] = k < len ? __ldg(p.cols + start + k) : -1;
            }
#pragma unroll
            for (int q = 0; q < 4; q++) nb[q] = f;
            ms_push4(p, nb, u, st, tq, tlen);
        }
    }
    m_block_flush(st, tq, tlen);
}

// Bottom-up pull: a warp owns 32 consecutive vertices; each lane ORs the
// frontier masks of its first 8 neighbours.  Rows with lanes still missing then
// go on in groups of 4 lanes, 8 rows per warp at a time, 16 neighbours a step
// until every missing lane is covered; a row that is not done after kPullSteps
// steps becomes chunk tasks of kPullChunk ids for all warps (ms_bu_tasks_phase):
// few steps here, as a group's are a chain (with 16 steps the groups of the level
// that reads most of R-MAT 22 took 469 us for 30 M ids, the tasks 276 for 100 M).
// A row that ends within kPullEnd steps is read to its end: its few ids as a task
// cost a warp, an atomic and a place in the list that longer rows need
// (Erdos-Renyi of 200 K vertices, 96 neighbours each, 40 roots: 469 us with such
// tasks, 296 without; R-MAT 22 with 64 roots 2160 and 1978).
// Bound by dependent reads (ids, then masks): one row at a time per warp left
// two thirds of the cycles waiting at the level's barrier for the warps whose
// vertices had long rows (R-MAT 20, 64 roots).
__device__ void ms_bu_phase(const MultiParams& p, MCtrl* c, int slot, unsigned long long active) {
    __shared__ unsigned char s_pend[kMBlock / 32][32];
    __shared__ unsigned long long s_acc[kMBlock / 32][32];
    const int lane = lane_id(), wib = threadIdx.x >> 5, grp = lane >> 2, gl = lane & 3;
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    for (long long base = gw * 32; base < p.n; base += nw * 32) {
        const long long u = base + lane;
        unsigned long long miss = 0, acc = 0;
        long long s = 0, e = 0, pos = 0;
        if (u < p.n) {
            miss = active & ~ldcg64(p.seen + u);
            if (miss) {
                s = __ldg(p.off + u);
                e = __ldg(p.off + u + 1);
                pos = s;   // a degree-0 row has nothing left to scan
            }
        }
        if (miss && e > s) {
            const long long a = s & ~3LL;
            const int4 x0 = __ldg(reinterpret_cast<const int4*>(p.cols_bu + a));
            const int4 x1 = __ldg(reinterpret_cast<const int4*>(p.cols_bu + a + 4));
            const int ids[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
            for (int t = 0; t < 8; t++) {
                const long long q = a + t;
                if (q >= s && q < e) acc |= ldcg64(p.front + ids[t]);
            }
            pos = a + 8;
        }
        const bool more = miss && (acc & miss) != miss && pos < e;
        const unsigned pend = __ballot_sync(kMFull, more);
        const int np = __popc(pend);
        if (more) s_pend[wib][__popc(pend & lanemask_lt())] = (unsigned char)lane;
        __syncwarp();
        for (int r0 = 0; r0 < np; r0 += 8) {
            const bool has = r0 + grp < np;
            const int L = has ? (int)s_pend[wib][r0 + grp] : 0;
            long long q = __shfl_sync(kMFull, pos, L);
            const long long qe = __shfl_sync(kMFull, e, L);
            const unsigned long long mL = __shfl_sync(kMFull, miss, L);
            unsigned long long aL = __shfl_sync(kMFull, acc, L);
            bool live = has;
            const int most = qe - q <= 16 * kPullEnd ? kPullEnd : kPullSteps;
            for (int step = 0; __any_sync(kMFull, live && step < most); step++) {
                unsigned long long x = 0;
                const long long q4 = q + 4 * gl;   // a multiple of 4: the window was aligned
                if (live && step < most && q4 < qe) {
                    const int4 y = __ldg(reinterpret_cast<const int4*>(p.cols_bu + q4));
                    const int ids[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int t = 0; t < 4; t++)
                        if (q4 + t < qe) x |= ldcg64(p.front + ids[t]);
                }
                x |= __shfl_xor_sync(kMFull, x, 1);
                x |= __shfl_xor_sync(kMFull, x, 2);
                if (live && step < most) {
                    aL |= x;
                    q += 16;
                    live = (aL & mL) != mL && q < qe;
                }
            }
            // the rest of a row: chunk tasks
            if (live && gl == 0) {
                const long long nch = (qe - q + kPullChunk - 1) / kPullChunk;
                const unsigned long long t0 = atomicAdd(&c->ntask[slot], (unsigned long long)nch);
                if ((long long)t0 + nch <= p.task_cap) {
                    for (long long k = 0; k < nch; k++) {
                        MTask t;
                        t.start = q + k * kPullChunk;
                        t.len = (int)min((long long)kPullChunk, qe - t.start);
                        t.v = (int)(base + L);
                        p.tasks[t0 + k] = t;
                    }
                    live = false;
                } else {
                    // what was reserved past the room left: tasks with nothing in them
                    MTask t;
                    t.start = 0;
                    t.len = 0;
                    t.v = (int)(base + L);
                    for (long long k = (long long)t0; k < p.task_cap; k++) p.tasks[k] = t;
                }
            }
            // rows that found the list full: the whole warp, 128 ids a step (left to its
            // four lanes, a hub behind many rows of a hundred ids is a chain of a step per 16)
            unsigned rest = __ballot_sync(kMFull, live && gl == 0);
            while (rest) {
                const int own = __ffs(rest) - 1;
                rest &= rest - 1;
                const long long re = __shfl_sync(kMFull, qe, own);
                const unsigned long long want = __shfl_sync(kMFull, mL, own);
                unsigned long long got = __shfl_sync(kMFull, aL, own);
                for (long long r = __shfl_sync(kMFull, q, own); r < re && (got & want) != want; r += 128) {
                    unsigned long long x = 0;
                    const long long r4 = r + 4 * lane;
                    if (r4 < re) {
                        const int4 y = __ldg(reinterpret_cast<const int4*>(p.cols_bu + r4));
                        const int ids[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                        for (int t = 0; t < 4; t++)
                            if (r4 + t < re) x |= ldcg64(p.front + ids[t]);
                    }
                    got |= warp_or64(x);
                }
                if (lane == own) aL = got;
            }
            if (has && gl == 0) s_acc[wib][L] = aL;
        }
        __syncwarp();
        if (more) acc = s_acc[wib][lane];
        const unsigned long long nb = acc & miss;
        if (nb) p.next[u] = nb;
        __syncwarp();
    }
}

// The chunks of long rows: a warp each, four ids per lane per step; a row's
// chunks meet in its next mask.
__device__ void ms_bu_tasks_phase(const MultiParams& p, MCtrl* c, int slot, unsigned long long active) {
    const int lane = lane_id();
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    const long long nt = min((long long)ld_relaxed64(&c->ntask[slot]), p.task_cap);
    for (long long t = gw; t < nt; t += nw) {
        const int4 raw = __ldcg(reinterpret_cast<const int4*>(p.tasks + t));
        const long long start = (long long)(unsigned)raw.x | ((long long)raw.y << 32);
        const int len = raw.z, v = raw.w;
        const unsigned long long miss = active & ~ldcg64(p.seen + v) & ~ldcg64(p.next + v);
        unsigned long long acc = 0;
        for (int k0 = 0; k0 < len && (acc & miss) != miss; k0 += 128) {
            int u[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int k = k0 + q * 32 + lane;
                u[q] = k < len ? __ldg(p.cols_bu + start + k) : -1;
            }
            unsigned long long x = 0;
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (u[q] >= 0) x |= ldcg64(p.front + u[q]);
            acc |= warp_or64(x);
        }
        if (lane == 0 && (acc & miss)) atomicOr(p.next + v, acc & miss);
    }
}

// Levels of the lanes in x at vertex v, found by iteration `iter`: into the
// planes while they hold it (one sector of v), else straight into the rows.
__device__ __forceinline__ void ms_set_planes(const MultiParams& p, long long v, unsigned long long x, int val) {
#pragma unroll
    for (int b = 0; b < 4; b++)
        if ((val >> b) & 1) p.planes[4 * v + b] = ldcg64(p.planes + 4 * v + b) | x;
}

// Apply over the touched vertices (after a top-down level, whose phase already
// removed the old frontier from front): seen |= next, front = next, next = 0,
// per-lane levels; counts the new frontier (n_f, m_f), the degree of vertices
// every active lane has now seen (subtracted from m_u) and which lanes found
// anything.
__device__ void ms_apply_phase(const MultiParams& p, MCtrl* c, int slot, int iter, unsigned long long active,
                               const LaneSmem& L, bool direct, const int* tq, long long tlen) {
    const long long tid = m_gtid(), nth = m_gthreads();
    unsigned long long am = 0, adone = 0, found = 0;
    for (long long i = tid; i < tlen; i += nth) {
        const int v = __ldcg(tq + i);
        const unsigned long long x = ldcg64(p.next + v);
        p.next[v] = 0ull;
        const unsigned long long s = ldcg64(p.seen + v);
        p.seen[v] = s | x;
        p.front[v] = x;
        found |= x;
        const long long deg = __ldg(p.off + v + 1) - __ldg(p.off + v);
        am += (unsigned long long)deg;
        if ((s & active) != active && ((s | x) & active) == active) adone += (unsigned long long)deg;
        if (!direct) ms_set_planes(p, v, x, iter + 2);
        unsigned long long bits = direct ? x : 0ull;
        while (bits) {
            const int i2 = __ffsll((long long)bits) - 1;
            bits &= bits - 1;
            L.rows[i2][v] = iter + 1 - L.start[i2];
        }
    }
    found = warp_or64(found);
    if (lane_id() == 0 && found) atomicOr(&c->found[slot], found);
    block_add4(0, am, adone, 0, nullptr, &c->accm[slot], &c->mdone[slot], nullptr);
    if (tid == 0) c->accn[slot] = (unsigned long long)tlen;
}

// Apply over all vertices: after a bottom-up level (which swept them all anyway),
// and after a top-down level that touched a large share of them: the same updates
// as ms_apply_phase, old frontier bits dropped in the same pass, and the new
// frontier listed in queue nq (null after a top-down level: the touched queue is
// that list).  Four vertices per lane are in flight; read by read, one vertex at a
// time, a nearly empty level took 95 us of latency at R-MAT 22.  A warp's four groups of
// 32 lie a whole grid apart, so that a graph of fewer vertices than the grid has threads
// is spread over all warps (128 in a row to a warp instead, and the empty groups walked
// too: a torus of 120^2, 40 roots, 121 levels, 2761 us; 1829 so).  Vertex by vertex in
// the touched queue's order the masks, planes and offsets (112 bytes a vertex) are
// random DRAM accesses: 918 K vertices of 4.2 M took 358 us.  In order, with few pull
// steps and four pushes in flight, R-MAT 22 with 64 roots went from 1843 to 1576 us
// (2217 to 2026 and 2274 to 2112 on other seeds).
constexpr int kApplyAll = 16;   // touched vertices from n / this many on are applied in order

__device__ void ms_apply_all_phase(const MultiParams& p, MCtrl* c, int slot, int iter, unsigned long long active,
                                   const LaneSmem& L, bool direct, int* nq, unsigned long long* nlen) {
    const int lane = lane_id();
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    MStage st = m_stage();
    unsigned long long an = 0, am = 0, adone = 0, found = 0;
    for (long long base = gw * 32; base < p.n; base += nw * 128) {
        unsigned long long x[4], f[4], s[4];
        long long deg[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const long long v = base + k * nw * 32 + lane;
            x[k] = v < p.n ? ldcg64(p.next + v) : 0ull;
            f[k] = v < p.n ? ldcg64(p.front + v) : 0ull;
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const long long v = base + k * nw * 32 + lane;
            s[k] = 0;
            deg[k] = 0;
            if (x[k]) {
                s[k] = ldcg64(p.seen + v);
                deg[k] = __ldg(p.off + v + 1) - __ldg(p.off + v);
            }
        }
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const long long v = base + k * nw * 32 + lane;
            if (v - lane >= p.n) break;   // (the same in every lane)
            if (x[k]) {
                p.next[v] = 0ull;
                p.seen[v] = s[k] | x[k];
                p.front[v] = x[k];
                found |= x[k];
                if (!direct) ms_set_planes(p, v, x[k], iter + 2);
                an += 1;
                am += (unsigned long long)deg[k];
                if ((s[k] & active) != active && ((s[k] | x[k]) & active) == active) adone += (unsigned long long)deg[k];
            } else if (f[k]) {
                p.front[v] = 0ull;
            }
            // level rows written as it goes: the warp walks the lanes any of its 32
            // vertices gained, one lane at a time, so each store instruction writes
            // consecutive vertices of one row (a lane-by-lane walk per thread would
            // scatter every store)
            unsigned long long ub = direct ? warp_or64(x[k]) : 0ull;
            while (ub) {
                const int i2 = __ffsll((long long)ub) - 1;
                ub &= ub - 1;
                if ((x[k] >> i2) & 1ull) L.rows[i2][v] = iter + 1 - L.start[i2];
            }
            if (nq) m_append(st, nq, nlen, x[k] != 0ull, (int)v);
        }
    }
    if (nq) m_block_flush(st, nq, nlen);
    found = warp_or64(found);
    if (lane == 0 && found) atomicOr(&c->found[slot], found);
    block_add4(an, am, adone, 0, &c->accn[slot], &c->accm[slot], &c->mdone[slot], nullptr);
}

// a[0..cnt) to zero (grid-stride; a is 16-byte aligned).
__device__ void ms_clear_words(unsigned long long* a, long long cnt) {
    const long long tid = m_gtid(), nth = m_gthreads();
    const ulonglong2 z = make_ulonglong2(0ull, 0ull);
    for (long long i = tid; i < cnt / 2; i += nth) reinterpret_cast<ulonglong2*>(a)[i] = z;
    if ((cnt & 1) && tid == 0) a[cnt - 1] = 0ull;
}

// The three masks, and the level planes where the launch keeps them.
__device__ void ms_clear_phase(const MultiParams& p) {
    ms_clear_words(p.seen, p.n);
    ms_clear_words(p.front, p.n);
    ms_clear_words(p.next, p.n);
    if (p.planes) ms_clear_words(p.planes, 4 * p.n);
}

// The level rows from the planes, every active lane's row whole: a warp takes
// 32 consecutive vertices and writes one line of each row in turn.  Bound by the
// rows' bytes (64 rows of R-MAT 22: 1.07 GB); a -1 fill and a scattered store
// per (lane, vertex) moved each line two or three times.  Eight lanes' four bits
// are first woven into one word of nibbles.
__device__ __forceinline__ unsigned ms_spread8(unsigned x) {
    x = (x | (x << 12)) & 0x000F000Fu;
    x = (x | (x << 6)) & 0x03030303u;
    return (x | (x << 3)) & 0x11111111u;
}

__device__ void ms_rows_phase(const MultiParams& p, unsigned long long active) {
    const long long tid = m_gtid(), nth = m_gthreads();
    const int k = __popcll(active);   // lanes 0..k-1
    for (long long v = tid; v < p.n; v += nth) {
        const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2*>(p.planes) + 2 * v);
        const ulonglong2 b = __ldcg(reinterpret_cast<const ulonglong2*>(p.planes) + 2 * v + 1);
        int* row = p.level0 + v;
        for (int i0 = 0; i0 < k; i0 += 8, row += 8 * p.n) {
            const unsigned w = ms_spread8((unsigned)(a.x >> i0) & 0xFFu) | ms_spread8((unsigned)(a.y >> i0) & 0xFFu) << 1 |
                               ms_spread8((unsigned)(b.x >> i0) & 0xFFu) << 2 |
                               ms_spread8((unsigned)(b.y >> i0) & 0xFFu) << 3;
            int* r = row;
#pragma unroll
            for (int i = 0; i < 8; i++, r += p.n)
                if (i0 + i < k) *r = (int)((w >> (4 * i)) & 15u) - 1;
        }
    }
}

// The levels of the frontier that iteration `iter` found (its `len` vertices listed in fq).
__device__ void ms_frontier_rows(const MultiParams& p, int iter, const LaneSmem& L, const int* fq, long long len) {
    const long long tid = m_gtid(), nth = m_gthreads();
    for (long long i = tid; i < len; i += nth) {
        const int v = __ldcg(fq + i);
        unsigned long long bits = ldcg64(p.front + v);
        while (bits) {
            const int i2 = __ffsll((long long)bits) - 1;
            bits &= bits - 1;
            L.rows[i2][v] = iter + 1 - L.start[i2];
        }
    }
}

// Fill the level rows of lanes in `mask` with -1 (rows of n entries).
__device__ void ms_fill_rows(const MultiParams& p, unsigned long long mask, const LaneSmem& L) {
    const long long tid = m_gtid(), nth = m_gthreads();
    unsigned long long bits = mask;
    while (bits) {
        const int i = __ffsll((long long)bits) - 1;
        bits &= bits - 1;
        int* row = L.rows[i];
        for (long long v = tid; v < p.n; v += nth) row[v] = -1;
    }
}

// Seed lanes in `mask` at their roots (atomics: several lanes may share a
// root); a root not yet in the frontier joins the frontier queue.  Run by the
// first warp (64 lanes at most -> two rounds).
__device__ void ms_seed_phase(const MultiParams& p, unsigned long long mask, const LaneSmem& L, bool direct, int* fq,
                              unsigned long long* flen) {
    if (m_gtid() >= 32) return;
    MStage st = m_stage();
    for (int i0 = 0; i0 < 64; i0 += 32) {
        const int i = i0 + lane_id();
        bool add = false;
        int r = 0;
        if ((mask >> i) & 1ull) {
            r = p.roots[i];
            atomicOr(p.seen + r, 1ull << i);
            add = atomicOr(p.front + r, 1ull << i) == 0ull;
            if (direct) L.rows[i][r] = 0;
            else atomicOr(p.planes + 4 * (long long)r, 1ull << i);
        }
        m_append(st, fq, flen, add, r);
    }
    m_flush(st, fq, flen);
}

__device__ __forceinline__ int ms_decide(const MultiParams& p, int prev, long long nf, long long mf, long long mu) {
    if (p.mode == BFS_MODE_TD_ONLY) return 0;
    if (p.mode == BFS_MODE_BU_ONLY) return 1;
    if (prev == 0) return (mf * (long long)p.alpha > mu) ? 1 : 0;
    return (nf * (long long)p.beta < p.n) ? 0 : 1;
}

// The barrier after a bottom-up phase, and its number of chunk tasks: read once per CTA
// (by every thread the counter's one line serves 16 times the requests), and not at
// all where no row is long enough for a task.
__device__ __forceinline__ bool bu_sync(const MultiParams& p, MCtrl* c, int slot, unsigned long long& ntask) {
    if (p.long_rows) return grid_sync_read(&c->b, p.expected, p.timeout_ns, &c->ntask[slot], &ntask, 1);
    if (threadIdx.x == 0) ntask = 0;
    return grid_sync(&c->b, p.expected, p.timeout_ns);
}

// ---------------------------------------------------------------- persistent driver

__global__ void __launch_bounds__(kMBlock, 2) bfs_multi_kernel(MultiParams p) {
    __shared__ LaneSmem L;
    load_lanes(p, L);
    __shared__ unsigned long long ntask;   // a bottom-up level's chunk tasks
    MCtrl* c = p.ctrl;
    const unsigned long long active = p.active;
    bool direct = p.planes == nullptr;
    ms_clear_phase(p);
    if (direct) ms_fill_rows(p, active, L);
    if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
    ms_seed_phase(p, active, L, direct, p.q0, &c->qlen[0]);
    if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
    // level-0 statistics from the (few) distinct roots, identical in every CTA
    long long mf = 0, mu = p.nnz;
    for (int i = 0; i < 64; i++) {
        if (!((active >> i) & 1ull)) continue;
        const int r = p.roots[i];
        bool dup = false;
        for (int j = 0; j < i; j++)
            if (((active >> j) & 1ull) && p.roots[j] == r) dup = true;
        if (dup) continue;
        const long long deg = __ldg(p.off + r + 1) - __ldg(p.off + r);
        mf += deg;
        if ((ldcg64(p.seen + r) & active) == active) mu -= deg;
    }
    int prev = 0, qsel = 0;
    for (int it = 0;; it++) {
        // counters of iteration `it` accumulate in slot it % 3 and are read by
        // every CTA after the closing barrier; the slot of iteration it + 1 is
        // cleared now (its last readers passed a barrier of iteration it - 1)
        const int slot = it % 3, sfree = (it + 1) % 3;
        if (blockIdx.x == 0 && threadIdx.x == 0) c->zero_slot(sfree);
        int* fq = qsel ? p.q1 : p.q0;
        int* tq = qsel ? p.q0 : p.q1;
        const long long flen = (long long)ld_relaxed64(&c->qlen[qsel]);
        unsigned long long* tlen = &c->qlen[qsel ^ 1];
        const int dir = ms_decide(p, prev, flen, mf, mu);
        if (dir == 0) {
            ms_td_phase(p, c, slot, fq, flen, tq, tlen);
            if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            if (ld_relaxed64(&c->ntask[slot]) > 0) {
                ms_tasks_phase(p, c, slot, tq, tlen);
                if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            }
            const long long touched = (long long)ld_relaxed64(tlen);
            if (touched * kApplyAll >= p.n)
                ms_apply_all_phase(p, c, slot, it, active, L, direct, nullptr, nullptr);
            else
                ms_apply_phase(p, c, slot, it, active, L, direct, tq, touched);
        } else {
            ms_bu_phase(p, c, slot, active);
            if (!bu_sync(p, c, slot, ntask)) return;
            if (ntask > 0) {
                ms_bu_tasks_phase(p, c, slot, active);
                if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            }
            ms_apply_all_phase(p, c, slot, it, active, L, direct, tq, tlen);
        }
        if (m_gtid() == 0) c->qlen[qsel] = 0;   // the old frontier's queue collects the next touched set
        if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
        const long long nt = (long long)ld_relaxed64(&c->accn[slot]);
        qsel ^= 1;
        if (nt == 0) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                c->iterations = it + 1;
                c->direct = direct ? 1u : 0u;
            }
            break;
        }
        mu -= (long long)ld_relaxed64(&c->mdone[slot]);
        mf = (long long)ld_relaxed64(&c->accm[slot]);
        prev = dir;
        if (!direct && it + 2 > kPlaneMax) {
            // vertices past the planes, which hold nothing of them: the rows as the planes
            // have them, then these vertices' levels
            ms_rows_phase(p, active);
            direct = true;
            if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            ms_frontier_rows(p, it, L, qsel ? p.q1 : p.q0, nt);
            if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
        }
    }
    if (!direct) ms_rows_phase(p, active);
}

// Minimum-id parents of a batch: parent_i[v] = min{u in adj(v) : level_i[u] =
// level_i[v] - 1} (rows sorted: the first such u), a root's its own, -1 where not
// reached.  From the planes: with t the bit-sliced (level + 1) - 1 of v's lanes,
// one sector read of a neighbour u says in a few word operations for which of the 64
// lanes u is a parent, so a row is read once for all lanes and left as soon as
// every lane has its parent (lane by lane over the level rows, one thread per
// vertex, R-MAT 18 with 40 roots took 47 ms).  A lane takes a vertex, a warp 32
// consecutive ones; their parents gather in shared memory so that every output
// row gets whole lines.  Lanes at level 1 need no search: their only parent is
// the root.  Rows above kMBigDeg become chunk tasks for ms_parent_tasks_kernel:
// a hub's parent in a lane with a small frontier may be anywhere in its row.
constexpr int kPBlock = 256;
constexpr int kPTileRow = 33;   // 32 vertices, padded against bank conflicts
constexpr size_t kParentSmem = sizeof(int) * 64 * kPTileRow * (kPBlock / 32);

struct LanePlanes {
    unsigned long long p0, p1, p2, p3;
};
__device__ __forceinline__ LanePlanes ms_planes(const MultiParams& p, long long v) {
    const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(p.planes) + 2 * v);
    const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(p.planes) + 2 * v + 1);
    return {a.x, a.y, b.x, b.y};
}
// bit-sliced decrement (lanes holding 0 wrap; callers mask them)
__device__ __forceinline__ LanePlanes ms_minus1(const LanePlanes& a) {
    const unsigned long long b1 = ~a.p0, b2 = b1 & ~a.p1, b3 = b2 & ~a.p2;
    return {~a.p0, a.p1 ^ b1, a.p2 ^ b2, a.p3 ^ b3};
}
__device__ __forceinline__ unsigned long long ms_equal(const LanePlanes& a, const LanePlanes& b) {
    return ~((a.p0 ^ b.p0) | (a.p1 ^ b.p1) | (a.p2 ^ b.p2) | (a.p3 ^ b.p3));
}
// lanes at level >= 2: the ones whose parent has to be looked for
__device__ __forceinline__ unsigned long long ms_searching(const LanePlanes& a) { return a.p2 | a.p3 | (a.p0 & a.p1); }

__global__ void __launch_bounds__(kPBlock) ms_parent_planes_kernel(MultiParams p, int* parent0) {
    extern __shared__ int s_tile[];
    __shared__ int s_root[64];
    MCtrl* c = p.ctrl;
    if (c->direct || c->b.status != kDevOk) return;
    if (threadIdx.x < 64) s_root[threadIdx.x] = p.roots[threadIdx.x];
    __syncthreads();
    const int lane = lane_id(), k = __popcll(p.active);
    int* tile = s_tile + (threadIdx.x >> 5) * 64 * kPTileRow;
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    for (long long base = gw * 32; base < p.n; base += nw * 32) {
        const long long v = base + lane;
        LanePlanes a = {0, 0, 0, 0};
        if (v < p.n) a = ms_planes(p, v);
        const unsigned long long reached = a.p0 | a.p1 | a.p2 | a.p3;
        const unsigned long long root = a.p0 & ~(a.p1 | a.p2 | a.p3), one = a.p1 & ~(a.p0 | a.p2 | a.p3);
        for (int i = 0; i < k; i++)
            tile[i * kPTileRow + lane] = (root >> i) & 1ull ? (int)v : (one >> i) & 1ull ? s_root[i] : -1;
        unsigned long long need = reached & ms_searching(a);
        if (need) {
            const LanePlanes t = ms_minus1(a);
            const long long s = __ldg(p.off + v), e = __ldg(p.off + v + 1);
            if (e - s > kMBigDeg) {
                const long long nch = (e - s + kPullChunk - 1) / kPullChunk;
                const unsigned long long t0 = atomicAdd(&c->nptask, (unsigned long long)nch);
                for (long long j = 0; j < nch && (long long)t0 + j < p.task_cap; j++) {
                    MTask m;
                    m.start = s + j * kPullChunk;
                    m.len = (int)min((long long)kPullChunk, e - m.start);
                    m.v = (int)v;
                    p.tasks[t0 + j] = m;
                }
                need = 0;
            }
            for (long long q = s; need && q < e; q += 4) {
                int u[4];
                LanePlanes b[4];
#pragma unroll
                for (int j = 0; j < 4; j++) u[j] = __ldg(p.cols + min(q + j, e - 1));
#pragma unroll
                for (int j = 0; j < 4; j++) b[j] = ms_planes(p, u[j]);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    unsigned long long hit = ms_equal(b[j], t) & need;
                    need &= ~hit;
                    while (hit) {
                        const int i = __ffsll((long long)hit) - 1;
                        hit &= hit - 1;
                        tile[i * kPTileRow + lane] = u[j];
                    }
                }
            }
        }
        __syncwarp();
        if (v < p.n) {
            int* o = parent0 + v;
            for (int i = 0; i < k; i++, o += p.n) *o = tile[i * kPTileRow + lane];
        }
        __syncwarp();
    }
}

// The long rows' chunks: a warp reads 32 ids and their sectors per step; the
// lowest warp lane that offers search lane i a parent is the chunk's smallest,
// and the chunks meet by atomicMin (unsigned: -1 is the largest).
__global__ void __launch_bounds__(kPBlock) ms_parent_tasks_kernel(MultiParams p, int* parent0) {
    const MCtrl* c = p.ctrl;
    if (c->direct || c->b.status != kDevOk) return;
    const int lane = lane_id();
    const long long gw = m_gtid() >> 5, nw = m_gthreads() >> 5;
    const long long nt = min((long long)c->nptask, p.task_cap);
    for (long long ti = gw; ti < nt; ti += nw) {
        const MTask m = p.tasks[ti];
        const LanePlanes a = ms_planes(p, m.v), t = ms_minus1(a);
        unsigned long long need = (a.p0 | a.p1 | a.p2 | a.p3) & ms_searching(a);
        for (int k0 = 0; k0 < m.len && need; k0 += 32) {
            const int kk = k0 + lane;
            int u = -1;
            unsigned long long hit = 0;
            if (kk < m.len) {
                u = __ldg(p.cols + m.start + kk);
                hit = ms_equal(ms_planes(p, u), t) & need;
            }
            const unsigned long long any = warp_or64(hit);
            if (!any) continue;
            need &= ~any;
            // drop the search lanes that a lower warp lane (a smaller id) offers too
            unsigned long long pre = hit;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(kMFull, pre, o);
                if (lane >= o) pre |= y;
            }
            pre = __shfl_up_sync(kMFull, pre, 1);
            if (lane > 0) hit &= ~pre;
            while (hit) {
                const int i = __ffsll((long long)hit) - 1;
                hit &= hit - 1;
                atomicMin(reinterpret_cast<unsigned*>(parent0 + (long long)i * p.n + m.v), (unsigned)u);
            }
        }
    }
}

// The same over the level rows, for a search that outgrew its planes.
__global__ void ms_parent_kernel(MultiParams p, int* const* prow) {
    __shared__ LaneSmem L;
    if (!p.ctrl->direct) return;
    load_lanes(p, L);
    const long long tid = m_gtid(), nth = m_gthreads();
    for (int i = 0; i < 64; i++) {
        if (!((p.active >> i) & 1ull)) continue;
        const int* lv = L.rows[i];
        int* pr = prow[i];
        for (long long v = tid; v < p.n; v += nth) {
            const int l = lv[v];
            int par = -1;
            if (l == 0) {
                par = (int)v;
            } else if (l > 0) {
                const long long s = __ldg(p.off + v), e = __ldg(p.off + v + 1);
                for (long long k = s; k < e; k++) {
                    const int u = __ldg(p.cols + k);
                    if (lv[u] == l - 1) {
                        par = u;
                        break;
                    }
                }
            }
            pr[v] = par;
        }
    }
}

// Clear the three masks of a slot (used when a server slot is created).
__global__ void __launch_bounds__(kMBlock) ms_clear_kernel(MultiParams p) { ms_clear_phase(p); }

// ---------------------------------------------------------------- server driver

// One launch of a server slot: optional admission of new lanes (drop the
// stale bits of `drop` lanes, fill new rows with -1, seed new roots), then
// levels iter0, iter0+1, ... for all `active` lanes until a lane's frontier
// comes back empty (its result is final), the union frontier is empty, or
// max_iters levels ran.  The direction per level follows the union frontier
// (top-down -> bottom-up when m_f * alpha > nnz / 2, back when n_f * beta < n;
// the per-lane unvisited degree m_u is not tracked when lanes start at
// different levels).  Results for the host: s_done, s_finished, s_nf, s_mf,
// s_dir in the control block (which persists across launches of the slot).
__global__ void __launch_bounds__(kMBlock, 2) bfs_serve_kernel(MultiParams p, int iter0, int max_iters,
                                                                unsigned long long newmask,
                                                                unsigned long long drop) {
    __shared__ LaneSmem L;
    load_lanes(p, L);
    __shared__ unsigned long long ntask;   // a bottom-up level's chunk tasks
    MCtrl* c = p.ctrl;
    const unsigned long long active = p.active;
    const long long tid = m_gtid(), nth = m_gthreads();
    int qsel = c->s_qsel;
    if (drop) {
        // lanes being reused: remove their previous query's bits
        const unsigned long long keep = ~drop;
        for (long long v = tid; v < p.n; v += nth) {
            const unsigned long long s = p.seen[v];
            if (s & drop) p.seen[v] = s & keep;
            const unsigned long long f = p.front[v];
            if (f & drop) p.front[v] = f & keep;
        }
    }
    if (newmask | drop) {
        ms_fill_rows(p, newmask, L);
        if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
        ms_seed_phase(p, newmask, L, true, qsel ? p.q1 : p.q0, &c->qlen[qsel]);
        if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
    }
    long long mf = c->s_mf;
    int prev = c->s_dir;
    int it = iter0, done = 0;
    long long nt = 0;
    unsigned long long finished = 0;
    for (; done < max_iters; it++) {
        const int slot = it % 3, sfree = (it + 1) % 3;
        if (blockIdx.x == 0 && threadIdx.x == 0) c->zero_slot(sfree);
        int* fq = qsel ? p.q1 : p.q0;
        int* tq = qsel ? p.q0 : p.q1;
        const long long flen = (long long)ld_relaxed64(&c->qlen[qsel]);
        unsigned long long* tlen = &c->qlen[qsel ^ 1];
        int dir;
        if (p.mode == BFS_MODE_TD_ONLY) dir = 0;
        else if (p.mode == BFS_MODE_BU_ONLY) dir = 1;
        else if (prev == 0) dir = (mf * (long long)p.alpha > p.nnz / 2) ? 1 : 0;
        else dir = (flen * (long long)p.beta < p.n) ? 0 : 1;
        if (dir == 0) {
            ms_td_phase(p, c, slot, fq, flen, tq, tlen);
            if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            if (ld_relaxed64(&c->ntask[slot]) > 0) {
                ms_tasks_phase(p, c, slot, tq, tlen);
                if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            }
            const long long touched = (long long)ld_relaxed64(tlen);
            if (touched * kApplyAll >= p.n)
                ms_apply_all_phase(p, c, slot, it, active, L, true, nullptr, nullptr);
            else
                ms_apply_phase(p, c, slot, it, active, L, true, tq, touched);
        } else {
            ms_bu_phase(p, c, slot, active);
            if (!bu_sync(p, c, slot, ntask)) return;
            if (ntask > 0) {
                ms_bu_tasks_phase(p, c, slot, active);
                if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
            }
            ms_apply_all_phase(p, c, slot, it, active, L, true, tq, tlen);
        }
        if (tid == 0) c->qlen[qsel] = 0;
        if (!grid_sync(&c->b, p.expected, p.timeout_ns)) return;
        nt = (long long)ld_relaxed64(&c->accn[slot]);
        qsel ^= 1;
        done++;
        prev = dir;
        mf = (long long)ld_relaxed64(&c->accm[slot]);
        finished = active & ~ld_relaxed64(&c->found[slot]);
        if (finished || nt == 0) break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->s_done = done;
        c->s_finished = finished;
        c->s_nf = nt;
        c->s_mf = mf;
        c->s_dir = prev;
        c->s_qsel = qsel;
    }
}

}  // namespace bfsk

// ====================================================================== host

namespace bfsrt {

using bfsk::MCtrl;
using bfsk::MTask;
using bfsk::MultiParams;

static size_t mask_bytes(const bfs_graph* g) { return sizeof(unsigned long long) * (size_t)g->n; }

bfs_status multi_alloc(bfs_graph* g, MultiWork& w, cudaStream_t s) {
    if (w.ready) return BFS_OK;
    const size_t nb = mask_bytes(g);
    // chunks of rows above kMBigDeg: at most nnz / chunk whole ones and one rest per row
    const long long task_cap = g->nnz / bfsk::kMChunk + g->nnz / bfsk::kMBigDeg + 1024;
    w.seen = (unsigned long long*)mem_of(g, w).alloc(nb, s);
    w.front = (unsigned long long*)mem_of(g, w).alloc(nb, s);
    w.next = (unsigned long long*)mem_of(g, w).alloc(nb, s);
    w.ctrl = mem_of(g, w).alloc(sizeof(MCtrl), s);
    w.tasks = mem_of(g, w).alloc(sizeof(MTask) * (size_t)task_cap, s);
    w.hubmask = mem_of(g, w).alloc(sizeof(unsigned long long) * (size_t)task_cap, s);
    w.lanes = mem_of(g, w).alloc(sizeof(bfsk::LaneTable), s);
    w.q0 = (int*)mem_of(g, w).alloc(sizeof(int) * (size_t)(g->n + 64), s);
    w.q1 = (int*)mem_of(g, w).alloc(sizeof(int) * (size_t)(g->n + 64), s);
    w.task_cap = task_cap;
    if (!w.seen || !w.front || !w.next || !w.ctrl || !w.tasks || !w.hubmask || !w.lanes || !w.q0 || !w.q1) {
        w.ready = true;
        multi_free(g, w);
        return fail(BFS_ERR_OOM, "multi-source work buffers: device allocation failed");
    }
    w.bytes = 3 * nb + sizeof(MCtrl) + (sizeof(MTask) + 8) * (size_t)task_cap + sizeof(bfsk::LaneTable) +
              2 * sizeof(int) * (size_t)(g->n + 64);
    int occ = 0;
    BFS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, bfsk::bfs_multi_kernel, bfsk::kMBlock, 0));
    if (occ < 1) return fail(BFS_ERR_UNSUPPORTED, "multi-source kernel cannot be resident");
    w.block = bfsk::kMBlock;
    w.grid = occ * g->sm_count;
    BFS_CUDA_TRY(cudaFuncSetAttribute(bfsk::ms_parent_planes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)bfsk::kParentSmem));
    BFS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, bfsk::ms_parent_planes_kernel, bfsk::kPBlock,
                                                               bfsk::kParentSmem));
    w.pgrid = std::max(1, occ) * g->sm_count;
    BFS_CUDA_TRY(cudaMemsetAsync(w.ctrl, 0, sizeof(MCtrl), s));
    BFS_CUDA_TRY(cudaMemsetAsync(w.lanes, 0, sizeof(bfsk::LaneTable), s));
    w.ready = true;
    return BFS_OK;
}

void multi_free(bfs_graph* g, MultiWork& w) {
    if (!w.ready) return;
    const size_t nb = mask_bytes(g);
    mem_of(g, w).release(w.seen, nb, nullptr);
    mem_of(g, w).release(w.front, nb, nullptr);
    mem_of(g, w).release(w.next, nb, nullptr);
    mem_of(g, w).release(w.planes, 4 * nb, nullptr);
    mem_of(g, w).release(w.ctrl, sizeof(MCtrl), nullptr);
    mem_of(g, w).release(w.tasks, sizeof(MTask) * (size_t)w.task_cap, nullptr);
    mem_of(g, w).release(w.hubmask, sizeof(unsigned long long) * (size_t)w.task_cap, nullptr);
    mem_of(g, w).release(w.lanes, sizeof(bfsk::LaneTable), nullptr);
    mem_of(g, w).release(w.q0, sizeof(int) * (size_t)(g->n + 64), nullptr);
    mem_of(g, w).release(w.q1, sizeof(int) * (size_t)(g->n + 64), nullptr);
    DeviceAlloc* keep = w.mem;   // the allocator choice outlives the buffers
    w = MultiWork();
    w.mem = keep;
}

bfs_status multi_prepare(bfs_graph* g, cudaStream_t s) {
    MultiWork& w = g->multi;
    if (w.ready) return BFS_OK;
    bfs_status st = multi_alloc(g, w, s);
    if (st != BFS_OK) return st;
    // 32 bytes per vertex of level planes; without room for them the rows are written directly
    w.planes = (unsigned long long*)mem_of(g, w).alloc(4 * mask_bytes(g), s);
    if (w.planes) w.bytes += 4 * mask_bytes(g);
    return BFS_OK;
}
void multi_release(bfs_graph* g) { multi_free(g, g->multi); }

static MultiParams multi_params(bfs_graph* g, MultiWork& w, const bfs_options& opt) {
    MultiParams p;
    memset(&p, 0, sizeof p);
    p.off = reinterpret_cast<const long long*>(g->offsets);
    p.cols = g->cols;
    p.cols_bu = (opt.bu_rows == BFS_BU_ROWS_HUB_FIRST && g->cols_hf) ? g->cols_hf : g->cols;
    p.n = g->n;
    p.nnz = g->nnz;
    p.seen = w.seen;
    p.front = w.front;
    p.next = w.next;
    p.ctrl = reinterpret_cast<MCtrl*>(w.ctrl);
    p.q0 = w.q0;
    p.q1 = w.q1;
    p.tasks = reinterpret_cast<MTask*>(w.tasks);
    p.hubmask = reinterpret_cast<unsigned long long*>(w.hubmask);
    p.task_cap = w.task_cap;
    bfsk::LaneTable* lt = reinterpret_cast<bfsk::LaneTable*>(w.lanes);
    p.rows = lt->rows;
    p.start = lt->start;
    p.roots = lt->roots;
    p.mode = opt.mode == BFS_MODE_RANDOM ? BFS_MODE_DO : opt.mode;
    p.alpha = opt.alpha;
    p.beta = opt.beta;
    p.planes = w.planes;
    p.big_deg = std::max(opt.td_big_degree, bfsk::kMBigDeg);
    // a pull reads at least five ids of a row in its first window, then 16 a step
    p.long_rows = g->max_degree > 5 + 16 * bfsk::kPullEnd;
    p.timeout_ns = (unsigned long long)(opt.timeout_ms > 0 ? opt.timeout_ms : 10000) * 1000000ull;
    p.expected = (unsigned)w.grid + (unsigned)(g->debug_barrier_extra > 0 ? g->debug_barrier_extra : 0);
    return p;
}

bfs_status multi_launch(bfs_graph* g, const int32_t* roots_host, int32_t k, int32_t* level, int32_t* parent,
                        const bfs_options& opt, cudaStream_t s) {
    MultiWork& w = g->multi;
    for (int32_t c0 = 0; c0 < k; c0 += 64) {
        const int kk = std::min(64, k - c0);
        bfsk::LaneTable t;
        memset(&t, 0, sizeof t);
        for (int i = 0; i < kk; i++) {
            t.rows[i] = level + (size_t)(c0 + i) * (size_t)g->n;
            t.prow[i] = parent ? parent + (size_t)(c0 + i) * (size_t)g->n : nullptr;
            t.start[i] = 0;
            t.roots[i] = roots_host[c0 + i];
        }
        // pageable source: staged by the driver before cudaMemcpyAsync returns,
        // and ordered on the stream before the launch that reads it
        BFS_CUDA_TRY(cudaMemcpyAsync(w.lanes, &t, sizeof t, cudaMemcpyHostToDevice, s));
        BFS_CUDA_TRY(cudaMemsetAsync(w.ctrl, 0, sizeof(MCtrl), s));
        MultiParams p = multi_params(g, w, opt);
        p.active = (kk == 64) ? ~0ull : ((1ull << kk) - 1ull);
        p.level0 = t.rows[0];
        if (!parent && kk <= bfsk::kDirectLanes) p.planes = nullptr;
        void* args[] = {&p};
        BFS_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)bfsk::bfs_multi_kernel, dim3(w.grid), dim3(w.block),
                                                 args, 0, s));
        if (parent) {
            if (p.planes) {
                bfsk::ms_parent_planes_kernel<<<w.pgrid, bfsk::kPBlock, bfsk::kParentSmem, s>>>(p, t.prow[0]);
                BFS_CUDA_TRY(cudaGetLastError());
                bfsk::ms_parent_tasks_kernel<<<w.pgrid, bfsk::kPBlock, 0, s>>>(p, t.prow[0]);
                BFS_CUDA_TRY(cudaGetLastError());
            }
            bfsk::LaneTable* lt = reinterpret_cast<bfsk::LaneTable*>(w.lanes);
            bfsk::ms_parent_kernel<<<w.grid, w.block, 0, s>>>(p, lt->prow);
            BFS_CUDA_TRY(cudaGetLastError());
        }
    }
    return BFS_OK;
}

bfs_status multi_collect_status(bfs_graph* g, cudaStream_t s) {
    MCtrl c;
    BFS_CUDA_TRY(cudaMemcpyAsync(&c, g->multi.ctrl, sizeof(MCtrl), cudaMemcpyDeviceToHost, s));
    BFS_CUDA_TRY(cudaStreamSynchronize(s));
    if (c.b.status == bfsk::kDevTimeout) return fail(BFS_ERR_TIMEOUT, "multi-source grid barrier ran out of time");
    if (c.b.status == bfsk::kDevOverflow) return fail(BFS_ERR_CUDA, "multi-source task list overflowed");
    return BFS_OK;
}

// ---------------------------------------------------------------- server driver (host side)

size_t ms_lane_table_bytes() { return sizeof(bfsk::LaneTable); }

void ms_lane_table_set(void* table_host, int lane, int32_t* row, int start, int root) {
    bfsk::LaneTable* t = reinterpret_cast<bfsk::LaneTable*>(table_host);
    t->rows[lane] = row;
    t->prow[lane] = nullptr;
    t->start[lane] = start;
    t->roots[lane] = root;
}

int ms_serve_max_grid(bfs_graph* g, MultiWork& w) { (void)g; return w.grid; }

bfs_status ms_serve_reset(bfs_graph* g, MultiWork& w, cudaStream_t s) {
    bfs_options o;
    bfs_options_default(&o);
    if (g->cols_hf) o.bu_rows = BFS_BU_ROWS_HUB_FIRST;
    MultiParams p = multi_params(g, w, o);
    bfsk::ms_clear_kernel<<<w.grid, w.block, 0, s>>>(p);
    BFS_CUDA_TRY(cudaGetLastError());
    BFS_CUDA_TRY(cudaMemsetAsync(w.ctrl, 0, sizeof(MCtrl), s));
    return BFS_OK;
}

bfs_status ms_serve_launch(bfs_graph* g, MultiWork& w, const void* lane_table_host, unsigned long long newmask,
                           unsigned long long drop, unsigned long long active, int iter0, int max_iters, int grid,
                           void* ctrl_pinned, cudaStream_t s) {
    bfs_options o;
    bfs_options_default(&o);
    if (g->cols_hf) o.bu_rows = BFS_BU_ROWS_HUB_FIRST;   // levels do not depend on the row order
    MultiParams p = multi_params(g, w, o);
    p.active = active;
    grid = std::max(1, std::min(grid, w.grid));
    p.expected = (unsigned)grid;
    if (newmask)
        BFS_CUDA_TRY(cudaMemcpyAsync(w.lanes, lane_table_host, sizeof(bfsk::LaneTable), cudaMemcpyHostToDevice, s));
    // the barrier state (first member of the control block) restarts at zero for
    // every launch, as the grid size varies between launches; the rest of the
    // control block carries over
    static_assert(offsetof(MCtrl, b) == 0, "barrier state leads the control block");
    BFS_CUDA_TRY(cudaMemsetAsync(w.ctrl, 0, sizeof(bfsk::BarrierState), s));
    void* args[] = {&p, &iter0, &max_iters, &newmask, &drop};
    BFS_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)bfsk::bfs_serve_kernel, dim3(grid), dim3(w.block), args, 0, s));
    BFS_CUDA_TRY(cudaMemcpyAsync(ctrl_pinned, w.ctrl, sizeof(MCtrl), cudaMemcpyDeviceToHost, s));
    return BFS_OK;
}

}  // namespace bfsrt
