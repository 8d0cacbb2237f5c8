// PeelOne's light levels on one thread-block cluster.
//
// Most levels of a skewed graph are light: a few dozen vertices leave, with
// some ten thousand arcs, long after most vertices are gone. On the whole grid
// such a level costs a residual scan, a grid barrier (2.9 us) and the detection
// that its asynchronous walk has ended, 17 to 40 us in all. A cluster of
// kTailCtas CTAs has a hardware barrier of 0.3 us and needs about 2 us for each
// generation of the level's frontier. So the grid kernel (peel::run_async) hands
// light levels over to it and takes heavy ones back: the launches alternate on
// the stream, each starting from the state (TailState) that the previous one
// left, and those with nothing to do return at once.
//
// Residual degrees stay in global memory, where the grid kernel needs them: L2
// serves a cluster of 16 SMs 0.83 returning atomics per clock and SM, distributed
// shared memory 0.32; one warp's chain of them takes 720 and 247 clocks each (measured,
// words that L2 holds).
//
// A level:
//   scan   Each CTA keeps its own part of the residual list (in global memory)
//          and of the near list (in shared memory): the residual vertices below
//          `hi`. A level below hi scans the near list only; when k reaches hi,
//          the residual list is filtered and a new window [k, hi) is listed.
//          A vertex that falls into the window later is listed by the one
//          decrement that takes it from hi to hi - 1. A near list that
//          overflows forces a scan of the residual list at the next level.
//   waves  The vertices that a CTA finds (in the scan, or by a decrement from
//          k + 1 to k) are queued in its shared memory; after a cluster barrier
//          that also exchanges the counts, all CTAs walk all queues together.
//          Every CTA lays the rows of a wave end to end (one thread per row, a
//          CTA-wide prefix sum of the degrees) and the cluster's warps take
//          segments of 128 arcs of that range in turn, whatever the degrees are.
//          Letting each CTA walk what it found itself needs no barrier per
//          wave, but a few rows of thousands of arcs then hold up the level
//          (measured: 43 us a level on Chung-Lu graphs). When a wave has more
//          rows than a CTA has threads, each CTA takes every kTailCtas-th row
//          for itself instead of all.
//          Vertices that do not fit a queue are listed in global memory and
//          walked with the next wave.
//   bail   A wave of more arcs than the launch's budget goes back to the grid
//          kernel, which finishes the level, unless this is the run's last launch
//          (no budget). A wave of at most kTailThreads vertices is laid out by every CTA, which
//          sees its arcs; those of a wider one are counted first (wave_arcs).
// The run ends when every vertex is queued: the rest of the last level's walk
// could only lower vertices that have their coreness.
#pragma once

#include "peel_local.cuh"
#include "peelone.cuh"

namespace pico {
namespace peel {

constexpr int kTailCtas = 16;
constexpr int kTailThreads = 512;
constexpr int kTailQueue = 4096;         // queue entries of a CTA and wave
constexpr int kTailNear = 8192;          // near-list entries of a CTA
constexpr int kTailWindow = 32;          // first width of the near window

// A row of d arcs in the sums that a wave is laid out by, which are 32 bits wide
// (graphs have up to 2^36 arcs). A wave of more than `budget` arcs goes back: a row of
// more is counted as budget + 1, and no sum over a tile's 512 rows wraps. Without a
// budget rows count whole, in graphs of at most kTailMaxGraph arcs.
__host__ __device__ inline int tail_row(long long d, unsigned budget)
{
    return d <= (long long)budget ? (int)d : (int)budget + 1;
}
static_assert(512ull * (kTailLateBudget + 1) < (1ull << 31) && kTailMaxGraph < kTailNoBudget,
              "a tile's sum wraps");

struct TailShared {
    long long off[kTailThreads];         // a wave's rows: row start minus position ...
    int start[kTailThreads + 32];        // ... and position in the wave's arc range
    int queue[2][kTailQueue];
    int near[2][kTailNear];
    uint4 x[2][kTailCtas][2];            // exchange: eight words per CTA, by parity
    unsigned qn[2];                      // vertices queued, by wave parity
    unsigned near_n[2];
    unsigned kept, overflow;
    int vmin;
    int wsum[kTailThreads / 32];
};

// What every CTA knows after an exchange.
struct TailTotals {
    unsigned before;    // lane r: vertices in the queues of the CTAs before r
    unsigned fitted;    // vertices in all queues
    unsigned queued;    // ... and those that did not fit, listed in fs
    unsigned kept, near_max;
    int vmin;
    bool overflow;
};

// Arcs per lane and step. The waves of a light level run through this code
// once per warp, so fetching the instructions is part of their latency: R-MAT
// scale 16 takes 1.39 ms with 1, 1.49 ms with 2 and 1.77 ms with 4, but R-MAT
// scale 22, whose waves hold more arcs, 12.6, 10.7 and 10.5 ms (all levels below
// 1 M arcs handed over).
constexpr int kTailU = 2;

template <typename Off>
struct TailPeel {
    static constexpr int U = kTailU;
    const Params<Off> &p;
    TailState *ts;
    TailShared &sh;
    unsigned rank;
    unsigned budget;   // arcs of a wave that this launch walks, at most
    int k = 0, hi = 0;
    unsigned par = 0, nb = 0, qb = 0;   // exchange parity, near buffer, queue buffer pushed to
    unsigned listed = 0;                // fs entries of the waves so far
    unsigned long long n_lowered = 0;   // decrements of vertices above the level

    // Positions for the lanes' marked elements of a list in shared memory: one
    // counter update per warp. Returns false when no lane has one.
    template <int N>
    __device__ __forceinline__ static bool reserve(const bool (&in)[N], unsigned *counter, unsigned (&pos)[N])
    {
        bool any = false;
#pragma unroll
        for (int j = 0; j < N; ++j) any |= in[j];
        if (!__any_sync(kFull, any)) return false;
        const unsigned lane = threadIdx.x & 31;
        unsigned total = 0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const unsigned b = __ballot_sync(kFull, in[j]);
            pos[j] = total + __popc(b & ((1u << lane) - 1u));
            total += __popc(b);
        }
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(counter, total);
        base = __shfl_sync(kFull, base, 0);
#pragma unroll
        for (int j = 0; j < N; ++j) pos[j] += base;
        return true;
    }

    template <int N>
    __device__ __forceinline__ void add_near(const bool (&in)[N], const int (&v)[N])
    {
        unsigned pos[N];
        if (!reserve(in, &sh.near_n[nb], pos)) return;
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (in[j]) {
                if (pos[j] < (unsigned)kTailNear) sh.near[nb][pos[j]] = v[j];
                else sh.overflow = 1;
            }
    }

    // Queues vertices at level k. Their coreness is written at the start of the
    // wave that walks them (settle): stores still in flight would hold up the
    // cluster barrier (985 clocks instead of 450). What does not fit is listed in global memory.
    template <int N>
    __device__ __forceinline__ void push(const bool (&in)[N], const int (&v)[N])
    {
        unsigned pos[N];
        if (!reserve(in, &sh.qn[qb], pos)) return;
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (in[j]) {
                if (pos[j] < (unsigned)kTailQueue) {
                    sh.queue[qb][pos[j]] = v[j];
                } else {
                    p.core[v[j]] = k;
                    const unsigned s = atomicAdd(&ts->spilled, 1u);
                    if (s < (unsigned)p.n) p.fs[s] = v[j];   // each vertex once in a run
                    else set_error(p.ctl, kErrNotConverged);
                }
            }
    }

    // Writes the coreness of the own vertices of a wave.
    __device__ __forceinline__ void settle(unsigned b, unsigned own)
    {
        for (unsigned i = threadIdx.x; i < own; i += blockDim.x) p.core[sh.queue[b][i]] = k;
    }

    // A step's arcs: all decrements are issued before the first result is used.
    __device__ __forceinline__ void arcs(const bool (&valid)[U], const int (&u)[U])
    {
        int old[U];
#pragma unroll
        for (int j = 0; j < U; ++j) old[j] = valid[j] ? atomicSub(p.work + u[j], 1) : INT_MIN;
        bool in[U], cross[U], any = false;
#pragma unroll
        for (int j = 0; j < U; ++j) {
            in[j] = old[j] == k + 1;
            cross[j] = old[j] == hi && !in[j];
            any |= in[j] || cross[j];
            n_lowered += old[j] > k;
        }
        if (!__any_sync(kFull, any)) return;
        push(in, u);
        add_near(cross, u);
    }

    // Cluster barrier after which every CTA knows every CTA's queue length, and
    // the sums and minima of the rest. What the next phase counts from zero is
    // cleared here, after it was sent and before the CTA arrives: a warp that has
    // left the barrier may count at once (a small wave has no CTA barrier of its
    // own). That is the count of the other queue buffer (the wave just walked it), the
    // scan's counters and, after a scan, the near buffer it read.
    __device__ __forceinline__ TailTotals exchange(bool of_scan)
    {
        __syncthreads();
        const unsigned lane = threadIdx.x & 31;
        if (threadIdx.x < (unsigned)kTailCtas) {
            const uint4 a = make_uint4(sh.qn[qb], (unsigned)sh.vmin, sh.overflow, sh.kept);
            const unsigned near = min(sh.near_n[nb], (unsigned)kTailNear);
            unsigned addr;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(addr)
                         : "r"(shared_addr(&sh.x[par][rank][0])), "r"(threadIdx.x));
            asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a.x),
                         "r"(a.y), "r"(a.z), "r"(a.w)
                         : "memory");
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr + 16), "r"(near) : "memory");
        }
        __syncwarp();
        if (threadIdx.x == 0) {
            sh.qn[qb ^ 1u] = 0;
            sh.kept = sh.overflow = 0;
            sh.vmin = INT_MAX;
            if (of_scan) sh.near_n[nb ^ 1u] = 0;
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        uint4 a = make_uint4(0, (unsigned)INT_MAX, 0, 0);
        if (lane < (unsigned)kTailCtas) a = sh.x[par][lane][0];
        TailTotals t;
        const unsigned fit = min(a.x, (unsigned)kTailQueue);   // lanes past the last CTA hold 0
        unsigned incl = fit;
#pragma unroll
        for (int o = 1; o < kTailCtas; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, incl, o);
            if ((int)lane >= o) incl += y;
        }
        t.before = incl - fit;
        t.fitted = t.queued = __shfl_sync(kFull, incl, kTailCtas - 1);
        if (__any_sync(kFull, fit != a.x)) t.queued = __reduce_add_sync(kFull, a.x);
        t.overflow = __any_sync(kFull, a.z);
        t.vmin = INT_MAX;
        t.kept = t.near_max = 0;
        if (of_scan) {
            t.vmin = __reduce_min_sync(kFull, (int)a.y);
            t.kept = __reduce_add_sync(kFull, a.w);
            t.near_max = __reduce_max_sync(
                kFull, lane < (unsigned)kTailCtas ? sh.x[par][lane][1].x : 0u);
        }
        par ^= 1u;
        return t;
    }

    // The i-th vertex of a wave: of all queues (buffer b), then of fs; -1 when not
    // `valid`. All lanes call.
    __device__ __forceinline__ int queued_vertex(unsigned b, const TailTotals &t, unsigned i, bool valid)
    {
        unsigned r = 0;
#pragma unroll
        for (unsigned s = kTailCtas / 2; s > 0; s >>= 1) {
            const unsigned x = __shfl_sync(kFull, t.before, r + s);
            if (x <= i) r += s;   // the last CTA that starts at or before i: not empty
        }
        const unsigned at = i - __shfl_sync(kFull, t.before, r);
        int v = -1;
        if (valid && i >= t.fitted) {
            v = ldcg(p.fs + listed + (i - t.fitted));
        } else if (valid) {
            unsigned addr;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(addr)
                         : "r"(shared_addr(&sh.queue[b][at])), "r"(r));
            asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
        }
        return v;
    }

    // Walks a wave of at most 32 vertices: every warp holds all rows in its
    // registers, one per lane, so no CTA barrier is needed before its segments.
    // Returns false as wave() does.
    __device__ __forceinline__ bool wave_small(unsigned b, const TailTotals &t)
    {
        const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const int v = queued_vertex(b, t, lane, lane < t.queued);
        Off rs = 0;
        int d = 0;
        if (v >= 0) {
            rs = p.rp[v];
            d = tail_row((long long)(p.rp[v + 1] - rs), budget);
        }
        int incl = d;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if ((int)lane >= o) incl += y;
        }
        const int total = __shfl_sync(kFull, incl, 31), excl = incl - d;
        if ((unsigned)total > budget) return false;
        const Off off = rs - (Off)excl;
        for (int a0 = (int)(warp * kTailCtas + rank) * 32 * U; a0 < total;
             a0 += (int)nw * kTailCtas * 32 * U) {
            // rows that start at or before a0, then one bit per row start
            int row = __popc(__ballot_sync(kFull, d > 0 && excl <= a0)) - 1;
            bool valid[U];
            int u[U];
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int w = a0 + 32 * j, e = w + (int)lane;
                const unsigned rel = (unsigned)(excl - w);
                const unsigned starts =
                    __reduce_or_sync(kFull, d > 0 && excl > a0 && rel < 32u ? 1u << rel : 0u);
                const int own = row + __popc(starts & (0xffffffffu >> (31 - lane)));
                row += __popc(starts);
                valid[j] = e < total;
                const Off o = __shfl_sync(kFull, off, own);
                u[j] = valid[j] ? __ldg(p.ci + o + e) : -1;
            }
            arcs(valid, u);
        }
        return true;
    }

    // Arcs of a wave of more than kTailThreads vertices, counted as at most
    // budget + 1 per warp (queue not walked yet: qb is the wave's buffer).
    // Without it one CTA would walk a hub in such a wave alone: a wave of 600
    // vertices, one of them with a million leaves, in a graph of 16.4 M arcs, 2.10 ms
    // against 0.84 with it (R-MAT scale 22 and Chung-Lu 2^22 unchanged within 1 %).
    __device__ __forceinline__ unsigned wave_arcs(const TailTotals &t, unsigned own)
    {
        unsigned sum = 0;
        const auto add = [&](int v) {
            sum = min(sum + (unsigned)tail_row((long long)(p.rp[v + 1] - p.rp[v]), budget), budget + 1);
        };
        for (unsigned i = threadIdx.x; i < own; i += blockDim.x) add(sh.queue[qb][i]);
        for (unsigned i = rank * blockDim.x + threadIdx.x; i < t.queued - t.fitted;
             i += (unsigned)kTailCtas * blockDim.x)
            add(ldcg(p.fs + listed + i));
        sum = min(__reduce_add_sync(kFull, sum), budget + 1);
        if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&sh.kept, sum);
        return exchange(true).kept;
    }

    // Walks the wave's vertices (buffer b). Returns false, with nothing walked,
    // when they have more than the budget's arcs (decided alike by every CTA); a wave
    // of more than kTailThreads vertices was counted before.
    __device__ __forceinline__ bool wave(unsigned b, const TailTotals &t)
    {
        const unsigned total = t.queued;
        const unsigned tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = T >> 5;
        const bool together = total <= T;
        const unsigned stride = together ? 1u : (unsigned)kTailCtas, first = together ? 0u : rank;
        for (unsigned base = 0; base * stride + first < total; base += T) {
            const unsigned i = (base + tid) * stride + first;
            const int v = queued_vertex(b, t, i, i < total);
            Off rs = 0;
            int d = 0;
            if (v >= 0) {
                rs = p.rp[v];
                d = tail_row((long long)(p.rp[v + 1] - rs), budget);
            }
            int incl = d;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, o);
                if ((int)lane >= o) incl += y;
            }
            if (lane == 31) sh.wsum[warp] = incl;
            __syncthreads();
            int ws = lane < nw ? sh.wsum[lane] : 0;
            const int arcs_total = (int)__reduce_add_sync(kFull, (unsigned)ws);
            const int before = (int)__reduce_add_sync(kFull, lane < warp ? (unsigned)ws : 0u);
            const int excl = before + incl - d;
            sh.start[tid] = excl;
            sh.off[tid] = (long long)rs - excl;
            if (tid < 32) sh.start[T + tid] = INT_MAX;
            __syncthreads();
            if (together && (unsigned)arcs_total > budget) return false;
            const int nseg = (arcs_total + 32 * U - 1) / (32 * U);
            const int step = (int)(together ? nw * (unsigned)kTailCtas : nw);
            for (int seg = (int)(together ? warp * (unsigned)kTailCtas + rank : warp); seg < nseg;
                 seg += step) {
                const int a0 = seg * 32 * U;
                // the last row that starts at or before a0: the lanes look at one
                // row in T / 32, then at the rows between two of those
                constexpr int kStride = kTailThreads / 32;
                int row = kStride * (__popc(__ballot_sync(kFull, sh.start[kStride * lane] <= a0)) - 1);
                row += __popc(__ballot_sync(
                           kFull, lane < (unsigned)kStride && sh.start[row + (int)lane] <= a0)) - 1;
                bool valid[U];
                int u[U];
#pragma unroll
                for (int j = 0; j < U; ++j) {
                    const int w = a0 + 32 * j, e = w + (int)lane;
                    valid[j] = e < arcs_total;
                    u[j] = -1;
                    if (w < arcs_total) {   // uniform
                        // rows that start in this window, one bit each
                        const unsigned rel = (unsigned)(sh.start[row + 1 + (int)lane] - w);
                        const unsigned starts = __reduce_or_sync(kFull, rel < 32u ? 1u << rel : 0u);
                        const int own = row + __popc(starts & (0xffffffffu >> (31 - lane)));
                        row += __popc(starts);
                        if (valid[j]) u[j] = __ldg(p.ci + sh.off[own] + e);
                    }
                }
                arcs(valid, u);
            }
            if (!together) __syncthreads();   // the rows are read before the next tile
        }
        return true;
    }

    // Scans the near list, or (full) the residual list lst[0, cnt) into
    // dst[0, ...): the vertices at k are queued. Ends without a barrier.
    template <bool full, int N>
    __device__ __forceinline__ void scan(const int *lst, unsigned cnt, int *dst)
    {
        const unsigned T = blockDim.x, lane = threadIdx.x & 31;
        const unsigned from = nb ^ 1u;   // near buffer read
        const unsigned total = full ? cnt : min(sh.near_n[from], (unsigned)kTailNear);
        int mn = INT_MAX;
        for (unsigned base = 0; base < total; base += N * T) {
            int v[N], r[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const unsigned i = base + j * T + threadIdx.x;
                v[j] = i < total ? (full ? ldcg(lst + i) : sh.near[from][i]) : -1;
            }
#pragma unroll
            for (int j = 0; j < N; ++j) r[j] = v[j] >= 0 ? ldcg(p.work + v[j]) : INT_MIN;
            bool at[N], keep[N], near[N];
            unsigned pos[N];
#pragma unroll
            for (int j = 0; j < N; ++j) {
                at[j] = r[j] == k;
                keep[j] = r[j] > k;
                near[j] = keep[j] && r[j] < hi;
                if (keep[j]) mn = min(mn, r[j]);
            }
            push(at, v);
            if (full && reserve(keep, &sh.kept, pos)) {
#pragma unroll
                for (int j = 0; j < N; ++j)
                    if (keep[j]) dst[pos[j]] = v[j];
            }
            add_near(near, v);
        }
        mn = __reduce_min_sync(kFull, mn);
        if (lane == 0 && mn != INT_MAX) atomicMin(&sh.vmin, mn);
    }

    // Returns whether the run is over (the same in every CTA).
    __device__ __forceinline__ bool run(unsigned long long *st)
    {
        const unsigned T = blockDim.x, lane = threadIdx.x & 31;
        const bool lead = rank == 0 && threadIdx.x == 0;
        const unsigned nres = ts->nres;
        unsigned cur = ts->cur;
        const unsigned per = (nres + kTailCtas - 1) / kTailCtas;
        const unsigned seg = min(rank * per, nres);
        unsigned cnt = min(per, nres - seg);
        int window = kTailWindow;
        unsigned left = nres;   // vertices not queued yet
        int mode = kTailDone;
        unsigned pend = 0;      // fs entries up to the end of those handed back
        k = hi = ts->k;
        if (threadIdx.x == 0) {
            sh.qn[0] = sh.qn[1] = 0;
            sh.near_n[0] = sh.near_n[1] = 0;
            sh.kept = sh.overflow = 0;
            sh.vmin = INT_MAX;
            if (rank == 0) ts->spilled = 0;
        }
        __syncthreads();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // every CTA is ready
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        const long long max_steps = 4ll * p.n + 64;
        for (long long steps = 0;; ++steps) {
            if (steps > max_steps) {
                if (threadIdx.x == 0) set_error(p.ctl, kErrNotConverged);
                break;
            }
            // ---- scan
            const bool full = k >= hi;
            const int *lst = (cur ? p.res1 : p.res0) + seg;
            int *dst = (cur ? p.res0 : p.res1) + seg;
            if (full) hi = k > INT_MAX - window ? INT_MAX : k + window;
            nb ^= 1u;
            if (full) scan<true, 4>(lst, cnt, dst);
            else scan<false, 1>(lst, cnt, dst);
            TailTotals t = exchange(true);
            if (full) {
                cnt = sh.x[par ^ 1u][rank][0].w;
                cur ^= 1u;
                left = t.kept;
                if (t.near_max < (unsigned)kTailNear / 8 && window < 4096) window *= 2;
                if (t.overflow && window > 1) window = max(1, window / 4);
            } else {
                left -= t.queued;
            }
            // a near list that overflowed is not read: the next scan is of the
            // residual list, and its exchange clears the buffer
            if (t.overflow) hi = k + 1;
            if (lead) {
                ++st[kStScans];
                st[kStScanned] += full ? t.kept + t.queued : t.near_max;
            }
            if (t.queued == 0) {   // empty level
                if (t.vmin != INT_MAX) k = t.vmin;
                else if (full) break;   // nothing is left
                else k = hi;
                continue;
            }
            if (lead) {
                ++st[kStLevels];
                if ((unsigned long long)k > st[kStKmax]) st[kStKmax] = (unsigned long long)k;
            }
            // ---- waves
            bool lost = false;   // a wave's additions to the near list did not fit
            while (t.queued > 0 && left > 0) {
                const unsigned b = qb, own = min(sh.x[par ^ 1u][rank][0].x, (unsigned)kTailQueue);
                settle(b, own);
                if ((unsigned long long)t.queued * (unsigned)k > budget ||
                    (budget != kTailNoBudget && t.queued > T && wave_arcs(t, own) > budget)) {
                    mode = kTailPending;
                } else {
                    qb ^= 1u;
                    if (!(t.queued <= 32u ? wave_small(b, t) : wave(b, t))) {
                        mode = kTailPending;
                        qb = b;
                    }
                }
                const unsigned beyond = listed + (t.queued - t.fitted);
                if (mode == kTailPending) {   // the grid kernel walks this wave
                    const unsigned at = beyond + __shfl_sync(kFull, t.before, rank);
                    for (unsigned i = threadIdx.x; i < own; i += T) p.fs[at + i] = sh.queue[b][i];
                    pend = beyond + t.fitted;
                    break;
                }
                listed = beyond;
                t = exchange(false);
                left -= t.queued;
                lost |= t.overflow;
                if (lead) ++st[kStSubrounds];
            }
            if (mode == kTailPending) break;
            if (left == 0) {
                settle(qb, min(sh.x[par ^ 1u][rank][0].x, (unsigned)kTailQueue));
                break;
            }
            if (lost) hi = k + 1;
            ++k;
        }
        if (mode == kTailDone) {
            if (lead) {
                ts->mode = kTailDone;
                ts->k = k;
            }
            return true;
        }
        // hand over: the residual list in one piece, the barrier and the scan
        // counters of the grid kernel at zero
        __syncthreads();
        if (threadIdx.x == 0) sh.qn[qb] = cnt;
        __syncthreads();
        (void)exchange(false);
        const unsigned mine = lane < (unsigned)kTailCtas ? sh.x[par ^ 1u][lane][0].x : 0u;
        const unsigned before = __reduce_add_sync(kFull, lane < rank ? mine : 0u);
        const unsigned total = __reduce_add_sync(kFull, mine);
        const int *src = (cur ? p.res1 : p.res0) + seg;
        int *dst = (cur ? p.res0 : p.res1) + before;
        for (unsigned i = threadIdx.x; i < cnt; i += T) dst[i] = ldcg(src + i);
        if (rank == 0) {
            if (threadIdx.x == 0) {
                ts->mode = mode;
                ts->k = k;
                ts->nres = total;
                ts->cur = cur ^ 1u;
                ts->lo = listed;
                ts->hi = pend;
                p.ctl->bar.w[0] = p.ctl->bar.w[1] = 0;
                p.ctl->gen.w[0] = 0;
            }
            if (threadIdx.x >= L_KEPT && threadIdx.x < L_FA + 3) p.ctl->live.w[threadIdx.x] = 0;
        }
        return false;
    }
};

}  // namespace peel
}  // namespace pico
