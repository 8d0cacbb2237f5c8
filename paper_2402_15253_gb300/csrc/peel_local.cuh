// PeelOne (Sec. III, Alg. 4) with the residual degrees in shared memory: one
// CTA, or the CTAs of one thread-block cluster, peel one graph.
//
// The levels and their dynamic frontier are those of peelone.cuh. What
// differs is where the decrements go. In global memory every decrement is an
// L2 round trip, and L2 serves 0.56 returning atomics per clock and SM when
// every SM issues them (measured, random words of 16 MB); shared memory
// serves at least 7 per clock and SM, 42 clocks each in a chain of one warp where L2
// takes 720. So each CTA keeps the residual degrees of the vertices it owns in shared
// memory, needs no guard read before a decrement (a decrement of a queued vertex
// returns at most k and is ignored), and a wave ends with __syncthreads.
//
//   one CTA    (n <= kLocalSlots) owns every vertex.
//   a cluster  of c CTAs (n <= c * kLocalSlots): CTA r owns the vertices
//              [r * per, (r + 1) * per). Every CTA walks every frontier arc
//              and applies the ones that end at its own vertices. Sharing the
//              walk and decrementing through distributed shared memory (0.37
//              atomics per clock and SM, measured) takes the same time: 184
//              graphs of 51,201 to 200,000 vertices 11.3 ms either way.
//
// Queue: each CTA queues its own vertices (each once over the run) in its
// part of a global array, level by level; a single CTA keeps the first
// entries of a level in shared memory. After a wave the CTAs tell
// each other how many vertices they queued (one remote store per pair, ordered
// by the cluster barrier). Counts rotate over three slots: in phase w a CTA
// adds to slot w, reads slot w - 1 and clears slot w + 1, whose last readers
// passed the barrier that ended phase w - 1.
//
// Work assignment in a wave: a warp takes up to 32 frontier vertices and walks
// their concatenated rows; longer rows are split into chunks listed in shared
// memory that all warps take after a CTA barrier.
//
// The run ends as soon as every vertex is queued: what is left of the last
// level's walk could only lower vertices that have their coreness. The
// statistics are Alg. 4's: every vertex's row is expanded once, and a vertex of
// degree d and coreness c is lowered d - c times, in any order of the frontier.
#pragma once

#include "pico_device.cuh"

namespace pico {
namespace peel {

constexpr int kLocalSlots = 51200;   // residual degrees per CTA (200 KB of shared memory)
// Rows longer than a piece are split over the CTA's warps: into 128 arcs (one
// step of a warp) when a wave has no more rows than warps, else 256.
__device__ __forceinline__ int local_piece(unsigned vb) { return vb == 1u ? 128 : 256; }
constexpr int kLocalMaxCtas = 4;

// Capacities of a CTA's shared lists: queue entries of a level kept in shared
// memory, and chunk entries listed at once.
struct LocalWide {
    static constexpr int kQueue = 2048, kChunks = 1024;
};
struct LocalTiny {
    static constexpr int kQueue = 512, kChunks = 128;
};

template <typename Off>
struct LocalParams {
    const Off *rp;
    const int *ci;
    int n;
    long long m;
    int *core;
    int *qs;      // n slots
    Ctrl *ctl;
};

// Fixed shared-memory part; the residual degrees follow it.
template <typename Cap>
struct LocalShared {
    unsigned long long c_start[Cap::kChunks];   // chunk entries: first arc, arcs
    int c_len[Cap::kChunks];
    int queue[Cap::kQueue];
    unsigned pushed[3];                         // own vertices queued, per phase
    int vmin[3];                                // smallest own residual degree above k
    unsigned nchunk[3];
    unsigned x_cnt[3][kLocalMaxCtas];           // every CTA's counts and minima, per phase
    int x_min[3][kLocalMaxCtas];
};

// Statistics of one graph, uniform over the CTA.
struct LocalStats {
    unsigned long long levels = 0, waves = 0, scans = 0, core_sum = 0;
    int kmax = 0;
};

// What a CTA that peels a graph alone keeps of it in shared memory besides the
// residual degrees: the row offsets, or all of it. A wave of a small graph is a
// chain of dependent accesses (row bounds, columns, decrements), and each of
// the first two takes some 500 clocks from L2 (440-535, a load of one warp) and 30 from
// shared memory.
enum : int { kKeepNone = 0, kKeepRows = 1, kKeepGraph = 2 };

// Dynamic shared memory of a CTA that owns `n` vertices (and the m arcs of the
// whole graph, if kept).
template <typename Cap>
__host__ __device__ inline size_t local_smem_bytes(long long n, int kept = kKeepNone, long long m = 0)
{
    const size_t slots = (size_t)((n + 3) & ~3ll);
    size_t b = ((sizeof(LocalShared<Cap>) + 15) & ~size_t(15)) + slots * sizeof(int);
    if (kept != kKeepNone) b += (slots + 4) * sizeof(int);
    if (kept == kKeepGraph) b += (size_t)m * sizeof(int);
    return b;
}

// The most that fits `bytes` of dynamic shared memory.
template <typename Cap>
__host__ __device__ inline int local_kept(long long n, long long m, size_t bytes)
{
    if (local_smem_bytes<Cap>(n, kKeepGraph, m) <= bytes) return kKeepGraph;
    return local_smem_bytes<Cap>(n, kKeepRows) <= bytes ? kKeepRows : kKeepNone;
}

constexpr size_t kLocalSmem = 227 * 1024 - 2048;   // dynamic shared memory of a wide CTA

__device__ __forceinline__ unsigned shared_addr(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

// Stores v at the same shared-memory location of CTA `rank` of the cluster.
__device__ __forceinline__ void store_remote(const void *p, unsigned rank, unsigned v)
{
    unsigned a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(shared_addr(p)), "r"(rank));
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

__device__ __forceinline__ int shared_dec(unsigned addr)
{
    int old;
    asm volatile("atom.relaxed.cta.shared::cta.add.s32 %0, [%1], -1;"
                 : "=r"(old)
                 : "r"(addr)
                 : "memory");
    return old;
}

// One warp walks the concatenated rows of its lanes' vertices (d = 0: none;
// lanes with d > 0 come first). A 32-arc window's owners follow from the
// rows that start in it: one warp-wide OR and a population count, where a
// search over the row starts would take five dependent shuffles. f takes
// F::kArcs windows at a time: f.arcs(valid, u), called by all 32 lanes.
// kShared: ci is in shared memory.
template <bool kShared, typename Off, typename F>
__device__ __forceinline__ void walk_rows(const int *__restrict__ ci, Off rs, int d, F &f)
{
    constexpr int U = F::kArcs;
    const int lane = threadIdx.x & 31;
    int incl = d;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    const int excl = incl - d;
    const int total = __shfl_sync(kFull, incl, 31);
    const Off off = rs - (Off)excl;
    int before = -1;   // rows started before the window, minus one
    for (int base = 0; base < total; base += 32 * U) {
        bool valid[U];
        int u[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int w = base + 32 * j, e = w + lane;
            valid[j] = e < total;
            u[j] = -1;
            if (w < total) {   // uniform
                const unsigned rel = (unsigned)(excl - w);
                const unsigned starts =
                    __reduce_or_sync(kFull, d > 0 && rel < 32u ? 1u << rel : 0u);
                const int owner = before + __popc(starts & (0xffffffffu >> (31 - lane)));
                before += __popc(starts);
                const Off o = __shfl_sync(kFull, off, owner & 31);
                if (valid[j]) u[j] = kShared ? ci[o + e] : __ldg(ci + o + e);
            }
        }
        f.arcs(valid, u);
    }
}

// One warp walks `len` consecutive arcs.
template <bool kShared, typename F>
__device__ __forceinline__ void walk_arcs(const int *__restrict__ c, int len, F &f)
{
    constexpr int U = F::kArcs;
    const int lane = threadIdx.x & 31;
    for (int base = 0; base < len; base += 32 * U) {
        bool valid[U];
        int u[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int e = base + 32 * j + lane;
            valid[j] = e < len;
            u[j] = valid[j] ? (kShared ? c[e] : __ldg(c + e)) : -1;
        }
        f.arcs(valid, u);
    }
}

// Moves the lanes with d > 0 to the front of the warp (walk_rows' order).
template <typename Off>
__device__ __forceinline__ void pack_rows(Off &rs, int &d)
{
    const unsigned have = __ballot_sync(kFull, d > 0);
    if ((have & (have + 1u)) == 0) return;   // no gap
    const unsigned lane = threadIdx.x & 31;
    unsigned src = 0;   // lane of the (lane + 1)-th row
#pragma unroll
    for (unsigned s = 16; s > 0; s >>= 1)
        if ((unsigned)__popc(have & ((1u << (src + s)) - 1u)) <= lane) src += s;
    const Off rs2 = __shfl_sync(kFull, rs, src);
    const int d2 = __shfl_sync(kFull, d, src);
    rs = rs2;
    d = lane < (unsigned)__popc(have) ? d2 : 0;
}

template <typename Off, typename Cap, bool kCluster, int kKept>
struct LocalPeel {
    // a whole graph in shared memory is small: its waves go through this code
    // once, and fetching the instructions is part of their latency
    static constexpr int kArcs = kKept == kKeepGraph ? 2 : 4;
    static constexpr bool kCols = kKept == kKeepGraph;
    const LocalParams<Off> &p;
    LocalShared<Cap> &sh;
    int *res;
    unsigned res_addr;     // its shared-memory address
    int *rows, *cols;      // copies of row_ptr and col_idx, if kept
    unsigned rank, ctas;   // this CTA in its cluster
    int per;               // vertices per CTA
    int vbase, cnt;        // own vertices
    int k = 0;
    unsigned ph = 0;       // phase slot (0..2)
    int q0 = 0;            // own entries of the level queued before this phase

    __device__ __forceinline__ static unsigned next(unsigned s) { return s == 2 ? 0 : s + 1; }

    // Queues the own vertices v[j] of the lanes with push[j] (one counter
    // update per warp; all lanes call).
    template <int U>
    __device__ __forceinline__ void queue_own(const bool (&push)[U], const int (&v)[U])
    {
        bool any = false;
#pragma unroll
        for (int j = 0; j < U; ++j) any |= push[j];
        if (!__any_sync(kFull, any)) return;
        const unsigned lane = threadIdx.x & 31;
        unsigned b[U], total = 0;
#pragma unroll
        for (int j = 0; j < U; ++j) {
            b[j] = __ballot_sync(kFull, push[j]);
            total += __popc(b[j]);
        }
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(&sh.pushed[ph], total);
        base = __shfl_sync(kFull, base, 0);
#pragma unroll
        for (int j = 0; j < U; ++j) {
            if (push[j]) {
                const int pos = q0 + (int)(base + __popc(b[j] & ((1u << lane) - 1u)));
                p.core[v[j]] = k;
                if (!kCluster && pos < Cap::kQueue) sh.queue[pos] = v[j];
                else p.qs[vbase + pos] = v[j];   // pos < cnt: each own vertex is queued once
            }
            base += __popc(b[j]);
        }
    }

    // The decrements of a step's arcs (walk_rows, walk_arcs): all issued
    // before the first result is used.
    __device__ __forceinline__ void arcs(const bool (&valid)[kArcs], const int (&u)[kArcs])
    {
        int old[kArcs];
#pragma unroll
        for (int j = 0; j < kArcs; ++j) {
            const unsigned x = (unsigned)(u[j] - vbase);
            old[j] = valid[j] && x < (unsigned)cnt ? shared_dec(res_addr + 4u * x) : 0;
        }
        bool push[kArcs];
#pragma unroll
        for (int j = 0; j < kArcs; ++j) {
            push[j] = old[j] == k + 1;   // k + 1 > 0
        }
        queue_own(push, u);
    }

    // Queues the own vertices whose residual degree is k, and records the
    // smallest one above k.
    __device__ __forceinline__ void collect()
    {
        const int tid = (int)threadIdx.x, T = (int)blockDim.x;
        int mn = INT_MAX;
        const int4 *r4 = reinterpret_cast<const int4 *>(res);
        for (int base = 0; base < cnt; base += 4 * T) {
            const int i = base + 4 * tid;
            int4 c = make_int4(0, 0, 0, 0);
            if (i < cnt) c = r4[i >> 2];   // the padding holds 0 < k
            const int cv[4] = {c.x, c.y, c.z, c.w};
            bool push[4];
            int v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                push[j] = cv[j] == k;
                if (cv[j] > k) mn = min(mn, cv[j]);
                v[j] = vbase + i + j;
            }
            queue_own(push, v);
        }
        mn = __reduce_min_sync(kFull, mn);
        if ((tid & 31) == 0 && mn != INT_MAX) atomicMin(&sh.vmin[ph], mn);
    }

    // Ends a phase: every CTA learns every CTA's count (and, after a scan, its
    // smallest residual degree) in slot ph, then the slots advance.
    template <bool kMin>
    __device__ __forceinline__ void end_phase()
    {
        __syncthreads();
        if (kCluster) {
            if (threadIdx.x < ctas) {
                store_remote(&sh.x_cnt[ph][rank], threadIdx.x, sh.pushed[ph]);
                if (kMin) store_remote(&sh.x_min[ph][rank], threadIdx.x, (unsigned)sh.vmin[ph]);
            }
            __syncwarp();
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
        ph = next(ph);
        if (threadIdx.x == 0) {   // the slot of the phase after this one
            const unsigned c = next(ph);
            sh.pushed[c] = 0;
            sh.vmin[c] = INT_MAX;
            sh.nchunk[c] = 0;
        }
    }

    __device__ __forceinline__ unsigned count_of(unsigned slot, unsigned r) const
    {
        return kCluster ? sh.x_cnt[slot][r] : sh.pushed[slot];
    }
    __device__ __forceinline__ unsigned total_of(unsigned slot) const
    {
        if (!kCluster) return sh.pushed[slot];
        unsigned t = 0;
        for (unsigned r = 0; r < ctas; ++r) t += sh.x_cnt[slot][r];
        return t;
    }
    __device__ __forceinline__ int min_of(unsigned slot) const
    {
        if (!kCluster) return sh.vmin[slot];
        int t = INT_MAX;
        for (unsigned r = 0; r < ctas; ++r) t = min(t, sh.x_min[slot][r]);
        return t;
    }

    __device__ __forceinline__ void row(int v, Off &rs, int &d) const
    {
        if (kKept != kKeepNone) {
            const int a = rows[v];
            rs = (Off)a;
            d = rows[v + 1] - a;
        } else {
            rs = p.rp[v];
            d = (int)(p.rp[v + 1] - rs);
        }
    }
    __device__ __forceinline__ const int *columns() const { return kCols ? cols : p.ci; }

    // Walks the vertices queued in phase slot `s`; q[r] is the level's queue
    // position of CTA r's first one.
    __device__ __forceinline__ void wave(unsigned s, unsigned total, const int (&q)[kLocalMaxCtas])
    {
        const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const unsigned vb = batch_width(total, 0, nw);
        const int piece = local_piece(vb);
        for (unsigned unit = warp; unit * vb < total; unit += nw) {
            unsigned i = unit * vb + lane;
            int v = -1;
            if (lane < vb && i < total) {
                if (kCluster) {
                    int pos = q[0];
                    unsigned r = 0;
#pragma unroll
                    for (unsigned t = 0; t + 1 < kLocalMaxCtas; ++t)
                        if (r == t && t + 1 < ctas && i >= sh.x_cnt[s][t]) {
                            i -= sh.x_cnt[s][t];
                            r = t + 1;
                            pos = q[t + 1];
                        }
                    v = ldcg(p.qs + (long long)r * per + pos + i);
                } else {
                    const int pos = q[0] + (int)i;
                    v = pos < Cap::kQueue ? sh.queue[pos] : ldcg(p.qs + pos);
                }
            }
            Off rs = 0;
            int d = 0;
            if (v >= 0) row(v, rs, d);
            unsigned bigs = __ballot_sync(kFull, d > piece);
            while (bigs) {   // list the chunks of long rows, or walk them here when the list is full
                const int src = __ffs(bigs) - 1;
                bigs &= bigs - 1;
                const Off s0 = __shfl_sync(kFull, rs, src);
                const int dd = __shfl_sync(kFull, d, src);
                const int size = max(piece, ((dd >> 8) + 127) & ~127);   // at most 257 pieces
                const unsigned nch = (unsigned)((dd + size - 1) / size);
                unsigned pos = 0;
                if (lane == 0) pos = atomicAdd(&sh.nchunk[ph], nch);
                pos = __shfl_sync(kFull, pos, 0);
                const bool fits = pos + nch <= Cap::kChunks;
                for (unsigned c = lane; c < nch && pos + c < Cap::kChunks; c += 32) {
                    sh.c_start[pos + c] = (unsigned long long)(s0 + (Off)c * size);
                    sh.c_len[pos + c] = fits ? min(size, dd - (int)c * size) : 0;
                }
                if (!fits) walk_arcs<kCols>(columns() + s0, dd, *this);
            }
            if (d > piece) d = 0;
            if (vb == 1u) {
                walk_arcs<kCols>(columns() + __shfl_sync(kFull, rs, 0), __shfl_sync(kFull, d, 0), *this);
            } else {
                pack_rows(rs, d);
                walk_rows<kCols>(columns(), rs, d, *this);
            }
        }
        __syncthreads();
        const unsigned nch = min(sh.nchunk[ph], (unsigned)Cap::kChunks);
        for (unsigned c = warp; c < nch; c += nw)
            walk_arcs<kCols>(columns() + sh.c_start[c], sh.c_len[c], *this);
    }

    // Peels the graph. Every thread of the CTA (cluster) calls it.
    __device__ __forceinline__ LocalStats run()
    {
        LocalStats st;
        const int tid = (int)threadIdx.x, T = (int)blockDim.x;
        const unsigned lane = threadIdx.x & 31;
        if (tid < 3) {
            sh.pushed[tid] = 0;
            sh.vmin[tid] = INT_MAX;
            sh.nchunk[tid] = 0;
        }
        __syncthreads();
        // init: residual degree = degree; pushed counts the non-isolated vertices here
        int mn = INT_MAX;
        unsigned linked = 0;
        for (int i = tid; i < ((cnt + 3) & ~3); i += T) {
            int d = 0;
            if (i < cnt) {
                const int v = vbase + i;
                const Off rs = p.rp[v];
                d = (int)(p.rp[v + 1] - rs);
                if (d == 0) p.core[v] = 0;
                if (kKept != kKeepNone) {
                    rows[v] = (int)rs;
                    if (v + 1 == cnt) rows[v + 1] = (int)rs + d;
                }
            }
            res[i] = d;
            if (d > 0) {
                mn = min(mn, d);
                ++linked;
            }
        }
        if (kCols) {
#pragma unroll 8
            for (int i = tid; i < (int)p.m; i += T) cols[i] = __ldg(p.ci + i);
        }
        linked = __reduce_add_sync(kFull, linked);
        if (lane == 0 && linked) atomicAdd(&sh.pushed[ph], linked);
        mn = __reduce_min_sync(kFull, mn);
        if (lane == 0 && mn != INT_MAX) atomicMin(&sh.vmin[ph], mn);
        end_phase<true>();
        unsigned prev = ph == 0 ? 2 : ph - 1;
        unsigned alive = total_of(prev);   // vertices not yet queued
        k = min_of(prev);
        long long steps = 0;
        while (alive > 0) {
            if (++steps > 2ll * p.n + 4) {
                if (tid == 0) set_error(p.ctl, kErrNotConverged);
                break;
            }
            // scan: own vertices at k are the level's static frontier
            q0 = 0;
            ++st.scans;
            collect();
            end_phase<true>();
            prev = ph == 0 ? 2 : ph - 1;
            unsigned total = total_of(prev);
            const int above = min_of(prev);
            if (total == 0) {   // empty level: jump to the smallest residual degree
                if (above == INT_MAX) {
                    if (tid == 0) set_error(p.ctl, kErrNotConverged);
                    break;
                }
                k = above;
                continue;
            }
            ++st.levels;
            st.kmax = k;
            int q[kLocalMaxCtas];
#pragma unroll
            for (int r = 0; r < kLocalMaxCtas; ++r) q[r] = 0;
            while (total > 0) {
                alive -= total;
                st.core_sum += (unsigned long long)total * (unsigned)k;
                ++st.waves;
                if (alive == 0) break;   // every vertex has its coreness
                q0 += (int)count_of(prev, rank);
                wave(prev, total, q);
                end_phase<false>();
                // the entries walked are behind the level's queue position now
                if (kCluster) {
#pragma unroll
                    for (int r = 0; r < kLocalMaxCtas; ++r)
                        if (r < (int)ctas) q[r] += (int)sh.x_cnt[prev][r];
                } else {
                    q[0] = q0;
                }
                prev = ph == 0 ? 2 : ph - 1;
                total = total_of(prev);
            }
            ++k;
        }
        return st;
    }
};

// smem: local_smem_bytes<Cap>(...) bytes of dynamic shared memory.
template <typename Off, typename Cap, bool kCluster, int kKept = kKeepNone>
__device__ __forceinline__ LocalStats run_local(const LocalParams<Off> &p, char *smem, unsigned rank,
                                                unsigned ctas)
{
    LocalShared<Cap> &sh = *reinterpret_cast<LocalShared<Cap> *>(smem);
    int *res = reinterpret_cast<int *>(smem + ((sizeof(LocalShared<Cap>) + 15) & ~size_t(15)));
    int *rows = res + ((p.n + 3) & ~3);
    LocalPeel<Off, Cap, kCluster, kKept> lp{p, sh, res, shared_addr(res), rows,
                                            rows + ((p.n + 3) & ~3) + 4, rank, ctas};
    lp.per = kCluster ? (int)(((p.n + (int)ctas - 1) / (int)ctas + 3) & ~3) : p.n;
    lp.vbase = (int)rank * lp.per;
    lp.cnt = max(0, min(lp.per, p.n - lp.vbase));
    return lp.run();
}

// Adds one graph's PeelOne statistics to the CTA's (thread 0 of one CTA).
__device__ __forceinline__ void add_stats(unsigned long long *st, const LocalStats &s, int n,
                                          long long m)
{
    st[kStLevels] += s.levels;
    st[kStSubrounds] += s.waves;
    st[kStScans] += s.scans;
    st[kStScanned] += s.scans * (unsigned long long)n;
    st[kStArcs] += (unsigned long long)m;
    st[kStAtomics] += (unsigned long long)m - s.core_sum;
    if ((unsigned long long)s.kmax > st[kStKmax]) st[kStKmax] = (unsigned long long)s.kmax;
}

}  // namespace peel
}  // namespace pico
