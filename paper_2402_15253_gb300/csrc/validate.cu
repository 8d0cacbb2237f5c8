// Input validation of a single-graph CSR: the paper's graphs are simple and
// undirected (Sec. II-A), and both methods rely on it (PeelOne decrements
// each neighbour once per arc, HistoCore's pulled rounds read an edit from
// the far end of each arc). Two launches on the caller's stream, or three:
//   rows   row_ptr[0] == 0, row_ptr non-decreasing, row_ptr[n] == m;
//   quick  (only when the rows passed, so that every row lies inside
//          col_idx) whether every neighbour id is in [0, n), no arc is a
//          self-loop, every row is strictly increasing and the graph is
//          symmetric. Symmetry takes one lookup per pair of arcs: of (v, u) and
//          (u, v), the one whose far end has the smaller (degree, id) is looked
//          up there by binary search. In strictly increasing rows two such
//          arcs never find the same partner, so when all are found and there
//          are as many of them as of the others, every arc has its reverse.
//   arcs   (only when the quick pass found something, which the host reads) every
//          arc's defects, each reverse looked up.
// The quick pass shares the arcs out evenly, up to 512 to a warp: one warp per row
// leaves a hub's row to a single warp (R-MAT scale 20, n 1.0 M, m 31 M: 9.2 ms).
// What remains is its gathers: two row bounds per arc, and a lookup in the
// shorter row for half of them. Valid Erdos-Renyi graphs of 2,000 rows of 200 arcs and
// 200,000 of 20: 52 and 113 us, 63 and 108 by the exact kernel alone; with one bad id 88
// and 196 us, 63 and 107. Each kernel ORs what it finds into one device
// word. Every load is bounds-checked first, so a malformed graph becomes a
// reported defect, never an out-of-range access.
#include <algorithm>

#include "pico.h"
#include "pico_device.cuh"
#include "pico_launch.h"

namespace pico {
namespace {

template <typename Off>
__global__ void __launch_bounds__(256)
    validate_rows(const Off *rp, long long n, long long m, unsigned *flag)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    bool bad = false;
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v <= n; v += stride) {
        const long long a = (long long)rp[v];
        if (v == 0 && a != 0) bad = true;
        if (v == n && a != m) bad = true;
        if (v < n) {
            const long long b = (long long)rp[v + 1];
            if (a < 0 || b < a || b > m) bad = true;
        }
    }
    if (bad) atomicOr(flag, PICO_DEFECT_ROWS);
}

constexpr int kSegment = 512;   // most arcs of a warp's turn in the quick pass

// The last row in [lo, hi) that starts at or before arc a, by 32-way search (one
// warp); rp[lo] <= a < rp[hi].
template <typename Off>
__device__ __forceinline__ long long row_at(const Off *rp, long long lo, long long hi, long long a)
{
    const int lane = threadIdx.x & 31;
    while (hi - lo > 1) {
        const long long step = (hi - lo + 31) / 32, at = lo + (lane + 1) * step;
        const unsigned b = __ballot_sync(kFull, at < hi && (long long)rp[at] <= a);
        lo += (long long)__popc(b) * step;   // the probes that pass come first
        hi = lo + step < hi ? lo + step : hi;
    }
    return lo;
}

// segment: arcs of a warp's turn, a multiple of 32
template <typename Off>
__global__ void __launch_bounds__(256)
    validate_quick(const Off *rp, const int *ci, long long n, long long m, int segment,
                   ValidateWords *words)
{
    __shared__ long long s_sum[8];
    // the rows kernel ran before on this stream: its word is final here
    if (ld_relaxed(&words->defects) & PICO_DEFECT_ROWS) return;
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long nseg = (m + segment - 1) / segment;
    bool bad = false;
    int excess = 0;   // arcs looked up minus the others
    for (long long seg = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; seg < nseg;
         seg += nw) {
        const long long a0 = seg * segment, a1 = a0 + segment < m ? a0 + segment : m;
        long long lo = row_at(rp, 0, n, a0);
        for (long long w = a0; w < a1; w += 32) {
            const long long e = w + lane;
            // the row of each arc: the starts of the next 32 rows, and again
            // while they all lie at or before the window's last arc
            const long long last = w + 31 < a1 ? w + 31 : a1 - 1;
            const long long mine = e < a1 ? e : last;
            long long v = lo;
            for (;;) {
                const long long r = lo + 1 + lane < n ? lo + 1 + lane : n;
                const long long start = (long long)rp[r];
                int c = 0;
#pragma unroll
                for (int s = 16; s > 0; s >>= 1)
                    if (__shfl_sync(kFull, start, c + s - 1) <= mine) c += s;
                if (__shfl_sync(kFull, start, c) <= mine) ++c;   // c <= 31 here
                if (c > 0) v = lo + c;
                const long long end = __shfl_sync(kFull, start, 31);
                if (end > last) break;
                lo += 32;
                if (__shfl_sync(kFull, start, 0) == end) {
                    // a run of empty rows, which may be millions of rows long (ids
                    // that are not used): its end is searched for
                    lo = row_at(rp, lo, n, end);
                    if (c > 0) v = lo;
                }
            }
            lo = __shfl_sync(kFull, v, 31);
            if (e >= a1) continue;
            const int u = ci[e];
            if (u < 0 || (long long)u >= n || (long long)u == v) {
                bad = true;
                continue;
            }
            const Off vs = rp[v], ve = rp[v + 1], us = rp[u], ue = rp[u + 1];
            if (e + 1 < (long long)ve && ci[e + 1] <= u) bad = true;
            const Off dv = ve - vs, du = ue - us;
            if (du < dv || (du == dv && (long long)u < v)) {
                Off x = us, y = ue;
                while (x < y) {
                    const Off mid = x + (y - x) / 2;
                    if ((long long)ci[mid] < v) x = mid + 1;
                    else y = mid;
                }
                if (x >= ue || (long long)ci[x] != v) bad = true;
                ++excess;
            } else {
                --excess;
            }
        }
    }
    if (__any_sync(kFull, bad) && lane == 0) atomicOr(&words->suspect, 1u);
    long long sum = __reduce_add_sync(kFull, excess);
    if (lane == 0) s_sum[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (unsigned i = 1; i < blockDim.x >> 5; ++i) sum += s_sum[i];
        if (sum)
            atomicAdd(reinterpret_cast<unsigned long long *>(&words->excess),
                      (unsigned long long)sum);
    }
}

template <typename Off>
__global__ void __launch_bounds__(256)
    validate_arcs(const Off *rp, const int *ci, long long n, unsigned *flag)
{
    const int lane = threadIdx.x & 31;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    unsigned bad = 0;
    // one warp per vertex, its lanes over the vertex's arcs
    for (long long v = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
        const Off a = rp[v], b = rp[v + 1];
        for (Off e = a + lane; e < b; e += 32) {
            const int u = ci[e];
            if (u < 0 || (long long)u >= n) {
                bad |= PICO_DEFECT_IDS;
                continue;
            }
            if ((long long)u == v) bad |= PICO_DEFECT_LOOP;
            if (e + 1 < b && ci[e + 1] <= u) bad |= PICO_DEFECT_ORDER;
            // (v, u) needs (u, v): v in u's row (an unsorted row of u may
            // hide it; that row is reported as unsorted anyway)
            Off lo = rp[u];
            const Off end = rp[u + 1];
            Off hi = end;
            while (lo < hi) {
                const Off mid = lo + (hi - lo) / 2;
                if ((long long)ci[mid] < v) lo = mid + 1;
                else hi = mid;
            }
            if (lo >= end || (long long)ci[lo] != v) bad |= PICO_DEFECT_ASYMMETRIC;
        }
    }
    bad = __reduce_or_sync(kFull, bad);
    if (bad && lane == 0) atomicOr(flag, bad);
}

}  // namespace

template <typename Off>
int launch_validate(const Off *rp, const int *ci, long long n, long long m, ValidateWords *words,
                    cudaStream_t stream, const LaunchCfg &cfg)
{
    // no more CTAs than the vertices, or the shares of arcs, occupy: on a small
    // graph most of a launch's time is setting up CTAs; and shares so small
    // that every warp has one: a share is walked 32 arcs at a time
    const long long most = cfg.sms > 0 ? cfg.sms * 8 : 1024;
    const int segment =
        (int)std::min<long long>(kSegment, std::max<long long>(32, (m / (8 * most) + 31) & ~31ll));
    const unsigned blocks = (unsigned)std::min<long long>(most, n / 256 + 1);
    const unsigned shares = (unsigned)std::min<long long>(most, m / (8 * segment) + 1);
    validate_rows<Off><<<blocks, 256, 0, stream>>>(rp, n, m, &words->defects);
    if (cudaGetLastError() != cudaSuccess) return -3;
    validate_quick<Off><<<shares, 256, 0, stream>>>(rp, ci, n, m, segment, words);
    if (cudaGetLastError() != cudaSuccess) return -3;
    return 0;
}

template <typename Off>
int launch_validate_exact(const Off *rp, const int *ci, long long n, ValidateWords *words,
                          cudaStream_t stream, const LaunchCfg &cfg)
{
    // a warp for every row
    const long long most = cfg.sms > 0 ? cfg.sms * 8 : 1024;
    validate_arcs<Off><<<(unsigned)std::min<long long>(most, n / 8 + 1), 256, 0, stream>>>(
        rp, ci, n, &words->defects);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template int launch_validate<int>(const int *, const int *, long long, long long, ValidateWords *,
                                  cudaStream_t, const LaunchCfg &);
template int launch_validate<long long>(const long long *, const int *, long long, long long,
                                        ValidateWords *, cudaStream_t, const LaunchCfg &);
template int launch_validate_exact<int>(const int *, const int *, long long, ValidateWords *,
                                        cudaStream_t, const LaunchCfg &);
template int launch_validate_exact<long long>(const long long *, const int *, long long,
                                              ValidateWords *, cudaStream_t, const LaunchCfg &);

}  // namespace pico
