// Batched form: the coreness of G independent graphs.
//
// Coreness is defined per connected component (Sec. I: the k-core is a
// maximal subgraph), so graphs packed side by side are solved independently.
// A schedule lists the graphs by class, and by decreasing arc count within a
// class (power-of-two buckets); CTAs and clusters draw tickets from it, so the
// largest graphs start first and the small ones fill in behind them.
//
// PeelOne keeps the residual degrees in shared memory (peel_local.cuh):
//   tiny    n <= kTinyVertices: CTAs of kTinyThreads threads, eight per SM, so
//           that one graph's barriers and chains overlap the others'.
//   middle  n <= kLocalSlots: one CTA of kWideThreads threads per graph; and tiny
//           graphs that the rest of the batch would wait for (straggles).
//   large   n <= kPeelCtas * kLocalSlots: a cluster of kPeelCtas CTAs per graph.
//   huge    the rest: a cluster of kClusterCtas CTAs per graph, in global memory
//           (peel::run over the cluster).
// Middle and large graphs share one launch: clusters first take the large
// graphs, then each CTA takes middle ones. It does not wait for the launch of
// the huge graphs before it, which leaves SMs free (24 graphs of 1 M vertices and
// 488 smaller ones, 1.2 G arcs: 28.6 ms one after the other, 25.6 ms side by side). The
// tiny graphs are the last launch, which waits for both (2,000 of them behind one graph
// of 1 M vertices add 0.3 ms).
//
// HistoCore runs the single-graph body (histo::run) in two phases: graphs of
// at least 2^cluster_log2 arcs (a tuning value) by clusters of kClusterCtas
// CTAs (ClusterDom: counters in the rank-0 CTA's shared memory, reached
// through distributed shared memory; hardware cluster barriers), the rest by
// one CTA each (CtaDom: counters in its own shared memory, __syncthreads).
//
// Scratch is sliced per graph: vertex-indexed arrays at vtx_off[g], the
// histogram at arc_off[g], and chunk lists at arc_off[g] / 16 + 2g with
// m_g / 16 + 2 entries (at least m_g / chunk + m_g / (small_deg + 1) + 2 for
// every allowed tuning: chunk >= 64 and small_deg >= 32).
#include <algorithm>

#include "histocore.cuh"
#include "peel_local.cuh"
#include "peelone.cuh"
#include "pico.h"
#include "pico_launch.h"

namespace pico {
namespace {

constexpr int kBuckets = 64;                    // arc-count buckets per class
constexpr int kClusterCtas = 8;                 // HistoCore: CTAs per cluster (portable size)
constexpr int kPeelCtas = 4;                    // PeelOne: CTAs per cluster
constexpr int kWideThreads = 1024;              // PeelOne: threads per CTA of large and middle graphs
constexpr int kTinyThreads = 128;               // ... and of tiny ones
constexpr int kTinyVertices = 2048;
constexpr size_t kTinySmem = 26 * 1024;         // eight CTAs share an SM's 228 KB
static_assert(kTinySmem >= 16 * kTinyVertices / 2 + 4096, "row offsets of a tiny graph must fit");

// control words of the batched launch (in Ctrl::live): tickets of the classes,
// and where the classes end in the schedule
enum : int { B_SMALL = 0, B_LARGE = 1, B_NLARGE = 2, B_TINY = 3, B_NMIDDLE = 4, B_HUGE = 5, B_NHUGE = 6 };

struct BatchParams {
    const long long *vtx_off, *arc_off;
    int G;
    const int *rp, *ci;
    int *core;
    int *order;
    int *res0, *res1, *qs;                          // PeelOne
    int *histo, *lists[6], *us;                     // HistoCore
    int2 *vinfo, *mv[2], *ichunks;
    int2 *chunks;                                   // both
    Ctrl *ctl;
    Tuning tn;
};

__device__ __forceinline__ int size_bucket(long long m)
{
    return m <= 0 ? 0 : 64 - __clzll(m);
}

// Whether a tiny graph takes a whole SM all the same: it has more arcs than an SM's
// share of the batch (`share`), so its 128 threads would be the last at work. Graphs of
// 2,000 vertices and 0.72 M arcs, Erdos-Renyi: 64 of them 1,432 us as tiny ones, 384 as
// middle ones (1,213 with 512 threads for each); 512 of them 1,468 and 1,233; with 0.2 M
// arcs 64 take 399 and 190 us, 512 take 423 and 510. Smaller graphs stay tiny: they take
// less time than with 512 threads each in any batch.
constexpr long long kTinyArcs = 32 << 10;
__device__ __forceinline__ bool straggles(long long m, long long share)
{
    return m > kTinyArcs && m > share;
}

// Class of a graph: 3 (listed first) to 0. PeelOne: by where its residual
// degrees fit; HistoCore: by its arcs (classes 2 and 0).
__device__ __forceinline__ int graph_class(long long n, long long m, int algo, int cluster_log2,
                                           long long share)
{
    if (algo != 0) return size_bucket(m) > cluster_log2 ? 2 : 0;
    return n > (long long)kPeelCtas * peel::kLocalSlots ? 3
           : n > peel::kLocalSlots                      ? 2
                                                        : (n > kTinyVertices || straggles(m, share) ? 1 : 0);
}

// Lists the graphs by class and decreasing arc-count bucket (one CTA) and
// records where classes 3, 2 and 1 end in the list (bucket b holds arc counts
// in [2^(b-1), 2^b)).
__global__ void __launch_bounds__(1024)
    schedule_kernel(const long long *vtx_off, const long long *arc_off, int G, int *order, Ctrl *ctl,
                    int algo, int cluster_log2, long long share)
{
    __shared__ unsigned cnt[4 * kBuckets];
    __shared__ unsigned start[4 * kBuckets];
    if (threadIdx.x < 4 * kBuckets) cnt[threadIdx.x] = 0;
    __syncthreads();
    auto key = [&](int g) {
        const long long n = vtx_off[g + 1] - vtx_off[g], m = arc_off[g + 1] - arc_off[g];
        return graph_class(n, m, algo, cluster_log2, share) * kBuckets + size_bucket(m);
    };
    for (int g = threadIdx.x; g < G; g += blockDim.x) atomicAdd(&cnt[key(g)], 1u);
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned run = 0;
        for (int b = 4 * kBuckets - 1; b >= 0; --b) {
            start[b] = run;
            run += cnt[b];
            if (b == 3 * kBuckets) ctl->live.w[B_NHUGE] = run;
            if (b == 2 * kBuckets) ctl->live.w[B_NLARGE] = run;
            if (b == kBuckets) ctl->live.w[B_NMIDDLE] = run;
        }
    }
    __syncthreads();
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        const unsigned pos = atomicAdd(&start[key(g)], 1u);
        order[pos] = g;
    }
}

// Solves graph g of the batch in domain `dom`, with its state in global memory.
template <int Algo, typename Dom>
__device__ __forceinline__ void solve_graph(const BatchParams &bp, int g, Dom &dom, unsigned *s_tmp,
                                            unsigned long long *st, PhaseClock &clk,
                                            unsigned long long &arcs, unsigned long long &atomics,
                                            unsigned long long &slots, unsigned long long &pulled,
                                            unsigned long long &extra)
{
    const long long v0 = bp.vtx_off[g], n = bp.vtx_off[g + 1] - v0;
    const long long a0 = bp.arc_off[g], m = bp.arc_off[g + 1] - a0;
    if (n <= 0) return;
    dom.reset();
    int2 *chunks = bp.chunks + (a0 / 16 + 2ll * g);
    const unsigned chunk_cap = (unsigned)(m / 16 + 2);
    if (Algo == 0) {
        peel::Params<int> p{bp.rp + v0 + g, bp.ci + a0,    n,      bp.core + v0,
                            bp.res0 + v0,   bp.res1 + v0,  bp.qs + v0, chunks,
                            chunk_cap,      bp.ctl,        bp.tn};
        peel::run<int, Dom, kPeelRepair, true>(p, dom, s_tmp, st, clk, arcs, atomics, extra);
        if (dom.leader()) arcs += (unsigned long long)m;   // every row is expanded once
    } else {
        histo::Params<int> p;
        p.rp = bp.rp + v0 + g;
        p.ci = bp.ci + a0;
        p.n = n;
        p.m = m;
        p.core = bp.core + v0;
        p.vinfo = bp.vinfo + v0;
        p.mv[0] = bp.mv[0] + v0;
        p.mv[1] = bp.mv[1] + v0;
        p.histo = bp.histo + a0;
        p.tl[0] = bp.lists[0] + v0;
        p.wl[0] = bp.lists[1] + v0;
        p.bl[0] = bp.lists[2] + v0;
        p.tl[1] = bp.lists[3] + v0;
        p.wl[1] = bp.lists[4] + v0;
        p.bl[1] = bp.lists[5] + v0;
        p.us = bp.us + v0;
        p.ub = chunks;
        p.ib = bp.ichunks + (a0 / 16 + 2ll * g);
        p.ub_cap = chunk_cap;
        p.ctl = bp.ctl;
        p.zero_histo = true;
        p.tn = bp.tn;
        histo::run(p, dom, s_tmp, st, clk, arcs, atomics, slots, pulled);
    }
}

// The CTA's next graph: a place in the schedule from `first` up to `end`, or -1
// when there is none left or the call has failed. One thread decides for all: an
// error that another CTA records meanwhile would otherwise send some warps out of
// the loop and leave the others waiting for them.
__device__ __forceinline__ int next_ticket(const BatchParams &bp, int word, int first, int end,
                                           int *s_ticket)
{
    if (threadIdx.x == 0) {
        const int t = first + (int)atomicAdd(&bp.ctl->live.w[word], 1u);
        *s_ticket = (t < end && status_of(bp.ctl) == 0) ? t : -1;
    }
    __syncthreads();
    const int t = *s_ticket;
    __syncthreads();
    return t;
}

// HistoCore.
template <int Threads>
__global__ void __launch_bounds__(Threads, 512 / Threads * 2)
    batched_histo_kernel(BatchParams bp, LastResult *last)
{
    namespace cg = cooperative_groups;
    __shared__ __align__(16) unsigned s_live[kLiveWords];   // 64-bit counters need 8-byte alignment
    __shared__ unsigned s_snap[kLiveWords + 1];
    __shared__ unsigned s_tmp[256];
    __shared__ unsigned long long s_red[32];
    __shared__ unsigned long long st[kStCount];
    __shared__ int s_ticket;
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    __syncthreads();
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned crank = cluster.block_rank(), csize = cluster.num_blocks();
    PhaseClock clk;
    unsigned long long arcs = 0, atomics = 0, slots = 0, pulled = 0, extra = 0;

    // phase 1: large graphs, one cluster per graph
    const int nlarge = (int)ld_relaxed(&bp.ctl->live.w[B_NLARGE]);
    {
        ClusterDom dom{bp.ctl, s_live, cluster.map_shared_rank(s_live, 0), s_snap, crank, csize,
                       0u};
        int *ticket0 = cluster.map_shared_rank(&s_ticket, 0);
        for (;;) {
            if (crank == 0 && threadIdx.x == 0) {
                const int t = (int)atomicAdd(&bp.ctl->live.w[B_LARGE], 1u);
                s_ticket = (t < nlarge && status_of(bp.ctl) == 0) ? t : -1;
            }
            cluster.sync();
            const int t = *ticket0;
            cluster.sync();
            if (t < 0) break;
            solve_graph<1>(bp, bp.order[t], dom, s_tmp, st, clk, arcs, atomics, slots, pulled, extra);
        }
    }
    // phase 2: the other graphs, one CTA per graph
    {
        CtaDom dom{bp.ctl, s_live, s_snap, 0u};
        for (;;) {
            const int t = next_ticket(bp, B_SMALL, nlarge, bp.G, &s_ticket);
            if (t < 0) break;
            solve_graph<1>(bp, bp.order[t], dom, s_tmp, st, clk, arcs, atomics, slots, pulled, extra);
            __syncthreads();
        }
    }
    block_sum_to(arcs, &bp.ctl->stats[kStArcs], s_red);
    block_sum_to(atomics, &bp.ctl->stats[kStAtomics], s_red);
    block_sum_to(slots, &bp.ctl->stats[kStSlots], s_red);
    block_sum_to(pulled, &bp.ctl->stats[kStPulled], s_red);
    finish_block(bp.ctl, last, 1, st, kStCount);
    cluster.sync();   // no CTA leaves while another may still read its shared memory
}

__device__ __forceinline__ peel::LocalParams<int> local_params(const BatchParams &bp, int g)
{
    const long long v0 = bp.vtx_off[g], a0 = bp.arc_off[g];
    return {bp.rp + v0 + g, bp.ci + a0,  (int)(bp.vtx_off[g + 1] - v0), bp.arc_off[g + 1] - a0,
            bp.core + v0,   bp.qs + v0, bp.ctl};
}

// PeelOne, huge graphs: one cluster per graph. Bound by the latency of L2 atomics
// and of the cluster barriers; 8 CTAs of 512 threads, two to an SM, keep twice the
// warps that 4 CTAs of 1,024 have, and leave room for a second graph beside them
// (one R-MAT graph of 2^20 vertices and 31 M arcs: 35 ms with those, 15.7 ms so; 24 of them
// and 488 smaller graphs: 41.8 and 25.6 ms).
// Its reads of residual degrees hit in L1, so it prefers all of an SM's memory as L1.
// Without that preference it starts on the SMs that another stream's wide CTAs
// have left with 28 KB of L1, and takes 43 ms instead of 21 (two or four streams of
// such batches: 35.7 ms a batch, 22.4 with it, 25.4 with one kernel for all classes; 21.5
// since the tickets below).
__global__ void __launch_bounds__(512, 2) batched_huge_kernel(BatchParams bp)
{
    namespace cg = cooperative_groups;
    // the next launch may start: it shares nothing with this one
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ __align__(16) unsigned s_live[kLiveWords];
    __shared__ unsigned s_snap[kLiveWords + 1];
    __shared__ unsigned s_tmp[256];
    __shared__ unsigned long long s_red[32];
    __shared__ unsigned long long st[kStCount];
    __shared__ int s_ticket;
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    __syncthreads();
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned crank = cluster.block_rank(), csize = cluster.num_blocks();
    PhaseClock clk;
    unsigned long long arcs = 0, atomics = 0, slots = 0, pulled = 0, extra = 0;
    const int nhuge = (int)ld_relaxed(&bp.ctl->live.w[B_NHUGE]);
    ClusterDom dom{bp.ctl, s_live, cluster.map_shared_rank(s_live, 0), s_snap, crank, csize, 0u};
    int *ticket0 = cluster.map_shared_rank(&s_ticket, 0);
    // The first tickets are dealt out in the clusters' order: there are often more
    // clusters than graphs, and the first ones, placed before SMs take a second
    // CTA, have SMs of their own (4 such graphs and 60 smaller ones: 16.1 ms, 18.8-19.6
    // when whichever clusters came first shared SMs).
    const int ncluster = (int)(gridDim.x / csize);
    for (int round = 0;; ++round) {
        if (crank == 0 && threadIdx.x == 0) {
            const int t = round == 0 ? (int)(blockIdx.x / csize)
                                     : ncluster + (int)atomicAdd(&bp.ctl->live.w[B_HUGE], 1u);
            s_ticket = (t < nhuge && status_of(bp.ctl) == 0) ? t : -1;
        }
        cluster.sync();
        const int t = *ticket0;
        cluster.sync();
        if (t < 0) break;
        solve_graph<0>(bp, bp.order[t], dom, s_tmp, st, clk, arcs, atomics, slots, pulled, extra);
    }
    block_sum_to(arcs, &bp.ctl->stats[kStArcs], s_red);
    block_sum_to(atomics, &bp.ctl->stats[kStAtomics], s_red);
    fold_block(bp.ctl, st);
    cluster.sync();   // no CTA leaves while another may still read its shared memory
}

// PeelOne, large and middle graphs (and tiny ones that straggle).
__global__ void __launch_bounds__(kWideThreads, 1) batched_peel_kernel(BatchParams bp)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) char smem[];
    __shared__ unsigned long long st[kStCount];
    __shared__ int s_ticket;
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    __syncthreads();
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned crank = cluster.block_rank();
    const int nhuge = (int)ld_relaxed(&bp.ctl->live.w[B_NHUGE]);
    const int nlarge = (int)ld_relaxed(&bp.ctl->live.w[B_NLARGE]);
    const int nmiddle = (int)ld_relaxed(&bp.ctl->live.w[B_NMIDDLE]);
    {   // large graphs, one cluster per graph
        int *ticket0 = cluster.map_shared_rank(&s_ticket, 0);
        for (;;) {
            if (crank == 0 && threadIdx.x == 0) {
                const int t = nhuge + (int)atomicAdd(&bp.ctl->live.w[B_LARGE], 1u);
                s_ticket = (t < nlarge && status_of(bp.ctl) == 0) ? t : -1;
            }
            cluster.sync();
            const int t = *ticket0;
            cluster.sync();
            if (t < 0) break;
            const peel::LocalParams<int> p = local_params(bp, bp.order[t]);
            const peel::LocalStats s =
                peel::run_local<int, peel::LocalWide, true>(p, smem, crank, kPeelCtas);
            if (crank == 0 && threadIdx.x == 0) peel::add_stats(st, s, p.n, p.m);
        }
    }
    for (;;) {   // middle graphs, one CTA per graph
        const int t = next_ticket(bp, B_SMALL, nlarge, nmiddle, &s_ticket);
        if (t < 0) break;
        const peel::LocalParams<int> p = local_params(bp, bp.order[t]);
        const bool rows = peel::local_smem_bytes<peel::LocalWide>(p.n, peel::kKeepRows) <=
                          peel::kLocalSmem;
        const peel::LocalStats s =
            rows ? peel::run_local<int, peel::LocalWide, false, peel::kKeepRows>(p, smem, 0, 1)
                 : peel::run_local<int, peel::LocalWide, false>(p, smem, 0, 1);
        if (threadIdx.x == 0) peel::add_stats(st, s, p.n, p.m);
        __syncthreads();
    }
    fold_block(bp.ctl, st);
    cluster.sync();   // no CTA leaves while another may still read its shared memory
    // this launch ends after the one before it, so that what follows waits for
    // both; one CTA waits, the others give their SMs to other streams
    if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// PeelOne, tiny graphs; the last launch of a batch, which publishes its status and
// statistics.
__global__ void __launch_bounds__(kTinyThreads, 8) batched_tiny_kernel(BatchParams bp, LastResult *last)
{
    extern __shared__ __align__(16) char smem[];
    __shared__ unsigned long long st[kStCount];
    __shared__ int s_ticket;
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    __syncthreads();
    const int nmiddle = (int)ld_relaxed(&bp.ctl->live.w[B_NMIDDLE]);
    for (;;) {
        const int t = next_ticket(bp, B_TINY, nmiddle, bp.G, &s_ticket);
        if (t < 0) break;
        const peel::LocalParams<int> p = local_params(bp, bp.order[t]);
        if (p.n <= 0) continue;
        const bool whole = peel::local_smem_bytes<peel::LocalTiny>(p.n, peel::kKeepGraph, p.m) <=
                           kTinySmem;
        const peel::LocalStats s =
            whole ? peel::run_local<int, peel::LocalTiny, false, peel::kKeepGraph>(p, smem, 0, 1)
                  : peel::run_local<int, peel::LocalTiny, false, peel::kKeepRows>(p, smem, 0, 1);
        if (threadIdx.x == 0) peel::add_stats(st, s, p.n, p.m);
        __syncthreads();
    }
    fold_kmax(bp.ctl, st);
    finish_block(bp.ctl, last, PICO_ALGO_PEELONE, st, kStCount);
}

// Launches a kernel over a persistent grid of clusters: every cluster that is
// resident at once, but no more than `need`. occ: the kernel's cached number
// of resident clusters (0: not known yet). beside: the launch may run beside the
// one before it on the stream. carveout: percent of an SM's shared memory the kernel
// prefers (-1: no preference).
cudaError_t launch_clusters(const void *fn, int cluster, int threads, size_t smem, int sms,
                            long long need, int &occ, void **args, cudaStream_t stream,
                            bool beside = false, int carveout = -1)
{
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    lc.attrs = attr;
    lc.numAttrs = 1;
    if (occ == 0) {
        if (smem > 0) {
            const cudaError_t e =
                cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        if (carveout >= 0) {
            const cudaError_t e =
                cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, carveout);
            if (e != cudaSuccess) return e;
        }
        lc.gridDim = dim3(cluster * sms);
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&occ, fn, &lc);
        if (e != cudaSuccess) return e;
        if (occ <= 0) return cudaErrorLaunchOutOfResources;
    }
    lc.gridDim = dim3(cluster * (unsigned)std::min<long long>(need, occ));
    if (beside) {
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        lc.numAttrs = 2;
    }
    return cudaLaunchKernelExC(&lc, fn, args);
}

}  // namespace

size_t batched_ws_bytes(int G, long long total_n, long long total_m, int algo)
{
    Carver c(nullptr);
    c.take<Ctrl>(1);
    c.take<int>(G);
    const size_t nchunks = (size_t)(total_m / 16 + 2ll * G + 2);
    if (algo == 0) {
        for (int i = 0; i < 3; ++i) c.take<int>(total_n);
    } else {
        c.take<int2>(total_n);  // vinfo
        c.take<int2>(total_n);  // mv[0]
        c.take<int2>(total_n);  // mv[1]
        c.take<int>(total_m);   // histo
        for (int i = 0; i < 7; ++i) c.take<int>(total_n);
        c.take<int2>(nchunks);  // chunk lists of every large vertex
    }
    c.take<int2>(nchunks);
    return c.size();
}

int launch_batched(const int64_t *vtx_off, const int64_t *arc_off, int G, const int32_t *rp,
                   const int32_t *ci, long long total_n, long long total_m, int32_t *core,
                   int algo, void *ws, LastResult *last, cudaStream_t stream, const LaunchCfg &cfg)
{
    Carver c(ws);
    BatchParams bp{};
    bp.vtx_off = reinterpret_cast<const long long *>(vtx_off);
    bp.arc_off = reinterpret_cast<const long long *>(arc_off);
    bp.G = G;
    bp.rp = rp;
    bp.ci = ci;
    bp.core = core;
    bp.ctl = c.take<Ctrl>(1);
    bp.order = c.take<int>(G);
    if (algo == 0) {
        bp.res0 = c.take<int>(total_n);
        bp.res1 = c.take<int>(total_n);
        bp.qs = c.take<int>(total_n);
    } else {
        bp.vinfo = c.take<int2>(total_n);
        bp.mv[0] = c.take<int2>(total_n);
        bp.mv[1] = c.take<int2>(total_n);
        bp.histo = c.take<int>(total_m);
        for (int i = 0; i < 6; ++i) bp.lists[i] = c.take<int>(total_n);
        bp.us = c.take<int>(total_n);
        bp.ichunks = c.take<int2>((size_t)(total_m / 16 + 2ll * G + 2));
    }
    bp.chunks = c.take<int2>((size_t)(total_m / 16 + 2ll * G + 2));
    bp.tn = cfg.tn;
    if (cudaMemsetAsync(bp.ctl, 0, sizeof(Ctrl), stream) != cudaSuccess) return -3;
    schedule_kernel<<<1, 1024, 0, stream>>>(bp.vtx_off, bp.arc_off, G, bp.order, bp.ctl, algo,
                                            cfg.tn.cluster_log2, total_m / std::max(1, cfg.sms));
    if (cudaGetLastError() != cudaSuccess) return -3;

    const int dev = cfg.device & 63;
    if (algo == 0) {
        static int occ_huge[64] = {}, occ_wide[64] = {}, occ_tiny[64] = {};
        void *args[] = {&bp, &last};
        // graphs of a class the batch can hold (its grid needs no more clusters)
        const long long huge =
            std::min<long long>(G, total_n / ((long long)kPeelCtas * peel::kLocalSlots + 1));
        if (huge > 0 && launch_clusters((const void *)batched_huge_kernel, kClusterCtas, 512, 0,
                                        cfg.sms, huge, occ_huge[dev], args, stream, false,
                                        cudaSharedmemCarveoutMaxL1) != cudaSuccess)
            return -3;
        const long long wide =
            std::min<long long>(G, total_n / (kTinyVertices + 1) + total_m / (kTinyArcs + 1));
        if (wide > 0 &&
            launch_clusters((const void *)batched_peel_kernel, kPeelCtas, kWideThreads,
                            peel::kLocalSmem, cfg.sms,
                            wide, occ_wide[dev], args, stream, huge > 0) != cudaSuccess)
            return -3;
        if (launch_clusters((const void *)batched_tiny_kernel, 1, kTinyThreads,
                            kTinySmem, cfg.sms * 8, G,
                            occ_tiny[dev], args, stream) != cudaSuccess)
            return -3;
        return 0;
    }
    static int occ[2][64] = {};
    const bool narrow = cfg.batched_threads == 256;
    void *args[] = {&bp, &last};
    const long long need = ((long long)G + kClusterCtas - 1) / kClusterCtas;
    if (launch_clusters(narrow ? (const void *)batched_histo_kernel<256>
                               : (const void *)batched_histo_kernel<512>,
                        kClusterCtas, narrow ? 256 : 512, 0, cfg.sms, need, occ[narrow][dev], args,
                        stream) != cudaSuccess)
        return -3;
    return 0;
}

}  // namespace pico
