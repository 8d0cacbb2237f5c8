// PeelOne (Sec. III, Alg. 4) on one graph as one persistent cooperative
// kernel: the algorithm body is peel::run_async (peelone.cuh) over the whole
// grid, or peel::run (a grid barrier per frontier wave) when asynchronous
// levels are switched off.
#include <algorithm>

#include "peel_local.cuh"
#include "peel_tail.cuh"
#include "peelone.cuh"
#include "pico.h"
#include "pico_launch.h"

namespace pico {
namespace {

// Percent of an SM's shared memory for the kernels that alternate: the same for
// both, so that the SMs are not set up anew between them.
constexpr int kTailCarveout = 50;

// The shared-memory form: threads of its CTA, and half as many for graphs that
// are kept there whole, whose waves are a few rows: idle warps take issue slots
// and the CTA barrier is cheaper (R-MAT scale 10: 124 us with 512, 135 with
// 1,024 threads; a path of 5,000 vertices: 2.34 and 2.67 ms).
constexpr int kLocalThreads = 1024;
// One SM walks about 1.5 arcs per clock, so it loses to the grid where there
// are many arcs and few levels (Erdos-Renyi, n 50,001, m 0.8 M, 9 levels: 504
// against 266 us) and wins on skewed graphs up to this size (R-MAT scale 14, m
// 0.43 M: 545 against 1,503 us; Chung-Lu, n 32,768, m 0.6 M: 794 against 1,229
// us with the cluster kernel and 2,028 us without).
constexpr long long kLocalMaxArcs = 640 << 10;
// Up to here whatever the degrees; beyond it a graph without skew has waves wide
// enough for the grid, which then looks at the degrees first and keeps such a graph
// (Erdos-Renyi, one CTA against the grid: n 10,000, mean degree 8: 166 and 218 us, 40:
// 329 and 338 us; n 15,000: 190 and 222, 386 and 361 us; n 20,000, degree 8: 220 and
// 226 us; 30,000: 292 and 234; 51,000: 438 and 228 us. With skew, R-MAT of 51,000
// vertices: 814 and 1,317 us; grids of 51,000 vertices: 888 and 1,083 us).
constexpr long long kLocalAnyVertices = 20480, kLocalAnyArcs = 400 << 10;   // both, ...
constexpr long long kLocalFewVertices = 12288;                              // ... or this few

// kTail: one of the launches that alternate with the cluster kernel. The one
// that ends the run publishes the status and the statistics (the `final` one
// ends it in any case); the launches after it return at once.
template <typename Off, int Mode, bool kAsync, bool kTail>
__global__ void __launch_bounds__(kThreads, 2)
    peelone_kernel(peel::Params<Off> p, LastResult *last, unsigned long long limit_ns,
                   long long m, int turn, bool final, bool local)
{
    __shared__ unsigned s_snap[kLiveWords + 1];
    __shared__ unsigned s_tmp[128];
    __shared__ unsigned long long s_red[32];
    __shared__ unsigned long long st[kStCount];   // statistics, written by thread 0
    if (kTail && p.tail->published) return;   // the same in every CTA
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long arcs = 0, atomics = 0, extra = 0;
    PhaseClock clk;
    if (blockIdx.x == 0 && threadIdx.x == 0 && last->trace_on) {
        if (!kTail || p.tail->mode == peel::kTailFresh) last->trace_len = 0;
        clk.trace = last->trace;
        clk.trace_len = &last->trace_len;
    }
    clk.start();
    GridDom dom{p.ctl, s_snap, limit_ns};
    bool over = true;
    if (kAsync)
        over = peel::run_async<Off, Mode, kTail>(p, dom, s_tmp, st, clk, arcs, atomics, extra, final,
                                                 local);
    else
        peel::run<Off, GridDom, Mode>(p, dom, s_tmp, st, clk, arcs, atomics, extra);
    if (kTail) {   // every row is expanded once, by one kernel or the other
        if (over && threadIdx.x == 0) st[kStArcs] = (unsigned long long)m;
    } else {
        block_sum_to(arcs, &p.ctl->stats[kStArcs], s_red);
    }
    block_sum_to(atomics, &p.ctl->stats[kStAtomics], s_red);
    block_sum_to(extra, &p.ctl->stats[kStExtra], s_red);
    if (blockIdx.x != 0 && threadIdx.x < kStCount) st[threadIdx.x] = 0;
    if (!over) {
        fold_block(p.ctl, st);
        return;
    }
    if (kTail) fold_kmax(p.ctl, st);
    const bool published = finish_block(
        p.ctl, last,
        Mode == kPeelRepair ? PICO_ALGO_PEELONE
                            : (Mode == kPeelCas ? PICO_ALGO_PEEL_CAS : PICO_ALGO_PEEL_ADDBACK),
        st, kStCount, turn);
    if (kTail && published) p.tail->published = 1;
}

// The light levels of a graph on one cluster, between two launches of the grid
// kernel (peel_tail.cuh).
template <typename Off>
__global__ void __launch_bounds__(peel::kTailThreads, 1)
    peelone_tail_kernel(peel::Params<Off> p, LastResult *last, long long m, int turn,
                        unsigned budget)
{
    extern __shared__ __align__(16) char smem[];
    __shared__ unsigned long long st[kStCount];
    __shared__ unsigned long long s_red[32];
    // nothing to do (the same in every CTA)
    if (p.tail->published) return;
    const bool failed = status_of(p.ctl) != 0;
    const bool final = budget == peel::kTailNoBudget;   // the run's last launch
    if (!final && (p.tail->mode != peel::kTailScan || failed)) return;
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    PhaseClock clk;
    if (blockIdx.x == 0 && threadIdx.x == 0 && last->trace_on) {
        clk.trace = last->trace;
        clk.trace_len = &last->trace_len;
    }
    __syncthreads();
    clk.start();
    peel::TailPeel<Off> tp{p, p.tail, *reinterpret_cast<peel::TailShared *>(smem), blockIdx.x,
                            budget};
    const bool over = failed || tp.run(st);
    if (over && blockIdx.x == 0 && threadIdx.x == 0) st[kStArcs] = (unsigned long long)m;
    clk.end(st, kPhWaveMid, (unsigned)st[kStLevels]);
    block_sum_to(tp.n_lowered, &p.ctl->stats[kStAtomics], s_red);
    if (over) {   // only CTA 0 counts levels and scans
        fold_kmax(p.ctl, st);
        if (finish_block(p.ctl, last, PICO_ALGO_PEELONE, st, kStCount, turn)) p.tail->published = 1;
    } else {
        fold_block(p.ctl, st);
    }
    cooperative_groups::this_cluster().sync();   // no CTA leaves while another may write to it
}

// A graph whose residual degrees fit the shared memory of one CTA
// (peel_local.cuh). tail: another launch may have solved it already (nullptr:
// none has).
template <typename Off, int kKept>
__global__ void __launch_bounds__(kLocalThreads, 1)
    peelone_local_kernel(peel::LocalParams<Off> p, const peel::TailState *tail, LastResult *last,
                         int turn)
{
    extern __shared__ __align__(16) char smem[];
    __shared__ unsigned long long st[kStCount];
    if (tail && tail->published) return;
    if (threadIdx.x < kStCount) st[threadIdx.x] = 0;
    PhaseClock clk;
    if (threadIdx.x == 0 && last->trace_on) {
        last->trace_len = 0;
        clk.trace = last->trace;
        clk.trace_len = &last->trace_len;
    }
    __syncthreads();
    clk.start();
    const peel::LocalStats s = peel::run_local<Off, peel::LocalWide, false, kKept>(p, smem, 0, 1);
    if (threadIdx.x == 0) peel::add_stats(st, s, p.n, p.m);
    clk.end(st, kPhWaveMid, (unsigned)s.waves);
    finish_block(p.ctl, last, PICO_ALGO_PEELONE, st, kStCount, turn);
}

// Sets a kernel's dynamic shared memory limit (and non-portable cluster size)
// once per device.
bool prepare_kernel(const void *fn, size_t smem, bool wide_cluster, bool &ready)
{
    if (ready) return true;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return false;
    if (wide_cluster &&
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return false;
    ready = true;
    return true;
}

template <typename Off>
cudaError_t launch_tail(peel::Params<Off> &p, long long m, LastResult *last, cudaStream_t stream,
                        int device, int turn, unsigned budget)
{
    static bool ready[64] = {};
    const void *fn = (const void *)peelone_tail_kernel<Off>;
    constexpr size_t smem = sizeof(peel::TailShared);
    if (!ready[device & 63] &&
        cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, kTailCarveout) !=
            cudaSuccess)
        return cudaErrorInvalidValue;
    if (!prepare_kernel(fn, smem, true, ready[device & 63])) return cudaErrorInvalidValue;
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = peel::kTailCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.gridDim = dim3(peel::kTailCtas);
    lc.blockDim = dim3(peel::kTailThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    lc.attrs = attr;
    lc.numAttrs = 1;
    void *args[] = {&p, &last, &m, &turn, &budget};
    return cudaLaunchKernelExC(&lc, fn, args);
}

// Launches that follow the grid kernel's first: cluster and grid kernel in turn. One
// with nothing to do takes 3.3 us, so small graphs get few. The cluster walks 7 G
// arcs/s, a fifth of what the grid does; the grid takes 17 us for a light level, the
// cluster 6. So what the last launches are left with decides:
//   below 6 Mi arcs one launch, on the cluster, which walks whatever is left. R-MAT
//   scale 16: 1.36 ms, 1.39 with a launch of the grid behind it; at worst, 5.6 M arcs
//   behind one heavy level, 0.96 ms (0.84 with it; one grid kernel 0.51).
//   below 20 Mi four; the second of the cluster keeps waves of up to 1 M arcs. R-MAT
//   scale 18, 19 and scale 20 with edge factor 8: 2.57, 3.20, 3.20 ms, with waves of
//   128 K 2.52, 3.15, 4.36, with three launches 2.57, 3.38, 3.31; 18 M arcs behind two
//   heavy levels 1.30 ms, with three launches 2.66 (one grid kernel 1.17).
//   then six, from 120 Mi twelve: R-MAT scale 20 takes 4.75 ms with six, 5.95 with four.
constexpr int kMostLaunches = 12;
static_assert(kMostLaunches + 1 < kMaxTurns, "every launch counts its CTAs in a word of its own");
constexpr long long kFourLaunches = 20ll << 20;
int tail_launches(long long m)
{
    return m < peel::kTailMaxGraph ? 1 : m < kFourLaunches ? 4 : m < (120 << 20) ? 6 : kMostLaunches;
}

// Arcs of a wave that the cluster kernel's launch i walks at most.
unsigned tail_budget(long long m, int i)
{
    if (m < peel::kTailMaxGraph) return peel::kTailNoBudget;
    return m < kFourLaunches && i == 3 ? peel::kTailLateBudget : peel::kTailBudget;
}

// Reads a range (16 bytes a thread per step); the values are not used.
__global__ void __launch_bounds__(256) touch_kernel(const int4 *p, size_t count, int *sink)
{
    int acc = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (size_t)gridDim.x * blockDim.x) {
        const int4 v = __ldcg(p + i);
        acc ^= v.x ^ v.y ^ v.z ^ v.w;
    }
    if (acc == 0x7fffffff && sink) *sink = acc;   // keeps the loads
}

}  // namespace

cudaError_t l2_release(const void *p, size_t bytes, cudaStream_t stream)
{
    const size_t count = bytes / sizeof(int4);
    if (!p || count == 0) return cudaSuccess;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)std::min<size_t>((count + 255) / 256, 1024));
    lc.blockDim = dim3(256);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[0].val.accessPolicyWindow.base_ptr = const_cast<void *>(p);
    attr[0].val.accessPolicyWindow.num_bytes = count * sizeof(int4);
    attr[0].val.accessPolicyWindow.hitRatio = 1.0f;
    attr[0].val.accessPolicyWindow.hitProp = cudaAccessPropertyNormal;
    attr[0].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    lc.attrs = attr;
    lc.numAttrs = 1;
    const int4 *q = static_cast<const int4 *>(p);
    int *sink = nullptr;
    void *args[] = {&q, (void *)&count, &sink};
    return cudaLaunchKernelExC(&lc, (const void *)touch_kernel, args);
}

size_t chunk_capacity(long long m) { return peel::chunk_list_capacity(m); }

size_t peelone_ws_bytes(long long n, long long m, bool async)
{
    Carver c(nullptr);
    peel::Params<int> p;
    peel::carve(p, c, n, m, async);
    return c.size();
}

namespace {

// Whether a graph of this size is peeled in one CTA's shared memory instead of by the
// grid kernel: whatever its degrees, or if they call for it (peel::local_degrees,
// known on the device).
bool peelone_local(long long n, long long m, bool any_degrees)
{
    if (n > peel::kLocalSlots || m > kLocalMaxArcs) return false;
    return !any_degrees || n <= kLocalFewVertices || (n <= kLocalAnyVertices && m <= kLocalAnyArcs);
}

// The shared-memory form. tail: the launch does nothing when *tail says that an
// earlier one has published the call (nullptr: there is none).
template <typename Off>
int launch_local(const peel::Params<Off> &p, long long m, const peel::TailState *tail,
                 LastResult *last, cudaStream_t stream, const LaunchCfg &cfg, int turn)
{
    static bool ready[3][64] = {};
    const void *fns[3] = {(const void *)peelone_local_kernel<Off, peel::kKeepNone>,
                          (const void *)peelone_local_kernel<Off, peel::kKeepRows>,
                          (const void *)peelone_local_kernel<Off, peel::kKeepGraph>};
    const int kept = peel::local_kept<peel::LocalWide>(p.n, m, peel::kLocalSmem);
    const void *fn = fns[kept];
    if (!prepare_kernel(fn, peel::kLocalSmem, false, ready[kept][cfg.device & 63])) return -3;
    peel::LocalParams<Off> lp{p.rp, p.ci, (int)p.n, m, p.core, p.qs, p.ctl};
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(1);
    lc.blockDim = dim3(kept == peel::kKeepGraph ? kLocalThreads / 2 : kLocalThreads);
    lc.dynamicSmemBytes = peel::local_smem_bytes<peel::LocalWide>(p.n, kept, m);
    lc.stream = stream;
    void *args[] = {&lp, &tail, &last, &turn};
    return cudaLaunchKernelExC(&lc, fn, args) == cudaSuccess ? 0 : -3;
}

template <typename Off>
const void *grid_kernel(int mode, bool async)
{
    const void *fns[2][3] = {{(const void *)peelone_kernel<Off, kPeelRepair, false, false>,
                              (const void *)peelone_kernel<Off, kPeelCas, false, false>,
                              (const void *)peelone_kernel<Off, kPeelAddBack, false, false>},
                             {(const void *)peelone_kernel<Off, kPeelRepair, true, true>,
                              (const void *)peelone_kernel<Off, kPeelCas, true, false>,
                              (const void *)peelone_kernel<Off, kPeelAddBack, true, false>}};
    return fns[async][mode];
}

// CTAs of the grid kernel, which is prepared by the first call on a device; 0: error.
template <typename Off>
int grid_ctas(int mode, bool async, const LaunchCfg &cfg)
{
    static int occ[2][3][64] = {};
    const void *fn = grid_kernel<Off>(mode, async);
    int &o = occ[async][mode][cfg.device & 63];
    if (o == 0) {
        if (async && mode == kPeelRepair &&
            cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, kTailCarveout) !=
                cudaSuccess)
            return 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, kThreads, 0) != cudaSuccess ||
            o <= 0)
            return 0;
    }
    return cfg.sms * (o < cfg.max_blocks_per_sm ? o : cfg.max_blocks_per_sm);
}

// The launches of one run, p carved and its control block zeroed; `turn` is the
// first one's place among the launches of the call. Behind another launch (turn > 0)
// asynchronous PeelOne does nothing when that one has published the call.
template <typename Off>
int launch_run(peel::Params<Off> &p, long long m, LastResult *last, cudaStream_t stream,
               const LaunchCfg &cfg, int mode, bool async, int turn)
{
    const bool tail = async && mode == kPeelRepair;
    if (tail && peelone_local(p.n, m, true))
        return launch_local(p, m, turn > 0 ? p.tail : nullptr, last, stream, cfg, turn);
    const int ctas = grid_ctas<Off>(mode, async, cfg);
    if (ctas == 0) return -3;
    unsigned long long limit = cfg.limit_ns;
    bool local = tail && peelone_local(p.n, m, false);   // this launch or one CTA, by the degrees
    const int launches = tail && !local ? tail_launches(m) : 0;   // ... and those that take turns
    // the residual degrees (the target of every decrement) stay in L2
    const size_t win = async ? std::min<size_t>((size_t)p.n * sizeof(int), cfg.l2_window) : 0;
    for (int i = 0; i <= launches; ++i, ++turn) {
        bool final = i == launches;
        bool by_degrees = local && i == 0;
        void *args[] = {&p, &last, &limit, &m, &turn, &final, &by_degrees};
        const cudaError_t e =
            i % 2 == 1 ? launch_tail(p, m, last, stream, cfg.device, turn, tail_budget(m, i))
                       : launch_cooperative(grid_kernel<Off>(mode, async), dim3(ctas), dim3(kThreads),
                                            args, 0, stream, p.work, win);
        if (e != cudaSuccess) return -3;
    }
    if (local && launch_local(p, m, p.tail, last, stream, cfg, turn) != 0) return -3;
    if (win > 0 && l2_release(p.work, win, stream) != cudaSuccess) return -3;
    return 0;
}

}  // namespace

template <typename Off>
bool peelone_async(const LaunchCfg &cfg)
{
    // beyond that the level-end flags have no room
    return cfg.peel_async && grid_ctas<Off>(kPeelRepair, true, cfg) <= peel::kMaxAsyncCtas;
}

template <typename Off>
int launch_peel_after(peel::Params<Off> &p, long long m, LastResult *last, cudaStream_t stream,
                      const LaunchCfg &cfg)
{
    return launch_run(p, m, last, stream, cfg, kPeelRepair, true, 1);
}

template <typename Off>
int launch_peelone(const Off *rp, const int *ci, long long n, long long m, int *core, void *ws,
                   LastResult *last, cudaStream_t stream, const LaunchCfg &cfg, int mode)
{
    if (mode < kPeelRepair || mode > kPeelAddBack) return -1;
    const bool async =
        cfg.peel_async && grid_ctas<Off>(mode, true, cfg) <= peel::kMaxAsyncCtas;
    Carver c(ws);
    peel::Params<Off> p;
    peel::carve(p, c, n, m, async);
    p.rp = rp;
    p.ci = ci;
    p.core = core;
    p.tn = cfg.tn;
    if (cudaMemsetAsync(p.ctl, 0, sizeof(Ctrl), stream) != cudaSuccess) return -3;
    return launch_run(p, m, last, stream, cfg, mode, async, 0);
}

template bool peelone_async<int>(const LaunchCfg &);
template bool peelone_async<long long>(const LaunchCfg &);
template int launch_peel_after<int>(peel::Params<int> &, long long, LastResult *, cudaStream_t,
                                    const LaunchCfg &);
template int launch_peel_after<long long>(peel::Params<long long> &, long long, LastResult *,
                                          cudaStream_t, const LaunchCfg &);
template int launch_peelone<int>(const int *, const int *, long long, long long, int *, void *,
                                 LastResult *, cudaStream_t, const LaunchCfg &, int);
template int launch_peelone<long long>(const long long *, const int *, long long, long long,
                                       int *, void *, LastResult *, cudaStream_t,
                                       const LaunchCfg &, int);

}  // namespace pico
