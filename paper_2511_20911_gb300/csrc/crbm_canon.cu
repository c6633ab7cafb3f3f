// SMEM-resident sweep, canonical SS fast path: a CTA holds one packed word
// (32 chains) -- the whole even, periodic lattice, its hidden layer and the
// lane-expanded tables -- in shared memory and runs a chunk of sweeps on it.
// The sweep body is in crbm_canon_body.cuh, the per-cell cores in
// crbm_row_core.cuh.
#include <algorithm>

#include "crbm_canon_body.cuh"
#include "crbm_launch.h"

#ifndef CRBM_SWEEP_MIN_BLOCKS
#define CRBM_SWEEP_MIN_BLOCKS (CRBM_SWEEP_MAX_THREADS <= 512 ? 2 : 1)  // 64 registers a thread either way
#endif

namespace crbm {
namespace {

using namespace dev;
using namespace canon;

// Persistent form: a grid that fits on the GPU at once works through items
// (word, chunk of `chunk` sweeps).  Chunks of a word run in order, one CTA at
// a time.  state[w] = 2 (chunks of w done) + (1 while a CTA holds w).  A CTA
// claims, with a compare-and-swap on state, the free word with the fewest
// chunks done (warp 0 scans all states with 16-byte loads; ties go to the
// first word in a CTA-dependent scan order), runs its next chunk, publishes
// the word's spins and sums, then releases it with the new count and claims
// again.  A CTA that finds no free unfinished word exits: every unfinished
// word is then held by a running CTA, which claims again after its chunk, so
// no work is left behind and nothing waits.  A launch with a CTA for every word
// has no states (nullptr) and one item per CTA.
//
// Three instantiations per variant: kCtaWide, CTAs of at most 512 threads alone
// on their SM, which may take 128 registers a thread (ladders of the L=18
// lattice, 96 words in CTAs of 16 warps: 4.67 us per sweep against 4.88 at 64
// registers); kCtaPair, CTAs of at most 384 threads at two or more per SM, 80
// registers (L=18 grid, 500 sweeps in CTAs of 8 warps: 5.28 ms; 5.41 at 128
// registers); kCtaAny, any CTA at 64 registers.
constexpr int kCtaAny = CRBM_SWEEP_MAX_THREADS, kCtaPair = 384, kCtaWide = 512;
template <int kMode, bool kPaper, int kMaxThreads>
__global__ void __launch_bounds__(kMaxThreads, kMaxThreads == kCtaPair ? 2 : CRBM_SWEEP_MIN_BLOCKS)
    k_sweep_canon_persistent(const SweepArgs a, int chunk, int* state) {
    extern __shared__ __align__(128) uint32_t smem[];  // (no static shared memory: see kReservedSmem)
    int& s_word = reinterpret_cast<int*>(smem + canon_smem(a.g, kMode).seg)[33];
    int& s_chunk = reinterpret_cast<int*>(smem + canon_smem(a.g, kMode).seg)[34];
    const int n_chunks = (a.n_sweeps + chunk - 1) / chunk;
    const int nw = a.n_words, nq = (nw + 3) / 4;
    const int K = a.measure_every;
    const int lane = threadIdx.x & 31;
    const unsigned int start = (blockIdx.x * 97u) % static_cast<unsigned int>(nw);
    for (bool first = true;; first = false) {
        if (state == nullptr) {  // a CTA per word: nothing to schedule
            if (threadIdx.x == 0) {
                s_word = first ? static_cast<int>(blockIdx.x) : -1;
                s_chunk = 0;
            }
        } else if (threadIdx.x < 32) {
            int word = -1, c = 0;
            for (int tries = 0; tries < (1 << 20) && word < 0; ++tries) {
                int best = 0x7fffffff, bk = 0x7fffffff, bw = -1;  // (chunks done, scan rank, word)
                for (int q = lane; q < nq; q += 32) {
                    const int4 v = __ldcg(reinterpret_cast<const int4*>(state) + q);
                    const int sv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int w = 4 * q + j;
                        const int dw = sv[j] >> 1;
                        const int rank = static_cast<int>((static_cast<unsigned int>(w) + nw - start) %
                                                          static_cast<unsigned int>(nw));
                        if (w < nw && (sv[j] & 1) == 0 && dw < n_chunks &&
                            (dw < best || (dw == best && rank < bk))) {
                            best = dw;
                            bk = rank;
                            bw = w;
                        }
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const int ob = __shfl_xor_sync(0xffffffffu, best, o);
                    const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                    const int ow = __shfl_xor_sync(0xffffffffu, bw, o);
                    if (ob < best || (ob == best && ok < bk)) {
                        best = ob;
                        bk = ok;
                        bw = ow;
                    }
                }
                if (bw < 0) break;  // every unfinished word is held by a running CTA
                if (lane == 0 && atomicCAS(state + bw, 2 * best, 2 * best + 1) == 2 * best) {
                    __threadfence();  // acquire: the previous chunk's stores precede its release
                    word = bw;
                    c = best;
                }
                word = __shfl_sync(0xffffffffu, word, 0);
                c = __shfl_sync(0xffffffffu, c, 0);
            }
            if (lane == 0) {
                s_word = word;
                s_chunk = c;
            }
        }
        __syncthreads();
        const int word = s_word, c = s_chunk;
        if (word < 0) break;
        const uint32_t t0 = a.t0 + static_cast<uint32_t>(c * chunk);
        const int n = min(chunk, a.n_sweeps - c * chunk);
        const int64_t meas0 =
            K > 0 ? a.meas0 + static_cast<int64_t>(t0 / K) - static_cast<int64_t>(a.t0 / K) : a.meas0;
        sweep_canon_body<kMode, false, kPaper>(a, word, t0, n, meas0, 0, 0, first);
        __syncthreads();  // every thread's state stores are issued
        if (threadIdx.x == 0 && state != nullptr) {
            __threadfence();
            st_release(state + word, 2 * (c + 1));
        }
    }
}

// Few words: each word's rows of cells split into bands over a cluster of
// a.n_bands CTAs, so that words that would hold an SM each use up to eight.
template <int kMode, bool kPaper>
__global__ void __launch_bounds__(kCtaWide, 1) k_sweep_canon_split(const SweepArgs a) {
    const int nb = a.n_bands, word = static_cast<int>(blockIdx.x) / nb;
    sweep_canon_body<kMode, true, kPaper>(a, word, a.t0, a.n_sweeps, a.meas0, static_cast<int>(blockIdx.x) - word * nb, 0);
}

}  // namespace

cudaError_t check_dynamic_smem_base(const void* kernel, int dev) {
    int reserved = 0;
    cudaFuncAttributes at{};
    cudaError_t e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, kernel);
    if (e == cudaSuccess && !dynamic_smem_at_base(reserved, at.sharedSizeBytes)) e = cudaErrorInvalidConfiguration;
    return e;
}

size_t smem_bytes_canon(const Geometry& g) {
    const size_t words = static_cast<size_t>(kAccWords) + kCanonTab + g.N + static_cast<size_t>(g.n_cells) * 32 + 96 + 33 +
                         32 + 64 + 3;
    return sizeof(uint32_t) * ((words & ~static_cast<size_t>(3)) + (g.paper ? static_cast<size_t>(g.n_cells) * 64 : 0));
}

// The segments' length.  Warp w takes segments w, w + warps, ... of a half-step
// and runs on SM sub-partition w % 4, so the half-step takes about what the
// fullest sub-partition has to issue (its segments, each half a cell on top of its
// cells), and a CTA alone on its SM also what its fullest warp has.
size_t canon_plan(Geometry& g, int warps, int* mode, int bands) {
    constexpr size_t kCtaMax = 227 * 1024;
    auto bytes = [&](int m) { return sizeof(uint32_t) * static_cast<size_t>(canon_smem(g, m).total); };
    auto cut = [&](int nseg) {
        g.seg_cells = (g.Wc + nseg - 1) / nseg;
        g.n_seg = (g.Wc + g.seg_cells - 1) / g.seg_cells;
    };
    const int min_seg = (g.Wc + kMaxSegCells - 1) / kMaxSegCells;
    cut(min_seg);
    for (*mode = kCanonRec; *mode < kCanonPacked && bytes(*mode) > kCtaMax;) ++*mode;
    int best = min_seg;
    double best_cost = 0.0;
    for (int nseg = min_seg; nseg <= g.Wc; ++nseg) {
        cut(nseg);
        // a band does its boundary row of cells first, then the others
        const int n = bands > 1 ? ((g.W + bands - 1) / bands - 1) * g.n_seg : g.W * g.n_seg;
        int rounds = (n + warps - 1) / warps, fullest = bands > 1 ? (g.n_seg + 3) / 4 : 0;
        if (bands > 1) rounds += (g.n_seg + warps - 1) / warps;
        int most = 0;
        for (int q = 0; q < 4; ++q) {
            int c = 0;
            for (int w = q; w < warps; w += 4) c += w < n ? (n - w + warps - 1) / warps : 0;
            most = std::max(most, c);
        }
        fullest += most;
        const double cost = (fullest + rounds) * (g.seg_cells + 0.5);
        if (nseg == min_seg || (cost < best_cost && bytes(*mode) <= kCtaMax)) {
            best = nseg;
            best_cost = cost;
        }
    }
    cut(best);
    return bytes(*mode);
}

namespace {
using PersistentKernel = void (*)(const SweepArgs, int, int*);
template <int kMaxThreads>
PersistentKernel persistent_kernel(int mode, int paper) {
    if (paper)
        return mode == kCanonRec     ? k_sweep_canon_persistent<kCanonRec, true, kMaxThreads>
               : mode == kCanonPlain ? k_sweep_canon_persistent<kCanonPlain, true, kMaxThreads>
                                     : k_sweep_canon_persistent<kCanonPacked, true, kMaxThreads>;
    return mode == kCanonRec     ? k_sweep_canon_persistent<kCanonRec, false, kMaxThreads>
           : mode == kCanonPlain ? k_sweep_canon_persistent<kCanonPlain, false, kMaxThreads>
                                 : k_sweep_canon_persistent<kCanonPacked, false, kMaxThreads>;
}
PersistentKernel persistent_kernel(int mode, int paper, int cta) {
    return cta == kCtaWide   ? persistent_kernel<kCtaWide>(mode, paper)
           : cta == kCtaPair ? persistent_kernel<kCtaPair>(mode, paper)
                             : persistent_kernel<kCtaAny>(mode, paper);
}

using SplitKernel = void (*)(const SweepArgs);
SplitKernel split_kernel(int mode, int paper) {
    if (paper)
        return mode == kCanonRec     ? k_sweep_canon_split<kCanonRec, true>
               : mode == kCanonPlain ? k_sweep_canon_split<kCanonPlain, true>
                                     : k_sweep_canon_split<kCanonPacked, true>;
    return mode == kCanonRec     ? k_sweep_canon_split<kCanonRec, false>
           : mode == kCanonPlain ? k_sweep_canon_split<kCanonPlain, false>
                                 : k_sweep_canon_split<kCanonPacked, false>;
}
cudaLaunchConfig_t split_config(int n_words, int bands, int warps, size_t smem, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(static_cast<unsigned int>(n_words * bands));
    c.blockDim = dim3(static_cast<unsigned int>(32 * warps));
    c.dynamicSmemBytes = smem;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = static_cast<unsigned int>(bands);
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}

// The bands a word is split into: the most (a power of two up to 8) with which
// every cluster is resident at once, an SM per CTA, and a band has at least 20
// cells (below that the cluster barriers cost more than the cells they save:
// L = 12 in two bands 2.2 us per sweep, whole 2.1).  1: no split.  Correlations
// need the whole lattice in one CTA.
int pick_bands(const Geometry& g0, int n_words, int warps, int sms, bool correlations) {
    if (correlations || 32 * warps > kCtaWide) return 1;
    for (int nb = 8; nb > 1; nb /= 2) {
        if (nb > g0.W || g0.n_cells < 20 * nb || n_words * nb > sms) continue;
        Geometry g = g0;
        int mode = 0, clusters = 0;
        const size_t smem = canon_plan(g, warps, &mode, nb);
        const SplitKernel k = split_kernel(mode, g.paper);
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t c = split_config(n_words, nb, warps, smem, &attr);
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, k, &c) == cudaSuccess && clusters >= n_words)
            return nb;
        cudaGetLastError();  // (not sticky: no split of this size)
    }
    return 1;
}

cudaError_t make_plan(const Geometry& g0, int n_words, int warps, int dev, bool correlations, CanonLaunch& p) {
    Geometry g = g0;
    p = CanonLaunch();
    p.smem = canon_plan(g, warps, &p.mode);
    p.seg_cells = g.seg_cells;
    p.n_seg = g.n_seg;
    cudaError_t e = cudaDeviceGetAttribute(&p.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    p.bands = pick_bands(g, n_words, warps, p.sms, correlations);
    if (p.bands > 1) {
        p.smem = canon_plan(g, warps, &p.mode, p.bands);
        if ((e = check_dynamic_smem_base(reinterpret_cast<const void*>(split_kernel(p.mode, g.paper)), dev)) != cudaSuccess)
            return e;
        p.seg_cells = g.seg_cells;
        p.n_seg = g.n_seg;
        p.warps = warps;
        p.device = dev;
        return cudaSuccess;
    }
    auto occupancy = [&](int cta, int* per_sm) {
        const PersistentKernel k = persistent_kernel(p.mode, g.paper, cta);
        // (always the most a CTA can have: contexts of other sizes share the kernel)
        cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        if (r == cudaSuccess) r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k, 32 * warps, p.smem);
        return r;
    };
    int per_sm[3] = {0, 0, 0};  // kCtaAny, kCtaPair, kCtaWide
    e = occupancy(kCtaAny, &per_sm[0]);
    if (e == cudaSuccess && 32 * warps <= kCtaPair) e = occupancy(kCtaPair, &per_sm[1]);
    if (e == cudaSuccess && 32 * warps <= kCtaWide) e = occupancy(kCtaWide, &per_sm[2]);
    if (e != cudaSuccess) return e;
    if (per_sm[2] > 0 && (n_words < 2 * p.sms || std::max(per_sm[0], per_sm[1]) == 1)) {
        p.cta = kCtaWide;
        p.per_sm = 1;
    } else if (per_sm[1] >= per_sm[0]) {
        p.cta = kCtaPair;
        p.per_sm = per_sm[1];
    } else {
        p.cta = kCtaAny;
        p.per_sm = per_sm[0];
    }
    if (p.per_sm < 1) return cudaErrorInvalidConfiguration;
    // a CTA per word: the instantiation with the most CTAs per SM (of as many, the one above)
    p.all_cta = p.cta;
    p.resident = p.per_sm;
    if (std::max(per_sm[0], per_sm[1]) > p.per_sm) {
        p.all_cta = per_sm[1] >= per_sm[0] ? kCtaPair : kCtaAny;
        p.resident = std::max(per_sm[0], per_sm[1]);
    }
    for (const int cta : {p.cta, p.all_cta})
        if ((e = check_dynamic_smem_base(reinterpret_cast<const void*>(persistent_kernel(p.mode, g.paper, cta)), dev)) != cudaSuccess)
            return e;
    p.warps = warps;
    p.device = dev;
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_sweep_canon_persistent(const SweepArgs& a0, int warps_per_cta, int* sched, CanonLaunch& plan,
                                          cudaStream_t st) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && (plan.warps != warps_per_cta || plan.device != dev))
        e = make_plan(a0.g, a0.n_words, warps_per_cta, dev, a0.sq_every > 0, plan);
    if (e != cudaSuccess) return e;
    SweepArgs a = a0;
    a.g.seg_cells = plan.seg_cells;
    a.g.n_seg = plan.n_seg;
    if (plan.bands > 1) {
        a.n_bands = plan.bands;
        cudaLaunchAttribute attr;
        cudaLaunchConfig_t c = split_config(a.n_words, plan.bands, warps_per_cta, plan.smem, &attr);
        c.stream = st;
        return cudaLaunchKernelEx(&c, split_kernel(plan.mode, a.g.paper), a);
    }
    // no more CTAs per SM than whole words: were every word held at once, SMs with one word more
    // than others would finish last with nothing to claim for the rest
    const int per_sm = std::max(1, std::min(plan.per_sm, a.n_words / plan.sms));
    int grid = std::min(a.n_words, per_sm * plan.sms), cta = plan.cta, chunk = a.n_sweeps;
    if (grid < a.n_words) {
        const CanonSchedule sc = canon_schedule(a.n_sweeps, a.n_words, a.g.n_cells, plan.sms, per_sm, plan.resident);
        chunk = sc.chunk;
        if (sc.all) {
            grid = a.n_words;
            cta = plan.all_cta;
        }
    }
    if (grid == a.n_words) {
        sched = nullptr;
    } else {
        e = cudaMemsetAsync(sched, 0, sizeof(int) * (4 + static_cast<size_t>(a.n_words)), st);
        if (e != cudaSuccess) return e;
    }
    persistent_kernel(plan.mode, a.g.paper, cta)<<<grid, warps_per_cta * 32, plan.smem, st>>>(a, chunk, sched);
    return cudaGetLastError();
}

}  // namespace crbm
