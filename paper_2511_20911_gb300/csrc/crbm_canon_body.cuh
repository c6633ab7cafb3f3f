// Body of the canonical SMEM-resident sweep (one CTA = one 32-chain word, or
// one band of cell rows of a word in a thread-block cluster), shared by the
// persistent kernel (crbm_canon.cu) and the batched kernel (crbm_batch.cu).
// The spins are kept in row form (crbm_row_core.cuh).
#pragma once

#include <cooperative_groups.h>

#include "crbm_row_core.cuh"

namespace crbm {
namespace canon {

namespace cg = cooperative_groups;

// Cell records: in shared memory (an address) or read through the read-only
// cache (a pointer).
template <int kMode>
struct CellRecs {
    const uint4* p;
    __device__ __forceinline__ CellRecs(uint32_t, const uint4* g, int cell) : p(g + static_cast<size_t>(cell) * kCellRec) {}
    template <int k>
    __device__ __forceinline__ uint4 get() const {
        return __ldg(p + k);
    }
};
template <>
struct CellRecs<kCanonRec> {
    uint32_t p;
    __device__ __forceinline__ CellRecs(uint32_t s, const uint4*, int cell) : p(s + 16u * kCellRec * static_cast<uint32_t>(cell)) {}
    template <int k>
    __device__ __forceinline__ uint4 get() const {
        return lds128<16 * k>(p);
    }
};

// The two halves of a cluster barrier, so that work no other CTA waits for
// can run between them: arrive (release: this thread's earlier shared-memory
// stores, local and remote) and wait (acquire).  Every thread of the CTA
// executes both, the same number of times on every rank.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// CTA barrier, or cluster barrier (release / acquire over the cluster's
// shared memory) when a word is split over the CTAs of a cluster.
template <bool kCluster>
__device__ __forceinline__ void body_sync() {
    if (kCluster)
        cg::this_cluster().sync();
    else
        __syncthreads();
}

// Whole-run body of the canonical SMEM-resident sweep for packed word `word`:
// load tables, spins and replica permutation into shared memory, run
// n_sweeps sweeps from global sweep t0 (measurement index meas0) with
// measurement / replica exchange / correlations, write the state back.
// State is read with L1-bypassing loads: under the persistent scheduler the
// previous chunk of this word may have been written by another SM.
// A warp's unit of work is a segment of a row of cells (a.g.seg_cells cells).
// kMode: how the word is kept in shared memory (kCanon*, crbm_internal.h).
// kCluster: the CTA holds band `band` of the word's a.n_bands bands of cell
// rows; the word's bands are the cluster ranks rank0 .. rank0 + n_bands - 1
// (a cluster may hold several words of one context, or padding ranks of that
// context with band >= n_bands).  Every rank holds the whole lattice;
// it updates its own rows and, as it goes, writes the hidden words of its
// last cell row into the next band (the upper neighbours of that band's first
// row) and the spins of its first spin row into the previous band (the last
// window row of that band's last cell row), wrapping around.  Half-steps end
// with a cluster barrier; measurement counts are summed into the word's
// band 0, which runs the measurement and the replica exchange.  Padding ranks
// (band >= n_bands) only keep the barrier count, which is the same for every
// rank because a cluster never mixes contexts.  Correlations need the whole
// lattice, so a word with sq_every > 0 is never split (n_bands == 1).
// A band does the cells other bands wait for first (its last cell row in
// the hidden half-step, its first in the visible one), arrives at the cluster
// barrier, does the rest and only then waits.  Those boundary cells are the
// only ones that read rows a neighbour writes, and they run after the
// previous barrier completed, so no band overwrites a row its neighbour has
// yet to read.
// first: false when this CTA's previous word was of the same context (its records
// and expansion table are then in place).
// kPaper: CRBM_PRECISION_PAPER draws (two Philox calls per cell, the visible
// uniforms passed from the hidden half-step through shared memory, or drawn
// again in the visible one with kCanonPacked).
template <int kMode, bool kCluster, bool kPaper = false>
__device__ __forceinline__ void sweep_canon_body(const SweepArgs& a, int word, uint32_t t0, int n_sweeps,
                                                 int64_t meas0, int band = 0, int rank0 = 0,
                                                 bool first = true) {
    extern __shared__ __align__(128) uint32_t smem[];
    constexpr bool kPacked = kMode == kCanonPacked && !kPaper;  // 16-bit hidden words
    constexpr bool kRedraw = kMode == kCanonPacked && kPaper;   // the visible call drawn again
    constexpr uint32_t kWCell = kPacked ? 64u : 128u;           // bytes of a cell's hidden words
    const Geometry& g = a.g;
    const int W = g.W, Wc = g.Wc;  // rows and columns of cells
    const int nseg = g.n_seg, uc = g.seg_cells;
    // (the shuffle tells the compiler that the warp index is warp-uniform: segment indices, loop counters
    // and cell addresses then run on the uniform pipe)
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);
    const int nwarp = blockDim.x >> 5;
    // The warp that keeps the running sums and finishes each measurement: the
    // last, which has the fewest segments when they do not divide evenly, so that
    // it can finish a measurement while the others start the next sweep.
    const int post_warp = nwarp - 1;
    const int nb = kCluster ? a.n_bands : 1;
    const bool active = band < nb;
    const int row0 = active ? band * W / nb : 0, row1 = active ? (band + 1) * W / nb : 0;
    const int u_begin = kCluster ? row0 * nseg : 0, u_end = kCluster ? row1 * nseg : W * nseg;
    const CanonSmem cs = canon_smem(g, kMode);
    int64_t* s_acc = reinterpret_cast<int64_t*>(smem + cs.acc);  // [kNSum][32] running sums
    int* s_cnt = reinterpret_cast<int*>(smem + cs.cnt);          // [3][32]
    int* s_sob = reinterpret_cast<int*>(smem + cs.sob);          // [32] slot of each rung
    int* s_bos = s_sob + 32;                                     // [32] rung of each slot
    uint32_t* s_u = smem + cs.u;                                 // [32] the swap round's uniforms
    uint32_t* s_segmask = smem + cs.segmask;
    int* s_seg = reinterpret_cast<int*>(smem + cs.seg);
    char* sm = reinterpret_cast<char*>(smem);
    char* s_tab = sm + 4 * kCanonTabWord;
    const uint32_t base = static_cast<uint32_t>(__cvta_generic_to_shared(smem));  // shared addresses from here on
    const uint32_t tab = base + 4u * kCanonTabWord;
    if (tab & 16383u) return;  // (the launchers have checked it: every CTA of the grid agrees)
    const uint32_t rec_addr = base + 4u * static_cast<uint32_t>(cs.rec);
    const uint32_t pw_addr = base + 4u * static_cast<uint32_t>(cs.pw);
    const uint32_t w_addr = base + 4u * static_cast<uint32_t>(cs.w);
    const uint32_t rows_addr = base + 4u * static_cast<uint32_t>(cs.rows);
    const uint32_t exp_addr = base + 4u * static_cast<uint32_t>(cs.expand);
    const uint32_t lane4 = 4u * static_cast<uint32_t>(lane);
    const uint32_t lane_w = kPacked ? 2u * static_cast<uint32_t>(lane) : lane4;
    const uint32_t seg_magic = nseg > 1 ? (0xFFFFFFFFu / static_cast<uint32_t>(nseg)) + 1u : 0u;
    // Segment u: cells j0 .. j0 + n - 1 of row i; the segment below it, and the one to its left
    struct Segment {
        int i, j0, n, below, left;
    };
    auto segment = [&](int u) {
        Segment r;
        r.i = nseg > 1 ? static_cast<int>(__umulhi(static_cast<uint32_t>(u), seg_magic)) : u;
        const int s = u - r.i * nseg;
        r.j0 = s * uc;
        r.n = min(uc, Wc - r.j0);
        r.below = r.i + 1 == W ? s : u + nseg;
        r.left = s > 0 ? u - 1 : u + nseg - 1;
        return r;
    };
    auto row_addr = [&](int u) { return rows_addr + 128u * static_cast<uint32_t>(u) + lane4; };
    // a segment's new nibbles, and its first column for the segment to its left
    auto store_row = [&](int u, const Segment& sg, uint32_t o) {
        sts16<2>(row_addr(u), o);
        sts8<1>(row_addr(sg.left), (o >> (4u * static_cast<uint32_t>(sg.n) - 2u)) << 6);
    };
    auto w_of = [&](int cell) { return w_addr + kWCell * static_cast<uint32_t>(cell) + lane_w; };
    auto load_w = [&](uint32_t addr) -> uint32_t { return kPacked ? lds32(exp_addr + 4u * lds16(addr)) : lds32(addr); };
    // cluster neighbours (unused without a split)
    char* sm_next = sm;
    char* sm_prev = sm;
    int* cnt0 = s_cnt;
    const int* bos0 = s_bos;
    if (kCluster && active) {
        cg::cluster_group cl = cg::this_cluster();
        if (nb > 1) {
            sm_next = cl.map_shared_rank(sm, static_cast<unsigned int>(rank0 + (band + 1) % nb));
            sm_prev = cl.map_shared_rank(sm, static_cast<unsigned int>(rank0 + (band + nb - 1) % nb));
        }
        cnt0 = cl.map_shared_rank(s_cnt, static_cast<unsigned int>(rank0));
        bos0 = cl.map_shared_rank(s_bos, static_cast<unsigned int>(rank0));
    }

    const uint32_t chain = static_cast<uint32_t>(word) * 32u + lane;
    const Round0Lane r0l = round0_lane(chain);
    const bool measuring = a.measure_every > 0;
    if (active) {
        // (every load of the staging is in flight before the first is waited for: a one-sweep launch
        // is mostly this)
        const uint32_t* gt = a.ctab + static_cast<size_t>(word) * kCanonTab;
        auto stage = [&](uint32_t dst, const uint4* src, int n) {
            for (int x = threadIdx.x; x < n; x += blockDim.x)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * static_cast<uint32_t>(x)), "l"(src + x)
                             : "memory");
        };
        stage(tab + kRowVis, reinterpret_cast<const uint4*>(gt + kCanonTh), 4 * 32 * 32 / 4);
        if (kMode == kCanonRec && first) {
            const int c0 = kCluster ? row0 * Wc : 0, c1 = kCluster ? row1 * Wc : g.n_cells;
            stage(rec_addr + 16u * kCellRec * static_cast<uint32_t>(c0), a.crec + static_cast<size_t>(c0) * kCellRec, (c1 - c0) * kCellRec);
        }
        // spins to row form: the site words of a segment's word (lane = bit), bit-transposed (lane = chain)
        const uint32_t* gv = a.v + static_cast<size_t>(word) * g.N;
        const Transpose32 transpose(lane);
        const SegmentSites site(g.Lc, lane);
        // (a band: its own rows and the one below them; the rest of the lattice is never read)
        const int n_staged = kCluster ? min(u_end - u_begin + nseg, W * nseg) : W * nseg;
        auto staged = [&](int x) { return !kCluster ? x : u_begin + x < W * nseg ? u_begin + x : u_begin + x - W * nseg; };
        for (int u0 = warp; u0 < n_staged; u0 += 4 * nwarp) {
            uint32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v[k] = 0u;
                if (u0 + k * nwarp < n_staged) {
                    const Segment sg = segment(staged(u0 + k * nwarp));
                    const int sx = site(lane, sg.i, sg.j0, sg.n, sg.j0 + sg.n == Wc ? 0 : sg.j0 + sg.n);
                    if (lane >= 14 && lane < 16 + 4 * sg.n) v[k] = __ldcg(gv + sx);
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (u0 + k * nwarp < n_staged) sts32(row_addr(staged(u0 + k * nwarp)), transpose(v[k]));
        }
        build_threshold_tables(s_tab, gt, threadIdx.x, blockDim.x);
        if (kPacked && first)
            for (int x = threadIdx.x; x < 1024; x += blockDim.x) smem[cs.expand + x] = expand_word(static_cast<uint32_t>(x));
        if (band == 0 && warp == post_warp && measuring) {
#pragma unroll
            for (int x = 0; x < kNSum; ++x)
                s_acc[x * 32 + lane] = __ldcg(a.sums + static_cast<size_t>(chain) * kNSum + x);
        }
        for (int x = threadIdx.x; x < 96; x += blockDim.x) s_cnt[x] = 0;
        if (a.sq_every > 0) {
            for (int x = threadIdx.x; x < 33; x += blockDim.x) s_seg[x] = a.seg[word * 33 + x];
            for (int x = threadIdx.x; x < 32; x += blockDim.x) s_segmask[x] = a.segmask[word * 32 + x];
        }
        if (warp == post_warp) {  // replica permutation (identity without tempering)
            const int sob = a.swap_every > 0 ? __ldcg(a.sob + word * 32 + lane) : lane;
            s_sob[lane] = sob;
            s_bos[sob] = lane;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncthreads();
    uint32_t tab4 = tab + 4u * static_cast<uint32_t>(s_bos[lane]);  // lane reads the column of its rung
    if (kCluster) body_sync<true>();  // every rank started before any shared memory crosses CTAs

    int64_t meas = meas0;
    EveryCounter every_meas(t0, a.measure_every), every_swap(t0, a.swap_every), every_sq(t0, kCluster ? 0 : a.sq_every);
    for (int it = 0; it < n_sweeps; ++it) {
        const uint32_t t = t0 + static_cast<uint32_t>(it);
        const Round1Sweep rs = round1_sweep(r0l.hi ^ t ^ a.rk[0], a.rk);
        if (every_swap.now() && band == 0 && warp == post_warp) s_u[lane] = swap_uniform(a, lane, word, t);
        // hidden half-step; a band's last cell row first (the next band waits for its hidden words),
        // arrive, the rest, then wait: the cluster barrier's latency overlaps the interior rows
        const int split = kCluster && nb > 1 ? u_end - nseg : u_begin;
        for (int ph = kCluster && nb > 1 ? 0 : 1; ph < 2; ++ph) {
            const int ub = ph == 0 ? split : u_begin, ue = ph == 0 || !(kCluster && nb > 1) ? u_end : split;
            if (!kCluster || active)
                for (int u = ub + warp; u < ue; u += nwarp) {
                    const Segment sg = segment(u);
                    Windows win(lds32(row_addr(u)), lds32(row_addr(sg.below)), sg.n);
                    const int cell = sg.i * Wc + sg.j0;
                    CellRecs<kMode> rec(rec_addr, a.crec, cell);
                    const uint32_t wo = w_of(cell), po = pw_addr + 256u * static_cast<uint32_t>(cell) + 2u * lane4;
                    const uint32_t tab8 = 2u * tab4 - tab;
                    auto one = [&](auto jc) {
                        constexpr int j = decltype(jc)::value;
                        const HiddenThresholds th(win, tab8, tab4);
                        const uint4 q0 = rec.template get<kCellRec * j>(), q1 = rec.template get<kCellRec * j + 1>();
                        uint32_t w;
                        if (kPaper) {
                            uint2 vis;
                            w = hidden_row_cell_paper(th, q0, q1, rs, r0l.lo, a.rk, vis);
                            if (!kRedraw) sts64<256 * j>(po, vis);
                        } else {
                            w = hidden_row_cell<kPacked>(th, q0, q1, rs, r0l.lo, a.rk);
                        }
                        if (kPacked)
                            sts16<static_cast<int>(kWCell) * j>(wo, w);
                        else
                            sts32<static_cast<int>(kWCell) * j>(wo, w);
                        if (kCluster && ph == 0) {  // what the cells below read
                            char* o = sm_next + (wo + kWCell * j - base);
                            if (kPacked)
                                *reinterpret_cast<uint16_t*>(o) = static_cast<uint16_t>(w);
                            else
                                *reinterpret_cast<uint32_t*>(o) = w;
                        }
                        win.next();
                    };
                    one(Cell<0>());
                    if (sg.n > 1) {
                        one(Cell<1>());
                        if (sg.n > 2) one(Cell<2>());
                    }
                }
            if (kCluster && ph == 0) cluster_arrive();
        }
        __syncthreads();
        if (kCluster && nb > 1) cluster_wait();
        // visible half-step; a band's first cell row first (the previous band waits for its spins)
        const int vsplit = kCluster && nb > 1 ? u_begin + nseg : u_begin;
        for (int ph = kCluster && nb > 1 ? 0 : 1; ph < 2; ++ph) {
            const int ub = ph == 0 ? u_begin : vsplit, ue = ph == 0 ? vsplit : u_end;
            if (!kCluster || active)
                for (int u = ub + warp; u < ue; u += nwarp) {
                    const Segment sg = segment(u);
                    const int cell = sg.i * Wc + sg.j0;
                    CellRecs<kMode> rec(rec_addr, a.crec, cell);
                    const uint32_t po = pw_addr + 256u * static_cast<uint32_t>(cell) + 2u * lane4;
                    const uint32_t wo = w_of(cell), wu = w_of(sg.i > 0 ? cell - Wc : cell + (W - 1) * Wc);
                    uint32_t left = load_w(w_of(sg.j0 > 0 ? cell - 1 : cell + Wc - 1)), o = 0u;
                    auto draw = [&](auto jc) {
                        constexpr int j = decltype(jc)::value;
                        if (kPaper) {
                            uint2 vis;
                            if (kRedraw) {
                                const U4 q = visible_draw(rec.template get<kCellRec * j + 2>(), rs, r0l.lo, a.rk);
                                vis = make_uint2(q.y, q.z);
                            } else {
                                vis = lds64<256 * j>(po);
                            }
                            return U4{vis.x << 16, vis.x, vis.y << 16, vis.y};
                        }
                        return visible_draw(rec.template get<kCellRec * j + 2>(), rs, r0l.lo, a.rk);
                    };
                    auto decide = [&](auto jc, const U4& q) {
                        constexpr uint32_t off = kWCell * decltype(jc)::value;
                        const uint32_t own = load_w(wo + off);
                        o = visible_row_cell<kRowVis>(merge_words(own, load_w(wu + off), left), q, tab4, o);
                        left = own;
                    };
                    if (sg.n == 3) {  // the three calls side by side
                        const U4 a0 = draw(Cell<0>()), a1 = draw(Cell<1>()), a2 = draw(Cell<2>());
                        decide(Cell<0>(), a0);
                        decide(Cell<1>(), a1);
                        decide(Cell<2>(), a2);
                    } else {
                        const U4 a0 = draw(Cell<0>());
                        decide(Cell<0>(), a0);
                        if (sg.n > 1) decide(Cell<1>(), draw(Cell<1>()));
                    }
                    store_row(u, sg, o);
                    if (kCluster && ph == 0) {  // the previous band reads this row as its row below
                        *reinterpret_cast<uint16_t*>(sm_prev + (row_addr(u) + 2u - base)) = static_cast<uint16_t>(o);
                        *reinterpret_cast<uint8_t*>(sm_prev + (row_addr(sg.left) + 1u - base)) =
                            static_cast<uint8_t>((o >> (4u * static_cast<uint32_t>(sg.n) - 2u)) << 6);
                    }
                }
            if (kCluster && ph == 0) cluster_arrive();
        }
        __syncthreads();
        if (kCluster && nb > 1) cluster_wait();
        const bool do_meas = every_meas.step();
        const bool do_swap = every_swap.step();
        if (do_meas || do_swap) {
            if (active) {
                int anti0 = 0, anti1 = 0, pos = 0;
                for (int u = u_begin + warp; u < u_end; u += nwarp) {
                    const Segment sg = segment(u);
                    count_segment(lds32(row_addr(u)), lds32(row_addr(sg.below)), sg.n, anti0, anti1, pos);
                }
                atomicAdd(&cnt0[lane], anti0);
                atomicAdd(&cnt0[32 + lane], anti1);
                atomicAdd(&cnt0[64 + lane], pos);
            }
            body_sync<kCluster>();
            const bool post = band == 0 && warp == post_warp;
            RungCounts rc{0, 0, 0};
            if (post) {
                rc = rung_counts(a, s_cnt, s_sob, lane);
                if (do_swap) swap_rungs(a, rc, s_sob, s_bos, lane, word, t, s_u[lane]);
            }
            // A swap round changes the permutation every warp reads next; a
            // measurement alone touches only warp post_warp's sums and the counts, which
            // the next measurement reaches after the next sweep's barriers.
            if (do_swap) {
                body_sync<kCluster>();
                if (active) tab4 = tab + 4u * static_cast<uint32_t>(bos0[lane]);
            }
            if (do_meas) {
                if (post) add_measurement(a, rc, lane, word, t, meas, s_acc);
                ++meas;
            }
        }
        if (every_sq.step()) {  // the hidden words are dead here: their space holds the lattice
            uint32_t* scratch = smem + cs.w;
            const int L = g.L;
            if (L <= 32) {  // one word per row and chain
                for (int R = warp; R < L; R += nwarp) {
                    uint32_t m = 0u;
                    for (int j0 = 0, s = 0; j0 < Wc; j0 += uc, ++s) {
                        const int n = min(uc, Wc - j0);
                        // bits 0, 2 of a nibble: columns 1, 0 of row R
                        const uint32_t x = lds32(row_addr((R >> 1) * nseg + s)) >> (17 - (R & 1));
                        for (int j = 0; j < n; ++j) {
                            const uint32_t c = x >> (4 * (n - 1 - j));
                            m |= (((c >> 2) & 1u) | ((c & 1u) << 1)) << (2 * (j0 + j));
                        }
                    }
                    scratch[R * 32 + lane] = m;
                }
                __syncthreads();
                accumulate_correlations_rows(a, scratch, s_seg, s_segmask, warp, nwarp, lane);
            } else {  // one word per site
                const SegmentSites site(g.Lc, lane);
                for (int u = warp; u < W * nseg; u += nwarp) {
                    const Segment sg = segment(u);
                    const uint32_t v = transpose32(lds32(row_addr(u)), lane);
                    if (lane >= 16 && lane < 16 + 4 * sg.n) scratch[site(lane, sg.i, sg.j0, sg.n, sg.j0 + sg.n)] = v;
                }
                __syncthreads();
                accumulate_correlations_sites(a, scratch, s_seg, s_segmask, warp, nwarp, lane);
            }
            __syncthreads();
        }
    }
    if (kCluster) body_sync<true>();  // no rank reads another's shared memory after this
    if (!active) return;
    uint32_t* gv = a.v + static_cast<size_t>(word) * g.N;
    const Transpose32 transpose(lane);
    const SegmentSites site(g.Lc, lane);
    for (int u = u_begin + warp; u < u_end; u += nwarp) {  // own rows
        const Segment sg = segment(u);
        const uint32_t v = transpose(lds32(row_addr(u)));
        if (lane >= 16 && lane < 16 + 4 * sg.n) gv[site(lane, sg.i, sg.j0, sg.n, sg.j0 + sg.n)] = v;
    }
    if (band == 0 && warp == post_warp && a.swap_every > 0) a.sob[word * 32 + lane] = s_sob[lane];
    if (band == 0 && warp == post_warp && measuring) {
        for (int x = 0; x < kNSum; ++x) a.sums[static_cast<size_t>(chain) * kNSum + x] = s_acc[x * 32 + lane];
    }
}

}  // namespace canon
}  // namespace crbm
