// Cores of the canonical SS sweeps in row form (the ten filters of Fig. 1 on
// an even, periodic lattice): warp = the 32 chains of a packed word, lane =
// chain, and a lane's 32-bit word holds the spins of n = 1 .. 3 neighbouring
// cells of one row of cells (a segment) of its chain: bits 16 .. 16 + 4 n - 1, a
// nibble per cell (bit 3 = spin (0,0), 2 = (1,0), 1 = (0,1), 0 = (1,1)), the first
// cell in the highest nibble, and at bits 15, 14 the two column-0 spins of the
// next segment's first cell.
//
// What bounds these sweeps (measured on sm_103a, cycles per warp instruction and
// SM sub-partition): LOP3, SHF, ISETP take 2.14 on the ALU; IMAD.WIDE takes 4.3
// on the FMA-heavy pipe and a 2.14 slot of the ALU as well; IMAD takes 2.14 on the
// FMA pipe, IADD 2.14 on either; shared-memory loads and uniform instructions
// take neither.  A cell's Philox calls are 61 wide products and 69 XORs, so every
// further integer instruction adds to a floor of 278 cycles.  Hence:
//  * a cell's window is six adjacent bits of one word (its nibble and the next
//    cell's column 0), and six bits of a second word that holds the odd spin rows
//    of its row of cells beside the even ones of the row below;
//  * the threshold tables are laid out sparsely so that the window, masked, IS
//    the table offset, and two filters' thresholds come with one load: six logic
//    operations per cell for ten thresholds (the site-word form took 50
//    instructions), the step to the next cell is a multiplication by 16;
//  * the ten decisions go to ONE per-lane word whose bits are the slots of the
//    visible indices that use them, merged by three logic operations;
//  * the visible decisions are shifted into the lane's new word: nothing is
//    balloted or stored per cell.
#pragma once

#include <type_traits>

#include "crbm_device.cuh"

namespace crbm {
namespace canon {

using namespace dev;

// Bits of the hidden word W for each filter unit k (kCanonSlot; l. the cell to
// the left, u. the cell above):
//   spin (0,0): b0 b4 b8 l.b1 u.b5 -> bits  7  8  9 10 11
//   spin (0,1): b0 b6 b1 u.b7 u.b9 -> bits 12 13 14 15 16
//   spin (1,0): b2 b4 b5 l.b3 l.b9 -> bits 17 18 19 20 21
//   spin (1,1): b2 b6 b8 b3 b7     -> bits 22 23 24 25 26
// A unit sets the bits of its own cell's spins and of the neighbours' that it
// meets (b1, b3, b9: the cell to the right; b5, b7, b9: the cell below).
__host__ __device__ constexpr uint32_t unit_word(int k) {
    constexpr uint32_t v[10] = {(1u << 7) | (1u << 12),  (1u << 14) | (1u << 10), (1u << 17) | (1u << 22),
                                (1u << 25) | (1u << 20), (1u << 8) | (1u << 18),  (1u << 19) | (1u << 11),
                                (1u << 13) | (1u << 23), (1u << 26) | (1u << 15), (1u << 9) | (1u << 24),
                                (1u << 16) | (1u << 21)};
    return v[k];
}
constexpr uint32_t kDownBits = (1u << 11) | (1u << 15) | (1u << 16);   // of the word form: for the cell below
constexpr uint32_t kRightBits = (1u << 10) | (1u << 20) | (1u << 21);  // for the cell to the right
constexpr uint32_t kOwnBits = ((1u << 27) - (1u << 7)) & ~kDownBits & ~kRightBits;

// The tables, byte offsets from their shared address (a multiple of 16384).
// Window bits 13 .. 8: columns 0, 0, 1, 1, 2, 2 of window rows 0, 1, 0, 1, 0, 1
// (first word) or rows 2, 1, 2, 1, 2, 1 (second word).  A table entry lies at the
// window's masked value; entries of [32 lanes] pairs (256 bytes) or words (128).
// The six sparse tables interleave (kThr*: their first entries), the running sums
// fill the gap before the visible tables [4][32 idx][32 lanes].
constexpr uint32_t kMask01 = 0x2A00u, kMask23 = 0x1500u, kMask46 = 0x3C00u, kMask57 = 0x3C00u, kMask8 = 0x2400u,
                   kMask9 = 0x0900u;
constexpr int kThr46 = 0, kThr01 = 256, kThr57 = 512, kThr8 = 13 * 256, kThr23 = 63 * 256, kThr9 = 65 * 256,
              kRowVis = 24576;
static_assert(kThr23 + 0x1500 + 256 <= kCanonAccByte && kCanonAccByte + 4 * kAccWords <= kRowVis &&
                  kRowVis + 16384 == kCanonTabBytes,
              "the tables' layout (crbm_internal.h)");
// Writes lane l's entries of the sparse tables from its hidden thresholds
// th[cls * 4 + e1 + 2 e2][32 lanes] (thread x of nthreads, all entries).
__device__ __forceinline__ void build_threshold_tables(char* tab, const uint32_t* __restrict__ th, int x0, int nthreads) {
#pragma unroll 4
    for (int x = x0; x < 56 * 32; x += nthreads) {
        const int l = x & 31, e = x >> 5;  // entry 0 .. 55 of the six tables
        auto T = [&](int cls, uint32_t e1, uint32_t e2) { return __ldg(th + (cls * 4 + static_cast<int>(e1 + 2u * e2)) * 32 + l); };
        const uint32_t i = static_cast<uint32_t>(e);
        const uint32_t a = i & 1u, b = (i >> 1) & 1u, c = (i >> 2) & 1u, d = (i >> 3) & 1u;
        if (e < 16) {  // (4,6): bits 13, 12 = filter 4's sites, 11, 10 = filter 6's
            *reinterpret_cast<uint2*>(tab + kThr46 + (a << 13 | b << 12 | c << 11 | d << 10) + 8 * l) = make_uint2(T(0, a, b), T(0, c, d));
        } else if (e < 32) {  // (5,7): their first sites are row 1
            *reinterpret_cast<uint2*>(tab + kThr57 + (a << 13 | b << 12 | c << 11 | d << 10) + 8 * l) = make_uint2(T(0, b, a), T(0, d, c));
        } else if (e < 40) {  // (0,1): columns 0-1 and 1-2 of row 0
            *reinterpret_cast<uint2*>(tab + kThr01 + (a << 13 | b << 11 | c << 9) + 8 * l) = make_uint2(T(0, a, b), T(0, b, c));
        } else if (e < 48) {  // (2,3): of row 1
            *reinterpret_cast<uint2*>(tab + kThr23 + (a << 12 | b << 10 | c << 8) + 8 * l) = make_uint2(T(0, a, b), T(0, b, c));
        } else if (e < 52) {  // 8: (0,0)-(1,1)
            *reinterpret_cast<uint32_t*>(tab + kThr8 + (a << 13 | b << 10) + 4 * l) = T(1, a, b);
        } else {  // 9: (1,2)-(2,1)
            *reinterpret_cast<uint32_t*>(tab + kThr9 + (a << 8 | b << 11) + 4 * l) = T(1, a, b);
        }
    }
}

// w | K when q < t, as one compare and one predicated OR.
template <uint32_t K>
__device__ __forceinline__ uint32_t or_if_less(uint32_t w, uint32_t q, uint32_t t) {
    asm("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p or.b32 %0, %0, %3;\n\t}"
        : "+r"(w)
        : "r"(q), "r"(t), "n"(K));
    return w;
}

// Shared-memory access by 32-bit shared address plus an immediate offset: the
// address is an operand of the load as it is, where a pointer is the base of
// shared memory plus an index.  tab32, tab64: thresholds, constant while a
// word is swept; lds32, lds64, lds128: state, ordered with the barriers.
template <int kOff>
__device__ __forceinline__ uint32_t tab32(uint32_t addr) {
    uint32_t x;
    asm("ld.shared.u32 %0, [%1+%2];" : "=r"(x) : "r"(addr), "n"(kOff));
    return x;
}
template <int kOff>
__device__ __forceinline__ uint2 tab64(uint32_t addr) {
    uint2 x;
    asm("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(x.x), "=r"(x.y) : "r"(addr), "n"(kOff));
    return x;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
    uint32_t x;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x) : "r"(addr));
    return x;
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr) {
    uint32_t x;
    asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(x) : "r"(addr));
    return x;
}
template <int kOff>
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 x;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(x.x), "=r"(x.y) : "r"(addr), "n"(kOff));
    return x;
}
template <int kOff>
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 x;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4+%5];"
                 : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                 : "r"(addr), "n"(kOff));
    return x;
}
template <int kOff = 0>
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t x) {
    asm volatile("st.shared.u32 [%0+%2], %1;" ::"r"(addr), "r"(x), "n"(kOff) : "memory");
}
template <int kOff = 0>
__device__ __forceinline__ void sts8(uint32_t addr, uint32_t x) {
    asm volatile("st.shared.u8 [%0+%2], %1;" ::"r"(addr), "r"(x), "n"(kOff) : "memory");
}
template <int kOff = 0>
__device__ __forceinline__ void sts16(uint32_t addr, uint32_t x) {
    asm volatile("st.shared.u16 [%0+%2], %1;" ::"r"(addr), "h"(static_cast<uint16_t>(x)), "n"(kOff) : "memory");
}
template <int kOff>
__device__ __forceinline__ void sts64(uint32_t addr, uint2 x) {
    asm volatile("st.shared.v2.u32 [%0+%3], {%1, %2};" ::"r"(addr), "r"(x.x), "r"(x.y), "n"(kOff) : "memory");
}

template <int j>
using Cell = std::integral_constant<int, j>;  // the j-th cell of a segment

// The windows of a segment of n cells from its word and the word of the segment
// below, the current cell's (the first's) at bits 13 .. 8; next() moves on.
struct Windows {
    uint32_t x, m;
    __device__ __forceinline__ Windows(uint32_t own, uint32_t below, int n) {
        const uint32_t s = 4u * static_cast<uint32_t>(n) + 2u;
        x = own >> s;
        // rows 1 of the segment beside rows 0 of the segment below (rows alternate from bit 15 up)
        m = ((own & 0x55555555u) | (below & 0xAAAAAAAAu)) >> s;
    }
    __device__ __forceinline__ void next() {
        x *= 16u;
        m *= 16u;
    }
};

// The thresholds of a cell's ten filters.  tab8, tab4 = the tables' shared
// address + 8 and 4 x the lane's column.
struct HiddenThresholds {
    uint2 t01, t23, t46, t57;
    uint32_t t8, t9;
    __device__ __forceinline__ HiddenThresholds(const Windows& w, uint32_t tab8, uint32_t tab4) {
        t01 = tab64<kThr01>((w.x & kMask01) | tab8);
        t23 = tab64<kThr23>((w.x & kMask23) | tab8);
        t46 = tab64<kThr46>((w.x & kMask46) | tab8);
        t57 = tab64<kThr57>((w.m & kMask57) | tab8);
        t8 = tab32<kThr8>((w.x & kMask8) | tab4);
        t9 = tab32<kThr9>((w.m & kMask9) | tab4);
    }
};

// The hidden word of a cell: W, or its ten decisions (bit k = unit k, kPacked).
template <bool kPacked>
struct HiddenWord {
    uint32_t w = 0u;
    template <int k>
    __device__ __forceinline__ void decide(uint32_t q, uint32_t t) {
        w = or_if_less<kPacked ? 1u << k : unit_word(k)>(w, q, t);
    }
};

// Hidden half-step of one cell: the thresholds against the cell's three
// Philox calls (record words q0, q1, see kCellRec).
template <bool kPacked>
__device__ __forceinline__ uint32_t hidden_row_cell(const HiddenThresholds& t, const uint4& q0, const uint4& q1,
                                                    const Round1Sweep& r1, uint32_t Y, const uint32_t (&rk)[20]) {
    const Round2Cell r2 = round2_cell(r1.hik ^ q0.x);  // shared by the cell's calls
    const U4 u0 = philox_from_call(Y, r1, r2, {q0.y, q0.z}, rk);
    const U4 u1 = philox_from_call(Y, r1, r2, {q0.w, q1.x}, rk);
    const U4 u2 = philox_from_call(Y, r1, r2, {q1.y, q1.z}, rk);
    HiddenWord<kPacked> h;
    h.template decide<0>(u0.x, t.t01.x);
    h.template decide<1>(u0.y, t.t01.y);
    h.template decide<2>(u0.z, t.t23.x);
    h.template decide<3>(u0.w, t.t23.y);
    h.template decide<4>(u1.x, t.t46.x);
    h.template decide<5>(u1.y, t.t57.x);
    h.template decide<6>(u1.z, t.t46.y);
    h.template decide<7>(u1.w, t.t57.y);
    h.template decide<8>(u2.x, t.t8);
    h.template decide<9>(u2.y, t.t9);
    return h.w;
}

// The same in paper precision: every Philox word carries two 16-bit uniforms
// and a threshold holds its 16-bit value in the upper half, so a word's
// high-half uniform compares as the whole word and its low half after a shift
// by 16.  Filter k takes half k & 1 of word k >> 1 of the tag-0 call, filters 8
// and 9 the halves of word 0 of the tag-1 call, whose words 1 and 2 (the cell's
// four visible uniforms) are returned in vis.
__device__ __forceinline__ uint32_t hidden_row_cell_paper(const HiddenThresholds& t, const uint4& q0, const uint4& q1,
                                                          const Round1Sweep& r1, uint32_t Y,
                                                          const uint32_t (&rk)[20], uint2& vis) {
    const Round2Cell r2 = round2_cell(r1.hik ^ q0.x);
    const U4 u0 = philox_from_call(Y, r1, r2, {q0.y, q0.z}, rk);
    const U4 u1 = philox_from_call(Y, r1, r2, {q0.w, q1.x}, rk);
    HiddenWord<false> h;
    h.decide<0>(u0.x << 16, t.t01.x);
    h.decide<1>(u0.x, t.t01.y);
    h.decide<2>(u0.y << 16, t.t23.x);
    h.decide<3>(u0.y, t.t23.y);
    h.decide<4>(u0.z << 16, t.t46.x);
    h.decide<5>(u0.z, t.t57.x);
    h.decide<6>(u0.w << 16, t.t46.y);
    h.decide<7>(u0.w, t.t57.y);
    h.decide<8>(u1.x << 16, t.t8);
    h.decide<9>(u1.x, t.t9);
    vis = make_uint2(u1.y, u1.z);
    return h.w;
}

// The visible call of a cell from its record words qv (lo, Q.h, Q.l).
__device__ __forceinline__ U4 visible_draw(const uint4& qv, const Round1Sweep& r1, uint32_t Y,
                                           const uint32_t (&rk)[20]) {
    return philox_from_call(Y, r1, round2_cell(r1.hik ^ qv.x), {qv.y, qv.z}, rk);
}

// The merged visible index bits of a cell from the hidden words of the cell, the
// cell above and the cell to the left.
__device__ __forceinline__ uint32_t merge_words(uint32_t own, uint32_t up, uint32_t left) {
    return (own & kOwnBits) | (up & kDownBits) | (left & kRightBits);
}
// W of a packed hidden word.
__device__ __forceinline__ uint32_t expand_word(uint32_t h) {
    uint32_t w = 0u;
#pragma unroll
    for (int k = 0; k < 10; ++k) w |= (0u - ((h >> k) & 1u)) & unit_word(k);
    return w;
}

// Visible half-step of one cell: its uniforms against the thresholds at the
// merged bits c; the four decisions are the next nibble of the new word o.
// kVis: the visible tables' offset from tab4's address.
template <int kVis>
__device__ __forceinline__ uint32_t visible_row_cell(uint32_t c, const U4& u, uint32_t tab4, uint32_t o) {
    constexpr uint32_t f = 31u << 7;
    const uint32_t t00 = tab32<kVis>((c & f) | tab4);
    const uint32_t t01 = tab32<kVis + 4096>(((c >> 5) & f) | tab4);
    const uint32_t t10 = tab32<kVis + 8192>(((c >> 10) & f) | tab4);
    const uint32_t t11 = tab32<kVis + 12288>(((c >> 15) & f) | tab4);
    o *= 16u;
    o = or_if_less<8u>(o, u.x, t00);
    o = or_if_less<2u>(o, u.y, t01);
    o = or_if_less<4u>(o, u.z, t10);
    o = or_if_less<1u>(o, u.w, t11);
    return o;
}

// Record words of cell `cell` (see kCellRec), formed on the device: the hidden
// calls', and the visible call's (in paper precision the tag-1 call).
__device__ __forceinline__ void hidden_call_words(uint32_t cell, const uint32_t (&rk)[20], uint4& q0, uint4& q1) {
    const Round0Cell rc = round0_cell(cell, rk[1]);
    const Round1Call c0 = round1_call(rc.a, rk), c1 = round1_call(rc.a ^ 1u, rk), c2 = round1_call(rc.a ^ 2u, rk);
    q0 = make_uint4(rc.b, c0.h, c0.l, c1.h);
    q1 = make_uint4(c1.l, c2.h, c2.l, 0u);
}
__device__ __forceinline__ uint4 visible_call_words(uint32_t cell, uint32_t tag, const uint32_t (&rk)[20]) {
    const Round0Cell rc = round0_cell(cell, rk[1]);
    const Round1Call cv = round1_call(rc.a ^ tag, rk);
    return make_uint4(rc.b, cv.h, cv.l, 0u);
}

// Measurement counts of a segment of n cells (words as for Windows): anti-aligned
// J and J' filters and +1 spins of the lane's chain.
__device__ __forceinline__ void count_segment(uint32_t own, uint32_t below, int n, int& anti0, int& anti1, int& pos) {
    const uint32_t x = own >> 14, s = own >> 16, b = below >> 17;
    const uint32_t m = (1u << (4 * n)) - 1u;
    // columns 0-1 and 1-2 of both rows, then rows 0-1 and 1-2 of both columns
    anti0 += __popc((x ^ (x >> 2)) & m) + __popc((s ^ (s >> 1)) & (m & 0x55555555u)) + __popc((s ^ b) & (m & 0x55555555u));
    anti1 += __popc((s ^ (s >> 3)) & (m & 0x11111111u)) + __popc((x ^ b) & (m & 0x11111111u));
    pos += __popc(s);
}

// The site of each bit 14 .. 16 + 4 n - 1 of a segment's word, lane = bit: cells
// j .. j + n - 1 of cell row i, jn the next segment's first cell (bits 15, 14).
// Full segments away from the right edge share their offsets from the first
// cell's site.
struct SegmentSites {
    int Lc, full;
    __device__ __forceinline__ SegmentSites(int Lc_, int lane) : Lc(Lc_) { full = offset(lane - 16, 3, 6); }
    // site of bit 16 + p less the first cell's; next = column of jn less the first cell's
    __device__ __forceinline__ int offset(int p, int n, int next) const {
        return p >= 0 ? (1 - (p & 1)) * Lc + 2 * (n - 1 - (p >> 2)) + 1 - ((p >> 1) & 1) : (-1 - p) * Lc + next;
    }
    // lanes < 14 and >= 16 + 4 n have no site
    __device__ __forceinline__ int operator()(int lane, int i, int j, int n, int jn) const {
        const int first = 2 * i * Lc + 2 * j;
        return first + (n == 3 && jn > j ? full : offset(lane - 16, n, 2 * (jn - j)));
    }
};

}  // namespace canon
}  // namespace crbm
