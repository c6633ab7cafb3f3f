// Word-parallel pieces of the bit-plane sweeps (CRBM_RNG_BITPLANE), shared by
// the SMEM sweep (crbm_bitplane.cu) and the streamed one (crbm_stream.cu).
// Every 32-bit value holds one bit per chain of a 32-chain word.
#pragma once

#include "crbm_device.cuh"

namespace crbm {
namespace bp {

using dev::transpose32;
using dev::U4;

// One plane of the comparison u < t, least significant bit first: lt collects
// the chains with u < t on the planes so far (the borrow of u - t), ne the
// chains with u != t there.  One LOP3 each; the other direction carries the
// open chains from plane to plane and takes three.  U, T: the plane of the
// uniforms and of the thresholds.
__device__ __forceinline__ void plane_step(uint32_t U, uint32_t T, uint32_t& lt, uint32_t& ne) {
    lt = (~U & T) | (~(U ^ T) & lt);
    ne |= U ^ T;
}
__device__ __forceinline__ void planes_step(const U4& q, const uint4& T, uint32_t& lt, uint32_t& ne) {
    plane_step(q.w, T.w, lt, ne);
    plane_step(q.z, T.z, lt, ne);
    plane_step(q.y, T.y, lt, ne);
    plane_step(q.x, T.x, lt, ne);
}
// The planes of a further call, below those compared so far: eq, the chains
// that agree on all of them, are decided by it where they differ.
__device__ __forceinline__ void planes_below(const U4& q, const uint4& T, uint32_t& lt, uint32_t& eq) {
    uint32_t l = 0u, ne = 0u;
    planes_step(q, T, l, ne);
    lt |= eq & l;
    eq &= ~ne;
}

// Four consecutive threshold planes of one row: the planes of one Philox
// call, read with one 16-byte shared-memory load (rows start on a 16-byte
// boundary and calls on a multiple of four planes).
__device__ __forceinline__ uint4 planes4(const uint32_t* p) { return *reinterpret_cast<const uint4*>(p); }

__device__ __forceinline__ uint4 mux4(uint32_t s, const uint4& x1, const uint4& x0) {
    return make_uint4((s & x1.x) | (~s & x0.x), (s & x1.y) | (~s & x0.y), (s & x1.z) | (~s & x0.z),
                      (s & x1.w) | (~s & x0.w));
}

// The four threshold planes of one Philox call of a hidden node with endpoints
// e1, e2: e1 picks m = 2 or m = -2 (tb points at the call's first plane of the
// m = -2 row, m = 2 row 64 words further).  Chains with m = 0 (e1 != e2) take no notice of them:
// their threshold 2^31 is the top plane of the uniform alone (hidden_first).
__device__ __forceinline__ uint4 hidden_planes(const uint32_t* tb, uint32_t e1) {
    return mux4(e1, planes4(tb + 64), planes4(tb));
}
// Calls 0 and 1 of a hidden node (Z: the chains with m = 0): lt the chains
// below their threshold, eq the chains still open.
__device__ __forceinline__ void hidden_first(const U4& q0, const U4& q1, const uint32_t* tb, uint32_t e1, uint32_t Z,
                                             uint32_t& lt, uint32_t& eq) {
    uint32_t l = 0u, ne = Z;
    planes_step(q1, hidden_planes(tb + 4, e1), l, ne);
    planes_step(q0, hidden_planes(tb, e1), l, ne);
    lt = (Z & ~q0.x) | (~Z & l);
    eq = ~ne;
}

// Count of set bits among h0..h3 per chain, c0 + 2 c1 + 4 c2, bit-sliced.
struct Count4 {
    uint32_t c0, c1, c2;
};
__device__ __forceinline__ Count4 count4(uint32_t h0, uint32_t h1, uint32_t h2, uint32_t h3) {
    const uint32_t s01 = h0 ^ h1, a01 = h0 & h1, s23 = h2 ^ h3, a23 = h2 & h3;
    const uint32_t cy = s01 & s23;
    return {s01 ^ s23, a01 ^ a23 ^ cy, (a01 & a23) | (cy & (a01 | a23))};
}

// The four threshold planes of one Philox call of a spin: tb points at the
// call's first plane in the [count][J' bit] rows (32 words apart); hp is the
// J' bit, n the count of the J incidences.  A mux tree per plane: the J' bit,
// then count bits 0, 1, 2 (a count of 4 has bits 0 and 1 clear).
__device__ __forceinline__ uint4 visible_planes(const uint32_t* tb, uint32_t hp, const Count4& n) {
    auto sel = [&](int c) { return mux4(hp, planes4(tb + (2 * c + 1) * 32), planes4(tb + 2 * c * 32)); };
    const uint4 m01 = mux4(n.c0, sel(1), sel(0));
    const uint4 m23 = mux4(n.c0, sel(3), sel(2));
    return mux4(n.c2, sel(4), mux4(n.c1, m23, m01));
}

// Appends the lanes whose comparison is still open (open != 0: its
// undecided chains) to a straggler list of (node, open chains) pairs, with
// one atomic per warp; returns true on the lanes whose node went to the list
// (false where the list is full: that lane finishes its node itself).
__device__ __forceinline__ bool push_straggler(uint32_t node, uint32_t open, int* count, uint2* list, int cap,
                                               int lane) {
    const uint32_t bal = __ballot_sync(0xffffffffu, open != 0u);
    if (bal == 0u) return false;
    int first = 0;
    if (lane == 0) first = atomicAdd(count, __popc(bal));
    first = __shfl_sync(0xffffffffu, first, 0);
    const int slot = first + __popc(bal & ((1u << lane) - 1u));
    if (open == 0u || slot >= cap) return false;
    list[slot] = make_uint2(node, open);
    return true;
}

}  // namespace bp
}  // namespace crbm
