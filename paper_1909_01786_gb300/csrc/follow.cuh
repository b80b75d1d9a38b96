// Checking one bucket nogood found through an occurrence list, by four lanes.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "device.cuh"
#include "store.h"

namespace aspgpu {

// The assignment codes that a check reads: global memory, or a CTA's copy of
// them in shared memory (half the chain of a check: 30 clocks instead of 300).
template <bool SHARED>
struct Codes {
    uint32_t *w;
    __device__ __forceinline__ uint32_t get(uint32_t i) const { return SHARED ? reinterpret_cast<volatile uint32_t *>(w)[i] : __ldcg(w + i); }
};

// What the four lanes of a quad know after a check: the same on all four, but
// for l.
struct QuadCheck {
    uint32_t id;        // the nogood
    uint32_t len;       // 0: at most eight literals, else its length
    uint32_t n_un;      // unassigned literals (counting stops at two or more)
    uint32_t ul;        // one of them
    bool sat;           // a literal's complement holds
    uint32_t l[2];      // of at most eight literals: this lane's two of the others (PAD_LIT: none)
};

template <class C>
__device__ __forceinline__ void quad_classify(const C &codes, uint32_t fresh, const uint32_t (&l)[2], QuadCheck &r)
{
    const uint32_t quad = threadIdx.x & 28u;
    uint32_t c[2];
#pragma unroll
    for (int q = 0; q < 2; q++) c[q] = l[q] != PAD_LIT ? codes.get(l[q] >> 4) >> ((l[q] >> 1 & 7u) * 4u) : 0u;
    bool un[2], opp = false;
#pragma unroll
    for (int q = 0; q < 2; q++) {
        // a variable claimed in this round (its fresh bit set) reads as unassigned
        const bool in = l[q] != PAD_LIT, free = (c[q] & 3u) == 0u || (c[q] & fresh);
        un[q] = in && free;
        opp |= in && !free && (c[q] & 3u) == ((l[q] & 1u) ? V_T : V_F);
    }
    const uint32_t b0 = (__ballot_sync(0xFFFFFFFFu, un[0]) >> quad) & 15u, b1 = (__ballot_sync(0xFFFFFFFFu, un[1]) >> quad) & 15u;
    const uint32_t bo = (__ballot_sync(0xFFFFFFFFu, opp) >> quad) & 15u;
    const uint32_t u0 = __shfl_sync(0xFFFFFFFFu, l[0], quad + (b0 ? __ffs(b0) - 1 : 0));
    const uint32_t u1 = __shfl_sync(0xFFFFFFFFu, l[1], quad + (b1 ? __ffs(b1) - 1 : 0));
    if (b0 | b1) r.ul = b0 ? u0 : u1;
    r.n_un += (uint32_t)(__popc(b0) + __popc(b1));
    r.sat |= bo != 0u;
}

// Occurrence o of D.occ against the codes, by the quad of lanes 4i .. 4i+3 (o
// the same on all four; 0xFFFFFFFF: nothing to check); all 32 lanes call it.
// An occurrence is 32 bytes, two words a lane: the nogood's id and its other
// literals (PAD_LIT past their number) if it has at most eight, so a check is
// two dependent loads (the words, the codes).  A longer one names its length
// and its literals' place in D.rows.
template <class C>
__device__ __forceinline__ QuadCheck quad_check(const Dev &D, const C &codes, uint32_t fresh, uint32_t o)
{
    const uint32_t sub = threadIdx.x & 3u, quad = threadIdx.x & 28u;
    const bool has = o != 0xFFFFFFFFu;
    const uint2 w = has ? __ldg(reinterpret_cast<const uint2 *>(D.occ) + 4ull * o + sub) : make_uint2(PAD_LIT, PAD_LIT);
    QuadCheck r{};
    r.id = __shfl_sync(0xFFFFFFFFu, w.x, quad);
    const uint32_t w1 = __shfl_sync(0xFFFFFFFFu, w.y, quad), row = __shfl_sync(0xFFFFFFFFu, w.x, quad + 1u);
    r.len = (w1 & END_BIT) ? w1 & 15u : 0u;
    r.l[0] = sub && !r.len ? w.x : PAD_LIT;
    r.l[1] = !r.len ? w.y : PAD_LIT;
    quad_classify(codes, fresh, r.l, r);
    for (uint32_t q = 0; __any_sync(0xFFFFFFFFu, q < r.len && !r.sat && r.n_un < 2u); q += 8u) {
        const bool go = !r.sat && r.n_un < 2u;
        const uint32_t l[2] = {go && q + sub < r.len ? __ldg(D.rows + row + q + sub) : PAD_LIT,
                               go && q + 4u + sub < r.len ? __ldg(D.rows + row + q + 4u + sub) : PAD_LIT};
        quad_classify(codes, fresh, l, r);
    }
    if (!has) r.sat = true;
    return r;
}

// The same by one lane, for rounds with many occurrences: a warp checks 32 at
// a time with about the instructions of a quad's eight, but each lane reads
// its literals one after another.
struct LaneCheck {
    uint32_t id, len, n_un, ul;
    bool sat;
    uint32_t l[7];      // of at most eight literals: the others (PAD_LIT: none)
};

template <class C>
__device__ __forceinline__ void lane_classify(const C &codes, uint32_t fresh, uint32_t l, uint32_t word, LaneCheck &r)
{
    if (l == PAD_LIT) return;
    const uint32_t c = word >> ((l >> 1 & 7u) * 4u);
    if ((c & 3u) == 0u || (c & fresh)) { r.n_un++; r.ul = l; }
    else r.sat |= (c & 3u) == ((l & 1u) ? V_T : V_F);
}

template <class C>
__device__ __forceinline__ LaneCheck lane_check(const Dev &D, const C &codes, uint32_t fresh, uint32_t o)
{
    const uint4 *e = reinterpret_cast<const uint4 *>(D.occ + o);
    const uint4 a = __ldg(e), b = __ldg(e + 1);
    LaneCheck r{};
    r.id = a.x;
    if (a.y & END_BIT) {
        r.len = a.y & 15u;
        for (uint32_t q = 0; q < r.len && !r.sat && r.n_un < 2u; q++) {
            const uint32_t l = __ldg(D.rows + a.z + q);
            lane_classify(codes, fresh, l, codes.get(l >> 4), r);
        }
        return r;
    }
    const uint32_t l[7] = {a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t w[7];
#pragma unroll
    for (int q = 0; q < 7; q++) w[q] = l[q] != PAD_LIT ? codes.get(l[q] >> 4) : 0u;
#pragma unroll
    for (int q = 0; q < 7; q++) {
        lane_classify(codes, fresh, l[q], w[q], r);
        r.l[q] = l[q];
    }
    return r;
}

// Calls f(o, i) for every occurrence o of up to 32 lists, the lanes of the
// warp taking one each at a time: lane i holds list i as [o0, o0 + c).
// f(0xFFFFFFFF, i) on lanes with none left; all 32 lanes call it.
template <class F>
__device__ __forceinline__ void warp_lists_lanes(uint32_t o0, uint32_t c, F f)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t end = c;
#pragma unroll
    for (uint32_t d = 1; d < 32u; d <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, end, d);
        if (lane >= d) end += x;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, end, 31);
    const uint32_t base = o0 - (end - c);
    for (uint32_t t0 = 0; t0 < total; t0 += 32u) {
        const uint32_t t = t0 + lane;
        uint32_t i = 0;
#pragma unroll
        for (uint32_t d = 16; d; d >>= 1)
            if (__shfl_sync(0xFFFFFFFFu, end, i + d - 1u) <= t) i += d;
        i = min(i, 31u);
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, base, i);
        f(t < total ? b + t : 0xFFFFFFFFu, i);
    }
}

// Calls f(o, i) for every occurrence o of up to eight lists, the quads of the
// warp taking one each at a time: lanes i < 8 hold list i as [o0, o0 + c) (c = 0
// on the others).  f(0xFFFFFFFF, i) on quads with none left; all 32 lanes call
// it.
template <class F>
__device__ __forceinline__ void warp_lists(uint32_t o0, uint32_t c, F f)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t end = c;
#pragma unroll
    for (uint32_t d = 1; d < 8u; d <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, end, d);
        if (lane >= d) end += x;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, end, 7);
    const uint32_t base = o0 - (end - c);            // occurrence t of the warp is base + t in its list
    for (uint32_t t0 = 0; t0 < total; t0 += 8u) {
        const uint32_t t = t0 + (lane >> 2);
        uint32_t i = 0;
#pragma unroll
        for (uint32_t q = 0; q < 7u; q++) i += __shfl_sync(0xFFFFFFFFu, end, q) <= t;
        const uint32_t b = __shfl_sync(0xFFFFFFFFu, base, i);
        f(t < total ? b + t : 0xFFFFFFFFu, i);
    }
}

}  // namespace aspgpu
