// Device-resident conflict-driven answer-set search (sm_103a).
//
// One persistent cooperative kernel runs the whole loop of Algorithm 1:
// InitialPropagation, propagate-and-check sweeps to fixpoint (Section 4.1),
// fwd-learning from decision-level dependency bitmaps (Section 4.2,
// Algorithm 4), Backjump, Decision over applicable rules (Section 2),
// CompleteAssignment, and the stability step.  Phases are separated by a
// grid barrier; the leader (CTA 0, thread 0) writes the control block for the
// next phase into the other half of a double buffer, so all CTAs read a
// stable copy while it is being updated.
//
// Propagation.  Claims are followed through occurrence lists by literal: one
// CTA while they are few (narrow_rounds), the grid when they are more
// (list_round).  Sweeps of the whole store run initial propagation, the round
// after a backjump, rounds with very many claims, and the confirmation of a
// full-sweep program's fixpoint, and lists too long for a warp.  One-CTA programs
// never sweep; programs whose lists did not fit in memory always do.
//
// Sweep design.  The static nogoods sit in one bucket per exact length
// (Section 4: one kernel per length class), stored structure-of-arrays, and
// are cut into contiguous ranges, one per CTA, along groups of nogoods (an
// atom's rules and the atom's own nogood).  Each CTA keeps a 2-bit view of
// the assignment in shared memory: all atoms, plus the auxiliary variables
// of the rules its ranges refer to.  One lane classifies one nogood against
// that view.  A claim (atomicOr on the global 4-bit codes) computes the
// claimed variable's dependency bitmap at once, from its reason, and is then
// published in the CTA's own view, so chains of implications inside a CTA
// can resolve within one sweep; other CTAs see the claim after the next
// barrier.  Long and learned nogoods are settled by a lane each through their
// watched literals, or scanned by one warp (ballot and popc over lanes),
// against the global codes.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "device.cuh"
#include "follow.cuh"
#include "mlp.cuh"
#include "store.h"

namespace aspgpu {

#define FULL_MASK 0xFFFFFFFFu

// CTA barrier that counts every thread on its own (PTX barrier.sync
// without .aligned).  The aligned form counts a warp as arrived when its
// first threads get there, which let warps pass while lane 0 of another
// warp was still finishing a section it runs alone (an atomic reservation,
// a control-block copy) and read shared values before they were written.
__device__ __forceinline__ void cta_sync()
{
    asm volatile("barrier.sync 0;" ::: "memory");
}

// ------------------------------------------------------------ primitives

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const unsigned int *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier number gen (0, 1, ... in every CTA) of a launch, with a
// bounded wait: returns false (and sets the sticky error flag) if the other
// CTAs do not arrive within limit_ns (20 s unless a test shortens it), or
// if another CTA gave up.  The host zeroes the counter before each launch,
// so barrier gen is complete once it reaches (gen + 1) x CTAs; a CTA
// arrives with a release add that returns nothing (the CTA's writes,
// ordered before it by the CTA barrier, become visible with it) and waits
// with acquire loads.
__device__ __forceinline__ bool grid_sync(Barrier *b, unsigned nblocks, unsigned long long limit_ns, uint32_t gen)
{
    __shared__ int s_ok;
    cta_sync();
    if (threadIdx.x == 0) {
        int ok = 1;
        if (nblocks > 1) {
            const unsigned long long target = ((unsigned long long)gen + 1ull) * nblocks;
            asm volatile("red.release.gpu.global.add.u64 [%0], %1;" :: "l"(&b->count), "l"(1ull) : "memory");
            unsigned long long t0 = 0;
            for (unsigned spins = 1; ld_acquire_u64(&b->count) < target; spins++) {
                if ((spins & 255u) == 0u) {
                    if (ld_acquire_u32(&b->err)) { ok = 0; break; }
                    const unsigned long long now = globaltimer_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > limit_ns) {
                        atomicExch(&b->err, 1u);
                        ok = 0;
                        break;
                    }
                }
            }
            __threadfence();
        }
        s_ok = ok;
    }
    cta_sync();
    return s_ok != 0;
}

__device__ __forceinline__ uint32_t nib(uint32_t word, uint32_t v) { return (word >> ((v & 7u) * 4u)) & 0xFu; }

// effective value during a round: fresh variables (claimed this round) read
// as unassigned
__device__ __forceinline__ uint32_t eff_val(uint32_t code, uint32_t fresh_cur)
{
    return (code & fresh_cur) ? 0u : (code & 3u);
}

__device__ __forceinline__ uint32_t global_val(const Dev &D, uint32_t v, uint32_t fresh_cur)
{
    return eff_val(nib(__ldcg(D.asg + (v >> 3)), v), fresh_cur);
}

// words of a dependency bitmap that can be non-zero for a variable at level L
__device__ __forceinline__ uint32_t deps_words(const Dev &D, uint32_t L)
{
    uint32_t w = (L + 63u) >> 6;
    return w < D.WW ? w : D.WW;
}

// bit of level L (levels >= Wlevels share the overflow bit Wlevels-1)
__device__ __forceinline__ uint32_t level_bit(const Dev &D, uint32_t L)
{
    return L < D.Wlevels ? L - 1u : D.Wlevels - 1u;
}

__device__ __forceinline__ uint32_t lit_at(const Dev &D, uint32_t idx)
{
    return idx < D.lits_static ? __ldg(D.lits + idx) : __ldcg(D.lits + idx);
}

// literal q (without end flag) and length of nogood `id`
__device__ __forceinline__ uint32_t ng_lit(const Dev &D, uint32_t id, uint32_t q)
{
    if (id & BUCKET_ID) {
        const uint32_t L = ((id >> 27) & 15u) + 1u, k = id & 0x7FFFFFFu;
        return __ldg(D.lits + D.bk_base[L] + (size_t)q * D.bk_n[L] + k);
    }
    return lit_at(D, id + q) & ~END_BIT;
}

__device__ __forceinline__ uint32_t ng_len(const Dev &D, uint32_t id)
{
    if (id & BUCKET_ID) return ((id >> 27) & 15u) + 1u;
    uint32_t n = 1;
    while (!(lit_at(D, id + n - 1u) & END_BIT)) n++;
    return n;
}

// ---------------------------------------------------------------- views

// The CTA's view (0 unassigned, 1 true, 2 false; 2 bits or one byte per
// entry) of the atoms [0, na_v) and of the auxiliary variables
// [auxlo, auxlo + auxn), which follow the atoms at entry aux_base (a
// multiple of 16).
struct View {
    volatile uint32_t *w;
    uint32_t na_v, aux_base, auxlo, auxn;
    bool bytes;

    // entry of v in the view, or 0xFFFFFFFF if v is not in it
    __device__ __forceinline__ uint32_t index(uint32_t v) const
    {
        if (v < na_v) return v;
        uint32_t k = v - auxlo;
        return k < auxn ? aux_base + k : 0xFFFFFFFFu;
    }
    // variable of entry i
    __device__ __forceinline__ uint32_t var(uint32_t i) const { return i < aux_base ? i : i - aux_base + auxlo; }
    __device__ __forceinline__ uint32_t get(uint32_t i) const
    {
        if (bytes) return reinterpret_cast<volatile const uint8_t *>(w)[i];
        return (w[i >> 4] >> (2u * (i & 15u))) & 3u;
    }
    // set entry i to val; true if it was unassigned
    __device__ __forceinline__ bool put(uint32_t i, uint32_t val) const
    {
        if (bytes) {
            volatile uint8_t *b = reinterpret_cast<volatile uint8_t *>(w);
            const uint32_t old = b[i];
            b[i] = (uint8_t)val;
            return old == 0u;
        }
        uint32_t sh = 2u * (i & 15u);
        uint32_t old = atomicOr((uint32_t *)(w + (i >> 4)), val << sh);
        return ((old >> sh) & 3u) == 0u;
    }
    __device__ __forceinline__ void clear(uint32_t i) const
    {
        if (bytes) reinterpret_cast<volatile uint8_t *>(w)[i] = 0;
        else atomicAnd((uint32_t *)(w + (i >> 4)), ~(3u << (2u * (i & 15u))));
    }
};

__device__ __forceinline__ uint32_t view_val(const Dev &D, const View &V, uint32_t v, uint32_t fresh_cur)
{
    uint32_t i = V.index(v);
    if (i != 0xFFFFFFFFu) return V.get(i);
    return global_val(D, v, fresh_cur);
}

__device__ __forceinline__ bool view_set(const View &V, uint32_t v, uint32_t val)
{
    uint32_t i = V.index(v);
    return i != 0xFFFFFFFFu && V.put(i, val);
}

__device__ __forceinline__ void view_clear(const View &V, uint32_t v)
{
    uint32_t i = V.index(v);
    if (i != 0xFFFFFFFFu) V.clear(i);
}

// 2-bit effective values of the 8 variables of one global code word
__device__ __forceinline__ uint32_t pack8(uint32_t word, uint32_t fresh_cur)
{
    uint32_t m = 0;
#pragma unroll
    for (uint32_t q = 0; q < 8u; q++) m |= eff_val((word >> (4u * q)) & 0xFu, fresh_cur) << (2u * q);
    return m;
}

// effective values of the 4 variables at nibbles sh..sh+3 of code words
// (a, b), one per byte
__device__ __forceinline__ uint32_t bytes4(uint32_t a, uint32_t b, uint32_t sh, uint32_t fresh_cur)
{
    const uint32_t x = (uint32_t)((((unsigned long long)b << 32) | a) >> (4u * sh));
    uint32_t m = 0;
#pragma unroll
    for (uint32_t q = 0; q < 4u; q++) m |= eff_val((x >> (4u * q)) & 0xFu, fresh_cur) << (8u * q);
    return m;
}

// Byte view: one view word holds 4 variables (half a global code word).
__device__ __forceinline__ void view_reload_bytes(const Dev &D, const View &V, uint32_t fresh_cur)
{
    const uint32_t wa = (V.na_v + 3u) >> 2, wx = (V.auxn + 3u) >> 2;
    for (uint32_t k = threadIdx.x; k < wa; k += blockDim.x) {
        const uint32_t v0 = 4u * k;
        uint32_t m = bytes4(__ldcg(D.asg + (v0 >> 3)), 0u, v0 & 7u, fresh_cur);
        const uint32_t valid = V.na_v - v0;
        if (valid < 4u) m &= (1u << (8u * valid)) - 1u;
        V.w[k] = m;
    }
    for (uint32_t k = wa + threadIdx.x; k < V.aux_base / 4u; k += blockDim.x) V.w[k] = 0u;
    for (uint32_t k = threadIdx.x; k < wx; k += blockDim.x) {
        const uint32_t v0 = V.auxlo + 4u * k, w0 = v0 >> 3;
        const uint32_t a = __ldcg(D.asg + w0);
        const uint32_t b = w0 + 1u < D.asg_words ? __ldcg(D.asg + w0 + 1u) : 0u;
        uint32_t m = bytes4(a, b, v0 & 7u, fresh_cur);
        const uint32_t valid = V.auxn - 4u * k;
        if (valid < 4u) m &= (1u << (8u * valid)) - 1u;
        V.w[V.aux_base / 4u + k] = m;
    }
}

// Rebuild the whole view from the global codes (fresh claims read as
// unassigned); one 2-bit view word holds 16 variables = two global code
// words.
__device__ __forceinline__ void view_reload(const Dev &D, const View &V, uint32_t fresh_cur)
{
    if (V.bytes) {
        view_reload_bytes(D, V, fresh_cur);
        return;
    }
    const uint32_t wa = (V.na_v + 15u) >> 4, wx = (V.auxn + 15u) >> 4;
    for (uint32_t k = threadIdx.x; k < wa; k += blockDim.x) {
        uint32_t lo = __ldcg(D.asg + 2u * k), hi = 2u * k + 1u < D.asg_words ? __ldcg(D.asg + 2u * k + 1u) : 0u;
        uint32_t m = pack8(lo, fresh_cur) | (pack8(hi, fresh_cur) << 16);
        uint32_t valid = V.na_v - 16u * k;    // entries of this word that are atoms
        if (valid < 16u) m &= (1u << (2u * valid)) - 1u;
        V.w[k] = m;
    }
    for (uint32_t k = threadIdx.x; k < wx; k += blockDim.x) {
        // variables auxlo + 16k .. +15: spread over up to three code words
        const uint32_t v0 = V.auxlo + 16u * k;
        const uint32_t w0 = v0 >> 3, sh = v0 & 7u;
        uint32_t a = __ldcg(D.asg + w0);
        uint32_t b = w0 + 1u < D.asg_words ? __ldcg(D.asg + w0 + 1u) : 0u;
        uint32_t c = w0 + 2u < D.asg_words ? __ldcg(D.asg + w0 + 2u) : 0u;
        // 24 nibbles starting at a; take 16 from nibble sh
        unsigned long long lo64 = ((unsigned long long)b << 32) | a;
        uint32_t first8 = (uint32_t)(lo64 >> (4u * sh));
        unsigned long long hi64 = ((unsigned long long)c << 32) | b;
        uint32_t next8 = (uint32_t)(hi64 >> (4u * sh));
        uint32_t m = pack8(first8, fresh_cur) | (pack8(next8, fresh_cur) << 16);
        uint32_t valid = V.auxn - 16u * k;
        if (valid < 16u) m &= (1u << (2u * valid)) - 1u;
        V.w[V.aux_base / 16u + k] = m;
    }
}

// ---------------------------------------------------------------- claims

// Claim the complement of an unassigned literal: 0 won, 1 agreed, 2 clash.
__device__ __forceinline__ int claim_var(uint32_t *asg, uint32_t v, uint32_t valbit, uint32_t fresh_cur)
{
    uint32_t sh = (v & 7u) * 4u;
    uint32_t old = atomicOr(asg + (v >> 3), (valbit | fresh_cur) << sh);
    uint32_t ov = (old >> sh) & 3u;
    if (ov == 0u) return 0;
    if (ov & valbit) return 1;
    return 2;
}

struct SweepCtx {
    const Dev *D;
    View V;
    uint32_t fresh;        // fresh bit of the current round
    uint32_t cdl;          // level of new claims
    uint32_t tbase;        // trail index of this phase's first claim
    Acc *acc;              // this phase's accumulators
    bool do_claim;
    bool use_view;
    uint32_t cta;          // this CTA's part of the static partition
    uint32_t gw, nw;       // warp index and warp count of the solving group
    // inside a sweep: claims are listed in shared memory and copied to the
    // trail once at the end of the sweep (one global atomic per CTA)
    bool listed = false;
};

constexpr uint32_t CLAIM_BUF = 256;
// first unit of each bucket in this CTA's part of the partition (units of
// unit_groups(L) groups of 32 nogoods); entry BUCKET_MAX + 1 = all units
__shared__ uint32_t s_ubase[BUCKET_MAX + 2];
// this CTA's range [s_krange[L][0], s_krange[L][1]) of bucket L
__shared__ uint32_t s_krange[BUCKET_MAX + 1][2];
__shared__ uint32_t s_claims[CLAIM_BUF];
__shared__ unsigned int s_ncl, s_cbase;
// next bucket unit of the CTA's queue in the current sweep (solver sweeps;
// sweeps that do not claim alternate between s_unit2[0] and s_unit2[1])
__shared__ unsigned int s_unit, s_unit2[2];
// CTA 0, thread 0: time in the sweeps on long and learned nogoods and on
// the buckets
__shared__ unsigned long long s_tlearned, s_tbuckets;
// the same two parts, max over the CTA's warps in the current sweep
__shared__ unsigned long long s_wmax[2];
__device__ __forceinline__ void report_conflict(const SweepCtx &X, uint32_t id, uint32_t len)
{
    const unsigned long long key = ((unsigned long long)len << 32) | id;
    atomicMin(&X.acc->ckey, key);
    atomicMin(&X.acc->cslot[id % 3u], key);    // read only with several conflicts per round
}

// Record a won claim: trail slot, level, reason.
__device__ __forceinline__ void record_claim(const SweepCtx &X, uint32_t v, uint32_t valbit, uint32_t id)
{
    const Dev &D = *X.D;
    D.dl[v] = (int32_t)X.cdl;
    D.reason[v] = id;
    const uint32_t entry = v | (valbit == V_F ? TRAIL_F : 0u);
    if (X.listed) {
        const uint32_t i = atomicAdd(&s_ncl, 1u);
        if (i < CLAIM_BUF) { s_claims[i] = entry; return; }
    }
    uint32_t pos = X.tbase + atomicAdd(&X.acc->nclaim, 1u);
    if (pos < D.nv) {
        D.trail[pos] = entry;
        if (D.tpos) D.tpos[v] = pos;
    }
}

// One lane per literal u of a reason (has = false on lanes holding none):
// the warp ORs Deps[u] over lanes with level > 1 and writes Deps[x]
// (Section 4.2, mk_dl_bitmap).  All 32 lanes call it.
__device__ __forceinline__ void warp_or_deps(const SweepCtx &X, bool has, uint32_t u, uint32_t x,
                                             int writer, bool accumulate)
{
    const Dev &D = *X.D;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t L = X.cdl;
    const uint32_t nw = deps_words(D, L);
    // a decision's bitmap is the bit of its own level: with the level, the
    // reason tells whether the bitmap words need loading at all (a learned
    // nogood of fwd-learning holds decisions only)
    int32_t Lu = has ? __ldcg(D.dl + u) : 0;
    const uint32_t ru = has ? __ldcg(D.reason + u) : 0u;
    uint32_t nwu = (has && Lu > 1) ? deps_words(D, (uint32_t)Lu) : 0u;
    const bool dec = has && Lu > 1 && ru == R_DECISION;
    const uint32_t dbit = level_bit(D, dec ? (uint32_t)Lu : L);
    for (uint32_t w = 0; w < nw; w++) {
        unsigned long long c = w >= nwu ? 0ull
                             : dec ? (w == (dbit >> 6) ? (1ull << (dbit & 63u)) : 0ull)
                             : __ldcg(D.deps + (size_t)u * D.WW + w);
        unsigned lo = __reduce_or_sync(FULL_MASK, (unsigned)c);
        unsigned hi = __reduce_or_sync(FULL_MASK, (unsigned)(c >> 32));
        if ((int)lane == writer) {
            unsigned long long m = ((unsigned long long)hi << 32) | lo;
            unsigned long long *dst = D.deps + (size_t)x * D.WW + w;
            *dst = accumulate ? (__ldcg(dst) | m) : m;
        }
    }
}

// value of a literal's variable during the sweep (view, else global codes)
__device__ __forceinline__ uint32_t lit_val(const SweepCtx &X, uint32_t l)
{
    return X.use_view ? view_val(*X.D, X.V, l >> 1, X.fresh) : global_val(*X.D, l >> 1, X.fresh);
}

// Dependency bitmap of x from the other variables of one lane's nogood
// (var), OR over those with level > 1 (Section 4.2, mk_dl_bitmap).
template <int L>
__device__ __forceinline__ void lane_deps(const SweepCtx &X, const uint32_t (&var)[L], uint32_t x)
{
    const Dev &D = *X.D;
    const uint32_t nw = deps_words(D, X.cdl);
    int32_t Lu[L];
#pragma unroll
    for (int q = 0; q < L; q++) Lu[q] = var[q] == x ? 0 : __ldcg(D.dl + var[q]);
    for (uint32_t w = 0; w < nw; w++) {
        unsigned long long acc = 0;
#pragma unroll
        for (int q = 0; q < L; q++) {
            uint32_t u = var[q];
            if (Lu[q] > 1 && w < deps_words(D, (uint32_t)Lu[q])) acc |= __ldcg(D.deps + (size_t)u * D.WW + w);
        }
        D.deps[(size_t)x * D.WW + w] = acc;
    }
}

// Dependency bitmaps (Section 4.2, mk_dl_bitmap) of every claim of a group of
// 32 nogoods at once: the claims take equal shares of the warp's lanes (32 / p2
// lanes each, p2 the claim count rounded up to a power of two), and the lanes
// of a claim split its bitmap words, so the group costs the two dependent
// loads of one claim whatever the number of claims.  All 32 lanes call it; won:
// this lane's nogood claimed x; tl: its literals as view entries.  Returns
// whether the group made a claim.
template <int L>
__device__ __forceinline__ bool group_claims(const SweepCtx &X, bool won, const uint32_t (&tl)[L], uint32_t x)
{
    const Dev &D = *X.D;
    const unsigned m = __ballot_sync(FULL_MASK, won);
    if (!m) return false;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t nc = (uint32_t)__popc(m);
    uint32_t p2 = 1u;
    while (p2 < nc) p2 <<= 1;
    const uint32_t gs = 32u / p2, c = lane / gs, sub = lane % gs;
    // the lane of the c-th claim
    unsigned mm = m;
    for (uint32_t i = 0; i < c && mm; i++) mm &= mm - 1u;
    const int src = mm ? __ffs(mm) - 1 : 0;
    uint32_t var[L];
#pragma unroll
    for (int q = 0; q < L; q++) var[q] = X.V.var(__shfl_sync(FULL_MASK, tl[q], src) >> 2);
    const uint32_t xs = __shfl_sync(FULL_MASK, x, src);
    if (c >= nc) return true;
    const uint32_t nw = deps_words(D, X.cdl);
    int32_t Lu[L];
#pragma unroll
    for (int q = 0; q < L; q++) Lu[q] = var[q] != xs ? __ldcg(D.dl + var[q]) : 0;
    for (uint32_t w = sub; w < nw; w += gs) {
        unsigned long long acc = 0;
#pragma unroll
        for (int q = 0; q < L; q++)
            if (Lu[q] > 1 && 64u * w < (uint32_t)Lu[q]) acc |= __ldcg(D.deps + (size_t)var[q] * D.WW + w);
        D.deps[(size_t)xs * D.WW + w] = acc;
    }
    return true;
}

// U groups of 32 nogoods of bucket L, lane = nogood k0 + t*stride + lane.
// All literals are loaded (coalesced, one row per literal position) and
// their values gathered before any is classified: a nogood is satisfied if
// some literal's complement holds, violated if all hold, unit if exactly one
// is unassigned and the rest hold (Section 2).  Repeats while a claim of
// this warp changed the view.
template <int L, int U>
__device__ __forceinline__ void bucket_tasks(const SweepCtx &X, uint32_t k0, uint32_t k1, uint32_t stride)
{
    const Dev &D = *X.D;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t *base = D.lits + D.bk_base[L];
    const uint32_t n = D.bk_n[L];
    uint32_t lit[U][L];
#pragma unroll
    for (int t = 0; t < U; t++) {
        const uint32_t k = k0 + (uint32_t)t * stride + lane;
#pragma unroll
        for (int q = 0; q < L; q++) lit[t][q] = k < k1 ? __ldg(base + (size_t)q * n + k) : PAD_LIT;
    }
    for (int pass = 0; pass < 2; pass++) {
        uint32_t val[U][L];
#pragma unroll
        for (int t = 0; t < U; t++)
#pragma unroll
            for (int q = 0; q < L; q++) val[t][q] = lit[t][q] == PAD_LIT ? 0u : lit_val(X, lit[t][q]);
        bool pub = false;
#pragma unroll
        for (int t = 0; t < U; t++) {
            const uint32_t k = k0 + (uint32_t)t * stride + lane;
            if (k >= k1) continue;
            bool sat = false;
            uint32_t n_un = 0, ul = 0;
#pragma unroll
            for (int q = 0; q < L; q++) {
                uint32_t v = val[t][q];
                sat |= v == ((lit[t][q] & 1u) ? V_T : V_F);
                if (v == 0u) { n_un++; ul = lit[t][q]; }
            }
            if (sat || n_un > 1u) continue;
            const uint32_t id = bucket_nogood_id((uint32_t)L, k);
            if (n_un == 0u) { report_conflict(X, id, (uint32_t)L); continue; }
            if (!X.do_claim) { atomicAdd(&X.acc->flag, 1u); continue; }
            const uint32_t x = ul >> 1, valbit = (ul & 1u) ? V_T : V_F;
            const int r = claim_var(D.asg, x, valbit, X.fresh);
            if (r == 2) { report_conflict(X, id, (uint32_t)L); continue; }
            if (r != 0) continue;
            record_claim(X, x, valbit, id);
            if (X.cdl > 1u) {
                uint32_t var[L];
#pragma unroll
                for (int q = 0; q < L; q++) var[q] = lit[t][q] >> 1;
                lane_deps<L>(X, var, x);
            }
            if (X.use_view) {
                __threadfence_block();
                pub |= view_set(X.V, x, valbit);
            }
        }
        if (!X.use_view || !X.do_claim || !__any_sync(FULL_MASK, pub)) break;
    }
}

// Contribution of one translated literal (entry << 2 | xmask) to its
// nogood's count: t = value ^ xmask is 1 if the literal holds, 2 if its
// complement holds, 0 or 3 if unassigned; the byte of 0x01100001 at t is
// 0, 16 or 1.  Over at most 15 literals the low byte of the sum is
// >= 16: satisfied; 0: violated; 1: unit; 2..15: two or more unassigned.
template <bool BYTES>
__device__ __forceinline__ uint32_t tlit_val(const View &V, uint32_t tl)
{
    const uint32_t i = tl >> 2;
    if (BYTES) return reinterpret_cast<volatile const uint8_t *>(V.w)[i];
    return V.w[i >> 4] >> (2u * (i & 15u));
}
template <bool BYTES>
__device__ __forceinline__ uint32_t tlit_count(const View &V, uint32_t tl)
{
    return __byte_perm(0x01100001u, 0u, (tlit_val<BYTES>(V, tl) ^ tl) & 3u);
}

// a if p, else b, as a predicated select (the group loop below picks a
// row of its register arrays with these, which keeps the arrays in
// registers)
__device__ __forceinline__ uint32_t sel_if(bool p, uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\tselp.b32 %0, %1, %2, q;\n\t}"
        : "=r"(r) : "r"(a), "r"(b), "r"((uint32_t)p));
    return r;
}

// The literals of one lane's nogood of a length-L bucket, as view entries.
template <int L>
struct Row { uint32_t q[L]; };

// The claim path of one group of 32 nogoods of bucket L, taken when the
// count found some lane's nogood unit or violated (cand): that lane
// classifies it again from the current view (a claim of this CTA may have
// changed it since the count), reports a violation, or claims the variable
// of its one unassigned literal; then the group's claims get their
// dependency bitmaps and are published in the view.  All 32 lanes call it.  Returns whether
// this lane claimed.
template <int L, bool BYTES>
__device__ __forceinline__ bool group_claim_path(const SweepCtx &X, const Row<L> &r, uint32_t k, bool cand)
{
    const Dev &D = *X.D;
    bool won = false;
    uint32_t e = 0, x = 0, valbit = 0;
    if (cand) {
        const uint32_t id = bucket_nogood_id((uint32_t)L, k);
        bool sat = false;
        uint32_t n_un = 0, ul = 0;
#pragma unroll
        for (int q = 0; q < L; q++) {
            const uint32_t tv = (tlit_val<BYTES>(X.V, r.q[q]) ^ r.q[q]) & 3u;
            sat |= tv == 2u;
            if (tv == 0u || tv == 3u) { n_un++; ul = r.q[q]; }
        }
        if (!sat && n_un == 0u) {
            report_conflict(X, id, (uint32_t)L);
        } else if (!sat && n_un == 1u) {
            if (!X.do_claim) {
                atomicAdd(&X.acc->flag, 1u);
            } else {
                e = ul >> 2;
                x = X.V.var(e);
                valbit = (ul & 1u) ? V_T : V_F;
                const int rc = claim_var(D.asg, x, valbit, X.fresh);
                if (rc == 2) report_conflict(X, id, (uint32_t)L);
                else if (rc == 0) { record_claim(X, x, valbit, id); won = true; }
            }
        }
    }
    if (L > 8 && won && X.cdl > 1u) {
        // long buckets (few claims): the claiming lane alone
        uint32_t var[L];
#pragma unroll
        for (int q = 0; q < L; q++) var[q] = X.V.var(r.q[q] >> 2);
        lane_deps<L>(X, var, x);
    }
    if (L <= 8 && X.cdl > 1u) {
        // bitmaps of this group's claims, all at once
        if (group_claims<L>(X, won, r.q, x)) {
            __threadfence_block();
            __syncwarp();
        }
    }
    if (won) {
        __threadfence_block();
        X.V.put(e, valbit);
    }
    return won;
}

// bucket_tasks over the translated copy of the store (view modes PACKED
// and BYTES): every literal is in the view, one shared-memory load and
// three integer operations classify it.  Lanes past the end of the range
// load the range's last nogood and drop the result.
template <int L, int U, bool BYTES>
__device__ __forceinline__ void bucket_tasks_view(const SweepCtx &X, uint32_t k0, uint32_t k1)
{
    const Dev &D = *X.D;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t *base = D.vlits + D.bk_base[L];
    const uint32_t n = D.bk_n[L];
    uint32_t lit[U][L];
#pragma unroll
    for (int t = 0; t < U; t++) {
        const uint32_t k = min(k0 + (uint32_t)t * 32u + lane, k1 - 1u);
#pragma unroll
        for (int q = 0; q < L; q++) lit[t][q] = __ldg(base + (size_t)q * n + k);
    }
    for (int pass = 0; pass < 2; pass++) {
        uint32_t cnt[U];
#pragma unroll
        for (int t = 0; t < U; t++) {
            cnt[t] = 0u;
#pragma unroll
            for (int q = 0; q < L; q++) cnt[t] += tlit_count<BYTES>(X.V, lit[t][q]);
        }
        // the groups with a nogood that is violated or unit by the count go
        // through the claim path, one at a time; the path is written out
        // once (the group's row is selected into registers), not once per
        // group, so the loops above stay small enough to stay in the
        // instruction cache from one round to the next
        unsigned cm = 0u;
#pragma unroll
        for (int t = 0; t < U; t++) {
            const uint32_t k = k0 + (uint32_t)t * 32u + lane;
            if (__any_sync(FULL_MASK, k < k1 && (cnt[t] & 0xFFu) <= 1u)) cm |= 1u << t;
        }
        bool pub = false;
        while (cm) {
            const int t = __ffs(cm) - 1;
            cm &= cm - 1u;
            Row<L> r;
            uint32_t c = cnt[0];
#pragma unroll
            for (int q = 0; q < L; q++) r.q[q] = lit[0][q];
#pragma unroll
            for (int tt = 1; tt < U; tt++) {
                c = sel_if(t == tt, cnt[tt], c);
#pragma unroll
                for (int q = 0; q < L; q++) r.q[q] = sel_if(t == tt, lit[tt][q], r.q[q]);
            }
            const uint32_t k = k0 + (uint32_t)t * 32u + lane;
            pub |= group_claim_path<L, BYTES>(X, r, k, k < k1 && (c & 0xFFu) <= 1u);
        }
        if (!X.do_claim || !__any_sync(FULL_MASK, pub)) break;
    }
}


template <bool BYTES>
__device__ __forceinline__ void run_unit_view(const SweepCtx &X, uint32_t L, uint32_t k0, uint32_t k1)
{
    switch (L) {
    case 2: bucket_tasks_view<2, unit_groups(2), BYTES>(X, k0, k1); break;
    case 3: bucket_tasks_view<3, unit_groups(3), BYTES>(X, k0, k1); break;
    case 4: bucket_tasks_view<4, unit_groups(4), BYTES>(X, k0, k1); break;
    case 5: bucket_tasks_view<5, unit_groups(5), BYTES>(X, k0, k1); break;
    case 6: bucket_tasks_view<6, unit_groups(6), BYTES>(X, k0, k1); break;
    case 7: bucket_tasks_view<7, unit_groups(7), BYTES>(X, k0, k1); break;
    case 8: bucket_tasks_view<8, unit_groups(8), BYTES>(X, k0, k1); break;
    case 9: bucket_tasks_view<9, unit_groups(9), BYTES>(X, k0, k1); break;
    case 10: bucket_tasks_view<10, unit_groups(10), BYTES>(X, k0, k1); break;
    case 11: bucket_tasks_view<11, unit_groups(11), BYTES>(X, k0, k1); break;
    case 12: bucket_tasks_view<12, unit_groups(12), BYTES>(X, k0, k1); break;
    case 13: bucket_tasks_view<13, unit_groups(13), BYTES>(X, k0, k1); break;
    case 14: bucket_tasks_view<14, unit_groups(14), BYTES>(X, k0, k1); break;
    default: bucket_tasks_view<15, unit_groups(15), BYTES>(X, k0, k1); break;
    }
}

__device__ __forceinline__ void run_unit(const SweepCtx &X, uint32_t L, uint32_t k0, uint32_t k1)
{
    switch (L) {
    case 2: bucket_tasks<2, unit_groups(2)>(X, k0, k1, 32u); break;
    case 3: bucket_tasks<3, unit_groups(3)>(X, k0, k1, 32u); break;
    case 4: bucket_tasks<4, unit_groups(4)>(X, k0, k1, 32u); break;
    case 5: bucket_tasks<5, unit_groups(5)>(X, k0, k1, 32u); break;
    case 6: bucket_tasks<6, unit_groups(6)>(X, k0, k1, 32u); break;
    case 7: bucket_tasks<7, unit_groups(7)>(X, k0, k1, 32u); break;
    case 8: bucket_tasks<8, unit_groups(8)>(X, k0, k1, 32u); break;
    case 9: bucket_tasks<9, unit_groups(9)>(X, k0, k1, 32u); break;
    case 10: bucket_tasks<10, unit_groups(10)>(X, k0, k1, 32u); break;
    case 11: bucket_tasks<11, unit_groups(11)>(X, k0, k1, 32u); break;
    case 12: bucket_tasks<12, unit_groups(12)>(X, k0, k1, 32u); break;
    case 13: bucket_tasks<13, unit_groups(13)>(X, k0, k1, 32u); break;
    case 14: bucket_tasks<14, unit_groups(14)>(X, k0, k1, 32u); break;
    default: bucket_tasks<15, unit_groups(15)>(X, k0, k1, 32u); break;
    }
}

// A nogood of any length, one warp, lanes over literals (ballot/popc),
// stopping once it is satisfied or has two unassigned literals; literals are
// checked against the global codes, 128 at a time (four loads and their
// gathers in flight before the first ballot).
// Watched literals (Algorithm 2, which uses them for long learned nogoods
// as well): *wslot holds two positions of the nogood (wp).  If neither watched
// literal holds -- one's complement is assigned, or both are unassigned --
// the nogood is neither unit nor violated, and two checks settle it (the
// caller's); otherwise this scan runs and moves the watches to literals that do
// not hold (the complement found, or the first unassigned ones).  Every such
// nogood is checked in list rounds and sweeps, and before each fixpoint (narrow
// rounds check none), whatever was assigned, so the watches need no per-variable
// lists and stay valid across backjumps.  Equal positions (a nogood of one literal)
// always scan.
__device__ __forceinline__ void classify_long(const SweepCtx &X, uint32_t id, unsigned long long &checks,
                                              uint2 *wslot, uint2 wp)
{
    const Dev &D = *X.D;
    const uint32_t lane = threadIdx.x & 31u;
    bool any_opp = false, done = false;
    uint32_t n_un = 0, ulit = 0, len = 0;
    uint32_t opos = 0, upos0 = 0, upos1 = 0;   // positions: a complement found, the first unassigned ones
    for (uint32_t off = id; !done && off < D.lits_cap; off += 128u) {
        uint32_t w[4], code[4];
#pragma unroll
        for (int q = 0; q < 4; q++) w[q] = lit_at(D, off + 32u * q + lane);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            uint32_t v = (w[q] & ~END_BIT) >> 1;
            code[q] = v < D.nv ? nib(__ldcg(D.asg + (v >> 3)), v) : 0u;
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (done) break;
            const uint32_t pos0 = off - id + 32u * (uint32_t)q;
            unsigned Bend = __ballot_sync(FULL_MASK, (w[q] & END_BIT) != 0u);
            unsigned valid = Bend ? ((2u << (__ffs(Bend) - 1)) - 1u) : FULL_MASK;
            uint32_t l = w[q] & ~END_BIT;
            bool mine = ((valid >> lane) & 1u) && (l >> 1) < D.nv;
            uint32_t val = mine ? eff_val(code[q], X.fresh) : 0u;
            bool opp = mine && val == ((l & 1u) ? V_T : V_F);
            bool un = mine && val == 0u;
            unsigned Bopp = __ballot_sync(FULL_MASK, opp);
            unsigned Bun = __ballot_sync(FULL_MASK, un);
            uint32_t first_un = __shfl_sync(FULL_MASK, l, Bun ? __ffs(Bun) - 1 : 0);
            if (Bun && n_un == 0) ulit = first_un;
            if (Bun) {
                const uint32_t b0 = (uint32_t)__ffs(Bun) - 1u;
                const unsigned rest = Bun & (Bun - 1u);
                if (n_un == 0) {
                    upos0 = pos0 + b0;
                    if (rest) upos1 = pos0 + (uint32_t)__ffs(rest) - 1u;
                } else if (n_un == 1) {
                    upos1 = pos0 + b0;
                }
            }
            if (Bopp) opos = pos0 + (uint32_t)__ffs(Bopp) - 1u;
            n_un += (uint32_t)__popc(Bun);
            len += (uint32_t)__popc(valid);
            checks += (uint32_t)__popc(valid);
            if (Bopp) { any_opp = true; done = true; }
            else if (Bend || n_un > 1) done = true;
        }
    }
    if (wslot && lane == 0 && (any_opp || n_un > 0)) {
        // the watches move to literals that do not hold
        uint2 nw;
        if (any_opp) nw = make_uint2(opos, n_un ? upos0 : (wp.x != opos ? wp.x : wp.y));
        else if (n_un > 1) nw = make_uint2(upos0, upos1);
        else nw = make_uint2(upos0, wp.x != upos0 ? wp.x : wp.y);
        if (nw.x != nw.y) *wslot = nw;
    }
    if (any_opp) return;
    int won = 0;
    if (lane == 0) {
        if (n_un == 0) {
            report_conflict(X, id, len);
        } else if (n_un == 1) {
            if (!X.do_claim) {
                atomicAdd(&X.acc->flag, 1u);
            } else {
                uint32_t v = ulit >> 1, valbit = (ulit & 1u) ? V_T : V_F;
                int r = claim_var(D.asg, v, valbit, X.fresh);
                if (r == 0) { record_claim(X, v, valbit, id); won = 1; }
                else if (r == 2) report_conflict(X, id, len);
            }
        }
    }
    won = __shfl_sync(FULL_MASK, won, 0);
    if (!won) return;
    const uint32_t x = ulit >> 1;
    if (X.cdl > 1u) {
        __threadfence_block();
        bool first = true;
        for (uint32_t off = id; off < D.lits_cap; off += 32u) {
            uint32_t w2 = lit_at(D, off + lane);
            unsigned Bend = __ballot_sync(FULL_MASK, (w2 & END_BIT) != 0u);
            unsigned valid = Bend ? ((2u << (__ffs(Bend) - 1)) - 1u) : FULL_MASK;
            uint32_t u2 = (w2 & ~END_BIT) >> 1;
            bool has = ((valid >> lane) & 1u) && u2 != x && u2 < D.nv;
            warp_or_deps(X, has, u2, x, 0, !first);
            first = false;
            if (Bend) break;
        }
    }
    if (lane == 0 && X.use_view) {
        __threadfence_block();
        view_set(X.V, x, (ulit & 1u) ? V_T : V_F);
    }
}

// OR into acc of word w of the bitmaps of variables u[0 .. C) other than x.
// The words are loaded beside the levels that say whether they count.
template <int C>
__device__ __forceinline__ unsigned long long deps_or(const Dev &D, const uint32_t (&u)[C], uint32_t x, uint32_t w)
{
    int32_t lev[C];
    unsigned long long word[C], acc = 0;
#pragma unroll
    for (int q = 0; q < C; q++) {
        lev[q] = u[q] != x ? __ldcg(D.dl + u[q]) : 0;
        word[q] = u[q] != x ? __ldcg(D.deps + (size_t)u[q] * D.WW + w) : 0ull;
    }
#pragma unroll
    for (int q = 0; q < C; q++)
        if (lev[q] > 1 && 64u * w < (uint32_t)lev[q]) acc |= word[q];
    return acc;
}

// Dependency bitmap (Section 4.2, mk_dl_bitmap) of variable x, assigned by
// bucket nogood id, by a group of `lanes` lanes, this one the sub-th: each
// takes every lanes-th word.  vars: the nogood's variables if it has at most eight literals and
// they are known, else null.
__device__ __forceinline__ void narrow_deps(const Dev &D, uint32_t x, uint32_t id, const uint4 *vars, uint32_t nw, uint32_t sub,
                                            uint32_t lanes)
{
    const uint32_t L = ((id >> 27) & 15u) + 1u, n = D.bk_n[L];
    if (vars && L <= 8u) {
        const uint4 v = vars[0];
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
        if (L <= 4u) {
            for (uint32_t w = sub; w < nw; w += lanes) D.deps[(size_t)x * D.WW + w] = deps_or<4>(D, u, x, w);
        } else {
            const uint4 t = vars[1];
            const uint32_t u2[4] = {t.x, t.y, t.z, t.w};
            for (uint32_t w = sub; w < nw; w += lanes) D.deps[(size_t)x * D.WW + w] = deps_or<4>(D, u, x, w) | deps_or<4>(D, u2, x, w);
        }
        return;
    }
    const uint32_t *base = D.lits + D.bk_base[L] + (id & 0x7FFFFFFu);
    for (uint32_t w = sub; w < nw; w += lanes) {
        unsigned long long acc = 0;
        for (uint32_t q0 = 0; q0 < L; q0 += 5u) {
            uint32_t u[5];
#pragma unroll
            for (uint32_t q = 0; q < 5u; q++) u[q] = q0 + q < L ? __ldg(base + (size_t)(q0 + q) * n) >> 1 : x;
            acc |= deps_or<5>(D, u, x, w);
        }
        D.deps[(size_t)x * D.WW + w] = acc;
    }
}

// One lane's action on a checked nogood of a list round: claim of its unit
// literal, or conflict; whether it claimed.
__device__ __forceinline__ bool list_act(const SweepCtx &X, uint32_t id, bool sat, uint32_t n_un, uint32_t ul, uint32_t &checks,
                                         uint32_t &visits)
{
    const uint32_t L = ((id >> 27) & 15u) + 1u;
    checks += L;
    visits++;
    if (sat || n_un > 1u) return false;
    const uint32_t x = ul >> 1, valbit = (ul & 1u) ? V_T : V_F;
    const int k = n_un == 0u ? 2 : claim_var(X.D->asg, x, valbit, X.fresh);
    if (k == 2) report_conflict(X, id, L);
    else if (k == 0) record_claim(X, x, valbit, id);
    return k == 0;
}

// Occurrence o of a literal of variable y by one lane: check, claim and, above
// the root level (nw > 0), the claim's bitmap.
__device__ __forceinline__ void list_check_lane(const SweepCtx &X, uint32_t o, uint32_t y, uint32_t nw, uint32_t &checks, uint32_t &visits)
{
    const Codes<false> codes{X.D->asg};
    const LaneCheck r = lane_check(*X.D, codes, X.fresh, o);
    if (!list_act(X, r.id, r.sat, r.n_un, r.ul, checks, visits) || !nw) return;
    const uint32_t x = r.ul >> 1;
    uint32_t u[8];
    u[0] = y;
#pragma unroll
    for (uint32_t q = 0; q < 7u; q++) u[q + 1u] = r.l[q] == PAD_LIT ? x : r.l[q] >> 1;
    const uint4 v[2] = {make_uint4(u[0], u[1], u[2], u[3]), make_uint4(u[4], u[5], u[6], u[7])};
    narrow_deps(*X.D, x, r.id, r.len ? nullptr : v, nw, 0u, 1u);
}

// The bucket nogoods of the literals on the trail entries [fr0, fr1) (the
// claims of the round before), by the whole grid: only these can have become
// unit or violated.  With up to eight entries a warp its quads share out their
// lists, for the shortest chain; with more its lanes do, 32 entries at a time.
// Values are the global codes, with this round's claims unseen.  For more
// claims than one CTA follows well and fewer than make a sweep of the store
// worth its bytes (Dev::list_max): on the 400k program a sweep takes 56 us, a
// round over 20k claims about 8 us.  A warp whose lists hold more than
// Dev::long_list occurrences passes them over and sets the phase's flag: the
// next round is then a sweep (an atom in half of the positive bodies of 320k
// rules kept one warp busy for 9 ms).
__device__ __forceinline__ void list_round(const SweepCtx &X, uint32_t fr0, uint32_t fr1, uint32_t &checks, uint32_t &visits)
{
    const Dev &D = *X.D;
    const uint32_t lane = threadIdx.x & 31u, sub = lane & 3u, quad = lane & 28u, n = fr1 - fr0;
    const uint32_t wpc = blockDim.x >> 5, slot = (X.gw % wpc) * (X.nw / wpc) + X.gw / wpc;
    const uint32_t each = min(32u, (n + X.nw - 1u) / X.nw), nw = X.cdl > 1u ? deps_words(D, X.cdl) : 0u;
    const Codes<false> codes{D.asg};
    for (uint32_t i0 = slot * each; i0 < n; i0 += X.nw * each) {
        const uint32_t i = i0 + lane;
        uint32_t y = 0, o0 = 0, c = 0;
        if (lane < each && i < n) {
            const uint32_t e = __ldcg(D.trail + fr0 + i), l = mk_lit(e & TRAIL_VAR, (e & TRAIL_F) != 0u);
            if ((l >> 1) < D.nv) {
                y = l >> 1;
                o0 = __ldg(D.occ_off + l);
                c = __ldg(D.occ_off + l + 1u) - o0;
            }
        }
        if (__reduce_add_sync(FULL_MASK, c) > D.long_list) {
            if (lane == 0) atomicOr(&X.acc->flag, 1u);
            continue;
        }
        if (each > 8u) {
            warp_lists_lanes(o0, c, [&](uint32_t o, uint32_t li) {
                const uint32_t yo = __shfl_sync(FULL_MASK, y, li);
                if (o != 0xFFFFFFFFu) list_check_lane(X, o, yo, nw, checks, visits);
                __syncwarp();
            });
            continue;
        }
        warp_lists(o0, c, [&](uint32_t o, uint32_t li) {
            const uint32_t yo = __shfl_sync(FULL_MASK, y, li);
            const QuadCheck r = quad_check(D, codes, X.fresh, o);
            const uint32_t x = r.ul >> 1;
            uint32_t won = sub == 0u && o != 0xFFFFFFFFu && list_act(X, r.id, r.sat, r.n_un, r.ul, checks, visits);
            if (!nw) return;
            won = __shfl_sync(FULL_MASK, won, quad);
            if (!__any_sync(FULL_MASK, won)) return;
            // the claim's bitmap by its quad, from the words of the occurrence
            uint32_t u[8];
#pragma unroll
            for (uint32_t q = 0; q < 8u; q++) u[q] = __shfl_sync(FULL_MASK, r.l[q & 1u], quad + (q >> 1));
#pragma unroll
            for (uint32_t q = 0; q < 8u; q++) u[q] = q == 0u ? yo : u[q] == PAD_LIT ? x : u[q] >> 1;
            if (won) {
                const uint4 v[2] = {make_uint4(u[0], u[1], u[2], u[3]), make_uint4(u[4], u[5], u[6], u[7])};
                narrow_deps(D, x, r.id, r.len ? nullptr : v, nw, sub, 4u);
            }
            __syncwarp();
        });
    }
}

// The CTA's unit table (s_ubase) from the static partition, once per
// launch; callers synchronise the CTA before the first sweep.
__device__ __forceinline__ void unit_table(const Dev &D, uint32_t cta, bool lists = false)
{
    if (threadIdx.x != 0) return;
    s_unit = 0u;
    s_ncl = 0u;
    s_unit2[0] = 0u;
    s_unit2[1] = 0u;
    if (lists) return;
    const uint32_t G1 = D.G + 1u;
    uint32_t acc = 0;
    for (uint32_t L = 2; L <= (uint32_t)BUCKET_MAX; L++) {
        s_ubase[L] = acc;
        s_krange[L][0] = __ldg(D.cta_boff + L * G1 + cta);
        s_krange[L][1] = __ldg(D.cta_boff + L * G1 + cta + 1u);
        const uint32_t n = s_krange[L][1] - s_krange[L][0];
        const uint32_t groups = (n + 31u) >> 5, per = unit_groups(L);
        acc += (groups + per - 1u) / per;
    }
    s_ubase[BUCKET_MAX + 1] = acc;
}

// Propagate-and-check over this CTA's ranges of every bucket (full), or
// over the lists of the trail entries [fr0, fr1) (list_round), then (grid-wide)
// the static long nogoods and the learned nogoods.  ONLY_LONG: the latter
// alone (one CTA follows the bucket nogoods in narrow rounds).
template <bool ONLY_LONG>
__device__ __forceinline__ void sweep(const SweepCtx &X0, uint32_t n_learned, bool full = true,
                                      uint32_t fr0 = 0u, uint32_t fr1 = 0u, uint32_t pass = 0u)
{
    SweepCtx X = X0;
    // Listed claims take their trail slots at the end of the sweep, after
    // any claim that overflowed the list; a claim can rest on an earlier
    // claim of its own CTA (published in the view), so listing breaks the
    // trail's dependency order once the list overflows.  Resolution
    // learning walks the trail backwards and needs that order: there every
    // claim takes its slot when it is made.
    X.listed = X0.do_claim && !X0.D->learning;
    const Dev &D = *X.D;
    const uint32_t lane = threadIdx.x & 31u;
    const bool timer = X.cta == 0 && threadIdx.x == 0 && X.do_claim;
    const bool wtimer = lane == 0 && X.do_claim;
    const unsigned long long t0 = wtimer ? globaltimer_ns() : 0ull;
    // Units of work (one bucket, unit_groups(L) consecutive groups of 32
    // nogoods) are taken from a per-CTA counter, bucket after bucket, so
    // every warp runs about the same number of load-gather-classify chains
    // whatever the mix of lengths.
    // The counters start at 0: reset at launch (unit_table) and, in the
    // solver, at the end of every sweep once no warp reads them any more.
    // Sweeps that do not claim (the sweep timed alone, `pass` = its index
    // in the launch) use two counters: after one barrier no warp is in the
    // previous sweep, so its counter can be cleared for the next one.
    unsigned int *uctr = &s_unit;
    if (!X.do_claim) {
        cta_sync();
        if (threadIdx.x == 0) s_unit2[(pass + 1u) & 1u] = 0u;
        uctr = &s_unit2[pass & 1u];
    }
    const uint32_t *const ubase = s_ubase;     // set up once per launch (unit_table)
    uint32_t units = full ? ubase[BUCKET_MAX + 1] : 0u;
    // Long and learned nogoods first (one warp each, round-robin over CTAs
    // first, then over the warps of a CTA); the warps that take one then
    // take fewer bucket units from the queue.
    unsigned long long checks = 0;
    const uint32_t nl = D.n_long + n_learned;
    const uint32_t wpc = blockDim.x >> 5, slot = (X.gw % wpc) * (X.nw / wpc) + X.gw / wpc;
    // a lane each for the two watched literals, which settle nearly all of
    // them; the whole warp scans the rest (with a warp each, the three
    // dependent loads of the watches were the cost of a round of a search with
    // thousands of learned nogoods)
    const uint32_t each = min(32u, (nl + X.nw - 1u) / X.nw);
    uint32_t wchecks = 0;
    for (uint32_t i0 = slot * each; i0 < nl; i0 += X.nw * each) {
        const uint32_t i = i0 + lane;
        uint32_t id = 0;
        uint2 wp = make_uint2(0u, 0u);
        bool scan = false;
        if (lane < each && i < nl) {
            id = i < D.n_long ? __ldg(D.long_ids + i) : __ldcg(D.learned_ids + (i - D.n_long));
            if (D.nwatch) wp = __ldcg(D.nwatch + i);
            scan = wp.x == wp.y;
            if (!scan) {
                const uint32_t l0 = lit_at(D, id + wp.x) & ~END_BIT, l1 = lit_at(D, id + wp.y) & ~END_BIT;
                const uint32_t v0 = (l0 >> 1) < D.nv ? global_val(D, l0 >> 1, X.fresh) : 0u;
                const uint32_t v1 = (l1 >> 1) < D.nv ? global_val(D, l1 >> 1, X.fresh) : 0u;
                const bool opp = v0 == ((l0 & 1u) ? V_T : V_F) || v1 == ((l1 & 1u) ? V_T : V_F);
                scan = !opp && (v0 != 0u || v1 != 0u);
                wchecks += 2u;
            }
        }
        for (unsigned m = __ballot_sync(FULL_MASK, scan); m; m &= m - 1u) {
            const int src = __ffs(m) - 1;
            classify_long(X, __shfl_sync(FULL_MASK, id, src), checks, D.nwatch ? D.nwatch + i0 + (uint32_t)src : nullptr,
                          make_uint2(__shfl_sync(FULL_MASK, wp.x, src), __shfl_sync(FULL_MASK, wp.y, src)));
        }
    }
    if (nl) checks += __reduce_add_sync(FULL_MASK, wchecks);
    const unsigned long long t1 = wtimer ? globaltimer_ns() : 0ull;
    while (!ONLY_LONG) {
        uint32_t u = 0;
        if (lane == 0) u = atomicAdd(uctr, 1u);
        u = __shfl_sync(FULL_MASK, u, 0);
        if (u >= units) break;
        uint32_t L = 2;
#pragma unroll
        for (uint32_t q = 3; q <= (uint32_t)BUCKET_MAX; q++)
            if (u >= ubase[q]) L = q;
        const uint32_t first = ubase[L];
        const uint32_t b0 = s_krange[L][0], b1 = s_krange[L][1];
        const uint32_t k0 = b0 + (u - first) * unit_groups(L) * 32u;
        if (D.view_mode == VIEW_BYTES) run_unit_view<true>(X, L, k0, b1);
        else if (D.view_mode == VIEW_PACKED) run_unit_view<false>(X, L, k0, b1);
        else run_unit(X, L, k0, b1);
    }
    uint32_t uvisits = 0;
    if (!ONLY_LONG && fr0 < fr1) {
        uint32_t c = 0, v = 0;
        list_round(X, fr0, fr1, c, v);
        checks += __reduce_add_sync(FULL_MASK, c);
        uvisits = __reduce_add_sync(FULL_MASK, v);
    }
    if (lane == 0 && checks) atomicAdd(&X.acc->checks, checks);
    if (lane == 0 && uvisits) atomicAdd(&X.acc->visits, (unsigned long long)uvisits);
    if (wtimer) {
        const unsigned long long t2 = globaltimer_ns();
        if (timer) {
            s_tlearned += t1 - t0;
            s_tbuckets += t2 - t1;
        }
        atomicMax(&s_wmax[0], t1 - t0);
        atomicMax(&s_wmax[1], t2 - t1);
    }
    if (X.do_claim) {
        // copy the listed claims to the trail: warp 0 reserves the slots,
        // then every thread copies (no barrier under a data-dependent branch)
        cta_sync();
        const uint32_t n = min(s_ncl, CLAIM_BUF);
        if (threadIdx.x == 0) {
            s_unit = 0u;                             // every warp has left the unit queue
            atomicMax(&X.acc->tlong, s_wmax[0]);
            atomicMax(&X.acc->tbuck, s_wmax[1]);
            s_wmax[0] = s_wmax[1] = 0ull;
        }
        if (threadIdx.x < 32u) {
            uint32_t base = 0;
            if (threadIdx.x == 0 && n) base = atomicAdd(&X.acc->nclaim, n);
            base = __shfl_sync(FULL_MASK, base, 0);
            if (threadIdx.x == 0) s_cbase = X.tbase + base;
        }
        cta_sync();
        const uint32_t b = s_cbase;
        if (threadIdx.x == 0) s_ncl = 0u;           // every thread has read n
        for (uint32_t k = threadIdx.x; k < n; k += blockDim.x)
            if (b + k < D.nv) {
                const uint32_t e = s_claims[k];
                D.trail[b + k] = e;
                if (D.tpos) D.tpos[e & TRAIL_VAR] = b + k;
            }
    }
}

// bitmap word w of "every decision level 2..L" (CompleteAssignment reading)
__device__ __forceinline__ unsigned long long all_levels_word(const Dev &D, uint32_t L, uint32_t w)
{
    // exact bits 1 .. min(L, Wlevels-1)-1, plus overflow if L >= Wlevels
    uint32_t hi = (L < D.Wlevels ? L : D.Wlevels - 1u);   // exclusive upper bit
    unsigned long long m = 0;
    uint32_t lo_bit = w * 64u, hi_bit = lo_bit + 64u;
    uint32_t a = lo_bit > 1u ? lo_bit : 1u, b = hi_bit < hi ? hi_bit : hi;
    if (a < b) {
        uint32_t n = b - a;
        unsigned long long ones = n >= 64u ? ~0ull : ((1ull << n) - 1ull);
        m = ones << (a - lo_bit);
    }
    if (L >= D.Wlevels && w == D.WW - 1u) m |= 1ull << 63;
    return m;
}

// OR of the dependency bitmaps of the literals of nogood `id` other than
// variable `skip` with level > 1, word w.
__device__ __forceinline__ unsigned long long or_deps_word(const Dev &D, uint32_t id, uint32_t skip, uint32_t w)
{
    unsigned long long acc = 0;
    const uint32_t len = ng_len(D, id);
    for (uint32_t q = 0; q < len; q++) {
        uint32_t u = ng_lit(D, id, q) >> 1;
        if (u == skip) continue;
        int32_t L = __ldcg(D.dl + u);
        if (L > 1 && w < deps_words(D, (uint32_t)L)) acc |= __ldcg(D.deps + (size_t)u * D.WW + w);
    }
    return acc;
}

__device__ __forceinline__ unsigned long long shfl_max_u64(unsigned long long x)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long y = __shfl_down_sync(FULL_MASK, x, o);
        x = y > x ? y : x;
    }
    return x;
}

struct Smem {
    unsigned long long *bm;     // [WW] conflict bitmap
    unsigned long long *red;    // [32]
    uint32_t *misc;             // [16]
    const __nv_bfloat16 *mlp;   // [MLP_PARAMS] after the view (heuristic 2)
    uint32_t *codes;            // [asg_words] after that (code_cache)
};

// The 16 features of candidate rule j (inputs of the learned heuristic):
// its 8 static features, then log1p activity, B- atoms still unassigned and
// already false, decision level / 64, log1p conflicts so far, fraction of
// variables assigned, two zeros.
__device__ __forceinline__ void cand_features(const Dev &D, uint32_t j, uint32_t cdl, uint32_t tend, float *x)
{
    const float *sf = D.rfeat + (size_t)j * 8u;
#pragma unroll
    for (int q = 0; q < 8; q++) x[q] = __ldg(sf + q);
    x[8] = log1pf((float)__ldcg(D.act + j));
    uint32_t un = 0, fa = 0;
    for (uint32_t q = __ldg(D.rneg_off + j); q < __ldg(D.rneg_off + j + 1); q++) {
        const uint32_t a = __ldg(D.rneg + q);
        const uint32_t v = (__ldcg(D.asg + (a >> 3)) >> ((a & 7u) * 4u)) & 3u;
        un += v == 0u;
        fa += v == V_F;
    }
    x[9] = (float)un;
    x[10] = (float)fa;
    x[11] = (float)cdl * (1.0f / 64.0f);
    x[12] = log1pf((float)__ldcg(&D.stats->conflicts));
    x[13] = (float)tend / (float)(D.nv ? D.nv : 1u);
    x[14] = 0.0f;
    x[15] = 0.0f;
}

// order-preserving map of a float to a positive 32-bit key
__device__ __forceinline__ uint32_t float_key(float f)
{
    uint32_t u = __float_as_uint(f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return u ? u : 1u;
}

// Decision (Section 2 / Section 4): among rules whose head is unassigned,
// with t_r true, n_r not false and b_r unassigned (applicable), pick the
// highest score, ties to the lowest rule index.  Every key is
// (score << 32) | (0xFFFFFFFF - j): the decision phase recovers the rule j
// from the low word.
__device__ __forceinline__ void decide(const Dev &D, const Smem &S, Acc *acc, uint32_t gtid, uint32_t nthreads,
                                       uint32_t cdl, uint32_t tend)
{
    unsigned long long best = 0;
    // the codes of b, t and n (three neighbours) of four rules load together;
    // the head's only for the few rules that these let pass
    for (uint32_t j4 = gtid; j4 < D.J; j4 += 4u * nthreads) {
        unsigned long long w[4];
#pragma unroll
        for (uint32_t q = 0; q < 4u; q++) {
            const uint32_t b = D.na + 3u * min(j4 + q * nthreads, D.J - 1u);
            w[q] = (((unsigned long long)__ldcg(D.asg + ((b + 2u) >> 3)) << 32) | __ldcg(D.asg + (b >> 3))) >> ((b & 7u) * 4u);
        }
        uint32_t pass = 0;
#pragma unroll
        for (uint32_t q = 0; q < 4u; q++)
            if ((w[q] & 3u) == 0u && ((w[q] >> 4) & 3u) == V_T && ((w[q] >> 8) & 3u) != V_F && j4 + q * nthreads < D.J) pass |= 1u << q;
        for (; pass; pass &= pass - 1u) {
            const uint32_t j = j4 + ((uint32_t)__ffs(pass) - 1u) * nthreads;
            const uint32_t h = (uint32_t)__ldg(D.rule_head + j);
            if ((nib(__ldcg(D.asg + (h >> 3)), h) & 3u) != 0u) continue;
            unsigned long long key;
            if (D.trace) {
                // sample about one candidate in eight per decision point
                uint32_t hsh = (j * 0x9E3779B1u) ^ (cdl * 0x85EBCA77u) ^ (tend * 0xC2B2AE3Du);
                hsh ^= hsh >> 15;
                hsh *= 0x2C1B3C6Du;
                hsh ^= hsh >> 12;
                if ((hsh & TRACE_SAMPLE_MASK) == 0u) {
                    const uint32_t r = atomicAdd(&D.stats->trace_n, 1u);
                    if (r < D.trace_cap) {
                        float x[N_FEATURES];
                        cand_features(D, j, cdl, tend, x);
                        uint32_t *rec = D.trace + (size_t)r * TRACE_WORDS;
                        for (int q = 0; q < N_FEATURES; q++) rec[q] = __float_as_uint(x[q]);
                        rec[16] = j;
                        rec[17] = cdl;
                        rec[18] = 0u;
                        rec[19] = 0u;
                    }
                }
            }
            if (D.heuristic == 3) {
                key = ((unsigned long long)float_key(__ldg(D.prior + j)) << 32) | (0xFFFFFFFFull - j);
            } else if (D.heuristic == 2) {
                // plain score (log1p occurrences of the head, feature 0) plus
                // the log of the learned probability that the rule's body
                // holds in an answer set
                float x[N_FEATURES];
                cand_features(D, j, cdl, tend, x);
                const float z = mlp_score(S.mlp, x);
                const float log_p = z >= 0.0f ? -log1pf(__expf(-z)) : z - log1pf(__expf(z));
                key = ((unsigned long long)float_key(x[0] + log_p) << 32) | (0xFFFFFFFFull - j);
            } else if (D.heuristic == 5) {
                // activity, plus the head's occurrences times a millionth of
                // the current increment (at most 4095 of them: less than one
                // bump) to order rules of equal activity; ties to the lowest
                // rule.  The low word stays ~j, which the decision phase decodes.
                const float *vact = reinterpret_cast<const float *>(D.act);
                const float a = __ldcg(vact + j);
                const float occ = (float)min(__ldg(D.score + j), 4095u);
                const float sc = a + occ * (__ldcg(vact + D.J) * 1e-6f);
                key = ((unsigned long long)float_key(sc) << 32) | (0xFFFFFFFFull - j);
            } else {
                unsigned long long sc = __ldg(D.score + j);
                if (D.heuristic == 1) sc += (unsigned long long)__ldcg(D.act + j) * 8ull;
                if (sc > 0x7FFFFFFFull) sc = 0x7FFFFFFFull;
                key = ((sc + 1ull) << 32) | (0xFFFFFFFFull - j);
            }
            best = key > best ? key : best;
        }
    }
    best = shfl_max_u64(best);
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    if (lane == 0) S.red[wid] = best;
    cta_sync();
    if (wid == 0) {
        unsigned long long x = lane < (blockDim.x >> 5) ? S.red[lane] : 0ull;
        x = shfl_max_u64(x);
        if (lane == 0 && x) atomicMax(&acc->dkey, x);
    }
}

// One pass of the immediate-consequence operator of the reduct on D.lm;
// whether this thread added an atom.  The assignment M is total and violates
// no nogood, so M is a model of the reduct, the least model stays inside M, and
// a rule can fire only if its body holds in M, which is the value of b_j: the
// other rules (most) are passed over by that one code, four at a time, and no
// negative body is read.
__device__ __forceinline__ bool least_model_pass(const Dev &D, uint32_t gtid, uint32_t nthreads)
{
    bool more = false;
    for (uint32_t j4 = gtid; j4 < D.J; j4 += 4u * nthreads) {
        uint32_t w[4], pass = 0;
#pragma unroll
        for (uint32_t q = 0; q < 4u; q++) {
            const uint32_t b = D.na + 3u * min(j4 + q * nthreads, D.J - 1u);
            w[q] = nib(__ldcg(D.asg + (b >> 3)), b) & 3u;
        }
#pragma unroll
        for (uint32_t q = 0; q < 4u; q++)
            if (w[q] == V_T && j4 + q * nthreads < D.J) pass |= 1u << q;
        for (; pass; pass &= pass - 1u) {
            const uint32_t j = j4 + ((uint32_t)__ffs(pass) - 1u) * nthreads, h = (uint32_t)__ldg(D.rule_head + j);
            if ((__ldcg(D.lm + (h >> 5)) >> (h & 31u)) & 1u) continue;
            bool ok = true;
            const uint32_t q1 = __ldg(D.rpos_off + j + 1);
            for (uint32_t q = __ldg(D.rpos_off + j); ok && q < q1; q++) {
                const uint32_t a = __ldg(D.rpos + q);
                ok = (__ldcg(D.lm + (a >> 5)) >> (a & 31u)) & 1u;
            }
            if (ok) {
                atomicOr(D.lm + (h >> 5), 1u << (h & 31u));
                more = true;
            }
        }
    }
    return more;
}

// Passes that one CTA makes in a phase (a grid makes one): the time budget is
// looked at between phases, and on a chain the least model takes a pass per
// atom (100k atoms: 8.7 s, all past the budget when they were one phase).  64
// passes of the 300k-rule program of that chain are about 6 ms.
constexpr uint32_t STAB_PASSES = 64u;

// The smallest true atom outside the least model, into acc->minU.
__device__ __forceinline__ void unfounded_min(const Dev &D, Acc *acc, uint32_t gtid, uint32_t nthreads)
{
    for (uint32_t p = gtid; p < D.na; p += nthreads) {
        const bool inM = (nib(__ldcg(D.asg + (p >> 3)), p) & 3u) == V_T;
        const bool inLM = (__ldcg(D.lm + (p >> 5)) >> (p & 31u)) & 1u;
        if (inM && !inLM) atomicMin(&acc->minU, p);
    }
}

// VSIDS-style activity (heuristic 5, not in the paper; the paper's
// Decision kernel names activity among its heuristics): every variable of a
// learned nogood bumps the rules it stands for -- b_j, t_j or n_j rule j, an
// atom the rules with it as head -- by the current increment, stored as a
// float after the J activities.  The increment grows by 1/0.95 per learned
// nogood (vsids_decay), so earlier bumps count less and less.
__device__ __forceinline__ void vsids_bump(const Dev &D, uint32_t var, float inc)
{
    float *vact = reinterpret_cast<float *>(D.act);
    if (var >= D.nv) return;
    if (var >= D.na) {
        atomicAdd(vact + (var - D.na) / 3u, inc);
        return;
    }
    for (uint32_t j = __ldg(D.head_first + var); j < __ldg(D.head_first + var + 1u); j++) atomicAdd(vact + j, inc);
}

// After each analysis (all threads of the analysing CTA): the increment
// grows by 1/0.95; above 1e20 every activity and the increment are scaled
// by 1e-20, which keeps their order.
__device__ __forceinline__ void vsids_decay(const Dev &D)
{
    __shared__ int s_rescale;
    float *vact = reinterpret_cast<float *>(D.act);
    cta_sync();
    if (threadIdx.x == 0) {
        float inc = __ldcg(vact + D.J) * (1.0f / 0.95f);
        s_rescale = inc > 1e20f;
        vact[D.J] = s_rescale ? inc * 1e-20f : inc;
    }
    cta_sync();
    if (s_rescale)
        for (uint32_t j = threadIdx.x; j < D.J; j += blockDim.x) vact[j] *= 1e-20f;
}

// fwd-learning (Algorithm 4) on CTA 0: OR the dependency bitmaps of the
// conflict's literals (plus those of the clashing variable's reason), take
// the highest level involved, and learn the nogood made of the decision
// literals of the levels in the bitmap.  Returns via S.misc:
//   misc[0] = 1 if the bitmap is empty (conflict at the root),
//   misc[1] = backjump target, misc[2] = learned length.
__device__ __forceinline__ void analyze(const Dev &D, const Smem &S, uint32_t g, uint32_t cdl, uint32_t lfill, bool find_clash)
{
    const uint32_t tid = threadIdx.x, nt = blockDim.x;
    const uint32_t nw = deps_words(D, cdl);
    for (uint32_t w = tid; w < D.WW; w += nt) S.bm[w] = 0ull;
    if (tid == 0) {
        // length of g and the clashing variable: the one with both values set
        uint32_t len = ng_len(D, g), clash = 0xFFFFFFFFu;
        for (uint32_t q = 0; q < len && find_clash; q++) {
            uint32_t u = ng_lit(D, g, q) >> 1;
            if ((nib(__ldcg(D.asg + (u >> 3)), u) & 3u) == 3u) clash = u;
        }
        S.misc[4] = len;
        S.misc[5] = clash;
    }
    cta_sync();
    const uint32_t len = S.misc[4], clash = S.misc[5];
    for (uint32_t t = tid; t < len * nw; t += nt) {
        uint32_t i = t / nw, w = t % nw;
        uint32_t u = ng_lit(D, g, i) >> 1;
        if (u == clash) continue;
        int32_t L = __ldcg(D.dl + u);
        if (L > 1 && w < deps_words(D, (uint32_t)L)) atomicOr(&S.bm[w], __ldcg(D.deps + (size_t)u * D.WW + w));
    }
    if (clash != 0xFFFFFFFFu) {
        uint32_t r = __ldcg(D.reason + clash);
        if (r == R_COMPLETE) {
            for (uint32_t w = tid; w < nw; w += nt) atomicOr(&S.bm[w], all_levels_word(D, cdl, w));
        } else if (r < R_INPUT) {
            for (uint32_t w = tid; w < nw; w += nt) atomicOr(&S.bm[w], or_deps_word(D, r, clash, w));
        } else if (r == R_DECISION) {
            int32_t L = __ldcg(D.dl + clash);
            for (uint32_t w = tid; w < nw; w += nt)
                if (L > 1 && w < deps_words(D, (uint32_t)L)) atomicOr(&S.bm[w], __ldcg(D.deps + (size_t)clash * D.WW + w));
        }
    }
    cta_sync();
    if (tid == 0) {
        bool overflow = cdl >= D.Wlevels && (S.bm[D.WW - 1] >> 63);
        int top = -1;
        for (int w = (int)nw - 1; w >= 0 && top < 0; w--) {
            unsigned long long m = S.bm[w];
            if (w == (int)D.WW - 1) m &= ~(1ull << 63);
            if (m) top = w * 64 + 63 - __clzll((long long)m);
        }
        if (!overflow && top < 0) {
            S.misc[0] = 1;
        } else {
            uint32_t h = overflow ? cdl : (uint32_t)top + 1u;
            S.misc[0] = 0;
            S.misc[1] = h - 1u;
            if (D.backjump == 1u && !overflow) {
                // the asserting level: the second-highest level of the bitmap
                // (1 if h is its only level); the learned nogood is unit there
                int second = -1;
                for (int w = top >> 6; w >= 0 && second < 0; w--) {
                    unsigned long long m = S.bm[w];
                    if (w == (int)D.WW - 1) m &= ~(1ull << 63);
                    if (w == (top >> 6)) m &= (1ull << (top & 63)) - 1ull;
                    if (m) second = w * 64 + 63 - __clzll((long long)m);
                }
                S.misc[1] = second >= 1 ? (uint32_t)second + 1u : 1u;
            }
            // write the decision literals, levels ascending
            uint32_t n = 0;
            for (uint32_t w = 0; w < nw; w++) {
                unsigned long long m = S.bm[w];
                if (w == D.WW - 1u) m &= ~(1ull << 63);
                while (m) {
                    uint32_t bit = (uint32_t)__ffsll((long long)m) - 1u;
                    m &= m - 1ull;
                    uint32_t level = w * 64u + bit + 1u;
                    if (level < 2u || level > cdl) continue;
                    uint32_t pos = lfill + n;
                    if (pos + 1u < D.lits_cap) D.lits[pos] = mk_lit(__ldcg(D.dec_var + level), false);
                    n++;
                }
            }
            if (overflow) {
                for (uint32_t level = D.Wlevels; level <= cdl; level++) {
                    uint32_t pos = lfill + n;
                    if (pos + 1u < D.lits_cap) D.lits[pos] = mk_lit(__ldcg(D.dec_var + level), false);
                    n++;
                }
            }
            if (n > 0 && lfill + n < D.lits_cap) D.lits[lfill + n - 1u] |= END_BIT;
            S.misc[2] = n;
            if (D.heuristic == 1) {
                for (uint32_t q = 0; q < n && lfill + q < D.lits_cap; q++) {
                    uint32_t bv = (D.lits[lfill + q] & ~END_BIT) >> 1;
                    if (bv >= D.na && (bv - D.na) % 3u == 0u) atomicAdd(D.act + (bv - D.na) / 3u, 1u);
                }
            }
        }
    }
    cta_sync();
    if (D.heuristic == 5 && !S.misc[0]) {
        const float inc = __ldcg(reinterpret_cast<const float *>(D.act) + D.J);
        for (uint32_t q = tid; q < S.misc[2] && lfill + q < D.lits_cap; q += nt)
            vsids_bump(D, (__ldcg(D.lits + lfill + q) & ~END_BIT) >> 1, inc);
        vsids_decay(D);
    }
}

// Register learned nogood number i (its first literal at `id`, len
// literals): the learned list, and its two watched positions (the first
// two literals; a nogood of one literal is always scanned).
__device__ __forceinline__ void add_learned(const Dev &D, uint32_t i, uint32_t id, uint32_t len)
{
    D.learned_ids[i] = id;
    if (D.nwatch) D.nwatch[D.n_long + i] = len > 1u ? make_uint2(0u, 1u) : make_uint2(0u, 0u);
}

// Record of the last conflict analysis, for consistency checks (leader).
__device__ __forceinline__ void debug_analysis(const Dev &D, uint32_t g, uint32_t tend, uint32_t lfill, uint32_t n,
                                               uint32_t target, uint32_t m)
{
    D.stats->dbg_conf = g;
    D.stats->dbg_tend = tend;
    D.stats->dbg_lfill = lfill;
    D.stats->dbg_len = n;
    D.stats->dbg_target = target;
    D.stats->dbg_level = m;
}

// ------------------------------------------------------ res-learning

// State of the resolution chain of res_analyze (uniform over its warp).
struct ResState {
    uint32_t m;             // level the nogood is resolved at
    uint32_t seg0, seg1;    // trail positions of level m
    uint32_t ep;            // stamp of this analysis
    uint32_t out0, nout;    // learned literals below level m: slots out0 ..
    uint32_t kappa;         // highest level among them (1 if none)
    bool err;
    uint32_t why, what;     // failed check (1..10) and the variable or value involved
};

__device__ __forceinline__ void res_fail(ResState &R, uint32_t why, uint32_t what)
{
    if (!R.err) { R.why = why; R.what = what; }
    R.err = true;
}

// The warp adds one literal per lane (has = false on lanes holding none) to
// the nogood being resolved.  Dropped: the variable `skip` (the one resolved
// upon), root-level literals and variables already in the nogood (stamped
// with R.ep).  A literal at level m is marked in the trail-position bitset;
// one below goes to the learned nogood.  Returns the number marked.
__device__ __forceinline__ uint32_t res_add(const Dev &D, ResState &R, bool has, uint32_t l, uint32_t skip)
{
    const uint32_t lane = threadIdx.x & 31u;
    bool cur = false, out = false;
    uint32_t L = 0, bad = 0u;
    if (has) {
        const uint32_t u = l >> 1;
        if (u >= D.nv) {
            bad = 1u;
        } else if (u != skip) {
            const int32_t Ls = __ldcg(D.dl + u);
            L = Ls > 0 ? (uint32_t)Ls : 0u;
            if (L == 0u) {
                bad = 2u;                // unassigned
            } else if (L > R.m) {
                bad = 3u;                // above the conflict level
            } else if (L > 1u && atomicExch(D.stamp + u, R.ep) != R.ep) {
                if (L == R.m) {
                    const uint32_t tp = __ldcg(D.tpos + u);
                    if (tp >= R.seg0 && tp < R.seg1) {
                        atomicOr(D.cand + (tp >> 5), 1u << (tp & 31u));
                        cur = true;
                    } else {
                        bad = 4u;        // trail position outside level m
                    }
                } else {
                    out = true;
                }
            }
        }
    }
    const unsigned bb = __ballot_sync(FULL_MASK, bad != 0u);
    if (bb) {
        const int src = __ffs(bb) - 1;
        res_fail(R, __shfl_sync(FULL_MASK, bad, src), __shfl_sync(FULL_MASK, l >> 1, src));
    }
    const unsigned bc = __ballot_sync(FULL_MASK, cur), bo = __ballot_sync(FULL_MASK, out);
    if (out) {
        const uint32_t pos = R.out0 + R.nout + (uint32_t)__popc(bo & ((1u << lane) - 1u));
        if (pos + 1u < D.lits_cap) D.lits[pos] = l;
    }
    R.nout += (uint32_t)__popc(bo);
    uint32_t k = out ? L : 0u;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(FULL_MASK, k, o));
    R.kappa = max(R.kappa, k);
    return (uint32_t)__popc(bc);
}

// The literals of nogood `id` but variable `skip`, 32 at a time.
__device__ __forceinline__ uint32_t res_add_nogood(const Dev &D, ResState &R, uint32_t id, uint32_t skip)
{
    const uint32_t lane = threadIdx.x & 31u;
    if (id & BUCKET_ID) {
        const uint32_t len = ng_len(D, id);               // at most BUCKET_MAX < 32
        const bool has = lane < len;
        return res_add(D, R, has, has ? ng_lit(D, id, lane) : 0u, skip);
    }
    uint32_t added = 0;
    for (uint32_t base = 0;; base += 32u) {
        if (id + base + 32u > D.lits_cap + 96u) { res_fail(R, 5u, id); break; }   // no end marker
        const uint32_t w = lit_at(D, id + base + lane);
        const unsigned Bend = __ballot_sync(FULL_MASK, (w & END_BIT) != 0u);
        const unsigned valid = Bend ? ((2u << (__ffs(Bend) - 1)) - 1u) : FULL_MASK;
        added += res_add(D, R, (valid >> lane) & 1u, w & ~END_BIT, skip);
        if (Bend) break;
    }
    return added;
}

// The antecedent of a literal set by CompleteAssignment at level Le: the
// decisions of levels 2 .. Le (each true).
__device__ __forceinline__ uint32_t res_add_decisions(const Dev &D, ResState &R, uint32_t Le, uint32_t skip)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t added = 0;
    for (uint32_t base = 2; base <= Le; base += 32u) {
        const uint32_t lv = base + lane;
        const bool has = lv <= Le;
        added += res_add(D, R, has, has ? mk_lit(__ldcg(D.dec_var + lv), false) : 0u, skip);
    }
    return added;
}

// Conflict analysis by resolution to the first UIP (Algorithm 3), by one
// warp of the analysing CTA.  delta starts as nogood g (every literal of it
// holds; a variable both values were claimed for in the conflict round is
// taken with its first claim) and m is its highest level.  Then, repeatedly:
// sigma = the literal of delta at level m assigned last (highest trail
// position); if no other literal of delta is at level m, sigma is the first
// UIP and delta is learned with kappa = the highest level of the others;
// else delta becomes the resolvent of delta and the reason of sigma (which
// holds the complement of sigma).  Root-level literals are left out of
// delta.  A literal set by CompleteAssignment has no reason nogood: its
// antecedent is taken to be every decision up to its level.  Writes the
// learned nogood at lfill, the first UIP first; S.misc: [0] = 1 conflict at
// the root, 2 internal inconsistency, else 0; [1] = kappa (the backjump
// target); [2] = length; [3] = m.
__device__ __forceinline__ void res_analyze(const Dev &D, const Smem &S, uint32_t g, uint32_t cdl, uint32_t tend,
                                            uint32_t lfill)
{
    const uint32_t tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) {
        S.misc[4] = ng_len(D, g);
        uint32_t e = atomicAdd(D.epoch, 1u) + 1u;
        S.misc[5] = e;
        S.misc[6] = 0u;
        S.misc[0] = 0u;
    }
    cta_sync();
    if (S.misc[5] == 0u) {
        // the stamp counter wrapped: clear every stamp, restart at 1
        for (uint32_t v = tid; v < D.nv; v += nt) D.stamp[v] = 0u;
        cta_sync();
        if (tid == 0) { *D.epoch = 1u; S.misc[5] = 1u; }
        cta_sync();
    }
    const uint32_t len = S.misc[4], ep = S.misc[5];
    for (uint32_t q = tid; q < len; q += nt) {
        const uint32_t u = ng_lit(D, g, q) >> 1;
        if (u < D.nv) atomicMax(&S.misc[6], (uint32_t)max(__ldcg(D.dl + u), 0));
    }
    cta_sync();
    const uint32_t m = S.misc[6];
    if (m <= 1u) {
        if (tid == 0) S.misc[0] = 1u;
        cta_sync();
        return;
    }
    const uint32_t seg0 = __ldcg(D.level_start + m);
    const uint32_t seg1 = m >= cdl ? tend : __ldcg(D.level_start + m + 1u);
    if (!(seg0 < seg1 && seg1 <= D.nv)) {
        if (tid == 0) { S.misc[0] = 2u; S.misc[1] = 10u; S.misc[2] = seg0; S.misc[3] = m; }
        cta_sync();
        return;
    }
    for (uint32_t w = (seg0 >> 5) + tid; w <= ((seg1 - 1u) >> 5); w += nt) D.cand[w] = 0u;
    cta_sync();
    if (tid < 32u) {
        const uint32_t lane = tid;
        ResState R{m, seg0, seg1, ep, lfill + 1u, 0u, 1u, false, 0u, 0u};
        uint32_t cnt = res_add_nogood(D, R, g, 0xFFFFFFFFu);
        __syncwarp();
        int p = (int)seg1 - 1;
        const int wlo = (int)(seg0 >> 5);
        uint32_t uip = 0xFFFFFFFFu;
        while (!R.err) {
            // the highest marked position <= p: 32 bitset words per step
            int q = -1;
            while (p >= (int)seg0) {
                const int wtop = p >> 5, w = wtop - (int)lane;
                uint32_t bits = 0;
                if (w >= wlo) {
                    bits = __ldcg(D.cand + w);
                    if (w == wtop) bits &= (2u << (p & 31)) - 1u;
                    if (w == wlo) bits &= ~0u << (seg0 & 31u);
                }
                const unsigned bal = __ballot_sync(FULL_MASK, bits != 0u);
                if (bal) {
                    const int src = __ffs(bal) - 1;
                    const uint32_t b = __shfl_sync(FULL_MASK, bits, src);
                    q = (wtop - src) * 32 + 31 - __clz(b);
                    break;
                }
                p = (wtop - 32) * 32 + 31;
            }
            if (q < 0) { res_fail(R, 6u, cnt); break; }
            if (cnt == 0u) { res_fail(R, 7u, (uint32_t)q); break; }
            const uint32_t entry = __ldcg(D.trail + q), e = entry & TRAIL_VAR;
            if (e >= D.nv) { res_fail(R, 8u, (uint32_t)q); break; }
            if (--cnt == 0u) { uip = entry; break; }     // sigma is the only literal at level m
            const uint32_t r = __ldcg(D.reason + e);
            if (r < R_INPUT) {
                cnt += res_add_nogood(D, R, r, e);
            } else if (r == R_COMPLETE) {
                cnt += res_add_decisions(D, R, (uint32_t)max(__ldcg(D.dl + e), 0), e);
            } else {
                res_fail(R, 9u, e);                       // a decision with others at its level
                break;
            }
            __syncwarp();
            p = q - 1;
        }
        const uint32_t n = 1u + R.nout;
        if (lane == 0) {
            if (R.err) {
                S.misc[0] = 2u;
                S.misc[1] = R.why;
                S.misc[2] = R.what;
                S.misc[3] = m;
            } else {
                if (lfill + 1u < D.lits_cap) D.lits[lfill] = mk_lit(uip & TRAIL_VAR, (uip & TRAIL_F) != 0u);
                if (lfill + n < D.lits_cap) D.lits[lfill + n - 1u] |= END_BIT;
                S.misc[1] = R.kappa;
                S.misc[2] = n;
                S.misc[3] = m;
            }
        }
        __syncwarp();
        if (!R.err && D.heuristic == 1) {
            for (uint32_t q = lane; q < n && lfill + q < D.lits_cap; q += 32u) {
                const uint32_t bv = (D.lits[lfill + q] & ~END_BIT) >> 1;
                if (bv >= D.na && (bv - D.na) % 3u == 0u) atomicAdd(D.act + (bv - D.na) / 3u, 1u);
            }
        }
        if (!R.err && D.heuristic == 5) {
            const float inc = __ldcg(reinterpret_cast<const float *>(D.act) + D.J);
            for (uint32_t q = lane; q < n && lfill + q < D.lits_cap; q += 32u)
                vsids_bump(D, (__ldcg(D.lits + lfill + q) & ~END_BIT) >> 1, inc);
        }
    }
    cta_sync();
    if (D.heuristic == 5 && S.misc[0] == 0u) vsids_decay(D);
}

__device__ __forceinline__ View make_view(const Dev &D, uint32_t *vbase, uint32_t cta)
{
    View V;
    V.w = vbase;
    V.na_v = D.view_atoms;
    V.aux_base = ((D.view_atoms + 15u) >> 4) << 4;
    V.bytes = D.view_mode == VIEW_BYTES;
    V.auxlo = __ldg(D.cta_auxlo + cta);
    V.auxn = __ldg(D.cta_auxn + cta);
    return V;
}

// Copy of a control struct read through L2 (other threads update it with
// plain stores and atomics), by the 32 lanes of a warp.
template <class T>
__device__ __forceinline__ void ldcg_copy(T *dst, const T *src)
{
    const uint32_t *s = reinterpret_cast<const uint32_t *>(src);
    uint32_t *d = reinterpret_cast<uint32_t *>(dst);
#pragma unroll
    for (uint32_t i = threadIdx.x & 31u; i < sizeof(T) / 4u; i += 32u) d[i] = __ldcg(s + i);
}

__device__ __forceinline__ Smem make_smem(const Dev &D, unsigned long long *raw)
{
    Smem S;
    S.bm = raw;
    S.red = S.bm + D.WW;
    S.misc = reinterpret_cast<uint32_t *>(S.red + 32);
    S.mlp = reinterpret_cast<const __nv_bfloat16 *>(S.misc + 16 + D.view_words);
    S.codes = S.misc + 16 + D.view_words + (2 * MLP_PARAMS + 15) / 16 * 4;
    return S;
}

// The i-th term (i >= 1) of the Luby sequence 1 1 2 1 1 2 4 1 1 2 ...: 2^(k-1)
// if i = 2^k - 1, else the term at i - 2^(k-1) + 1 for the k with
// 2^(k-1) <= i < 2^k - 1 (Luby, Sinclair and Zuckerman's restart schedule).
__device__ __forceinline__ uint32_t luby(uint32_t i)
{
    for (;;) {
        uint32_t k = 1;
        while (k < 31u && (1u << k) - 1u < i) k++;
        if ((1u << k) - 1u == i || k == 31u) return 1u << (k - 1u);
        i = i - (1u << (k - 1u)) + 1u;
    }
}

// Phase barrier of the solving group: the whole grid (one program on every
// SM) or one CTA (one program of a batch).
template <bool BATCH>
__device__ __forceinline__ bool group_sync(const Dev &D, uint32_t gen)
{
    if (BATCH) {
        cta_sync();
        return true;
    }
    return grid_sync(D.bar, gridDim.x, D.barrier_ns, gen);
}

// ------------------------------------------------------------ narrow rounds

// Long lists of a round that its warps put off; with more of them (64k literals
// hold at most 250) the others go to a warp each.
constexpr uint32_t LONG_LISTS = 16u;

// What a round leaves to the next one: claims, items drawn, whether some lists
// are not among the items, whether there was a conflict, lists in lng (found;
// LONG_LISTS of them are kept).  Read at once, after the round's barrier.
struct __align__(16) NarrowCount { uint32_t n, m; uint16_t rest, conf; uint32_t nlong; };

// Claims of the previous and of the current narrow round, cached in shared
// memory (the trail holds all of them): e = trail entry, reason, and its
// literal's occurrence list [z, w) unless the list is among the round's items;
// u = the reason's variables, where it has at most eight literals (the entry's
// own variable where there are fewer).
template <uint32_t ENTRIES, uint32_t ITEMS>
struct NarrowQueue {
    static constexpr uint32_t N = ENTRIES, M = ITEMS;
    uint4 e[2][N], u[2][N][2];
    uint2 item[2][M];             // position in D.occ, variable it is the list of
    uint4 lng[LONG_LISTS];        // lists of more than Dev::long_list outside the items: [x, y) of variable z
    NarrowCount count[3];         // of round i, at (i + 1) % 3
};

// Entry k of a round's queue (k and at: its place among the items, drawn by
// the caller) by `lanes` lanes, this one the sub-th.
template <class Queue>
__device__ __forceinline__ void narrow_queue(Queue &Q, uint32_t buf, uint32_t slot, uint32_t k, uint32_t at, uint32_t entry,
                                             uint32_t id, uint32_t o0, uint32_t o1, uint32_t sub, uint32_t lanes)
{
    const uint32_t c = o1 - o0;
    const bool fits = k < Queue::N && at <= Queue::M && c <= Queue::M - at;
    if (fits)
        for (uint32_t j = sub; j < c; j += lanes) Q.item[buf][at + j] = make_uint2(o0 + j, entry & TRAIL_VAR);
    else
        for (uint32_t j = at + sub; j < Queue::M && j - at < c; j += lanes) Q.item[buf][j] = make_uint2(0xFFFFFFFFu, 0u);   // drawn, not used
    if (sub == 0u) {
        if (k < Queue::N) Q.e[buf][k] = make_uint4(entry, id, o0, fits ? o0 : o1);
        if (!fits) Q.count[slot].rest = 1u;
    }
}

// What a round counts and where its claims go.
struct NarrowRound {
    uint32_t cdl, fresh, buf, slot, out;      // buf, slot: of the next round's queue; out: trail index of its first claim
    uint32_t checks, visits;
};

// A claim made in a narrow round: its place in the queue (0xFFFFFFFF: none
// made) and among the items, its occurrence list.
struct NarrowClaim { uint32_t k, at, a0, a1; };

// One lane's action on a checked nogood: claims its unit literal's complement,
// or reports the conflict.  CACHED: the codes are the CTA's copy, and a claim
// goes to global memory too, where nothing of the round waits for it.
template <bool CACHED, class Queue>
__device__ __forceinline__ NarrowClaim narrow_claim(const Dev &D, const Codes<CACHED> &codes, Acc *acc, Queue &Q, NarrowRound &R,
                                                    uint32_t id, bool sat, uint32_t n_un, uint32_t ul)
{
    NarrowClaim C{0xFFFFFFFFu, 0u, 0u, 0u};
    const uint32_t L = ((id >> 27) & 15u) + 1u;
    R.checks += L;
    R.visits++;
    if (sat || n_un > 1u) return C;
    bool clash = n_un == 0u;
    if (!clash) {
        const uint32_t x = ul >> 1, valbit = (ul & 1u) ? V_T : V_F;
        // the claimed literal's list bounds load beside the claim
        C.a0 = __ldg(D.occ_off + (ul ^ 1u));
        C.a1 = __ldg(D.occ_off + (ul ^ 1u) + 1u);
        const int c = claim_var(codes.w, x, valbit, R.fresh);
        if (CACHED && c != 1) atomicOr(D.asg + (x >> 3), (valbit | R.fresh) << ((x & 7u) * 4u));
        if (c == 0) {
            C.k = atomicAdd(&Q.count[R.slot].n, 1u);
            C.at = atomicAdd(&Q.count[R.slot].m, C.a1 - C.a0);
            D.dl[x] = (int32_t)R.cdl;
            D.reason[x] = id;
            const uint32_t pos = R.out + C.k;
            if (pos < D.nv) {
                D.trail[pos] = x | (valbit == V_F ? TRAIL_F : 0u);
                if (D.tpos) D.tpos[x] = pos;
            }
        }
        clash = c == 2;
    }
    if (clash) {
        const unsigned long long key = ((unsigned long long)L << 32) | id;
        atomicMin(&acc->ckey, key);
        atomicMin(&acc->cslot[id % 3u], key);
        Q.count[R.slot].conf = 1u;
    }
    return C;
}

// Checks occurrence o (0xFFFFFFFF: none) of a literal of variable y by a quad
// of lanes; the first acts on it, and all four write a claim's queue entry.
// All 32 lanes call it.
template <bool CACHED, class Queue>
__device__ __forceinline__ void narrow_check(const Dev &D, const Codes<CACHED> &codes, Acc *acc, Queue &Q, NarrowRound &R, uint32_t o,
                                             uint32_t y)
{
    const uint32_t sub = threadIdx.x & 3u, quad = threadIdx.x & 28u;
    const QuadCheck r = quad_check(D, codes, R.fresh, o);
    NarrowClaim C{0xFFFFFFFFu, 0u, 0u, 0u};
    if (sub == 0u && o != 0xFFFFFFFFu) C = narrow_claim(D, codes, acc, Q, R, r.id, r.sat, r.n_un, r.ul);
    const uint32_t k = __shfl_sync(FULL_MASK, C.k, quad);
    if (!__any_sync(FULL_MASK, k != 0xFFFFFFFFu)) return;
    const uint32_t at = __shfl_sync(FULL_MASK, C.at, quad), a0 = __shfl_sync(FULL_MASK, C.a0, quad), a1 = __shfl_sync(FULL_MASK, C.a1, quad);
    if (k != 0xFFFFFFFFu) {
        const uint32_t x = r.ul >> 1;
        narrow_queue(Q, R.buf, R.slot, k, at, x | ((r.ul & 1u) ? 0u : TRAIL_F), r.id, a0, a1, sub, 4u);
        // the reason's variables for the bitmap, two per lane of the quad
        if (k < Queue::N && !r.len)
            reinterpret_cast<uint2 *>(&Q.u[R.buf][k][0])[sub] =
                make_uint2(sub == 0u ? y : r.l[0] == PAD_LIT ? x : r.l[0] >> 1, r.l[1] == PAD_LIT ? x : r.l[1] >> 1);
    }
    __syncwarp();
}

// The same by one lane.
template <bool CACHED, class Queue>
__device__ __forceinline__ void narrow_check_lane(const Dev &D, const Codes<CACHED> &codes, Acc *acc, Queue &Q, NarrowRound &R,
                                                  uint32_t o, uint32_t y)
{
    const LaneCheck r = lane_check(D, codes, R.fresh, o);
    const NarrowClaim C = narrow_claim(D, codes, acc, Q, R, r.id, r.sat, r.n_un, r.ul);
    if (C.k == 0xFFFFFFFFu) return;
    const uint32_t x = r.ul >> 1;
    narrow_queue(Q, R.buf, R.slot, C.k, C.at, x | ((r.ul & 1u) ? 0u : TRAIL_F), r.id, C.a0, C.a1, 0u, 1u);
    if (C.k < Queue::N && !r.len) {
        uint32_t u[8];
        u[0] = y;
#pragma unroll
        for (uint32_t q = 0; q < 7u; q++) u[q + 1u] = r.l[q] == PAD_LIT ? x : r.l[q] >> 1;
        Q.u[R.buf][C.k][0] = make_uint4(u[0], u[1], u[2], u[3]);
        Q.u[R.buf][C.k][1] = make_uint4(u[4], u[5], u[6], u[7]);
    }
}

// Bitmaps of entries [i0, i0 + step, ...) of the n in queue buf (trail from qs).
template <class Queue>
__device__ __forceinline__ void narrow_bitmaps(const Dev &D, const Queue &Q, uint32_t buf, uint32_t qs, uint32_t n, uint32_t i0,
                                               uint32_t step, uint32_t nw)
{
    for (uint32_t i = i0; i < n; i += step) {
        if (i < Queue::N) {
            const uint4 c = Q.e[buf][i];
            narrow_deps(D, c.x & TRAIL_VAR, c.y, &Q.u[buf][i][0], nw, threadIdx.x & 7u, 8u);
        } else {
            const uint32_t x = __ldcg(D.trail + qs + i) & TRAIL_VAR;
            narrow_deps(D, x, __ldcg(D.reason + x), nullptr, nw, threadIdx.x & 7u, 8u);
        }
    }
}

// Rounds of one narrow phase.  The search's time budget is looked at between
// phases, and the grid's other CTAs wait for the end of this one at a barrier
// that gives up (20 s): a chain a_i :- a_(i-1) claims one variable a round for
// three rounds an atom, so a phase that ran to the fixpoint overran a budget of
// 200 ms by 350 ms on a chain of 100k atoms, and from about 2M atoms on it
// would have outlasted the barrier.  1024 rounds are about 2.5 ms; the phase
// that follows costs a few us.
constexpr uint32_t NARROW_ROUNDS = 1024u;

// Occurrences of a round that one CTA of a grid follows, and why it ends its
// phase: the next round has more of them, or (LEAVE_LONG + their number) long
// lists were put off.  Closures with 960, 1920, 3840 and 7680 occurrences in one
// round, by one CTA and by the grid: 122 and 130, 147 and 146, 167 and 155, 253
// and 166 us (1.1M literals); 206 and 197, 244 and 198, 316 and 199, 388 and 215
// (22M).  A round of narrow_max claims has about 1000.
constexpr uint32_t NARROW_OCC = 2048u, LEAVE_WIDE = 1u, LEAVE_LONG = 2u;

// Propagation by one CTA, following the claims instead of sweeping the store
// (Algorithm 2's Last/Next): the trail entries [first, tend) are the
// assignments whose nogoods have not been checked yet (claims of the phase
// before, or the decision, whose level and bitmap are in memory); every other
// static nogood is as a sweep left it.  A round takes each entry's occurrence
// list for the literal that now holds -- only those nogoods can have become
// unit or violated -- and claims become the next round's entries, at
// tbase, tbase + 1, ... of the trail.  Ends when a round claims nothing, on a
// conflict, after NARROW_ROUNDS rounds, or when a round claims more than
// D.narrow_max (every CTA following a part is then the faster way).  A list of
// more than D.long_list occurrences that is not among the items is not walked by
// its warp: it ends the phase (*leave = LEAVE_LONG + such lists), after which all
// of one CTA's warps walk it (long_lists) or a grid sweeps the store.  In a grid
// a phase also ends, at once if need be, when a round's lists hold more than
// NARROW_OCC (LEAVE_WIDE).
//
// Why: a search round assigns a few dozen variables (62 on average in the
// 100k-atom program), and a sweep round costs its chain of barriers and loads
// (15 us there on 152 CTAs) whatever its claims.  Here a round is bound by a
// chain of list entry, codes, claim (two loads and an atomic from L2, about
// 0.6 us) and the instructions around it.  A claim puts its list's positions
// into the next round's items, so a quad of lanes checks one nogood whatever
// the lists' lengths (a program whose codes fit keeps a copy of them in shared
// memory, which halves the chain); two thirds of the warps check while the
// others compute the bitmaps of the round's entries (nothing in the round reads
// those), from the variables that the claim left in shared memory.
// The fresh bits alternate by round exactly as in sweeps: an entry's bit is
// cleared while its round runs, when only the other parity's bit hides a
// variable.  Returns the number of rounds; *n_claims is the number of claims,
// *n_left that of the last ones, still to be checked.
template <bool CACHED, class Queue>
__device__ __forceinline__ uint32_t narrow_rounds(const Dev &D, uint32_t *cache, Queue &Q, Acc *acc, uint32_t cdl, uint32_t round,
                                                  uint32_t first, uint32_t tend, uint32_t tbase, uint32_t *n_claims, uint32_t *n_left,
                                                  uint32_t *leave)
{
    constexpr uint32_t N = Queue::N, M = Queue::M;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nwarp = blockDim.x >> 5;
    const uint32_t nw = cdl > 1u ? deps_words(D, cdl) : 0u;
    const Codes<CACHED> codes{CACHED ? cache : D.asg};
    // warps [0, wa) check nogoods, the others compute bitmaps; all do both
    // when there is one warp, and all check at the root level
    const bool split = nw && nwarp > 1u;
    const uint32_t wa = split ? max(1u, nwarp * 2u / 3u) : nwarp;
    if (tid < 3u) Q.count[tid] = NarrowCount{};
    if (CACHED)
        for (uint32_t w = tid; w < D.asg_words; w += blockDim.x) cache[w] = __ldcg(D.asg + w);
    cta_sync();
    if (tid == 0 && tend - first > N) Q.count[0].rest = 1u;
    for (uint32_t i = tid; i < min(tend - first, N); i += blockDim.x) {
        const uint32_t e = __ldcg(D.trail + first + i), l = mk_lit(e & TRAIL_VAR, (e & TRAIL_F) != 0u);
        if ((l >> 1) >= D.nv) { atomicExch(&D.bar->err, 2u); Q.e[0][i] = make_uint4(0u, 0u, 0u, 0u); continue; }   // corrupt trail
        const uint32_t a0 = __ldg(D.occ_off + l), a1 = __ldg(D.occ_off + l + 1u);
        narrow_queue(Q, 0u, 0u, i, atomicAdd(&Q.count[0].m, a1 - a0), e, 0u, a0, a1, 0u, 1u);
    }
    cta_sync();
    const uint32_t occ_max = D.G > 1u ? NARROW_OCC : 0xFFFFFFFFu;
    uint32_t qs = first, qn = tend - first, it = 0;
    NarrowCount count = Q.count[0];
    NarrowRound R{cdl, 0u, 0u, 0u, tbase, 0u, 0u};
    for (bool done = count.m > occ_max; !done;) {
        const uint32_t cur = it & 1u, stale = 4u << ((round + 1u) & 1u), items = min(count.m, M), rest = count.rest;
        R.fresh = 4u << (round & 1u);
        R.buf = cur ^ 1u;
        R.slot = (it + 1u) % 3u;
        // cleared for the next round's claims; last read two barriers ago
        if (tid == 0) Q.count[(it + 2u) % 3u] = NarrowCount{};
        if (warp < wa) {
            for (uint32_t i0 = warp * 8u; i0 < items; i0 += wa * 8u) {
                const uint32_t i = i0 + (lane >> 2);
                const uint2 t = i < items ? Q.item[cur][i] : make_uint2(0xFFFFFFFFu, 0u);
                narrow_check(D, codes, acc, Q, R, t.x, t.y);
            }
            // lists past the items, and entries past the queue: many, so a lane
            // each
            for (uint32_t i0 = warp * 32u; rest && i0 < qn; i0 += wa * 32u) {
                const uint32_t i = i0 + lane;
                uint32_t y = 0, o = 0, o1 = 0;
                if (i < qn) {
                    if (i < N) {
                        const uint4 c = Q.e[cur][i];
                        y = c.x & TRAIL_VAR; o = c.z; o1 = c.w;
                    } else {
                        const uint32_t e = __ldcg(D.trail + qs + i), l = mk_lit(e & TRAIL_VAR, (e & TRAIL_F) != 0u);
                        y = e & TRAIL_VAR;
                        if (y >= D.nv) { atomicExch(&D.bar->err, 2u); y = 0u; }
                        else { o = __ldg(D.occ_off + l); o1 = __ldg(D.occ_off + l + 1u); }
                    }
                }
                if (o1 - o > D.long_list) {
                    const uint32_t k = atomicAdd(&Q.count[R.slot].nlong, 1u);
                    if (k < LONG_LISTS) { Q.lng[k] = make_uint4(o, o1, y, 0u); o1 = o; }
                }
                warp_lists_lanes(o, o1 - o, [&](uint32_t oc, uint32_t li) {
                    const uint32_t yo = __shfl_sync(FULL_MASK, y, li);
                    if (oc != 0xFFFFFFFFu) narrow_check_lane(D, codes, acc, Q, R, oc, yo);
                    __syncwarp();
                });
            }
        }
        // the entries' fresh bits, from the last warps backwards (they
        // have the fewest items)
        for (uint32_t i = blockDim.x - 1u - tid; i < qn; i += blockDim.x) {
            const uint32_t y = (i < N ? Q.e[cur][i].x : __ldcg(D.trail + qs + i)) & TRAIL_VAR;
            if (y >= D.nv) continue;
            const uint32_t clear = ~(stale << ((y & 7u) * 4u));
            if (CACHED) atomicAnd(cache + (y >> 3), clear);
            atomicAnd(D.asg + (y >> 3), clear);
        }
        // bitmaps of this round's entries (the first round's have theirs)
        if (nw && it > 0u && (!split || warp >= wa))
            narrow_bitmaps(D, Q, cur, qs, qn, (split ? warp - wa : warp) * 4u + (lane >> 3), (split ? nwarp - wa : nwarp) * 4u, nw);
        cta_sync();
        count = Q.count[R.slot];
        const uint32_t n_new = count.n;
        done = n_new - 1u >= D.narrow_max || (count.conf | count.nlong) || R.out + n_new > D.nv || count.m > occ_max || it + 1u >= NARROW_ROUNDS;
        qs = R.out;
        qn = n_new;
        R.out += n_new;
        round++;
        it++;
    }
    *leave = count.nlong ? LEAVE_LONG + min(count.nlong, LONG_LISTS) : count.m > occ_max ? LEAVE_WIDE : 0u;
    // the last claims' bitmaps, by every warp
    if (nw && it) narrow_bitmaps(D, Q, it & 1u, qs, qn, warp * 4u + (lane >> 3), nwarp * 4u, nw);
    cta_sync();
    const uint32_t c32 = __reduce_add_sync(FULL_MASK, R.checks), v32 = __reduce_add_sync(FULL_MASK, R.visits);
    if (lane == 0 && v32) {
        atomicAdd(&acc->checks, (unsigned long long)c32);
        atomicAdd(&acc->visits, (unsigned long long)v32);
    }
    *n_claims = R.out - tbase;
    *n_left = qn;
    return it;
}

// The lists that one CTA's narrow rounds put off, by all of its warps, as the
// tail of the last round (X.fresh is that round's, so its claims stay unseen).
// Apart from the rounds, whose every instruction counts: shared out there, the
// lists cost 2 to 7 % of searches that have none.  A closure with a list of 800
// occurrences takes 166 us, and took 187 with one warp on it.
__device__ __forceinline__ void long_lists(const SweepCtx &X, const uint4 *lists, uint32_t n)
{
    const uint32_t nw = X.cdl > 1u ? deps_words(*X.D, X.cdl) : 0u;
    uint32_t checks = 0, visits = 0;
    for (uint32_t i = 0; i < n; i++) {
        const uint4 t = lists[i];
        for (uint32_t o = t.x + threadIdx.x; o < t.y; o += blockDim.x) list_check_lane(X, o, t.z, nw, checks, visits);
    }
    __syncwarp();
    checks = __reduce_add_sync(FULL_MASK, checks);
    visits = __reduce_add_sync(FULL_MASK, visits);
    if ((threadIdx.x & 31u) == 0u && visits) {
        atomicAdd(&X.acc->checks, (unsigned long long)checks);
        atomicAdd(&X.acc->visits, (unsigned long long)visits);
    }
}

// Test-only failure injection: CTA D.stall_cta (thread 0) waits on a flag
// that nothing sets, so it does not reach the first phase barrier in time.
// The wait ends when another CTA has given up on that barrier (its error
// flag) or after three times the barrier's limit, whichever comes first.
__device__ __forceinline__ void injected_stall(const Dev &D)
{
    if (blockIdx.x != D.stall_cta || threadIdx.x != 0) return;
    const unsigned long long t0 = globaltimer_ns();
    while (ld_acquire_u32(&D.bar->stall) == 0u) {
        if (ld_acquire_u32(&D.bar->err)) break;
        if (globaltimer_ns() - t0 > 3ull * D.barrier_ns) break;
        __nanosleep(1000);
    }
}

// Algorithm 1 on the device.  rank/size: thread index and thread count of
// the solving group; cta: this CTA's part of the program's static partition;
// cta0/leader: the CTA and thread that run conflict analysis and write the
// next control block.  LISTS: bucket nogoods are followed through the
// occurrence lists only, as in programs with D.lists (no sweep code, no view).
template <bool BATCH, bool LISTS>
__device__ __forceinline__ void solver_loop(const Dev &D, const Smem &S, const View &V, uint32_t rank,
                                            uint32_t size, bool cta0, bool leader, uint32_t cta)
{
    __shared__ Ctl sC;
    __shared__ Acc sA;
    const uint32_t gtid = rank, nthreads = size;
    const bool lists = LISTS || D.lists;
    // leader-only counters (shared memory, not registers of every thread),
    // written to the stats when the search ends
    __shared__ unsigned long long t_start, t_phase, n_conf, n_phases, ns_bar, ns_sw, ns_an, ns_de, ns_st;
    __shared__ unsigned long long ns_slow, ns_slow_sw, ns_slow_long, ns_slow_buck, t_cta0;
    // restarts: learned nogoods since the last restart, restarts so far
    __shared__ uint32_t r_conf, r_idx;
    if (leader) {
        t_start = globaltimer_ns();
        t_phase = t_start;
        n_conf = n_phases = ns_bar = ns_sw = ns_an = ns_de = ns_st = ns_slow = ns_slow_sw = 0ull;
        ns_slow_long = ns_slow_buck = 0ull;
        r_conf = 0u;
        r_idx = 0u;
    }
    if (threadIdx.x == 0) { s_tlearned = 0ull; s_tbuckets = 0ull; s_wmax[0] = s_wmax[1] = 0ull; t_cta0 = globaltimer_ns(); }

    if (threadIdx.x < 32u) ldcg_copy(&sC, D.ctl);
    if (D.heuristic == 2) {
        uint16_t *w = const_cast<uint16_t *>(reinterpret_cast<const uint16_t *>(S.mlp));
        for (uint32_t i = threadIdx.x; i < (uint32_t)MLP_PARAMS; i += blockDim.x) w[i] = __ldg(D.mlp + i);
    }
    cta_sync();
    if (!lists) view_reload(D, V, 4u << (sC.round & 1u));
    unit_table(D, cta, lists);
    cta_sync();

    for (uint32_t k = 0;; k++) {
        if (threadIdx.x < 32u) {
            ldcg_copy(&sC, D.ctl + (k & 1u));
            ldcg_copy(&sA, D.acc + ((k + 3u) & 3u));
        }
        cta_sync();
        const Ctl C = sC;
        const Acc A = sA;
        if (leader) { ns_slow += A.tbusy; ns_slow_sw += A.tsweep; ns_slow_long += A.tlong; ns_slow_buck += A.tbuck; }
        if (C.op == OP_DONE) break;
        Acc *acc = D.acc + (k & 3u);
        // the next control block, written by the leader only (kept in
        // shared memory rather than in every thread's registers)
        __shared__ Ctl sN;
        Ctl &N = sN;
        if (leader) N = C;
        int kind = 0;   // 0 sweep, 1 analysis, 2 decision, 3 stability
        const uint32_t tend = C.tb + A.nclaim;
        const uint32_t fresh_cur = 4u << (C.round & 1u);
        const uint32_t fresh_prev = 4u << ((C.round + 1u) & 1u);

        // the propagate-and-check sweep of ROUND and APPLY runs after the
        // switch (one copy of its code)
        bool sw = false, sw_full = true, nar = false;
        uint32_t sw_cdl = 0, sw_tbase = 0, sw_fr0 = 0, sw_fr1 = 0;
        switch (C.op) {
        case OP_INIT: {
            SweepCtx X{&D, V, fresh_cur, 1u, tend, acc, true, false, cta, rank >> 5, size >> 5};
            if (leader && D.heuristic == 5) reinterpret_cast<float *>(D.act)[D.J] = 1.0f;   // the first increment
            for (uint32_t i = gtid; i < D.n_units; i += nthreads) {
                uint32_t id = D.units_base + i;
                uint32_t l = __ldg(D.lits + id) & ~END_BIT;
                uint32_t v = l >> 1;
                uint32_t val = global_val(D, v, fresh_cur);
                uint32_t own = (l & 1u) ? V_F : V_T;
                if (val == 0u) {
                    const uint32_t valbit = (l & 1u) ? V_T : V_F;
                    int r = claim_var(D.asg, v, valbit, fresh_cur);
                    if (r == 0) record_claim(X, v, valbit, id);
                    else if (r == 2) report_conflict(X, id, 1u);
                } else if (val == own) {
                    report_conflict(X, id, 1u);
                }
            }
            if (leader) {
                N.op = OP_ROUND; N.round = C.round + 1u; N.tb = tend; N.tc = C.tc; N.tcom = C.tc; N.clean = 0; N.full = 1;
            }
            break;
        }
        case OP_ROUND: {
            if (A.ckey != NO_KEY) {
                kind = 1;
                if (D.mode == MODE_PROPAGATE || C.cdl <= 1u) {
                    if (leader) {
                        N.op = OP_DONE;
                        N.conflict = 1;
                        N.status = C.n_models > 0 ? 10 : 20;
                        atomicAdd(&D.stats->conflicts, 1ull);
                        n_conf++;
                    }
                    break;
                }
                if (cta0) {
                    // the conflicts to analyse: the shortest one, then (several
                    // per round) the shortest of each id class, shorter first
                    __shared__ unsigned long long s_keys[4];
                    __shared__ uint32_t s_nk, s_stop;
                    if (leader) {
                        uint32_t nk = 0;
                        s_keys[nk++] = A.ckey;
                        for (int j = 0; j < 3; j++) {
                            unsigned long long key = A.cslot[j];
                            if (key == NO_KEY || key == A.ckey) continue;
                            uint32_t i = nk++;
                            while (i > 1u && s_keys[i - 1u] > key) { s_keys[i] = s_keys[i - 1u]; i--; }
                            s_keys[i] = key;
                        }
                        s_nk = min(nk, max(D.conf_per_round, 1u));
                        s_stop = 0u;
                        atomicAdd(&D.stats->conflict_rounds, 1ull);
                        N.target = 0xFFFFFFFFu;
                    }
                    cta_sync();
                    const uint32_t nk = s_nk;
                    for (uint32_t c = 0; c < nk; c++) {
                        const uint32_t g = (uint32_t)(s_keys[c] & 0xFFFFFFFFull);
                        const uint32_t lf = N.lfill;
                        if (D.learning) res_analyze(D, S, g, C.cdl, tend, lf);
                        else analyze(D, S, g, C.cdl, lf, true);
                        if (leader) {
                            atomicAdd(&D.stats->conflicts, 1ull);
                            n_conf++;
                            if (S.misc[0] == 2u) {
                                N.op = OP_DONE; N.err = -6; N.status = 0;
                                debug_analysis(D, g, tend, lf, 0u, S.misc[1], S.misc[3]);
                                D.stats->dbg_lfill = S.misc[2];
                                s_stop = 1u;
                            } else if (S.misc[0]) {
                                N.op = OP_DONE;
                                N.status = C.n_models > 0 ? 10 : 20;
                                s_stop = 1u;
                            } else {
                                uint32_t n = S.misc[2];
                                if (lf + n + 64u >= D.lits_cap || N.n_learned + 1u >= D.learned_ng_cap) {
                                    N.op = OP_DONE; N.err = -6; N.status = 0;
                                    s_stop = 1u;
                                } else {
                                    add_learned(D, N.n_learned, lf, n);
                                    N.n_learned = N.n_learned + 1u;
                                    N.lfill = lf + n;
                                    N.op = OP_BACKJUMP;
                                    N.target = min(N.target, S.misc[1]);
                                    N.tb = tend;
                                    atomicAdd(&D.stats->learned, 1ull);
                                    atomicAdd(&D.stats->learned_lits, (unsigned long long)n);
                                    debug_analysis(D, g, tend, lf, n, S.misc[1], D.learning ? S.misc[3] : 0u);
                                }
                            }
                        }
                        cta_sync();
                        if (s_stop) break;
                    }
                    if (leader && N.op == OP_BACKJUMP && D.restart_unit &&
                        ++r_conf >= luby(r_idx + 1u) * D.restart_unit) {
                        r_conf = 0u;
                        r_idx++;
                        N.target = 1u;
                        atomicAdd(&D.stats->restarts, 1ull);
                    }
                }
                break;
            }
            // without sweeps the caller's partial assignment is followed too
            const bool input = lists && D.mode == MODE_PROPAGATE && C.round == 1u;
            const bool quiet = A.nclaim == 0u && !input;   // no assignment is left to follow
            const bool owed = A.flag != 0u;                // lists passed over in the last round
            if (quiet && C.clean && !owed) {
                // fixpoint
                if (D.mode == MODE_PROPAGATE) {
                    if (leader) { N.op = OP_DONE; N.status = 0; }
                    break;
                }
                if (tend >= D.nv) {
                    kind = 3;
                    if (leader) N.op = OP_STAB_INIT;
                    break;
                }
                kind = 2;
                decide(D, S, acc, gtid, nthreads, C.cdl, tend);
                if (leader) N.op = OP_APPLY;
                break;
            }
            if (!quiet && (lists || (!C.full && !C.wide && !owed && A.nclaim <= D.narrow_max))) {
                nar = true; sw_cdl = C.cdl; sw_fr0 = input ? 0u : C.tb; sw_fr1 = sw_tbase = tend;
                if (leader) atomicAdd(&D.stats->props, (unsigned long long)A.nclaim);
                break;
            }
            // a full sweep, or the claims' lists, by the whole grid
            sw_full = !lists && (C.full != 0u || owed || (D.frontier == 0u && quiet) || (!quiet && A.nclaim > D.list_max));
            // make last round's claims visible: clear their fresh bit
            // (grid-wide) and put them in this CTA's view, which only sweeps
            // read
            for (uint32_t i = (quiet ? tend : C.tb) + gtid; i < tend; i += nthreads) {
                uint32_t v = __ldcg(D.trail + i) & TRAIL_VAR;
                if (v >= D.nv) { atomicExch(&D.bar->err, 2u); continue; }   // corrupt trail: stop with an error
                atomicAnd(D.asg + (v >> 3), ~(fresh_prev << ((v & 7u) * 4u)));
            }
            if (sw_full) {
                if (tend - C.tc > 4096u) {
                    view_reload(D, V, fresh_cur);
                } else {
                    for (uint32_t i = C.tc + threadIdx.x; i < tend; i += blockDim.x) {
                        const uint32_t e = __ldcg(D.trail + i);
                        view_set(V, e & TRAIL_VAR, (e & TRAIL_F) ? V_F : V_T);
                    }
                }
            }
            cta_sync();
            sw = true; sw_cdl = C.cdl; sw_tbase = tend;
            if (!sw_full && !quiet) { sw_fr0 = C.tb; sw_fr1 = tend; }
            if (leader) {
                N.op = OP_ROUND; N.round = C.round + 1u; N.tc = sw_full ? tend : C.tc; N.tb = tend; N.tcom = tend; N.full = 0; N.wide = 0;
                N.clean = lists || D.frontier != 0u || sw_full;
                atomicAdd(&D.stats->rounds, 1ull);
                atomicAdd(&D.stats->props, (unsigned long long)A.nclaim);
                if (sw_full) atomicAdd(&D.stats->checks, D.static_checks);
                atomicAdd(&D.stats->visits, (sw_full ? D.static_nogoods : 0ull) + D.n_long + C.n_learned);
            }
            break;
        }
        case OP_APPLY: {
            if (A.dkey == 0ull) {
                // CompleteAssignment: falsify the unassigned atoms; their
                // dependency bitmap is every decision level so far
                kind = 2;
                SweepCtx X{&D, V, fresh_cur, C.cdl, tend, acc, true, false, cta, rank >> 5, size >> 5};
                const uint32_t nw = deps_words(D, C.cdl);
                for (uint32_t p = gtid; p < D.na; p += nthreads) {
                    if ((nib(__ldcg(D.asg + (p >> 3)), p) & 3u) != 0u) continue;
                    if (claim_var(D.asg, p, V_F, fresh_cur) == 0) {
                        record_claim(X, p, V_F, R_COMPLETE);
                        if (C.cdl > 1u)
                            for (uint32_t w = 0; w < nw; w++)
                                D.deps[(size_t)p * D.WW + w] = all_levels_word(D, C.cdl, w);
                    }
                }
                if (leader) {
                    N.op = OP_ROUND; N.round = C.round + 1u; N.tb = tend; N.tcom = tend; N.clean = 0;
                    N.full = 0;
                    atomicAdd(&D.stats->completions, 1ull);
                }
                break;
            }
            const uint32_t j = 0xFFFFFFFFu - (uint32_t)(A.dkey & 0xFFFFFFFFull);
            if (j >= D.J || C.cdl + 1u > D.J + 1u) {
                // a decision key that names no rule: stop with an error
                // rather than write outside the arrays
                if (leader) { N.op = OP_DONE; N.err = -6; N.status = 0; }
                break;
            }
            const uint32_t L = C.cdl + 1u;
            const uint32_t bv = D.na + 3u * j;
            if (leader) {
                D.level_start[L] = tend;
                D.dec_var[L] = bv;
                D.trail[tend] = bv;
                if (D.tpos) D.tpos[bv] = tend;
                D.dl[bv] = (int32_t)L;
                D.reason[bv] = R_DECISION;
                uint32_t nw = deps_words(D, L), bit = level_bit(D, L);
                for (uint32_t w = 0; w < nw; w++)
                    D.deps[(size_t)bv * D.WW + w] = (w == (bit >> 6)) ? (1ull << (bit & 63u)) : 0ull;
                __threadfence();
                atomicOr(D.asg + (bv >> 3), V_T << ((bv & 7u) * 4u));
            }
            // the decision's consequences by narrow rounds: the store is at a
            // fixpoint, so only the decision's nogoods can change it
            nar = true; sw_cdl = L; sw_fr0 = tend; sw_fr1 = sw_tbase = tend + 1u;
            if (leader) {
                N.cdl = L;
                atomicAdd(&D.stats->decisions, 1ull);
                if ((unsigned long long)L > D.stats->max_level) D.stats->max_level = L;
            }
            break;
        }
        case OP_BACKJUMP: {
            kind = 1;
            const uint32_t newend = __ldcg(D.level_start + C.target + 1u);
            for (uint32_t i = newend + gtid; i < tend; i += nthreads) {
                uint32_t v = __ldcg(D.trail + i) & TRAIL_VAR;
                if (v >= D.nv) { atomicExch(&D.bar->err, 2u); continue; }
                atomicAnd(D.asg + (v >> 3), ~(0xFu << ((v & 7u) * 4u)));
                D.dl[v] = 0;
            }
            if (!lists)
                for (uint32_t i = newend + threadIdx.x; i < tend; i += blockDim.x)
                    view_clear(V, __ldcg(D.trail + i) & TRAIL_VAR);
            if (leader) {
                N.op = OP_ROUND; N.cdl = C.target; N.tc = min(C.tc, newend); N.tb = newend; N.tcom = newend; N.clean = 0; N.full = 1;
            }
            break;
        }
        case OP_STAB_INIT: {
            kind = 3;
            const uint32_t words = (D.na + 31u) >> 5;
            for (uint32_t w = gtid; w < words; w += nthreads) D.lm[w] = 0u;
            if (leader) { N.op = OP_STAB_ITER; N.stab_first = 1; N.tb = tend; }
            if (!BATCH && gridDim.x > 1u) break;
            // one CTA goes on in this phase
        }
        [[fallthrough]];
        case OP_STAB_ITER: {
            kind = 3;
            if (BATCH || gridDim.x == 1u) {
                // one CTA: several passes in a phase
                __shared__ uint32_t s_more;
                uint32_t more = 1u;
                for (uint32_t i = 0; more && i < STAB_PASSES; i++) {
                    cta_sync();
                    if (threadIdx.x == 0) s_more = 0u;
                    cta_sync();
                    if (least_model_pass(D, gtid, nthreads)) s_more = 1u;
                    cta_sync();
                    more = s_more;
                }
                if (!more) {
                    unfounded_min(D, acc, gtid, nthreads);
                    if (leader) N.op = OP_STAB_RESULT;
                }
                break;
            }
            if (!C.stab_first && A.flag == 0u) {
                // least model reached: look for true atoms outside it
                unfounded_min(D, acc, gtid, nthreads);
                if (leader) N.op = OP_STAB_RESULT;
                break;
            }
            if (least_model_pass(D, gtid, nthreads)) atomicOr(&acc->flag, 1u);
            if (leader) { N.op = OP_STAB_ITER; N.stab_first = 0; }
            break;
        }
        case OP_STAB_RESULT: {
            kind = 3;
            if (A.minU == 0xFFFFFFFFu) {
                // answer set: record it, then block it with the decision literals
                const long long row = C.n_models;
                const uint32_t words = (D.na + 63u) >> 6;
                if (D.trace && row == 0) {
                    // label each sampled candidate: does its body hold in the answer set
                    const uint32_t nrec = min(__ldcg(&D.stats->trace_n), D.trace_cap);
                    for (uint32_t r = gtid; r < nrec; r += nthreads) {
                        uint32_t *rec = D.trace + (size_t)r * TRACE_WORDS;
                        const uint32_t b = D.na + 3u * rec[16];
                        rec[18] = (nib(__ldcg(D.asg + (b >> 3)), b) & 3u) == V_T ? 1u : 0u;
                        rec[19] = 1u;
                    }
                }
                if (row < D.models_cap) {
                    for (uint32_t w = gtid; w < words; w += nthreads) {
                        unsigned long long m = 0;
                        for (uint32_t q = 0; q < 64u; q++) {
                            uint32_t p = w * 64u + q;
                            if (p < D.na && (nib(__ldcg(D.asg + (p >> 3)), p) & 3u) == V_T) m |= 1ull << q;
                        }
                        D.models[(size_t)row * words + w] = m;
                    }
                }
                if (leader) {
                    atomicAdd(&D.stats->models, 1ull);
                    N.n_models = C.n_models + 1;
                    if ((D.max_models > 0 && N.n_models >= D.max_models) || C.cdl <= 1u) {
                        N.op = OP_DONE; N.status = 10;
                    } else if (C.lfill + C.cdl + 64u >= D.lits_cap || C.n_learned + 1u >= D.learned_ng_cap) {
                        N.op = OP_DONE; N.err = -6; N.status = 10;
                    } else {
                        uint32_t n = 0;
                        for (uint32_t level = 2; level <= C.cdl; level++)
                            D.lits[C.lfill + n++] = mk_lit(__ldcg(D.dec_var + level), false);
                        D.lits[C.lfill + n - 1u] |= END_BIT;
                        add_learned(D, C.n_learned, C.lfill, n);
                        N.n_learned = C.n_learned + 1u;
                        N.lfill = C.lfill + n;
                        N.op = OP_BACKJUMP;
                        N.target = C.cdl - 1u;
                        atomicAdd(&D.stats->learned, 1ull);
                        atomicAdd(&D.stats->learned_lits, (unsigned long long)n);
                    }
                }
                break;
            }
            // not an answer set: loop nogood {Tp} u {Fb_j : head(j) in U,
            // body+(j) disjoint from U} for U = M \ LM(reduct), p = min U
            const uint32_t p = A.minU;
            for (uint32_t j = gtid; j < D.J; j += nthreads) {
                uint32_t h = (uint32_t)__ldg(D.rule_head + j);
                bool hU = ((nib(__ldcg(D.asg + (h >> 3)), h) & 3u) == V_T) && !((__ldcg(D.lm + (h >> 5)) >> (h & 31u)) & 1u);
                if (!hU) continue;
                bool ext = true;
                for (uint32_t q = __ldg(D.rpos_off + j); ext && q < __ldg(D.rpos_off + j + 1); q++) {
                    uint32_t a = __ldg(D.rpos + q);
                    bool aU = ((nib(__ldcg(D.asg + (a >> 3)), a) & 3u) == V_T) && !((__ldcg(D.lm + (a >> 5)) >> (a & 31u)) & 1u);
                    if (aU) ext = false;
                }
                if (ext) {
                    uint32_t pos = C.lfill + 1u + atomicAdd(&acc->nlits, 1u);
                    if (pos + 64u < D.lits_cap) D.lits[pos] = mk_lit(D.na + 3u * j, true);
                }
            }
            if (leader) {
                D.lits[C.lfill] = mk_lit(p, false);
                N.op = OP_ANALYZE_ID;
                N.conf_id = C.lfill;
                atomicAdd(&D.stats->loops, 1ull);
            }
            break;
        }
        case OP_ANALYZE_ID: {
            kind = 1;
            const uint32_t len = 1u + A.nlits;
            if (C.lfill + len + C.cdl + 64u >= D.lits_cap || C.n_learned + 2u >= D.learned_ng_cap) {
                if (leader) { N.op = OP_DONE; N.err = -6; N.status = C.n_models > 0 ? 10 : 0; }
                break;
            }
            if (cta0) {
                if (leader) {
                    D.lits[C.lfill + len - 1u] |= END_BIT;
                    add_learned(D, C.n_learned, C.lfill, len);
                    __threadfence();
                }
                cta_sync();
                const uint32_t lf = C.lfill + len;
                if (D.learning) res_analyze(D, S, C.conf_id, C.cdl, tend, lf);
                else analyze(D, S, C.conf_id, C.cdl, lf, false);
                if (leader) {
                    atomicAdd(&D.stats->conflicts, 1ull);
                    n_conf++;
                    atomicAdd(&D.stats->learned, 1ull);
                    atomicAdd(&D.stats->learned_lits, (unsigned long long)len);
                    if (S.misc[0] == 2u) {
                        N.op = OP_DONE; N.err = -6; N.status = 0;
                        debug_analysis(D, C.conf_id, tend, lf, 0u, S.misc[1], S.misc[3]);
                        D.stats->dbg_lfill = S.misc[2];
                    } else if (S.misc[0]) {
                        N.op = OP_DONE;
                        N.status = C.n_models > 0 ? 10 : 20;
                        N.n_learned = C.n_learned + 1u;
                        N.lfill = lf;
                    } else {
                        uint32_t n = S.misc[2];
                        add_learned(D, C.n_learned + 1u, lf, n);
                        N.n_learned = C.n_learned + 2u;
                        N.lfill = lf + n;
                        N.op = OP_BACKJUMP;
                        N.target = S.misc[1];
                        atomicAdd(&D.stats->learned, 1ull);
                        atomicAdd(&D.stats->learned_lits, (unsigned long long)n);
                        debug_analysis(D, C.conf_id, tend, lf, n, S.misc[1], D.learning ? S.misc[3] : 0u);
                        if (D.restart_unit && ++r_conf >= luby(r_idx + 1u) * D.restart_unit) {
                            r_conf = 0u;
                            r_idx++;
                            N.target = 1u;
                            atomicAdd(&D.stats->restarts, 1ull);
                        }
                    }
                }
            }
            break;
        }
        default:
            if (leader) { N.op = OP_DONE; N.err = -6; }
            break;
        }
        if (nar && cta0) {
            // few claims (or the decision): CTA 0 follows them, the others wait
            // at the barrier; their views catch up with the trail
            // at the next sweep.  A full-sweep program confirms the fixpoint
            // with a sweep; so does a program with long or learned nogoods,
            // which no list holds
            // (several CTAs share an SM in batches, with their views beside it)
            constexpr uint32_t QN = !BATCH ? 192u : LISTS ? 96u : 24u;
            __shared__ NarrowQueue<QN, 4u * QN> Q;
            cta_sync();
            uint32_t n = 0, left = 0, leave = 0;
            // without lists (only decisions come here then) it is left to a sweep
            uint32_t its = 0;
            if (D.narrow_max == 0u) { left = sw_fr1 - sw_fr0; leave = LEAVE_LONG + 1u; }
            else its = D.code_cache
                ? narrow_rounds<true>(D, S.codes, Q, acc, sw_cdl, C.round, sw_fr0, sw_fr1, sw_tbase, &n, &left, &leave)
                : narrow_rounds<false>(D, S.codes, Q, acc, sw_cdl, C.round, sw_fr0, sw_fr1, sw_tbase, &n, &left, &leave);
            if (leave > LEAVE_LONG && D.G == 1u && its) {
                SweepCtx X{&D, V, 4u << ((C.round + its - 1u) & 1u), sw_cdl, sw_tbase + n, acc, true, false, cta, rank >> 5, size >> 5};
                long_lists(X, Q.lng, leave - LEAVE_LONG);
                cta_sync();
                leave = 0u;
            }
            if (leader) {
                // the trail's last `left` claims, and those of the long lists
                // after them, are still to be followed
                N.op = OP_ROUND; N.round = C.round + its; N.tb = N.tcom = sw_tbase + n - left;
                N.full = leave > LEAVE_LONG; N.wide = leave == LEAVE_WIDE;
                N.clean = (lists || D.frontier != 0u) && D.n_long + C.n_learned == 0u && leave <= LEAVE_LONG;
                atomicAdd(&acc->nclaim, left);
                atomicAdd(&D.stats->props, (unsigned long long)((long long)n - (long long)left));
                atomicAdd(&D.stats->rounds, (unsigned long long)its);
            }
        }
        if (sw) {
            const unsigned long long ts = threadIdx.x == 0 ? globaltimer_ns() : 0ull;
            SweepCtx X{&D, V, fresh_cur, sw_cdl, sw_tbase, acc, true, !lists, cta, rank >> 5, size >> 5};
            sweep<LISTS>(X, C.n_learned, sw_full, sw_fr0, sw_fr1);
            if (threadIdx.x == 0) atomicMax(&acc->tsweep, globaltimer_ns() - ts);
        }

        if (leader) {
            if (D.mode == MODE_SOLVE && N.op != OP_DONE) {
                unsigned long long now = globaltimer_ns();
                bool over_time = D.time_budget_ns > 0 && (long long)(now - t_start) > D.time_budget_ns;
                bool over_conf = D.conflict_budget > 0 && (long long)n_conf >= D.conflict_budget;
                if (over_time || over_conf) { N.op = OP_DONE; N.status = N.n_models > 0 ? 10 : 0; }
            }
            D.ctl[(k + 1u) & 1u] = N;
            Acc z;
            z.ckey = NO_KEY; z.cslot[0] = z.cslot[1] = z.cslot[2] = NO_KEY; z.dkey = 0; z.nclaim = 0; z.flag = 0; z.minU = 0xFFFFFFFFu; z.nlits = 0; z.checks = 0; z.visits = 0;
            z.tbusy = 0; z.tsweep = 0; z.tlong = 0; z.tbuck = 0;
            D.acc[(k + 1u) & 3u] = z;
            // fold long-nogood checks of the previous phase into the stats
            if (A.checks) atomicAdd(&D.stats->checks, A.checks);
            if (A.visits) atomicAdd(&D.stats->visits, A.visits);
            unsigned long long now = globaltimer_ns();
            unsigned long long dt = now - t_phase;
            t_phase = now;
            if (kind == 0) ns_sw += dt;
            else if (kind == 1) ns_an += dt;
            else if (kind == 2) ns_de += dt;
            else ns_st += dt;
            n_phases++;
            if (!BATCH && gridDim.x > 1u) __threadfence();
        }
        const unsigned long long tb0 = threadIdx.x == 0 ? globaltimer_ns() : 0ull;
        if (threadIdx.x == 0) atomicMax(&acc->tbusy, tb0 - t_cta0);
        if (!BATCH && k == 0 && D.stall_cta != 0xFFFFFFFFu) injected_stall(D);
        if (!group_sync<BATCH>(D, k)) break;
        if (threadIdx.x == 0) t_cta0 = globaltimer_ns();
        if (leader) ns_bar += t_cta0 - tb0;
    }
    if (leader) {
        const Ctl F = sC;
        D.stats->pad = F.tcom;
        D.stats->ns_total = globaltimer_ns() - t_start;
        D.stats->ns_sweep = ns_sw;
        D.stats->ns_analysis = ns_an;
        D.stats->ns_decision = ns_de;
        D.stats->ns_stab = ns_st;
        D.stats->phases = n_phases;
        D.stats->ns_barrier = ns_bar;
        D.stats->ns_learned = s_tlearned;
        D.stats->ns_buckets = s_tbuckets;
        D.stats->ns_slowest = ns_slow;
        D.stats->ns_slowest_sweep = ns_slow_sw;
        D.stats->ns_slowest_long = ns_slow_long;
        D.stats->ns_slowest_buckets = ns_slow_buck;
        int err = F.err;
        if (__ldcg(&D.bar->err)) err = -6;
        D.result[0] = F.status;
        D.result[1] = F.n_models;
        D.result[2] = err;
        D.result[3] = F.conflict;
    }
}

// The dynamic shared-memory limit is a property of each kernel, shared by
// every program: it is set to the largest size any program may use, and
// occupancy is computed for a program's own size.
constexpr int MAX_DYN_SMEM = (int)SOLVE_SMEM_BUDGET;

}  // namespace aspgpu
