// Allocation-free unit propagation (asp_propagate_noalloc).
//
// Some callers cannot allocate device memory on the path where they need
// propagation: real-time loops that must not enter the allocator (an
// allocation can block on the driver or trigger a synchronising free of
// cached blocks), and processes whose device memory is handed out up front
// by a pool or a framework that owns all of it.  This entry point computes the
// same closure as asp_debug_propagate, but all of its working memory (the
// assignment codes, the list of assigned literals, the round counters and the
// grid barrier) lives in one fixed static device array defined below.  It
// reads the program's nogood store and occurrence lists (created earlier by
// asp_load_ground) and the caller's device buffers, and allocates nothing.
//
// The array is shared by every call in the process: calls that overlap on
// the GPU (two streams, or two host threads) race on it and give wrong
// results.  Each call re-initialises what must start at zero.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "aspgpu.h"
#include "device.cuh"
#include "follow.cuh"
#include "store.h"

namespace aspgpu {

constexpr uint32_t NOALLOC_CTL_WORDS = 64;
// largest program the static array serves: 2^20 variables (4-bit codes)
constexpr uint32_t NOALLOC_MAX_VARS = 1u << 20;
constexpr uint32_t NOALLOC_CODES = NOALLOC_MAX_VARS / 8u;
constexpr uint32_t NOALLOC_WORDS = NOALLOC_CTL_WORDS + NOALLOC_CODES + NOALLOC_MAX_VARS;

// 512 KB of codes, 4 MB of list and 256 B of control words; every GPU that
// loads the library holds them until the process exits.
static __device__ __align__(256) uint32_t g_noalloc_scratch[NOALLOC_WORDS];

namespace {

struct NaCtl {                 // first words of the scratch array
    unsigned int count, err, conflict;
    // of the grid's rounds, by their number modulo 3 (a round clears the next
    // one's, whose last readers are two barriers back): literals listed, why to
    // stop following them (NA_CONFLICT, NA_LONG)
    unsigned int nclaim[3], stop[3];
    // CTA 0's narrow rounds: number of the next round, literals it left to
    // follow, why it stopped; and the counter of literals past its shared lists
    unsigned int next, left, nstop, nover;
};
// a nogood is violated; lists too long for a warp were passed over
constexpr unsigned int NA_CONFLICT = 1u, NA_LONG = 2u;

constexpr uint32_t NA_THREADS = 768, NA_LIST = 1024;
// claims that CTA 0 follows alone: a round of the grid costs its barrier and
// list copy (about 3 us) over the chain of loads of a narrow round, in which
// 192 claims go at a time
constexpr uint32_t NA_NARROW = 384;

__device__ __forceinline__ unsigned long long na_timer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t na_ld_acquire(const unsigned int *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// CTA barrier that counts every thread on its own: warps arrive from loops
// with different trip counts
__device__ __forceinline__ void na_cta_sync() { asm volatile("barrier.sync 0;" ::: "memory"); }

// grid barrier number gen on the scratch control words (its counter is zeroed
// before each launch); bounded wait (~20 s)
__device__ bool na_sync(NaCtl *c, uint32_t gen)
{
    __shared__ int s_ok;
    na_cta_sync();
    if (threadIdx.x == 0) {
        int ok = 1;
        if (gridDim.x > 1) {
            const uint32_t target = (gen + 1u) * gridDim.x;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(&c->count) : "memory");
            unsigned long long t0 = 0;
            for (unsigned spins = 1; (int)(na_ld_acquire(&c->count) - target) < 0; spins++) {
                if ((spins & 255u) != 0u) continue;
                const unsigned long long now = na_timer();
                if (t0 == 0) t0 = now;
                if (na_ld_acquire(&c->err) || now - t0 > 20000000000ull) {
                    atomicExch(&c->err, 1u);
                    ok = 0;
                    break;
                }
            }
            __threadfence();
        }
        s_ok = ok;
    }
    na_cta_sync();
    return s_ok != 0;
}

// value of variable v with claims of the current round (fresh bit) unseen
__device__ __forceinline__ uint32_t na_val(const uint32_t *asg, uint32_t v, uint32_t fresh)
{
    uint32_t c = (__ldcg(asg + (v >> 3)) >> ((v & 7u) * 4u)) & 0xFu;
    return (c & fresh) ? 0u : (c & 3u);
}

// The CTA's literals listed in the current round: shared memory first, then
// straight to the list (slots of counter *n after base).
struct NaList {
    uint32_t *list;            // of the scratch array
    uint32_t base;             // its first free word
    unsigned int *n;           // counter of the round
    uint32_t *s_lit;           // [NA_LIST]
    unsigned int *s_n;
    unsigned int *stop;        // the round's reasons to stop
};

__device__ __forceinline__ void na_push(const NaList &O, uint32_t l)
{
    const uint32_t i = atomicAdd(O.s_n, 1u);
    if (i < NA_LIST) { O.s_lit[i] = l; return; }
    const uint32_t pos = O.base + atomicAdd(O.n, 1u);
    if (pos < NOALLOC_MAX_VARS) O.list[pos] = l;
}

// Copies the CTA's literals to the list, one global atomic a CTA.
__device__ __forceinline__ void na_flush(const NaList &O)
{
    __shared__ uint32_t s_base;
    na_cta_sync();
    const uint32_t n = min(*O.s_n, NA_LIST);
    if (threadIdx.x == 0) s_base = O.base + (n ? atomicAdd(O.n, n) : 0u);
    na_cta_sync();
    const uint32_t b = s_base;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x)
        if (b + i < NOALLOC_MAX_VARS) O.list[b + i] = O.s_lit[i];
    if (threadIdx.x == 0) *O.s_n = 0u;
}

__device__ __forceinline__ void na_conflict(NaCtl *c, const NaList &O)
{
    atomicExch(&c->conflict, 1u);
    atomicOr(O.stop, NA_CONFLICT);
}

// claim the complement of literal l; conflict flag on a clash
__device__ __forceinline__ void na_claim(uint32_t *asg, NaCtl *c, uint32_t l, uint32_t fresh, const NaList &O)
{
    const uint32_t v = l >> 1, valbit = (l & 1u) ? V_T : V_F, sh = (v & 7u) * 4u;
    const uint32_t old = (atomicOr(asg + (v >> 3), (valbit | fresh) << sh) >> sh) & 3u;
    if (old == 0u) na_push(O, l ^ 1u);
    else if (!(old & valbit)) na_conflict(c, O);
}

// Checks the bucket nogoods of the n literals at `from` (each holds since the
// round before; no other nogood can have become unit or violated).  With up to
// eight literals a warp its quads share out their lists, for the shortest
// chain; with more its lanes do, 32 literals at a time.  A literal's own fresh
// bit, of the other parity, is cleared meanwhile.  SHARED: `from` is in shared
// memory.  A warp whose lists hold more than `longest` occurrences passes them
// over and stops the rounds for a sweep of the store (a literal of 130k nogoods
// kept one warp busy for 26 ms).
template <bool SHARED>
__device__ __forceinline__ void na_follow(const Dev &D, uint32_t *asg, NaCtl *c, const uint32_t *from, uint32_t n, uint32_t w,
                                          uint32_t nw, uint32_t fresh, uint32_t stale, uint32_t longest, const NaList &O)
{
    const uint32_t lane = threadIdx.x & 31u, each = min(32u, (n + nw - 1u) / nw);
    const Codes<false> codes{asg};
    for (uint32_t i0 = w * each; i0 < n; i0 += nw * each) {
        const uint32_t i = i0 + lane;
        uint32_t o0 = 0, count = 0;
        if (lane < each && i < n) {
            const uint32_t l = SHARED ? from[i] : __ldcg(from + i), y = l >> 1;
            o0 = __ldg(D.occ_off + l);
            count = __ldg(D.occ_off + l + 1u) - o0;
            atomicAnd(asg + (y >> 3), ~(stale << ((y & 7u) * 4u)));
        }
        if (__reduce_add_sync(0xFFFFFFFFu, count) > longest) {
            if (lane == 0) atomicOr(O.stop, NA_LONG);
            continue;
        }
        if (each <= 8u) {
            warp_lists(o0, count, [&](uint32_t o, uint32_t) {
                const QuadCheck r = quad_check(D, codes, fresh, o);
                if ((lane & 3u) == 0u && !r.sat && r.n_un < 2u) {
                    if (r.n_un == 0u) na_conflict(c, O);
                    else na_claim(asg, c, r.ul, fresh, O);
                }
                __syncwarp();
            });
        } else {
            warp_lists_lanes(o0, count, [&](uint32_t o, uint32_t) {
                if (o != 0xFFFFFFFFu) {
                    const LaneCheck r = lane_check(D, codes, fresh, o);
                    if (!r.sat && r.n_un == 0u) na_conflict(c, O);
                    else if (!r.sat && r.n_un == 1u) na_claim(asg, c, r.ul, fresh, O);
                }
                __syncwarp();
            });
        }
    }
}

// Checks every bucket nogood of the store, a lane each, and clears the fresh
// bits of the n literals at `from`.
__device__ __forceinline__ void na_sweep(const Dev &D, uint32_t *asg, NaCtl *c, const uint32_t *from, uint32_t n, uint32_t gt,
                                         uint32_t nth, uint32_t fresh, uint32_t stale, const NaList &O)
{
    for (uint32_t i = gt; i < n; i += nth) {
        const uint32_t y = __ldcg(from + i) >> 1;
        atomicAnd(asg + (y >> 3), ~(stale << ((y & 7u) * 4u)));
    }
    for (uint32_t L = 2; L <= (uint32_t)BUCKET_MAX; L++) {
        const uint32_t *base = D.lits + D.bk_base[L];
        const uint32_t m = D.bk_n[L];
        for (uint32_t k = gt; k < m; k += nth) {
            bool sat = false;
            uint32_t n_un = 0, ul = 0;
            for (uint32_t q0 = 0; q0 < L && !sat && n_un < 2u; q0 += 4u) {
                uint32_t l[4], v[4];
#pragma unroll
                for (uint32_t q = 0; q < 4u; q++) l[q] = q0 + q < L ? __ldg(base + (size_t)(q0 + q) * m + k) : PAD_LIT;
#pragma unroll
                for (uint32_t q = 0; q < 4u; q++) v[q] = l[q] != PAD_LIT ? na_val(asg, l[q] >> 1, fresh) : 3u;
#pragma unroll
                for (uint32_t q = 0; q < 4u; q++) {
                    if (v[q] == 0u) { n_un++; ul = l[q]; }
                    sat |= v[q] == ((l[q] & 1u) ? V_T : V_F);
                }
            }
            if (!sat && n_un == 0u) na_conflict(c, O);
            else if (!sat && n_un == 1u) na_claim(asg, c, ul, fresh, O);
        }
    }
}

// The unit nogoods.
__device__ __forceinline__ void na_units(const Dev &D, uint32_t *asg, NaCtl *c, uint32_t gt, uint32_t nth, uint32_t fresh,
                                         const NaList &O)
{
    for (uint32_t i = gt; i < D.n_units; i += nth) {
        const uint32_t l = __ldg(D.lits + D.units_base + i) & ~END_BIT;
        const uint32_t v = na_val(asg, l >> 1, fresh);
        if (v == 0u) na_claim(asg, c, l, fresh, O);
        else if (v == ((l & 1u) ? V_F : V_T)) na_conflict(c, O);
    }
}

// Long nogoods: one warp per nogood, lanes over literals.
__device__ __forceinline__ void na_long(const Dev &D, uint32_t *asg, NaCtl *c, uint32_t gw, uint32_t nw, uint32_t fresh, const NaList &O)
{
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t i = gw; i < D.n_long; i += nw) {
        __syncwarp();
        const uint32_t id = __ldg(D.long_ids + i);
        bool sat = false;
        uint32_t n_un = 0, ul = 0;
        for (uint32_t off = id;; off += 32u) {
            const uint32_t w = __ldg(D.lits + off + lane);
            const unsigned Bend = __ballot_sync(0xFFFFFFFFu, (w & END_BIT) != 0u);
            const unsigned valid = Bend ? ((2u << (__ffs(Bend) - 1)) - 1u) : 0xFFFFFFFFu;
            const uint32_t l = w & ~END_BIT;
            const bool mine = (valid >> lane) & 1u;
            const uint32_t v = mine ? na_val(asg, l >> 1, fresh) : 0u;
            const unsigned Bopp = __ballot_sync(0xFFFFFFFFu, mine && v == ((l & 1u) ? V_T : V_F));
            const unsigned Bun = __ballot_sync(0xFFFFFFFFu, mine && v == 0u);
            const uint32_t first = __shfl_sync(0xFFFFFFFFu, l, Bun ? __ffs(Bun) - 1 : 0);
            if (Bun && n_un == 0) ul = first;
            n_un += (uint32_t)__popc(Bun);
            if (Bopp) { sat = true; break; }
            if (Bend || n_un > 1u) break;
        }
        if (lane == 0 && !sat) {
            if (n_un == 0u) na_conflict(c, O);
            else if (n_un == 1u) na_claim(asg, c, ul, fresh, O);
        }
    }
}

// The fixpoint by following assignments: a round checks the nogoods of the
// literals listed by the round before (first the caller's assignment), found
// through the occurrence lists, instead of every nogood of the store; with at
// most NA_NARROW of them CTA 0 goes on alone, with CTA barriers.  Nogoods in
// no list (more than BUCKET_MAX literals) are checked in the grid's rounds,
// and the last round is one.  After lists too long for a warp the grid's next
// round is a sweep of the store.  A round is bound by its chain of dependent
// loads (list, list bounds, occurrence, codes, claim) and its barrier.
__global__ void __launch_bounds__(NA_THREADS, 1) noalloc_propagate_kernel(Dev D, const int8_t *partial, int8_t *closure,
                                                                          int32_t *conflict_out, uint32_t *scratch)
{
    __shared__ uint32_t s_lit[2][NA_LIST];
    __shared__ unsigned int s_n[3], s_stop;
    NaCtl *c = reinterpret_cast<NaCtl *>(scratch);
    uint32_t *asg = scratch + NOALLOC_CTL_WORDS, *list = asg + NOALLOC_CODES;
    const uint32_t nth = gridDim.x * blockDim.x, gt = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u, nw = nth >> 5;
    // consecutive warps of the grid sit on different CTAs, so short lists
    // spread over the SMs
    const uint32_t gw = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const uint32_t words = (D.nv + 7u) >> 3;
    if (threadIdx.x == 0) s_n[0] = s_n[1] = s_n[2] = s_stop = 0u;
    na_cta_sync();
    NaList O{list, 0u, &c->nclaim[2], s_lit[0], &s_n[0], &c->stop[2]};
    // the caller's partial assignment, committed (no fresh bits); round -1
    const bool aligned = ((reinterpret_cast<uintptr_t>(partial) | reinterpret_cast<uintptr_t>(closure)) & 7u) == 0u;
    for (uint32_t w = gt; w < words; w += nth) {
        unsigned long long x = 0;
        if (aligned && 8u * w + 8u <= D.nv) x = reinterpret_cast<const unsigned long long *>(partial)[w];
        else
            for (uint32_t q = 0; q < 8u && 8u * w + q < D.nv; q++) x |= (unsigned long long)(uint8_t)partial[8u * w + q] << (8u * q);
        uint32_t m = 0;
        for (uint32_t q = 0; x >> (8u * q); q++) {
            const int8_t p = (int8_t)(x >> (8u * q));
            if (p) {
                m |= (p > 0 ? V_T : V_F) << (4u * q);
                na_push(O, mk_lit(8u * w + q, p < 0));
            }
            if (q == 7u) break;
        }
        asg[w] = m;
    }
    na_flush(O);
    uint32_t gen = 0, from = 0, to = 0;       // literals [from, to) are to be followed
    bool ok = na_sync(c, gen++);
    if (ok) to = __ldcg(&c->nclaim[2]);
    // what a warp walks in the time of a sweep.  A call with one list of n
    // occurrences, walked and with a sweep instead: 335k literals, n = 100 74 and 66
    // us, 200 114 and 109, 400 136 and 86; 5.9M literals, 200 92 and 89, 400 118
    // and 84
    const uint32_t longest = 128u + (uint32_t)(D.static_checks / (16u * nw));
    // r: rounds so far (its parity names the fresh bit), k: the grid's rounds;
    // the first also applies the unit nogoods
    uint32_t r = 0, k = 0, stop = 0;
    if (D.narrow_max == 0u) {
        // no lists: every round reads the whole store
        for (; ok; k++, r++) {
            const uint32_t fresh = 4u << (r & 1u), slot = k % 3u;
            if (gt == 0) c->nclaim[(k + 1u) % 3u] = c->stop[(k + 1u) % 3u] = 0u;
            O = NaList{list, to, &c->nclaim[slot], s_lit[0], &s_n[0], &c->stop[slot]};
            if (k == 0) na_units(D, asg, c, gt, nth, fresh, O);
            na_sweep(D, asg, c, list + from, to - from, gt, nth, fresh, 4u << ((r + 1u) & 1u), O);
            na_long(D, asg, c, gw, nw, fresh, O);
            na_flush(O);
            if (!(ok = na_sync(c, gen++))) break;
            const uint32_t n = __ldcg(&c->nclaim[slot]);
            if (__ldcg(&c->stop[slot]) || n == 0u) break;
            from = to;
            to += n;
        }
        goto done;
    }
follow:
    for (; ok; k++) {
        const uint32_t fresh = 4u << (r & 1u), stale = 4u << ((r + 1u) & 1u), slot = k % 3u;
        if (gt == 0) c->nclaim[(k + 1u) % 3u] = c->stop[(k + 1u) % 3u] = 0u;
        O = NaList{list, to, &c->nclaim[slot], s_lit[0], &s_n[0], &c->stop[slot]};
        if (k == 0) na_units(D, asg, c, gt, nth, fresh, O);
        na_follow<false>(D, asg, c, list + from, to - from, gw, nw, fresh, stale, longest, O);
        na_long(D, asg, c, gw, nw, fresh, O);
        na_flush(O);
        if (!(ok = na_sync(c, gen++))) break;
        // every thread sees the same counters after the barrier
        const uint32_t n = __ldcg(&c->nclaim[slot]);
        stop = __ldcg(&c->stop[slot]);
        from = to;
        to += n;
        r++;
        if (stop || n == 0u) break;
        if (n > NA_NARROW) continue;
        if (blockIdx.x == 0) {
            // narrow rounds: a round's literals stay in shared memory, two
            // lists in turn; if the last one lists too many, or lists were
            // passed over, they go to the list after `to`, for the grid
            for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) s_lit[0][i] = __ldcg(list + from + i);
            if (threadIdx.x == 0) c->nover = 0u;
            uint32_t m = n, i = 0;
            O.base = to;
            O.n = &c->nover;
            O.stop = &s_stop;
            do {
                na_cta_sync();
                if (threadIdx.x == 0) s_n[(i + 2u) % 3u] = 0u;     // the next round's counter
                O.s_lit = s_lit[(i + 1u) & 1u];
                O.s_n = &s_n[(i + 1u) % 3u];
                na_follow<true>(D, asg, c, s_lit[i & 1u], m, threadIdx.x >> 5, blockDim.x >> 5, 4u << ((r + i) & 1u),
                                4u << ((r + i + 1u) & 1u), longest, O);
                na_cta_sync();
                m = *O.s_n;
                i++;
            } while (m != 0u && m <= NA_NARROW && !s_stop);
            const bool over = m > NA_NARROW || (m != 0u && s_stop);
            if (over) na_flush(O);
            na_cta_sync();
            if (threadIdx.x == 0) {
                c->next = r + i;
                c->left = over ? m : 0u;
                c->nstop = s_stop;
                s_n[0] = s_n[1] = s_n[2] = s_stop = 0u;
            }
        }
        if (!(ok = na_sync(c, gen++))) break;
        r = __ldcg(&c->next);
        from = to;
        to += __ldcg(&c->left);
        stop = __ldcg(&c->nstop);
        if (stop || (from == to && D.n_long == 0u)) break;
    }
    if (ok && stop == NA_LONG) {
        // a round of the whole store.  Apart from the others: as a case among
        // them, with a test in each, it took 6 % of an 80k-atom program's
        // propagation, which has no such list
        k++;
        const uint32_t slot = k % 3u;
        if (gt == 0) c->nclaim[(k + 1u) % 3u] = c->stop[(k + 1u) % 3u] = 0u;
        O = NaList{list, to, &c->nclaim[slot], s_lit[0], &s_n[0], &c->stop[slot]};
        na_sweep(D, asg, c, list + from, to - from, gt, nth, 4u << (r & 1u), 4u << ((r + 1u) & 1u), O);
        na_flush(O);
        if ((ok = na_sync(c, gen++))) {
            const uint32_t n = __ldcg(&c->nclaim[slot]);
            stop = __ldcg(&c->stop[slot]);
            from = to;
            to += n;
            r++;
            k++;
            if (!stop) goto follow;
        }
    }
done:
    if (!ok && !gt) *conflict_out = -1;
    if (!ok) return;
    for (uint32_t w = gt; w < words; w += nth) {
        const uint32_t m = __ldcg(asg + w);
        unsigned long long x = 0;
        for (uint32_t q = 0; q < 8u; q++) {
            const uint32_t code = (m >> (4u * q)) & 3u;
            x |= (unsigned long long)(uint8_t)(code == V_F ? -1 : code == 3u ? 2 : (int)code) << (8u * q);
        }
        if (aligned && 8u * w + 8u <= D.nv) reinterpret_cast<unsigned long long *>(closure)[w] = x;
        else
            for (uint32_t q = 0; q < 8u && 8u * w + q < D.nv; q++) closure[8u * w + q] = (int8_t)(x >> (8u * q));
    }
    if (gt == 0) *conflict_out = __ldcg(&c->conflict) ? 1 : 0;
}

std::mutex g_noalloc_mu;
void *g_noalloc_ptr[128];
int g_noalloc_grid[128];

}  // namespace

const Dev *internal_dev(const asp_prog *p);
cudaStream_t internal_stream(const asp_prog *p);
int internal_device(const asp_prog *p);
int internal_fail(int code, const char *msg);

}  // namespace aspgpu

extern "C" int asp_propagate_noalloc(const asp_prog *p, const int8_t *d_partial, int8_t *d_closure,
                                     int32_t *d_conflict)
{
    using namespace aspgpu;
    if (!p || !d_partial || !d_closure || !d_conflict) return internal_fail(ASP_E_ARG, "null argument");
    const Dev *D = internal_dev(p);
    if (D->nv > NOALLOC_MAX_VARS)
        return internal_fail(ASP_E_CAPACITY, "program has more than 2^20 variables, the static working array's limit");
    // the program's stream and store belong to the device it was loaded on;
    // the static array's address is looked up on the current device, so the
    // two must agree
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return internal_fail(ASP_E_CUDA, "no current device");
    if (dev != internal_device(p))
        return internal_fail(ASP_E_ARG, "the current device is not the device the program was loaded on");
    void *scratch = nullptr;
    int grid = 0;
    {
        // once per device, with that device current: the device address of
        // the static array (its host-side name is only a stand-in)
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr)
                return internal_fail(ASP_E_CUDA, "cudaGetSymbolAddress of the static working array failed");
            int sms = 0, per_sm = 0;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
                return internal_fail(ASP_E_CUDA, "reading the multiprocessor count failed");
            // The kernel is compiled for one 768-thread block per SM
            // (__launch_bounds__(768, 1)), so a grid of one CTA per SM always
            // fits a cooperative launch; the occupancy query confirms that
            // at least one block is resident per SM.
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, noalloc_propagate_kernel, NA_THREADS, 0) != cudaSuccess ||
                per_sm < 1)
                return internal_fail(ASP_E_CUDA, "the propagation kernel cannot be resident on an SM");
            g_noalloc_grid[dev] = sms;
            g_noalloc_ptr[dev] = ptr;
        }
        scratch = g_noalloc_ptr[dev];
        grid = g_noalloc_grid[dev];
    }
    // small programs take fewer CTAs: their barriers are shorter
    grid = std::min<int>(grid, 1 + (int)(D->nv / 4096u));
    cudaStream_t st = internal_stream(p);
    // the control words start at zero on every call
    if (cudaMemsetAsync(scratch, 0, NOALLOC_CTL_WORDS * sizeof(uint32_t), st) != cudaSuccess)
        return internal_fail(ASP_E_CUDA, "clearing the counters failed");
    Dev copy = *D;
    uint32_t *s = static_cast<uint32_t *>(scratch);
    void *args[] = {(void *)&copy, (void *)&d_partial, (void *)&d_closure, (void *)&d_conflict, (void *)&s};
    if (cudaLaunchCooperativeKernel((void *)noalloc_propagate_kernel, dim3(grid), dim3(NA_THREADS), args, 0, st) != cudaSuccess)
        return internal_fail(ASP_E_CUDA, "launch failed");
    return ASP_OK;
}
