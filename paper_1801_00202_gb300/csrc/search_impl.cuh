// Bit-parallel Bron-Kerbosch search (Alg. 4, BKPivotOrdered with
// ChoosePivotOrdered) as a persistent, work-stealing CUDA kernel for sm_103a.
//
// Two tiers (Section 4.1 describes the CPU bitset encoding this replaces):
//  * The top of the search tree: a warp owns one frame (P, X, pivot, end, |R|,
//    S(R)), which stands for "expand the children v in L = P & ~N(pivot) &
//    [0, end) in increasing position".  Lane l holds words [l*K, l*K + K) of
//    every set; the current frame lives in registers, its ancestors on an
//    explicit stack in local memory (no recursion).  A frame is pushed only
//    while it has children left, so single-child chains (e.g. a complete
//    graph) do not grow the stack.
//  * The warp tier, where nearly all nodes are: subtrees of at most 128
//    vertices, compressed to small sets and searched a child per lane (see
//    "The warp tier" below).
//  * The renumbered adjacency (Section 4.2) is read from L2 above the warp
//    tier, which leaves the shared memory to that tier (staging rows of up to
//    32 words there gained 5 % on G(700, 0.18) and nothing elsewhere).
//  * Work moves at two levels.  Idle warps take frames from their block's
//    ring in shared memory or from the device-wide ring (a bounded MPMC ring
//    in global memory whose tickets are taken by fetch-and-add at both ends);
//    busy warps refill the block's ring while it has more idle warps than
//    queued frames, and the device-wide ring while the GPU has.
//    Cutting a branching set L into a front part L1 (given) and the rest as
//    (P, X, end = first kept element) and (P \ L1, X u L1, end) reproduces
//    exactly the sequential P/X updates of Alg. 4, so node counts do not
//    depend on how the work was split.
//  * Leaves update per-lane register counters; sizes go to a shared-memory
//    histogram; everything is integer arithmetic modulo 2^64, so the
//    reduction order does not matter and results are bit-exact.
//
// Every spin (queue tickets, idle wait) is bounded and
// ends in an error status plus a global abort flag, never a hang or a trap.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "mce_internal.h"

namespace mce {

constexpr unsigned FULL = 0xffffffffu;
constexpr unsigned kCasTries = 1u << 14; // bound of one queue ticket loop

// Work-distribution thresholds by edge density p = i/40 (i = 1..39): the
// smallest candidate-set size k whose random subgraph G(k, p) has at least
// 256, 2048 or 16384 maximal cliques in expectation
// (sum_j C(k,j) p^C(j,2) (1-p^j)^(k-j)).  A frame is given to the block ring
// or the device-wide ring when its candidate set reaches the first: what moves
// must carry enough work to pay for the move.  The second and third bound the
// warp tier's subproblems, and a new subtree of the third (at most half of the
// vertices) is published breadth-first (see density_thresholds).
__constant__ unsigned short kShareLocalByDensity[39] = {147, 111, 96, 87, 80, 73, 68, 63, 58, 55, 52, 49, 47,
                                                        44,  42,  41, 39, 37, 36, 35, 33, 32, 31, 30, 29, 29,
                                                        28,  27,  26, 26, 25, 25, 25, 25, 25, 25, 26, 28, 34};
__constant__ unsigned short kShareGlobalByDensity[39] = {440, 343, 283, 234, 199, 174, 155, 141, 129, 119, 110,
                                                         102, 94,  88,  82,  77,  73,  69,  65,  62,  58,  55,
                                                         53,  50,  48,  46,  44,  42,  41,  39,  38,  37,  36,
                                                         35,  34,  34,  35,  36,  42};
__constant__ unsigned short kSplitByDensity[39] = {1363, 907, 651, 515, 433, 376, 329, 290, 257, 230, 208, 189, 173,
                                                   159,  146, 135, 125, 116, 108, 101, 94,  88,  83,  78,  73,  69,
                                                   65,   61,  58,  55,  52,  50,  48,  46,  45,  44,  43,  45,  51};

struct Thresholds {
    unsigned share;        // smallest |P| of a frame given to the block's idle warps
    unsigned share_far;    // smallest |P| of a frame given to the device-wide ring
    unsigned split;        // smallest |P| of a new subtree that is published breadth-first
    unsigned task;         // warp tier: largest |P| of a subproblem
    unsigned cls;          // warp tier: words per set (P u X of at most 32 cls vertices)
};

// Thresholds from the graph's edge density (deg_sum = twice the edges);
// non-zero caller values win.  batch_cls != 0: one of a batch's graphs, which
// share sets of that size.
__device__ __forceinline__ Thresholds density_thresholds(unsigned deg_sum, uint32_t n, const Tuning &tune,
                                                         unsigned fixed_split, bool scores, unsigned batch_cls = 0u)
{
    Thresholds t{0xffffffffu, 0xffffffffu, 0xffffffffu, 128u, max(batch_cls, 1u)};
    if (n >= 2u) {
        const float pd = (float)deg_sum / ((float)n * (float)(n - 1u));
        int i = (int)(pd * 40.0f + 0.5f);
        i = i < 1 ? 1 : (i > 39 ? 39 : i);
        t.share = kShareLocalByDensity[i - 1];
        t.share_far = t.share;
        // dense structured graphs (Moon-Moser: every child keeps all but three
        // vertices) would never reach the density's split size; cap it at
        // half of n
        t.split = min((unsigned)kSplitByDensity[i - 1], max(20u, n / 2u));
        // Largest subproblem of the warp tier: about a 4,096th of the whole
        // search (log2 of its expected maximal cliques continued from the
        // table on a log-log line), so that every warp gets some before
        // frames have to be given away; the whole graph when that is small
        // (fewer than 50,000: handing out the parts takes longer than it
        // saves).  In dense graphs, where a subtree can hold far more cliques
        // than a random graph's (Moon-Moser), a third of the vertices.
        // Measured with limits of 24 / 32 / 48 / 64 / 128 vertices, ms:
        // G(106, 0.71) 0.40 / 0.43 / 0.49 / - / 0.57, G(100, 0.8) 1.5 / 1.1 /
        // 1.5 / 1.8 / 1.4, G(300, 0.5) 3.7 / 2.5 / 1.5 / 1.3 / 1.4, G(100, 0.5)
        // 0.20 / 0.18 / 0.19 / 0.16 / 0.16; Moon-Moser 45 with 16 / 20 / 24 /
        // 32: 0.69 / 0.63 / 0.77 / 1.06.
        const float k2 = (float)kShareGlobalByDensity[i - 1], k3 = (float)kSplitByDensity[i - 1];
        const float size = 14.0f + 3.0f * __logf((float)n / k3) / __logf(k3 / k2);
        if (i >= 30) t.task = min((unsigned)kShareGlobalByDensity[i - 1], max(20u, n / 3u));
        else if (n > 128u) t.task = min((unsigned)kSplitByDensity[i - 1], max(48u, 3u * n / 10u));
        else if (size >= 15.6f || (size >= 12.5f && i >= 24))
            t.task = size < 21.5f ? kShareLocalByDensity[i - 1]
                                  : (size < 24.5f ? kShareGlobalByDensity[i - 1] : kSplitByDensity[i - 1]);
        // Set size of the warp tier: k levels below the root P u X has about
        // n p^k vertices.  The first level of at most 102 (128 in a long
        // search, which has frames enough beside the larger half) gets the tier, or
        // the one below where the children of the root would hold more than
        // about 256 cliques each (then they are too few and too uneven).  (At
        // n p = 97 / 99 / 101 the four words for all children beat the level
        // below, G(750, 0.13) 0.34 / 0.37, G(660, 0.15) 0.28 / 0.36, G(560, 0.18)
        // 0.25 / 0.33 ms; at 103 / 104 / 106 too many children do not fit them,
        // G(622, 0.165) 0.42 / 0.35, G(600, 0.174) 0.39 / 0.35, G(640, 0.165) 0.51 /
        // 0.36.  With 600 cliques in place of 256: G(260, 0.32) 0.27 / 0.21, G(190,
        // 0.44) 0.26 / 0.22, G(310, 0.32) under TomitaBB 0.34 / 0.28.)
        // Room for all of the level's frames: three standard deviations for
        // the children of the root, two below; none in dense graphs, where
        // one level further down still holds enough work per frame.  One
        // size for the whole search keeps one instance of the tier's code in
        // the instruction caches: with all four sizes in use the SM's
        // instruction fetches were what bounded the search.
        float sz = (float)n, pk = 1.0f;
        const float pf = pd < 0.95f ? pd : 0.95f;
        int level = 0;
        const float most = size < 22.5f ? 102.0f : 128.0f;
        while (sz > most || (level == 1 && size - __log2f((float)n) > 8.0f)) {
            sz *= pf;
            pk *= pf;
            ++level;
        }
        if (level <= 1) sz += 3.0f * sqrtf(sz * (1.0f - pk));
        else if (pf < 0.48f) sz += 2.0f * sqrtf(sz * (1.0f - pk));
        // Below the root's children two words at least, where rows are short
        // (one word builds eight subproblems side by side, but gives up a level
        // more often: G(640, 0.165) 0.39 / 0.36 ms, G(1000, 0.14) 0.58 / 0.55);
        // rows of more than 32 words cost the build a load per word (G(1600,
        // 0.1): one word 0.78, two 0.83).
        if (level > 1 && n <= 1024u) sz = fmaxf(sz, 32.0f);
        // Just above 128 vertices a search of up to 2^19 cliques has fewer
        // frames on that level than the GPU has warps; subproblems of at most
        // 32 vertices, one level further down, spread it.  Under rules that
        // score pivots a node takes longer, and it pays up to 2^21.  Two words /
        // one, ms: G(129, 0.56) 0.28 / 0.20, under TomitaBB 0.34 / 0.23, G(140,
        // 0.62) 0.44 / 0.45, under TomitaBB 0.65 / 0.47.
        if (level > 1 && n <= 160u && size < (scores ? 21.0f : 19.0f)) sz = 1.0f;
        t.cls = n <= 128u ? (n + 31u) / 32u : (unsigned)((sz + 32.0f) * (1.0f / 32.0f));
        t.cls = min(max(t.cls, 1u), 4u);
        // A batch has work for every warp without cutting subtrees small, and
        // one set size for all of its graphs keeps to one instance of the
        // code: 512 graphs of 32 to 512 vertices took 17.7 ms with the limits
        // of a graph searched alone, 13.0 with 128 vertices as the limit and
        // four words above 128 vertices, 12.5 with four words throughout.
        // Dense graphs, two thirds of the vertices (a third, as alone / a half /
        // two thirds / all, ms, 700 graphs: G(64, 0.8) 18.3 / 7.2 / 7.2 / 6.6,
        // G(50, 0.9) 10.5 / 6.5 / 4.2 / 4.8, Moon-Moser 36 10.2 / 10.2 / 9.2 /
        // 9.2, 160 G(130, 0.75) 178 / 145 / 145 / 146).
        if (batch_cls) {
            t.cls = batch_cls;
            t.task = i < 30 ? 128u : max(20u, 2u * n / 3u);
        }
    }
    if (tune.share_local) t.share = tune.share_local;
    if (tune.share_global) t.share_far = tune.share_global;
    if (fixed_split) {
        // (a caller's split size is honoured: larger subtrees are published,
        // not searched by the warp tier)
        t.split = fixed_split;
        t.task = min(t.task, fixed_split - 1u);
    }
    if (tune.t2_task) t.task = min(t.task, tune.t2_task);
    if (tune.t2_cls && n > 128u) t.cls = min(tune.t2_cls, 4u);
    return t;
}

// SplitMix64 finaliser (Steele, Lea and Flood, OOPSLA 2014), the mixing step
// of the clique hash h(K) = mix64(S(K) ^ mix64(|K|)).
__device__ __forceinline__ uint64_t mix64(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void set_status(uint64_t *out, Ctl *ctl, int code)
{
    atomicCAS(reinterpret_cast<unsigned long long *>(out + MCE_OUT_STATUS), 0ull,
              static_cast<unsigned long long>(static_cast<long long>(code)));
    atomicExch(&ctl->abort, 1u);
}

// ---------------------------------------------------------------------------
// Bounded MPMC ring of frames (per-slot sequence numbers: a slot with
// seq == ticket is free for producer `ticket`, seq == ticket + 1 holds the
// frame for consumer `ticket`).

// Reserve a producer ticket: check the room left -- producer tickets at
// most qcap - margin ahead of the consumers', margin = the warps that can
// reserve at once (one ticket each) -- and take the ticket with one
// fetch-and-add, so producers race no compare-and-swap either.  The room
// check puts the ticket's slot behind a consumer ticket already claimed, so
// the slot is free as soon as that frame has been taken (microseconds;
// waited for, with a bound).  On false the caller keeps its frame; a ticket
// taken but never filled (the bounded wait ran out, or the search aborted)
// only leaves its consumer idle.
__device__ __forceinline__ bool q_reserve_push(Ctl *ctl, unsigned *seq, unsigned mask, unsigned &ticket,
                                               unsigned margin)
{
    const unsigned hd = ld_relaxed(&ctl->head), tl = ld_relaxed(&ctl->tail);
    if ((int)(tl - hd) >= (int)(mask + 1u) - (int)margin) return false;
    const unsigned tk = atomicAdd(&ctl->tail, 1u);
#pragma unroll 1
    for (unsigned t = 0; ld_acquire(&seq[tk & mask]) != tk; ++t) {
        if (t >= (kCasTries << 8) || ld_relaxed(&ctl->abort)) return false;
        __nanosleep(32);
    }
    ticket = tk;
    return true;
}

// Take the oldest published frame of a block-private ring (batched form:
// the only contenders are the block's own warps, so a compare-and-swap on
// the head is cheap there).
__device__ __forceinline__ bool q_reserve_pop(Ctl *ctl, unsigned *seq, unsigned mask, unsigned &ticket,
                                              unsigned long long *fails, unsigned tries = kCasTries)
{
    unsigned pos = ld_relaxed(&ctl->head);
#pragma unroll 1
    for (unsigned t = 0; t < tries; ++t) {
        unsigned s = ld_acquire(&seq[pos & mask]);
        int dif = (int)(s - (pos + 1));
        if (dif == 0) {
            unsigned prev = atomicCAS(&ctl->head, pos, pos + 1);
            if (prev == pos) { ticket = pos; return true; }
            atomicAdd(fails, 1ull);
            pos = prev;
        } else if (dif < 0) {
            return false;  // empty
        } else {
            pos = ld_relaxed(&ctl->head);
        }
    }
    return false;
}

// Room kept free in a frame ring for producers that reserve at once: every
// warp of the launch on the device-wide ring (the plain form sizes the ring
// at four frames per warp and more), the block's warps on a block-private
// ring (batched form).
__device__ __forceinline__ unsigned push_margin(const SearchParams &prm)
{
    const unsigned block_warps = blockDim.x >> 5;
    return (prm.total_groups > block_warps ? prm.total_groups : block_warps) + 32u;
}

// Claim up to `want` consecutive consumer tickets of the device-wide ring
// with one fetch-and-add: first .. first + k - 1.  Only frames seen in the
// ring are claimed, so claimers never race a compare-and-swap on the head
// (under a compare-and-swap, most of the idle blocks' attempts failed and
// were retried, and the ring's head was the search's bottleneck); two
// claimers that saw the same frames can take tickets past the producers'.
// A claimed ticket is the claimer's alone: its frame is taken once the
// producer has published it (seq == ticket + 1), or never if the search ends
// first -- the search ends only when no frame is queued or held anywhere
// (pending == 0), so no published frame is ever left behind.  Returns k.
__device__ __forceinline__ unsigned q_claim(Ctl *ctl, unsigned want, unsigned &first)
{
    const unsigned h = ld_relaxed(&ctl->head), t = ld_relaxed(&ctl->tail);
    const int avail = (int)(t - h);
    if (avail <= 0) return 0u;
    const unsigned k = min(want, (unsigned)avail);
    first = atomicAdd(&ctl->head, k);
    return k;
}

// ---------------------------------------------------------------------------
// Warp-wide set primitives: lane l holds words [l*K, l*K + K) of a set.  All
// are reached by all 32 lanes in warp-uniform control flow.

// Position of the lowest set bit (= the vertex first in the order), or -1.
template <int K>
__device__ __forceinline__ int set_first(const uint32_t (&s)[K], unsigned lane)
{
    int loc = -1;
#pragma unroll
    for (int k = K - 1; k >= 0; --k)
        if (s[k]) loc = (int)((lane * K + k) * 32u) + __ffs(s[k]) - 1;
    return (int)__reduce_min_sync(FULL, (unsigned)loc);
}
template <int K>
__device__ __forceinline__ uint32_t set_or(const uint32_t (&s)[K])
{
    uint32_t o = s[0];
#pragma unroll
    for (int k = 1; k < K; ++k) o |= s[k];
    return o;
}
template <int K>
__device__ __forceinline__ unsigned set_count(const uint32_t (&s)[K])
{
    unsigned c = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) c += (unsigned)__popc(s[k]);
    return c;
}
// Bits [0, end) of this lane's k-th word.
template <int K>
__device__ __forceinline__ uint32_t set_below(int k, unsigned end, unsigned lane)
{
    const unsigned base = (lane * K + k) * 32u;
    if (end >= base + 32u) return FULL;
    if (end <= base) return 0u;
    return (1u << (end - base)) - 1u;
}
// The bit of vertex v in this lane's k-th word.
template <int K>
__device__ __forceinline__ uint32_t set_bit(int k, unsigned v, unsigned lane)
{
    return (v >> 5) == lane * K + k ? 1u << (v & 31u) : 0u;
}
// Elements in lower lanes.
__device__ __forceinline__ unsigned lanes_below_sum(unsigned x, unsigned lane)
{
    unsigned incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(FULL, incl, o);
        incl += (int)lane >= o ? y : 0u;
    }
    return incl - x;
}

template <int K>
__device__ __forceinline__ void load_row(uint32_t (&r)[K], const uint32_t *p)
{
    if (K == 1) {
        r[0] = __ldg(p);
    } else if (K == 2) {
        uint2 t = __ldg(reinterpret_cast<const uint2 *>(p));
        r[0] = t.x;
        r[1] = t.y;
    } else {
        uint4 t = __ldg(reinterpret_cast<const uint4 *>(p));
        r[0] = t.x;
        r[1] = t.y;
        r[2] = t.z;
        r[3] = t.w;
    }
}

// ---------------------------------------------------------------------------
// Block-local frame ring (shared memory): the same per-slot sequence-number
// protocol as the global ring, with block-scope atomics.

__device__ __forceinline__ unsigned vld(const unsigned *p) { return *reinterpret_cast<const volatile unsigned *>(p); }
__device__ __forceinline__ void vst(unsigned *p, unsigned v) { *reinterpret_cast<volatile unsigned *>(p) = v; }

__device__ __forceinline__ bool lq_reserve_push(LocalHdr *h, unsigned *seq, unsigned mask, unsigned &ticket)
{
    unsigned pos = vld(&h->tail);
#pragma unroll 1
    for (unsigned t = 0; t < 256; ++t) {
        const unsigned s = vld(&seq[pos & mask]);
        const int dif = (int)(s - pos);
        if (dif == 0) {
            const unsigned prev = atomicCAS(&h->tail, pos, pos + 1);
            if (prev == pos) { ticket = pos; return true; }
            pos = prev;
        } else if (dif < 0) {
            return false;
        } else {
            pos = vld(&h->tail);
        }
    }
    return false;
}

__device__ __forceinline__ bool lq_reserve_pop(LocalHdr *h, unsigned *seq, unsigned mask, unsigned &ticket)
{
    unsigned pos = vld(&h->head);
#pragma unroll 1
    for (unsigned t = 0; t < 256; ++t) {
        const unsigned s = vld(&seq[pos & mask]);
        const int dif = (int)(s - (pos + 1));
        if (dif == 0) {
            const unsigned prev = atomicCAS(&h->head, pos, pos + 1);
            if (prev == pos) { ticket = pos; return true; }
            pos = prev;
        } else if (dif < 0) {
            return false;
        } else {
            pos = vld(&h->head);
        }
    }
    return false;
}

struct LocalQ {
    LocalHdr *h;
    unsigned *seq;
    uint32_t *frames;
    unsigned mask;  // slots - 1
};

__device__ __forceinline__ LocalQ local_queue_at(unsigned char *base)
{
    LocalQ q;
    q.h = reinterpret_cast<LocalHdr *>(base);
    q.seq = reinterpret_cast<unsigned *>(base + sizeof(LocalHdr));
    q.frames = reinterpret_cast<uint32_t *>(base + sizeof(LocalHdr) + kLocalSlots * 4u);
    q.mask = kLocalSlots - 1u;
    return q;
}

// Reset the block's ring (whole block; a barrier must follow).
__device__ __forceinline__ void local_queue_reset(const LocalQ &q, unsigned warps)
{
#pragma unroll 1
    for (unsigned i = threadIdx.x; i <= q.mask; i += blockDim.x) q.seq[i] = i;
    if (threadIdx.x == 0) {
        q.h->head = 0u;
        q.h->tail = 0u;
        q.h->idle = warps;
        q.h->bwork = 0u;
        q.h->poller = 0u;
        q.h->done = 0u;
        q.h->refreshing = 0u;
        q.h->g_head = 0u;
        q.h->g_tail = 0u;
        q.h->g_starving = 0u;
        q.h->stamp = 0ull;
        q.h->trace_n = 0u;
        for (int i = 0; i < kDiagCount; ++i) q.h->diag[i] = 0ull;
    }
}

// Per-lane result counters (summed over the warp at the end; nodes is formed
// at the flush as leaves + dead ends + internal nodes).  The block's
// work-distribution diagnostics live in shared memory (diag).
struct Counters {
    uint64_t cnt = 0, nodes = 0, intl = 0, dead = 0, hash = 0;
    unsigned max = 0;
    unsigned long long *diag = nullptr;
    __device__ __forceinline__ void note(int i, unsigned long long v = 1ull) const { atomicAdd(diag + i, v); }
};

// Warp-reduce the counters and add them to out[] (one atomic per counter per
// warp).  Called by all 32 lanes.
__device__ __forceinline__ void flush_counters(Counters &c, uint64_t *out)
{
    c.nodes = c.cnt + c.dead + c.intl;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        c.cnt += __shfl_xor_sync(FULL, c.cnt, o);
        c.nodes += __shfl_xor_sync(FULL, c.nodes, o);
        c.intl += __shfl_xor_sync(FULL, c.intl, o);
        c.dead += __shfl_xor_sync(FULL, c.dead, o);
        c.hash += __shfl_xor_sync(FULL, c.hash, o);
        c.max = max(c.max, __shfl_xor_sync(FULL, c.max, o));
    }
    if ((threadIdx.x & 31u) == 0) {
        unsigned long long *o = reinterpret_cast<unsigned long long *>(out);
        if (c.cnt) atomicAdd(o + MCE_OUT_COUNT, c.cnt);
        if (c.nodes) atomicAdd(o + MCE_OUT_NODES, c.nodes);
        if (c.intl) atomicAdd(o + MCE_OUT_INTERNAL, c.intl);
        if (c.dead) atomicAdd(o + MCE_OUT_DEAD_ENDS, c.dead);
        if (c.hash) atomicAdd(o + MCE_OUT_HASH, c.hash);
        if (c.max) atomicMax(o + MCE_OUT_MAX_SIZE, (unsigned long long)c.max);
    }
}

// The block's diagnostics to out[] (one thread, after the block's warps are
// done).
__device__ __forceinline__ void flush_diag(const unsigned long long *diag, uint64_t *out)
{
    unsigned long long *o = reinterpret_cast<unsigned long long *>(out);
    const int word[kDiagCount] = {MCE_OUT_DONATIONS, MCE_OUT_STEALS,   MCE_OUT_GLOBAL,    MCE_OUT_BUSY_NS,
                                  MCE_OUT_GPUSH,     MCE_OUT_GTRY,     MCE_OUT_CAS_FAIL,  MCE_OUT_LANE_TASKS};
#pragma unroll
    for (int i = 0; i < kDiagCount; ++i)
        if (diag[i]) atomicAdd(o + word[i], diag[i]);
}

// ---------------------------------------------------------------------------
// The warp tier.  Most nodes of the search tree lie where few vertices are
// left: once a frame's P u X has at most 128 vertices, nothing outside that
// set can ever enter a descendant's P or X (Alg. 4 only intersects them with
// rows of vertices of P).  Such a frame is compressed: U = P u X in
// increasing position is relabelled 0..u-1 -- order-preserving, so "first in
// the order" is still the lowest set bit and every pivot rule (first of X or
// P; the TX / TomitaBB argmax with ties to the earliest) picks the same
// vertex -- and its induced adjacency becomes u rows of W = ceil(u/32) words
// in the warp's shared memory.  The whole warp then searches the subtree from
// a stack of frames: a step hands the next 32 unexpanded children, counted
// from the top of the stack down, to the 32 lanes, whatever frames they
// belong to, and every lane computes its child from the frame's sets and
// pushes it if it has children itself.  No lane keeps a frame between steps,
// so a frame with many children that are leaves (most frames near the bottom)
// takes as few steps as its children fill.  The tree, the leaves and the hash
// terms are exactly those of the search by frames; only who expands which
// node differs.
//
// What bounds it: a step of 29 nodes takes about 340 instructions with
// four-word sets, most of them in one chain (scan of the children counts,
// frame -> pivot row -> child row -> pivot row from shared memory); the SM
// issues on a third of its cycles, and the rest are that chain's latencies and
// fetches of instructions.  Building a subproblem costs about as much as 300
// nodes.  Before, a warp searched 32 subproblems of at most 32 vertices, each
// by one lane with a stack of its own, and everything above 32 vertices a node
// per warp; now against then, ms: G(1000, 0.3) 2.9 / 5.8, G(500, 0.5) 9.6 /
// 21.4, G(300, 0.5) 1.2 / 2.0, Moon-Moser 45 0.63 / 0.85, G(45, 0.5) 0.045 /
// 0.125, G(100, 0.8) 1.0 / 1.5.  It gains least where a search is nothing but
// subproblems of ten nodes or so (G(700, 0.18) 0.46 / 0.45).
//
// Graphs of at most 128 vertices need no compression: their rows (and hash
// terms) are laid out once per block and every frame goes to the warp tier as
// it is.
//
// The warp's region of shared memory: local rows | hash terms of the local
// vertices | their positions | leaf buffer | stack of frames.
// A frame on the stack: P and X as they were when it was pushed (W words each),
// then meta = pivot (7 bits) | subproblem slot (3) | |R| less the start
// frame's (7) | children |L| (7) | children already taken (7), then S(R) in two
// words.  L = P \ N(pivot) is recomputed; child i is its i-th element v, with
// the earlier ones moved from P to X (Alg. 4's loop).  Frames are an odd
// number of words, so lanes on consecutive frames touch different banks.
template <int W>
struct PoolShape {
    static constexpr unsigned kFields = 2 * W + 3;
    static constexpr unsigned kStride = W == 3 ? 4u : (unsigned)W;         // words of a local row
    static constexpr unsigned kSlots = W == 1 ? 8u : (W == 2 ? 4u : 1u);   // subproblems searched together
    static constexpr unsigned kSlotRows = 32u * W * kStride;               // row words of one subproblem
    static constexpr unsigned kSlotVerts = 32u * W;
    // byte offsets in the warp's region
    static constexpr unsigned kHashOff = kSlots * kSlotRows * 4u;
    static constexpr unsigned kPosOff = kHashOff + kSlots * kSlotVerts * 8u;
    static constexpr unsigned kLeafOff = kPosOff + kSlots * kSlotVerts * 2u;
    static constexpr unsigned kRs0Off = kLeafOff + kPoolLeafBytes;   // |R| of every slot's start frame
    static constexpr unsigned kScratchOff = kRs0Off + 32u;           // one frame
    static constexpr unsigned kStackOff = kScratchOff + 48u;
    static_assert(kStackOff <= (unsigned)kPoolFixedBytes && kStackOff % 16u == 0u && kFields * 4u <= 48u,
                  "the region's fixed part");
    static_assert(kStackOff + 64u * kFields * 4u <= kPoolBytesMin, "a stack of at least 64 frames");
};
// The same for a size known at run time.
struct PoolOffsets {
    uint32_t hash, pos, leaf, rs0, stack;
};
template <int W>
__device__ __forceinline__ PoolOffsets pool_offsets_of()
{
    using Sh = PoolShape<W>;
    return {Sh::kHashOff, Sh::kPosOff, Sh::kLeafOff, Sh::kRs0Off, Sh::kStackOff};
}
__device__ __forceinline__ PoolOffsets pool_offsets(unsigned cls)
{
    return cls == 1u ? pool_offsets_of<1>()
                     : (cls == 2u ? pool_offsets_of<2>() : (cls == 3u ? pool_offsets_of<3>() : pool_offsets_of<4>()));
}

// Flags beside the position (12 bits) of a vertex that is handed over.
constexpr unsigned kPosInP = 0x8000u, kPosPivot = 0x4000u, kPosMask = 0x0fffu;

// Where a warp's tier finds things (byte offsets in shared memory): the local
// rows, hash terms and positions (the warp's own, or the block's when the
// whole graph is small), the warp's region and the block ring.
struct PoolAt {
    uint32_t rows, hash, pos, region, lq, hist;
};

// Result counters of one warp-tier run (per lane; at most one of each a step).
// A run may take any number of steps: every kFoldSteps of them the counters go
// to the result array (pool_fold) and start anew.  64-bit counters, or a fold
// into the caller's, cost every search 1 to 5 %, a fold by pool_watch 2.6 % of
// G(1000, 0.3), this call 1 %.
constexpr unsigned kFoldSteps = 1u << 14;
struct PoolCounters {
    uint64_t hash = 0;
    unsigned cnt = 0, intl = 0, dead = 0, max = 0;
};

template <int W>
__device__ __forceinline__ void pool_row(uint32_t (&r)[W], const uint32_t *a)
{
    if constexpr (W == 1) {
        r[0] = a[0];
    } else if constexpr (W == 2) {
        const uint2 t = *reinterpret_cast<const uint2 *>(a);
        r[0] = t.x;
        r[1] = t.y;
    } else {
        const uint4 t = *reinterpret_cast<const uint4 *>(a);
        r[0] = t.x;
        r[1] = t.y;
        r[2] = t.z;
        if constexpr (W == 4) r[3] = t.w;
    }
}

template <int W>
__device__ __forceinline__ bool pool_any(const uint32_t (&s)[W])
{
    uint32_t o = s[0];
#pragma unroll
    for (int k = 1; k < W; ++k) o |= s[k];
    return o != 0u;
}

// Lowest element of a set (of an empty one: some value below 32 W after the
// caller's mask).
template <int W>
__device__ __forceinline__ unsigned pool_first(const uint32_t (&s)[W])
{
    uint32_t w = s[W - 1];
    unsigned base = 32u * (W - 1);
#pragma unroll
    for (int k = W - 2; k >= 0; --k)
        if (s[k]) {
            w = s[k];
            base = 32u * (unsigned)k;
        }
    return base + (unsigned)__ffs(w) - 1u;
}

// Hand one subproblem to the warp's tier (all 32 lanes): `mine` is this
// lane's (first) word of U = P u X; the caller has written the positions of U with
// their flags to the slot.  Lane i builds the local rows of U[i], U[i + 32],
// ...: it walks its rows in word order, four words a load, and for every
// vertex U[j] of a word (the same word and bit in every lane) rotates that
// bit to place j of the row being assembled -- two instructions a column for
// 32 rows, against a shuffle, a test and a ballot a row and 32 columns.  Rows
// of more than 32 words (K > 1) would cost a sector of every lane's row for a
// few bits (G(3000, 0.1): some 40 KB from L2 for 30 vertices); there the warp
// reads one row at a time, lane i the word that holds U[i + 32 k], and a ballot
// makes the local row.  The start frame goes on the stack as frame `slot`.
template <int W, int K>
__device__ __noinline__ void pool_build(const uint32_t *rows, uint32_t rw, const uint32_t *order, uint32_t region,
                                        unsigned slot, uint32_t mine, unsigned u, unsigned children, unsigned rs,
                                        uint64_t S)
{
    using Sh = PoolShape<W>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const unsigned lane = threadIdx.x & 31u;
    uint32_t *A = reinterpret_cast<uint32_t *>(smem_raw + region) + slot * Sh::kSlotRows;
    uint64_t *lhv = reinterpret_cast<uint64_t *>(smem_raw + region + Sh::kHashOff) + slot * Sh::kSlotVerts;
    const uint16_t *pos = reinterpret_cast<const uint16_t *>(smem_raw + region + Sh::kPosOff) + slot * Sh::kSlotVerts;
    uint32_t *f = reinterpret_cast<uint32_t *>(smem_raw + region + Sh::kStackOff) + slot * Sh::kFields;
    const uint32_t *row[W];
    uint32_t qw[W], qm[W];  // word and bit of this lane's columns
    unsigned pl = 0;
#pragma unroll
    for (int g = 0; g < W; ++g) {
        const bool in = lane + 32u * g < u;
        const unsigned e = in ? (unsigned)pos[lane + 32u * g] : 0u;
        const unsigned q = e & kPosMask;
        row[g] = rows + (size_t)q * rw;
        qw[g] = q >> 5;
        qm[g] = in ? 1u << (q & 31u) : 0u;
        if (in) lhv[lane + 32u * g] = mix64((uint64_t)order[q] + 1u);
        const unsigned valid = __ballot_sync(FULL, in), p = __ballot_sync(FULL, (e & kPosInP) != 0u);
        const unsigned pb = __ballot_sync(FULL, (e & kPosPivot) != 0u);
        if (pb) pl = 32u * g + (unsigned)__ffs(pb) - 1u;
        if (lane == 0) {
            f[g] = p;
            f[W + g] = valid & ~p;
        }
    }
    if constexpr (K == 1) {
        uint32_t acc[W];
#pragma unroll
        for (int g = 0; g < W; ++g) acc[g] = 0u;
        unsigned j = 0;  // columns done
        auto store = [&](unsigned kw) {
#pragma unroll
            for (int g = 0; g < W; ++g) {
                A[(lane + 32u * g) * Sh::kStride + kw] = acc[g];
                acc[g] = 0u;
            }
        };
        const unsigned V = rw >= 4u ? 4u : rw;  // words of a load (rows are 1, 2 or a multiple of 4 words)
        const unsigned sw = min(rw, 32u);
#pragma unroll 1
        for (unsigned w0 = 0; w0 < sw && j < u; w0 += 4u) {
            // U's next four words (uniform), and the rows' (skipped where U has none)
            uint32_t m[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const unsigned wi = w0 + t;
                m[t] = __shfl_sync(FULL, mine, (int)(wi & 31u));
                if (wi >= sw) m[t] = 0u;
            }
            if ((m[0] | m[1] | m[2] | m[3]) == 0u) continue;
            uint32_t x[W][4];
#pragma unroll
            for (int g = 0; g < W; ++g) {
                if (V == 4u) {
                    const uint4 t = __ldg(reinterpret_cast<const uint4 *>(row[g] + w0));
                    x[g][0] = t.x;
                    x[g][1] = t.y;
                    x[g][2] = t.z;
                    x[g][3] = t.w;
                } else {
                    x[g][0] = __ldg(row[g]);
                    x[g][1] = V > 1u ? __ldg(row[g] + 1) : 0u;
                    x[g][2] = x[g][3] = 0u;
                }
            }
#pragma unroll 1
            for (int t = 0; t < 4; ++t) {
                uint32_t mt = m[0];
#pragma unroll 1
                while (mt) {
                    const unsigned rot = (j - (unsigned)__ffs(mt) + 1u) & 31u, bit = 1u << (j & 31u);
                    mt &= mt - 1u;
#pragma unroll
                    for (int g = 0; g < W; ++g) acc[g] |= __funnelshift_l(x[g][0], x[g][0], rot) & bit;
                    ++j;
                    if ((j & 31u) == 0u) store(j / 32u - 1u);
                }
                m[0] = m[1];
                m[1] = m[2];
                m[2] = m[3];
#pragma unroll
                for (int g = 0; g < W; ++g) {
                    x[g][0] = x[g][1];
                    x[g][1] = x[g][2];
                    x[g][2] = x[g][3];
                }
            }
        }
        if ((j & 31u) != 0u) store(j / 32u);
        // words past the last column
#pragma unroll 1
        for (unsigned kw = (u + 31u) / 32u; kw < (unsigned)W; ++kw) store(kw);
    } else {
        constexpr int B = 4;  // rows at a time
#pragma unroll 1
        for (unsigned j0 = 0; j0 < u; j0 += B) {
            uint32_t w[B][W];
#pragma unroll
            for (int t = 0; t < B; ++t) {
                const unsigned qj = j0 + t < u ? pos[j0 + t] & kPosMask : 0u;
#pragma unroll
                for (int g = 0; g < W; ++g) w[t][g] = __ldg(rows + (size_t)qj * rw + qw[g]);
            }
#pragma unroll
            for (int t = 0; t < B; ++t) {
                uint32_t b[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int g = 0; g < W; ++g) b[g] = __ballot_sync(FULL, (w[t][g] & qm[g]) != 0u);
                if (lane == 0 && j0 + t < u) {
                    uint32_t *a = A + (j0 + t) * Sh::kStride;
                    if (W == 1) a[0] = b[0];
                    else if (W == 2) *reinterpret_cast<uint2 *>(a) = make_uint2(b[0], b[1]);
                    else *reinterpret_cast<uint4 *>(a) = make_uint4(b[0], b[1], b[2], b[3]);
                }
            }
        }
    }
    if (lane == 0) {
        f[2 * W] = pl | (slot << 7) | (children << 17);
        f[2 * W + 1] = (uint32_t)S;
        f[2 * W + 2] = (uint32_t)(S >> 32);
        reinterpret_cast<uint32_t *>(smem_raw + region + Sh::kRs0Off)[slot] = rs;
    }
    __syncwarp();
}

// Position of the r-th (0-based) set bit of w, r < popc(w).
__device__ __forceinline__ unsigned select_bit(uint32_t w, unsigned r)
{
    unsigned at = 0u;
#pragma unroll
    for (unsigned h = 16u; h != 0u; h >>= 1) {
        const unsigned c = (unsigned)__popc((w >> at) & ((1u << h) - 1u));
        const bool up = r >= c;
        r -= up ? c : 0u;
        at += up ? h : 0u;
    }
    return at;
}

// Give the frame at byte offset `frame`, as it stands, to the block ring
// (`local`) or the device-wide ring as an ordinary frame over positions; the
// copy there is left without children.  False when the ring is full.
// Called by all 32 lanes; the warp holds a unit of block work.
template <int W>
__device__ __noinline__ bool pool_give(const PoolAt at, uint32_t frame, bool local)
{
    using Sh = PoolShape<W>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const unsigned lane = threadIdx.x & 31u;
    LocalHdr *h = reinterpret_cast<LocalHdr *>(smem_raw + at.lq);
    const LocalQ lq = local_queue_at(smem_raw + at.lq);
    uint32_t *f = reinterpret_cast<uint32_t *>(smem_raw + frame);
    const uint32_t meta = f[2 * W];
    const unsigned slot = (meta >> 7) & 7u, left = ((meta >> 17) & 127u) - (meta >> 24);
    if (left == 0u) return true;  // nothing there
    unsigned got = 0u, ticket = 0u;
    if (lane == 0) {
        if (local) {
            atomicAdd(&h->bwork, 1u);
            got = lq_reserve_push(h, lq.seq, lq.mask, ticket) ? 1u : 0u;
            if (!got) atomicSub(&h->bwork, 1u);
        } else {
            atomicAdd(&h->ctl->pending, 1u);
            got = q_reserve_push(h->ctl, h->gseq, h->qcap - 1u, ticket, h->margin) ? 1u : 0u;
            if (!got) atomicSub(&h->ctl->pending, 1u);
        }
    }
    got = __shfl_sync(FULL, got, 0);
    ticket = __shfl_sync(FULL, ticket, 0);
    if (!got) return false;
    uint32_t *fr = local ? lq.frames + (size_t)(ticket & lq.mask) * frame_words(h->wp)
                         : h->gframes + (size_t)(ticket & (h->qcap - 1u)) * h->fs;
#pragma unroll 1
    for (unsigned w = lane; w < 2u * h->wp; w += 32u) fr[kFrameHdr + w] = 0u;
    __threadfence();
    __syncwarp();
    const uint16_t *pos = reinterpret_cast<const uint16_t *>(smem_raw + at.pos) + slot * Sh::kSlotVerts;
    const uint32_t *a = reinterpret_cast<const uint32_t *>(smem_raw + at.rows) + slot * Sh::kSlotRows +
                        (meta & 127u) * Sh::kStride;
    unsigned taken = meta >> 24;  // the children already taken: from P to X
    // The frame's own children end before its branching set does when it is
    // the front of a set that was cut: `end` is the first position not its own.
    unsigned ahead = left, end = h->n;
#pragma unroll 1
    for (int k = 0; k < W; ++k) {
        uint32_t P = f[k], X = f[W + k];
        uint32_t L = P & ~a[k], gone = 0u;
        for (; taken != 0u && L != 0u; --taken) {
            gone |= L & (0u - L);
            L &= L - 1u;
        }
        P &= ~gone;
        X |= gone;
        const unsigned c = (unsigned)__popc(L);
        if (ahead < c) {
            end = pos[32 * k + select_bit(L, ahead)] & kPosMask;
            ahead = 0xffffffffu;
        } else if (ahead != 0xffffffffu) {
            ahead -= c;
        }
        if (((P | X) >> lane) & 1u) {
            const unsigned q = pos[32 * k + lane] & kPosMask;
            atomicOr(fr + kFrameHdr + (((P >> lane) & 1u) ? 0u : h->wp) + (q >> 5), 1u << (q & 31u));
        }
    }
    if (lane == 0) {
        const uint32_t *rs0 = reinterpret_cast<const uint32_t *>(smem_raw + at.region + Sh::kRs0Off);
        fr[0] = (uint32_t)(pos[meta & 127u] & kPosMask) | (end << 16);
        fr[1] = rs0[slot] + ((meta >> 10) & 127u);
        fr[2] = f[2 * W + 1];
        fr[3] = f[2 * W + 2];
        f[2 * W] = meta + (left << 24);
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) {
        if (local) {
            vst(&lq.seq[ticket & lq.mask], ticket + 1u);
        } else {
            st_release(&h->gseq[ticket & (h->qcap - 1u)], ticket + 1u);
            atomicAdd(&h->diag[kDiagGpush], 1ull);
        }
        atomicAdd(&h->diag[kDiagDonations], 1ull);
    }
    __syncwarp();
    return true;
}

// Hash terms and sizes of up to 32 buffered leaves: lane i takes the entry at
// e + 3 i; rs0 holds |R| of every slot's start frame.
__device__ __forceinline__ void pool_leaves(const uint32_t *e, unsigned n, unsigned lane, const uint32_t *rs0,
                                            uint32_t *hist, uint64_t *out, PoolCounters &c)
{
    const bool on = lane < n;
    unsigned k = 0u;
    if (on) {
        const uint64_t S = (uint64_t)e[3 * lane] | ((uint64_t)e[3 * lane + 1] << 32);
        const unsigned z = e[3 * lane + 2];
        k = rs0[z >> 8] + (z & 255u);
        ++c.cnt;
        c.hash += mix64(S ^ mix64((uint64_t)k));
        c.max = k > c.max ? k : c.max;
    }
    unsigned todo = __ballot_sync(FULL, on);
#pragma unroll 1
    while (todo) {  // one addition per size
        const unsigned k0 = __shfl_sync(FULL, k, __ffs(todo) - 1);
        const unsigned m = __ballot_sync(FULL, on && k == k0);
        todo &= ~m;
        if (lane == 0) {
            const unsigned add = (unsigned)__popc(m), old = atomicAdd(&hist[k0], add);
            if (old + add < old)
                atomicAdd(reinterpret_cast<unsigned long long *>(out + MCE_OUT_HIST + k0), 1ull << 32);
        }
    }
    __syncwarp();
}

// Pages of a warp's stack in local memory (32 frames each: a word per lane and
// field); beyond kSoftPages a step takes one child at a time.
constexpr unsigned kSoftPages = 8, kPages = kSoftPages + 128 / 32 + 1;

// The bottom 32 frames of a full stack to a page, or the last page back to an
// empty stack.
template <int W>
__device__ __noinline__ void pool_page(const PoolAt &at, uint32_t (*paged)[PoolShape<W>::kFields], unsigned &pages,
                                       unsigned &cnt)
{
    constexpr unsigned F = PoolShape<W>::kFields;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const unsigned lane = threadIdx.x & 31u;
    uint32_t *stk = reinterpret_cast<uint32_t *>(smem_raw + at.region + PoolShape<W>::kStackOff);
    unsigned n = cnt, pg = pages;
    if (n != 0u) {
#pragma unroll 1
        for (unsigned w = 0; w < F; ++w) paged[pg][w] = stk[w * 32u + lane];
        ++pg;
        n -= 32u;
#pragma unroll 1
        for (unsigned i = 0; i < n * F; i += 32u) {
            __syncwarp();
            const bool on = i + lane < n * F;
            const uint32_t t = on ? stk[32u * F + i + lane] : 0u;
            __syncwarp();
            if (on) stk[i + lane] = t;
        }
    } else {
        --pg;
#pragma unroll 1
        for (unsigned w = 0; w < F; ++w) stk[w * 32u + lane] = paged[pg][w];
        n = 32u;
    }
    __syncwarp();
    pages = pg;
    cnt = n;
}

// A run's counters so far to the result array (all 32 lanes).
template <int D = 0>
__device__ __noinline__ void pool_fold(uint64_t *out, unsigned cnt, unsigned intl, unsigned dead)
{
    Counters c;
    c.cnt = cnt;
    c.intl = intl;
    c.dead = dead;
    flush_counters(c, out);
}

// What a long run looks at every few steps: it gives its oldest frames (of
// the fullest subtrees; at most half of all it has) to idle warps -- the
// block's own first, then any -- and watches for an abort and the search's
// time limit.  True when the search has been aborted.
template <int W>
__device__ __noinline__ bool pool_watch(const PoolAt &at, uint32_t (*paged)[PoolShape<W>::kFields], unsigned pages,
                                        unsigned cnt, unsigned &gave_io, uint64_t deadline, uint64_t *out)
{
    constexpr unsigned F = PoolShape<W>::kFields;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const unsigned lane = threadIdx.x & 31u;
    LocalHdr *h = reinterpret_cast<LocalHdr *>(smem_raw + at.lq);
    unsigned near = 0u, far = 0u;
    if (lane == 0) {
        Ctl *ctl = h->ctl;
        const unsigned ab = ld_relaxed(&ctl->abort), gh = ld_relaxed(&ctl->head), gt = ld_relaxed(&ctl->tail);
        const unsigned id = vld(&h->idle);
        const bool shared_ring = h->total > blockDim.x / 32u;
        const unsigned st = shared_ring ? ld_relaxed(&ctl->starving) : id;
        const int l = (int)id - (int)(vld(&h->tail) - vld(&h->head));
        const int g = (int)st - max((int)(gt - gh), 0) - max(l, 0);
        near = (unsigned)min(max(l, 0), 4);
        far = shared_ring ? (unsigned)min(max(g, 0), 4) : 0u;
        if (4u * st > h->total) near |= 16u;  // draining (or filling): smaller frames too
        if (deadline != ~0ull && global_ns() > deadline) set_status(out, ctl, MCE_ETIMEOUT);
        if (ab) near = 32u;
    }
    near = __shfl_sync(FULL, near, 0);
    far = __shfl_sync(FULL, far, 0);
    if (near == 32u) return true;
    const unsigned min_p = (near & 16u) != 0u ? h->give_p / 2u : h->give_p;
    near &= 15u;
    unsigned gave = gave_io;
    const unsigned keep = (cnt + 32u * pages - gave + 1u) / 2u;  // frames this warp keeps
#pragma unroll 1
    for (; near + far != 0u && gave + keep < cnt + 32u * pages; ++gave) {
        uint32_t frame = at.region + PoolShape<W>::kStackOff + (gave - 32u * pages) * F * 4u;
        const bool out_page = gave < 32u * pages;
        const unsigned pg = gave / 32u, q0 = (gave & 31u) * F;
        if (out_page) {  // a frame that was paged out: through the scratch words
            frame = at.region + PoolShape<W>::kScratchOff;
            uint32_t *sc = reinterpret_cast<uint32_t *>(smem_raw + frame);
#pragma unroll 1
            for (unsigned w = 0; w < F; ++w) {
                const unsigned q = w * 32u + lane - q0;
                if (q < F) sc[q] = paged[pg][w];
            }
            __syncwarp();
        }
        const uint32_t *f = reinterpret_cast<const uint32_t *>(smem_raw + frame);
        unsigned np = 0;
#pragma unroll
        for (int k = 0; k < W; ++k) np += (unsigned)__popc(f[k]);
        const bool local = near != 0u;
        if (np < min_p || !pool_give<W>(at, frame, local)) break;
        near -= local ? 1u : 0u;
        far -= local ? 0u : 1u;
        if (out_page) {
            const uint32_t m = f[2 * W];
            __syncwarp();
#pragma unroll 1
            for (unsigned w = 0; w < F; ++w)
                if (w * 32u + lane - q0 == 2u * W) paged[pg][w] = m;
        }
    }
    gave_io = gave;
    return false;
}

// Search the `cnt` start frames on the warp's stack to the end (all 32
// lanes).  Leaves go to a buffer that is worked off 32 at a time, so that the
// two 64-bit mixes of a clique's hash run on full warps.  cap = frames the
// stack holds (at least 64).  Frames that would overflow it page out: the
// bottom 32 go to local memory, a word per lane and field, and come back when
// the stack is empty.  How many frames there can be: the frames pushed by one
// step (at most 32) lie on top of the ones they are children of, so while
// several steps' frames are on the stack their subtrees' heights fall from
// step to step, and there are at most 32 per level of the tree.  Beyond
// kSoftPages pages a step takes one child at a time, and the stack then grows
// by less than one frame per level (at most 128), which the last pages hold.
// Ends early, with the rest unsearched, only when the whole search has been
// aborted.
template <int W, int PIVOT>
__device__ __noinline__ void pool_run(const PoolAt at, unsigned cnt, unsigned cap, uint64_t *out, uint64_t deadline,
                                      PoolCounters &pc)
{
    using Sh = PoolShape<W>;
    constexpr unsigned F = Sh::kFields;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const unsigned lane = threadIdx.x & 31u;
    const unsigned below = (1u << lane) - 1u;
    const uint32_t *A0 = reinterpret_cast<const uint32_t *>(smem_raw + at.rows);
    const uint64_t *lhv = reinterpret_cast<const uint64_t *>(smem_raw + at.hash);
    uint32_t *leaf = reinterpret_cast<uint32_t *>(smem_raw + at.region + PoolShape<W>::kLeafOff);
    const uint32_t *rs0 = reinterpret_cast<const uint32_t *>(smem_raw + at.region + Sh::kRs0Off);
    uint32_t *stk = reinterpret_cast<uint32_t *>(smem_raw + at.region + PoolShape<W>::kStackOff);
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw + at.hist);
    uint32_t paged[kPages][F];
    unsigned pages = 0;
    unsigned nleaf = 0;  // buffered leaves
    unsigned gave = 0;   // frames at the bottom (of the first page, if any) that were given away
    // (a step that scores pivots takes several times as long)
    const unsigned give_mask = reinterpret_cast<const LocalHdr *>(smem_raw + at.lq)->give_mask >>
                               (PIVOT == MCE_PIVOT_GREEDY ? 0 : 2);
    PoolCounters c;

#pragma unroll 1
    for (unsigned step = 1;; ++step) {
        if (cnt + 32u > cap || (cnt == 0u && pages != 0u)) pool_page<W>(at, paged, pages, cnt);
        if (nleaf >= 32u || (cnt == 0u && nleaf != 0u)) {
            const unsigned n = nleaf < 32u ? nleaf : 32u;
            nleaf -= n;
            pool_leaves(leaf + 3u * nleaf, n, lane, rs0, hist, out, c);
        }
        if (cnt == 0u) {
            if (nleaf == 0u) break;
            continue;
        }
        if ((step & give_mask) == 0u || (step <= 12u && (step & 3u) == 0u)) {
            const bool look = (step & 511u) == 0u;
            if (pool_watch<W>(at, paged, pages, cnt, gave, look ? deadline : ~0ull, out)) break;
            if (look && (step & (kFoldSteps - 1u)) == 0u) {
                pool_fold<>(out, c.cnt, c.intl, c.dead);
                c.cnt = c.intl = c.dead = 0u;
            }
        }

        // ---- hand out children: lane j looks at the j-th frame from the top
        const uint32_t mj = lane < cnt ? stk[(cnt - 1u - lane) * F + 2 * W] : 0u;
        const unsigned cj = ((mj >> 17) & 127u) - (mj >> 24);  // children left
        unsigned incl = cj;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(FULL, incl, o);
            incl += (int)lane >= o ? y : 0u;
        }
        const unsigned excl = incl - cj;
        const unsigned most = pages < kSoftPages ? 32u : 1u;
        // first lane of every frame's run of children
        const unsigned firsts = __reduce_or_sync(FULL, cj != 0u && excl < most ? 1u << excl : 0u);
        const unsigned total = min(most, __shfl_sync(FULL, incl, 31));
        const unsigned upto = firsts & (below | (1u << lane));
        const unsigned fi = (unsigned)__popc(upto) - 1u;  // this lane's frame from the top
        const bool act = lane < total;
        const unsigned gone_frames = (unsigned)__popc(__ballot_sync(FULL, lane < cnt && incl <= total));
        const uint32_t *f = stk + (cnt - 1u - (act ? fi : 0u)) * F;
        uint32_t P[W], X[W], L[W], a[W];
#pragma unroll
        for (int k = 0; k < W; ++k) {
            P[k] = f[k];
            X[k] = f[W + k];
        }
        const uint32_t meta = f[2 * W];
        const uint64_t S = (uint64_t)f[2 * W + 1] | ((uint64_t)f[2 * W + 2] << 32);
        __syncwarp();
        if (cj != 0u && excl < total && incl > total)  // the frame that keeps children
            stk[(cnt - 1u - lane) * F + 2 * W] = mj + ((total - excl) << 24);
        cnt -= gone_frames;
        gave = min(gave, cnt + 32u * pages);

        // ---- this lane's child v: element i of L, the earlier ones to X
        // (lanes without one compute on the top frame, and none of it counts)
        const unsigned slot = (meta >> 7) & 7u;
        const uint32_t *A = A0 + slot * Sh::kSlotRows;
        pool_row<W>(a, A + (meta & 127u) * Sh::kStride);
        unsigned i = act ? (meta >> 24) + lane - (31u - (unsigned)__clz((int)upto)) : 0u;
        // past[k]: the child lies past word k of L
        bool past[W];
        uint32_t lw;
        unsigned vk = 0u;
        {
            unsigned run = 0u, skip = 0u;
#pragma unroll
            for (int k = 0; k < W; ++k) L[k] = P[k] & ~a[k];
            lw = L[0];
#pragma unroll
            for (int k = 0; k < W - 1; ++k) {
                run += (unsigned)__popc(L[k]);
                past[k] = i >= run;
                lw = past[k] ? L[k + 1] : lw;
                skip = past[k] ? run : skip;
                vk = past[k] ? 32u * (k + 1) : vk;
            }
            past[W - 1] = false;
            i -= skip;
        }
        const unsigned vb = select_bit(lw, i) & 31u;
        const unsigned v = vk + vb;
        const uint32_t low = (1u << vb) - 1u;
        pool_row<W>(a, A + v * Sh::kStride);
        const uint64_t Sc = S + lhv[slot * Sh::kSlotVerts + v];
        uint32_t op = 0u, ox = 0u;
#pragma unroll
        for (int k = 0; k < W; ++k) {
            const uint32_t g = L[k] & (past[k] ? FULL : (k == 0 || past[k > 0 ? k - 1 : 0] ? low : 0u));
            P[k] = P[k] & ~g & a[k];    // (P minus the earlier children) n N(v)
            X[k] = (X[k] | g) & a[k];   // (X and the earlier children) n N(v)
            op |= P[k];
            ox |= X[k];
        }
        const bool bp = act && op != 0u, bx = ox != 0u;
        c.intl += bp ? 1u : 0u;
        c.dead += act && !bp && bx ? 1u : 0u;
        unsigned p = 0u;
        if (PIVOT == MCE_PIVOT_GREEDY) {
#pragma unroll
            for (int k = 0; k < W; ++k) L[k] = bx ? X[k] : P[k];
            p = bp ? pool_first<W>(L) : 0u;
        } else if (bp) {
            // argmax |P' n N(u)| over X' (TX, NX) or P' u X' (TomitaBB),
            // candidates in increasing position with '>' keeping the earliest;
            // one that covers all of P' cannot be beaten, which ends the scan
            // under every rule (as Naude's early exit does)
            p = pool_first<W>(P);  // TX with X' empty: first of P'
            int best = -1, all = 0;
#pragma unroll
            for (int k = 0; k < W; ++k) all += __popc(P[k]);
            bool open = true;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                uint32_t cand = (PIVOT == MCE_PIVOT_GREEDY_TX) ? X[k] : (P[k] | X[k]);
#pragma unroll 1
                while (cand != 0u && open) {
                    const unsigned w = 32u * k + (unsigned)__ffs(cand) - 1u;
                    cand &= cand - 1u;
                    uint32_t r[W];
                    pool_row<W>(r, A + w * Sh::kStride);
                    int n = 0;
#pragma unroll
                    for (int j = 0; j < W; ++j) n += __popc(P[j] & r[j]);
                    if (n > best) {
                        best = n;
                        p = w;
                    }
                    open = best != all;
                }
            }
        }
        pool_row<W>(a, A + p * Sh::kStride);
        unsigned n = 0;
#pragma unroll
        for (int k = 0; k < W; ++k) n += (unsigned)__popc(P[k] & ~a[k]);  // |L'|, L' = P' \ N(p)

        // ---- P' u X' empty: R u {v} is a maximal clique
        const unsigned rel = ((meta >> 10) & 127u) + 1u;
        const bool lf = act && !bp && !bx;
        const unsigned lm = __ballot_sync(FULL, lf);
        if (lf) {
            uint32_t *e = leaf + 3u * (nleaf + (unsigned)__popc(lm & below));
            e[0] = (uint32_t)Sc;
            e[1] = (uint32_t)(Sc >> 32);
            e[2] = (slot << 8) | rel;
        }
        nleaf += (unsigned)__popc(lm);
        // ---- a child with children of its own goes on the stack
        const bool push = bp && n != 0u;
        const unsigned pm = __ballot_sync(FULL, push);
        if (push) {
            uint32_t *fr = stk + (cnt + (unsigned)__popc(pm & below)) * F;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                fr[k] = P[k];
                fr[W + k] = X[k];
            }
            fr[2 * W] = p | (slot << 7) | (rel << 10) | (n << 17);
            fr[2 * W + 1] = (uint32_t)Sc;
            fr[2 * W + 2] = (uint32_t)(Sc >> 32);
        }
        cnt += (unsigned)__popc(pm);
        __syncwarp();
    }
    pc = c;
}

// The warp tier with sets of `cls` words (the same for the whole search, so
// that one instance of the code is in the instruction caches).
template <int K, int PIVOT>
__device__ __forceinline__ void pool_run_class(unsigned cls, const PoolAt &at, unsigned cnt, uint32_t bytes,
                                               uint64_t *out, uint64_t deadline, PoolCounters &c)
{
    if (cls == 1u) pool_run<1, PIVOT>(at, cnt, (bytes - PoolShape<1>::kStackOff) / (4u * PoolShape<1>::kFields), out, deadline, c);
    else if (cls == 2u) pool_run<2, PIVOT>(at, cnt, (bytes - PoolShape<2>::kStackOff) / (4u * PoolShape<2>::kFields), out, deadline, c);
    else if (cls == 3u) pool_run<3, PIVOT>(at, cnt, (bytes - PoolShape<3>::kStackOff) / (4u * PoolShape<3>::kFields), out, deadline, c);
    else pool_run<4, PIVOT>(at, cnt, (bytes - PoolShape<4>::kStackOff) / (4u * PoolShape<4>::kFields), out, deadline, c);
}

// The search proper: this warp expands frames until the search is over or
// aborts.  rows, order: the renumbered adjacency (rows of prm.wp words) and
// the labels; hist, lq, region: this block's
// clique-size histogram and ring and this warp's region of shared memory.
// direct: the block holds the whole graph's rows, hash terms and positions in
// the warp tier's layout (graphs of at most 128 vertices).  Called by all 32
// lanes of every warp of the block.
template <int K, int PIVOT, bool LIST>
__device__ __forceinline__ void search_loop(const SearchParams &prm, const uint32_t *rows, uint32_t *hist,
                                            const LocalQ &lq, const Thresholds th, const PoolAt at, bool direct,
                                            Counters &cn)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr bool POOL = !LIST;
    const uint32_t n = prm.n, rw = prm.wp;     // rw: words from row to row
    const uint32_t sw = min(rw, 32u * K);      // words of a set
    Ctl *ctl = prm.ctl;
    LocalHdr *h = lq.h;
    const unsigned lane = threadIdx.x & 31u;
    const bool mine = lane * K < sw;  // this lane's words exist
    const unsigned warps = blockDim.x >> 5;
    const bool ring_shared = prm.total_groups > warps;
    const unsigned qmask = prm.qcap - 1u;
    uint32_t P[K], X[K], L[K];
#pragma unroll
    for (int k = 0; k < K; ++k) P[k] = X[k] = L[k] = 0u;
    unsigned pe = 0, rs = 0;
    uint64_t S = 0;
    int d = 0, dbase = 0;
    bool work = false;
    bool lempty = true;     // the current frame's branching set is exhausted
    bool fresh = false;     // the frame was just taken from a ring
    bool open = true;       // the device-wide ring was short of frames when last seen
    unsigned pslots = 0u;   // subproblems waiting on this warp's stack
    // lane 0 only: the polling role, and a claimed ticket of the device-wide
    // ring whose frame this (idle) warp takes once it is published
    bool poller = false, held = false;
    unsigned hticket = 0;
    // Clique listing (ListParams): this warp's index, the |R| of the frame it
    // took last, and (lane 0) the chunk it appends records to.
    const unsigned gidx = blockIdx.x * warps + (threadIdx.x >> 5);
    unsigned rsb = 0, cpos = 0, cend = 0;
    bool cfull = false;

    // ancestors of the current frame: P and X, and the scalars, one each in
    // lanes 0..3 (pivot | end, |R|, S low, S high)
    uint32_t stack[kStackDepth][2 * K + 1];
    const PoolOffsets po = pool_offsets(th.cls);
    uint16_t *ppos = reinterpret_cast<uint16_t *>(smem_raw + at.region + po.pos);

    uint64_t quiet_since = 0, t_busy = 0;
    const uint64_t t_start = global_ns();
    // (~0: none, also where the sum does not fit)
    const uint64_t deadline = prm.limit_ns < ~0ull - t_start ? t_start + prm.limit_ns : ~0ull;
    unsigned last_pend = 0xffffffffu, last_head = 0xffffffffu;
    unsigned backoff = 64;

    if (POOL && threadIdx.x == 0) {  // what the warp tier needs to give frames away
        h->ctl = ctl;
        h->gseq = prm.seq;
        h->gframes = prm.frames;
        h->qcap = prm.qcap;
        h->fs = prm.fs;
        h->margin = push_margin(prm);
        h->wp = rw;
        h->n = n;
        h->give_p = prm.tune.give_p ? prm.tune.give_p : th.share;
        h->total = ring_shared ? prm.total_groups : warps;
        h->give_mask = prm.tune.give_steps - 1u;
    }
    __syncthreads();

    auto get_row = [&](uint32_t (&r)[K], unsigned v) {
        if (mine) {
            load_row<K>(r, rows + (size_t)v * rw + lane * K);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) r[k] = 0u;
        }
    };
    auto scalars = [&]() -> uint32_t {
        return lane == 0u ? pe : (lane == 1u ? rs : (lane == 2u ? (uint32_t)S : (uint32_t)(S >> 32)));
    };

    // This lane's words of R for a frame of this warp with |R| = r, plus
    // vertex `extra` when it is >= 0 (listing only).
    auto r_bits = [&](unsigned r, int extra, uint32_t (&out)[K]) {
        const uint32_t *b = prm.lst.base + (size_t)gidx * rw + lane * K;
#pragma unroll
        for (int k = 0; k < K; ++k) out[k] = mine ? b[k] : 0u;
        const uint16_t *pp = prm.lst.path + (size_t)gidx * n;
#pragma unroll 1
        for (unsigned j = rsb; j < r; ++j)
#pragma unroll
            for (int k = 0; k < K; ++k) out[k] |= set_bit<K>(k, pp[j], lane);
        if (extra >= 0)
#pragma unroll
            for (int k = 0; k < K; ++k) out[k] |= set_bit<K>(k, (unsigned)extra, lane);
    };

    // Append the maximal clique R u {v} (|R| = rs) as a record to this warp's
    // chunk.
    auto emit_clique = [&](int v) {
        const unsigned k = rs + 1u;
        unsigned ok = 0u, wpos = 0u;
        if (lane == 0) {
            const unsigned need = k + 1u, CW = prm.lst.chunk_words;
            if (cpos + need > cend && !cfull) {
                if (cend) prm.lst.fill[cend / CW - 1u] = cpos - (cend - CW);  // retire the chunk
                const unsigned c = atomicAdd(prm.lst.next_chunk, 1u);
                if (c < prm.lst.n_chunks) {
                    cpos = c * CW;
                    cend = cpos + CW;
                } else {
                    cpos = cend = 0u;
                    cfull = true;
                    atomicExch(prm.lst.overflow, 1u);
                }
            }
            if (!cfull && cpos + need <= cend) {
                ok = 1u;
                wpos = cpos;
                cpos += need;
            }
        }
        ok = __shfl_sync(FULL, ok, 0);
        wpos = __shfl_sync(FULL, wpos, 0);
        if (!ok) return;
        uint32_t rb[K];
        const uint32_t *b = prm.lst.base + (size_t)gidx * rw + lane * K;
#pragma unroll
        for (int kk = 0; kk < K; ++kk) rb[kk] = mine ? b[kk] : 0u;
        unsigned o = lanes_below_sum(set_count<K>(rb), lane);
        // R of the taken frame fills slots [0, rsb), the path [rsb, rs), the
        // leaf vertex slot rs
        uint32_t *rec = prm.lst.rec + wpos + 1u;
#pragma unroll
        for (int kk = 0; kk < K; ++kk) {
            uint32_t w = rb[kk];
            while (w) {
                if (o < rsb) rec[o] = (lane * K + kk) * 32u + (unsigned)(__ffs(w) - 1);
                ++o;
                w &= w - 1u;
            }
        }
        const uint16_t *pp = prm.lst.path + (size_t)gidx * n;
        for (unsigned j = rsb + lane; j < rs; j += 32u) rec[j] = pp[j];
        if (lane == 0) {
            rec[rs] = (uint32_t)v;
            prm.lst.rec[wpos] = 0x80000000u | k;
        }
    };

    // Write a frame (and R when listing) to slot `ticket` of a ring and
    // publish it.
    auto publish = [&](bool local, unsigned ticket, const uint32_t (&fP)[K], const uint32_t (&fX)[K], unsigned fpe,
                       unsigned frs, uint64_t fS, const uint32_t (&fR)[K]) {
        uint32_t *fr = local ? lq.frames + (size_t)(ticket & lq.mask) * frame_words(rw, LIST)
                             : prm.frames + (size_t)(ticket & qmask) * prm.fs;
        if (mine) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                fr[kFrameHdr + lane * K + k] = fP[k];
                fr[kFrameHdr + rw + lane * K + k] = fX[k];
                if (LIST) fr[kFrameHdr + 2 * rw + lane * K + k] = fR[k];
            }
        }
        if (lane == 0) {
            fr[0] = fpe;
            fr[1] = frs;
            fr[2] = (uint32_t)fS;
            fr[3] = (uint32_t)(fS >> 32);
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) {
            if (local) vst(&lq.seq[ticket & lq.mask], ticket + 1u);
            else st_release(&prm.seq[ticket & qmask], ticket + 1u);
            cn.note(kDiagDonations);
        }
        __syncwarp();
    };
    // A ticket of the block ring or the device-wide ring for a frame about to
    // be published, or false.  A frame in the block ring is block work (the
    // giver keeps the block active); one in the device-wide ring is a unit of
    // global pending.
    auto reserve = [&](bool local, unsigned &ticket) -> bool {
        unsigned got = 0u;
        ticket = 0u;
        if (lane == 0) {
            if (local) {
                atomicAdd(&h->bwork, 1u);
                got = lq_reserve_push(h, lq.seq, lq.mask, ticket) ? 1u : 0u;
                if (!got) atomicSub(&h->bwork, 1u);
            } else {
                atomicAdd(&ctl->pending, 1u);
                got = q_reserve_push(ctl, prm.seq, qmask, ticket, push_margin(prm)) ? 1u : 0u;
                if (got) cn.note(kDiagGpush);
                else atomicSub(&ctl->pending, 1u);
            }
        }
        got = __shfl_sync(FULL, got, 0);
        ticket = __shfl_sync(FULL, ticket, 0);
        return got != 0u;
    };

    // Give away the front of the branching set of the shallowest frame this
    // warp owns (the stack bottom, else the current frame): the taker gets
    // the first half of L as the frame (P, X, pivot, end = first kept
    // element), the giver keeps (P \ L1, X u L1).  Walking L1 then the rest is
    // exactly the sequential loop of Alg. 4.  A stacked frame with one child
    // left goes whole; a frame with |P| < min_p is kept.
    auto share = [&](bool local, unsigned min_p) {
        const bool from_stack = d > dbase;
        uint32_t sP[K], sX[K], sL[K], sR[K];
        unsigned spe = pe, srs = rs;
        uint64_t sS = S;
        if (from_stack) {
            uint32_t rp[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                sP[k] = stack[dbase][k];
                sX[k] = stack[dbase][K + k];
            }
            const uint32_t m = stack[dbase][2 * K];
            spe = __shfl_sync(FULL, m, 0);
            srs = __shfl_sync(FULL, m, 1);
            sS = (uint64_t)__shfl_sync(FULL, m, 2);
            sS |= (uint64_t)__shfl_sync(FULL, m, 3) << 32;
            get_row(rp, spe & 0xffffu);
#pragma unroll
            for (int k = 0; k < K; ++k) sL[k] = sP[k] & ~rp[k] & set_below<K>(k, spe >> 16, lane);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                sP[k] = P[k];
                sX[k] = X[k];
                sL[k] = L[k];
            }
        }
        const unsigned cl = set_count<K>(sL);
        const unsigned both = __reduce_add_sync(FULL, (set_count<K>(sP) << 16) | cl);
        const unsigned c = both & 0xffffu;
        const unsigned give = c >= 2u ? c / 2u : (c == 1u && from_stack ? 1u : 0u);
        if (give == 0u || (both >> 16) < min_p) return;
        // the position of element #give of L (the first one kept), or the
        // frame's end when everything goes
        unsigned split = spe >> 16;
        if (give < c) {
            const unsigned pre = lanes_below_sum(cl, lane);
            unsigned at_pos = 0xffffffffu;
            if (pre <= give && give < pre + cl) {
                unsigned r = give - pre;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const unsigned cw = (unsigned)__popc(sL[k]);
                    if (at_pos == 0xffffffffu) {
                        if (r < cw) at_pos = (lane * K + k) * 32u + select_bit(sL[k], r);
                        else r -= cw;
                    }
                }
            }
            split = __reduce_min_sync(FULL, at_pos);
        }
        unsigned ticket;
        if (!reserve(local, ticket)) return;
#pragma unroll
        for (int k = 0; k < K; ++k) sR[k] = 0u;
        if (LIST) r_bits(srs, -1, sR);
        publish(local, ticket, sP, sX, (spe & 0xffffu) | (split << 16), srs, sS, sR);
        if (from_stack && give >= c) {
            ++dbase;
            return;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t l1 = sL[k] & set_below<K>(k, split, lane);
            if (from_stack) {
                stack[dbase][k] = sP[k] & ~l1;
                stack[dbase][K + k] = sX[k] | l1;
            } else {
                P[k] &= ~l1;
                X[k] |= l1;
                L[k] &= ~l1;
            }
        }
    };

    // Search what waits on this warp's stack.
    auto pool_flush = [&]() {
        PoolCounters c;
        PoolAt a = at;
        if (!direct) {
            a.rows = at.region;
            a.hash = at.region + po.hash;
            a.pos = at.region + po.pos;
        }
        pool_run_class<K, PIVOT>(th.cls, a, pslots, prm.pool_bytes, prm.out, deadline, c);
        cn.cnt += c.cnt;
        cn.intl += c.intl;
        cn.dead += c.dead;
        cn.hash += c.hash;
        cn.max = c.max > cn.max ? c.max : cn.max;
        pslots = 0u;
    };

    // Hand the frame (tP, tX, tL, pivot tp, |R| = trs, S = tS) to the warp
    // tier; what does not fit beside the subproblems already waiting has
    // those searched first.
    auto pool_take = [&](const uint32_t (&tP)[K], const uint32_t (&tX)[K], unsigned children, unsigned u, unsigned tp,
                         unsigned trs, uint64_t tS) {
        if (lane == 0) cn.note(kDiagLaneTasks);
        if (direct) {
            if (pslots != 0u) pool_flush();
            uint32_t *f = reinterpret_cast<uint32_t *>(smem_raw + at.region + po.stack);
            if (lane < th.cls) {
                f[lane] = tP[0];
                f[th.cls + lane] = tX[0];
            }
            if (lane == 0) {
                f[2 * th.cls] = tp | (trs << 10) | (children << 17);
                f[2 * th.cls + 1] = (uint32_t)tS;
                f[2 * th.cls + 2] = (uint32_t)(tS >> 32);
                reinterpret_cast<uint32_t *>(smem_raw + at.region + po.rs0)[0] = 0u;
            }
            __syncwarp();
            pslots = 1u;
            return;
        }
        const unsigned slots = th.cls == 1u ? PoolShape<1>::kSlots : (th.cls == 2u ? PoolShape<2>::kSlots : 1u);
        if (pslots >= slots) pool_flush();
        const unsigned slot = pslots++;
        uint32_t U[K];
        unsigned cnt = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            U[k] = tP[k] | tX[k];
            cnt += (unsigned)__popc(U[k]);
        }
        unsigned i = slot * 32u * th.cls + lanes_below_sum(cnt, lane);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            uint32_t w = U[k];
#pragma unroll 1
            while (w) {
                const unsigned b = (unsigned)(__ffs(w) - 1);
                w &= w - 1u;
                const unsigned q = (lane * K + k) * 32u + b;
                ppos[i++] = (uint16_t)(q | (((tP[k] >> b) & 1u) ? kPosInP : 0u) | (q == tp ? kPosPivot : 0u));
            }
        }
        __syncwarp();
        if (th.cls == 1u)
            pool_build<1, K>(rows, rw, prm.order, at.region, slot, U[0], u, children, trs, tS);
        else if (th.cls == 2u)
            pool_build<2, K>(rows, rw, prm.order, at.region, slot, U[0], u, children, trs, tS);
        else if (th.cls == 3u)
            pool_build<3, K>(rows, rw, prm.order, at.region, slot, U[0], u, children, trs, tS);
        else
            pool_build<4, K>(rows, rw, prm.order, at.region, slot, U[0], u, children, trs, tS);
    };
    // whether a frame of |P| = np, |P u X| = u and c children fits the tier
    auto pool_fits = [&](unsigned np, unsigned u, unsigned c) -> bool {
        return POOL && prm.t2_max_p != 0u && u <= 32u * th.cls && np <= min(prm.t2_max_p, th.task) && c <= 127u;
    };

#pragma unroll 1
    for (unsigned it = 1;; ++it) {
        // ---- A: a frame whose branching set is exhausted returns to its
        // parent (a stacked level always has children left), or the warp's
        // work is done.  (Subproblems of the warp tier are searched first: the
        // frames they give away are block work, which this warp's unit keeps
        // alive.)
        if (work && lempty) {
            if (d > dbase) {
                --d;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    P[k] = stack[d][k];
                    X[k] = stack[d][K + k];
                }
                const uint32_t m = stack[d][2 * K];
                pe = __shfl_sync(FULL, m, 0);
                rs = __shfl_sync(FULL, m, 1);
                S = (uint64_t)__shfl_sync(FULL, m, 2);
                S |= (uint64_t)__shfl_sync(FULL, m, 3) << 32;
                uint32_t rp[K];
                get_row(rp, pe & 0xffffu);
#pragma unroll
                for (int k = 0; k < K; ++k) L[k] = P[k] & ~rp[k] & set_below<K>(k, pe >> 16, lane);
                lempty = false;
            } else {
                if (POOL && pslots != 0u) pool_flush();
                work = false;
                if (lane == 0) {
                    cn.note(kDiagBusyNs, global_ns() - t_busy);
                    atomicAdd(&h->idle, 1u);
                    if (ring_shared) atomicAdd(&ctl->starving, 1u);
                    // the last work of the block gives back its unit
                    if (atomicSub(&h->bwork, 1u) == 1u) atomicSub(&ctl->pending, 1u);
                }
                backoff = 64;
            }
        }

        // ---- B: idle warps take a frame (block ring first, then the
        // device-wide ring), or end with the search; the block's polling warp
        // refreshes the cached global state for the others
        if (!work) {
            unsigned code = 0u, ticket = 0u;  // 1: block ring, 2: device-wide ring, 3: the end
            if (lane == 0) {
                // (nothing to be seen: sleep on, in a loop of a few instructions)
#pragma unroll 1
                for (unsigned naps = 0; naps < 64u && !poller && !held; ++naps) {
                    if (vld(&h->done) != 0u || vld(&h->tail) != vld(&h->head) || vld(&h->poller) == 0u ||
                        (int)(vld(&h->g_tail) - vld(&h->g_head)) > 0)
                        break;
                    __nanosleep(backoff);
                    backoff = backoff < prm.tune.idle_sleep_ns ? backoff * 2u : prm.tune.idle_sleep_ns;
                }
                if (vld(&h->done)) code = 3u;
                if (code == 0u && held && ld_acquire(&prm.seq[hticket & qmask]) == hticket + 1u) {
                    code = 2u;
                    ticket = hticket;
                    held = false;
                }
                if (code == 0u && !held && vld(&h->tail) != vld(&h->head) && lq_reserve_pop(h, lq.seq, lq.mask, ticket))
                    code = 1u;
                if (code == 0u && !poller) poller = atomicCAS(&h->poller, 0u, 1u) == 0u;
                if (code == 0u && poller) {
                    const uint64_t now = global_ns();
                    const unsigned ab = ld_relaxed(&ctl->abort), pend = ld_relaxed(&ctl->pending);
                    const unsigned gh = ld_relaxed(&ctl->head), gt = ld_relaxed(&ctl->tail);
                    const unsigned st = ld_relaxed(&ctl->starving);
                    vst(&h->g_head, gh);
                    vst(&h->g_tail, gt);
                    vst(&h->g_starving, st);
                    *reinterpret_cast<volatile unsigned long long *>(&h->stamp) = now;
                    if (ab || pend == 0u) {
                        vst(&h->done, ab ? 2u : 1u);
                        code = 3u;
                    }
                    // a stalled search: nothing moved for the whole budget
                    if (pend != last_pend || gh != last_head || quiet_since == 0) {
                        quiet_since = now;
                        last_pend = pend;
                        last_head = gh;
                    } else if (now - quiet_since > prm.timeout_ns) {
                        set_status(prm.out, ctl, MCE_ETIMEOUT);
                    }
                    if (now - t_start > prm.limit_ns) set_status(prm.out, ctl, MCE_ETIMEOUT);
                    if (prm.trace) {
                        const unsigned ti = atomicAdd(&h->trace_n, 1u);
                        if (ti < prm.trace_per_block) {
                            const unsigned busy = warps - min(warps, vld(&h->idle));
                            const unsigned qg = (int)(gt - gh) > 0 ? min(gt - gh, 65535u) : 0u;
                            unsigned long long *rec = prm.trace + 2ull * ((size_t)blockIdx.x * prm.trace_per_block + ti);
                            rec[0] = now;
                            rec[1] = (unsigned long long)busy | ((unsigned long long)qg << 32) |
                                     ((unsigned long long)min(st, 65535u) << 48);
                        }
                    }
                }
                if (code == 0u && !held && (int)(vld(&h->g_tail) - vld(&h->g_head)) > 0) {
                    cn.note(kDiagGtry);
                    if (ring_shared) {
                        if (q_claim(ctl, 1u, hticket) != 0u) {
                            if (ld_acquire(&prm.seq[hticket & qmask]) == hticket + 1u) {
                                code = 2u;
                                ticket = hticket;
                            } else {
                                held = true;
                            }
                        } else {
                            vst(&h->g_head, vld(&h->g_tail));  // (seen empty: wait for the next refresh)
                        }
                    } else if (q_reserve_pop(ctl, prm.seq, qmask, ticket, cn.diag + kDiagCasFail, prm.tune.pop_tries)) {
                        code = 2u;
                    }
                }
            }
            code = __shfl_sync(FULL, code, 0);
            ticket = __shfl_sync(FULL, ticket, 0);
            if (code == 3u) break;
            if (code == 0u) {
                // the poller (or holder of a ticket) backs off too
                if (lane == 0 && (poller || held)) {
                    __nanosleep(backoff < 512u ? backoff : 512u);
                    backoff = backoff < 512u ? backoff * 2u : 512u;
                }
                __syncwarp();
                continue;
            }
            const bool local = code == 1u;
            const uint32_t *fr = local ? lq.frames + (size_t)(ticket & lq.mask) * frame_words(rw, LIST)
                                       : prm.frames + (size_t)(ticket & qmask) * prm.fs;
            __threadfence();
            if (local) {
                const volatile uint32_t *v = fr;
                pe = v[0];
                rs = v[1];
                S = (uint64_t)v[2] | ((uint64_t)v[3] << 32);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    P[k] = mine ? v[kFrameHdr + lane * K + k] : 0u;
                    X[k] = mine ? v[kFrameHdr + rw + lane * K + k] : 0u;
                    if (LIST && mine)
                        prm.lst.base[(size_t)gidx * rw + lane * K + k] = v[kFrameHdr + 2 * rw + lane * K + k];
                }
            } else {
                pe = __ldcg(fr + 0);
                rs = __ldcg(fr + 1);
                S = (uint64_t)__ldcg(fr + 2) | ((uint64_t)__ldcg(fr + 3) << 32);
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    P[k] = mine ? __ldcg(fr + kFrameHdr + lane * K + k) : 0u;
                    X[k] = mine ? __ldcg(fr + kFrameHdr + rw + lane * K + k) : 0u;
                    if (LIST && mine)
                        prm.lst.base[(size_t)gidx * rw + lane * K + k] = __ldcg(fr + kFrameHdr + 2 * rw + lane * K + k);
                }
            }
            __syncwarp();
            if (lane == 0) {
                if (local) {
                    __threadfence_block();
                    vst(&lq.seq[ticket & lq.mask], ticket + lq.mask + 1u);
                } else {
                    st_release(&prm.seq[ticket & qmask], ticket + prm.qcap);
                    // an already active block absorbs the frame's unit
                    if (atomicAdd(&h->bwork, 1u) != 0u) atomicSub(&ctl->pending, 1u);
                    cn.note(kDiagGlobal);
                }
                atomicSub(&h->idle, 1u);
                if (ring_shared) atomicSub(&ctl->starving, 1u);
                cn.note(kDiagSteals);
                if (poller) {  // busy now: another idle warp polls
                    atomicExch(&h->poller, 0u);
                    poller = false;
                }
                t_busy = global_ns();
            }
            quiet_since = 0;
            work = true;
            fresh = true;
            lempty = false;
            rsb = rs;
            d = dbase = 0;
            uint32_t rp[K];
            get_row(rp, pe & 0xffffu);
#pragma unroll
            for (int k = 0; k < K; ++k) L[k] = P[k] & ~rp[k] & set_below<K>(k, pe >> 16, lane);
        }

        // ---- a frame just taken that fits the warp tier goes there whole
        if (fresh) {
            fresh = false;
            uint32_t u = 0;
#pragma unroll
            for (int k = 0; k < K; ++k) u += (unsigned)__popc(P[k] | X[k]);
            const unsigned pu = __reduce_add_sync(FULL, (set_count<K>(P) << 16) | u);
            const unsigned c = __reduce_add_sync(FULL, set_count<K>(L));
            if (pool_fits(pu >> 16, pu & 0xffffu, c)) {
                if (c != 0u) pool_take(P, X, c, pu & 0xffffu, pe & 0xffffu, rs, S);
                lempty = true;
                continue;
            }
        }

        // ---- busy warps refill the block ring while the block has more idle
        // warps than queued frames, and the device-wide ring while the GPU has
        if ((it & (prm.tune.local_check - 1u)) == 0u) {
            unsigned want = 0u;
            bool half = false;  // draining (or filling): smaller frames too
            if (lane == 0) {
                const int l = (int)vld(&h->idle) - (int)(vld(&h->tail) - vld(&h->head));
                if (l > 0) {
                    want = 1u;
                    half = 4u * vld(&h->idle) > warps;
                } else if ((it & (prm.tune.global_check - 1u)) == 0u) {
                    const uint64_t now = global_ns();
                    if (now - *reinterpret_cast<volatile unsigned long long *>(&h->stamp) > prm.tune.refresh_ns &&
                        atomicCAS(&h->refreshing, 0u, 1u) == 0u) {
                        const unsigned ab = ld_relaxed(&ctl->abort);
                        vst(&h->g_head, ld_relaxed(&ctl->head));
                        vst(&h->g_tail, ld_relaxed(&ctl->tail));
                        vst(&h->g_starving, ld_relaxed(&ctl->starving));
                        if (ab) vst(&h->done, 2u);
                        if (now - t_start > prm.limit_ns) set_status(prm.out, ctl, MCE_ETIMEOUT);
                        *reinterpret_cast<volatile unsigned long long *>(&h->stamp) = now;
                        atomicExch(&h->refreshing, 0u);
                    }
                    if ((int)vld(&h->g_starving) > max((int)(vld(&h->g_tail) - vld(&h->g_head)), 0)) want = 2u;
                    half = 4u * vld(&h->g_starving) > prm.total_groups;
                }
                if (vld(&h->done) == 2u) want = 3u;
                if ((int)(vld(&h->g_tail) - vld(&h->g_head)) < (int)prm.split_target) want |= 4u;
                if (half) want |= 8u;
            }
            want = __shfl_sync(FULL, want, 0);
            open = (want & 4u) != 0u;
            half = (want & 8u) != 0u;
            want &= 3u;
            if (want == 3u) break;
            if (want != 0u) share(want == 1u, (want == 1u ? th.share : th.share_far) >> (half ? 1 : 0));
        }

        // ---- C: expand one child v = first(L).  (Pops and queued frames
        // always carry children, and giving work away always leaves the giver
        // at least one; a frame without would just be returned from.)
        const int v = set_first<K>(L, lane);
        if (v < 0) {
            lempty = true;
            continue;
        }
        uint32_t Pc[K], Xc[K], r[K];
        get_row(r, (unsigned)v);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t b = set_bit<K>(k, (unsigned)v, lane);
            Pc[k] = P[k] & r[k];  // P n N(v)
            Xc[k] = X[k] & r[k];  // X n N(v)
            L[k] &= ~b;
            P[k] &= ~b;  // P <- P \ {v}
            X[k] |= b;   // X <- X u {v}
        }
        const bool bp = __ballot_sync(FULL, set_or<K>(Pc) != 0u) != 0u;
        const bool bx = __ballot_sync(FULL, set_or<K>(Xc) != 0u) != 0u;
        const uint64_t Sc = S + mix64((uint64_t)prm.order[v] + 1u);
        lempty = __ballot_sync(FULL, set_or<K>(L) != 0u) == 0u;
        if (!bp) {
            if (bx) {
                cn.dead += lane == 0 ? 1u : 0u;
            } else {  // P u X empty: R u {v} is a maximal clique
                if (lane == 0) {
                    const unsigned k = rs + 1u;
                    ++cn.cnt;
                    cn.hash += mix64(Sc ^ mix64((uint64_t)k));
                    cn.max = k > cn.max ? k : cn.max;
                    const unsigned old = atomicAdd(&hist[k], 1u);
                    if (old == 0xffffffffu)
                        atomicAdd(reinterpret_cast<unsigned long long *>(prm.out + MCE_OUT_HIST + k), 1ull << 32);
                }
                if (LIST) emit_clique(v);
            }
            continue;
        }
        cn.intl += lane == 0 ? 1u : 0u;

        // ChoosePivotOrdered on the child (P', X')
        unsigned pc;
        if (PIVOT == MCE_PIVOT_GREEDY) {
            pc = (unsigned)(bx ? set_first<K>(Xc, lane) : set_first<K>(Pc, lane));
        } else if (PIVOT == MCE_PIVOT_GREEDY_TX && !bx) {
            pc = (unsigned)set_first<K>(Pc, lane);
        } else {
            // argmax |P' n N(u)| over X' (TX, NX) or P' u X' (TomitaBB), all
            // candidates at once: the lanes' words of P' go to the warp's
            // scratch (the leaf buffer, empty here), every lane scores the
            // candidates in its own words against the whole of P' (16-byte
            // loads starting at a chunk rotated by lane, so a phase of eight
            // lanes hits distinct banks), and one packed max (score + 1,
            // 0xffff - position) keeps the highest score, earliest on ties.
            // NX has TX's pivot (its early exit only saves work).
            uint32_t *pw = reinterpret_cast<uint32_t *>(smem_raw + at.region + (LIST ? 0u : po.leaf));
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (mine) pw[lane * K + k] = Pc[k];
            __syncwarp();
            unsigned best = 0u;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                uint32_t w = (PIVOT == MCE_PIVOT_GREEDY_TX) ? Xc[k] : (Pc[k] | Xc[k]);
#pragma unroll 1
                while (w) {
                    const unsigned b = (unsigned)(__ffs(w) - 1);
                    w &= w - 1u;
                    const unsigned u = (lane * K + k) * 32u + b;
                    const uint32_t *ru = rows + (size_t)u * rw;
                    unsigned c = 0;
                    if (sw >= 4u) {
                        const unsigned nc = sw / 4u;
#pragma unroll 4
                        for (unsigned j = 0; j < nc; ++j) {
                            const unsigned jj = ((j + lane) & (nc - 1u)) * 4u;
                            const uint4 a = *reinterpret_cast<const uint4 *>(pw + jj);
                            const uint4 q = __ldg(reinterpret_cast<const uint4 *>(ru + jj));
                            c += (unsigned)(__popc(a.x & q.x) + __popc(a.y & q.y) + __popc(a.z & q.z) + __popc(a.w & q.w));
                        }
                    } else {
                        for (unsigned j = 0; j < sw; ++j) c += (unsigned)__popc(pw[j] & __ldg(ru + j));
                    }
                    const unsigned key = ((c + 1u) << 16) | (0xffffu - u);
                    best = key > best ? key : best;
                }
            }
            best = __reduce_max_sync(FULL, best);
            __syncwarp();
            pc = 0xffffu - (best & 0xffffu);
        }
        uint32_t Lc[K];
        unsigned u = 0;
        get_row(r, pc);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            Lc[k] = Pc[k] & ~r[k];  // L' = P' \ N(p)
            u += (unsigned)__popc(Pc[k] | Xc[k]);
        }
        const unsigned c = __reduce_add_sync(FULL, set_count<K>(Lc));
        if (c == 0u) continue;
        const unsigned pu = __reduce_add_sync(FULL, (set_count<K>(Pc) << 16) | u);
        if (pool_fits(pu >> 16, pu & 0xffffu, c)) {
            pool_take(Pc, Xc, c, pu & 0xffffu, pc, rs + 1u, Sc);
            continue;
        }
        // Breadth-first split of the top of the tree: a new subtree with a
        // large candidate set goes to the device-wide ring (while that is
        // short of frames) instead of being descended into here.  With the
        // stack full, the rest of this frame (L is non-empty) goes there as it
        // stands, and the warp descends without it.
        const bool split = open && (pu >> 16) >= th.split;
        const bool spill = !split && !lempty && d >= (int)prm.stack_levels;
        if (split || spill) {
            uint32_t fP[K], fX[K], fR[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                fP[k] = split ? Pc[k] : P[k];
                fX[k] = split ? Xc[k] : X[k];
                fR[k] = 0u;
            }
            unsigned ticket;
            const bool got = reserve(false, ticket);
            if (got) {
                if (LIST) r_bits(rs, split ? v : -1, fR);
                publish(false, ticket, fP, fX, split ? (pc | (n << 16)) : pe, split ? rs + 1u : rs, split ? Sc : S, fR);
            }
            if (got && split) continue;
            if (!got && !lempty && d >= (int)prm.stack_levels && lane == 0) set_status(prm.out, ctl, MCE_EOVERFLOW);
            if (!got && !lempty && d >= (int)prm.stack_levels) lempty = true;
        }
        if (!lempty && !spill) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                stack[d][k] = P[k];
                stack[d][K + k] = X[k];
            }
            stack[d][2 * K] = scalars();
            ++d;
        }
        if (LIST && lane == 0) prm.lst.path[(size_t)gidx * n + rs] = (uint16_t)v;  // R grows by v at |R| = rs
        if (LIST) __syncwarp();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            P[k] = Pc[k];
            X[k] = Xc[k];
            L[k] = Lc[k];
        }
        pe = pc | (n << 16);
        rs = rs + 1u;
        S = Sc;
        lempty = false;
    }
    if (LIST && lane == 0 && cend)  // retire the last chunk
        prm.lst.fill[cend / prm.lst.chunk_words - 1u] = cpos - (cend - prm.lst.chunk_words);
}

// Direct layout (n <= 128): rows of `cls` words (stride 4 for three), hash
// terms and positions of the whole graph, once per block, in the order the
// warp tier reads them.  Whole block; a barrier must follow.
__device__ __forceinline__ void direct_layout(const uint32_t *rows, uint32_t rw, const uint32_t *order, uint32_t n,
                                              unsigned cls, uint32_t *drows, uint64_t *dhash, uint16_t *dpos)
{
    const unsigned stride = cls == 3u ? 4u : cls;
    for (unsigned i = threadIdx.x; i < n * stride; i += blockDim.x) {
        const unsigned v = i / stride, w = i % stride;
        drows[i] = w < rw && w < cls ? rows[(size_t)v * rw + w] : 0u;
    }
    for (unsigned i = threadIdx.x; i < n; i += blockDim.x) {
        dhash[i] = mix64((uint64_t)order[i] + 1u);
        dpos[i] = (uint16_t)i;
    }
}

template <int K, int PIVOT, bool LIST, int T>
__global__ void __launch_bounds__(T) search_kernel(const SearchParams prm)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const uint32_t n = prm.n;
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw);
    const uint32_t lq_off = (uint32_t)smem_local_offset(n);
    const LocalQ lq = local_queue_at(smem_raw + lq_off);
    local_queue_reset(lq, blockDim.x / 32u);

#pragma unroll 1
    for (uint32_t i = threadIdx.x; i <= n; i += blockDim.x) hist[i] = 0u;
    const Thresholds th = density_thresholds(prm.ctl->pad3[0], n, prm.tune, prm.split_min_p, PIVOT != MCE_PIVOT_GREEDY);
    const uint32_t *rows = prm.rows;
    const bool direct = !LIST && K == 1 && n <= 128u && prm.t2_max_p != 0u;
    PoolAt at{};
    at.rows = prm.direct_offset;
    at.hash = at.rows + kDirectRows * 4;
    at.pos = at.hash + kDirectVerts * 8;
    at.region = prm.t2_offset + (threadIdx.x >> 5) * prm.pool_bytes;
    at.lq = lq_off;
    at.hist = 0u;
    __syncthreads();
    if (direct)
        direct_layout(rows, prm.wp, prm.order, n, th.cls, reinterpret_cast<uint32_t *>(smem_raw + at.rows),
                      reinterpret_cast<uint64_t *>(smem_raw + at.hash), reinterpret_cast<uint16_t *>(smem_raw + at.pos));
    Counters cn;
    cn.diag = lq.h->diag;
    search_loop<K, PIVOT, LIST>(prm, rows, hist, lq, th, at, direct, cn);
    flush_counters(cn, prm.out);
    __syncthreads();
    if (threadIdx.x == 0) flush_diag(lq.h->diag, prm.out);
#pragma unroll 1
    for (uint32_t i = threadIdx.x; i <= n; i += blockDim.x)
        if (hist[i]) atomicAdd(reinterpret_cast<unsigned long long *>(prm.out + MCE_OUT_HIST + i), (unsigned long long)hist[i]);
}

// Batched form: each block takes graphs of its bucket one at a time, most
// expensive first, and searches each with its own block-local queue region
// (the same frame ring as the single-graph kernel, private to the block).
// Per graph: the root counted (status kept), frames of its children (or a
// subproblem's root) queued, search, reduction into the graph's own result
// array.
template <int K, int PIVOT, int T>
__global__ void __launch_bounds__(T) batch_kernel(const BatchParams bp)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ unsigned cur, root_key;

    unsigned char *region = bp.qbase + (size_t)blockIdx.x * bp.qstride;
    Ctl *ctl = reinterpret_cast<Ctl *>(region);
    unsigned *seq = reinterpret_cast<unsigned *>(region + batch_seq_offset());
    uint32_t *frames = reinterpret_cast<uint32_t *>(region + batch_frames_offset(bp.qcap));
    for (;;) {
        if (threadIdx.x == 0) cur = atomicAdd(bp.next, 1u);
        __syncthreads();
        const unsigned idx = cur;
        if (idx >= bp.count) break;
        // a work item: graph index | part << 16 | parts << 24; a graph split
        // into parts (parts >= 2) spreads over several blocks, each searching
        // the root's children t = part, part + parts, ... (independent
        // subtrees; the root node is counted by part 0)
        const unsigned item = bp.list[idx];
        const unsigned part = (item >> 16) & 0xffu, parts = max(item >> 24, 1u);
        const BatchGraph gd = bp.graphs[item & 0xffffu];
        const uint32_t n = gd.n, WP = gd.wp;
        uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw);
        const LocalQ lq = local_queue_at(smem_raw + smem_local_offset(n));
        local_queue_reset(lq, bp.groups_per_block);
        const bool valid = gd.out[MCE_OUT_STATUS] == 0ull;
        // The root's P and X over positions: all of V and nothing, or, for a
        // subproblem of the outer loop (Alg. 3), the given sets carried
        // through the order, with R = {rv} already chosen.
        const bool sub = gd.root != nullptr;
        bool pne = false, xne = false;
        for (uint32_t w = threadIdx.x; w < WP; w += blockDim.x) {
            uint32_t pw = 0u, xw = 0u;
            if (!sub) {
                const uint32_t base = w * 32u;
                if (n >= base + 32u) pw = FULL;
                else if (n > base) pw = (1u << (n - base)) - 1u;
            } else {
                for (uint32_t b = 0; b < 32u && w * 32u + b < n; ++b) {
                    const uint32_t loc = gd.order[w * 32u + b];
                    pw |= ((gd.root[loc >> 5] >> (loc & 31u)) & 1u) << b;
                    xw |= ((gd.root[gd.w + (loc >> 5)] >> (loc & 31u)) & 1u) << b;
                }
            }
            frames[kFrameHdr + w] = pw;
            frames[kFrameHdr + WP + w] = xw;
            pne = pne || pw != 0u;
            xne = xne || xw != 0u;
        }
        pne = __syncthreads_or(pne) != 0;
        xne = __syncthreads_or(xne) != 0;
        const unsigned r0 = sub ? 1u : 0u;
        const uint64_t s0 = sub ? mix64((uint64_t)gd.label[gd.rv] + 1u) : 0ull;

        // the root is one node: internal, a leaf (R is maximal) or a dead end;
        // the graph's result array starts zeroed (cleared with the batch) and
        // every part adds to it
        // every graph starts from its root's children, but the outer loop's
        // subproblems of up to 128 vertices, which one warp takes whole
        const bool split = !sub || n > 128u;
        if (threadIdx.x == 0 && (!split || part == 0u)) {
            unsigned long long *o = reinterpret_cast<unsigned long long *>(gd.out);
            atomicAdd(o + MCE_OUT_NODES, 1ull);
            if (pne) atomicAdd(o + MCE_OUT_INTERNAL, 1ull);
            if (!pne && xne) atomicAdd(o + MCE_OUT_DEAD_ENDS, 1ull);
            if (!pne && !xne) {
                atomicAdd(o + MCE_OUT_COUNT, 1ull);
                atomicAdd(o + MCE_OUT_HIST + r0, 1ull);
                atomicAdd(o + MCE_OUT_HASH, (unsigned long long)mix64(s0 ^ mix64((uint64_t)r0)));
                atomicMax(o + MCE_OUT_MAX_SIZE, (unsigned long long)r0);
            }
        }
        // (a subproblem's order becomes the original labels: the search reads
        // it for the hash terms alone)
        if (sub) {
            __syncthreads();
#pragma unroll 1
            for (uint32_t j = threadIdx.x; j < n; j += blockDim.x) gd.order[j] = gd.label[gd.order[j]];
        }
#pragma unroll 1
        for (uint32_t j = threadIdx.x; j <= n; j += blockDim.x) hist[j] = 0u;

        // ChoosePivotOrdered at the root: the key (score + 1) << 12 | (4095 -
        // position) is largest for the best score, earliest on ties; GreedyBB
        // scores nothing (first of X, else of P), GreedyBBTX/NX score
        // |P n N(u)| over X (else first of P), TomitaBB over P u X.
        if (threadIdx.x == 0) root_key = 0u;
        __syncthreads();
        {
            unsigned mine = 0u;
            for (uint32_t u = threadIdx.x; u < n; u += blockDim.x) {
                const bool inp = (frames[kFrameHdr + (u >> 5)] >> (u & 31u)) & 1u;
                const bool inx = (frames[kFrameHdr + WP + (u >> 5)] >> (u & 31u)) & 1u;
                const bool cand = (PIVOT == MCE_PIVOT_TOMITA) ? (inp || inx) : (xne ? inx : inp);
                if (!cand) continue;
                unsigned score = 0;
                if (PIVOT == MCE_PIVOT_TOMITA || (PIVOT == MCE_PIVOT_GREEDY_TX && xne))
                    for (uint32_t w = 0; w < WP; ++w)
                        score += __popc(frames[kFrameHdr + w] & gd.ren[(size_t)u * WP + w]);
                const unsigned key = ((score + 1u) << 12) | (4095u - u);
                mine = key > mine ? key : mine;
            }
            atomicMax(&root_key, mine);
        }
        __syncthreads();
        // the root frame is queued only with children to expand: with X
        // non-empty the pivot may cover all of P (an internal node without
        // children), and a queued frame must always carry a branching vertex
        const unsigned p0 = root_key ? (4095u - (root_key & 4095u)) : 0u;
        bool lne = false;
        if (pne)
            for (uint32_t w = threadIdx.x; w < WP; w += blockDim.x)
                lne = lne || (frames[kFrameHdr + w] & ~gd.ren[(size_t)p0 * WP + w]) != 0u;
        lne = __syncthreads_or(lne) != 0;
        const bool root = valid && pne && lne;
        // frames of `per` consecutive root children each: with v_t the t-th
        // vertex of L = P \ N(p0), children a..b-1 are the frame (P minus v_0
        // ..v_{a-1}, X and those, p0, end = v_b); a part takes every parts-th of
        // them.  Frames go to slots 1.. (slot 0 keeps the root's P and X).
        // per: what makes a frame worth taking, and what the ring has room for.
        unsigned queued = root ? 1u : 0u;
        if (split) {
            __shared__ unsigned lpre[kBatchPartWords + 1];
            const uint32_t *rp0 = gd.ren + (size_t)p0 * WP;
            if (threadIdx.x == 0) {
                unsigned acc = 0;
                for (uint32_t w = 0; w < WP; ++w) {
                    lpre[w] = acc;
                    acc += (unsigned)__popc(frames[kFrameHdr + w] & ~rp0[w]);
                }
                lpre[WP] = acc;
            }
            __syncthreads();
            const unsigned nl = lpre[WP];
            unsigned per = sub ? max(1u, nl / bp.groups_per_block) : gd.per;
            if (parts == 1u) per = max(per, (nl + bp.root_frames - 1u) / bp.root_frames);
            const unsigned all = (nl + per - 1u) / per;
            const unsigned mine = all > part ? (all - part + parts - 1u) / parts : 0u;
            auto child = [&](unsigned t) -> unsigned {  // v_t
                unsigned w = 0;
                while (w + 1u < WP && lpre[w + 1] <= t) ++w;
                uint32_t lw = frames[kFrameHdr + w] & ~rp0[w];
                for (unsigned r = t - lpre[w]; r > 0u; --r) lw &= lw - 1u;
                return w * 32u + (unsigned)(__ffs(lw) - 1);
            };
            for (unsigned j = threadIdx.x; j < mine && j + 1u < bp.qcap; j += blockDim.x) {
                const unsigned t = (part + j * parts) * per;
                const unsigned v = child(t), end = t + per < nl ? child(t + per) : n;
                uint32_t *fr = frames + (size_t)(j + 1u) * bp.fs;
                for (uint32_t q = 0; q < WP; ++q) {
                    const uint32_t pw = frames[kFrameHdr + q];
                    uint32_t below = 0u;
                    if (v >= q * 32u + 32u) below = FULL;
                    else if (v > q * 32u) below = (1u << (v - q * 32u)) - 1u;
                    const uint32_t x = pw & ~rp0[q] & below;
                    fr[kFrameHdr + q] = pw & ~x;
                    fr[kFrameHdr + WP + q] = frames[kFrameHdr + WP + q] | x;
                }
                fr[0] = (p0 & 0xffffu) | (end << 16);
                fr[1] = r0;
                fr[2] = (uint32_t)s0;
                fr[3] = (uint32_t)(s0 >> 32);
                fr[4] = 0u;
            }
            queued = valid && pne ? min(mine, bp.qcap - 1u) : 0u;
            if (threadIdx.x == 0 && valid && mine + 1u > bp.qcap)  // the host sizes the ring for this
                atomicCAS(reinterpret_cast<unsigned long long *>(gd.out + MCE_OUT_STATUS), 0ull,
                          static_cast<unsigned long long>(static_cast<long long>(MCE_EOVERFLOW)));
        }
        // ring state: a subproblem's root frame is consumer ticket 0 in slot 0;
        // root children are consumer tickets 1..queued in slots 1..queued (slot 0 is
        // then free for producer ticket qcap)
        for (uint32_t j = threadIdx.x; j < bp.qcap; j += blockDim.x) {
            unsigned sv = j;
            if (!split && j == 0u && root) sv = 1u;
            if (split && j == 0u) sv = bp.qcap;
            if (split && j >= 1u && j <= queued) sv = j + 1u;
            seq[j] = sv;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            frames[0] = (p0 & 0xffffu) | (n << 16);
            frames[1] = r0;
            frames[2] = (uint32_t)s0;
            frames[3] = (uint32_t)(s0 >> 32);
            ctl->head = split ? 1u : 0u;
            ctl->abort = 0u;
            ctl->tail = split ? queued + 1u : (root ? 1u : 0u);
            ctl->pending = split ? queued : (root ? 1u : 0u);
            ctl->starving = 0u;
        }
        __threadfence();
        __syncthreads();

        SearchParams prm;
        prm = SearchParams{};
        prm.n = n;
        prm.wp = WP;
        prm.rows = gd.ren;
        prm.order = gd.order;
        prm.ctl = ctl;
        prm.seq = seq;
        prm.frames = frames;
        prm.qcap = bp.qcap;
        prm.fs = bp.fs;
        prm.out = gd.out;
        prm.timeout_ns = bp.timeout_ns;
        prm.limit_ns = bp.limit_ns;
        prm.total_groups = bp.groups_per_block;
        prm.pivot_mode = bp.pivot_mode;
        prm.stack_levels = bp.stack_levels;
        prm.split_min_p = bp.split_min_p;
        prm.split_target = bp.split_target;
        prm.tune = bp.tune;
        prm.count_root = 1;
        prm.t2_offset = bp.t2_offset;
        prm.pool_bytes = bp.pool_bytes;
        prm.t2_max_p = bp.t2_max_p;
        prm.direct_offset = bp.direct_offset;
        const uint32_t *rows = gd.ren;
        if (threadIdx.x == 0) root_key = 0u;
        __syncthreads();
        {
            unsigned mine = 0;
            for (uint32_t i = threadIdx.x; i < n * WP; i += blockDim.x) mine += (unsigned)__popc(rows[i]);
            atomicAdd(&root_key, mine);
        }
        __syncthreads();
        // (the outer loop's subproblems of more than 128 vertices are sparse and
        // alike: the size that fits their children, several side by side.
        // G(10000, 0.03): 18.5 -> 15.7 ms on the device)
        const Thresholds th = density_thresholds(root_key, n, bp.tune, bp.split_min_p, PIVOT != MCE_PIVOT_GREEDY, sub && n > 128u ? 0u : bp.cls);
        const bool direct = K == 1 && n <= 128u && bp.t2_max_p != 0u;
        PoolAt at{};
        at.rows = bp.direct_offset;
        at.hash = at.rows + kDirectRows * 4;
        at.pos = at.hash + kDirectVerts * 8;
        at.region = bp.t2_offset + (threadIdx.x >> 5) * bp.pool_bytes;
        at.lq = (uint32_t)smem_local_offset(n);
        at.hist = 0u;
        if (direct)
            direct_layout(rows, WP, gd.order, n, th.cls, reinterpret_cast<uint32_t *>(smem_raw + at.rows),
                          reinterpret_cast<uint64_t *>(smem_raw + at.hash), reinterpret_cast<uint16_t *>(smem_raw + at.pos));
        Counters cn;
        cn.diag = lq.h->diag;
        search_loop<K, PIVOT, false>(prm, rows, hist, lq, th, at, direct, cn);
        flush_counters(cn, gd.out);
        __syncthreads();
        if (threadIdx.x == 0) flush_diag(lq.h->diag, gd.out);
        for (uint32_t j = threadIdx.x; j <= n; j += blockDim.x)
            if (hist[j]) atomicAdd(reinterpret_cast<unsigned long long *>(gd.out + MCE_OUT_HIST + j), (unsigned long long)hist[j]);
        __syncthreads();
    }
}

// The result array with the root already counted: one node, internal when
// n > 0; for n = 0 the root is a leaf and the empty set is the one maximal
// clique; and an empty queue (the kernel that follows queues the root's
// children, or a part of them).  A part counts the root only when asked to.
// A non-zero status left by an earlier step (invalid input) suppresses the
// frames, so the search returns at once.
template <int D = 0>
__global__ void search_init_kernel(const SearchParams prm)
{
    const uint32_t n = prm.n;
    const unsigned tid = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned nth = gridDim.x * blockDim.x;
    const bool part = prm.part != nullptr;
    const unsigned queued = part ? prm.part_k : 0u;
    const bool root = !part || prm.count_root;
    for (unsigned i = tid; i < prm.qcap; i += nth) prm.seq[i] = i < queued ? i + 1u : i;
    for (unsigned i = tid; i < MCE_OUT_WORDS(n); i += nth) {
        if (i == MCE_OUT_STATUS) continue;  // sticky: an earlier step's error stays
        uint64_t v = 0ull;
        if (root && i == MCE_OUT_NODES) v = 1ull;
        if (root && n > 0u && i == MCE_OUT_INTERNAL) v = 1ull;
        if (root && n == 0u && (i == MCE_OUT_COUNT || i == MCE_OUT_HIST)) v = 1ull;
        if (root && n == 0u && i == MCE_OUT_HASH) v = mix64(0ull ^ mix64(0ull));
        if (i == MCE_OUT_GROUPS) v = prm.total_groups;
        prm.out[i] = v;
    }
    if (tid == 0) {
        Ctl *c = prm.ctl;
        c->head = 0u;
        c->abort = 0u;
        const bool go = queued > 0u && prm.out[MCE_OUT_STATUS] == 0ull;
        c->tail = go ? queued : 0u;
        c->pending = go ? queued : 0u;
        c->starving = prm.total_groups;  // warps without a frame: all of them
        c->pad3[0] = 0u;                 // degree sum, added by the kernel that follows
    }
}

// Root pivot for TomitaBB: the vertex of maximum degree, earliest on ties.
template <int D = 0>
__global__ void root_tomita_pivot_kernel(const uint32_t *rows, uint32_t n, uint32_t wp, unsigned *dst)
{
    __shared__ unsigned best;
    if (threadIdx.x == 0) best = 0u;
    __syncthreads();
    unsigned mine = 0u;
    for (uint32_t v = threadIdx.x; v < n; v += blockDim.x) {
        unsigned deg = 0;
        for (uint32_t w = 0; w < wp; ++w) deg += __popc(rows[(size_t)v * wp + w]);
        const unsigned key = ((deg + 1u) << 12) | (4095u - v);
        mine = key > mine ? key : mine;
    }
    atomicMax(&best, mine);
    __syncthreads();
    if (threadIdx.x == 0) *dst = n ? (4095u - (best & 4095u)) : 0u;
}

}  // namespace mce
