// Preprocessing steps of the search path on the device:
//  * input canonicalisation (Section 2: simple undirected graph) from an edge
//    list or a bitset,
//  * the maximum-degree-first ordering (Section 4.2),
//  * renumbering by position (Section 4.2, "How we use the vertex ordering").
#include <algorithm>
#include <cstdint>
#include <mutex>
#include <utility>
#include <vector>
#include <cuda_runtime.h>

#include "mce_internal.h"

namespace mce {
namespace {

constexpr unsigned FULLM = 0xffffffffu;

__device__ __forceinline__ void flag_invalid(uint64_t *out)
{
    atomicCAS(reinterpret_cast<unsigned long long *>(out + MCE_OUT_STATUS), 0ull,
              static_cast<unsigned long long>(static_cast<long long>(MCE_EINVAL)));
}

// Edge list -> symmetric bitset (rows cleared beforehand).
__global__ void edges_kernel(uint32_t n, uint64_t m, const uint32_t *__restrict__ uv, uint32_t w,
                             uint32_t *__restrict__ rows, uint64_t *out)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
        const uint32_t a = uv[2 * e], b = uv[2 * e + 1];
        if (a >= n || b >= n || a == b) {
            flag_invalid(out);
            continue;
        }
        atomicOr(rows + (size_t)a * w + (b >> 5), 1u << (b & 31));
        atomicOr(rows + (size_t)b * w + (a >> 5), 1u << (a & 31));
    }
}

// Bitset checks of one word: zero diagonal, zero bits at positions >= n,
// symmetry.
__device__ __forceinline__ bool valid_word(uint32_t n, uint32_t w, const uint32_t *rows, uint64_t idx)
{
    const uint32_t i = (uint32_t)(idx / w), j = (uint32_t)(idx % w);
    uint32_t word = rows[idx];
    if (word == 0u) return true;
    const uint32_t base = j * 32u;
    uint32_t valid = FULLM;
    if (base >= n) valid = 0u;
    else if (n - base < 32u) valid = (1u << (n - base)) - 1u;
    if (word & ~valid) return false;
    if (i >= base && i < base + 32u && ((word >> (i - base)) & 1u)) return false;
    while (word) {
        const uint32_t b = (uint32_t)__ffs(word) - 1u;
        word &= word - 1u;
        const uint32_t u = base + b;
        if (!((rows[(size_t)u * w + (i >> 5)] >> (i & 31)) & 1u)) return false;
    }
    return true;
}

__global__ void validate_kernel(uint32_t n, uint32_t w, const uint32_t *__restrict__ rows, uint64_t *out)
{
    const uint64_t total = (uint64_t)n * w;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += stride)
        if (!valid_word(n, w, rows, idx)) flag_invalid(out);
}

// Maximum-degree-first order (Section 4.2) by one block of T threads: highest
// remaining degree first, smallest label on ties.
//
// The order is sequential by definition, but most of a pick's cost is finding
// the maximum over all vertices and reading rows.  So vertices are placed in
// rounds.  A round gathers the up to 128 vertices of highest remaining degree
// (whole degree classes, by a histogram below the maximum), their 128 x 128
// adjacency bits, and lets one warp pick from them alone, four candidates a
// lane: a pick is one max-reduction and the removal of one row of bits.  It
// is the right pick as long as it beats every vertex outside, and those can
// only fall: the warp stops when the best candidate has fallen to the
// highest degree outside.  (When the highest degree alone has more than 128
// vertices, the candidates are the 128 of smallest label, and the first one
// left out is the one to beat.)  Then all degrees are lowered by the picks'
// rows at once.  G(1000, 0.3) takes 46 rounds of 22 picks, G(3000, 0.1) 97 of
// 31, a graph of up to 128 vertices one round.  What bounds it is the chain of
// picks, about 0.1 us each (max-reduction, one broadcast load, four
// subtractions), and 3 to 5 us of gathering and barriers a round.  A search of
// all vertices for one or two picks a round took, per call by events (G(n, p),
// now in brackets): n = 100 32 us (24), 300 96 (62), 500 152 (118), 1000 359
// (238), 2000 1993 (452), 3000 4369 (843; rows in L2, two dependent reads a
// round).  The pass that lowers the degrees counts them for the next round's
// classes as well: 4 % of the launch against a pass and a barrier of its own.
constexpr unsigned kOrderCand = 128;
constexpr unsigned kSmallPrepThreads = 256, kSmallPrepVerts = 128, kSmallPrepWords = 4;

struct OrderShared {
    uint32_t adj[kOrderCand][4];   // adjacency among the candidates
    uint32_t hist[2][kOrderCand];  // vertices by (base - degree), of this round and the next
    uint32_t chunk[4096 / 32];     // vertices of maximum degree by 32 labels (crowded rounds)
    uint16_t label[kOrderCand];    // the candidates
    uint16_t placed[kOrderCand];   // this round's picks
    uint32_t cands, picks, top, beat;
};

// Bit j of lane i becomes bit i of lane j.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, uint32_t lane)
{
    const uint32_t mask[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const uint32_t d = 16u >> s;
        const uint32_t y = __shfl_xor_sync(FULLM, x, (int)d);
        x = (lane & d) ? ((x & ~mask[s]) | ((y >> d) & mask[s])) : ((x & mask[s]) | ((y << d) & ~mask[s]));
    }
    return x;
}

// deg[u] = remaining degree + 1, 0 once placed (n entries in shared memory).
// Rows that are not a simple graph's (flagged by the validation) give some
// order and stay in bounds: degrees are clamped and never fall below 1.
template <unsigned T>
__device__ __forceinline__ void order_rounds(uint32_t n, uint32_t w, const uint32_t *R, uint32_t *__restrict__ order,
                                             uint16_t *deg, OrderShared &sh)
{
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    constexpr uint32_t NW = T / 32u;
    const uint32_t chunks = (n + 31u) / 32u;
    if (t == 0) sh.top = 0u;
    for (uint32_t i = t; i < 2u * kOrderCand; i += T) sh.hist[i / kOrderCand][i % kOrderCand] = 0u;
    __syncthreads();
    {
        uint32_t mx = 0u;
        for (uint32_t u = t; u < n; u += T) {
            uint32_t d = 0;
#pragma unroll 4
            for (uint32_t j = 0; j < w; ++j) d += (uint32_t)__popc(R[(size_t)u * w + j]);
            d = (d < 4095u ? d : 4095u) + 1u;
            deg[u] = (uint16_t)d;
            mx = d > mx ? d : mx;
        }
        mx = __reduce_max_sync(FULLM, mx);
        if (lane == 0) atomicMax(&sh.top, mx);
    }
    __syncthreads();
    if (t == 0) {
        sh.cands = 0u;
        sh.beat = 0u;
    }
    uint32_t base = 0u, h = 0u;  // hist[h] counts vertices by (base - degree)
    for (uint32_t done = 0; done < n;) {
        const uint32_t M = sh.top;
        // The pass that lowers the degrees also counts them for the next
        // round, by the distance from this round's maximum, which no degree
        // exceeds; counted anew where the maximum has fallen too far below it.
        if (done == 0u || base - M > kOrderCand / 2u) {
            base = M;
            for (uint32_t i = t; i < kOrderCand; i += T) sh.hist[h][i] = 0u;
            __syncthreads();
            for (uint32_t u = t; u < n; u += T) {
                const uint32_t d = deg[u];
                if (d != 0u && base - d < kOrderCand) atomicAdd(&sh.hist[h][base - d], 1u);
            }
            __syncthreads();
        }
        const uint32_t above = base - M;  // leading classes without a vertex
        // degree classes base, base - 1, ... that fit together (every warp
        // computes the same number)
        uint32_t classes;
        {
            const uint4 hc = *reinterpret_cast<const uint4 *>(&sh.hist[h][4u * lane]);
            const uint32_t s4 = hc.x + hc.y + hc.z + hc.w;
            uint32_t incl = s4;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULLM, incl, o);
                incl += (int)lane >= o ? y : 0u;
            }
            const uint32_t e = incl - s4, c0 = e + hc.x, c1 = c0 + hc.y, c2 = c1 + hc.z, c3 = c2 + hc.w;
            classes = (c0 <= kOrderCand) + (c1 <= kOrderCand) + (c2 <= kOrderCand) + (c3 <= kOrderCand);
            classes = __reduce_add_sync(FULLM, classes);
        }
        const bool whole = classes > above;
        if (whole) {
            for (uint32_t c = warp; c < chunks; c += NW) {
                const uint32_t u = c * 32u + lane, d = u < n ? deg[u] : 0u;
                const uint32_t in = __ballot_sync(FULLM, d != 0u && base - d < classes);
                if (in == 0u) continue;
                uint32_t at = 0u;
                if (lane == 0) at = atomicAdd(&sh.cands, (uint32_t)__popc(in));
                at = __shfl_sync(FULLM, at, 0) + (uint32_t)__popc(in & ((1u << lane) - 1u));
                if ((in >> lane) & 1u) sh.label[at] = (uint16_t)u;
            }
        } else {  // more than 128 vertices of the maximum degree: the smallest labels
            for (uint32_t c = warp; c < chunks; c += NW) {
                const uint32_t u = c * 32u + lane;
                const uint32_t b = __ballot_sync(FULLM, u < n && deg[u] == M);
                if (lane == 0) sh.chunk[c] = (uint32_t)__popc(b);
            }
            __syncthreads();
            for (uint32_t c = warp; c < chunks; c += NW) {
                uint32_t before = 0u;
                for (uint32_t x = lane; x < c; x += 32u) before += sh.chunk[x];
                before = __reduce_add_sync(FULLM, before);
                const uint32_t u = c * 32u + lane;
                const bool in = u < n && deg[u] == M;
                const uint32_t at = before + (uint32_t)__popc(__ballot_sync(FULLM, in) & ((1u << lane) - 1u));
                if (in && at < kOrderCand) sh.label[at] = (uint16_t)u;
                if (in && at == kOrderCand) sh.beat = (M << 12) | (4095u - u);
            }
            if (t == 0) sh.cands = kOrderCand;
        }
        __syncthreads();
        const uint32_t m = sh.cands;
        for (uint32_t i = t; i < kOrderCand; i += T) sh.hist[h ^ 1u][i] = 0u;
        // their adjacency, four rows a warp at a time (16 loads in flight)
        {
            uint32_t wd[4], sf[4];  // word and bit of this lane's columns
            bool on[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t c = lane + 32u * k;
                on[k] = c < m;
                const uint32_t u = on[k] ? sh.label[c] : 0u;
                wd[k] = u >> 5;
                sf[k] = u & 31u;
            }
            for (uint32_t r0 = warp * 4u; r0 < m; r0 += NW * 4u) {
                uint32_t x[4][4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t *row = R + (size_t)sh.label[r0 + q < m ? r0 + q : 0u] * w;
#pragma unroll
                    for (int k = 0; k < 4; ++k) x[q][k] = row[wd[k]];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t b[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) b[k] = __ballot_sync(FULLM, on[k] && ((x[q][k] >> sf[k]) & 1u));
                    if (lane == 0 && r0 + q < m)
                        *reinterpret_cast<uint4 *>(sh.adj[r0 + q]) = make_uint4(b[0], b[1], b[2], b[3]);
                }
            }
        }
        __syncthreads();
        if (warp == 0) {
            // key: degree + 1 (13 bits) | 4095 - label (12) | candidate (7)
            uint32_t key[4], open[4];  // open: 1 until the candidate is picked
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t c = lane + 32u * k;
                const uint32_t u = c < m ? sh.label[c] : 0u;
                open[k] = c < m ? 1u : 0u;
                key[k] = c < m ? ((uint32_t)deg[u] << 19) | ((4095u - u) << 7) | c : 0u;
            }
            // the (degree + 1, 4095 - label) to beat; whole classes: any
            // degree above the classes taken
            const uint32_t beat = whole ? ((base - classes < base ? base - classes : 0u) << 12) | 4095u : sh.beat;
            // (a row that is not a simple graph's can take a degree field below
            // zero: the candidate is then picked out of turn, and nothing else)
            uint32_t picks = 0u, floor_key = 0u;  // the first pick always stands
#pragma unroll 2
            for (; picks < m; ++picks) {
                const uint32_t a = key[0] > key[1] ? key[0] : key[1], b = key[2] > key[3] ? key[2] : key[3];
                const uint32_t best = __reduce_max_sync(FULLM, a > b ? a : b);
                if (best <= floor_key) break;
                floor_key = (beat << 7) | 127u;
                const uint4 row = *reinterpret_cast<const uint4 *>(sh.adj[best & 127u]);
                if (lane == 0) sh.placed[picks] = (uint16_t)(4095u - ((best >> 7) & 4095u));
                const uint32_t rw[4] = {row.x, row.y, row.z, row.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool own = key[k] == best;
                    const uint32_t lower = key[k] - (((rw[k] >> lane) & open[k]) << 19);
                    key[k] = own ? 0u : lower;
                    open[k] = own ? 0u : open[k];
                }
            }
            __syncwarp();
            for (uint32_t x = lane; x < picks; x += 32u) {
                const uint32_t u = sh.placed[x];
                order[done + x] = u;
                deg[u] = 0u;
            }
            if (lane == 0) {
                sh.picks = picks;
                sh.top = 0u;
                sh.cands = 0u;
                sh.beat = 0u;
            }
        }
        __syncthreads();
        const uint32_t picks = sh.picks;
        done += picks;
        // lower the degrees: lane j reads its pick's word for 32 vertices (four
        // such words in flight), a transposition gives lane i the picks'
        // bits of vertex i, and their population count is its loss
        uint32_t mx = 0u;
        for (uint32_t c0 = warp; c0 < chunks; c0 += NW * 4u) {
            uint32_t dec[4] = {0u, 0u, 0u, 0u};
            for (uint32_t p0 = 0; p0 < picks; p0 += 32u) {
                const bool on = p0 + lane < picks;
                const uint32_t *row = R + (size_t)sh.placed[on ? p0 + lane : 0u] * w;
                uint32_t x[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) x[q] = on && c0 + q * NW < chunks ? row[c0 + q * NW] : 0u;
#pragma unroll
                for (int q = 0; q < 4; ++q) dec[q] += (uint32_t)__popc(transpose_bits(x[q], lane));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t u = (c0 + q * NW) * 32u + lane;
                uint32_t d = u < n ? deg[u] : 0u;
                if (d != 0u) {
                    d = d > dec[q] + 1u ? d - dec[q] : 1u;
                    deg[u] = (uint16_t)d;
                    if (M - d < kOrderCand) atomicAdd(&sh.hist[h ^ 1u][M - d], 1u);
                }
                mx = d > mx ? d : mx;
            }
        }
        mx = __reduce_max_sync(FULLM, mx);
        if (lane == 0) atomicMax(&sh.top, mx);
        base = M;
        h ^= 1u;
        __syncthreads();
    }
}

// Shared memory of an ordering block: its state, the degrees, and the rows
// when they fit.
__host__ __device__ inline size_t order_fixed_bytes(uint32_t n)
{
    return (sizeof(OrderShared) + 15) / 16 * 16 + ((size_t)n * 2 + 15) / 16 * 16;
}

template <unsigned T>
__device__ __forceinline__ void order_block(uint32_t n, uint32_t w, const uint32_t *__restrict__ rows,
                                            uint32_t *__restrict__ order, bool rows_in_smem, unsigned char *sm)
{
    OrderShared &sh = *reinterpret_cast<OrderShared *>(sm);
    uint16_t *deg = reinterpret_cast<uint16_t *>(sm + (sizeof(OrderShared) + 15) / 16 * 16);
    if (rows_in_smem) {
        uint32_t *srows = reinterpret_cast<uint32_t *>(sm + order_fixed_bytes(n));
#pragma unroll 8
        for (uint32_t i = threadIdx.x; i < n * w; i += T) srows[i] = rows[i];
        __syncthreads();
        order_rounds<T>(n, w, srows, order, deg, sh);
    } else {
        order_rounds<T>(n, w, rows, order, deg, sh);
    }
}

template <unsigned T>
__global__ void __launch_bounds__(T) order_kernel(uint32_t n, uint32_t w, const uint32_t *__restrict__ rows,
                                                  uint32_t *__restrict__ order, int rows_in_smem)
{
    extern __shared__ __align__(16) unsigned char osm[];
    order_block<T>(n, w, rows, order, rows_in_smem != 0, osm);
}

// Everything before the search of a graph of at most 128 vertices, by one
// block: validation, the order, the renumbered rows, the result array and the
// queue as the search starts from them (the root counted, its children's
// frames queued; nothing queued for rows that are not a simple graph's).  As
// separate launches these were seven short kernels in a row, some 20 us of
// launch gaps and of global memory written and read back: G(45, 0.5) 62 us
// from rows to result, now 50; G(100, 0.5) 145 and 137.  TomitaBB's root
// pivot is position 0, too: the order's first vertex has the largest degree.
__global__ void __launch_bounds__(kSmallPrepThreads) small_prep_kernel(const SearchParams prm, uint32_t w,
                                                                       const uint32_t *__restrict__ rows_in,
                                                                       uint32_t *order, uint32_t *rows)
{
    extern __shared__ __align__(16) unsigned char osm[];
    __shared__ uint32_t so[kSmallPrepVerts], nrows[kSmallPrepVerts * kSmallPrepWords], bad, degrees;
    OrderShared &sh = *reinterpret_cast<OrderShared *>(osm);
    uint16_t *deg = reinterpret_cast<uint16_t *>(osm + (sizeof(OrderShared) + 15) / 16 * 16);
    uint32_t *srows = reinterpret_cast<uint32_t *>(osm + order_fixed_bytes(prm.n));
    const uint32_t n = prm.n, wp = prm.wp, t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    constexpr uint32_t T = kSmallPrepThreads;
    if (t == 0) bad = degrees = 0u;
    for (uint32_t i = t; i < n * w; i += T) srows[i] = rows_in[i];
    // the ticket words past the queued frames
    for (uint32_t i = t; i < prm.qcap; i += T)
        if (i >= kSmallPrepVerts) prm.seq[i] = i;
    __syncthreads();
    for (uint32_t i = t; i < n * w; i += T)
        if (!valid_word(n, w, srows, i)) bad = 1u;
    order_rounds<T>(n, w, srows, order, deg, sh);
    for (uint32_t i = t; i < n; i += T) so[i] = order[i];
    __syncthreads();
    for (uint32_t x = warp; x < n * wp; x += T / 32u) {
        const uint32_t i = x / wp, j = x % wp * 32u + lane;
        bool bit = false;
        if (j < n) {
            const uint32_t col = so[j];
            bit = (srows[so[i] * w + (col >> 5)] >> (col & 31u)) & 1u;
        }
        const uint32_t word = __ballot_sync(FULLM, bit);
        if (lane == 0) {
            rows[x] = word;
            nrows[x] = word;
        }
    }
    __syncthreads();
    uint32_t sum = 0u;
    for (uint32_t x = t; x < n * wp; x += T) sum += (uint32_t)__popc(nrows[x]);
    sum = __reduce_add_sync(FULLM, sum);
    if (lane == 0 && sum != 0u) atomicAdd(&degrees, sum);
    __syncthreads();
    // L = V \ N(position 0): child k branches on its k-th vertex v, the ones
    // before in X
    const bool go = bad == 0u;
    auto all_of = [&](uint32_t q) -> uint32_t { return n >= q * 32u + 32u ? FULLM : (n > q * 32u ? (1u << (n - q * 32u)) - 1u : 0u); };
    uint32_t c = 0u;
    for (uint32_t q = 0; q < wp; ++q) c += (uint32_t)__popc(all_of(q) & ~nrows[q]);
    for (uint32_t k = t; k < kSmallPrepVerts && k < prm.qcap; k += T) prm.seq[k] = go && k < c ? k + 1u : k;
    for (uint32_t k = t; k < c && go; k += T) {
        uint32_t v = 0u;
        for (uint32_t q = 0, before = 0; q < wp; ++q) {
            uint32_t l = all_of(q) & ~nrows[q];
            const uint32_t here = (uint32_t)__popc(l);
            if (k >= before && k < before + here) {
                for (uint32_t r = k - before; r > 0u; --r) l &= l - 1u;
                v = q * 32u + (uint32_t)__ffs(l) - 1u;
            }
            before += here;
        }
        uint32_t *fr = prm.frames + (size_t)k * prm.fs;
        for (uint32_t q = 0; q < wp; ++q) {
            const uint32_t below = v >= q * 32u + 32u ? FULLM : (v > q * 32u ? (1u << (v - q * 32u)) - 1u : 0u);
            const uint32_t X = all_of(q) & ~nrows[q] & below;
            fr[kFrameHdr + q] = all_of(q) & ~X;
            fr[kFrameHdr + wp + q] = X;
            if (prm.lst.rec) fr[kFrameHdr + 2u * wp + q] = 0u;
        }
        fr[0] = (v + 1u) << 16;
        fr[1] = fr[2] = fr[3] = fr[4] = 0u;
    }
    for (uint32_t i = t; i < MCE_OUT_WORDS(n); i += T) {
        uint64_t x = 0ull;
        if (i == MCE_OUT_NODES || i == MCE_OUT_INTERNAL) x = 1ull;
        if (i == MCE_OUT_GROUPS) x = prm.total_groups;
        if (i == MCE_OUT_STATUS && !go) x = static_cast<uint64_t>(static_cast<int64_t>(MCE_EINVAL));
        prm.out[i] = x;
    }
    if (t == 0) {
        Ctl *ctl = prm.ctl;
        ctl->head = 0u;
        ctl->abort = 0u;
        ctl->tail = ctl->pending = go ? c : 0u;
        ctl->starving = prm.total_groups;
        ctl->pad3[0] = degrees;
    }
}

// One block per graph of a batch; the rows go to shared memory when they fit
// in the launch's dynamic shared memory.
__global__ void __launch_bounds__(256) order_batch_kernel(const BatchGraph *__restrict__ graphs, size_t smem_bytes)
{
    extern __shared__ __align__(16) unsigned char osm[];
    const BatchGraph gd = graphs[blockIdx.x];
    const size_t need = order_fixed_bytes(gd.n) + (size_t)gd.n * gd.w * 4;
    order_block<256>(gd.n, gd.w, gd.rows, gd.order, need <= smem_bytes, osm);
}

__global__ void identity_kernel(uint32_t n, uint32_t *order)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) order[i] = i;
}

// A'[i][j] = A[order[i]][order[j]]: one warp per output word, each lane
// fetching one bit and a ballot assembling the word.
__global__ void renumber_kernel(uint32_t n, uint32_t w, const uint32_t *__restrict__ rows,
                                const uint32_t *__restrict__ order, uint32_t wout, uint32_t *__restrict__ out)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t total = (uint64_t)n * wout;
    const uint64_t nwarps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t t = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < total; t += nwarps) {
        const uint32_t i = (uint32_t)(t / wout), jw = (uint32_t)(t % wout);
        const uint32_t j = jw * 32u + lane;
        bool bit = false;
        if (j < n) {
            const uint32_t src = __ldg(order + i), col = __ldg(order + j);
            bit = (__ldg(rows + (size_t)src * w + (col >> 5)) >> (col & 31)) & 1u;
        }
        const uint32_t word = __ballot_sync(FULLM, bit);
        if (lane == 0) out[t] = word;
    }
}

// Renumbering for a batch: blockIdx.y selects the graph, the block's warps
// stride over its output words.
__global__ void renumber_batch_kernel(const BatchGraph *__restrict__ graphs)
{
    const BatchGraph gd = graphs[blockIdx.y];
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t total = (uint64_t)gd.n * gd.wp;
    const uint64_t nwarps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    for (uint64_t t = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < total; t += nwarps) {
        const uint32_t i = (uint32_t)(t / gd.wp), jw = (uint32_t)(t % gd.wp);
        const uint32_t j = jw * 32u + lane;
        bool bit = false;
        if (j < gd.n) {
            const uint32_t src = gd.order[i], col = gd.order[j];
            bit = (__ldg(gd.rows + (size_t)src * gd.w + (col >> 5)) >> (col & 31)) & 1u;
        }
        const uint32_t word = __ballot_sync(FULLM, bit);
        if (lane == 0) gd.ren[t] = word;
    }
}

unsigned grid_for(uint64_t work, unsigned threads)
{
    uint64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 65535u) g = 65535u;
    return (unsigned)g;
}

}  // namespace

cudaError_t launch_edges_to_rows(uint32_t n, uint64_t m, const uint32_t *uv, uint32_t w, uint32_t *rows,
                                 uint64_t *out, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(rows, 0, (size_t)n * w * 4, s);
    if (e != cudaSuccess || m == 0) return e;
    edges_kernel<<<grid_for(m, 256), 256, 0, s>>>(n, m, uv, w, rows, out);
    return cudaGetLastError();
}

cudaError_t launch_validate_rows(uint32_t n, uint32_t w, const uint32_t *rows, uint64_t *out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    validate_kernel<<<grid_for((uint64_t)n * w, 256), 256, 0, s>>>(n, w, rows, out);
    return cudaGetLastError();
}

cudaError_t launch_order(uint32_t n, uint32_t w, const uint32_t *rows, uint32_t *order, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    // rows in shared memory up to 200 KB; 512 threads, fewer where barriers
    // cost more than they save (256 / 512 / 1024 threads, us by events: n = 500
    // 116 / 118 / 124, 1000 245 / 238 / 265, 2000 521 / 452 / 519, 3000 952 / 843 /
    // 915; 512 / 1024: 4096 1346 / 1443)
    const size_t fixed = order_fixed_bytes(n), rbytes = (size_t)n * w * 4;
    const int in_smem = fixed + rbytes <= 200u * 1024u;
    const size_t smem = fixed + (in_smem ? rbytes : 0);
    const unsigned threads = n <= 128 ? 128u : 512u;
    void (*f)(uint32_t, uint32_t, const uint32_t *, uint32_t *, int) = n <= 128 ? order_kernel<128> : order_kernel<512>;
    cudaError_t e = kernel_smem_setup((const void *)f);
    if (e != cudaSuccess) return e;
    f<<<1, threads, smem, s>>>(n, w, rows, order, in_smem);
    return cudaGetLastError();
}

bool small_prep_fits(uint32_t n, uint32_t w, uint32_t wp)
{
    return n >= 1u && n <= kSmallPrepVerts && wp <= kSmallPrepWords && order_fixed_bytes(n) + (size_t)n * w * 4 <= 40u * 1024u;
}

cudaError_t launch_small_prep(const SearchParams &prm, uint32_t w, const uint32_t *rows_in, uint32_t *order,
                              uint32_t *rows, cudaStream_t s)
{
    small_prep_kernel<<<1, kSmallPrepThreads, order_fixed_bytes(prm.n) + (size_t)prm.n * w * 4, s>>>(prm, w, rows_in,
                                                                                                order, rows);
    return cudaGetLastError();
}

cudaError_t launch_identity(uint32_t n, uint32_t *order, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    identity_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, order);
    return cudaGetLastError();
}

cudaError_t launch_renumber(uint32_t n, uint32_t w, const uint32_t *rows, const uint32_t *order, uint32_t wout,
                            uint32_t *rows_out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const uint64_t warps = (uint64_t)n * wout;
    renumber_kernel<<<grid_for(warps * 32, 256), 256, 0, s>>>(n, w, rows, order, wout, rows_out);
    return cudaGetLastError();
}


cudaError_t kernel_smem_setup(const void *func, bool prefer_l1)
{
    constexpr int kMaxDev = 64;
    static std::mutex mu;
    static std::vector<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    for (const auto &d : done)
        if (d.first == func && d.second == dev) return cudaSuccess;
    int optin = 0;
    cudaFuncAttributes fa{};
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, func);
    if (e == cudaSuccess)  // static shared memory counts against the same limit
        e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess && !prefer_l1)
        e = cudaFuncSetAttribute(func, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && (int)done.size() < kMaxDev * 256) done.emplace_back(func, dev);
    return e;
}

cudaError_t prepare_order_batch(uint32_t max_n, uint32_t max_w, size_t *smem)
{
    const size_t fixed = order_fixed_bytes(max_n), rbytes = (size_t)max_n * max_w * 4;
    *smem = fixed + (fixed + rbytes <= 200u * 1024u ? rbytes : 0);
    return kernel_smem_setup((const void *)order_batch_kernel);
}

cudaError_t launch_order_batch(const BatchGraph *graphs, uint32_t count, size_t smem, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    order_batch_kernel<<<count, 256, smem, s>>>(graphs, smem);
    return cudaGetLastError();
}

cudaError_t launch_renumber_batch(const BatchGraph *graphs, uint32_t count, uint32_t max_n, uint32_t max_wp,
                                  cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    const uint64_t warps = (uint64_t)max_n * max_wp;
    unsigned gx = (unsigned)std::min<uint64_t>((warps + 7) / 8, 1024);
    if (gx == 0) gx = 1;
    renumber_batch_kernel<<<dim3(gx, count), 256, 0, s>>>(graphs);
    return cudaGetLastError();
}

}  // namespace mce
