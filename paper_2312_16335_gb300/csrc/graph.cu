// Graph construction on the primary vectors (App. A: search + prune for every node;
// App. D: Vamana with R, L, alpha), batch-synchronous and bit-reproducible:
//   1. beam search of every batch node on the graph as it was at the batch start
//      (beam_kernel in build mode, exact integer-core pair scores);
//   2. RobustPrune of pool = beam u old out-list (one CTA per node, pool records
//      staged in shared memory);
//   3. the batch's out-lists are replaced;
//   4. reverse edges grouped by target with a count / scan / scatter pass, each
//      target's sources sorted ascending, appended, and the target pruned if it
//      exceeds R.
#include <cuda_runtime.h>

#include <cstring>
#include <vector>

#include "beam.cuh"
#include "common.cuh"
#include "index.cuh"

namespace lv {

// -------------------------------------------------------------------- helpers
static inline float host_fsub(float a, float b) { return a - b; }  // IEEE float32 (host SSE/NEON)
__host__ __device__ __forceinline__ uint64_t splitmix(uint64_t seed, uint64_t a, uint64_t b) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ULL * (1ULL + (a << 32) + b);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

__device__ __forceinline__ bool entry_better(float ga, int ia, float gb, int ib) {
    if (isnan(ga)) return false;
    if (isnan(gb)) return true;
    return ga > gb || (ga == gb && ia < ib);
}

// Remove out-of-range and repeated ids of every row (first occurrence kept).
__global__ void graph_sanitize_kernel(int32_t *g, int64_t n, int R, int *status) {
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    int32_t *row = g + v * R;
    for (int s = 0; s < R; ++s) {
        int32_t u = row[s];
        if (u < -1 || u >= n) {
            atomicOr(status, ST_CORRUPT);
            row[s] = -1;
            continue;
        }
        if (u < 0) continue;
        for (int t = 0; t < s; ++t)
            if (row[t] == u) {
                row[s] = -1;
                break;
            }
    }
}

// argmax_i G_i (ties -> smaller id): G is the third float of the record constants; with the L2
// metric argmax_i 2 G_i - N_i (the primary nearest the mean; N = first float of the second chunk).
__global__ void entry_partial_kernel(const uint8_t *rec, int64_t n, int64_t stride, int cb, int metric, float *bg,
                                     int *bi) {
    __shared__ float sg[256];
    __shared__ int si[256];
    float best = -INFINITY;
    int bid = 0x7fffffff;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float gv = *reinterpret_cast<const float *>(rec + i * stride + cb + 8);
        if (metric) gv = __fsub_rn(__fmul_rn(2.0f, gv), *reinterpret_cast<const float *>(rec + i * stride + cb + 16));
        if (entry_better(gv, (int)i, best, bid) || bid == 0x7fffffff) {
            if (!isnan(gv) || bid == 0x7fffffff) {
                best = isnan(gv) ? -INFINITY : gv;
                bid = (int)i;
            }
        }
    }
    sg[threadIdx.x] = best;
    si[threadIdx.x] = bid;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o && entry_better(sg[threadIdx.x + o], si[threadIdx.x + o], sg[threadIdx.x], si[threadIdx.x])) {
            sg[threadIdx.x] = sg[threadIdx.x + o];
            si[threadIdx.x] = si[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        bg[blockIdx.x] = sg[0];
        bi[blockIdx.x] = si[0];
    }
}

__global__ void entry_final_kernel(const float *bg, const int *bi, int nb, int32_t *out) {
    __shared__ float sg[256];
    __shared__ int si[256];
    float best = -INFINITY;
    int bid = 0x7fffffff;
    for (int t = threadIdx.x; t < nb; t += blockDim.x)
        if (entry_better(bg[t], bi[t], best, bid)) {
            best = bg[t];
            bid = bi[t];
        }
    sg[threadIdx.x] = best;
    si[threadIdx.x] = bid;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o && entry_better(sg[threadIdx.x + o], si[threadIdx.x + o], sg[threadIdx.x], si[threadIdx.x])) {
            sg[threadIdx.x] = sg[threadIdx.x + o];
            si[threadIdx.x] = si[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = si[0] == 0x7fffffff ? 0 : si[0];
}

// Initial graph: node v keeps the first min(R, n-1) draws splitmix(seed, v, j) mod n
// that are neither v nor repeated.  One warp per node, 32 draws at a time, the row in shared memory (a
// thread per node, which searched and filled its row in global memory: 200,000 x 64 in 1.63 ms, 0.11 ms now).
constexpr int RG_WARPS = 8;
__global__ void __launch_bounds__(32 * RG_WARPS) random_graph_kernel(int32_t *g, int64_t n, int R, uint64_t seed,
                                                                     int *status) {
    __shared__ int32_t s_row[RG_WARPS][RMAX];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t v = (int64_t)blockIdx.x * RG_WARPS + wid;
    if (v >= n) return;  // whole warps
    int32_t *const row = s_row[wid];
    const int want = (int)((n - 1) < R ? (n - 1) : R);
    int cnt = 0;
    const uint64_t limit = 1ull << 24;
    for (uint64_t j = 0; cnt < want; j += 32) {
        if (j >= limit) {
            if (lane == 0) atomicOr(status, ST_TIMEOUT);
            break;
        }
        const int32_t u = (int32_t)(splitmix(seed, (uint64_t)v, j + lane) % (uint64_t)n);
        const unsigned same = __match_any_sync(FULL, u);  // every lane takes part, the node itself drawn or not
        bool keep = u != v && (same & ((1u << lane) - 1u)) == 0u;  // first of its kind here
        for (int t = 0; t < cnt; ++t) keep &= row[t] != u;
        const unsigned bal = __ballot_sync(FULL, keep);
        const int pos = cnt + __popc(bal & ((1u << lane) - 1u));
        if (keep && pos < want) row[pos] = u;
        cnt = min(want, cnt + __popc(bal));
        __syncwarp();
    }
    for (int t = lane; t < R; t += 32) g[v * R + t] = t < cnt ? row[t] : -1;
}

// --------------------------------------------------------------- RobustPrune
// Pair score of two records held in shared memory (exact build score; L2: -||y_a - y_b||^2).
template <int BITS, bool L2>
__device__ __forceinline__ float smem_pair_score(const uint8_t *ra, const uint8_t *rb, int CH, int cb, float mu2,
                                                 float fdim) {
    int P = 0;
    for (int c = 0; c < CH; ++c)
        P += code_dot<BITS>(*reinterpret_cast<const uint4 *>(ra + 16 * c), *reinterpret_cast<const uint4 *>(rb + 16 * c));
    const float4 ka = *reinterpret_cast<const float4 *>(ra + cb);
    const float4 kb = *reinterpret_cast<const float4 *>(rb + cb);
    const float ip = build_pair_score(mu2, fdim, ka.x, ka.y, ka.z, ka.w, kb.x, kb.y, kb.z, kb.w, P);
    if (!L2) return ip;
    return l2_from_ip(ip, *reinterpret_cast<const float *>(ra + cb + 16), *reinterpret_cast<const float *>(rb + cb + 16));
}

// The same score by four lanes (g = lane mod 4), each with every fourth chunk; every lane of the group
// gets it.  All 32 lanes take part.
template <int BITS, bool L2>
__device__ __forceinline__ float smem_pair_score4(const uint8_t *ra, const uint8_t *rb, int g, int CH, int cb, float mu2,
                                                  float fdim) {
    int P = 0;
#pragma unroll 4
    for (int c = g; c < CH; c += 4)
        P += code_dot<BITS>(*reinterpret_cast<const uint4 *>(ra + 16 * c), *reinterpret_cast<const uint4 *>(rb + 16 * c));
    P += __shfl_xor_sync(FULL, P, 1);
    P += __shfl_xor_sync(FULL, P, 2);
    const float4 ka = *reinterpret_cast<const float4 *>(ra + cb);
    const float4 kb = *reinterpret_cast<const float4 *>(rb + cb);
    const float ip = build_pair_score(mu2, fdim, ka.x, ka.y, ka.z, ka.w, kb.x, kb.y, kb.z, kb.w, P);
    if (!L2) return ip;
    return l2_from_ip(ip, *reinterpret_cast<const float *>(ra + cb + 16), *reinterpret_cast<const float *>(rb + cb + 16));
}

struct PruneParams {
    const uint8_t *prim;
    int64_t stride;  // record stride (multiple of 32)
    int CH, cb, dim;
    float mu2, alpha, shift;
    int metric;  // 1: L2 pair scores -||y_a - y_b||^2
    int R, PMAX;
    int slot;  // shared bytes of a staged record (see prune_slot)
    int64_t n;
    int32_t *graph;        // n x R
    // mode 0: batch nodes
    const int32_t *nodes;  // perm + b0
    const int32_t *beams;  // nb x Lb, best first, -1 at the end
    const float *bscores;  // nb x Lb: the beams' build scores
    int Lb;
    int32_t *newl;         // nb x R
    // mode 1: reverse edges; targets whose new sources number lo < .. <= hi
    const int64_t *offs;   // n + 1 exclusive scan (hi: sources, lo: touched count)
    const int32_t *srcs;
    const int32_t *touched;
    const int64_t *total;  // lo 32 bits: number of touched targets
    int lo, hi;
    int *status;
};

// an unsigned key that orders like the score (-0 and 0 alike), and back
__device__ __forceinline__ unsigned score_key(float s) {
    const unsigned u = __float_as_uint(s + 0.0f);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float key_score(unsigned k) {
    return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}
// (score, id) in one word: the larger the better, ties by the smaller id; NaN as -infinity, as in the beam
__device__ __forceinline__ unsigned long long pool_key(float s, int id) {
    return (unsigned long long)score_key(fmaxf(s, -INFINITY)) << 32 | (unsigned)~id;
}

// Writes the values of the block's kept threads, in thread order, to dst[base ..) while they fit below
// cap; returns base + their number.  wcnt: one int per warp.  Every thread of the block calls it.
template <int NT>
__device__ __forceinline__ int block_append(bool keep, int value, int *dst, int base, int cap, int *wcnt) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned bal = __ballot_sync(FULL, keep);
    __syncthreads();
    if (lane == 0) wcnt[wid] = __popc(bal);
    __syncthreads();
    int pos = base + __popc(bal & ((1u << lane) - 1u)), all = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        if (w < wid) pos += wcnt[w];
        all += wcnt[w];
    }
    if (keep && pos < cap) dst[pos] = value;
    return base + all;
}

// MODE 0: pool = beam (minus p) u old out-list of p; output to newl[t].
// MODE 1: pool = current out-list of u + its new sources (ascending, not present);
//         pruned only when it exceeds R; output to graph[u].
// One block per node.  The pool's records are staged in shared memory by 16-byte asynchronous
// copies; ranks put the pool in order (score desc, id asc); then the kept members are taken one by
// one, each striking out the members of the rest that it covers.  Bound by the latency of that
// chain (one barrier per kept member) and by the shared-memory reads of the pair scores, so nothing
// in it is serial over the pool: lists are compacted by ballots, the beam's part of the pool comes
// with its scores and its order from the search (only the old neighbours are scored and merged in),
// and the members still standing are bits of ballot words in rank order, one thread per member.
// Two passes over 200,000 nodes of 160 codes (R = 64, L_build = 128): 30.4 -> 8.8 ms (mode 0) and 18.1
// -> 6.1 ms (mode 1) against lists walked by one thread and the whole pool ranked and rescored; over
// 50,000 nodes of 768 codes, four lanes per record: 41.6 -> 13.3 ms and 10.4 -> 5.2 ms (a thread per
// record: 23.1 and 5.4 ms).
template <int BITS, int MODE, bool L2, bool LONG, int NT>
__global__ void __launch_bounds__(NT) prune_kernel(const PruneParams pp) {
    constexpr int POOL = MODE == 0 ? LCAP_MAX + RMAX : 4 * RMAX + 256;  // the largest PMAX
    constexpr int E = (POOL + NT - 1) / NT;                             // pool members of a lane
    constexpr int WORDS = E * NT / 32;
    static_assert(WORDS <= 32, "a lane reads one word");
    extern __shared__ __align__(16) unsigned char sm[];
    uint8_t *const recs = sm;                                                            // PMAX records
    uint8_t *const prec = recs + (size_t)pp.PMAX * pp.slot;                              // own record
    unsigned long long *const key = reinterpret_cast<unsigned long long *>(prec + pp.slot);  // PMAX keys
    int *const pid = reinterpret_cast<int *>(key + pp.PMAX);                             // PMAX ids
    unsigned short *const ord = reinterpret_cast<unsigned short *>(pid + pp.PMAX);       // PMAX: rank -> member
    __shared__ int s_out[RMAX], s_wcnt[NT / 32], s_np, s_self;
    __shared__ unsigned s_mask[2][WORDS];
    __shared__ unsigned char s_list[NT / 32][32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

    int64_t p;
    int32_t *dst;
    if (MODE == 0) {
        p = pp.nodes[blockIdx.x];
        dst = pp.newl + (int64_t)blockIdx.x * pp.R;
    } else {
        if ((int64_t)blockIdx.x >= (*pp.total & 0xffffffff)) return;
        p = pp.touched[blockIdx.x];
        dst = pp.graph + p * pp.R;
    }
    const int32_t *old = pp.graph + p * pp.R;

    // records [from, to) of the pool (to == np + 1: and p's own) in 16-byte chunks, 16 or 32 lanes a record
    const int chunks = (pp.cb + (L2 ? 32 : 16)) / 16;
    auto stage = [&](int from, int to, bool own) {
        const int g = chunks <= 16 ? 16 : 32;
        for (int r = from + tid / g; r < to + (own ? 1 : 0); r += NT / g) {
            const uint8_t *src = pp.prim + (r < to ? (int64_t)pid[r] : p) * pp.stride;
            const uint8_t *d = r < to ? recs + (size_t)r * pp.slot : prec;
            for (int c = tid & (g - 1); c < chunks; c += g)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(d + 16 * c)),
                             "l"(src + 16 * c)
                             : "memory");
        }
    };

    // ---- gather the pool: members [0, n0) come sorted and scored (mode 0: the beam) ----
    int np, n0 = 0;
    if (MODE == 0) {
        // beam members except p (distinct), then old neighbours not in the beam
        const int32_t *beam = pp.beams + (int64_t)blockIdx.x * pp.Lb;
        const float *bsc = pp.bscores + (int64_t)blockIdx.x * pp.Lb;
        if (tid == 0) {
            s_np = 0;
            s_self = 0x7fffffff;
        }
        __syncthreads();
        for (int t = tid; t < pp.Lb; t += NT) {
            const int u = beam[t];
            if (u >= 0 && (t + 1 == pp.Lb || beam[t + 1] < 0)) s_np = t + 1;
            if (u == p) s_self = t;
        }
        __syncthreads();
        const int nb = s_np, self = s_self;
        n0 = nb - (self < nb ? 1 : 0);
        for (int t = tid; t < nb; t += NT) {
            if (t == self) continue;
            const int u = beam[t], o = t - (t > self ? 1 : 0);
            pid[o] = u;
            key[o] = pool_key(bsc[t], u);
        }
        __syncthreads();
        if (tid == 0) s_np = n0;
        stage(0, n0, false);
        // four threads look for each old neighbour in the beam
        __syncthreads();
        for (int s0 = 0; s0 < pp.R; s0 += NT / 4) {
            const int s = s0 + (tid >> 2);
            const int u = s < pp.R ? old[s] : -1;
            unsigned in = 0;
            if (u >= 0)
                for (int t = tid & 3; t < n0; t += 4) in |= pid[t] == u ? 1u : 0u;
            in |= __shfl_xor_sync(FULL, in, 1);
            in |= __shfl_xor_sync(FULL, in, 2);
            if ((tid & 3) == 0 && u >= 0 && u != p && !in) pid[atomicAdd(&s_np, 1)] = u;
        }
        __syncthreads();
        np = s_np;
        stage(n0, np, true);
    } else {
        const int64_t o0 = pp.offs[p] >> 32, o1 = pp.offs[p + 1] >> 32;
        const int nsrc = (int)(o1 - o0);
        if (nsrc <= pp.lo || nsrc > pp.hi) return;  // the whole block: another launch's
        // current list (compacted)
        int nl = 0;
        for (int s0 = 0; s0 < pp.R; s0 += NT) {
            const int s = s0 + tid, u = s < pp.R ? old[s] : -1;
            nl = block_append<NT>(u >= 0, u, pid, nl, pp.PMAX, s_wcnt);
        }
        // the sources ascending (ranks; they are distinct), without those present
        if (nsrc > pp.PMAX && tid == 0) atomicOr(pp.status, ST_CAPACITY);
        int *const tmp = reinterpret_cast<int *>(key);  // PMAX ids by rank
        int *const src = tmp + pp.PMAX;                 // the sources, when they fit
        const bool fit = nsrc <= pp.PMAX;
        for (int t = tid; fit && t < nsrc; t += NT) src[t] = pp.srcs[o0 + t];
        __syncthreads();
        for (int t = tid; t < nsrc; t += NT) {
            const int s = fit ? src[t] : pp.srcs[o0 + t];
            int rank = 0;
            for (int w = 0; w < nsrc; ++w) rank += (fit ? src[w] : pp.srcs[o0 + w]) < s ? 1 : 0;
            bool keep = s != p;
            for (int w = 0; w < nl; ++w) keep &= pid[w] != s;
            if (rank < pp.PMAX) tmp[rank] = keep ? s : -1;
        }
        __syncthreads();
        np = nl;
        for (int t0 = 0; t0 < min(nsrc, pp.PMAX); t0 += NT) {
            const int t = t0 + tid, s = t < min(nsrc, pp.PMAX) ? tmp[t] : -1;
            np = block_append<NT>(s >= 0, s, pid, np, pp.PMAX, s_wcnt);
        }
        __syncthreads();
        if (np > pp.PMAX) {
            if (tid == 0) atomicOr(pp.status, ST_CAPACITY);
            np = pp.PMAX;
        }
        if (np <= pp.R) {
            for (int s = tid; s < pp.R; s += NT) dst[s] = s < np ? pid[s] : -1;
            return;
        }
        stage(0, np, true);
    }

    // ---- score the rest, order by (score desc, id asc) ----
    for (int i = tid; i < np; i += NT) ord[i] = (unsigned short)i;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const float fdim = (float)pp.dim;
    if constexpr (LONG) {
        for (int i0 = n0; i0 < np; i0 += NT / 4) {  // whole warps
            const int i = i0 + (tid >> 2), j = min(i, np - 1);
            const float f = smem_pair_score4<BITS, L2>(prec, recs + (size_t)j * pp.slot, tid & 3, pp.CH, pp.cb, pp.mu2, fdim);
            if (i < np && (tid & 3) == 0) key[i] = pool_key(f, pid[i]);
        }
    } else {
        for (int i = n0 + tid; i < np; i += NT)
            key[i] = pool_key(smem_pair_score<BITS, L2>(prec, recs + (size_t)i * pp.slot, pp.CH, pp.cb, pp.mu2, fdim), pid[i]);
    }
    __syncthreads();
    for (int i = tid; i < np; i += NT) {
        const unsigned long long k = key[i];
        int rank = 0;
        if (i < n0) {
            rank = i;
        } else {  // sorted members ahead of it
            int hi = n0;
            while (rank < hi) {
                const int mid = (rank + hi) >> 1;
                if (key[mid] > k)
                    rank = mid + 1;
                else
                    hi = mid;
            }
        }
#pragma unroll 4
        for (int t = n0; t < np; ++t) rank += key[t] > k ? 1 : 0;
        ord[rank] = (unsigned short)i;
    }
    __syncthreads();
    // ---- greedy selection: word e of a warp holds the members of ranks NT e + 32 wid .. + 31 ----
    int mine[E];         // lane's member
    unsigned word[E];    // members of the warp still standing (the same in every lane)
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int q = tid + NT * e;
        mine[e] = q < np ? ord[q] : 0;
        word[e] = __ballot_sync(FULL, q < np);
    }
    int nsel = 0, cur = 0;
    for (int buf = 0; cur < np; buf ^= 1) {
        const int i = ord[cur];
        if (tid == 0) s_out[nsel] = pid[i];
        if (++nsel >= pp.R) break;
        const uint8_t *ri = recs + (size_t)i * pp.slot;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (NT * e >= np) break;
            const int first = NT * e + 32 * wid;
            unsigned m = word[e];  // those after the member taken
            if (first + 31 <= cur)
                m = 0;
            else if (first <= cur)
                m &= ~((2u << (cur - first)) - 1u);
            auto covered = [&](int j, float s) {
                return __fmul_rn(pp.alpha, s) >= __fadd_rn(key_score((unsigned)(key[j] >> 32)), pp.shift);
            };
            if constexpr (LONG) {  // eight members at a time, four lanes each
                const int cnt = __popc(m);
                if (m >> lane & 1u) s_list[wid][__popc(m & ((1u << lane) - 1u))] = (unsigned char)lane;
                __syncwarp();
                for (int b = 0; b < cnt; b += 8) {
                    const int src = s_list[wid][min(b + (lane >> 2), cnt - 1)];
                    const int j = __shfl_sync(FULL, mine[e], src);
                    const float s = smem_pair_score4<BITS, L2>(ri, recs + (size_t)j * pp.slot, lane & 3, pp.CH, pp.cb,
                                                               pp.mu2, fdim);
                    m &= ~__reduce_or_sync(FULL, covered(j, s) ? 1u << src : 0u);
                }
                __syncwarp();  // the list is read before the next one is written
            } else {  // a thread each
                bool a = m >> lane & 1u;
                if (a) {
                    const int j = mine[e];
                    a = !covered(j, smem_pair_score<BITS, L2>(ri, recs + (size_t)j * pp.slot, pp.CH, pp.cb, pp.mu2, fdim));
                }
                m = __ballot_sync(FULL, a);
            }
            word[e] = m;
            if (lane == 0) s_mask[buf][e * (NT / 32) + wid] = m;
        }
        __syncthreads();  // the words of the other buffer are read before it is written again
        // the next member standing: the lowest bit of the words
        const unsigned w = lane < (np + 31) / 32 ? s_mask[buf][lane] : 0u;
        const unsigned nz = __ballot_sync(FULL, w != 0u);
        if (nz == 0u) break;
        const int wi = __ffs(nz) - 1;
        cur = 32 * wi + __ffs(__shfl_sync(FULL, w, wi)) - 1;
    }
    __syncthreads();
    for (int s = tid; s < pp.R; s += NT) dst[s] = s < nsel ? s_out[s] : -1;
}

__global__ void scatter_rows_kernel(const int32_t *newl, const int32_t *nodes, int nb, int R, int32_t *graph) {
    const int t = blockIdx.x;
    if (t >= nb) return;
    const int64_t p = nodes[t];
    for (int s = threadIdx.x; s < R; s += blockDim.x) graph[p * R + s] = newl[(int64_t)t * R + s];
}

__global__ void count_pairs_kernel(const int32_t *newl, int64_t total, int *cnt) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    int u = newl[i];
    if (u >= 0) atomicAdd(cnt + u, 1);
}

__global__ void scatter_pairs_kernel(const int32_t *newl, const int32_t *nodes, int nb, int R, const int64_t *offs,
                                     int *cnt, int32_t *srcs) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)nb * R) return;
    int u = newl[i];
    if (u < 0) return;
    const int t = (int)(i / R);
    const int64_t pos = (offs[u] >> 32) + atomicSub(cnt + u, 1) - 1;
    srcs[pos] = nodes[t];
}

// Exclusive scan of packed (count << 32 | (count > 0)) over n nodes: 8192 per block.
constexpr int SCAN_T = 1024, SCAN_E = 8;
__global__ void scan_local_kernel(const int *cnt, int64_t n, int64_t *offs, int64_t *bsum) {
    __shared__ int64_t sh[SCAN_T];
    const int64_t base = (int64_t)blockIdx.x * SCAN_T * SCAN_E + (int64_t)threadIdx.x * SCAN_E;
    int64_t v[SCAN_E];
    int64_t s = 0;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e) {
        const int64_t i = base + e;
        const int c = i < n ? cnt[i] : 0;
        v[e] = ((int64_t)c << 32) | (c > 0 ? 1 : 0);
        s += v[e];
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < SCAN_T; o <<= 1) {
        int64_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    int64_t run = sh[threadIdx.x] - s;
#pragma unroll
    for (int e = 0; e < SCAN_E; ++e) {
        const int64_t i = base + e;
        if (i < n) offs[i] = run;
        run += v[e];
    }
    if (threadIdx.x == SCAN_T - 1) bsum[blockIdx.x] = sh[SCAN_T - 1];
}

__global__ void scan_blocks_kernel(int64_t *bsum, int nb, int64_t *total) {
    __shared__ int64_t sh[SCAN_T];
    int64_t carry = 0;
    for (int b0 = 0; b0 < nb; b0 += SCAN_T) {
        const int i = b0 + threadIdx.x;
        const int64_t v = i < nb ? bsum[i] : 0;
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < SCAN_T; o <<= 1) {
            int64_t t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
            __syncthreads();
            sh[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nb) bsum[i] = carry + sh[threadIdx.x] - v;
        const int64_t tot = sh[SCAN_T - 1];
        __syncthreads();
        carry += tot;
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void scan_add_kernel(int64_t *offs, int64_t n, const int64_t *bsum, const int64_t *total,
                                const int *cnt, int32_t *touched) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n) return;
    if (i == n) {
        offs[n] = *total;
        return;
    }
    const int64_t v = offs[i] + bsum[i / (SCAN_T * SCAN_E)];
    offs[i] = v;
    if (cnt[i] > 0) touched[(int)(v & 0xffffffff)] = (int32_t)i;
}

// ---------------------------------------------------------------- launchers
int launch_graph_sanitize(int32_t *graph, int64_t n, int R, int *status, cudaStream_t st) {
    graph_sanitize_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(graph, n, R, status);
    LV_CHECK_LAUNCH("graph_sanitize_kernel");
    return LV_OK;
}

int launch_entry_argmax(const uint8_t *rec, int64_t n, int64_t stride, int code_bytes, int metric, int32_t *out,
                        cudaStream_t st) {
    const int nb = 256;
    float *bg = nullptr;
    int *bi = nullptr;
    int rc = tmp_alloc((void **)&bg, sizeof(float) * nb, st);
    if (rc == LV_OK) rc = tmp_alloc((void **)&bi, sizeof(int) * nb, st);
    if (rc) {
        tmp_free(bg, st);
        return rc;
    }
    entry_partial_kernel<<<nb, 256, 0, st>>>(rec, n, stride, code_bytes, metric, bg, bi);
    entry_final_kernel<<<1, 256, 0, st>>>(bg, bi, nb, out);
    cudaError_t e = cudaGetLastError();
    tmp_free(bg, st);
    tmp_free(bi, st);
    if (e != cudaSuccess) return cuda_fail(e, "entry kernels");
    return LV_OK;
}

// ------------------------------------------------------------------ driver
// the size that decides how many reverse edges of a batch a target can take (part of the result)
static int prune_pool_bytes(int PMAX, int64_t stride) { return (int)(PMAX * (stride + 17) + stride + 16); }
// shared bytes of the prune kernel's arrays
static int prune_smem(int PMAX, int slot) { return PMAX * (slot + 14) + slot; }
// records of more code chunks than this are scored by four lanes each
constexpr int PRUNE_LONG = 16;
// A staged record takes its codes and constants.  Where there is room its chunks are an odd number (a
// thread per record: the 16-byte reads of consecutive records fall on different banks; 12 chunks have
// 4-way conflicts) or 4 mod 8 (four lanes per record: those of two consecutive records do).
static int prune_slot(int PMAX, int chunks, int metric) {
    const int used = chunks + 1 + metric, pad = chunks > PRUNE_LONG ? (used + 3) / 8 * 8 + 4 : used | 1;
    return prune_smem(PMAX, 16 * pad) <= 225 * 1024 ? 16 * pad : 16 * used;
}

template <int BITS, int MODE, bool L2, bool LONG, int NT>
static int go_prune(const PruneParams &pp, unsigned grid, cudaStream_t st) {
    const int sm = prune_smem(pp.PMAX, pp.slot);
    if (grid == 0) return LV_OK;
    auto k = prune_kernel<BITS, MODE, L2, LONG, NT>;
    LV_CUDA(allow_smem(k));
    k<<<grid, NT, sm, st>>>(pp);
    LV_CHECK_LAUNCH("prune_kernel");
    return LV_OK;
}

template <int BITS, bool L2>
static int launch_prune_m(const PruneParams &pp, int mode, unsigned grid, cudaStream_t st) {
    // long records leave room for one block of a batch node's pool on an SM: eight warps
    if (pp.CH > PRUNE_LONG)
        return mode == 0 ? go_prune<BITS, 0, L2, true, 256>(pp, grid, st) : go_prune<BITS, 1, L2, true, 128>(pp, grid, st);
    return mode == 0 ? go_prune<BITS, 0, L2, false, 128>(pp, grid, st) : go_prune<BITS, 1, L2, false, 128>(pp, grid, st);
}

template <int BITS>
static int launch_prune(const PruneParams &pp, int mode, unsigned grid, cudaStream_t st) {
    return pp.metric ? launch_prune_m<BITS, true>(pp, mode, grid, st) : launch_prune_m<BITS, false>(pp, mode, grid, st);
}

int build_graph_impl(lv_index *idx, int R, int Lb, float alpha, int passes, int batch, uint64_t seed, int rule,
                     cudaStream_t st) {
    const int64_t n = idx->n;
    batch = (int)std::min<int64_t>(batch, n);
    const int PMAX = Lb + R;
    if (prune_pool_bytes(PMAX, idx->pg.stride) > 227 * 1024) return fail(LV_ERR_CAPACITY, "build: L_build + R too large");
    // reverse-edge pool: the target's list plus its new sources of one batch
    int PMAX1 = std::max(PMAX, 4 * R + 256);
    // (two prune blocks per SM for short records; long records may take most of an SM's shared memory)
    const int cap1 = idx->pg.stride > 256 ? 200 * 1024 : 120 * 1024;
    while (PMAX1 > PMAX && prune_pool_bytes(PMAX1, idx->pg.stride) > cap1) PMAX1 -= 32;
    cudaFree(idx->graph);
    idx->graph = nullptr;
    idx->R = 0;
    idx->entry = -1;
    LV_CUDA(cudaMalloc(&idx->graph, sizeof(int32_t) * (size_t)n * R));

    // workspace layout
    const int64_t nblk = (n + SCAN_T * SCAN_E - 1) / (SCAN_T * SCAN_E);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += round_up((int64_t)bytes, 256);
        return o;
    };
    const size_t o_perm = take(sizeof(int32_t) * n);
    const size_t o_bid = take(sizeof(int32_t) * (size_t)batch * Lb);
    const size_t o_bsc = take(sizeof(float) * (size_t)batch * Lb);
    const size_t o_newl = take(sizeof(int32_t) * (size_t)batch * R);
    const size_t o_cnt = take(sizeof(int) * n);
    const size_t o_offs = take(sizeof(int64_t) * (n + 1));
    const size_t o_bsum = take(sizeof(int64_t) * (nblk + 1));
    const size_t o_tot = take(sizeof(int64_t));
    const size_t o_touch = take(sizeof(int32_t) * (size_t)std::min<int64_t>(n, (int64_t)batch * R));
    const size_t o_srcs = take(sizeof(int32_t) * (size_t)batch * R);
    const size_t o_ent = take(sizeof(int32_t));
    int rc = ensure_ws(&idx->bws, &idx->bws_bytes, off);
    if (rc) return rc;
    uint8_t *ws = reinterpret_cast<uint8_t *>(idx->bws);
    int32_t *perm_d = reinterpret_cast<int32_t *>(ws + o_perm);
    int32_t *bid = reinterpret_cast<int32_t *>(ws + o_bid);
    float *bsc = reinterpret_cast<float *>(ws + o_bsc);
    int32_t *newl = reinterpret_cast<int32_t *>(ws + o_newl);
    int *cnt = reinterpret_cast<int *>(ws + o_cnt);
    int64_t *offs = reinterpret_cast<int64_t *>(ws + o_offs);
    int64_t *bsum = reinterpret_cast<int64_t *>(ws + o_bsum);
    int64_t *tot = reinterpret_cast<int64_t *>(ws + o_tot);
    int32_t *touched = reinterpret_cast<int32_t *>(ws + o_touch);
    int32_t *srcs = reinterpret_cast<int32_t *>(ws + o_srcs);
    int32_t *ent_d = reinterpret_cast<int32_t *>(ws + o_ent);

    // initial graph, entry point, order
    random_graph_kernel<<<(unsigned)((n + RG_WARPS - 1) / RG_WARPS), 32 * RG_WARPS, 0, st>>>(idx->graph, n, R, seed,
                                                                                             idx->status);
    LV_CHECK_LAUNCH("random_graph_kernel");
    rc = launch_entry_argmax(idx->prim, n, idx->pg.stride, idx->pg.code_bytes, idx->metric, ent_d, st);
    if (rc) return rc;
    int32_t entry = 0;
    LV_CUDA(cudaMemcpyAsync(&entry, ent_d, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    std::vector<int32_t> perm((size_t)n);
    for (int64_t i = 0; i < n; ++i) perm[i] = (int32_t)i;
    for (int64_t i = n - 1; i >= 1; --i) {
        int64_t j = (int64_t)(splitmix(seed + 1, (uint64_t)i, 0) % (uint64_t)(i + 1));
        std::swap(perm[i], perm[j]);
    }
    LV_CUDA(cudaMemcpyAsync(perm_d, perm.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, st));
    LV_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * n, st));
    LV_CUDA(cudaStreamSynchronize(st));

    // search in build mode
    BeamParams bp;
    memset(&bp, 0, sizeof(bp));
    bp.prim = idx->prim;
    bp.prim_stride = idx->pg.stride;
    bp.prim_chunks = idx->pg.code_chunks;
    bp.prim_dim = idx->d;
    bp.graph = idx->graph;
    bp.R = R;
    bp.n = n;
    bp.entry = entry;
    bp.uni = make_int4(Lb, Lb, 0, 0);
    bp.mu2 = idx->mu2;
    bp.metric = idx->metric;
    bp.ids = bid;
    bp.scores = bsc;
    bp.ldo = Lb;
    bp.status = idx->status;
    bp.work = idx->status + 1;
    bp.Lcap = (int)round_up(Lb, 32);
    int hs = 1024;
    while (hs < 8 * Lb && hs < 8192) hs <<= 1;
    while (hs < 2 * bp.Lcap) hs <<= 1;
    bp.Hcap = hs;
    bp.hbits = 0;
    while ((1 << bp.hbits) < hs) bp.hbits++;
    bp.W = 1;
    bp.T = 1;
    bp.Rcap = beam_rcap(1, 1, R);
    bp.vbits = 32;
    bp.warp_smem = beam_warp_smem(bp.Lcap, bp.Hcap, 32, bp.Rcap, 0);  // the build scorer keeps its query in registers
    int warps = 8;
    while (warps > 1 && (size_t)warps * bp.warp_smem > 227 * 1024) warps >>= 1;
    const size_t bsmem = (size_t)warps * bp.warp_smem;
    const int nc = (idx->pg.code_chunks + 1 + idx->metric + 3) / 4;

    PruneParams pp;
    memset(&pp, 0, sizeof(pp));
    pp.prim = idx->prim;
    pp.stride = idx->pg.stride;
    pp.CH = idx->pg.code_chunks;
    pp.cb = idx->pg.code_bytes;
    pp.dim = idx->d;
    pp.mu2 = idx->mu2;
    pp.metric = idx->metric;
    pp.R = R;
    pp.PMAX = PMAX;
    pp.slot = prune_slot(PMAX, idx->pg.code_chunks, idx->metric);
    pp.n = n;
    pp.graph = idx->graph;
    pp.beams = bid;
    pp.Lb = Lb;
    pp.bscores = bsc;
    pp.newl = newl;
    pp.offs = offs;
    pp.srcs = srcs;
    pp.touched = touched;
    pp.total = tot;
    pp.status = idx->status;

    for (int pass = 0; pass < passes; ++pass) {
        pp.alpha = pass < passes - 1 ? 1.0f : alpha;
        pp.shift = rule ? host_fsub(pp.alpha, 1.0f) : 0.0f;
        for (int64_t b0 = 0; b0 < n; b0 += batch) {
            const int nb = (int)std::min<int64_t>(batch, n - b0);
            bp.qnodes = perm_d + b0;
            bp.m = nb;
            LV_CUDA(cudaMemsetAsync(bp.work, 0, sizeof(int), st));
            rc = launch_build_search(bp, idx->pbits, nc, warps * 32, bsmem, idx->num_sms, st);
            if (rc) return rc;
            pp.nodes = perm_d + b0;
            rc = idx->pbits == 8 ? launch_prune<8>(pp, 0, nb, st) : launch_prune<4>(pp, 0, nb, st);
            if (rc) return rc;
            scatter_rows_kernel<<<nb, 64, 0, st>>>(newl, perm_d + b0, nb, R, idx->graph);
            const int64_t tp = (int64_t)nb * R;
            count_pairs_kernel<<<(unsigned)((tp + 255) / 256), 256, 0, st>>>(newl, tp, cnt);
            scan_local_kernel<<<(unsigned)nblk, SCAN_T, 0, st>>>(cnt, n, offs, bsum);
            scan_blocks_kernel<<<1, SCAN_T, 0, st>>>(bsum, (int)nblk, tot);
            scan_add_kernel<<<(unsigned)((n + 1 + 255) / 256), 256, 0, st>>>(offs, n, bsum, tot, cnt, touched);
            scatter_pairs_kernel<<<(unsigned)((tp + 255) / 256), 256, 0, st>>>(newl, perm_d + b0, nb, R, offs, cnt, srcs);
            LV_CHECK_LAUNCH("reverse-edge kernels");
            const unsigned g1 = (unsigned)std::min<int64_t>(n, tp);
            // most targets gain a few edges: the pools of those with at most 32 sources fit many blocks on an
            // SM; the rest (a target may receive many reverse edges in one batch) take a second launch.  The
            // line is drawn on the sources alone, which the first launch does not change: a list it rewrote
            // must not be taken a second time.  Where the largest pool is small, one launch takes all: the second
            // one's blocks cost more to start than the occupancy gives (50,000 nodes of 24 codes, R = 16, pools of
            // 20 KB: 7.97 ms with two launches, 7.26 with one; 64 codes, R = 32, 36 KB: 13.8 and 13.3; 64 codes,
            // R = 64, 48 KB: equal; 128 codes, R = 32, 61 KB: 14.8 and 15.1; 160 codes, R = 64, 97 KB: 21.7 and 24.1).
            const bool one = prune_smem(PMAX1, prune_slot(PMAX1, idx->pg.code_chunks, idx->metric)) <= 40 * 1024;
            const int small = one ? PMAX1 : std::min(R + 32, PMAX1);
            for (int tier = 0; tier < (small < PMAX1 ? 2 : 1) && !rc; ++tier) {
                PruneParams pr = pp;
                pr.PMAX = tier ? PMAX1 : small;
                pr.slot = prune_slot(pr.PMAX, idx->pg.code_chunks, idx->metric);
                pr.lo = tier ? 32 : -1;
                pr.hi = tier || small == PMAX1 ? 0x7fffffff : 32;
                rc = idx->pbits == 8 ? launch_prune<8>(pr, 1, g1, st) : launch_prune<4>(pr, 1, g1, st);
            }
            if (rc) return rc;
        }
    }
    LV_CUDA(cudaStreamSynchronize(st));
    idx->R = R;
    idx->entry = entry;
    return LV_OK;
}

}  // namespace lv
