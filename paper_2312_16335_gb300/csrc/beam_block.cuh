// Beam search of small batches: one block of four warps per query, the same rounds, scores and
// results as beam_kernel (beam.cuh).
//
// A batch of a few queries per SM is bound by the latency of one walk, not by the chip: with a
// warp per query a round's phases (128 adjacency ids, about 20 records, the merge over the beam) run
// one after the other on 32 lanes, in passes, while the other schedulers idle.  Here a round is one
// pass of each phase: a thread per adjacency id, eight records a warp (each warp filters and places
// the records it scored), a thread per candidate and per beam position in the merge, five block
// barriers.  A round waits for two dependent global loads (adjacency row, record) and little else.
// The visited cache holds 32-bit ids in buckets of 4, filled by compare-and-swap, so that two threads
// that meet one id in a round do not both take it; it may forget ids when a bucket is full, as the
// caches of beam_kernel may.
// One query on 200k x 768 (L = 128, width 2, 72 rounds): 186 us for the whole search against 249 us with a
// warp per query; 100 queries 315 and 361 us, 608 375 and 452.  Of a round's 3900 cycles the adjacency
// row and visited test take 1180, the records 1190, the places 510, the parents 430, ranks and merge 510.
// Measured and left out: every warp scoring its own new ids (a barrier less, uneven passes: equal), a
// search for places by four probes a step and L1 prefetches of the likely next rows (slower).
#pragma once

#include "beam.cuh"

namespace lv {

constexpr int BB_WARPS = 4, BB_T = 32 * BB_WARPS;
constexpr int BB_SLOTS = 4096;  // visited cache of a query

// shared bytes of a block: beam (8 Lcap), visited cache (4 Hcap), ids and scores of the new records and
// id, score and place of the candidates (20 Rcap), the scorer's query
constexpr int block_query_smem(int Lcap, int Hcap, int Rcap, int qbytes) {
    return 8 * Lcap + 4 * Hcap + 20 * Rcap + qbytes;
}
static_assert(block_query_smem(LCAP_MAX, BB_SLOTS, CMAX, 2048) <= 47 * 1024, "fits without asking for more");

template <class PS, int WT>
__global__ void __launch_bounds__(BB_T) beam_block_kernel(const BeamParams p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_cnt[2], s_cv;  // new ids of the round (by turns), candidates
    __shared__ unsigned s_ranks;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    int *const hash = reinterpret_cast<int *>(smem_raw);       // visited cache
    void *const qsm = hash + p.Hcap;                           // the scorer's query
    float *const bS = reinterpret_cast<float *>(reinterpret_cast<unsigned char *>(qsm) + PS::QBYTES);  // beam scores
    int *const bI = reinterpret_cast<int *>(bS + p.Lcap);      // beam ids, top bit = expanded
    int *const wI = bI + p.Lcap;                               // new ids of the round and their scores
    float *const wS = reinterpret_cast<float *>(wI + p.Rcap);
    int *const cI = reinterpret_cast<int *>(wS + p.Rcap);      // the candidates that enter
    float *const cS = reinterpret_cast<float *>(cI + p.Rcap);
    int *const cP = reinterpret_cast<int *>(cS + p.Rcap);      // beam members ahead of each, then its place
    const int64_t qi = blockIdx.x;
    const int bshift = 34 - p.hbits;  // 32 - log2(buckets)

    const int4 dq = p.desc ? p.desc[qi] : p.uni;
    int k = dq.x, L = dq.y, r = dq.z;
    if (L > p.Lcap || L < 1 || k > p.ldo || k < 0) {
        if (tid == 0) atomicOr(p.status, ST_CAPACITY);
        L = min(max(L, 1), p.Lcap);
        k = min(max(k, 0), p.ldo);
    }
    r = min(max(r, 0), L);
    const int maxh = dq.w > 0 ? dq.w : (int)(p.n < 0x7fffffff ? p.n : 0x7fffffff);
    const int entry = p.entry;
    for (int t = 4 * tid; t < p.Hcap; t += 4 * BB_T) *reinterpret_cast<int4 *>(hash + t) = make_int4(-1, -1, -1, -1);
    if (tid == 0) wI[0] = entry;
    PS ps;
    ps.setup(p, qi, lane, qsm, wid == 0);
    __syncthreads();
    if (wid == 0) {
        if (lane == 0) hash[4 * (int)(((unsigned)entry * 0x9E3779B1u) >> bshift)] = entry;
        ps.score(wI, wS, 1, lane);
        __syncwarp();
        if (lane == 0) {
            bS[0] = fmaxf(wS[0], -INFINITY);  // NaN ranks last: keys stay ordered
            bI[0] = entry;
            s_cnt[0] = 0;
        }
    }
    __syncthreads();
    int size = 1, hops = 0, F = 0, turn = 0;
    for (; hops < maxh; turn ^= 1) {
        // the WT best unexpanded members: every warp finds the same ones
        int par[WT];
        int npar = 0;
        const int want = min(WT, maxh - hops);
        for (int base = F & ~31; base < size && npar < want; base += 32) {
            const int i = base + lane;
            unsigned bal = __ballot_sync(FULL, i >= F && i < size && !(bI[i] & (int)EXPANDED));
#pragma unroll
            for (int w = 0; w < WT; ++w)
                if (bal && npar < want && w == npar) {
                    par[w] = base + __ffs(bal) - 1;
                    bal &= bal - 1;
                    ++npar;
                }
        }
        if (npar == 0) break;
        F = par[0] + 1;
#pragma unroll
        for (int w = 1; w < WT; ++w)
            if (w < npar) F = par[w] + 1;
        hops += npar;
        // ---- adjacency and visited test, a thread per id ----
        const int nst = npar * p.R;
        for (int j0 = 0; j0 < nst; j0 += BB_T) {
            const int j = j0 + tid;
            int u = -1;
            if (j < nst) {
                const bool second = WT > 1 && j >= p.R;
                const int parent = bI[second ? par[WT - 1] : par[0]] & ~(int)EXPANDED;
                u = __ldg(p.graph + (int64_t)parent * p.R + (second ? j - p.R : j));
                if (u >= p.n) {
                    atomicOr(p.status, ST_CORRUPT);
                    u = -1;
                }
            }
            bool isnew = false;
            if (u >= 0) {
                const unsigned hv = (unsigned)u * 0x9E3779B1u;
                int *const b = hash + 4 * (int)(hv >> bshift);
                const int4 v = *reinterpret_cast<const int4 *>(b);
                if (v.x != u && v.y != u && v.z != u && v.w != u) {
                    // take the first empty slot; another thread may take it first, with this id or another
                    bool open = true;
                    for (int s = v.x < 0 ? 0 : v.y < 0 ? 1 : v.z < 0 ? 2 : v.w < 0 ? 3 : 4; s < 4 && open; ++s) {
                        const int was = atomicCAS(b + s, -1, u);
                        if (was == -1) isnew = true;
                        open = was != -1 && was != u;
                    }
                    if (open) isnew = atomicExch(b + (int)((hv >> (bshift - 2)) & 3u), u) != u;  // full
                }
            }
            const unsigned bal = __ballot_sync(FULL, isnew);
            int base = 0;
            if (lane == 0 && bal) base = atomicAdd(&s_cnt[turn], __popc(bal));
            base = __shfl_sync(FULL, base, 0);
            if (isnew) wI[base + __popc(bal & lt)] = u;
        }
        if (tid == 0) s_cv = 0;
        __syncthreads();
        const int cnt = s_cnt[turn];
        if (tid == 0) {  // the flags travel with the members in the merge
#pragma unroll
            for (int w = 0; w < WT; ++w)
                if (w < npar) bI[par[w]] |= (int)EXPANDED;
            s_ranks = 0;
            s_cnt[turn ^ 1] = 0;  // read before the last round's second barrier, added to after this one's
        }
        // ---- score, eight records a warp (sixteen when there are many); the warp that scored a record
        // tests it against the beam's last member and finds its place ----
        const bool full = size >= L;
        float tS = 0.f;
        int tI = 0;
        if (full) {
            tS = bS[L - 1];
            tI = bI[L - 1] & ~(int)EXPANDED;
        }
        const int per = cnt > 8 * BB_WARPS ? 16 : 8;
        for (int b = per * wid; b < cnt; b += per * BB_WARPS) {
            if (per == 16)
                ps.template pass<2>(wI, wS, b, cnt, lane);
            else
                ps.template pass<1>(wI, wS, b, cnt, lane);
            __syncwarp();
            const int j = b + lane;
            bool valid = false;
            float s = 0.f;
            int id = 0, pb = 0;
            if (lane < per && j < cnt) {
                s = fmaxf(wS[j], -INFINITY);
                id = wI[j];
                valid = !full || key_better(s, id, tS, tI);
                if (valid) {
                    int hi = size;
                    while (pb < hi) {
                        const int mid = (pb + hi) >> 1;
                        const float ms = bS[mid];
                        bool better = ms > s;
                        if (ms == s) better = (bI[mid] & ~(int)EXPANDED) < id;
                        if (better)
                            pb = mid + 1;
                        else
                            hi = mid;
                    }
                    if (pb < size && (bI[pb] & ~(int)EXPANDED) == id) valid = false;
                }
            }
            const unsigned bal = __ballot_sync(FULL, valid);
            int base = 0;
            if (lane == 0 && bal) base = atomicAdd(&s_cv, __popc(bal));
            base = __shfl_sync(FULL, base, 0);
            if (valid) {
                const int o = base + __popc(bal & lt);
                cI[o] = id;
                cS[o] = s;
                cP[o] = pb;
            }
        }
        __syncthreads();
        int cv = s_cv;
        if (cv == 0) continue;
        // ---- place of each candidate: the beam members ahead and its rank (see beam_kernel: copies of an
        // id share a rank, and only then are they looked for) ----
        for (;;) {
            unsigned ranks = 0;
            for (int j = tid; j < cv; j += BB_T) {
                const float s = cS[j];
                const int id = cI[j];
                int rank = 0;
                for (int u = 0; u < cv; ++u) rank += key_better(cS[u], cI[u], s, id) ? 1 : 0;
                cP[j] = (cP[j] & 0xffff) | rank << 16;
                ranks += (unsigned)rank;
            }
            if (WT > 1) {
                ranks = __reduce_add_sync(FULL, ranks);
                if (lane == 0 && ranks) atomicAdd(&s_ranks, ranks);
            }
            __syncthreads();
            if (WT == 1 || s_ranks == (unsigned)(cv * (cv - 1) / 2)) break;
            __syncthreads();
            if (wid == 0) {  // rare: one warp drops the copies
                int cv2 = 0;
                for (int j0 = 0; j0 < cv; j0 += 32) {
                    const int j = j0 + lane;
                    bool keep = j < cv;
                    float s = 0.f;
                    int id = 0, pb = 0;
                    if (keep) {
                        s = cS[j];
                        id = cI[j];
                        pb = cP[j] & 0xffff;
                        for (int u = 0; u < cv2; ++u) keep &= cI[u] != id;
                        for (int u = j0; u < j; ++u) keep &= cI[u] != id;
                    }
                    const unsigned bal = __ballot_sync(FULL, keep);
                    __syncwarp();
                    if (keep) {
                        const int o = cv2 + __popc(bal & lt);
                        cI[o] = id;
                        cS[o] = s;
                        cP[o] = pb;
                    }
                    cv2 += __popc(bal);
                    __syncwarp();
                }
                if (lane == 0) {
                    s_cv = cv2;
                    s_ranks = 0;
                }
            }
            __syncthreads();
            cv = s_cv;
        }
        // ---- merge in place, a thread per beam position: a position that no candidate takes holds the
        // member that is as many positions further up as candidates come before it ----
        constexpr int E = LCAP_MAX / BB_T;
        const int nsize = min(L, size + cv);
        float ms[E];
        int mi[E];
        bool move[E];
        int first = LCAP_MAX;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            move[e] = false;
            if (BB_T * e < nsize) {
                const int d = tid + BB_T * e;
                int before = 0;
                bool taken = false;
                for (int u = 0; u < cv; ++u) {
                    const int x = cP[u], np = (x & 0xffff) + (x >> 16);
                    before += np < d ? 1 : 0;
                    taken |= np == d;
                    first = min(first, np);
                }
                if (d < nsize && before && !taken) {
                    move[e] = true;
                    ms[e] = bS[d - before];
                    mi[e] = bI[d - before];
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (move[e]) {
                bS[tid + BB_T * e] = ms[e];
                bI[tid + BB_T * e] = mi[e];
            }
        for (int j = tid; j < cv; j += BB_T) {
            const int x = cP[j], np = (x & 0xffff) + (x >> 16);
            if (np < L) {
                bS[np] = cS[j];
                bI[np] = cI[j];
            }
        }
        __syncthreads();
        size = nsize;
        F = min(F, first);
    }
    __syncthreads();  // a round without candidates ends without one

    int32_t *oid = p.ids + qi * p.ldo;
    float *osc = p.scores + qi * p.ldo;
    if (r > 0 && p.cand) {
        // the rerank kernel scores these with the secondary store and writes the results
        const int nr = min(r, size);
        int32_t *cd = p.cand + qi * p.ldc;
        for (int t = tid; t < nr; t += BB_T) cd[t] = bI[t] & ~(int)EXPANDED;
        if (tid == 0) p.cand_n[qi] = nr;
        return;
    }
    if (p.cand_n && tid == 0) p.cand_n[qi] = -1;
    const int nres = min(k, size);
    for (int t = tid; t < p.ldo; t += BB_T) {
        oid[t] = t < nres ? bI[t] & ~(int)EXPANDED : -1;
        osc[t] = t < nres ? bS[t] : -INFINITY;
    }
}

// launcher: one block per query (p.m of them)
template <class PS, int WT>
int launch_block(const BeamParams &p, size_t smem, cudaStream_t st) {
    auto k = beam_block_kernel<PS, WT>;
    if (p.slots) {  // every query has its block at once: no waves to cut the batch by
        *p.slots = INT64_MAX;
        return LV_OK;
    }
    k<<<(unsigned)p.m, BB_T, smem, st>>>(p);
    LV_CHECK_LAUNCH("beam_block_kernel");
    return LV_OK;
}

template <int NC, int BITS>
int launch_block_nc(const BeamParams &p, size_t smem, cudaStream_t st) {
    if (p.metric)
        return p.W == 1 ? launch_block<LvqIntScorer<NC, BITS, true>, 1>(p, smem, st)
                        : launch_block<LvqIntScorer<NC, BITS, true>, 2>(p, smem, st);
    return p.W == 1 ? launch_block<LvqIntScorer<NC, BITS, false>, 1>(p, smem, st)
                    : launch_block<LvqIntScorer<NC, BITS, false>, 2>(p, smem, st);
}

}  // namespace lv
