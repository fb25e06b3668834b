// Rerank kernel (Sec. 2 "Search": the final candidates of the primary search are rescored
// with the full-dimensional LVQ-8 or FP16 secondary vectors against the unreduced query, and the
// best k are kept).  The beam kernel hands over the top-r ids of every query (BeamParams::cand);
// here a block of four warps (two for long FP16 records) takes one query.
//
// Bound by the random reads of the secondary records (r x about D bytes per query).  A record
// goes through a shared-memory ring by cp.async.bulk, one copy per record, RR_GROUP records to a
// stage, so a warp keeps two stages in flight without holding them in registers.  The warps of a
// block share a query's candidates (group w, w + warps, ...) and its byte limbs: the set-up and the
// top-k of one query then hide behind the copies of the other blocks of the SM.
// 152 candidates of 784 bytes per query from a 1M-row store, L2 flushed (time, share of the copy
// bandwidth): 10,000 queries 213 us (82 %), 3,069 86 us (63 %), 100 20 us; with one warp per query
// 217, 106 and 40 us; with three stages (five instead of seven blocks per SM) 248, 96 and 20 us;
// with 16-byte cp.async instead of bulk copies 299 us at 10,000.  In the benchmark's search the
// second sub-batch's 3,069 queries took 137 us when a warp loaded its records into registers.
#include <cuda_fp16.h>

#include "beam.cuh"

namespace lv {

constexpr int RR_GROUP = 4;   // records of a stage (their four sums share one reduction)
constexpr int RR_STAGES = 2;  // ring stages of a warp
constexpr uint32_t RR_TRY_NS = 1000000;  // longest suspension of one try of a wait

struct RerankParams {
    const uint8_t *sec;
    int64_t sec_stride;
    int sec_chunks;  // 16-byte code chunks of a record
    int rec_bytes;   // bytes of a record that are read (codes and constants)
    const float *Q;  // unreduced queries m x D
    int D;
    const float *smean;    // secondary mean mu (D): cQ = <q, mu>, sQ = sum q per query; NULL with FP16 records
    const int4 *desc;      // per query (k, L, r, max_hops) or NULL
    int4 uni;
    int64_t m;
    const int32_t *cand;  // m x ldc candidate ids
    const int *cand_n;    // per query: candidates, or -1 = results already written
    int ldc;
    int32_t *ids;
    float *scores;
    int ldo;
    int *status;
    int tries;  // limit of one wait for a stage's copies
};

// --------------------------------------------------------------------------------
// Scorers: per query setup() (the whole block; the query's form in `qsm`, shared memory), load()
// (a warp's share of it into registers), then dot(), a lane's part of the score of a record in
// shared memory, and finish(), the score from the warp's sum of the parts.
// --------------------------------------------------------------------------------
// LVQ-8 records against the unreduced query held as 24-bit fixed point in three byte limbs (same
// scheme and error bound as LvqIntScorer, with D in place of d).  Lane l holds code chunks l and
// l + 32 (D <= 1008).
template <bool L2 = false>
struct SecIntScorer {
    static constexpr int WARPS = 4;  // of a block, all on one query
    static constexpr int NCW = 2;
    uint4 qh[NCW], qm[NCW], ql[NCW];
    float c0, s0, scale;
    int CH;

    static constexpr __host__ __device__ int query_bytes(int chunks) { return 3 * 16 * chunks; }

    // Each warp reads the whole query and forms the constants in its lanes' fixed order; the WARPS warps
    // share the limbs: byte j of the limb arrays h, m, l belongs to entry j, that is to code j of a
    // record.  Loads go out 16 at a time; the loops stay rolled beyond that, since a small batch
    // runs this code once per SM and pays for every instruction line it fetches.
    __device__ __forceinline__ void setup(const float *q, const RerankParams &p, unsigned char *qsm) {
        constexpr int U = 16;
        CH = p.sec_chunks;
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        float amax = 0.f, cQ = 0.f, sQ = 0.f;
#pragma unroll 1
        for (int j0 = lane; j0 < p.D; j0 += 32 * U) {
            float v[U], mu[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const bool in = j0 + 32 * i < p.D;
                v[i] = in ? __ldg(q + j0 + 32 * i) : 0.f;
                mu[i] = in ? __ldg(p.smean + j0 + 32 * i) : 0.f;
            }
#pragma unroll
            for (int i = 0; i < U; ++i)
                if (j0 + 32 * i < p.D) {
                    amax = fmaxf(amax, fabsf(v[i]));
                    cQ = fmaf(v[i], mu[i], cQ);
                    sQ += v[i];
                }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, o));
            cQ += __shfl_xor_sync(FULL, cQ, o);
            sQ += __shfl_xor_sync(FULL, sQ, o);
        }
        c0 = cQ;
        s0 = sQ;
        scale = amax > 0.f ? amax / 8388607.0f : 1.0f;
        const float inv = amax > 0.f ? 8388607.0f / amax : 0.f;
#pragma unroll 4
        for (int j = lane + 32 * wid; j < 16 * CH; j += 32 * WARPS) {  // entries past D are zero
            int qv = j < p.D ? __float2int_rn(__ldg(q + j) * inv) : 0;
            qv = max(-8388607, min(8388607, qv));
            qsm[j] = (unsigned char)(qv >> 16);
            qsm[16 * CH + j] = (unsigned char)(qv >> 8);
            qsm[32 * CH + j] = (unsigned char)qv;
        }
    }

    __device__ __forceinline__ void load(const unsigned char *qsm, int lane) {
        const uint4 *q4 = reinterpret_cast<const uint4 *>(qsm);
#pragma unroll
        for (int t = 0; t < NCW; ++t) {
            const int c = lane + 32 * t;
            const uint4 z = make_uint4(0, 0, 0, 0);
            qh[t] = c < CH ? q4[c] : z;
            qm[t] = c < CH ? q4[CH + c] : z;
            ql[t] = c < CH ? q4[2 * CH + c] : z;
        }
    }

    __device__ __forceinline__ float dot(const unsigned char *rec, int lane) const {
        int sh = 0, sm = 0, sl = 0;
#pragma unroll
        for (int t = 0; t < NCW; ++t) {
            // lanes past the codes hold zero limbs and read some chunk of the record
            const uint4 v = *reinterpret_cast<const uint4 *>(rec + 16 * min(lane + 32 * t, CH));
            sh = dp4a_su(qh[t].x, v.x, sh);
            sm = dp4a_uu(qm[t].x, v.x, sm);
            sl = dp4a_uu(ql[t].x, v.x, sl);
            sh = dp4a_su(qh[t].y, v.y, sh);
            sm = dp4a_uu(qm[t].y, v.y, sm);
            sl = dp4a_uu(ql[t].y, v.y, sl);
            sh = dp4a_su(qh[t].z, v.z, sh);
            sm = dp4a_uu(qm[t].z, v.z, sm);
            sl = dp4a_uu(ql[t].z, v.z, sl);
            sh = dp4a_su(qh[t].w, v.w, sh);
            sm = dp4a_uu(qm[t].w, v.w, sm);
            sl = dp4a_uu(ql[t].w, v.w, sl);
        }
        return fmaf((float)sh, 65536.0f, fmaf((float)sm, 256.0f, (float)sl));
    }

    __device__ __forceinline__ float finish(float s, const unsigned char *rec) const {
        const float2 k = *reinterpret_cast<const float2 *>(rec + 16 * CH);  // delta, lower
        const float sc = fmaf(k.x * scale, s, fmaf(k.y, s0, c0));
        if (!L2) return sc;
        // the original vector's squared norm: second constants chunk
        return fmaf(2.0f, sc, -*reinterpret_cast<const float *>(rec + 16 * CH + 20));
    }
};

// FP16 records: the unreduced query in float32 registers, lane l holds half chunks l, l + 32, ...
// (8 halves each; D <= 32 NCW 8); the halves are widened exactly to float32 and accumulated in
// float32.
template <int NCW, bool L2 = false>
struct Fp16SecScorer {
    // Above 256 dimensions two warps a block: records of 1.5 KB leave an SM four blocks of four warps, too few
    // queries at once where r is small.  200k x 768, r = 20 / 64 / 152, whole searches against four warps: 2000
    // queries 1.03 / 1.03 / 1.05 times the speed, 20,000 1.09 / 1.05 / 1.02; up to 256 dimensions equal.
    static constexpr int WARPS = NCW > 1 ? 2 : 4;
    float q[NCW][8];
    int CH;

    static constexpr __host__ __device__ int query_bytes(int chunks) { return 32 * chunks; }

    __device__ __forceinline__ void setup(const float *qrow, const RerankParams &p, unsigned char *qsm) {
        CH = p.sec_chunks;
        float *dst = reinterpret_cast<float *>(qsm);
        for (int j = threadIdx.x; j < 8 * CH; j += 32 * WARPS) dst[j] = j < p.D ? qrow[j] : 0.f;
    }

    __device__ __forceinline__ void load(const unsigned char *qsm, int lane) {
        const float *src = reinterpret_cast<const float *>(qsm);
#pragma unroll
        for (int t = 0; t < NCW; ++t) {
            const int c = lane + 32 * t;
#pragma unroll
            for (int e = 0; e < 8; ++e) q[t][e] = c < CH ? src[8 * c + e] : 0.f;
        }
    }

    __device__ __forceinline__ float dot(const unsigned char *rec, int lane) const {
        float a0 = 0.f, a1 = 0.f, nn = 0.f;
#pragma unroll
        for (int t = 0; t < NCW; ++t) {
            const int c = lane + 32 * t;
            const uint4 v = c < CH ? *reinterpret_cast<const uint4 *>(rec + 16 * c) : make_uint4(0, 0, 0, 0);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 x = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
                a0 = fmaf(q[t][2 * i], x.x, a0);
                a1 = fmaf(q[t][2 * i + 1], x.y, a1);
                if (L2) nn = fmaf(x.y, x.y, fmaf(x.x, x.x, nn));
            }
        }
        const float s = a0 + a1;
        return L2 ? fmaf(2.0f, s, -nn) : s;  // 2 <q, x16> - ||x16||^2, summed over the warp
    }

    __device__ __forceinline__ float finish(float s, const unsigned char *) const { return s; }
};

// --------------------------------------------------------------------------------
// bulk copies
// --------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t rr_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Wait for the phase with parity `parity`; false when it gave up.  A try suspends the warp for RR_TRY_NS at
// most (the hint replaces the system's own limit), so `tries` bounds the wait in time.
__device__ __forceinline__ bool rr_wait(uint64_t *bar, uint32_t parity, int tries) {
    for (int it = 0; it < tries; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(rr_smem(bar)), "r"(parity), "r"(RR_TRY_NS)
            : "memory");
        if (done) return true;
    }
    return false;
}

// --------------------------------------------------------------------------------
// top k
// --------------------------------------------------------------------------------
// an unsigned key that orders like the score (-0 and 0 alike)
__device__ __forceinline__ unsigned order_key(float s) {
    const unsigned u = __float_as_uint(s + 0.0f);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}

constexpr int TOPK_ROUNDS = 32;  // up to this k: rounds of a warp maximum; above: ranks by the block

// The best k of n entries by (score desc, id asc) into oid / osc[0 .. min(k, n)).  key[t] holds the
// order of entry t, score above id; S its score.  Small k: one warp, a round per result -- two redux
// instructions for the maximum, its entry cleared.  Larger k: every thread ranks its entries against
// all (n^2 / blockDim.x comparisons a thread, independent of k).
__device__ __forceinline__ void block_topk(unsigned long long *key, const float *S, int n, int k, int32_t *oid,
                                           float *osc) {
    const int tid = threadIdx.x, lane = tid & 31;
    if (k <= TOPK_ROUNDS) {
        if (tid >= 32) return;
        for (int r = 0; r < k && r < n; ++r) {
            unsigned long long best = 0;
            int bt = lane;
#pragma unroll 4
            for (int t = lane; t < n; t += 32) {
                const unsigned long long x = key[t];
                if (x > best) {
                    best = x;
                    bt = t;
                }
            }
            const unsigned hi = (unsigned)(best >> 32), top = __reduce_max_sync(FULL, hi);
            const unsigned lo = hi == top ? (unsigned)best : 0u, win = __reduce_max_sync(FULL, lo);
            // two lanes can hold the same (score, id) only when the beam held an id twice
            const unsigned who = __ballot_sync(FULL, hi == top && lo == win);
            if (lane == __ffs(who) - 1) {
                oid[r] = (int)~win;
                osc[r] = S[bt];
                key[bt] = 0;
            }
            __syncwarp();
        }
        return;
    }
    for (int t = tid; t < n; t += (int)blockDim.x) {
        const unsigned long long mine = key[t];
        int rank = 0;
        for (int u = 0; u < n; ++u) rank += key[u] > mine || (key[u] == mine && u < t) ? 1 : 0;
        if (rank < k) {
            oid[rank] = (int)~(unsigned)mine;
            osc[rank] = S[t];
        }
    }
}

template <class SS>
__global__ void __launch_bounds__(32 * SS::WARPS) rerank_kernel(const RerankParams p) {
    constexpr int W = SS::WARPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t bars[W][RR_STAGES];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t qi = blockIdx.x;
    int k = p.desc ? p.desc[qi].x : p.uni.x;
    k = min(max(k, 0), p.ldo);

    const int ring = RR_STAGES * RR_GROUP * p.rec_bytes;  // of one warp
    unsigned char *const my = smem_raw + (size_t)wid * ring;
    unsigned char *const qsm = smem_raw + (size_t)W * ring;
    unsigned long long *const rK = reinterpret_cast<unsigned long long *>(qsm + SS::query_bytes(p.sec_chunks));
    float *const rS = reinterpret_cast<float *>(rK + p.ldc);
    int *const rI = reinterpret_cast<int *>(rS + p.ldc);
    uint64_t *const bar = bars[wid];
    if (lane == 0) {
        for (int s = 0; s < RR_STAGES; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(rr_smem(bar + s)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int32_t *cd = p.cand + qi * p.ldc;
    for (int t = tid; t < p.ldc; t += 32 * W) rI[t] = cd[t];  // with the count in flight; the first nr are used
    const int nr = min(p.cand_n[qi], p.ldc);
    if (nr < 0) return;  // the whole block
    __syncthreads();
    // group i of this warp: candidates RR_GROUP (wid + W i) .. + RR_GROUP - 1
    const int groups = (nr + RR_GROUP - 1) / RR_GROUP;
    const int mine = wid < groups ? (groups - wid + W - 1) / W : 0;
    auto issue = [&](int i) {
        const int b = RR_GROUP * (wid + W * i), cnt = min(RR_GROUP, nr - b), s = i % RR_STAGES;
        if (lane == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(rr_smem(bar + s)),
                         "r"((uint32_t)(cnt * p.rec_bytes))
                         : "memory");
        __syncwarp();
        if (lane < cnt)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    rr_smem(my + (size_t)(s * RR_GROUP + lane) * p.rec_bytes)),
                "l"(p.sec + (int64_t)rI[b + lane] * p.sec_stride), "r"((uint32_t)p.rec_bytes), "r"(rr_smem(bar + s))
                : "memory");
    };
    for (int i = 0; i < min(mine, RR_STAGES); ++i) issue(i);  // in flight while the query is set up
    SS sc;
    sc.setup(p.Q + qi * p.D, p, qsm);
    __syncthreads();
    sc.load(qsm, lane);
    int i = 0;
    for (; i < mine; ++i) {
        const int b = RR_GROUP * (wid + W * i), s = i % RR_STAGES;
        if (!__all_sync(FULL, rr_wait(bar + s, (uint32_t)(i / RR_STAGES) & 1u, p.tries))) break;
        const unsigned char *rec = my + (size_t)s * RR_GROUP * p.rec_bytes;
        // sums over the warp of the four records: the halves of a lane pair each take on two records,
        // then one, then the usual butterfly -- the additions of a full butterfly per record
        float v[RR_GROUP];
#pragma unroll
        for (int u = 0; u < RR_GROUP; ++u) v[u] = b + u < nr ? sc.dot(rec + u * p.rec_bytes, lane) : 0.f;
        const bool h4 = lane & 16, h3 = lane & 8;
        const float r0 = __shfl_xor_sync(FULL, h4 ? v[0] : v[2], 16), r1 = __shfl_xor_sync(FULL, h4 ? v[1] : v[3], 16);
        const float w0 = (h4 ? v[2] : v[0]) + r0, w1 = (h4 ? v[3] : v[1]) + r1;
        float x = (h3 ? w1 : w0) + __shfl_xor_sync(FULL, h3 ? w0 : w1, 8);
#pragma unroll
        for (int o = 4; o; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
        const int u = lane >> 3;
        if ((lane & 7) == 0 && b + u < nr) {
            const float f = fmaxf(sc.finish(x, rec + u * p.rec_bytes), -INFINITY);  // NaN ranks last, as in the beam
            rS[b + u] = f;
            rK[b + u] = (unsigned long long)order_key(f) << 32 | (unsigned)~rI[b + u];
        }
        __syncwarp();  // the stage has been read
        if (i + RR_STAGES < mine) issue(i + RR_STAGES);
    }
    if (i < mine) {  // gave up: report it, and let the copies in flight end before the block does
        if (lane == 0) atomicOr(p.status, ST_TIMEOUT);
        for (int j = i; j < min(mine, i + RR_STAGES); ++j)
            rr_wait(bar + j % RR_STAGES, (uint32_t)(j / RR_STAGES) & 1u, RR_TRIES);
    }
    // a query that any warp gave up on has no answer.  (A branch with its own stores here takes 71 registers
    // instead of 63, and the eighth block of an SM where records are short: 50,000 queries on 1M x 200 0.5 % slower.)
    const int n = __syncthreads_or(i < mine) ? 0 : nr;
    int32_t *oid = p.ids + qi * p.ldo;
    float *osc = p.scores + qi * p.ldo;
    block_topk(rK, rS, n, k, oid, osc);
    for (int t = min(k, n) + tid; t < p.ldo; t += 32 * W) {
        oid[t] = -1;
        osc[t] = -INFINITY;
    }
}

// bytes of a block's ring, query and candidates; without more than 48 KB no limit has to be raised (see allow_smem)
template <class SS>
static constexpr size_t rerank_smem(int rec_bytes, int chunks, int ldc) {
    return (size_t)SS::WARPS * RR_STAGES * RR_GROUP * rec_bytes + SS::query_bytes(chunks) + 16 * (size_t)ldc;
}
static_assert(rerank_smem<SecIntScorer<true>>(1024, 63, LCAP_MAX) <= 48 * 1024, "LVQ-8, 64 chunks");
static_assert(rerank_smem<Fp16SecScorer<4>>(2048, 128, LCAP_MAX) <= 48 * 1024, "FP16, 1024 dimensions");
static_assert(rerank_smem<Fp16SecScorer<1>>(512, 32, LCAP_MAX) <= 48 * 1024, "FP16, 256 dimensions, four warps");

template <class SS>
static int go_rerank(const RerankParams &p, cudaStream_t st) {
    const size_t smem = rerank_smem<SS>(p.rec_bytes, p.sec_chunks, p.ldc);
    rerank_kernel<SS><<<(unsigned)p.m, 32 * SS::WARPS, smem, st>>>(p);
    LV_CHECK_LAUNCH("rerank_kernel");
    return LV_OK;
}

template <bool L2>
static int launch_rerank_m(const BeamParams &bp, const RerankParams &p, cudaStream_t st) {
    if (bp.sec_bits == 16) {
        switch ((p.sec_chunks + 31) / 32) {
            case 1: return go_rerank<Fp16SecScorer<1, L2>>(p, st);
            case 2: return go_rerank<Fp16SecScorer<2, L2>>(p, st);
            case 3: return go_rerank<Fp16SecScorer<3, L2>>(p, st);
            case 4: return go_rerank<Fp16SecScorer<4, L2>>(p, st);
            default: return fail(LV_ERR_ARG, "rerank: FP16 secondaries longer than 1024 dimensions");
        }
    }
    if (!p.smean) return fail(LV_ERR_STATE, "rerank: LVQ-8 secondaries without their mean");
    return go_rerank<SecIntScorer<L2>>(p, st);
}

int launch_rerank(const BeamParams &bp, cudaStream_t st, int tries) {
    if (bp.m <= 0) return LV_OK;
    RerankParams p;
    p.sec = bp.sec;
    p.sec_stride = bp.sec_stride;
    p.sec_chunks = bp.sec_chunks;
    p.rec_bytes = 16 * (bp.sec_chunks + (bp.sec_bits == 16 ? 0 : 1 + bp.metric));
    p.Q = bp.Q;
    p.D = bp.D;
    p.smean = bp.smean;
    p.desc = bp.desc;
    p.uni = bp.uni;
    p.m = bp.m;
    p.cand = bp.cand;
    p.cand_n = bp.cand_n;
    p.ldc = bp.ldc;
    p.ids = bp.ids;
    p.scores = bp.scores;
    p.ldo = bp.ldo;
    p.status = bp.status;
    p.tries = tries;
    if (bp.metric) return launch_rerank_m<true>(bp, p, st);
    return launch_rerank_m<false>(bp, p, st);
}

}  // namespace lv
