// The nout leading eigenpairs of a symmetric FP64 matrix.  LeanVec-ID (Sec. 2.1) and the
// eigenvector search (Algorithm 2) use only the d leading eigenvectors of a D x D second moment,
// so instead of diagonalising the whole matrix (cyclic Jacobi, fit.cu) this path
//   1. reduces K to tridiagonal form T = Q^T K Q by D - 2 Householder reflections (one persistent
//      kernel, all SMs, one grid barrier per reflection);
//   2. finds the nout largest eigenvalues of T by multisection on Sturm counts (two warps each);
//   3. finds their eigenvectors of T by inverse iteration on the pivoted tridiagonal factorisation
//      of T - lambda I, with Gram-Schmidt inside clusters of close eigenvalues (one block per
//      cluster);
//   4. maps them back through the reflections (x = Q z, one block per eigenvector) and fixes the
//      sign (largest-magnitude entry positive, first index on ties).
// FP64, with float32 only where FP64 decides the result: three rounds of the multisection narrow an interval
// whose ends an FP64 round then checks.  Reciprocals and roots as in fp64.cuh.  Every grid-wide wait is
// bounded: a block that waits too long records ST_TIMEOUT and returns.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "fp64.cuh"

namespace lv {

constexpr int TRI_THREADS = 256, TRI_WARPS = TRI_THREADS / 32;
constexpr long long TRI_SPIN = 1ll << 25;  // with a 64 ns sleep per try: a give-up within seconds
constexpr int EIGH_TOP_MAX_D = 4096;

__device__ __forceinline__ double warp_sum_d(double x) {
#pragma unroll
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

// sum over the block in a fixed order (the same in every block for the same data)
__device__ double block_sum_d(double x, double *red) {
    x = warp_sum_d(x);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    double t = 0.0;
    const int nw = blockDim.x >> 5;
    for (int i = 0; i < nw; ++i) t += red[i];
    __syncthreads();
    return t;
}

// Grid barrier on a cumulative arrival counter: barrier number `target` completes when
// gridDim.x * target blocks have arrived.  False when this block gave up waiting.
__device__ bool grid_barrier(unsigned *count, volatile unsigned *gen, unsigned &target) {
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        ++target;
        __threadfence();
        const unsigned arrived = atomicAdd(count, 1u) + 1u;
        if (arrived == gridDim.x * target) {
            __threadfence();
            atomicExch(const_cast<unsigned *>(gen), target);
        } else {
            long long it = 0;
            while (*gen < target) {
                if (++it > TRI_SPIN) {
                    ok = 0;
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// The grid barrier again, polled without sleeping on the arrival counter itself.
__device__ bool grid_barrier_spin(unsigned *count, unsigned &target) {
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        target += gridDim.x;
        unsigned seen;
        asm volatile("atom.add.release.gpu.global.u32 %0, [%1], 1;" : "=r"(seen) : "l"(count) : "memory");
        ++seen;
        for (int it = 0; seen < target; ++it) {
            if (it > (1 << 22)) {  // about a second
                ok = 0;
                break;
            }
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// sum over the block of TS_T threads in a fixed order, in every thread; `slot` alternates between calls
constexpr int TS_T = 128, TS_W = TS_T / 32;
__device__ __forceinline__ double ts_block_sum(double x, double (*red)[TS_W], int slot) {
    x = warp_sum_d(x);
    if ((threadIdx.x & 31) == 0) red[slot][threadIdx.x >> 5] = x;
    __syncthreads();
    return (red[slot][0] + red[slot][1]) + (red[slot][2] + red[slot][3]);
}

// f(0), f(1), .. f(N - 1) with compile-time arguments.  The loops over a vector's register slots leave out
// the slots that hold no entry any more, and they do it at compile time: an FP64 instruction whose
// predicate is off still takes the pipe for its 64 cycles.
template <int I = 0, int N, class F>
__device__ __forceinline__ void phases(std::integral_constant<int, N> n, F &&f) {
    f(std::integral_constant<int, I>());
    if constexpr (I + 1 < N) phases<I + 1>(n, f);
}

// The tridiagonalisation of tridiag_kernel (below) with every block's rows kept in shared memory (row
// i in block i mod G, local row i / G) and the step's vectors in registers (entry tid + 128 u in
// slot u, zero where the step has no entry).  A step k then goes:
//   1. from step k - 1: p (entries by every block) and row k as it stood before that step's update,
//      published by its owner, both read from L2 at once; every block forms w, row k of A^(k), its
//      norm and v_k;
//   2. every block updates its rows with (v_{k-1}, w) and forms its entries of p = tau_k A^(k) v_k, all
//      four warps on four rows at a time, the sums by exchanging halves;
//   3. one grid barrier.
// D = 768: 9.08 ms (11.9 us a step) with rows in L2, eight warps a block that all took the step's root and
// divisions, and a sleeping barrier; 5.10 ms (6.7 us) now, of it about 1.2 us in the barrier, 1.7 in the
// two sums and the root, 1.4 in the rows.
template <int E>
__global__ void __launch_bounds__(TS_T) tridiag_sm_kernel(const double *__restrict__ K, int D, double *dg, double *ofd,
                                                           double *Hv, double *tau, double *pbuf, double *rowbuf,
                                                           unsigned *bar_count, int *status) {
    extern __shared__ double sh[];
    const int G = (int)gridDim.x, c = (int)blockIdx.x, nl = c < D ? (D - c + G - 1) / G : 0;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, maxl = (D + G - 1) / G;
    double *const A = sh;                        // maxl rows
    double *vp_s = A + (size_t)maxl * D;         // v_{k-1}, v_k and w of step k - 1 by row, for the own rows'
    double *vc_s = vp_s + D;                     // coefficients
    double *const w_s = vc_s + D;
    double *const part = w_s + D;                // TS_W x maxl partial sums of p
    __shared__ double red[2][TS_W], s_b[2];
    unsigned target = 0;
    for (int l = 0; l < nl; ++l)
        for (int j = tid; j < D; j += TS_T) A[(size_t)l * D + j] = K[(int64_t)(c + l * G) * D + j];
    double vp[E], vc[E], w[E], x[E];
#pragma unroll
    for (int u = 0; u < E; ++u) vp[u] = w[u] = 0.0;
    for (int j = tid; j < D; j += TS_T) vp_s[j] = w_s[j] = 0.0;
    double t = 0.0;
    bool alive = true;
    __syncthreads();
    // phase U0: the steps k with k / TS_T = U0; their vectors have entries in slots U0 .. E - 1
    phases(std::integral_constant<int, E>(), [&](auto u0c) {
        constexpr int U0 = decltype(u0c)::value;
        const int kend = min(D - 2, TS_T * (U0 + 1));
        for (int k = TS_T * U0; alive && k < kend; ++k) {
            const double *const pb = pbuf + (size_t)((k & 1) ^ 1) * D;      // p of step k - 1
            const double *const rb = k ? rowbuf + (size_t)(k & 1) * D : K;  // row k before its update
            // ---- w of step k - 1 and x = row k of A^(k) (v_{k-1}[k] = 1) ----
#pragma unroll
            for (int u = U0; u < E; ++u) {
                const int j = tid + TS_T * u;
                const bool in = j >= k && j < D;
                x[u] = in ? __ldcg(rb + j) : 0.0;
                w[u] = in && k ? __ldcg(pb + j) : 0.0;
            }
            if (k) {
                double pv = 0.0;
#pragma unroll
                for (int u = U0; u < E; ++u) pv = fma(w[u], vp[u], pv);
                if (tid + TS_T * U0 == k) s_b[0] = w[U0];
                pv = ts_block_sum(pv, red, 0);
                const double gam = 0.5 * t * pv, wk = s_b[0] - gam;
#pragma unroll
                for (int u = U0; u < E; ++u) {
                    w[u] = fma(-gam, vp[u], w[u]);
                    x[u] = fma(-wk, vp[u], x[u] - w[u]);
                }
            }
            double s = 0.0;
#pragma unroll
            for (int u = U0; u < E; ++u) {
                const int j = tid + TS_T * u;
                const double y = u > U0 + 1 || j >= k + 2 ? x[u] : 0.0;
                s = fma(y, y, s);
                if (j == k + 1) s_b[1] = x[u];
            }
            if (tid + TS_T * U0 == k && c == 0) dg[k] = x[U0];
            const double xn2 = ts_block_sum(s, red, 1), x0 = s_b[1];
            double beta = x0, scal = 0.0;
            t = 0.0;
            if (xn2 > 0.0) {
                const double S = fma(x0, x0, xn2);
                if (S > 1e-290 && S < 1e290) {
                    const double y = fast_rsqrt(S), b = S * y;
                    t = fma(fabs(x0), y, 1.0);  // (beta - x0) / beta with beta = -sign(x0) sqrt(S)
                    beta = -copysign(b, x0);
                    scal = copysign(fast_rcp(fabs(x0) + b), x0);
                } else {
                    beta = -copysign(sqrt(S), x0);
                    t = (beta - x0) / beta;
                    scal = 1.0 / (x0 - beta);
                }
            }
#pragma unroll
            for (int u = U0; u < E; ++u) {
                const int j = tid + TS_T * u;
                vc[u] = x[u] * scal;
                if (u <= U0 + 1) vc[u] = j == k + 1 ? 1.0 : j > k ? vc[u] : 0.0;
                if (j > k && j < D) {
                    vc_s[j] = vc[u];
                    w_s[j] = w[u];
                    if (c == 0) Hv[(int64_t)k * D + j] = vc[u];
                }
            }
            if (c == 0 && tid == 0) {
                tau[k] = t;
                ofd[k] = beta;
            }
            __syncthreads();
            // ---- own rows i > k: the pending update, then p_i = t (row_i . v_k); NR rows at a time ----
            const int l0 = k >= c ? (k - c) / G + 1 : 0;
            auto pass = [&](auto nrc, int lc) {
                constexpr int NR = decltype(nrc)::value;
                double acc[4] = {}, vi[NR], wi[NR];
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    vi[r] = vp_s[c + (lc + r) * G];
                    wi[r] = w_s[c + (lc + r) * G];
                }
                const bool pub = c + lc * G == k + 1;  // the next pivot row is always the first one left
                double *const base = A + (size_t)lc * D + tid;
                double *const prow = rowbuf + (size_t)((k + 1) & 1) * D + tid;
#pragma unroll
                for (int u = U0; u < E; ++u) {
                    const bool in = tid + TS_T * u < D;
                    double a[NR];
#pragma unroll
                    for (int r = 0; r < NR; ++r) a[r] = in ? base[(size_t)r * D + TS_T * u] : 0.0;
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        a[r] = fma(-vi[r], w[u], a[r]);
                        a[r] = fma(-wi[r], vp[u], a[r]);
                        acc[r] = fma(a[r], vc[u], acc[r]);
                        if (in) base[(size_t)r * D + TS_T * u] = a[r];
                    }
                    if (pub && in) __stcg(prow + TS_T * u, a[0]);
                }
                // sums over the warp: with four rows lane's row is 2 (bit 4) + (bit 3), with two bit 4
                const bool h4 = lane & 16, h3 = lane & 8;
                double y;
                int row = 0;
                if constexpr (NR == 4) {
                    const double a0 = (h4 ? acc[2] : acc[0]) + __shfl_xor_sync(FULL, h4 ? acc[0] : acc[2], 16);
                    const double a1 = (h4 ? acc[3] : acc[1]) + __shfl_xor_sync(FULL, h4 ? acc[1] : acc[3], 16);
                    y = (h3 ? a1 : a0) + __shfl_xor_sync(FULL, h3 ? a0 : a1, 8);
                    row = (h4 ? 2 : 0) + (h3 ? 1 : 0);
                } else {
                    if constexpr (NR == 2) {
                        y = (h4 ? acc[1] : acc[0]) + __shfl_xor_sync(FULL, h4 ? acc[0] : acc[1], 16);
                        row = h4 ? 1 : 0;
                    } else {
                        y = acc[0] + __shfl_xor_sync(FULL, acc[0], 16);
                    }
                    y += __shfl_xor_sync(FULL, y, 8);
                }
#pragma unroll
                for (int o = 4; o; o >>= 1) y += __shfl_xor_sync(FULL, y, o);
                if ((lane & (NR == 4 ? 7 : NR == 2 ? 15 : 31)) == 0) part[wid * maxl + lc + row] = y;
            };
            int lc = l0;
            for (; lc + 4 <= nl; lc += 4) pass(std::integral_constant<int, 4>(), lc);
            if (lc + 2 <= nl) {
                pass(std::integral_constant<int, 2>(), lc);
                lc += 2;
            }
            if (lc < nl) pass(std::integral_constant<int, 1>(), lc);
            __syncthreads();
            for (int l = l0 + tid; l < nl; l += TS_T)
                __stcg(pbuf + (size_t)(k & 1) * D + c + l * G,
                       t * ((part[l] + part[maxl + l]) + (part[2 * maxl + l] + part[3 * maxl + l])));
            if (!grid_barrier_spin(bar_count, target)) {
                if (tid == 0) atomicOr(status, ST_TIMEOUT);
                alive = false;  // the whole block
            }
            // v_k becomes v_{k-1}
            double *const o = vp_s;
            vp_s = vc_s;
            vc_s = o;
#pragma unroll
            for (int u = U0; u < E; ++u) vp[u] = vc[u];
        }
    });
    if (!alive) return;
    // the last 2 x 2 block: row a from its owner's published copy, the corner from the owner itself
    const int a = D - 2, b = D - 1, k = D - 2;
    const double *const pb = pbuf + (size_t)((k & 1) ^ 1) * D, *const rb = rowbuf + (size_t)(k & 1) * D;
    if (tid == 0) {
        const double va = vp_s[a], vb = vp_s[b], pa = __ldcg(pb + a), pbb = __ldcg(pb + b), pv = fma(pa, va, pbb * vb);
        const double gam = 0.5 * t * pv, wa = fma(-gam, va, pa), wb = fma(-gam, vb, pbb);
        if (c == 0) {
            dg[a] = __ldcg(rb + a) - 2.0 * va * wa;
            ofd[a] = __ldcg(rb + b) - va * wb - wa * vb;
            tau[a] = 0.0;
        }
        if (b % G == c) dg[b] = A[(size_t)(b / G) * D + b] - 2.0 * vb * wb;
    }
}

// Householder tridiagonalisation of the symmetric D x D matrix A (device, full storage).  Reflection
// k (k = 0 .. D - 3) maps the column below the diagonal, x = A^(k)[k + 1 .., k], to (beta, 0, ..):
// H_k = I - tau_k v_k v_k^T with v_k[0] = 1, stored as Hv[k][k + 1 ..].  The trailing matrix
// changes by A^(k+1) = A^(k) - v w^T - w v^T with p = tau A^(k) v, w = p - (tau / 2)(p . v) v.
// That update is applied one step late, inside the next step's pass over the rows, so that a
// step needs one grid barrier: step k rebuilds row k of A^(k) from the stored row and the pending
// (v, w) of step k - 1, forms v_k, then each block updates its rows (owner = row % gridDim.x, one
// warp per row), writes them back and forms their entries of p = tau_k A^(k) v_k; after the barrier
// every block forms w_k.  Outputs: diagonal dg (D), off-diagonal ofd (D - 1), Hv, tau.  Everything
// that crosses blocks goes through L2 (ld.cg / st.cg).
__global__ void __launch_bounds__(TRI_THREADS) tridiag_kernel(double *A, int D, double *dg, double *ofd,
                                                               double *Hv, double *tau, double *pbuf,
                                                               unsigned *bar_count, unsigned *bar_gen, int *status) {
    extern __shared__ double sh[];
    double *vp = sh, *wp = sh + D, *vc = sh + 2 * D, *red = sh + 3 * D;  // global row indices
    const int G = (int)gridDim.x, c = (int)blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    unsigned target = 0;
    for (int g = tid; g < D; g += TRI_THREADS) vp[g] = wp[g] = 0.0;
    __syncthreads();
    for (int k = 0; k + 2 < D; ++k) {
        const double *rowk = A + (int64_t)k * D;
        const double vk = vp[k], wk = wp[k];
        // x_j = A^(k)[k][j], j > k: the stored row k with step k - 1's update
        double s = 0.0;
        for (int j = k + 2 + tid; j < D; j += TRI_THREADS) {
            const double xj = __ldcg(rowk + j) - vk * wp[j] - wk * vp[j];
            vc[j] = xj;
            s = fma(xj, xj, s);
        }
        const double xn2 = block_sum_d(s, red);
        const double x0 = __ldcg(rowk + k + 1) - vk * wp[k + 1] - wk * vp[k + 1];
        double beta = x0, t = 0.0, scal = 0.0;
        if (xn2 > 0.0) {
            beta = -copysign(sqrt(fma(x0, x0, xn2)), x0);
            t = (beta - x0) / beta;
            scal = 1.0 / (x0 - beta);
        }
        for (int j = k + 1 + tid; j < D; j += TRI_THREADS) vc[j] = j == k + 1 ? 1.0 : vc[j] * scal;
        __syncthreads();
        if (c == 0) {
            for (int j = k + 1 + tid; j < D; j += TRI_THREADS) Hv[(int64_t)k * D + j] = vc[j];
            if (tid == 0) {
                tau[k] = t;
                ofd[k] = beta;
                dg[k] = __ldcg(rowk + k) - 2.0 * vk * wk;
            }
        }
        // rows i > k of this block: apply step k - 1's update, store, p_i = t (row_i . v_k)
        const int first = k + 1 + (((c - (k + 1)) % G) + G) % G;
        for (int i = first + wid * G; i < D; i += TRI_WARPS * G) {
            double *ar = A + (int64_t)i * D;
            const double vi = vp[i], wi = wp[i];
            double acc = 0.0;
            for (int j = k + 1 + lane; j < D; j += 32) {
                const double a = __ldcg(ar + j) - vi * wp[j] - wi * vp[j];
                __stcg(ar + j, a);
                acc = fma(a, vc[j], acc);
            }
            acc = warp_sum_d(acc);
            if (lane == 0) __stcg(pbuf + i, t * acc);
        }
        if (!grid_barrier(bar_count, bar_gen, target)) {
            if (tid == 0) atomicOr(status, ST_TIMEOUT);
            return;
        }
        // w_k = p - (t / 2)(p . v_k) v_k, pending for the next step
        double pv = 0.0;
        for (int j = k + 1 + tid; j < D; j += TRI_THREADS) pv = fma(__ldcg(pbuf + j), vc[j], pv);
        pv = block_sum_d(pv, red);
        const double gam = 0.5 * t * pv;
        for (int j = k + 1 + tid; j < D; j += TRI_THREADS) {
            wp[j] = fma(-gam, vc[j], __ldcg(pbuf + j));
            vp[j] = vc[j];
        }
        __syncthreads();
    }
    if (c == 0 && tid == 0) {
        const int a = D - 2, b2 = D - 1;
        dg[a] = __ldcg(A + (int64_t)a * D + a) - 2.0 * vp[a] * wp[a];
        ofd[a] = __ldcg(A + (int64_t)a * D + b2) - vp[a] * wp[b2] - wp[a] * vp[b2];
        dg[b2] = __ldcg(A + (int64_t)b2 * D + b2) - 2.0 * vp[b2] * wp[b2];
        tau[a] = 0.0;
    }
}

// number of eigenvalues of T below x: negative pivots of T - x I (e2: squared off-diagonals).  The pivot's
// reciprocal is fast_rcp; signs and the pivot floor are read off the high word, which costs no FP64
// instruction: five of them a pivot instead of about twelve.
__device__ __forceinline__ int sturm_below(const double *dg, const double *e2, int D, double x, double pivmin) {
    const int ph = __double2hiint(pivmin);
    double q = dg[0] - x;
    int neg = 0;
#pragma unroll 4
    for (int j = 1; j < D; ++j) {
        const int h = __double2hiint(q);
        if ((h & 0x7fffffff) < ph) q = -pivmin;
        neg -= __double2hiint(q) >> 31;
        q = fma(-e2[j - 1], fast_rcp(q), dg[j] - x);
    }
    if ((__double2hiint(q) & 0x7fffffff) < ph) q = -pivmin;
    return neg - (__double2hiint(q) >> 31);
}
// the same in float32 for T / ||T||: the counts of a matrix within about 1e-6 ||T|| of T
__device__ __forceinline__ int sturm_below_f(const float *dg, const float *e2, int D, float x) {
    float q = dg[0] - x;
    int neg = 0;
#pragma unroll 4
    for (int j = 1; j < D; ++j) {
        if (fabsf(q) < 1e-30f) q = -1e-30f;
        neg += q < 0.f;
        q = dg[j] - x - __fdividef(e2[j - 1], q);
    }
    return neg + (q < 0.f);
}

// lam[i] = the (i + 1)-th largest eigenvalue of T, i < nout; one block of two warps per eigenvalue.
// Multisection: a round counts at 63 points of [lo, hi] and keeps the interval around the change of
// "at least i + 1 eigenvalues at or above".  float32 rounds narrow the interval to about 1e-5 ||T|| first
// (a float32 count takes a seventh of the time); the first FP64 round then checks both its ends and
// falls back to the Gershgorin interval's part beyond an end that does not hold.
// 160 eigenvalues of D = 768: 4.93 ms with 31 points, FP64 throughout and a division a pivot; 1.31 ms now.
__global__ void __launch_bounds__(64) bisect_kernel(const double *dg, const double *ofd, int D, int nout, double lo0,
                                                    double hi0, double pivmin, double *lam) {
    extern __shared__ double sb[];
    double *const sd = sb, *const se = sb + D;
    float *const fd = reinterpret_cast<float *>(se + D), *const fe = fd + D;
    __shared__ unsigned s_bal[2][2];
    const int i = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const double norm = fmax(fabs(lo0), fabs(hi0)), inv = 1.0 / norm;
    for (int j = tid; j < D; j += 64) {
        const double d = dg[j], e = j + 1 < D ? ofd[j] : 0.0;
        sd[j] = d;
        se[j] = e * e;
        fd[j] = (float)(d * inv);
        const float ef = (float)(e * inv);
        fe[j] = ef * ef;
    }
    __syncthreads();
    int buf = 0;
    // number of leading true predicates of the 64 threads (they form a prefix)
    auto prefix = [&](bool pred) {
        const unsigned bal = __ballot_sync(FULL, pred);
        if (lane == 0) s_bal[buf][wid] = bal;
        __syncthreads();
        const int n0 = __popc(s_bal[buf][0]);
        const int n = n0 < 32 ? n0 : 32 + __popc(s_bal[buf][1]);
        buf ^= 1;
        return n;
    };
    auto point = [&](double lo, double hi, int p, int parts) { return lo + (hi - lo) * ((double)p / (double)parts); };
    double lo = lo0, hi = hi0;
    const bool scaled = norm > 1e-150 && norm < 1e150;
    if (scaled) {
        float l = (float)(lo0 * inv), h = (float)(hi0 * inv);
        for (int r = 0; r < 3; ++r) {
            auto at = [&](int p) { return l + (h - l) * ((float)p / 64.0f); };
            const int n = prefix(tid < 63 && D - sturm_below_f(fd, fe, D, at(tid + 1)) >= i + 1);
            const float nl = n > 0 ? at(n) : l, nh = n < 63 ? at(n + 1) : h;
            l = nl;
            h = nh;
        }
        const double g = 1e-5 * norm;
        const double cl = fmax(lo0, (double)l * norm - g), ch = fmin(hi0, (double)h * norm + g);
        const int n = prefix(D - sturm_below(sd, se, D, point(cl, ch, tid, 63), pivmin) >= i + 1);
        lo = n > 0 ? point(cl, ch, n - 1, 63) : lo0;
        hi = n < 64 ? point(cl, ch, n, 63) : hi0;
    }
    for (int round = 0; round < 64; ++round) {
        const double x = point(lo, hi, tid + 1, 64);
        bool pred;
        if (tid == 63 || x >= hi)
            pred = false;
        else if (x <= lo)
            pred = true;
        else
            pred = D - sturm_below(sd, se, D, x, pivmin) >= i + 1;
        const int n = prefix(pred);
        const double nlo = n > 0 ? fmax(lo, point(lo, hi, n, 64)) : lo, nhi = n < 63 ? fmin(hi, point(lo, hi, n + 1, 64)) : hi;
        if (nlo == lo && nhi == hi) break;
        lo = nlo;
        hi = nhi;
    }
    if (tid == 0) lam[i] = 0.5 * (lo + hi);
}

// a deterministic start vector entry in [-1, 1)
__device__ __forceinline__ double start_entry(int i, int e) {
    unsigned h = (unsigned)i * 0x9E3779B1u ^ ((unsigned)e + 0x7F4A7C15u) * 0x85EBCA77u;
    h ^= h >> 15;
    h *= 0x2C1B3C6Du;
    h ^= h >> 12;
    return (double)(h >> 8) * (2.0 / 16777216.0) - 1.0;
}

// Inverse iteration, one block per cluster [cb[c], ce[c]) of eigenvalues (descending, close ones
// together).  For eigenvalue e: T - lam I = P L U by Gaussian elimination with partial pivoting
// (thread 0; pivots below tol replaced by +-tol, kept as reciprocals), then: solve, orthogonalise
// against the cluster's earlier vectors (modified Gram-Schmidt), normalise -- three rounds (the
// eigenvalue is accurate to the last bits, so one solve already nearly converges).  Z: nout x D.
// The factors and the vector sit in shared memory and the recurrences in registers, so that a chain step
// costs its FP64 instructions alone; three warps a block, so that the chains of two blocks on an SM
// fall on different schedulers: 160 vectors of D = 768 1.15 ms with the factors in L2 and two
// divisions a row, 0.69 ms now.
__global__ void __launch_bounds__(96) inviter_kernel(const double *dg, const double *ofd, int D, const double *lam,
                                                      const int *cb, const int *ce, double tol, double *Z) {
    extern __shared__ double si[];
    __shared__ double red[4];
    const int c = blockIdx.x, tid = threadIdx.x;
    double *const mu = si, *const iv = mu + D, *const du = iv + D, *const du2 = du + D, *const x = du2 + D;
    unsigned char *const piv = reinterpret_cast<unsigned char *>(x + D);
    auto mag = [](double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; };  // orders like |v|
    for (int e = cb[c]; e < ce[c]; ++e) {
        // distinct shifts inside a cluster (equal eigenvalues would give the same vector)
        double le = lam[e];
        if (e > cb[c]) le = fmin(le, lam[e - 1] - 4.0 * DBL_EPSILON * fabs(lam[e - 1]) - tol * 1e-3);
        // T in place of what it will be replaced by: iv = diagonal - lam, mu = off-diagonal
        for (int j = tid; j < D; j += blockDim.x) {
            iv[j] = dg[j] - le;
            mu[j] = j + 1 < D ? ofd[j] : 0.0;
            x[j] = start_entry(j, e);
        }
        __syncthreads();
        if (tid == 0) {
            double d = iv[0], u = mu[0];  // the current row's diagonal and superdiagonal
            const long long tm = mag(tol);
            for (int j = 0; j + 1 < D; ++j) {
                const double l = mu[j], dn = iv[j + 1], un = mu[j + 1];
                if (mag(d) >= mag(l) || mag(l) < tm) {
                    if (mag(d) < tm) d = d < 0.0 ? -tol : tol;
                    const double r = fast_rcp(d), m = l * r;
                    mu[j] = m;
                    iv[j] = r;
                    du[j] = u;
                    du2[j] = 0.0;
                    piv[j] = 0;
                    d = fma(-m, u, dn);
                    u = un;
                } else {
                    const double r = fast_rcp(l), m = d * r;
                    mu[j] = m;
                    iv[j] = r;
                    du[j] = dn;
                    du2[j] = un;
                    piv[j] = 1;
                    d = fma(-m, dn, u);
                    u = -m * un;
                }
            }
            if (mag(d) < tm) d = d < 0.0 ? -tol : tol;
            iv[D - 1] = fast_rcp(d);
        }
        __syncthreads();
        for (int round = 0; round < 3; ++round) {
            if (tid == 0) {
                double cur = x[0];
#pragma unroll 4
                for (int j = 0; j + 1 < D; ++j) {
                    const double nx = x[j + 1], m = mu[j];
                    const bool p = piv[j];
                    const double keep = p ? nx : cur, other = p ? cur : nx;
                    x[j] = keep;
                    cur = fma(-m, keep, other);
                }
                double x1 = cur * iv[D - 1], x2 = 0.0;
                x[D - 1] = x1;
#pragma unroll 4
                for (int j = D - 2; j >= 0; --j) {
                    const double v = fma(-du[j], x1, fma(-du2[j], x2, x[j])) * iv[j];
                    x[j] = v;
                    x2 = x1;
                    x1 = v;
                }
            }
            __syncthreads();
            for (int f = cb[c]; f < e; ++f) {
                const double *zf = Z + (size_t)f * D;
                double s = 0.0;
                for (int i = tid; i < D; i += blockDim.x) s = fma(zf[i], x[i], s);
                s = block_sum_d(s, red);
                for (int i = tid; i < D; i += blockDim.x) x[i] = fma(-s, zf[i], x[i]);
                __syncthreads();
            }
            double s = 0.0;
            for (int i = tid; i < D; i += blockDim.x) s = fma(x[i], x[i], s);
            s = block_sum_d(s, red);
            const double inv = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
            for (int i = tid; i < D; i += blockDim.x) x[i] *= inv;
            __syncthreads();
        }
        double *ze = Z + (size_t)e * D;
        for (int i = tid; i < D; i += blockDim.x) ze[i] = x[i];
        __syncthreads();
    }
}

template <int T>
__device__ __forceinline__ double bt_block_sum(double x, double (*red)[T / 32], int slot) {
    x = warp_sum_d(x);
    if ((threadIdx.x & 31) == 0) red[slot][threadIdx.x >> 5] = x;
    __syncthreads();
    double s = red[slot][0];
#pragma unroll
    for (int w = 1; w < T / 32; ++w) s += red[slot][w];
    return s;
}

// evecs[r] = Q z_r = H_0 H_1 .. H_{D-3} z_r, unit norm, largest-magnitude entry positive (first
// index on ties); evals[r] = lam[r] (evals nullable).  One block of T threads per eigenvector, its
// entries in registers (tid + T u), the next reflection's vector loaded while the current one's sum goes
// round: 160 vectors of D = 768 2.04 ms with one warp per vector, 1.12 ms with the slots below the
// reflection predicated off instead of left out, 0.87 ms now.
template <int T, int E>
__global__ void __launch_bounds__(T) backtrans_kernel(const double *__restrict__ Z, const double *__restrict__ Hv,
                                                         const double *__restrict__ tau, int D, const double *lam,
                                                         double *evals, double *evecs) {
    __shared__ double red[2][(T / 32)];
    __shared__ double s_best[(T / 32)];
    __shared__ int s_bi[(T / 32)];
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double x[E], v[E];
#pragma unroll
    for (int u = 0; u < E; ++u) x[u] = tid + T * u < D ? Z[(size_t)r * D + tid + T * u] : 0.0;
    auto fetch = [&](int k) {
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int j = tid + T * u;
            v[u] = k >= 0 && j > k && j < D ? __ldg(Hv + (int64_t)k * D + j) : 0.0;
        }
    };
    fetch(D - 3);
    // phase U0, from the last: the reflections k with (k + 1) / T = U0, whose entries sit in slots U0 ..
    phases(std::integral_constant<int, E>(), [&](auto ic) {
        constexpr int U0 = E - 1 - decltype(ic)::value;
        for (int k = min(D - 3, T * (U0 + 1) - 2); k >= max(0, T * U0 - 1); --k) {
            double w[E], s = 0.0;
#pragma unroll
            for (int u = U0; u < E; ++u) {
                w[u] = v[u];
                s = fma(w[u], x[u], s);
            }
            const double t = __ldg(tau + k);
            fetch(k - 1);
            s = -bt_block_sum<T>(s, red, k & 1) * t;
#pragma unroll
            for (int u = U0; u < E; ++u) x[u] = fma(s, w[u], x[u]);
        }
    });
    double s = 0.0, best = -1.0;
    int bi = D;
#pragma unroll
    for (int u = 0; u < E; ++u) {
        s = fma(x[u], x[u], s);
        const double a = fabs(x[u]);
        if (tid + T * u < D && a > best) {
            best = a;
            bi = tid + T * u;
        }
    }
    __syncthreads();
    s = bt_block_sum<T>(s, red, 0);
    // largest |x_i|, first index on ties
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        const double ob = __shfl_xor_sync(FULL, best, o);
        const int oi = __shfl_xor_sync(FULL, bi, o);
        if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
        }
    }
    if (lane == 0) {
        s_best[wid] = best;
        s_bi[wid] = bi;
    }
    __syncthreads();
    for (int w = 0; w < (T / 32); ++w)
        if (s_best[w] > best || (s_best[w] == best && s_bi[w] < bi)) {
            best = s_best[w];
            bi = s_bi[w];
        }
    __shared__ double s_sign;
#pragma unroll
    for (int u = 0; u < E; ++u)
        if (tid + T * u == bi) s_sign = x[u] < 0.0 ? -1.0 : 1.0;
    __syncthreads();
    const double scale = (s > 0.0 ? 1.0 / sqrt(s) : 0.0) * (bi < D ? s_sign : 1.0);
#pragma unroll
    for (int u = 0; u < E; ++u)
        if (tid + T * u < D) evecs[(size_t)r * D + tid + T * u] = x[u] * scale;
    if (tid == 0 && evals) evals[r] = lam[r];
}

static int launch_backtrans(const double *Z, const double *Hv, const double *tau, int D, int nout, const double *lam,
                            double *evals, double *evecs, cudaStream_t st) {
    auto go = [&](auto k, int threads) -> int {
        k<<<nout, threads, 0, st>>>(Z, Hv, tau, D, lam, evals, evecs);
        LV_CHECK_LAUNCH("backtrans_kernel");
        return LV_OK;
    };
    if (D <= 256) return go(backtrans_kernel<128, 2>, 128);
    if (D <= 512) return go(backtrans_kernel<128, 4>, 128);
    if (D <= 768) return go(backtrans_kernel<128, 6>, 128);
    if (D <= 1024) return go(backtrans_kernel<128, 8>, 128);
    if (D <= 2048) return go(backtrans_kernel<128, 16>, 128);
    return go(backtrans_kernel<128, 32>, 128);
}

// the path applies: 8 <= D <= 4096, 1 <= nout <= D
bool eigh_top_ok(int D, int nout) { return D >= 8 && D <= EIGH_TOP_MAX_D && nout >= 1 && nout <= D; }

int eigh_top(const double *K, int D, int nout, double *evals, double *evecs, cudaStream_t st) {
    if (!eigh_top_ok(D, nout)) return fail(LV_ERR_ARG, "eigh_top: need 8 <= D <= 4096 and 1 <= nout <= D");
    double *A = nullptr, *Hv = nullptr, *tau = nullptr, *dg = nullptr, *ofd = nullptr, *pbuf = nullptr;
    double *lam = nullptr, *Z = nullptr, *rowbuf = nullptr;
    unsigned *bar = nullptr;
    int *status = nullptr, *cl = nullptr;
    int rc = LV_OK;
    const size_t DD = (size_t)D * D;
    std::vector<double> hd(D), he(D), hl(nout);
    std::vector<int> hcb, hce;
    int dev = 0, sms = 0, per_sm = 0, nclus = 0, hstatus = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return fail(LV_ERR_CUDA, "eigh_top: no device");
    // rows in shared memory while they fit (D <= about 1800); two rows a block at least
    const int gs = std::min(sms, (D + 1) / 2), maxl = (D + gs - 1) / gs;
    const size_t ssm = sizeof(double) * ((size_t)maxl * D + 3 * (size_t)D + (size_t)TS_W * maxl);
    const bool in_sm = ssm <= 220 * 1024 && D <= 16 * TS_T;
    const size_t tsm = sizeof(double) * (3 * (size_t)D + TRI_WARPS);
    const size_t bsm = 2 * sizeof(double) * (size_t)D + 2 * sizeof(float) * (size_t)D, ism = (5 * sizeof(double) + 1) * (size_t)D;
    if ((!in_sm && tmp_alloc((void **)&A, sizeof(double) * DD, st)) || tmp_alloc((void **)&Hv, sizeof(double) * DD, st) ||
        tmp_alloc((void **)&tau, sizeof(double) * D, st) || tmp_alloc((void **)&dg, sizeof(double) * D, st) ||
        tmp_alloc((void **)&ofd, sizeof(double) * D, st) || tmp_alloc((void **)&pbuf, sizeof(double) * 2 * D, st) ||
        tmp_alloc((void **)&rowbuf, sizeof(double) * 2 * D, st) ||
        tmp_alloc((void **)&lam, sizeof(double) * nout, st) || tmp_alloc((void **)&Z, sizeof(double) * nout * (size_t)D, st) ||
        tmp_alloc((void **)&bar, 2 * sizeof(unsigned), st) || tmp_alloc((void **)&status, sizeof(int), st)) {
        rc = fail(LV_ERR_OOM, "eigh_top: allocation failed");
        goto done;
    }
    if ((!in_sm && cudaMemcpyAsync(A, K, sizeof(double) * DD, cudaMemcpyDeviceToDevice, st) != cudaSuccess) ||
        cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st) != cudaSuccess ||
        cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) {
        rc = fail(LV_ERR_CUDA, "eigh_top: copy failed");
        goto done;
    }
    // 1. tridiagonal form: one block per SM, all co-resident (cooperative launch)
    {
        const void *kern = !in_sm            ? (const void *)tridiag_kernel
                           : D <= 2 * TS_T  ? (const void *)tridiag_sm_kernel<2>
                           : D <= 4 * TS_T  ? (const void *)tridiag_sm_kernel<4>
                           : D <= 6 * TS_T  ? (const void *)tridiag_sm_kernel<6>
                           : D <= 8 * TS_T  ? (const void *)tridiag_sm_kernel<8>
                                            : (const void *)tridiag_sm_kernel<16>;
        const size_t sm = in_sm ? ssm : tsm;
        const int threads = in_sm ? TS_T : TRI_THREADS, blocks = in_sm ? gs : sms;
        if (allow_smem(kern) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, sm) != cudaSuccess || per_sm < 1) {
            rc = fail(LV_ERR_CUDA, "eigh_top: cannot size the tridiagonalisation");
            goto done;
        }
        int Dv = D;
        unsigned *bar_gen = bar + 1;
        void *args_sm[] = {(void *)&K, &Dv, &dg, &ofd, &Hv, &tau, &pbuf, &rowbuf, &bar, &status};
        void *args_gl[] = {&A, &Dv, &dg, &ofd, &Hv, &tau, &pbuf, &bar, &bar_gen, &status};
        if (cudaLaunchCooperativeKernel(kern, dim3((unsigned)blocks), dim3((unsigned)threads), in_sm ? args_sm : args_gl,
                                        sm, st) != cudaSuccess) {
            cudaGetLastError();
            rc = fail(LV_ERR_CUDA, "eigh_top: tridiagonalisation launch failed");
            goto done;
        }
    }
    if (cudaMemcpyAsync(hd.data(), dg, sizeof(double) * D, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(he.data(), ofd, sizeof(double) * (D - 1), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&hstatus, status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        rc = fail(LV_ERR_CUDA, "eigh_top: tridiagonalisation failed");
        goto done;
    }
    if (hstatus) {
        rc = fail(LV_ERR_TIMEOUT, "eigh_top: a grid barrier of the tridiagonalisation timed out");
        goto done;
    }
    {
        // 2. eigenvalues: Gershgorin interval, pivot floor as in the usual Sturm-count bisection
        double lo = hd[0], hi = hd[0], e2max = 0.0;
        for (int j = 0; j < D; ++j) {
            const double r = (j > 0 ? fabs(he[j - 1]) : 0.0) + (j + 1 < D ? fabs(he[j]) : 0.0);
            lo = std::min(lo, hd[j] - r);
            hi = std::max(hi, hd[j] + r);
            if (j + 1 < D) e2max = std::max(e2max, he[j] * he[j]);
        }
        const double tnorm = std::max(fabs(lo), fabs(hi));
        const double pad = 4.0 * DBL_EPSILON * tnorm + DBL_MIN;
        lo -= pad;
        hi += pad;
        const double pivmin = DBL_MIN * std::max(1.0, e2max);
        if (allow_smem(bisect_kernel) != cudaSuccess ||
            allow_smem(inviter_kernel) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh_top: shared-memory attribute failed");
            goto done;
        }
        bisect_kernel<<<nout, 64, bsm, st>>>(dg, ofd, D, nout, lo, hi, pivmin, lam);
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(hl.data(), lam, sizeof(double) * nout, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh_top: bisection failed");
            goto done;
        }
        // 3. clusters: consecutive eigenvalues closer than 1e-5 ||T||
        const double ctol = 1e-5 * tnorm;
        for (int i = 0; i < nout; ++i) {
            if (i == 0 || hl[i - 1] - hl[i] > ctol) {
                hcb.push_back(i);
                hce.push_back(i + 1);
            } else {
                hce.back() = i + 1;
            }
        }
        nclus = (int)hcb.size();
        if (tmp_alloc((void **)&cl, sizeof(int) * 2 * nclus, st)) {
            rc = fail(LV_ERR_OOM, "eigh_top: allocation failed");
            goto done;
        }
        if (cudaMemcpyAsync(cl, hcb.data(), sizeof(int) * nclus, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaMemcpyAsync(cl + nclus, hce.data(), sizeof(int) * nclus, cudaMemcpyHostToDevice, st) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh_top: cluster copy failed");
            goto done;
        }
        const double tol = std::max(DBL_EPSILON * tnorm, DBL_MIN);
        inviter_kernel<<<nclus, 96, ism, st>>>(dg, ofd, D, lam, cl, cl + nclus, tol, Z);
        if (cudaGetLastError() != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh_top: inverse iteration launch failed");
            goto done;
        }
        // 4. back to K's basis
        if ((rc = launch_backtrans(Z, Hv, tau, D, nout, lam, evals, evecs, st))) goto done;
        if (cudaStreamSynchronize(st) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh_top: back-transformation failed");
            goto done;
        }
    }
done:
    tmp_free(A, st);
    tmp_free(Hv, st);
    tmp_free(tau, st);
    tmp_free(dg, st);
    tmp_free(ofd, st);
    tmp_free(pbuf, st);
    tmp_free(lam, st);
    tmp_free(Z, st);
    tmp_free(bar, st);
    tmp_free(status, st);
    tmp_free(cl, st);
    tmp_free(rowbuf, st);
    return rc;
}

}  // namespace lv

extern "C" int leanvec_eigh_top(const double *K, int D, int nout, double *evals, double *evecs, lv_stream_t stream) {
    if (!K || !evecs) return lv::fail(LV_ERR_ARG, "eigh_top: null pointer");
    return lv::eigh_top(K, D, nout, evals, evecs, (cudaStream_t)stream);
}
