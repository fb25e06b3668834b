// Learning the projections: second moments K = sum x x^T (Sec. 2.2 "Efficiency"),
// an FP64 symmetric eigensolver (cyclic Jacobi rotations, round-robin pair order so
// that the D/2 rotations of a round are independent), and LeanVec-ID (Sec. 2.1:
// A = B = the d leading eigenvectors of K_X).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <vector>

#include "common.cuh"
#include "fp64.cuh"

namespace lv {

// ------------------------------------------------------------ Gram matrix (FP32)
constexpr int GT = 64, GK = 32;

// K[a][b] = sum_i X[i][a] X[i][b]; 256 threads, 4 x 4 outputs per thread.
__global__ void __launch_bounds__(256) gram_fp32_kernel(const float *__restrict__ X, int64_t n, int D,
                                                        float *__restrict__ K) {
    __shared__ float As[GK][GT + 4];
    __shared__ float Bs[GK][GT + 4];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int a0 = blockIdx.y * GT, b0 = blockIdx.x * GT;
    float acc[4][4] = {};
    for (int64_t i0 = 0; i0 < n; i0 += GK) {
        for (int t = threadIdx.x; t < GK * GT; t += 256) {
            const int r = t / GT, c = t % GT;
            const int64_t gi = i0 + r;
            As[r][c] = (gi < n && a0 + c < D) ? X[gi * D + a0 + c] : 0.0f;
            Bs[r][c] = (gi < n && b0 + c < D) ? X[gi * D + b0 + c] : 0.0f;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < GK; ++kk) {
            float a[4], b[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = As[kk][ty * 4 + u];
#pragma unroll
            for (int v = 0; v < 4; ++v) b[v] = Bs[kk][tx * 4 + v];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = a0 + ty * 4 + u;
        if (r >= D) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int c = b0 + tx * 4 + v;
            if (c < D) K[(int64_t)r * D + c] = acc[u][v];
        }
    }
}

int launch_gram_fp32(const float *X, int64_t n, int D, float *K, cudaStream_t st) {
    dim3 grd((D + GT - 1) / GT, (D + GT - 1) / GT);
    gram_fp32_kernel<<<grd, 256, 0, st>>>(X, n, D, K);
    LV_CHECK_LAUNCH("gram_fp32_kernel");
    return LV_OK;
}

// ---------------------------------------------------------- FP64 Jacobi eigh
// Round r of the round-robin schedule on Dp (even) indices pairs slot i:
//   i = 0: (r, Dp - 1);  i > 0: ((r + i) mod (Dp - 1), (r - i) mod (Dp - 1)).
__device__ __forceinline__ void rr_pair(int r, int i, int Dp, int &p, int &q) {
    const int m = Dp - 1;
    if (i == 0) {
        p = r % m;
        q = m;
    } else {
        p = (r + i) % m;
        q = ((r - i) % m + m) % m;
    }
    if (p > q) {
        int t = p;
        p = q;
        q = t;
    }
}

// Rotation J (J_pp = J_qq = c, J_pq = s, J_qp = -s) that zeroes A'_pq of J^T A J.
__global__ void jacobi_rot_kernel(const double *__restrict__ A, int Dp, int r, double2 *__restrict__ cs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Dp / 2) return;
    int p, q;
    rr_pair(r, i, Dp, p, q);
    const double apq = A[(int64_t)p * Dp + q];
    double c = 1.0, s = 0.0;
    const double app = A[(int64_t)p * Dp + p], aqq = A[(int64_t)q * Dp + q];
    if (apq != 0.0 && fabs(apq) > 1e-300) {
        const double theta = (aqq - app) / (2.0 * apq);
        const double t = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
        c = 1.0 / sqrt(t * t + 1.0);
        s = t * c;
    }
    cs[i] = make_double2(c, s);
}

// rows p, q of A  <-  (c A_p - s A_q, s A_p + c A_q)   for every pair of the round
__global__ void jacobi_rows_kernel(double *__restrict__ A, int Dp, int r, const double2 *__restrict__ cs) {
    const int i = blockIdx.y;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= Dp) return;
    int p, q;
    rr_pair(r, i, Dp, p, q);
    const double2 k = cs[i];
    const double a = A[(int64_t)p * Dp + j], b = A[(int64_t)q * Dp + j];
    A[(int64_t)p * Dp + j] = k.x * a - k.y * b;
    A[(int64_t)q * Dp + j] = k.y * a + k.x * b;
}

// columns p, q of A and V  <-  (c X_p - s X_q, s X_p + c X_q)
__global__ void jacobi_cols_kernel(double *__restrict__ A, double *__restrict__ V, int Dp, int r,
                                   const double2 *__restrict__ cs) {
    const int i = blockIdx.y;
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= Dp) return;
    int p, q;
    rr_pair(r, i, Dp, p, q);
    const double2 k = cs[i];
    double *ar = A + (int64_t)row * Dp;
    double a = ar[p], b = ar[q];
    ar[p] = k.x * a - k.y * b;
    ar[q] = k.y * a + k.x * b;
    double *vr = V + (int64_t)row * Dp;
    a = vr[p];
    b = vr[q];
    vr[p] = k.x * a - k.y * b;
    vr[q] = k.y * a + k.x * b;
}

// One whole round in one kernel: block i owns the pair (p, q) = rr_pair(r, i) and writes rows
// p and q of J^T A J (its own rotation mixes the two rows, then every pair's rotation mixes
// the columns of both rows) and rows p and q of V J.  The pairs partition the indices, so
// the blocks touch disjoint rows; the arithmetic is the row pass followed by the column pass
// of the two kernels above, with coalesced row accesses only.
__global__ void __launch_bounds__(256) jacobi_round_kernel(double *__restrict__ A, double *__restrict__ V, int Dp,
                                                           int r, const double2 *__restrict__ cs) {
    extern __shared__ double rows_sm[];
    double *rp = rows_sm, *rq = rows_sm + Dp, *vp = rows_sm + 2 * Dp, *vq = rows_sm + 3 * Dp;
    int p, q;
    rr_pair(r, blockIdx.x, Dp, p, q);
    const double2 k = cs[blockIdx.x];
    double *Ap = A + (int64_t)p * Dp, *Aq = A + (int64_t)q * Dp;
    double *Vp = V + (int64_t)p * Dp, *Vq = V + (int64_t)q * Dp;
    for (int j = threadIdx.x; j < Dp; j += blockDim.x) {
        const double a = Ap[j], b = Aq[j];
        rp[j] = k.x * a - k.y * b;
        rq[j] = k.y * a + k.x * b;
        vp[j] = Vp[j];
        vq[j] = Vq[j];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < Dp / 2; t += blockDim.x) {
        int pp, qq;
        rr_pair(r, t, Dp, pp, qq);
        const double2 kk = cs[t];
        double a = rp[pp], b = rp[qq];
        rp[pp] = kk.x * a - kk.y * b;
        rp[qq] = kk.y * a + kk.x * b;
        a = rq[pp];
        b = rq[qq];
        rq[pp] = kk.x * a - kk.y * b;
        rq[qq] = kk.y * a + kk.x * b;
        a = vp[pp];
        b = vp[qq];
        vp[pp] = kk.x * a - kk.y * b;
        vp[qq] = kk.y * a + kk.x * b;
        a = vq[pp];
        b = vq[qq];
        vq[pp] = kk.x * a - kk.y * b;
        vq[qq] = kk.y * a + kk.x * b;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < Dp; j += blockDim.x) {
        Ap[j] = rp[j];
        Aq[j] = rq[j];
        Vp[j] = vp[j];
        Vq[j] = vq[j];
    }
}

// out[0] = sum of squared off-diagonal entries, out[1] = sum of squared diagonal entries
__global__ void jacobi_offnorm_kernel(const double *__restrict__ A, int Dp, double *__restrict__ out) {
    __shared__ double so[256], sd[256];
    double o = 0.0, d = 0.0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (int64_t)Dp * Dp;
         t += (int64_t)gridDim.x * blockDim.x) {
        const double v = A[t];
        if (t / Dp == t % Dp)
            d += v * v;
        else
            o += v * v;
    }
    so[threadIdx.x] = o;
    sd[threadIdx.x] = d;
    __syncthreads();
    for (int s = 128; s; s >>= 1) {
        if (threadIdx.x < s) {
            so[threadIdx.x] += so[threadIdx.x + s];
            sd[threadIdx.x] += sd[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicAdd(out, so[0]);
        atomicAdd(out + 1, sd[0]);
    }
}

__global__ void pad_copy_kernel(const double *__restrict__ K, int D, double *__restrict__ A, double *__restrict__ V,
                                int Dp) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)Dp * Dp) return;
    const int i = (int)(t / Dp), j = (int)(t % Dp);
    A[t] = (i < D && j < D) ? K[(int64_t)i * D + j] : 0.0;
    V[t] = i == j ? 1.0 : 0.0;
}

// evecs[r] = column idx[r] of V (first D entries), sign: largest-|.| entry positive
// (first index on ties); evals[r] = A[idx[r]][idx[r]].
__global__ void gather_eig_kernel(const double *__restrict__ A, const double *__restrict__ V, int Dp, int D,
                                  const int *__restrict__ idx, int nout, double *__restrict__ evals,
                                  double *__restrict__ evecs) {
    const int r = blockIdx.x;
    if (r >= nout) return;
    const int c = idx[r];
    __shared__ double sv[256];
    __shared__ int si[256];
    double best = -1.0;
    int bi = 0x7fffffff;
    for (int i = threadIdx.x; i < D; i += blockDim.x) {
        const double v = fabs(V[(int64_t)i * Dp + c]);
        if (v > best || (v == best && i < bi)) {
            best = v;
            bi = i;
        }
    }
    sv[threadIdx.x] = best;
    si[threadIdx.x] = bi;
    __syncthreads();
    for (int s = blockDim.x / 2; s; s >>= 1) {
        if (threadIdx.x < s) {
            const double v = sv[threadIdx.x + s];
            const int j = si[threadIdx.x + s];
            if (v > sv[threadIdx.x] || (v == sv[threadIdx.x] && j < si[threadIdx.x])) {
                sv[threadIdx.x] = v;
                si[threadIdx.x] = j;
            }
        }
        __syncthreads();
    }
    const double sign = V[(int64_t)si[0] * Dp + c] < 0.0 ? -1.0 : 1.0;
    for (int i = threadIdx.x; i < D; i += blockDim.x) evecs[(int64_t)r * D + i] = sign * V[(int64_t)i * Dp + c];
    if (threadIdx.x == 0 && evals) evals[r] = A[(int64_t)c * Dp + c];
}

__global__ void diag_kernel(const double *__restrict__ A, int Dp, double *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < Dp) out[i] = A[(int64_t)i * Dp + i];
}

__global__ void f32_to_f64_kernel(const float *__restrict__ a, int64_t n, double *__restrict__ b) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) b[t] = (double)a[t];
}

__global__ void f64_to_f32_kernel(const double *__restrict__ a, int64_t n, float *__restrict__ b) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) b[t] = (float)a[t];
}

// ------------------------------------------------- Jacobi eigh of small matrices
// The whole decomposition of a matrix of up to JC_MAX rows in one launch: a cluster of JC_CL blocks
// keeps A in its shared memory (row i in block i mod JC_CL, entries j > i; two copies, one read and
// one written in turn) and goes from round to round over the cluster barrier.  A round on the
// pairs (p_k, q_k) splits A into 2 x 2 blocks (pair I x pair J), each owned by one thread, which reads it
// from the old copy, applies both rotations and writes it to the new one.  Every block forms all
// rotations itself from copies of its own: the diagonal, which it updates for itself, and the
// round's a_pq, which their owners send to all blocks as they write them.  The rotations are kept, and
// jacobi_vectors_kernel applies them to the rows of V, which do not depend on one another, over all SMs.
//
// FP64 bounds this: the pipe takes a warp instruction every 64 cycles, so a division or a root
// costs 550 and no extra warp hides it.  Hence the angle comes from float32 (any t serves that
// brings a_pq down -- 1e-7 of it remains, the next sweep's share), converted by integer instructions, and
// only c = 1 / sqrt(1 + t^2) and s = t c are made accurate to FP64: an approximate root with one cubic
// step.  The update multiplies by t and scales by c_I c_J at the end (12 instead of 16 operations).
// 128 rows, 7 sweeps of 127 rounds: 5.4 ms of kernels and 2 ms of graph building with two launches a
// round replayed from a graph made per call; 2.7 ms with the angles' entries read from the other
// blocks in every round; 1.9 ms now, and 0.2 ms for the vectors.
constexpr int JC_CL = 16, JC_MAX = 256, JC_SWEEPS = 40;

__device__ __forceinline__ double ld_cluster(uint32_t addr, int rank) {
    uint32_t ra;
    double v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra) : "memory");
    return v;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, int rank, double v) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// pair k of round r on Dp (even) indices, as rr_pair, with 0 <= r < Dp - 1
__device__ __forceinline__ void rr_pair_fast(int r, int k, int Dp, int &p, int &q) {
    const int m = Dp - 1;
    int a = r + k, b = r - k;
    if (a >= m) a -= m;
    if (b < 0) b += m;
    if (k == 0) {
        a = r;
        b = m;
    }
    p = min(a, b);
    q = max(a, b);
}

// T threads (h = Dp / 2 <= T / 2); NB: 2 x 2 blocks of a thread at most
template <int T, int NB>
__global__ void __launch_bounds__(T) jacobi_cluster_kernel(double *__restrict__ A, int Dp, double2 *__restrict__ rot,
                                                           int *__restrict__ sweeps) {
    extern __shared__ double sm_a[];
    __shared__ double s_dg[2][JC_MAX], s_apq[2][JC_MAX / 2];
    __shared__ double2 s_tc[JC_MAX / 2];
    __shared__ double s_red[T / 32][2], s_part[2];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint32_t crank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(crank));
    const int rank = (int)crank, h = Dp / 2, rows = (Dp + JC_CL - 1) / JC_CL, rounds = Dp - 1;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm_a);
    const uint32_t part = (uint32_t)__cvta_generic_to_shared(s_part);
    const uint32_t apq_a = (uint32_t)__cvta_generic_to_shared(&s_apq[0][0]);
    auto at = [&](int i, int j) { return base + 8u * (uint32_t)((i >> 4) * Dp + j); };  // i < j
    static_assert(JC_CL == 16, "row to block by shifts");
    for (int l = wid; l < rows; l += T / 32) {
        const int i = rank + JC_CL * l;
        if (i < Dp)
            for (int j = i + lane; j < Dp; j += 32) sm_a[l * Dp + j] = A[(int64_t)i * Dp + j];
    }
    for (int i = tid; i < Dp; i += T) s_dg[0][i] = A[(int64_t)i * Dp + i];
    if (tid < h) {
        int p, q;
        rr_pair_fast(0, tid, Dp, p, q);
        s_apq[0][tid] = A[(int64_t)p * Dp + q];
    }
    // this thread's 2 x 2 blocks: pairs I < J of the round's list, the same positions in every round
    int bI[NB], bJ[NB];
#pragma unroll
    for (int e = 0; e < NB; ++e) {
        int b = (rank * T + tid) + e * JC_CL * T, i = 0;
        if (b < h * (h - 1) / 2) {
            while (b >= h - 1 - i) {
                b -= h - 1 - i;
                ++i;
            }
            bI[e] = i;
            bJ[e] = i + 1 + b;
        } else {
            bI[e] = -1;
            bJ[e] = 0;
        }
    }
    cluster_barrier();
    int buf = 0, sweep = 0;
    for (;; ++sweep) {
        // off-diagonal and diagonal sums of squares, added in one order by every block
        double off = 0.0, diag = 0.0;
        for (int l = wid; l < rows; l += T / 32) {
            const int i = rank + JC_CL * l;
            if (i < Dp)
                for (int j = i + 1 + lane; j < Dp; j += 32) {
                    const double v = sm_a[(buf * rows + l) * Dp + j];
                    off = fma(v, v, off);
                }
        }
        for (int i = rank + JC_CL * tid; i < Dp; i += JC_CL * T) diag = fma(s_dg[buf][i], s_dg[buf][i], diag);
        for (int o = 16; o; o >>= 1) {
            off += __shfl_xor_sync(FULL, off, o);
            diag += __shfl_xor_sync(FULL, diag, o);
        }
        if (lane == 0) {
            s_red[wid][0] = off;
            s_red[wid][1] = diag;
        }
        __syncthreads();
        if (tid < 2) {
            double v = 0.0;
            for (int w = 0; w < T / 32; ++w) v += s_red[w][tid];
            s_part[tid] = v;
        }
        cluster_barrier();
        off = diag = 0.0;
        for (int c = 0; c < JC_CL; ++c) {
            off += ld_cluster(part, c);
            diag += ld_cluster(part + 8, c);
        }
        off *= 2.0;
        const double tot = off + diag;
        if (!(off > 1e-28 * tot) || tot == 0.0 || sweep == JC_SWEEPS) break;
        for (int r = 0; r < rounds; ++r, buf ^= 1) {
            const uint32_t from = 8u * (uint32_t)(buf * rows * Dp), to = 8u * (uint32_t)((buf ^ 1) * rows * Dp);
            // entries (p_I, p_J), (p_I, q_J), (q_I, p_J), (q_I, q_J), on their way while the angles are formed
            double v[NB][4];
            int ei[NB][4], ej[NB][4];
#pragma unroll
            for (int e = 0; e < NB; ++e) {
                if (bI[e] < 0) continue;
                int i2[2], j2[2];
                rr_pair_fast(r, bI[e], Dp, i2[0], i2[1]);
                rr_pair_fast(r, bJ[e], Dp, j2[0], j2[1]);
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    ei[e][x] = min(i2[x >> 1], j2[x & 1]);
                    ej[e][x] = max(i2[x >> 1], j2[x & 1]);
                    v[e][x] = ld_cluster(at(ei[e][x], ej[e][x]) + from, ei[e][x] & 15);
                }
            }
            if (tid < h) {
                int p, q;
                rr_pair_fast(r, tid, Dp, p, q);
                double t, c;
                jacobi_angle(s_dg[buf][p], s_dg[buf][q], s_apq[buf][tid], t, c);
                s_tc[tid] = make_double2(t, c);
            }
            __syncthreads();
            // the pairs' own 2 x 2 blocks, by the other half of the threads: the diagonal in every block's copy,
            // what is left of a_pq and the rotation by one block
            const int k = tid - T / 2;
            if (k >= 0 && k < h) {
                int p, q;
                rr_pair_fast(r, k, Dp, p, q);
                const double app = s_dg[buf][p], aqq = s_dg[buf][q], apq = s_apq[buf][k];
                const double2 tc = s_tc[k];
                const double c2 = tc.y * tc.y, x2 = apq + apq;
                s_dg[buf ^ 1][p] = c2 * fma(tc.x, fma(tc.x, aqq, -x2), app);
                s_dg[buf ^ 1][q] = c2 * fma(tc.x, fma(tc.x, app, x2), aqq);
                if ((k & 15) == rank) {
                    st_cluster(at(p, q) + to, p & 15, c2 * fma(tc.x, fma(-tc.x, apq, app - aqq), apq));
                    rot[((int64_t)sweep * rounds + r) * h + k] = make_double2(tc.y, tc.x * tc.y);
                }
            }
            const int rn = r + 1 == rounds ? 0 : r + 1;  // the next round
#pragma unroll
            for (int e = 0; e < NB; ++e) {
                double n[4] = {0.0, 0.0, 0.0, 0.0};
                int nk[4] = {-1, -1, -1, -1};
                if (bI[e] >= 0) {
                    const double2 ti = s_tc[bI[e]], tj = s_tc[bJ[e]];
                    const double a = fma(-ti.x, v[e][2], v[e][0]), b = fma(-ti.x, v[e][3], v[e][1]);
                    const double c = fma(ti.x, v[e][0], v[e][2]), d = fma(ti.x, v[e][1], v[e][3]);
                    const double cc = ti.y * tj.y;
                    n[0] = cc * fma(-tj.x, b, a);
                    n[1] = cc * fma(tj.x, a, b);
                    n[2] = cc * fma(-tj.x, d, c);
                    n[3] = cc * fma(tj.x, c, d);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int i = ei[e][x], j = ej[e][x];
                        st_cluster(at(i, j) + to, i & 15, n[x]);
                        // the pair's position in the next round, if (i, j) is one: i + j = 2 rn mod m, or (rn, m)
                        int u = i - rn;
                        if (u < 0) u += rounds;
                        int w = j - rn;
                        if (w < 0) w += rounds;
                        if (j == rounds ? u == 0 : u + w == rounds) nk[x] = j == rounds ? 0 : min(u, w);
                    }
                }
                // the next round's a_pq to every block
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    unsigned bal = __ballot_sync(FULL, nk[x] >= 0);
                    while (bal) {
                        const int src = __ffs(bal) - 1;
                        bal &= bal - 1;
                        const double y = __shfl_sync(FULL, n[x], src);
                        const int kk = __shfl_sync(FULL, nk[x], src);
                        if (lane < JC_CL) st_cluster(apq_a + 8u * (uint32_t)((buf ^ 1) * (JC_MAX / 2) + kk), lane, y);
                    }
                }
            }
            cluster_barrier();
        }
    }
    if (rank == 0)
        for (int i = tid; i < Dp; i += T) A[(int64_t)i * Dp + i] = s_dg[buf][i];
    if (rank == 0 && tid == 0) *sweeps = sweep;
    cluster_barrier();  // no block leaves while another may read its partial sums
}

// Row blockIdx.x of V: the unit row times all rotations in order; one thread per pair.
__global__ void jacobi_vectors_kernel(const double2 *__restrict__ rot, const int *__restrict__ sweeps, int Dp,
                                      double *__restrict__ V) {
    __shared__ double v[JC_MAX];
    const int k = threadIdx.x, h = Dp / 2;
    v[k] = k == (int)blockIdx.x ? 1.0 : 0.0;
    v[k + h] = k + h == (int)blockIdx.x ? 1.0 : 0.0;
    const int64_t total = (int64_t)*sweeps * (Dp - 1);
    double2 next = total > 0 ? rot[k] : make_double2(1.0, 0.0);
    __syncthreads();
    int r = 0;
    for (int64_t g = 0; g < total; ++g) {
        const double2 cs = next;
        if (g + 1 < total) next = rot[(g + 1) * h + k];
        int p, q;
        rr_pair_fast(r, k, Dp, p, q);
        const double a = v[p], b = v[q];
        v[p] = fma(cs.x, a, -(cs.y * b));
        v[q] = fma(cs.y, a, cs.x * b);
        if (++r == Dp - 1) r = 0;
        __syncthreads();
    }
    V[(int64_t)blockIdx.x * Dp + k] = v[k];
    V[(int64_t)blockIdx.x * Dp + k + h] = v[k + h];
}

// Runs the cluster path on the padded matrix A (diagonal replaced by the eigenvalues) and writes V.
// False when the device cannot hold the cluster (nothing launched).
static int jacobi_cluster(double *A, double *V, int Dp, int *sweeps_dev, double2 *rot, cudaStream_t st, bool *ran) {
    *ran = false;
    const int rows = (Dp + JC_CL - 1) / JC_CL;
    const size_t smem = sizeof(double) * 2 * (size_t)rows * Dp;
    auto go = [&](auto kern, int threads) -> int {
        LV_CUDA(allow_smem(kern));
        LV_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(JC_CL);
        cfg.blockDim = dim3((unsigned)threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = JC_CL;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess || clusters < 1) {
            cudaGetLastError();
            return LV_OK;
        }
        LV_CUDA(cudaLaunchKernelEx(&cfg, kern, A, Dp, rot, sweeps_dev));
        *ran = true;
        return LV_OK;
    };
    // blocks of a thread: h (h - 1) / 2 of them, h = Dp / 2, over 16 T threads
    int rc = Dp <= 128 ? go(jacobi_cluster_kernel<128, 1>, 128) : go(jacobi_cluster_kernel<256, 2>, 256);
    if (rc || !*ran) return rc;
    jacobi_vectors_kernel<<<Dp, Dp / 2, 0, st>>>(rot, sweeps_dev, Dp, V);
    LV_CHECK_LAUNCH("jacobi_vectors_kernel");
    return LV_OK;
}

bool eigh_top_ok(int D, int nout);
int eigh_top(const double *K, int D, int nout, double *evals, double *evecs, cudaStream_t st);

// Eigen-decomposition of symmetric K (D x D FP64, device).  Writes the nout leading
// eigenpairs (descending eigenvalue) to evals (nullable) / evecs (nout x D).  Fewer than D pairs
// of a matrix of 8 .. 4096 rows: tridiagonal reduction + bisection + inverse iteration
// (eigh_tri.cu); all of them: cyclic Jacobi.
int eigh_impl(const double *K, int D, int nout, double *evals, double *evecs, cudaStream_t st, int *sweeps_out) {
    if (nout < D && eigh_top_ok(D, nout)) {
        if (sweeps_out) *sweeps_out = 0;
        return eigh_top(K, D, nout, evals, evecs, st);
    }
    const int Dp = D + (D & 1);
    double *A = nullptr, *V = nullptr, *acc = nullptr, *dg = nullptr;
    double2 *cs = nullptr;
    double2 *rot = nullptr;
    int *idx_d = nullptr, *nsw = nullptr;
    int rc = LV_OK;
    std::vector<double> diag(Dp);
    std::vector<int> order(Dp);
    double host_acc[2];
    int sweep = 0;
    bool fused = (size_t)Dp * 32 <= 200 * 1024;  // four rows of Dp doubles in shared memory
    cudaGraphExec_t sweep_exec = nullptr;
    auto launch_sweep = [&](cudaStream_t s) {
        for (int r = 0; r < Dp - 1; ++r) {
            jacobi_rot_kernel<<<(Dp / 2 + 127) / 128, 128, 0, s>>>(A, Dp, r, cs);
            if (fused) {
                jacobi_round_kernel<<<Dp / 2, 256, (size_t)Dp * 32, s>>>(A, V, Dp, r, cs);
            } else {
                jacobi_rows_kernel<<<dim3((Dp + 127) / 128, Dp / 2), 128, 0, s>>>(A, Dp, r, cs);
                jacobi_cols_kernel<<<dim3((Dp + 127) / 128, Dp / 2), 128, 0, s>>>(A, V, Dp, r, cs);
            }
        }
    };
    if (tmp_alloc((void **)&A, sizeof(double) * Dp * Dp, st) || tmp_alloc((void **)&V, sizeof(double) * Dp * Dp, st) ||
        tmp_alloc((void **)&acc, 2 * sizeof(double), st) || tmp_alloc((void **)&cs, sizeof(double2) * Dp / 2, st) ||
        tmp_alloc((void **)&idx_d, sizeof(int) * Dp, st) || tmp_alloc((void **)&dg, sizeof(double) * Dp, st)) {
        rc = fail(LV_ERR_OOM, "eigh: allocation failed");
        goto done;
    }
    pad_copy_kernel<<<(unsigned)(((int64_t)Dp * Dp + 255) / 256), 256, 0, st>>>(K, D, A, V, Dp);
    if (Dp >= 4 && Dp <= JC_MAX) {
        bool ran = false;
        const size_t rots = (size_t)JC_SWEEPS * (Dp - 1) * (Dp / 2);
        if (tmp_alloc((void **)&rot, sizeof(double2) * rots, st) || tmp_alloc((void **)&nsw, sizeof(int), st)) {
            rc = fail(LV_ERR_OOM, "eigh: allocation failed");
            goto done;
        }
        if ((rc = jacobi_cluster(A, V, Dp, nsw, rot, st, &ran))) goto done;
        if (ran) {
            if (sweeps_out && (cudaMemcpyAsync(&sweep, nsw, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                               cudaStreamSynchronize(st) != cudaSuccess)) {
                rc = fail(LV_ERR_CUDA, "eigh: kernel failure");
                goto done;
            }
            goto sorted;
        }
    }
    // one sweep = Dp - 1 rounds of (rotation angles, fused round); captured once into a CUDA
    // graph (launched per sweep), else launched directly
    if (fused && Dp * 32 > 48 * 1024 &&
        allow_smem(jacobi_round_kernel) != cudaSuccess) {
        cudaGetLastError();
        fused = false;
    }
    {
        cudaStream_t cap = nullptr;
        cudaGraph_t graph = nullptr;
        if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            launch_sweep(cap);
            if (cudaStreamEndCapture(cap, &graph) != cudaSuccess ||
                cudaGraphInstantiate(&sweep_exec, graph, 0) != cudaSuccess)
                sweep_exec = nullptr;
        }
        cudaGetLastError();  // a failed capture falls back to direct launches
        if (graph) cudaGraphDestroy(graph);
        if (cap) cudaStreamDestroy(cap);
    }
    for (sweep = 0; sweep < 40; ++sweep) {
        cudaMemsetAsync(acc, 0, 2 * sizeof(double), st);
        jacobi_offnorm_kernel<<<128, 256, 0, st>>>(A, Dp, acc);
        cudaMemcpyAsync(host_acc, acc, 2 * sizeof(double), cudaMemcpyDeviceToHost, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh: kernel failure");
            goto done;
        }
        const double tot = host_acc[0] + host_acc[1];
        if (!(host_acc[0] > 1e-28 * tot) || tot == 0.0) break;
        if (sweep_exec) {
            if (cudaGraphLaunch(sweep_exec, st) != cudaSuccess) {
                rc = fail(LV_ERR_CUDA, "eigh: sweep graph launch failed");
                goto done;
            }
        } else {
            launch_sweep(st);
        }
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "jacobi kernels");
            goto done;
        }
    }
sorted:
    // sort eigenvalues descending (stable by index); the padding index (D) is dropped
    {
        diag_kernel<<<(Dp + 255) / 256, 256, 0, st>>>(A, Dp, dg);
        cudaMemcpyAsync(diag.data(), dg, sizeof(double) * Dp, cudaMemcpyDeviceToHost, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh: diagonal copy failed");
            goto done;
        }
        std::iota(order.begin(), order.end(), 0);
        std::stable_sort(order.begin(), order.begin() + D, [&](int a, int b) { return diag[a] > diag[b]; });
        cudaMemcpyAsync(idx_d, order.data(), sizeof(int) * D, cudaMemcpyHostToDevice, st);
        gather_eig_kernel<<<nout, 256, 0, st>>>(A, V, Dp, D, idx_d, nout, evals, evecs);
        if (cudaStreamSynchronize(st) != cudaSuccess) {
            rc = fail(LV_ERR_CUDA, "eigh: gather failed");
            goto done;
        }
    }
done:
    if (sweep_exec) {
        cudaStreamSynchronize(st);
        cudaGraphExecDestroy(sweep_exec);
    }
    if (sweeps_out) *sweeps_out = sweep;
    tmp_free(A, st);
    tmp_free(V, st);
    tmp_free(acc, st);
    tmp_free(cs, st);
    tmp_free(idx_d, st);
    tmp_free(dg, st);
    tmp_free(rot, st);
    tmp_free(nsw, st);
    return rc;
}

int second_moment_bf16(const float *X, int64_t n, int D, float *K, int *status, cudaStream_t st);

int launch_f32_to_f64(const float *a, int64_t n, double *b, cudaStream_t st) {
    f32_to_f64_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, n, b);
    LV_CHECK_LAUNCH("f32_to_f64_kernel");
    return LV_OK;
}

int launch_f64_to_f32(const double *a, int64_t n, float *b, cudaStream_t st) {
    f64_to_f32_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, n, b);
    LV_CHECK_LAUNCH("f64_to_f32_kernel");
    return LV_OK;
}

}  // namespace lv

using namespace lv;

extern "C" {

int leanvec_second_moment(const float *X, int64_t n, int D, float *K, int precision, lv_stream_t stream) {
    if (!X || !K || n <= 0 || D <= 0) return fail(LV_ERR_ARG, "second_moment: invalid sizes or null pointer");
    if (precision == LV_PREC_FP32) return launch_gram_fp32(X, n, D, K, (cudaStream_t)stream);
    if (precision != LV_PREC_BF16) return fail(LV_ERR_ARG, "second_moment: precision must be LV_PREC_FP32 or LV_PREC_BF16");
    cudaStream_t st = (cudaStream_t)stream;
    int *status = nullptr, h = 0;
    if (tmp_alloc((void **)&status, sizeof(int), st)) return fail(LV_ERR_OOM, "second_moment: allocation failed");
    int rc = cudaMemsetAsync(status, 0, sizeof(int), st) == cudaSuccess ? LV_OK : fail(LV_ERR_CUDA, "memset failed");
    if (rc == LV_OK) rc = second_moment_bf16(X, n, D, K, status, st);
    if (rc == LV_OK && cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        rc = fail(LV_ERR_CUDA, "second_moment: status copy failed");
    if (rc == LV_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = fail(LV_ERR_CUDA, "second_moment: sync failed");
    if (rc == LV_OK && h) rc = fail(LV_ERR_TIMEOUT, "second_moment: a tensor-core pipeline wait timed out");
    tmp_free(status, st);
    return rc;
}

int leanvec_eigh(const double *K, int D, double *evals, double *evecs, lv_stream_t stream) {
    if (!K || !evecs || D <= 1) return fail(LV_ERR_ARG, "eigh: invalid sizes or null pointer");
    return eigh_impl(K, D, D, evals, evecs, (cudaStream_t)stream, nullptr);
}

int leanvec_fit_id(const float *X, int64_t n, int D, int d, float *A_out, float *B_out, int precision,
                   lv_stream_t stream) {
    if (!X || !A_out || n <= 0 || D <= 1 || d <= 0 || d > D)
        return fail(LV_ERR_ARG, "fit_id: invalid sizes or null pointer");
    cudaStream_t st = (cudaStream_t)stream;
    float *K = nullptr;
    double *K64 = nullptr, *P = nullptr;
    int rc = LV_OK;
    if (tmp_alloc((void **)&K, sizeof(float) * D * D, st) || tmp_alloc((void **)&K64, sizeof(double) * D * D, st) ||
        tmp_alloc((void **)&P, sizeof(double) * (size_t)d * D, st)) {
        rc = fail(LV_ERR_OOM, "fit_id: allocation failed");
    }
    if (rc == LV_OK) rc = leanvec_second_moment(X, n, D, K, precision, stream);
    if (rc == LV_OK) rc = launch_f32_to_f64(K, (int64_t)D * D, K64, st);
    if (rc == LV_OK) rc = eigh_impl(K64, D, d, nullptr, P, st, nullptr);
    if (rc == LV_OK) rc = launch_f64_to_f32(P, (int64_t)d * D, A_out, st);
    if (rc == LV_OK && B_out && B_out != A_out)
        if (cudaMemcpyAsync(B_out, A_out, sizeof(float) * (size_t)d * D, cudaMemcpyDeviceToDevice, st) != cudaSuccess)
            rc = fail(LV_ERR_CUDA, "fit_id: copy failed");
    if (rc == LV_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = fail(LV_ERR_CUDA, "fit_id: sync failed");
    tmp_free(K, st);
    tmp_free(K64, st);
    tmp_free(P, st);
    return rc;
}

}  // extern "C"
