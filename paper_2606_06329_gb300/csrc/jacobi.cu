// jacobi.cu - Step 3 (eq. svd_cov; Alg. 1 SVD_p): eigendecomposition of the
// k x k patch Gram G = X_c X_c^T = U diag(s^2) U^T, whose top p eigenpairs give
// the truncated SVD X_c = U_p diag(s) V_r^T (V_r = X_c^T U_p diag(s)^-1).
//
// Parallel-order (round-robin) two-sided Jacobi.  A round pairs every index
// once (the circle method: index kp-1 fixed, the others rotating), so its kp/2
// plane rotations touch disjoint row/column pairs and commute.  Per round:
//   1. the table threads compute each pair's rotation from the current 2 x 2
//      block: tau = (a_qq - a_pp) / (2 a_pq), t = sign(tau) / (|tau| +
//      sqrt(1 + tau^2)), c = 1/sqrt(1 + t^2), s = t c (the rotation zeroing
//      a_pq); pairs with |a_pq| <= eps sqrt(|a_pp a_qq|) are skipped (eps =
//      2^-22 in FP32, 2^-50 in FP64), and the
//      rotating pairs are compacted into the round's table (late sweeps are
//      cheap because few pairs still rotate);
//   2. A <- A J (each thread walks one row over its share of the pairs),
//   3. A <- J^T A (one column per thread), a_pq := 0 for rotated pairs,
//   4. U <- U J.
// kp - 1 rounds form a sweep; a sweep without any rotation ends the solve.
// One CTA of JT threads per patch keeps 4x more warps resident than one warp
// per patch at the same shared-memory footprint (A and U with row stride
// kp + 1 so column walks are bank-conflict free), which the latency-bound
// updates need.  The sweep count is capped; the cap sets
// MECUCO_ERR_NOT_CONVERGED in the device status word and keeps the current
// eigenpairs - it never traps.  Real = float (plain form) or double.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace mecuco {

template <typename Real>
struct JacobiEps;
template <>
struct JacobiEps<float> {
    static __host__ __device__ __forceinline__ float rel() { return 2.384185791015625e-07f; }  // 2^-22
};
template <>
struct JacobiEps<double> {
    static __host__ __device__ __forceinline__ double rel() { return 8.8817841970012523e-16; }  // 2^-50
};

// sqrt(|a b|); by the factors' roots where the product leaves FP32's normal range
// (entries beyond 2^64 and below 2^-63: the Grams of points beyond 1e9 or below 1e-9),
// where the sweeps would not rotate at all, or by anything.
__device__ __forceinline__ float geometric_mean(float a, float b) {
    const float p = fabsf(a * b);
    return p < INFINITY && p > 1.17549435e-38f ? sqrtf(p) : sqrtf(fabsf(a)) * sqrtf(fabsf(b));
}
__device__ __forceinline__ double geometric_mean(double a, double b) { return sqrt(fabs(a * b)); }

constexpr int JT = 128;  // threads per patch

// One rotation of a round's table, read by every walker as one 16-byte (FP32)
// or 32-byte (FP64) shared load: the kernel is bound by shared-memory
// wavefronts, and four separate table loads per rotation cost as many as its
// data accesses.
template <typename Real>
struct alignas(2 * sizeof(Real) + 2 * sizeof(int) > 16 ? 32 : 16) JRot {
    Real c, s;
    int p, q;
};

template <typename Real>
__global__ void __launch_bounds__(JT)
jacobi_kernel(const __grid_constant__ PatchSeg one, const PatchSeg *__restrict__ tab, int ntab, int blk0,
              int max_sweeps, Real eps, DevCounters *ctr) {
    extern __shared__ __align__(16) unsigned char jsm[];
    int local;
    const PatchSeg &seg = find_seg(one, tab, ntab, blk0 + (int)blockIdx.x, local);
    const int k = seg.k;
    const float *G = seg.G;
    float *sigma = seg.sig, *U = seg.U;
    const int kp = (k + 1) & ~1;
    const int h = kp / 2;
    const int ld = kp + 1;
    Real *A = reinterpret_cast<Real *>(jsm);
    Real *V = A + (size_t)kp * ld;
    // [h] rotations of the round, after A and V (rounded up to the entry alignment)
    JRot<Real> *rtab = reinterpret_cast<JRot<Real> *>(
        (reinterpret_cast<uintptr_t>(V + (size_t)kp * ld) + alignof(JRot<Real>) - 1) & ~(uintptr_t)(alignof(JRot<Real>) - 1));
    __shared__ int s_rot;
    __shared__ int s_act;  // rotations in the current round (compacted table length)

    const int tid = threadIdx.x;
    const int64_t patch = local;
    const float *g = G + patch * (int64_t)k * k;
    for (int e = tid; e < kp * kp; e += JT) {
        int r = e / kp, c = e % kp;
        A[r * ld + c] = (r < k && c < k) ? (Real)g[r * k + c] : (Real)0;
        V[r * ld + c] = (r == c) ? (Real)1 : (Real)0;
    }
    if (tid == 0) { s_rot = 0; s_act = 0; }
    __syncthreads();
    // thread -> (line, pair group) for the row/column/U walks: kp lines, JT/kp groups
    const int groups = JT / kp > 0 ? JT / kp : 1;
    const int line = tid % kp;
    const int grp = tid / kp;
    const bool walker = tid < kp * groups;

    int sweep = 0;
    bool converged = false;
    unsigned long long rotations = 0;  // tid 0's running total (counters only)
    for (; sweep < max_sweeps; ++sweep) {
        for (int round = 0; round < kp - 1; ++round) {
            if (tid < h) {
                int a, b;
                if (tid == 0) { a = kp - 1; b = round; }
                else { a = (round + tid) % (kp - 1); b = (round + kp - 1 - tid) % (kp - 1); }
                const int p = a < b ? a : b, q = a < b ? b : a;
                const Real app = A[p * ld + p], aqq = A[q * ld + q], apq = A[p * ld + q];
                if (fabs(apq) > eps * geometric_mean(app, aqq) && apq != (Real)0) {
                    const Real tau = (aqq - app) / (2 * apq);
                    const Real t = (tau >= 0 ? (Real)1 : (Real)-1) / (fabs(tau) + sqrt((Real)1 + tau * tau));
                    const Real c = (Real)1 / sqrt((Real)1 + t * t);
                    // rotations of one round commute: keep only those that rotate, in any order
                    const int slot = atomicAdd(&s_act, 1);
                    rtab[slot] = JRot<Real>{c, t * c, p, q};
                }
            }
            __syncthreads();
            const int nact = s_act;
            const int per = (nact + groups - 1) / groups;
            const int i0 = grp * per, i1 = min(nact, i0 + per);
            // A <- A J (thread walks row `line`)
            if (walker && line < kp) {
                Real *row = A + line * ld;
#pragma unroll 4
                for (int i = i0; i < i1; ++i) {
                    const JRot<Real> rt = rtab[i];
                    const int p = rt.p, q = rt.q;
                    const Real c = rt.c, s = rt.s;
                    const Real x = row[p], y = row[q];
                    row[p] = c * x - s * y;
                    row[q] = s * x + c * y;
                }
            }
            __syncthreads();
            // A <- J^T A (thread walks column `line`), U <- U J (row `line`)
            if (walker && line < kp) {
                Real *urow = V + line * ld;
#pragma unroll 4
                for (int i = i0; i < i1; ++i) {
                    const JRot<Real> rt = rtab[i];
                    const int p = rt.p, q = rt.q;
                    const Real c = rt.c, s = rt.s;
                    const Real x = A[p * ld + line], y = A[q * ld + line];
                    A[p * ld + line] = c * x - s * y;
                    A[q * ld + line] = s * x + c * y;
                    const Real u = urow[p], w = urow[q];
                    urow[p] = c * u - s * w;
                    urow[q] = s * u + c * w;
                }
            }
            __syncthreads();
            if (tid < nact) {
                const JRot<Real> rt = rtab[tid];
                A[rt.p * ld + rt.q] = 0;
                A[rt.q * ld + rt.p] = 0;
            }
            if (tid == 0) { s_rot += nact; s_act = 0; }
            __syncthreads();
        }
        const int rot = s_rot;
        rotations += (unsigned long long)rot;
        __syncthreads();
        if (tid == 0) s_rot = 0;
        __syncthreads();
        if (rot == 0) { converged = true; break; }
    }
    // sort eigenpairs (indices < k) descending by rank counting
    float *sg = sigma + patch * (int64_t)k;
    float *u = U + patch * (int64_t)k * k;
    for (int i = tid; i < k; i += JT) {
        const Real di = A[i * ld + i];
        int rank = 0;
        for (int j = 0; j < k; ++j) {
            const Real dj = A[j * ld + j];
            rank += pair_before(dj, j, di, i);
        }
        sg[rank] = (float)di;
        for (int r = 0; r < k; ++r) u[r * k + rank] = (float)V[r * ld + i];
    }
    if (tid == 0) {
        atomicMax(&ctr->jacobi_max_sweeps, (unsigned long long)(converged ? sweep : max_sweeps));
        atomicAdd(&ctr->jacobi_rotations, rotations);
        if (!converged) {
            atomicAdd(&ctr->jacobi_not_converged, 1ull);
            atomicOr(&ctr->status, (unsigned)DEV_NOT_CONVERGED);
        }
    }
}

// ---------------------------------------------------------------------------
// The same parallel-order Jacobi (same pairing, thresholds, rotations and
// sweep cap) with a round's updates fused into one pass over 2 x 2 blocks.
// Per round, lanes i < kp/2 of warp 0 compute pair i's rotation J_i and
// publish (c, s, p, q) in a table; then every rotating pair j is taken by one
// of the NW warps of the patch (round-robin over the ballot of rotating pairs,
// JW_UNROLL pairs in flight per warp), whose lane i replaces the block
// A[{p_i,q_i}, {p_j,q_j}] by J_i^T (A_ij J_j) (J_i = I when pair i does not
// rotate; for i = j the off-diagonal pair is set to 0) and, when pair i does
// not rotate, also writes the transposed result into A[{p_j,q_j}, {p_i,q_i}],
// the block whose column pair is not visited in this round; the same warp
// applies J_j to columns p_j, q_j of U (kept transposed: rows of U^T
// contiguous, two entries per lane, 8-byte accesses).  Every block is read and
// written by one lane in one iteration and no iteration reads a block another
// one writes, so a round needs two barriers (table published; updates done)
// and none inside.  Per rotation of a full round this moves 8 words of A (plus
// 4 transposed for pairs that do not rotate) and 8 of U, against 16 plus 3
// table reads in the one-CTA form's three passes with three barriers.
// ---------------------------------------------------------------------------
namespace {
constexpr int JW_UNROLL = 4;  // rotating pairs whose block updates are in flight together per warp
// Threshold strategy (Rutishauser's, for the cyclic Jacobi method): in the
// first JW_THR_SWEEPS sweeps a pair rotates only if |a_pq| also exceeds
// JW_THR_FACTOR S / kp^2, S the sum of |a_pq| over p < q at the sweep's start.
// 100k patches at k = 64: 21-22% fewer rotations, 192 -> 182 ms; the
// 256-dataset batch 2094 -> 1918 ms (factor 0.2: 1969 ms)
constexpr int JW_THR_SWEEPS = 3;
constexpr float JW_THR_FACTOR = 0.5f;
__host__ __device__ inline size_t jw_smem_bytes(int kmax) {
    const int kp = (kmax + 1) & ~1;
    // A (row stride kp + 1), U^T (row stride kp), 8-byte pad, 16-byte pad, table
    return ((size_t)kp * (kp + 1) + (size_t)kp * kp + 2 + 4) * sizeof(float) + 32 * sizeof(float4);
}
template <int NW>
__device__ __forceinline__ void jw_sync() {
    if constexpr (NW == 1) __syncwarp();
    else __syncthreads();
}
}  // namespace

template <int NW>
__global__ void __launch_bounds__(NW * 32)
jacobi_warp_kernel(const __grid_constant__ PatchSeg one, const PatchSeg *__restrict__ tab, int ntab, int blk0,
                   int max_sweeps, float eps, DevCounters *ctr) {
    extern __shared__ __align__(16) float jw_sm[];
    __shared__ unsigned ctl_mask;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int local;
    const PatchSeg &seg = find_seg(one, tab, ntab, blk0 + (int)blockIdx.x, local);
    const int k = seg.k;
    const int kp = (k + 1) & ~1;
    const int h = kp / 2;
    const int ld = kp + 1;
    const int n1 = kp - 1;
    float *A = jw_sm;
    float *Ut = A + (size_t)kp * ld;
    Ut += (reinterpret_cast<uintptr_t>(Ut) & 7) ? 1 : 0;  // 8-byte aligned rows (kp is even)
    float4 *T = reinterpret_cast<float4 *>((reinterpret_cast<uintptr_t>(Ut + (size_t)kp * kp) + 15) & ~(uintptr_t)15);
    const int64_t patch = local;
    const float *g = seg.G + patch * (int64_t)k * k;
    for (int e = threadIdx.x; e < kp * kp; e += NW * 32) {
        const int r = e / kp, c = e % kp;
        A[r * ld + c] = (r < k && c < k) ? g[r * k + c] : 0.f;
        Ut[e] = (r == c) ? 1.f : 0.f;
    }
    jw_sync<NW>();
    const unsigned FULL = 0xffffffffu;
    int sweep = 0;
    bool converged = false;
    unsigned long long rotations = 0;
    for (; sweep < max_sweeps; ++sweep) {
        int rot = 0;
        // threshold strategy in the first sweeps: small off-diagonal entries are
        // left for later sweeps, whose rotations would disturb them anyway
        float thr = 0.f;
        if (sweep < JW_THR_SWEEPS && warp == 0) {
            float part = 0.f;
            for (int e = lane; e < kp * kp; e += 32) {
                const int r = e / kp, c = e % kp;
                if (r < c) part += fabsf(A[r * ld + c]);
            }
            thr = JW_THR_FACTOR * warp_sum(part) / (float)(kp * kp);
        }
        // circle method (warp 0): index kp - 1 fixed (lane 0's a), the others rotate
        int a = lane == 0 ? n1 : lane % n1, b = lane == 0 ? 0 : (n1 - lane) % n1;
        for (int round = 0; round < n1; ++round) {
            if (warp == 0) {
                bool act = false;
                if (lane < h) {
                    const int p = a < b ? a : b, q = a < b ? b : a;
                    float c = 1.f, sn = 0.f;
                    const float app = A[p * ld + p], aqq = A[q * ld + q], apq = A[p * ld + q];
                    if (fabsf(apq) > eps * geometric_mean(app, aqq) && fabsf(apq) > thr && apq != 0.f) {
                        const float tau = (aqq - app) / (2 * apq);
                        const float t = (tau >= 0 ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
                        c = 1.f / sqrtf(1.f + t * t);
                        sn = t * c;
                        act = true;
                    }
                    T[lane] = make_float4(c, sn, __int_as_float(p), __int_as_float(q));
                }
                const unsigned m = __ballot_sync(FULL, act);
                if (lane == 0) ctl_mask = m;
                // next round's pair
                if (lane == 0) b = b + 1;
                else { a = a + 1 == n1 ? 0 : a + 1; b = b + 1 == n1 ? 0 : b + 1; }
            }
            jw_sync<NW>();  // the round's table
            unsigned mask = ctl_mask;
            rot += __popc(mask);
            if (mask != 0u && lane < h) {
                const float4 ti = T[lane];
                const float c = ti.x, sn = ti.y;
                const int p = __float_as_int(ti.z), q = __float_as_int(ti.w);
                const bool act = (mask >> lane) & 1u;
                float *rp = A + p * ld, *rq = A + q * ld;
                // this warp's share: every NW-th rotating pair, starting at the warp's index
                for (int w = 0; w < warp && mask; ++w) mask &= mask - 1;
                while (mask) {
                    int js[JW_UNROLL];
                    float4 tj[JW_UNROLL];
                    float av[JW_UNROLL][4];
                    float2 uv[JW_UNROLL], wv[JW_UNROLL];
#pragma unroll
                    for (int u = 0; u < JW_UNROLL; ++u) {
                        js[u] = mask ? __ffs(mask) - 1 : -1;
#pragma unroll
                        for (int w = 0; w < NW; ++w) mask &= mask - 1;
                    }
                    // every load of the group before its first store (no element
                    // loaded in a round is stored by another pair's update)
#pragma unroll
                    for (int u = 0; u < JW_UNROLL; ++u) {
                        if (js[u] < 0) continue;
                        tj[u] = T[js[u]];
                        const int pj = __float_as_int(tj[u].z), qj = __float_as_int(tj[u].w);
                        av[u][0] = rp[pj];
                        av[u][1] = rp[qj];
                        av[u][2] = rq[pj];
                        av[u][3] = rq[qj];
                        uv[u] = reinterpret_cast<const float2 *>(Ut + pj * kp)[lane];
                        wv[u] = reinterpret_cast<const float2 *>(Ut + qj * kp)[lane];
                    }
#pragma unroll
                    for (int u = 0; u < JW_UNROLL; ++u) {
                        if (js[u] < 0) continue;
                        const float c1 = tj[u].x, s1 = tj[u].y;
                        const int pj = __float_as_int(tj[u].z), qj = __float_as_int(tj[u].w);
                        // A J_j on the block's columns, then J_i^T on its rows
                        const float t00 = c1 * av[u][0] - s1 * av[u][1], t01 = s1 * av[u][0] + c1 * av[u][1];
                        const float t10 = c1 * av[u][2] - s1 * av[u][3], t11 = s1 * av[u][2] + c1 * av[u][3];
                        float r00 = t00, r01 = t01, r10 = t10, r11 = t11;
                        if (act) {
                            r00 = c * t00 - sn * t10;
                            r10 = sn * t00 + c * t10;
                            r01 = c * t01 - sn * t11;
                            r11 = sn * t01 + c * t11;
                        }
                        if (lane == js[u]) { r01 = 0.f; r10 = 0.f; }
                        rp[pj] = r00;
                        rp[qj] = r01;
                        rq[pj] = r10;
                        rq[qj] = r11;
                        if (!act) {
                            A[pj * ld + p] = r00;
                            A[qj * ld + p] = r01;
                            A[pj * ld + q] = r10;
                            A[qj * ld + q] = r11;
                        }
                        // U J_j: rows p_j, q_j of U^T
                        reinterpret_cast<float2 *>(Ut + pj * kp)[lane] =
                            make_float2(c1 * uv[u].x - s1 * wv[u].x, c1 * uv[u].y - s1 * wv[u].y);
                        reinterpret_cast<float2 *>(Ut + qj * kp)[lane] =
                            make_float2(s1 * uv[u].x + c1 * wv[u].x, s1 * uv[u].y + c1 * wv[u].y);
                    }
                }
            }
            jw_sync<NW>();  // the round's updates
        }
        rotations += (unsigned long long)rot;
        if (rot == 0) { converged = true; break; }
    }
    // eigenpairs (indices < k) sorted descending by rank counting
    float *sg = seg.sig + patch * (int64_t)k;
    float *u = seg.U + patch * (int64_t)k * k;
    for (int i = threadIdx.x; i < k; i += NW * 32) {
        const float di = A[i * ld + i];
        int rank = 0;
        for (int j = 0; j < k; ++j) {
            const float dj = A[j * ld + j];
            rank += pair_before(dj, j, di, i);
        }
        sg[rank] = di;
        for (int r = 0; r < k; ++r) u[r * k + rank] = Ut[i * kp + r];
    }
    if (threadIdx.x == 0) {
        atomicMax(&ctr->jacobi_max_sweeps, (unsigned long long)(converged ? sweep : max_sweeps));
        atomicAdd(&ctr->jacobi_rotations, rotations);
        if (!converged) {
            atomicAdd(&ctr->jacobi_not_converged, 1ull);
            atomicOr(&ctr->status, (unsigned)DEV_NOT_CONVERGED);
        }
    }
}

namespace {
// blk0: launch point of the first block (the points before it are solved elsewhere)
template <int NW>
cudaError_t launch_jw(const PatchSeg &one, const PatchSeg *tab, int ntab, int kmax, int64_t np, int blk0,
                      int max_sweeps, float eps, DevCounters *ctr, cudaStream_t s) {
    const size_t smem = jw_smem_bytes(kmax);
    cudaError_t e = cudaFuncSetAttribute(jacobi_warp_kernel<NW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    jacobi_warp_kernel<NW><<<(unsigned)np, NW * 32, smem, s>>>(one, tab, ntab, blk0, max_sweeps, eps, ctr);
    return cudaGetLastError();
}

// warps per patch of the fused form (1, 2 or 4)
cudaError_t launch_jacobi_warp(const PatchSeg &one, const PatchSeg *tab, int ntab, int kmax, int64_t np, int blk0,
                               int max_sweeps, float eps, DevCounters *ctr, cudaStream_t s, int nw) {
    if (nw == 4) return launch_jw<4>(one, tab, ntab, kmax, np, blk0, max_sweeps, eps, ctr, s);
    if (nw == 2) return launch_jw<2>(one, tab, ntab, kmax, np, blk0, max_sweeps, eps, ctr, s);
    return launch_jw<1>(one, tab, ntab, kmax, np, blk0, max_sweeps, eps, ctr, s);
}
}  // namespace

// ---------------------------------------------------------------------------
// Refinement of an FP32 eigendecomposition: one step of the iterative
// refinement for symmetric eigenproblems of Ogita & Aishima (Japan J. Indust.
// Appl. Math. 35, 2018).  With X the k x k eigenvector estimate from the FP32
// sweeps and A = G:
//   R = I - X^T X,   S = X^T A X,   lam_i = S_ii / (1 - R_ii),
//   E_ij = (S_ij + lam_j R_ij) / (lam_j - lam_i)  if |lam_i - lam_j| > delta,
//   E_ij = R_ij / 2 otherwise (and on the diagonal),   X' = X + X E.
// From FP32-accurate X one step squares the eigenvector error and
// re-orthogonalises X.  delta = 2^-18 max|lam| treats eigenvalues closer than
// the FP32 estimate resolves as a cluster (only orthogonalised); with rel != 0
// the test is relative to the pair, |lam_i - lam_j| <= 2^-18 max(|lam_i|,
// |lam_j|), for Grams whose FP32 eigenpairs are accurate relative to each
// eigenvalue (a nearly diagonal Gram, as in the adjoint's rotated basis).  With rel =
// 0 a pair whose correction would exceed REFINE_MAX_E is taken as one of a cluster
// too, and from REFINE_FIRST_ORDER on the second order is added, X' = X + X E + X E^2 /
// 2.  With rel = 1 neither: among the null vectors of a rank-deficient patch any
// noise is a gap relative to the pair, their corrections are as large as they like, and
// a second order would square them (nothing that the adjoint uses reads them).
// (With delta alone and the first order, 64 eigenvalues 2^-12 or 2^-16 apart came out
// with U^T U - I up to 700: what the sweeps leave off the diagonal is not small beside
// such gaps.)
// The O(k^3) products R, S and T = A X need more than FP32.  They are carried
// in two-term FP32 arithmetic ("double-float": a value is hi + lo, |lo| <=
// ulp(hi) / 2) because GB300 issues FP32 at ~60x its FP64 rate: A and X are
// FP32 values, so each product a x is exact as p + e (TwoProd: p = a x
// rounded, e = fma(a, x, -p)); the running sum takes p with Knuth's TwoSum
// (exact error term, no ordering assumption) and gathers e and the TwoSum
// errors in lo.  The accumulated error is ~n 2^-48 of the sum of |terms|
// (FP64: ~n 2^-53), far below what the FP32 eigenvectors written back can
// show: on 100k curved patches (m = 4096, k = 64) kappa came out bit-identical
// to an FP64 refinement, in 32% less stage time.  T is kept as hi + lo; S
// uses both parts (X T_lo as a plain FP32 product: it is 2^-24 of the term).
// The O(k^2) part (lambda, E) runs in FP64 from hi + lo, the correction X E
// (relative size ~2^-23) in FP32.  Every EFT step uses the _rn intrinsics,
// which the compiler never contracts into an FMA.  One CTA (256 threads,
// ~100 KB of shared memory, two per SM) per patch; results re-sorted
// descending.
// ---------------------------------------------------------------------------
namespace {
__device__ __forceinline__ void ff_mac(float &hi, float &lo, float a, float x) {
    const float p = __fmul_rn(a, x);
    const float e = __fmaf_rn(a, x, -p);
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(err, e));
}
// upper-triangle packed index of (a, b), a <= b < k
__device__ __forceinline__ int tri(int a, int b, int k) { return a * k - (a * (a - 1)) / 2 + (b - a); }
}  // namespace

constexpr int FT_REFINE = 256;
// Largest correction E_ij of a pair, and the largest up to which X (I + E) will do: the
// step is of first order and leaves E^2 of U^T U - I; beyond, E^2 / 2 is added, which
// leaves E^4 / 4 (the skew part's exponential to second order).  Eigenvectors that only
// rotate a patch (the adjoint's U0) take the second order from REFINE_ROTATION on: it
// moves the last bits of U0, and the gradient with them, for what 2^-16 of
// orthogonality in a near-degenerate pair is worth.
constexpr float REFINE_MAX_E = 0.0078125f;              // 2^-7
constexpr float REFINE_FIRST_ORDER = 2.44140625e-04f;   // 2^-12
constexpr float REFINE_ROTATION = 0.00390625f;          // 2^-8

template <int NT>
__device__ __forceinline__ void refine_ff_patch(const PatchSeg &seg, int local, int rel, float first_order,
                                                unsigned char *fsm) {
    const int k = seg.k;
    const float *G = seg.G;
    float *sigma = seg.sig, *U = seg.U;
    const int ld = k + 1;
    const int ntri = k * (k + 1) / 2;
    float *A = reinterpret_cast<float *>(fsm);  // [k][ld], later E
    float *X = A + k * ld;                      // [k][ld]
    float *Th = X + k * ld;                     // [k][ld]  T = A X, high part; later X'
    float *Tl = Th + k * ld;                    // [k][ld]  low part
    float *Sh = Tl + k * ld;                    // [ntri] S = X^T A X (upper)
    float *Sl = Sh + ntri;
    float *Rh = Sl + ntri;                      // [ntri] X^T X (upper)
    float *Rl = Rh + ntri;
    double *lam = reinterpret_cast<double *>(reinterpret_cast<uintptr_t>(Rl + ntri + 1) & ~(uintptr_t)7);  // [k]
    __shared__ double s_lmax;
    const int tid = threadIdx.x;
    const int64_t pt = local;
    const float *g = G + pt * (int64_t)k * k;
    float *u = U + pt * (int64_t)k * k;
    const int kk = k * k;
    for (int e = tid; e < kk; e += NT) {
        const int r = e / k, c = e - r * k;
        A[r * ld + c] = g[e];
        X[r * ld + c] = u[e];
    }
    __syncthreads();
    // T = A X: four outputs of one row per thread pass (independent chains)
    for (int q = tid; q * 4 < kk; q += NT) {
        const int e0 = q * 4;
        float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
        int rr[4], cc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = e0 + i < kk ? e0 + i : kk - 1;
            rr[i] = e / k;
            cc[i] = e - rr[i] * k;
        }
        for (int j = 0; j < k; ++j) {
#pragma unroll
            for (int i = 0; i < 4; ++i) ff_mac(hi[i], lo[i], A[rr[i] * ld + j], X[j * ld + cc[i]]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (e0 + i < kk) {
                Th[rr[i] * ld + cc[i]] = hi[i];
                Tl[rr[i] * ld + cc[i]] = lo[i];
            }
    }
    __syncthreads();
    // S = X^T T and R = X^T X on the upper triangle, two outputs per thread pass
    for (int q = tid; q * 2 < ntri; q += NT) {
        int ra[2], ca[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            int t = q * 2 + i < ntri ? q * 2 + i : ntri - 1;
            int a = 0;
            while (t >= k - a) { t -= k - a; ++a; }
            ra[i] = a;
            ca[i] = a + t;
        }
        float sh[2] = {0.f, 0.f}, sl[2] = {0.f, 0.f}, rh[2] = {0.f, 0.f}, rl[2] = {0.f, 0.f};
        for (int j = 0; j < k; ++j) {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float xr = X[j * ld + ra[i]];
                ff_mac(sh[i], sl[i], xr, Th[j * ld + ca[i]]);
                sl[i] = __fmaf_rn(xr, Tl[j * ld + ca[i]], sl[i]);
                ff_mac(rh[i], rl[i], xr, X[j * ld + ca[i]]);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (q * 2 + i < ntri) {
                const int t = q * 2 + i;
                Sh[t] = sh[i];
                Sl[t] = sl[i];
                Rh[t] = rh[i];
                Rl[t] = rl[i];
            }
    }
    __syncthreads();
    auto Sd = [&](int a, int b) { const int t = tri(a, b, k); return (double)Sh[t] + (double)Sl[t]; };
    // I - X^T X: the identity minus hi, then minus lo, in FP64
    auto Rd = [&](int a, int b) {
        const int t = tri(a, b, k);
        return ((a == b ? 1.0 : 0.0) - (double)Rh[t]) - (double)Rl[t];
    };
    if (tid < k) lam[tid] = Sd(tid, tid) / (1.0 - Rd(tid, tid));
    __syncthreads();
    if (tid == 0) {
        double mx = 0.0;
        for (int i = 0; i < k; ++i) mx = fmax(mx, fabs(lam[i]));
        s_lmax = mx;
    }
    __syncthreads();
    const double delta = 3.814697265625e-06 * s_lmax;  // 2^-18 max|lam|
    float *Ef = A;  // A is no longer needed
    bool large = false;
    for (int e = tid; e < kk; e += NT) {
        const int i = e / k, j = e - i * k;
        const int a = i < j ? i : j, b = i < j ? j : i;
        const double rij = Rd(a, b);
        const double sij = Sd(a, b);
        const double dij = rel ? 3.814697265625e-06 * fmax(fabs(lam[i]), fabs(lam[j])) : delta;
        const double gap = lam[j] - lam[i];
        // the mean of E_ij's numerator and E_ji's, so that both take the same branch
        const double num = fabs(sij + 0.5 * (lam[i] + lam[j]) * rij);
        double v;
        if (i == j || fabs(gap) <= dij || (!rel && num > (double)REFINE_MAX_E * fabs(gap))) v = 0.5 * rij;
        else v = (sij + lam[j] * rij) / gap;  // (a NaN stays one)
        large = large || fabs(v) > (double)first_order;
        Ef[i * ld + j] = (float)v;
    }
    const bool second = __syncthreads_or(large);
    // X' = X + X E (FP32), into Th; X E kept for the second order
    float *Xn = Th, *Y = Tl;
    for (int e = tid; e < kk; e += NT) {
        const int r = e / k, c = e - r * k;
        float t = 0.f;
        for (int j = 0; j < k; ++j) t = fmaf(X[r * ld + j], Ef[j * ld + c], t);
        Xn[r * ld + c] = X[r * ld + c] + t;
        Y[r * ld + c] = t;
    }
    __syncthreads();
    if (second) {
        for (int e = tid; e < kk; e += NT) {
            const int r = e / k, c = e - r * k;
            float t = 0.f;
            for (int j = 0; j < k; ++j) t = fmaf(Y[r * ld + j], Ef[j * ld + c], t);
            Xn[r * ld + c] = fmaf(0.5f, t, Xn[r * ld + c]);
        }
        __syncthreads();
    }
    float *sg = sigma + pt * (int64_t)k;
    for (int i = tid; i < k; i += NT) {
        int rank = 0;
        for (int j = 0; j < k; ++j) rank += pair_before(lam[j], j, lam[i], i);
        sg[rank] = (float)lam[i];
        for (int r = 0; r < k; ++r) u[r * k + rank] = Xn[r * ld + i];
    }
}

template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT)
jacobi_refine_ff_kernel(const __grid_constant__ PatchSeg one, const PatchSeg *__restrict__ tab, int ntab, int rel,
                        float first_order) {
    extern __shared__ __align__(16) unsigned char fsm[];
    int local;
    const PatchSeg &seg = find_seg(one, tab, ntab, (int)blockIdx.x, local);
    refine_ff_patch<NT>(seg, local, rel, first_order, fsm);
}

size_t refine_ff_smem_bytes(int k) {
    return (size_t)4 * k * (k + 1) * sizeof(float) + (size_t)2 * k * (k + 1) * sizeof(float) + 16 +
           (size_t)k * sizeof(double);
}


// ---------------------------------------------------------------------------
// The same refinement step through the residual T = A X - X diag(l), l the
// sweeps' eigenvalues, for callers that use only the refined eigenpairs:
//   N = X^T T = S + R diag(l) - diag(l)      (R = I - X^T X, S = X^T A X),
// so N_ij is the numerator of E_ij for i != j (it decides, with N_ji, whether the pair
// is one of a cluster), and lam_i = l_i + N_ii / (1 -
// R_ii).  Only T needs more than FP32: it is small (the sweeps' residual, 1e-6
// to 1e-4 of lam_1), so N from FP32 products carries 2^-24 of a small matrix,
// which is a relative error of the correction E, not of the eigenvectors.  R is
// formed (two-term) only where E uses it alone: the diagonal and pairs inside
// a cluster.  A product a x is added to a two-term sum in four operations: hi
// carries an offset of 1.5 2^e that every partial sum stays below a third of
// (|A X| <= lam_1 by Cauchy, so 2^e >= 4 lam_1; 2^e = 4 for the sums of R), so
// hi never leaves its binade, d = fma(a, x, hi) - hi is exact and fma(a, x, -d)
// is what the sum lost, to 2^-24 of one unit in the last place of the offset:
// about 2^-41 lam_1 over 64 terms.
// One k^3 two-term product and two FP32 ones, no FP64, against two and a half
// two-term products at ten operations a term, one FP32 product and k^2 FP64
// divisions (GB300 has 1/64 of the FP32 rate in FP64).
// Measured on GB300 per 100k patches, first order alone: k = 64 9.4 ms (two-term
// products: 52), k = 37 3.3 (12), k = 32 1.6 (6.7); the exchange of the numerators and
// the second order add 0.5% to a forward pass.  U^T U - I and the off-diagonals of U^T
// A U as with the two-term products (5e-7, 1.3e-8 lam_1).  FMA-issue bound.
// Every thread forms 4 x 4 blocks from 16-byte shared loads, two columns per
// packed FP32 instruction.
// ---------------------------------------------------------------------------
namespace {
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float lo, float hi) {
    f2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// (hi, lo) += a x, two independent sums with the offset in hi; minus = (-1, -1)
__device__ __forceinline__ void off_mac2(f2 &hi, f2 &lo, f2 a, f2 x, f2 minus) {
    const f2 h = fma2(a, x, hi);
    lo = add2(lo, fma2(a, x, fma2(h, minus, hi)));
    hi = h;
}
// sum of a_r b_r - base over r < k (|sum| <= 1 or so), rounded once
__device__ __forceinline__ float off_dot(const float *a, const float *b, int stride, int k, float base) {
    float hi = 6.f, lo = 0.f;
    for (int r = 0; r < k; ++r) {
        const float h = __fmaf_rn(a[r * stride], b[r * stride], hi);
        lo = __fadd_rn(lo, __fmaf_rn(a[r * stride], b[r * stride], __fsub_rn(hi, h)));
        hi = h;
    }
    return __fadd_rn(__fsub_rn(hi, 6.f + base), lo);
}
__host__ __device__ inline int rr_ld(int k) { return (k + 3) / 4 * 4 + 4; }
__host__ __device__ inline size_t refine_res_smem_bytes(int k) {
    const int k4 = (k + 3) / 4 * 4;
    return ((size_t)3 * k4 * rr_ld(k) + 4 * k4) * sizeof(float);
}
}  // namespace

template <int NT>
__device__ __forceinline__ void refine_res_patch(const PatchSeg &seg, int local, float *rsm) {
    const int k = seg.k;
    const int k4 = (k + 3) / 4 * 4, ld = rr_ld(k), nt = k4 / 4;
    float *A = rsm;            // [k4][ld] G, later X^T
    float *X = A + k4 * ld;    // [k4][ld]
    float *T = X + k4 * ld;    // [k4][ld] A X - X diag(l), later E
    float *l0 = T + k4 * ld;   // [k4] the sweeps' eigenvalues
    float *dl = l0 + k4;       // [k4] lam - l0
    float *rd = dl + k4;       // [k4] R_ii
    float *lam = rd + k4;      // [k4]
    const int tid = threadIdx.x;
    const int64_t pt = local;
    const float *g = seg.G + pt * (int64_t)k * k;
    float *u = seg.U + pt * (int64_t)k * k;
    float *sg = seg.sig + pt * (int64_t)k;
    for (int r = tid / 32; r < k4; r += NT / 32)
        for (int c = tid & 31; c < k4; c += 32) {
            const bool in = r < k && c < k;
            A[r * ld + c] = in ? g[r * k + c] : 0.f;
            X[r * ld + c] = in ? u[r * k + c] : 0.f;
        }
    if (tid < k4) l0[tid] = tid < k ? sg[tid] : 0.f;
    __syncthreads();
    const f2 minus = pack2(-1.f, -1.f);
    // T = A X - X diag(l): A's rows stand for its columns (symmetric)
    const bool mine = tid < nt * nt;  // one 4 x 4 block per thread (nt^2 <= NT)
    const int i0 = tid / nt * 4, c0 = tid % nt * 4;
    if (mine) {
        float l1 = 9.4039548e-38f;
        for (int j = 0; j < k; ++j) l1 = fmaxf(l1, fabsf(l0[j]));
        // 1.5 2^e, 4 l1 <= 2^e < 8 l1 (the largest binade at the end of the range)
        const float off = 1.5f * __uint_as_float(min((__float_as_uint(l1) >> 23) + 3u, 253u) << 23);
        const f2 off2 = pack2(off, off), noff2 = pack2(-off, -off);
        f2 hi[4][2], lo[4][2] = {};
#pragma unroll
        for (int i = 0; i < 4; ++i) hi[i][0] = hi[i][1] = off2;
        for (int j = 0; j < k; ++j) {
            const float4 a = *reinterpret_cast<const float4 *>(A + j * ld + i0);
            const float4 x = *reinterpret_cast<const float4 *>(X + j * ld + c0);
            const f2 x0 = pack2(x.x, x.y), x1 = pack2(x.z, x.w);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const f2 a2 = pack2(av[i], av[i]);
                off_mac2(hi[i][0], lo[i][0], a2, x0, minus);
                off_mac2(hi[i][1], lo[i][1], a2, x1, minus);
            }
        }
        const float4 l = *reinterpret_cast<const float4 *>(l0 + c0);
        const f2 n0 = pack2(-l.x, -l.y), n1 = pack2(-l.z, -l.w);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 x = *reinterpret_cast<const float4 *>(X + (i0 + i) * ld + c0);
            off_mac2(hi[i][0], lo[i][0], n0, pack2(x.x, x.y), minus);
            off_mac2(hi[i][1], lo[i][1], n1, pack2(x.z, x.w), minus);
            const float2 p = unpack2(add2(add2(hi[i][0], noff2), lo[i][0])),
                         q = unpack2(add2(add2(hi[i][1], noff2), lo[i][1]));
            *reinterpret_cast<float4 *>(T + (i0 + i) * ld + c0) = make_float4(p.x, p.y, q.x, q.y);
        }
    }
    // R_ii
    if (tid < k4) rd[tid] = -off_dot(X + tid, X + tid, ld, k, 1.f);
    __syncthreads();
    // N = X^T T, kept in registers
    f2 n[4][2] = {};
    if (mine) {
        for (int r = 0; r < k; ++r) {
            const float4 x = *reinterpret_cast<const float4 *>(X + r * ld + i0);
            const float4 v = *reinterpret_cast<const float4 *>(T + r * ld + c0);
            const f2 v0 = pack2(v.x, v.y), v1 = pack2(v.z, v.w);
            const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const f2 x2 = pack2(xv[i], xv[i]);
                n[i][0] = fma2(x2, v0, n[i][0]);
                n[i][1] = fma2(x2, v1, n[i][1]);
            }
        }
        if (i0 == c0) {
            const float d[4] = {unpack2(n[0][0]).x, unpack2(n[1][0]).y, unpack2(n[2][1]).x, unpack2(n[3][1]).y};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                dl[i0 + i] = d[i] / (1.f - rd[i0 + i]);
                lam[i0 + i] = l0[i0 + i] + dl[i0 + i];
            }
        }
    }
    // X^T over A
    for (int r = tid / 32; r < k4; r += NT / 32)
        for (int c = tid & 31; c < k4; c += 32) A[c * ld + r] = X[r * ld + c];
    __syncthreads();
    float lmax = 0.f;
    for (int i = 0; i < k; ++i) lmax = fmaxf(lmax, fabsf(lam[i]));
    const float delta = 3.814697265625e-06f * lmax;  // 2^-18 max|lam|
    // N over T (every thread is past its reads of T): E_ij needs N_ji too
    float v[4][4];
    bool large = false;
    if (mine) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 p = unpack2(n[i][0]), q = unpack2(n[i][1]);
            v[i][0] = p.x, v[i][1] = p.y, v[i][2] = q.x, v[i][3] = q.y;
            *reinterpret_cast<float4 *>(T + (i0 + i) * ld + c0) = make_float4(p.x, p.y, q.x, q.y);
        }
    }
    __syncthreads();
    if (mine) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float4 t4 = *reinterpret_cast<const float4 *>(T + (c0 + c) * ld + i0);  // N_ji
            const float nt[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int ii = i0 + i, jj = c0 + c;
                const float d = (l0[jj] - l0[ii]) + (dl[jj] - dl[ii]);
                // the mean of both numerators, so that E_ij and E_ji take the same branch
                const float num = 0.5f * fabsf(v[i][c] + nt[i]);
                if (ii == jj) {
                    v[i][c] = 0.5f * rd[ii];
                } else if (!(fabsf(d) > delta) || !(num <= REFINE_MAX_E * fabsf(d))) {
                    v[i][c] = ii < k && jj < k ? -0.5f * off_dot(X + ii, X + jj, ld, k, 0.f) : 0.f;
                } else {
                    v[i][c] = v[i][c] / d;
                    large = large || fabsf(v[i][c]) > REFINE_FIRST_ORDER;
                }
            }
        }
    }
    const bool second = __syncthreads_or(large);
    // E over N
    if (mine) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(T + (i0 + i) * ld + c0) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
    }
    __syncthreads();
    // X' = X + X E, and with corrections beyond the first order + (X E) E / 2
    for (int order = 1;; ++order) {
        f2 acc[4][2] = {};
        if (mine) {
            for (int j = 0; j < k; ++j) {
                const float4 x = *reinterpret_cast<const float4 *>(A + j * ld + i0);
                const float4 e = *reinterpret_cast<const float4 *>(T + j * ld + c0);
                const f2 e0 = pack2(e.x, e.y), e1 = pack2(e.z, e.w);
                const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f2 x2 = pack2(xv[i], xv[i]);
                    acc[i][0] = fma2(x2, e0, acc[i][0]);
                    acc[i][1] = fma2(x2, e1, acc[i][1]);
                }
            }
            const f2 part = order == 1 ? pack2(1.f, 1.f) : pack2(0.5f, 0.5f);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 *xr = reinterpret_cast<float4 *>(X + (i0 + i) * ld + c0);
                const float4 x = *xr;
                const float2 p = unpack2(fma2(part, acc[i][0], pack2(x.x, x.y))),
                             q = unpack2(fma2(part, acc[i][1], pack2(x.z, x.w)));
                *xr = make_float4(p.x, p.y, q.x, q.y);
            }
        }
        if (order == 2 || !second) break;
        __syncthreads();  // every thread is past its reads of A
        if (mine) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {  // (X E)^T over X^T
                float t[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 a = unpack2(acc[i][c >> 1]);
                    t[i] = c & 1 ? a.y : a.x;
                }
                *reinterpret_cast<float4 *>(A + (c0 + c) * ld + i0) = make_float4(t[0], t[1], t[2], t[3]);
            }
        }
        __syncthreads();
    }
    // ranks (descending, lowest index first on ties), over dl
    int *rk = reinterpret_cast<int *>(dl);
    if (tid < k) {
        const float li = lam[tid];
        int rank = 0;
        for (int j = 0; j < k; ++j) rank += pair_before(lam[j], j, li, tid);
        sg[rank] = li;
        rk[tid] = rank;
    }
    __syncthreads();
    for (int r = tid / 32; r < k; r += NT / 32)
        for (int c = tid & 31; c < k; c += 32) u[r * k + rk[c]] = X[r * ld + c];
}

// nres: segments (of a table; they lead) refined through the residual, the rest
// by the two-term products
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
jacobi_refine_res_kernel(const __grid_constant__ PatchSeg one, const PatchSeg *__restrict__ tab, int ntab, int nres) {
    extern __shared__ __align__(16) float rsm[];
    int local;
    const PatchSeg &seg = find_seg(one, tab, ntab, (int)blockIdx.x, local);
    if (ntab == 0 || (int)(&seg - tab) < nres) refine_res_patch<NT>(seg, local, rsm);
    else refine_ff_patch<NT>(seg, local, 0, REFINE_FIRST_ORDER, reinterpret_cast<unsigned char *>(rsm));
}

size_t jacobi_smem_bytes(int k, int fp64) {
    const int kp = (k + 1) & ~1;
    const size_t real = fp64 ? sizeof(double) : sizeof(float);
    const size_t ent = fp64 ? sizeof(JRot<double>) : sizeof(JRot<float>);
    return (size_t)2 * kp * (kp + 1) * real + ent + (size_t)(kp / 2) * ent;
}

cudaError_t launch_jacobi_seg(const PatchSeg &one, const PatchSeg *tab, int ntab, int kmax, int64_t np, int fp64,
                              int max_sweeps, DevCounters *ctr, cudaStream_t s, int warp_form, const JacobiReg &reg) {
    if (np <= 0) return cudaSuccess;
    if (kmax > 64 || kmax < 1) return cudaErrorInvalidValue;
    cudaError_t e;
    // FP32 sweeps: one or more warps per patch, or one CTA per patch
    auto sweeps32 = [&](const PatchSeg *t, int nt, int kb, int64_t n, int64_t blk0) -> cudaError_t {
        const float eps = JacobiEps<float>::rel();
        if (n <= 0) return cudaSuccess;
        if (warp_form)
            return launch_jacobi_warp(one, t, nt, kb, n, (int)blk0, max_sweeps, eps, ctr, s,
                                      warp_form < 0 ? 2 : warp_form);
        const size_t smem = jacobi_smem_bytes(kb, 0);
        cudaError_t r = cudaFuncSetAttribute(jacobi_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (r != cudaSuccess) return r;
        jacobi_kernel<float><<<(unsigned)n, JT, smem, s>>>(one, t, nt, (int)blk0, max_sweeps, eps, ctr);
        return cudaGetLastError();
    };
    if (fp64 == 1 || fp64 == 3 || fp64 == 4) {
        // FP32 sweeps, then one refinement step (3: relative cluster test; 4: a rotation)
        const bool fast = reg.np > 0 && fp64 == 1 && warp_form < 0;
        if (fast) {
            PatchSeg seg = one;
            seg.npts = (int)np;
            seg.jfirst = 0;
            e = launch_jacobi_reg(seg, tab, ntab ? reg.nseg : 0, reg.kmax, reg.warps, max_sweeps, ctr, s);
            if (e != cudaSuccess) return e;
            e = sweeps32(tab + reg.nseg, ntab - reg.nseg, reg.kmax_rest, np - reg.np, reg.np);
        } else {
            e = sweeps32(tab, ntab, kmax, np, 0);
        }
        if (e != cudaSuccess) return e;
        if (fast) {
            // threads per patch: one 4 x 4 block each; one launch, which takes the
            // two-term products for the points solved by the two-sided sweeps
            const bool rest = reg.np < np;
            const size_t rs = std::max(refine_res_smem_bytes(reg.kmax), rest ? refine_ff_smem_bytes(reg.kmax_rest) : 0);
            auto refine = [&](auto kern, int nt) -> cudaError_t {
                cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rs);
                if (r != cudaSuccess) return r;
                kern<<<(unsigned)np, nt, rs, s>>>(one, tab, ntab, reg.nseg);
                return cudaGetLastError();
            };
            if (kmax <= 32) return refine(jacobi_refine_res_kernel<64, 12>, 64);
            if (kmax <= 44) return refine(jacobi_refine_res_kernel<128, 6>, 128);
            return refine(jacobi_refine_res_kernel<256, 3>, 256);
        }
        // threads per patch: 64 (k <= 16), 128 (k <= 32) or 256, so that small
        // patches are not limited to 8 per SM by idle threads
        const size_t rs = refine_ff_smem_bytes(kmax);
        auto refine = [&](auto kern, int nt) -> cudaError_t {
            cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rs);
            if (r != cudaSuccess) return r;
            const float first = fp64 == 3 ? INFINITY : fp64 == 4 ? REFINE_ROTATION : REFINE_FIRST_ORDER;
            kern<<<(unsigned)np, nt, rs, s>>>(one, tab, ntab, fp64 == 3, first);
            return cudaGetLastError();
        };
        if (kmax <= 16) return refine(jacobi_refine_ff_kernel<64>, 64);
        if (kmax <= 32) return refine(jacobi_refine_ff_kernel<128>, 128);
        return refine(jacobi_refine_ff_kernel<FT_REFINE>, FT_REFINE);
    }
    if (fp64 == 2) {
        const size_t smem = jacobi_smem_bytes(kmax, fp64);
        e = cudaFuncSetAttribute(jacobi_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        jacobi_kernel<double><<<(unsigned)np, JT, smem, s>>>(one, tab, ntab, 0, max_sweeps, JacobiEps<double>::rel(), ctr);
        return cudaGetLastError();
    }
    return sweeps32(tab, ntab, kmax, np, 0);
}

cudaError_t launch_jacobi(const float *G, int k, int64_t np, int fp64, int max_sweeps, float *sigma, float *U,
                          DevCounters *ctr, cudaStream_t s, int warp_form, bool reg) {
    PatchSeg one{};
    one.k = k;
    one.G = const_cast<float *>(G);
    one.sig = sigma;
    one.U = U;
    return launch_jacobi_seg(one, nullptr, 0, k, np, fp64, max_sweeps, ctr, s, warp_form,
                             reg ? jacobi_reg_all(k, np) : JacobiReg());
}

}  // namespace mecuco
