// moments.cu - Steps 2-3 (Sec. 3 Step 2; Alg. 1 Fast branch: centring, and the
// k x k Gram that replaces SVD_p(X_c), eq. svd_cov) plus the patch moments the
// one-pass estimator needs.  Plain FP32 on the CUDA cores.
//
// Every estimator term of Alg. 1 is a k-space function of three moments of
// the centred patch X_c (derivation in the estimator kernel):
//   G = X_c X_c^T,  R = X_c 1_m,  M[j,r,t] = sum_a X_c[j,a] X_c[r,a] X_c[t,a],
// and, for the Haar-consistent variant, Q = X_c diag(c) X_c^T with
// c_a = sum_j X_c[j,a]^2.  Centring is per column (x_ja - mean_j x_ja), so the
// kernels stream the patch through shared memory in column chunks, centre each
// chunk and accumulate.
//
// The kernels optionally take a per-point orthogonal k x k matrix U0 (row r,
// column l) and then accumulate the moments of Z = U0^T X_c instead of X_c.
// Every estimator term is invariant under such a rotation of the point axis
// (tau, t_range, t_A, |G_tens|^2 and the Haar sum are sums of squares over j),
// and with U0 the eigenvectors of a first Gram the rotated Gram is nearly
// diagonal, so its small eigenvalues come out with small relative error in
// FP32 (error of order eps s_max/s_min instead of eps (s_max/s_min)^2).  The
// adjoint uses this.
//
// A chunk is MCH columns: gathered row by row (a warp per row, a lane per
// column, the next chunk's values on their way in registers), centred (a lane per
// column, the rows shared between the warps: in two-term FP32 for the rotated form,
// whose small directions would show the rounding of the means), then rotated, or
// copied, into column-major order, which is what 16-byte operand loads want.  Every
// sum of a result runs in ascending order of the column in one thread.
#include <math.h>

#include "common.cuh"
#include "fast_terms.cuh"
#include "kernels.h"

namespace mecuco {

namespace {
typedef unsigned long long f2;  // two FP32 values of a packed instruction
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

// A neighbour index outside [0, N) is read as row 0 and flagged, never followed.
__device__ __forceinline__ int checked_row(int r, int64_t N, DevCounters *ctr) {
    if (r < 0 || (int64_t)r >= N) {
        atomicOr(&ctr->status, (unsigned)DEV_INVALID);
        return 0;
    }
    return r;
}

constexpr int MCH = 32;  // columns per chunk
constexpr int XLD = 34;  // row stride of a row-major chunk (even: 8-byte loads)

// Rows warp, warp + NT / 32, ... (NR at most) of a chunk in registers: loaded while
// the chunk before is worked on, then stored.
template <int NT, int NR>
struct ChunkRows {
    float v[NR];
    template <typename T>
    __device__ __forceinline__ void load(const T *__restrict__ X, int64_t ld, const int *rows, int k, int64_t a0,
                                         int64_t m) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const bool in = a0 + lane < m;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int r = warp + i * (NT / 32);
            v[i] = in && r < k ? load_elem(X + (int64_t)rows[r] * ld + a0 + lane) : 0.f;
        }
    }
    __device__ __forceinline__ void store(float *Xr, int k) const {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int r = warp + i * (NT / 32);
            if (r < k) Xr[r * XLD + lane] = v[i];
        }
    }
};

// x - mean, rounded once (two-term sums); part: NT floats x 2.  Ends before a barrier.
template <int NT>
__device__ __forceinline__ void centre_two_term(float *Xr, int k, float2 *part) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    ff s{0.f, 0.f};
    for (int r = warp; r < k; r += NW) s = ff_add(s, ff{Xr[r * XLD + lane], 0.f});
    part[threadIdx.x] = make_float2(s.hi, s.lo);
    __syncthreads();
    s = ff{0.f, 0.f};
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const float2 v = part[w * 32 + lane];
        s = ff_add(s, ff{v.x, v.y});
    }
    const float kf = (float)k, q1 = s.hi / kf, q2 = (fmaf(-q1, kf, s.hi) + s.lo) / kf;
    for (int r = warp; r < k; r += NW) {
        float h, e;
        two_sum(Xr[r * XLD + lane], -q1, h, e);
        Xr[r * XLD + lane] = h + (e - q2);
    }
}

// FP32 means, rows in ascending order.  Ends before a barrier.
template <int NT>
__device__ __forceinline__ void centre_plain(float *Xr, int k, float2 *part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0) {
        float s = 0.f;
        for (int r = 0; r < k; ++r) s += Xr[r * XLD + lane];
        part[lane].x = s / (float)k;
    }
    __syncthreads();
    const float mean = part[lane].x;
    for (int r = warp; r < k; r += NT / 32) Xr[r * XLD + lane] -= mean;
}

// U[r][l] = u[r * k + l] (r < k; 0 for k <= l < kp), row stride ldu
template <int NT>
__device__ __forceinline__ void load_matrix(float *Us, const float *__restrict__ u, int k, int kp, int ldu) {
    for (int r = threadIdx.x >> 5; r < k; r += NT / 32)
        for (int l = threadIdx.x & 31; l < kp; l += 32) Us[r * ldu + l] = l < k ? u[r * k + l] : 0.f;
}

// Z = U^T X for a chunk: 4 rows x 2 columns per thread, packed along the rows,
// r ascending.  COL: Z column-major with stride ldu, else row-major like X.
template <int NT, bool COL>
__device__ __forceinline__ void rotate_chunk(const float *Xr, const float *Us, float *Z, int k, int kp, int ldu) {
    const int nl = kp >> 2;
    for (int u = threadIdx.x; u < nl * (MCH / 2); u += NT) {
        const int c2 = u / nl, l4 = u - c2 * nl;
        f2 z[2][2] = {};
#pragma unroll 4
        for (int r = 0; r < k; ++r) {
            const ulonglong2 ur = *reinterpret_cast<const ulonglong2 *>(Us + r * ldu + 4 * l4);
            const float2 x = *reinterpret_cast<const float2 *>(Xr + r * XLD + 2 * c2);
            const f2 x0 = pack2(x.x, x.x), x1 = pack2(x.y, x.y);
            z[0][0] = fma2(ur.x, x0, z[0][0]);
            z[0][1] = fma2(ur.y, x0, z[0][1]);
            z[1][0] = fma2(ur.x, x1, z[1][0]);
            z[1][1] = fma2(ur.y, x1, z[1][1]);
        }
        if (COL) {
#pragma unroll
            for (int c = 0; c < 2; ++c)
                *reinterpret_cast<ulonglong2 *>(Z + (2 * c2 + c) * ldu + 4 * l4) = make_ulonglong2(z[c][0], z[c][1]);
        } else {
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float2 a = unpack2(z[0][i]), b = unpack2(z[1][i]);
                *reinterpret_cast<float2 *>(Z + (4 * l4 + 2 * i) * XLD + 2 * c2) = make_float2(a.x, b.x);
                *reinterpret_cast<float2 *>(Z + (4 * l4 + 2 * i + 1) * XLD + 2 * c2) = make_float2(a.y, b.y);
            }
        }
    }
}

// Column-major copy of a chunk, rows k..kp-1 zero.
template <int NT>
__device__ __forceinline__ void transpose_chunk(const float *Xr, float *Z, int k, int kp, int ldz) {
    for (int c = threadIdx.x >> 5; c < MCH; c += NT / 32)
        for (int r = threadIdx.x & 31; r < kp; r += 32) Z[c * ldz + r] = r < k ? Xr[r * XLD + c] : 0.f;
}
}  // namespace

// ---------------------------------------------------------------------------
// Gram kernel: one CTA per point.  Thread u owns one 4 x 4 block (bi <= bj) of G,
// and of Q when it is wanted (both symmetric), as packed sums; 64 threads hold
// the 55 blocks of k = 40, 128 the 120 of k = 60, 160 the 136 of k = 64, and small
// CTAs leave room for many points on an SM, which hides the barriers between the
// steps of a chunk.  Measured (the plain and the rotated Gram of 20,000 points, 256
// columns, k = 32): 4.7 ms with FP64 centring by 64 threads, scalar operand loads
// and 64 of 256 threads at work, 1.7 without the next chunk under way, 1.5 with it
// (1.6 without the bound on the registers).
// ---------------------------------------------------------------------------
__host__ __device__ inline size_t gram_smem_floats(int k, bool rot, int nt) {
    const int kp = (k + 3) / 4 * 4, ldz = kp + 4;
    return (size_t)(rot ? k * ldz : 0) + MCH * ldz + kp * XLD + 2 * nt;
}

// largest k of a CTA of NT threads over its warps
constexpr int GRAM_NR(int nt) { return nt == 64 ? 20 : nt == 128 ? 15 : 13; }

template <typename T, int NT, bool ROT, bool WQ>
__global__ void __launch_bounds__(NT, NT == 64 ? 10 : NT == 128 ? 5 : 4)
patch_gram_kernel(const T *__restrict__ X, int64_t N, int64_t m, int64_t ld, const int32_t *__restrict__ idx,
                  int k, int64_t p0, const float *__restrict__ rot, float *__restrict__ G, float *__restrict__ R,
                  float *__restrict__ Q, DevCounters *ctr) {
    extern __shared__ __align__(16) float gsm[];
    const int kp = (k + 3) / 4 * 4, ldz = kp + 4, nb = kp / 4;
    float *Zc = gsm, *Us = Zc + MCH * ldz, *Xr = Us + (ROT ? k * ldz : 0);
    float2 *part = reinterpret_cast<float2 *>(Xr + kp * XLD);
    __shared__ float cw[MCH];
    __shared__ int rows[64];
    const int tid = threadIdx.x;
    const int64_t p = p0 + blockIdx.x;
    for (int j = tid; j < k; j += NT) rows[j] = checked_row(idx[p * k + j], N, ctr);
    if (ROT) load_matrix<NT>(Us, rot + (p - p0) * (int64_t)k * k, k, kp, ldz);
    int bi = 0, bj = tid;
    const bool active = tid < nb * (nb + 1) / 2;
    if (active)
        while (bj >= nb - bi) bj -= nb - bi++;
    bj += bi;
    f2 g[4][2] = {}, qq[4][2] = {};
    float rsum = 0.f;
    __syncthreads();
    ChunkRows<NT, GRAM_NR(NT)> next;
    next.load(X, ld, rows, k, 0, m);
    for (int64_t a0 = 0; a0 < m; a0 += MCH) {
        next.store(Xr, k);
        if (a0 + MCH < m) next.load(X, ld, rows, k, a0 + MCH, m);
        __syncthreads();
        if (ROT) centre_two_term<NT>(Xr, k, part);
        else centre_plain<NT>(Xr, k, part);
        __syncthreads();
        if (WQ && tid < MCH) {
            float w = 0.f;
            for (int r = 0; r < k; ++r) {
                const float v = Xr[r * XLD + tid];
                w = fmaf(v, v, w);
            }
            cw[tid] = w;
        }
        if (ROT) rotate_chunk<NT, true>(Xr, Us, Zc, k, kp, ldz);
        else transpose_chunk<NT>(Xr, Zc, k, kp, ldz);
        __syncthreads();
        if (active) {
#pragma unroll 4
            for (int c = 0; c < MCH; ++c) {
                const float4 a = *reinterpret_cast<const float4 *>(Zc + c * ldz + 4 * bi);
                const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(Zc + c * ldz + 4 * bj);
                const float xr[4] = {a.x, a.y, a.z, a.w};
                const float w = WQ ? cw[c] : 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const f2 x = pack2(xr[i], xr[i]);
                    g[i][0] = fma2(x, b.x, g[i][0]);
                    g[i][1] = fma2(x, b.y, g[i][1]);
                    if (WQ) {
                        const float z = xr[i] * w;
                        const f2 zz = pack2(z, z);
                        qq[i][0] = fma2(zz, b.x, qq[i][0]);
                        qq[i][1] = fma2(zz, b.y, qq[i][1]);
                    }
                }
            }
        }
        if (NT >= 64 && tid < k)
            for (int c = 0; c < MCH; ++c) rsum += Zc[c * ldz + tid];
        // the next write of Zc and cw follows two barriers, that of Xr comes after its last read
    }
    const int64_t kk = (int64_t)k * k;
    if (active) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 gv = unpack2(g[i][h]), qv = unpack2(qq[i][h]);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int r = 4 * bi + i, t = 4 * bj + 2 * h + e;
                    if (r < k && t < k && r <= t) {
                        const float v = e ? gv.y : gv.x;
                        G[(p - p0) * kk + (int64_t)r * k + t] = v;
                        G[(p - p0) * kk + (int64_t)t * k + r] = v;
                        if (WQ) {
                            const float q = e ? qv.y : qv.x;
                            Q[(p - p0) * kk + (int64_t)r * k + t] = q;
                            Q[(p - p0) * kk + (int64_t)t * k + r] = q;
                        }
                    }
                }
            }
    }
    if (tid < k) R[(p - p0) * k + tid] = rsum;
}

namespace {
template <typename T, int NT>
cudaError_t gram_launch(const T *X, int64_t N, int64_t m, int64_t ld, const int32_t *idx, int k, int64_t p0,
                        int64_t np, const float *rot, float *G, float *R, float *Q, DevCounters *ctr,
                        cudaStream_t s) {
    const size_t smem = gram_smem_floats(k, rot != nullptr, NT) * sizeof(float);  // 36.9 KB at most
    const unsigned n = (unsigned)np;
    if (rot && Q)
        patch_gram_kernel<T, NT, true, true><<<n, NT, smem, s>>>(X, N, m, ld, idx, k, p0, rot, G, R, Q, ctr);
    else if (rot)
        patch_gram_kernel<T, NT, true, false><<<n, NT, smem, s>>>(X, N, m, ld, idx, k, p0, rot, G, R, Q, ctr);
    else if (Q)
        patch_gram_kernel<T, NT, false, true><<<n, NT, smem, s>>>(X, N, m, ld, idx, k, p0, rot, G, R, Q, ctr);
    else
        patch_gram_kernel<T, NT, false, false><<<n, NT, smem, s>>>(X, N, m, ld, idx, k, p0, rot, G, R, Q, ctr);
    return cudaGetLastError();
}
template <typename T>
cudaError_t gram_dispatch(const T *X, int64_t N, int64_t m, int64_t ld, const int32_t *idx, int k, int64_t p0,
                          int64_t np, const float *rot, float *G, float *R, float *Q, DevCounters *ctr,
                          cudaStream_t s) {
    if (k <= 40) return gram_launch<T, 64>(X, N, m, ld, idx, k, p0, np, rot, G, R, Q, ctr, s);
    if (k <= 60) return gram_launch<T, 128>(X, N, m, ld, idx, k, p0, np, rot, G, R, Q, ctr, s);
    return gram_launch<T, 160>(X, N, m, ld, idx, k, p0, np, rot, G, R, Q, ctr, s);
}
}  // namespace

cudaError_t launch_patch_gram(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld,
                              const int32_t *idx, int k, int64_t p0, int64_t np, const float *rot,
                              float *G, float *R, float *Q, DevCounters *ctr, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    if (k > 64) return cudaErrorInvalidValue;
    if (dt == MECUCO_BF16)
        return gram_dispatch((const __nv_bfloat16 *)X, N, m, ld, idx, k, p0, np, rot, G, R, Q, ctr, s);
    return gram_dispatch((const float *)X, N, m, ld, idx, k, p0, np, rot, G, R, Q, ctr, s);
}

// ---------------------------------------------------------------------------
// Third moments.  Work items (j, Rb, Tb), Rb >= j/8, Tb >= Rb, over
// nb = ceil(k/8) blocks of 8 cover every sorted triple j <= r <= t; an item
// accumulates acc[r][t] = M[j][8Rb + r][8Tb + t] (64 accumulators, packed along
// t) and is one thread's.  A pass over the patch serves one item per thread; the
// CTA is the smallest of 96, 160, 288 and 480 threads that holds the items of k in
// one pass (80 items at k = 24, 160 at 32, 280 at 40, 448 at 48, 960 at 64: two).
//
// Two forms share the passes:
//  * MOMENTS: M is stored (the gradient and the randomised SVD need it), one CTA
//    per point and pass.
//    Storage is pair-major: D[pair(a, b)][c] = M[a][b][c] for a <= b and every c,
//    pair(a, b) = a k - a (a - 1)/2 + (b - a), so the slice M_j (k x k) is the k
//    contiguous rows pair(min(j, r), max(j, r)), r = 0..k-1.  Each sorted triple
//    a <= b <= c is written to its three images D[pair(a,b)][c], D[pair(a,c)][b]
//    and D[pair(b,c)][a] (the same value; coinciding images rewrite it).
//  * KAPPA: with V, s the eigenpairs of the Gram of Z, the chunk is rotated once
//    more, Y = V^T Z, and the items are S[a,b,c] = sum Y_a Y_b Y_c.  The estimator
//    terms then need no product with W: T^[(r,t), l] = S_rtl / (s_r s_t), and with
//    all images of a sorted triple |G_tens|^2 takes 2 (T^_ab,c^2 + T^_ac,b^2 +
//    T^_bc,a^2) from a < b < c (half of that with two equal indices, a sixth with
//    three), so M is neither written nor read and the pass over M that formed
//    W^T M_j W (k^3 p multiply-adds, as many as the third moments at m = 6 k)
//    is gone.
// Bound by the FP32 lanes: 64 multiply-adds a column and item in 32 packed
// instructions, and the steps between the barriers of a chunk.
// Measured (20,000 points, 256 columns, k = 32): 8.1 ms for M and 6.3 for the pass
// over it, 4.4 for KAPPA, 4.2 with the next chunk under way; the gradient's M (8,000
// points) 3.3 -> 1.6 ms.
// ---------------------------------------------------------------------------
int m3_items(int k) {
    int nb = (k + 7) / 8, n = 0;
    for (int j = 0; j < k; ++j) {
        int r0 = j / 8;
        n += (nb - r0) * (nb - r0 + 1) / 2;
    }
    return n;
}

void m3_build_items(int k, int32_t *items) {
    int nb = (k + 7) / 8, n = 0;
    for (int j = 0; j < k; ++j)
        for (int rb = j / 8; rb < nb; ++rb)
            for (int tb = rb; tb < nb; ++tb) items[n++] = j | (rb << 8) | (tb << 16);
}

namespace {
struct ThirdOut {
    float *M;                             // MOMENTS
    const float *V, *sigma, *R, *Q;       // KAPPA: eigenpairs, R and Q of Z
    int variant;
    float rank_eps;
    float *kappa, *lambda, *s;            // lambda, s nullable
};

__host__ __device__ inline size_t third_smem_floats(int k, bool kappa, int nt) {
    const int kp = (k + 7) / 8 * 8, ldz = kp + 4;
    return (size_t)(kappa ? 3 : 1) * kp * ldz + MCH * ldz + (kappa ? 2 : 1) * kp * XLD + 2 * nt;
}
}  // namespace

// largest k of a CTA of NT threads over its warps
constexpr int THIRD_NR(int nt) { return nt == 96 ? 8 : nt == 160 ? 7 : 5; }

template <typename T, int NT, int MINB, bool KAPPA>
__global__ void __launch_bounds__(NT, MINB)
patch_m3_kernel(const T *__restrict__ X, int64_t N, int64_t m, int64_t ld, const int32_t *__restrict__ idx,
                int k, int64_t p0, const float *__restrict__ rot, const int32_t *__restrict__ items, int nitems,
                ThirdOut out, DevCounters *ctr) {
    extern __shared__ __align__(16) float tsm[];
    const int kp = (k + 7) / 8 * 8, ldz = kp + 4;
    float *Yc = tsm, *Us = Yc + MCH * ldz, *Vs = Us + kp * ldz, *diag = Vs + (KAPPA ? kp * ldz : 0);
    float *Xr = diag + (KAPPA ? kp * ldz : 0), *Zr = Xr + kp * XLD;
    float2 *part = reinterpret_cast<float2 *>(Zr + (KAPPA ? kp * XLD : 0));
    __shared__ int rows[64];
    __shared__ float is_s[64], c_s[64];
    __shared__ float2 red[NT / 32][5];
    __shared__ int s_p;
    const int tid = threadIdx.x;
    const int64_t pt = blockIdx.x;  // the point within the launch
    const int64_t kk = (int64_t)k * k;
    for (int j = tid; j < k; j += NT) rows[j] = checked_row(idx[(p0 + pt) * k + j], N, ctr);
    if (rot) load_matrix<NT>(Us, rot + pt * kk, k, kp, ldz);
    int p = 0;
    if (KAPPA) {
        load_matrix<NT>(Vs, out.V + pt * kk, k, kp, ldz);
        if (tid < 32) {
            const int rank = fast_rank(out.sigma + pt * k, k, m, out.rank_eps, ctr);
            if (tid == 0) s_p = rank;
        }
        __syncthreads();
        p = s_p;
        if (tid < 64) is_s[tid] = tid < p ? __frsqrt_rn(out.sigma[pt * k + tid]) : 0.f;
    }
    ff gsum{0.f, 0.f};
    __syncthreads();
    for (int first = KAPPA ? 0 : (int)blockIdx.y * NT; first < nitems; first += NT) {
        int j = 0, rb = 0, tb = 0;
        const bool active = first + tid < nitems;
        if (active) {
            const int code = items[first + tid];
            j = code & 0xff;
            rb = (code >> 8) & 0xff;
            tb = (code >> 16) & 0xff;
        }
        f2 acc[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int t = 0; t < 4; ++t) acc[r][t] = 0ull;
        ChunkRows<NT, THIRD_NR(NT)> next;
        next.load(X, ld, rows, k, 0, m);
        for (int64_t a0 = 0; a0 < m; a0 += MCH) {
            next.store(Xr, k);
            if (a0 + MCH < m) next.load(X, ld, rows, k, a0 + MCH, m);
            __syncthreads();
            if (rot) centre_two_term<NT>(Xr, k, part);
            else centre_plain<NT>(Xr, k, part);
            __syncthreads();
            if (KAPPA) {
                rotate_chunk<NT, false>(Xr, Us, Zr, k, kp, ldz);
                __syncthreads();
                rotate_chunk<NT, true>(Zr, Vs, Yc, k, kp, ldz);
            } else if (rot) {
                rotate_chunk<NT, true>(Xr, Us, Yc, k, kp, ldz);
            } else {
                transpose_chunk<NT>(Xr, Yc, k, kp, ldz);
            }
            __syncthreads();
            if (active) {
#pragma unroll 2
                for (int c = 0; c < MCH; ++c) {
                    const float *col = Yc + c * ldz;
                    const float4 r0 = *reinterpret_cast<const float4 *>(col + 8 * rb);
                    const float4 r1 = *reinterpret_cast<const float4 *>(col + 8 * rb + 4);
                    const ulonglong2 t0 = *reinterpret_cast<const ulonglong2 *>(col + 8 * tb);
                    const ulonglong2 t1 = *reinterpret_cast<const ulonglong2 *>(col + 8 * tb + 4);
                    const float xj = col[j];
                    const float xr[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const float z = xj * xr[r];
                        const f2 zz = pack2(z, z);
                        acc[r][0] = fma2(zz, t0.x, acc[r][0]);
                        acc[r][1] = fma2(zz, t0.y, acc[r][1]);
                        acc[r][2] = fma2(zz, t1.x, acc[r][2]);
                        acc[r][3] = fma2(zz, t1.y, acc[r][3]);
                    }
                }
            }
            // the next write of Yc follows two barriers, that of Xr comes after its last read
        }
        if (active) {
            float *D = KAPPA ? nullptr : out.M + pt * m3_pair_floats_d(k);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int rr = 8 * rb + r;
                float part_sq = 0.f;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int tt = 8 * tb + t;
                    if (rr < j || tt < rr || tt >= k) continue;  // sorted triples j <= rr <= tt < k
                    const float2 v2 = unpack2(acc[r][t >> 1]);
                    const float v = (t & 1) ? v2.y : v2.x;
                    if (!KAPPA) {
                        D[(int64_t)pair_index(j, rr, k) * k + tt] = v;
                        D[(int64_t)pair_index(j, tt, k) * k + rr] = v;
                        D[(int64_t)pair_index(rr, tt, k) * k + j] = v;
                    } else {
                        const float ab = v * (is_s[j] * is_s[rr]), ac = v * (is_s[j] * is_s[tt]),
                                    bc = v * (is_s[rr] * is_s[tt]);
                        const bool e1 = j == rr, e2 = rr == tt;
                        const float sq = e1 && e2 ? ab * ab : fmaf(ab, ab, fmaf(ac, ac, bc * bc));
                        part_sq = fmaf(e1 || e2 ? 1.f : 2.f, sq, part_sq);
                        if (e1) diag[j * ldz + tt] = ab;   // T^[(j,j), tt]
                        if (e2) diag[rr * ldz + j] = bc;   // T^[(rr,rr), j]
                    }
                }
                if (KAPPA) gsum = sum_add(gsum, ff{part_sq, 0.f});
            }
        }
        if (!KAPPA) break;
    }
    if (!KAPPA) return;
    __syncthreads();
    float *Qs = Xr;  // k rows of ldz floats in the two chunk buffers (2 kp XLD >= k (kp + 4))
    if (out.variant == MECUCO_FAST_HAAR) load_matrix<NT>(Qs, out.Q + pt * kk, k, kp, ldz);
    __syncthreads();
    const float *sg = out.sigma + pt * k;
    fast_kappa<NT>(k, p, m, out.variant, gsum, sg, out.R + pt * k, diag, ldz, Vs, ldz, Qs, ldz, c_s, red,
                   out.kappa + pt);
    if (out.lambda && tid < k)
        out.lambda[pt * k + tid] = lambda_of(sg[tid], tid, p, k);
    if (out.s && tid < k) out.s[pt * k + tid] = sqrtf(pos_part(sg[tid]));
}

namespace {
template <typename T, int NT, int MINB, bool KAPPA>
cudaError_t third_launch(const T *X, int64_t N, int64_t m, int64_t ld, const int32_t *idx, int k, int64_t p0,
                         int64_t np, const float *rot, const int32_t *items, const ThirdOut &out, DevCounters *ctr,
                         cudaStream_t s) {
    const int n = m3_items(k);
    const size_t smem = third_smem_floats(k, KAPPA, NT) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(patch_m3_kernel<T, NT, MINB, KAPPA>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(third_smem_floats(64, KAPPA, NT) * sizeof(float)));
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)np, KAPPA ? 1u : (unsigned)((n + NT - 1) / NT));
    patch_m3_kernel<T, NT, MINB, KAPPA><<<grid, NT, smem, s>>>(X, N, m, ld, idx, k, p0, rot, items, n, out, ctr);
    return cudaGetLastError();
}
template <typename T, bool KAPPA>
cudaError_t third_dispatch(const T *X, int64_t N, int64_t m, int64_t ld, const int32_t *idx, int k, int64_t p0,
                           int64_t np, const float *rot, const int32_t *items, const ThirdOut &out,
                           DevCounters *ctr, cudaStream_t s) {
    if (k <= 24) return third_launch<T, 96, 5, KAPPA>(X, N, m, ld, idx, k, p0, np, rot, items, out, ctr, s);
    if (k <= 32) return third_launch<T, 160, 3, KAPPA>(X, N, m, ld, idx, k, p0, np, rot, items, out, ctr, s);
    if (k <= 40) return third_launch<T, 288, 2, KAPPA>(X, N, m, ld, idx, k, p0, np, rot, items, out, ctr, s);
    return third_launch<T, 480, 1, KAPPA>(X, N, m, ld, idx, k, p0, np, rot, items, out, ctr, s);
}
}  // namespace

cudaError_t launch_patch_m3(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld,
                            const int32_t *idx, int k, int64_t p0, int64_t np, const float *rot,
                            float *M, const int32_t *items, DevCounters *ctr, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    if (k > 64) return cudaErrorInvalidValue;
    ThirdOut out{};
    out.M = M;
    if (dt == MECUCO_BF16)
        return third_dispatch<__nv_bfloat16, false>((const __nv_bfloat16 *)X, N, m, ld, idx, k, p0, np, rot, items, out,
                                                    ctr, s);
    return third_dispatch<float, false>((const float *)X, N, m, ld, idx, k, p0, np, rot, items, out, ctr, s);
}

cudaError_t launch_patch_kappa(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld,
                               const int32_t *idx, int k, int64_t np, const float *rot, const float *sigma,
                               const float *V, const float *R, const float *Q, int variant, float rank_eps,
                               const int32_t *items, float *kappa, float *lambda_out, float *s_out,
                               DevCounters *ctr, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    if (k > 64 || !rot) return cudaErrorInvalidValue;
    ThirdOut out{};
    out.V = V;
    out.sigma = sigma;
    out.R = R;
    out.Q = Q;
    out.variant = variant;
    out.rank_eps = rank_eps;
    out.kappa = kappa;
    out.lambda = lambda_out;
    out.s = s_out;
    if (dt == MECUCO_BF16)
        return third_dispatch<__nv_bfloat16, true>((const __nv_bfloat16 *)X, N, m, ld, idx, k, 0, np, rot, items, out,
                                                   ctr, s);
    return third_dispatch<float, true>((const float *)X, N, m, ld, idx, k, 0, np, rot, items, out, ctr, s);
}

}  // namespace mecuco
