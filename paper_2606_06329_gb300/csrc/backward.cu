// backward.cu - adjoint of the Fast-mode estimator: d(sum_i g_i K_i)/dX with the
// neighbour lists frozen (K_i from eqs. tnull, tA, tB, fast_curv; Alg. 1).
//
// Per point the forward is a function of the patch moments G = X_c X_c^T,
// R = X_c 1, M (third moments), Q (Haar) and of the eigenpairs (s_l^2, u_l) of
// G (see the estimator kernel).  With W = U_p diag(s)^-1, S_j = W^T M_j W,
// A_jl = (S_j)_ll, xd_j = R_j - sum_l A_jl, gt2 = sum_j |S_j|_F^2,
// h = sum_l w_l^T Q w_l, c = 1/q (printed) or 1/(q+2) (Haar), km1 = k - 1 and
// f = (t_range + t_null)/2 + tau/2, K = |f|, g~ = g sign(f):
//   dA_jl   = g~ (A_jl - c xd_j) / km1          dR_j = g~ c xd_j / km1
//   dgt2    = g~ c / km1                        dh   = -2 g~ c / km1     (Haar)
//   dtau    = g~ (1/2 - c) (printed) or g~ (1/2 + c) (Haar)
//   dS_j    = 2 dgt2 S_j + diag(dA_j.)
//   dM_j    = W dS_j W^T,   dW += 2 M_j W dS_j,   dQ = dh W W^T,  dW += 2 dh Q W
//   ds2_l   = dtau/km1 - (1/2) s_l^-3 u_l^T dw_l,  du_l = dw_l / s_l   (l < p)
//   dG      = U (diag(ds2) + F o (U^T dU)) U^T (symmetrised), F_ij = 1/(s_j^2 - s_i^2)
// (the derivative of a symmetric eigendecomposition).  Back to the patch:
//   dX_c[i,a] = 2 (dG x_a)_i + dR_i + x_a^T C_i x_a
//               + 2 w_a (dQ x_a)_i + 2 X_c[i,a] x_a^T dQ x_a            (Haar)
// with x_a = X_c[:, a], w_a = sum_j X_c[j,a]^2 and C_i[r][t] = dM[i,r,t] +
// dM[r,i,t] + dM[t,i,r] (the fully symmetric use of M), then the centring
// adjoint dX_p = dX_c - 1 (1^T dX_c)/k and a scatter-add into dX rows idx[i,:].
// Degenerate eigenvalue pairs make F unbounded; the difference is clamped at
// 2^-40 max|s^2| in magnitude (the derivative there is not defined).
//
// Conditioning.  With s_min/s_max = 1e-3 the small eigenpairs of an FP32 Gram
// carry relative errors near eps (s_max/s_min)^2 = 1e-1 and the s^-3 terms of
// the adjoint amplify them.  K is invariant under any orthogonal rotation
// Z = U0^T X_c of the point axis (tau, t_range, t_A, |G_tens|^2 and the Haar
// sum are sums of squares over j), so the adjoint works on the rotated patch:
// U0 = eigenvectors of the plain FP32 Gram (held fixed: K does not depend on
// it; refined (Ogita-Aishima step), since a U0 that is not orthogonal to FP32 rounding
// perturbs the patch), the moments of Z (whose Gram is nearly diagonal, error
// near eps s_max/s_min) and the eigenpairs of that Gram; the formulas above
// give dZ, and dX_c = U0 dZ.
#include <math.h>

#include "common.cuh"
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

// k x k matrices in shared memory: rows of ld = k rounded up to 4, plus 4 floats.
__host__ __device__ inline int bw_ld(int k) { return (k + 3) / 4 * 4 + 4; }
__host__ __device__ inline size_t bw_smem_bytes(int k) {
    return (size_t)5 * ((k + 3) / 4 * 4) * bw_ld(k) * sizeof(float);
}

// Asynchronous copies into shared memory; a thread waits for its own groups.
template <int B>
__device__ __forceinline__ void cp_async(float *dst, const float *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// k rows of k floats, row r from src(r), to dst (row stride ld): 16-byte copies
// where the rows are aligned to them.  All NT threads; no commit.
template <int NT, typename F>
__device__ __forceinline__ void copy_rows_async(float *dst, int ld, int k, F src) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if ((k & 3) == 0) {
        const int q4 = k >> 2, rpw = 32 / q4, rr = lane / q4, c = 4 * (lane - rr * q4);
        if (rr < rpw)
            for (int r = warp * rpw + rr; r < k; r += NT / 32 * rpw) cp_async<16>(dst + r * ld + c, src(r) + c);
    } else {
        for (int r = warp; r < k; r += NT / 32)
            for (int c = lane; c < k; c += 32) cp_async<4>(dst + r * ld + c, src(r) + c);
    }
}

// v[i][c] = sum_{x < n} A[x][i0 + i] B[x][c0 + c], x ascending (rows of A and B
// stand for the product's contracted index).
__device__ __forceinline__ void tile_mul(const float *A, const float *B, int ld, int n, int i0, int c0,
                                         float (&v)[4][4]) {
    f2 acc[4][2] = {};
    for (int x = 0; x < n; ++x) {
        const float4 a = *reinterpret_cast<const float4 *>(A + x * ld + i0);
        const float4 b = *reinterpret_cast<const float4 *>(B + x * ld + c0);
        const f2 b0 = pack2(b.x, b.y), b1 = pack2(b.z, b.w);
        const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const f2 a2 = pack2(av[i], av[i]);
            acc[i][0] = fma2(a2, b0, acc[i][0]);
            acc[i][1] = fma2(a2, b1, acc[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 p = unpack2(acc[i][0]), q = unpack2(acc[i][1]);
        v[i][0] = p.x, v[i][1] = p.y, v[i][2] = q.x, v[i][3] = q.y;
    }
}
__device__ __forceinline__ void tile_store(float *D, int ld, int i0, int c0, const float (&v)[4][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4 *>(D + (i0 + i) * ld + c0) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
}
__device__ __forceinline__ void tile_store_t(float *D, int ld, int i0, int c0, const float (&v)[4][4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
        *reinterpret_cast<float4 *>(D + (c0 + c) * ld + i0) = make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
}
}  // namespace

// k-space adjoint: one CTA per point, a thread per 4 x 4 block of the k x k
// products (NT >= (k / 4)^2).  Outputs per point: dG (k x k), dR (k), dQ (k x k,
// Haar only), C (k x k rows of k rounded up to 8) as described above.
// One pass over j: every output is linear in g~ = g sign(f), and f (the forward
// value) only decides the sign, so the pass runs with g and the outputs take the
// sign at the end.  Per j five k x k x k products (M_j W, W^T B, B dS, W dS,
// (W dS) W^T) from 16-byte shared loads and packed FMAs, every sum in ascending
// order of its index.  Bound by the FP32 lanes and the shared reads that feed
// them; M_{j+1} is copied into shared memory behind the products of j.  Both
// adjoint kernels of 8,000 points at 256 columns, k = 32: 42.2 ms with two passes
// over j and scalar products, 11.8 with one pass on packed FMAs, 6.2 with the
// copies of M, dM and C (below) under way while the rows before are worked on.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
adjoint_kspace_kernel(const float *__restrict__ sigma, const float *__restrict__ U, const float *__restrict__ M,
                      const float *__restrict__ R, const float *__restrict__ Q, const float *__restrict__ gk, int k,
                      int64_t m, int variant, float rank_eps, float *__restrict__ dG, float *__restrict__ dR, float *__restrict__ dQ,
                      float *__restrict__ Cout, float *__restrict__ dMbuf) {
    extern __shared__ __align__(16) float bsm[];
    const int k4 = (k + 3) / 4 * 4, ld = bw_ld(k), nt = k4 / 4;
    float *W = bsm;              // W[r][l]
    float *Wt = W + k4 * ld;     // W[l][r]
    float *Ms = Wt + k4 * ld;    // M_j
    float *Bs = Ms + k4 * ld;    // M_j W, then dS_j
    float *Bt = Bs + k4 * ld;    // (M_j W)^T, then (W dS_j)^T
    __shared__ float Adiag[64], xd[64], sg[64];
    __shared__ double red[NT / 32][2];
    __shared__ float s_scal[8];
    __shared__ int s_p;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t pt = blockIdx.x;
    const float *u = U + pt * (int64_t)k * k;
    const float *D = M + pt * m3_pair_floats_d(k);
    const bool mine = tid < nt * nt;
    const int i0 = tid / nt * 4, c0 = tid % nt * 4;
    if (tid < k) sg[tid] = sigma[pt * k + tid];
    if (tid < 64) Adiag[tid] = 0.f;
    __syncthreads();
    const double km1 = (double)(k - 1);
    if (tid == 0) {
        int pmax = k - 1;
        if ((int64_t)pmax > m) pmax = (int)m;
        const float s0 = fmaxf(sg[0], 0.f);
        int rank = 0;
        for (int l = 0; l < k; ++l) rank += (sg[l] > rank_eps * s0) && (sg[l] > 0.f);
        const int p = rank < pmax ? rank : pmax;
        s_p = p;
        const int64_t q = m - p;
        const double cnull = q > 0 ? 1.0 / (double)(variant == MECUCO_FAST_HAAR ? q + 2 : q) : 0.0;
        const double g = (double)gk[pt];
        s_scal[0] = (float)(g * cnull / km1);  // dgt2
        s_scal[1] = (float)(g / km1);          // scale of dA
        s_scal[2] = (float)cnull;              // c
        s_scal[3] = (float)(g * (variant == MECUCO_FAST_HAAR ? 0.5 + cnull : 0.5 - cnull));  // dtau
        s_scal[4] = (float)(variant == MECUCO_FAST_HAAR ? -2.0 * g * cnull / km1 : 0.0);      // dh
    }
    __syncthreads();
    const int p = s_p;
    const int64_t q = m - p;
    const double cnull = q > 0 ? 1.0 / (double)(variant == MECUCO_FAST_HAAR ? q + 2 : q) : 0.0;
    for (int r = warp; r < k4; r += NT / 32)
        for (int l = lane; l < k4; l += 32) {
            const float w = (r < k && l < p) ? u[r * k + l] * rsqrtf(sg[l]) : 0.f;
            W[r * ld + l] = w;
            Wt[l * ld + r] = w;
            if (r >= k || l >= k) Ms[r * ld + l] = 0.f;
        }
    const float dg2 = s_scal[0], ga = s_scal[1], gc = s_scal[2];
    float dW[4][4] = {};
    double acc_range = 0.0, acc_gt2 = 0.0, acc_A = 0.0;
    auto load_m = [&](int j) {
        copy_rows_async<NT>(Ms, ld, k, [&](int r) {
            return D + (int64_t)pair_index(j < r ? j : r, j < r ? r : j, k) * k;
        });
        cp_async_commit();
    };
    load_m(0);
    for (int j = 0; j < k; ++j) {
        cp_async_wait<0>();
        __syncthreads();
        float v[4][4];
        // B = M_j W (M_j symmetric)
        if (mine) {
            tile_mul(Ms, W, ld, k, i0, c0, v);
            tile_store(Bs, ld, i0, c0, v);
            tile_store_t(Bt, ld, i0, c0, v);
        }
        __syncthreads();
        if (j + 1 < k) load_m(j + 1);  // M_j has been read
        // S = W^T B
        if (mine) {
            tile_mul(W, Bs, ld, k, i0, c0, v);
            float part = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) part += v[i][c] * v[i][c];
            acc_gt2 += part;
            if (i0 == c0)
#pragma unroll
                for (int i = 0; i < 4; ++i) Adiag[i0 + i] = v[i][i];
        }
        __syncthreads();
        float sa = 0.f, s2 = 0.f;
        for (int l = lane; l < p; l += 32) { const float a = Adiag[l]; sa += a; s2 += a * a; }
        sa = warp_sum(sa);
        s2 = warp_sum(s2);
        const float x = R[pt * k + j] - sa;
        if (tid == 0) {
            acc_range += s2;
            xd[j] = x;
            acc_A += (double)x * x;
        }
        // dS_j = 2 dgt2 S_j + diag(dA_j.), over B
        if (mine) {
            float ds[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    ds[i][c] = 2.f * dg2 * v[i][c];
                    if (i0 + i == c0 + c && i0 + i < p) ds[i][c] += ga * (v[i][c] - gc * x);
                }
            tile_store(Bs, ld, i0, c0, ds);
        }
        __syncthreads();
        if (mine) {
            // dW += 2 B dS_j; (W dS_j)^T over B^T
            tile_mul(Bt, Bs, ld, p, i0, c0, v);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) dW[i][c] = fmaf(2.f, v[i][c], dW[i][c]);
            tile_mul(Wt, Bs, ld, p, i0, c0, v);
        }
        __syncthreads();
        if (mine) tile_store_t(Bt, ld, i0, c0, v);
        __syncthreads();
        // dM_j = (W dS_j) W^T
        if (mine) {
            tile_mul(Bt, Wt, ld, p, i0, c0, v);
            float *dMj = dMbuf + (pt * (int64_t)k + j) * k * k;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i0 + i < k) {
                    float *row = dMj + (i0 + i) * k + c0;
                    if ((k & 3) == 0) {
                        *reinterpret_cast<float4 *>(row) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (c0 + c < k) row[c] = v[i][c];
                    }
                }
        }
    }
    // ---- the forward value's sign
    double v0 = acc_gt2, hpart = 0.0;
    const float *qm = Q + pt * (int64_t)k * k;
    if (variant == MECUCO_FAST_HAAR) {
        for (int e = tid; e < k * p; e += NT) {
            const int r = e / p, l = e % p;
            float t = 0.f;
            for (int c = 0; c < k; ++c) t = fmaf(qm[r * k + c], W[c * ld + l], t);
            hpart += (double)W[r * ld + l] * t;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        hpart += __shfl_xor_sync(0xffffffffu, hpart, o);
    }
    if (lane == 0) {
        red[warp][0] = v0;
        red[warp][1] = hpart;
    }
    __syncthreads();
    if (tid == 0) {
        double gt2 = 0.0, hsum = 0.0;
        for (int w = 0; w < NT / 32; ++w) {
            gt2 += red[w][0];
            hsum += red[w][1];
        }
        double tau = 0.0;
        for (int l = 0; l < p; ++l) tau += (double)sg[l];
        tau /= km1;
        const double t_range = acc_range / km1, t_A = acc_A / km1;
        double t_null = 0.0;
        if (q > 0) {
            const double tB = (variant == MECUCO_FAST_HAAR) ? tau - 2.0 * hsum / km1 + gt2 / km1 : -tau + gt2 / km1;
            t_null = (t_A + 2.0 * tB) * cnull;
        }
        const double f = 0.5 * (t_range + t_null) + 0.5 * tau;
        s_scal[6] = f > 0.0 ? 1.f : (f < 0.0 ? -1.f : 0.f);
        s_scal[5] = (float)((double)gk[pt] * cnull / km1);  // dR scale
    }
    __syncthreads();
    const float sgn = s_scal[6];
    if (tid < k) dR[pt * k + tid] = sgn * (s_scal[5] * xd[tid]);
    // ---- Haar: dQ = dh W W^T, dW += 2 dh Q W
    const float dh = s_scal[4];
    float v[4][4];
    if (variant == MECUCO_FAST_HAAR) {
        for (int r = warp; r < k; r += NT / 32)
            for (int t = lane; t < k; t += 32) Ms[r * ld + t] = qm[r * k + t];
        __syncthreads();
        if (mine) {
            tile_mul(Wt, Wt, ld, p, i0, c0, v);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (i0 + i < k && c0 + c < k)
                        dQ[pt * (int64_t)k * k + (i0 + i) * k + c0 + c] = sgn * (dh * v[i][c]);
            // Q symmetric: its rows stand for its columns
            tile_mul(Ms, W, ld, k, i0, c0, v);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int c = 0; c < 4; ++c) dW[i][c] += 2.f * dh * v[i][c];
        }
        __syncthreads();
    }
    // ---- eigen adjoint.  U over Ms, U^T over Wt, dW over Bt, then dU over Bs
    for (int r = warp; r < k4; r += NT / 32)
        for (int l = lane; l < k4; l += 32) {
            const float e = (r < k && l < k) ? u[r * k + l] : 0.f;
            Ms[r * ld + l] = e;
            Wt[l * ld + r] = e;
        }
    if (mine) {
        tile_store(Bt, ld, i0, c0, dW);
        float du[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float is = c0 + c < p ? rsqrtf(sg[c0 + c]) : 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) du[i][c] = c0 + c < p ? dW[i][c] * is : 0.f;
        }
        tile_store(Bs, ld, i0, c0, du);
    }
    __syncthreads();
    const float dtau = s_scal[3];
    if (tid < k) {
        const int l = tid;
        float e = 0.f;
        if (l < p) {
            float uw = 0.f;
            for (int r = 0; r < k; ++r) uw = fmaf(Ms[r * ld + l], Bt[r * ld + l], uw);
            const float s = sqrtf(sg[l]);
            e = dtau / (float)km1 - 0.5f * uw / (sg[l] * s);
        }
        Adiag[l] = e;
    }
    __syncthreads();
    // K = diag(ds2) + F o (U^T dU), over W
    float smax = 0.f;
    for (int l = 0; l < k; ++l) smax = fmaxf(smax, fabsf(sg[l]));
    const float floor_gap = smax * 9.094947017729282e-13f;  // 2^-40 max|s^2|
    if (mine) {
        tile_mul(Ms, Bs, ld, k, i0, c0, v);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int a = i0 + i, b = c0 + c;
                if (a >= k || b >= k) {
                    v[i][c] = 0.f;
                } else if (a == b) {
                    v[i][c] = Adiag[a];
                } else {
                    float dif = sg[b] - sg[a];
                    if (fabsf(dif) < floor_gap) dif = dif < 0.f ? -floor_gap : floor_gap;
                    v[i][c] = v[i][c] / dif;
                }
            }
        tile_store(W, ld, i0, c0, v);
    }
    __syncthreads();
    // dG = U K U^T, symmetrised: (U K)^T over Bs, then (U K) U^T over Bt
    if (mine) {
        tile_mul(Wt, W, ld, k, i0, c0, v);
        tile_store_t(Bs, ld, i0, c0, v);
    }
    __syncthreads();
    if (mine) {
        tile_mul(Bs, Wt, ld, k, i0, c0, v);
        tile_store(Bt, ld, i0, c0, v);
    }
    __syncthreads();
    for (int r = warp; r < k; r += NT / 32)
        for (int t = lane; t < k; t += 32)
            dG[pt * (int64_t)k * k + r * k + t] = sgn * (0.5f * (Bt[r * ld + t] + Bt[t * ld + r]));
    // ---- C_i[r][t] = dM[i,r,t] + dM[r,i,t] + dM[t,i,r]: the rows dM[r, i, .] and
    // dM[i, r, .] staged in shared memory, those of i + 1 on the way while C_i is
    // written, so that every global access is along a row
    const float *dMp = dMbuf + pt * (int64_t)k * k * k;
    const int k8 = (k + 7) / 8 * 8;  // C's rows, zero past k
    float *Cp = Cout + pt * (int64_t)k * k * k8;
    float *across[2] = {W, Ms}, *along[2] = {Wt, Bs};
    auto load_c = [&](int i) {
        copy_rows_async<NT>(i & 1 ? across[1] : across[0], ld, k, [&](int r) { return dMp + (r * k + i) * k; });
        copy_rows_async<NT>(i & 1 ? along[1] : along[0], ld, k, [&](int r) { return dMp + (i * k + r) * k; });
        cp_async_commit();
    };
    load_c(0);  // W, Ms, Wt and Bs were last read before the barrier above; dM_j was written before many
    for (int i = 0; i < k; ++i) {
        cp_async_wait<0>();
        __syncthreads();
        if (i + 1 < k) load_c(i + 1);  // its buffers were read in the step before
        const float *ac = i & 1 ? across[1] : across[0], *al = i & 1 ? along[1] : along[0];
        for (int r = warp; r < k; r += NT / 32)
            for (int t = lane; t < k8; t += 32)
                Cp[(i * k + r) * k8 + t] =
                    t < k ? sgn * (al[r * ld + t] + ac[r * ld + t] + ac[t * ld + r]) : 0.f;
    }
}

// Patch-space adjoint and scatter: one CTA (256 threads) per point; the patch
// is re-gathered, centred and rotated (Z = U0^T X_c) in chunks of 128 columns
// (four per lane of every warp).  Warp w forms rows i = w, w + 8, ... of dZ:
// 2 dG z + dR and the quadratic form z^T C_i z, whose matrix is symmetric, by 8 x
// 8 blocks on and above the diagonal (the ones above count twice) - 8 rows of C_i
// z for 4 columns in registers, packed along the rows.  The warp copies the next
// AP_ROWS rows of such a block column into its own pair of buffers while it works
// on the present ones, whose entries it reads as uniform 16-byte loads.  Then dX_c = U0 dZ, the centring adjoint subtracts
// the column mean, and the result is atomically added to dX rows idx[pt, :].
// Bound by the FP32 lanes (the quadratic forms: k^3 multiply-adds a column); the
// figures stand at adjoint_kspace_kernel.
constexpr int AP_CH = 128;
constexpr int AP_ROWS = 32;  // rows of C_i per buffer
__host__ __device__ inline size_t adjoint_patch_smem(int k) {
    const size_t k8 = (k + 7) / 8 * 8;
    return sizeof(float) * (2 * k8 * AP_CH + 8 * 2 * AP_ROWS * 8 + 2 * AP_CH + 64 * 65);
}

// A run of rows [s0, s1) of the block column r0 of C_i: the rows right of the
// diagonal block (i.e. below it, C_i being symmetric) in runs of AP_ROWS, then the
// diagonal block's own, then the next block column, then the warp's next i.
struct AdjRun {
    int i, r0, s0, s1;
    bool diag;
    __device__ void start(int k) {
        s0 = r0 + 8;
        diag = s0 >= k;
        if (diag) s0 = r0;
        s1 = diag ? k : min(s0 + AP_ROWS, k);
    }
    __device__ void next(int k) {
        if (!diag && s1 < k) {
            s0 = s1;
            s1 = min(s0 + AP_ROWS, k);
        } else if (!diag) {
            diag = true;
            s0 = r0;
            s1 = r0 + 8;
        } else {
            r0 += 8;
            if (r0 >= k) {
                r0 = 0;
                i += 8;
            }
            start(k);
        }
    }
};

// sum over rows l < k of Us(l) * Z[l][4 lane ..], as two packed pairs
template <typename F>
__device__ __forceinline__ float4 row_mix(const float *Z, int k, int lane, F coef) {
    f2 a0 = 0, a1 = 0;
    for (int l = 0; l < k; ++l) {
        const float u = coef(l);
        const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(Z + l * AP_CH + 4 * lane);
        const f2 u2 = pack2(u, u);
        a0 = fma2(u2, z.x, a0);
        a1 = fma2(u2, z.y, a1);
    }
    const float2 p = unpack2(a0), q = unpack2(a1);
    return make_float4(p.x, p.y, q.x, q.y);
}

template <typename T>
__global__ void __launch_bounds__(256, 2)
adjoint_patch_kernel(const T *__restrict__ X, int64_t N, int64_t m, int64_t ld, const int32_t *__restrict__ idx, int k,
                     int variant, const float *__restrict__ rot, const float *__restrict__ dG,
                     const float *__restrict__ dR,
                     const float *__restrict__ dQ, const float *__restrict__ C, float *__restrict__ dX, int64_t ldd) {
    extern __shared__ __align__(16) float psm[];
    const int kk = k * k, k8 = (k + 7) / 8 * 8;
    float *Xs = psm;                  // [k8][AP_CH] X_c, then dZ
    float *Zs = Xs + k8 * AP_CH;      // [k8][AP_CH] Z (rows k .. zero), then dX_c
    float *Cs = Zs + k8 * AP_CH;      // per warp: two buffers of AP_ROWS x 8 of C_i
    float *wa = Cs + 8 * 2 * AP_ROWS * 8, *xq = wa + AP_CH;  // Haar: |z|^2, z^T dQ z per column
    float(*Us)[65] = reinterpret_cast<float(*)[65]>(xq + AP_CH);
    __shared__ int rows[64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t pt = blockIdx.x;
    const bool haar = variant == MECUCO_FAST_HAAR;
    if (tid < k) {
        int r = idx[pt * k + tid];
        rows[tid] = (r < 0 || (int64_t)r >= N) ? 0 : r;
    }
    load_rotation(rot + pt * (int64_t)kk, k, Us);
    __syncthreads();
    const float *Cp = C + pt * (int64_t)kk * k8;
    const float *Gp = dG + pt * (int64_t)kk, *Qp = dQ + pt * (int64_t)kk;
    const float *dRp = dR + pt * k;
    for (int64_t a0 = 0; a0 < m; a0 += AP_CH) {
        for (int j = warp; j < k; j += 8)
            for (int c = lane; c < AP_CH; c += 32)
                Xs[j * AP_CH + c] = a0 + c < m ? load_elem(X + (int64_t)rows[j] * ld + a0 + c) : 0.f;
        __syncthreads();
        if (tid < AP_CH) {
            // centred values rounded once from a two-term mean
            ff sd{0.f, 0.f};
            for (int j = 0; j < k; ++j) sd = ff_add(sd, ff{Xs[j * AP_CH + tid], 0.f});
            // sd / k: quotient, then the remainder's quotient
            const float kf = (float)k, qh = sd.hi / kf;
            const float ql = (fmaf(-qh, kf, sd.hi) + sd.lo) / kf;
            for (int j = 0; j < k; ++j) {
                float h, e;
                two_sum(Xs[j * AP_CH + tid], -qh, h, e);
                Xs[j * AP_CH + tid] = h + (e - ql);
            }
        }
        __syncthreads();
        for (int l = warp; l < k8; l += 8) {  // Z = U0^T X_c (rows past k come out zero)
            const float4 z = row_mix(Xs, k, lane, [&](int r) { return Us[r][l]; });
            *reinterpret_cast<float4 *>(Zs + l * AP_CH + 4 * lane) = z;
        }
        __syncthreads();
        if (haar) {
            if (tid < AP_CH) {
                float w = 0.f, t = 0.f;
                for (int j = 0; j < k; ++j) w = fmaf(Zs[j * AP_CH + tid], Zs[j * AP_CH + tid], w);
                for (int r = 0; r < k; ++r) {
                    float s = 0.f;
                    for (int c = 0; c < k; ++c) s = fmaf(__ldg(Qp + r * k + c), Zs[c * AP_CH + tid], s);
                    t = fmaf(Zs[r * AP_CH + tid], s, t);
                }
                wa[tid] = w;
                xq[tid] = t;
            }
            __syncthreads();
        }
        float *Cw = Cs + warp * 2 * AP_ROWS * 8;
        int buf = 0;
        AdjRun nx{warp, 0, 0, 0, false};
        nx.start(k);
        auto load_run = [&](const AdjRun &run, float *dst) {
            if (run.i < k && run.s0 + lane < run.s1) {
                const float *src = Cp + ((int64_t)run.i * k + run.s0 + lane) * k8 + run.r0;
                cp_async<16>(dst + lane * 8, src);
                cp_async<16>(dst + lane * 8 + 4, src + 4);
            }
            cp_async_commit();
        };
        load_run(nx, Cw);
        for (int i = warp; i < k; i += 8) {
            const float4 g = row_mix(Zs, k, lane, [&](int r) { return __ldg(Gp + i * k + r); });
            float y[4] = {2.f * g.x, 2.f * g.y, 2.f * g.z, 2.f * g.w};
            if (haar) {
                const float4 qv = row_mix(Zs, k, lane, [&](int r) { return __ldg(Qp + i * k + r); });
                const float qe[4] = {qv.x, qv.y, qv.z, qv.w};
                const float4 zi = *reinterpret_cast<const float4 *>(Zs + i * AP_CH + 4 * lane);
                const float ze[4] = {zi.x, zi.y, zi.z, zi.w};
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    y[c] += 2.f * wa[4 * lane + c] * qe[c] + 2.f * ze[c] * xq[4 * lane + c];
            }
            f2 cq[4] = {};
            for (int r0 = 0; r0 < k; r0 += 8) {
                f2 t[4][4] = {};  // [row pair][column]
                bool diag;
                do {
                    const AdjRun run = nx;  // of this i and r0
                    nx.next(k);
                    load_run(nx, Cw + (buf ^ 1) * AP_ROWS * 8);
                    cp_async_wait<1>();  // the present run has landed
                    __syncwarp();
                    const float *cb = Cw + buf * AP_ROWS * 8, *zs = Zs + run.s0 * AP_CH + 4 * lane;
                    diag = run.diag;
                    if (diag) {  // what came before counts twice
                        const f2 two = pack2(2.f, 2.f);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
#pragma unroll
                            for (int c = 0; c < 4; ++c) t[e][c] = fma2(t[e][c], two, 0ull);
                    }
#pragma unroll 4
                    for (int s = 0; s < run.s1 - run.s0; ++s) {
                        const float4 z = *reinterpret_cast<const float4 *>(zs + s * AP_CH);
                        const ulonglong2 c0 = *reinterpret_cast<const ulonglong2 *>(cb + s * 8);
                        const ulonglong2 c1 = *reinterpret_cast<const ulonglong2 *>(cb + s * 8 + 4);
                        const f2 cp[4] = {c0.x, c0.y, c1.x, c1.y};
                        const float zc[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const f2 z2 = pack2(zc[c], zc[c]);
#pragma unroll
                            for (int e = 0; e < 4; ++e) t[e][c] = fma2(cp[e], z2, t[e][c]);
                        }
                    }
                    __syncwarp();  // the buffer has been read
                    buf ^= 1;
                } while (!diag);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float4 za = *reinterpret_cast<const float4 *>(Zs + (r0 + 2 * e) * AP_CH + 4 * lane);
                    const float4 zb = *reinterpret_cast<const float4 *>(Zs + (r0 + 2 * e + 1) * AP_CH + 4 * lane);
                    cq[0] = fma2(pack2(za.x, zb.x), t[e][0], cq[0]);
                    cq[1] = fma2(pack2(za.y, zb.y), t[e][1], cq[1]);
                    cq[2] = fma2(pack2(za.z, zb.z), t[e][2], cq[2]);
                    cq[3] = fma2(pack2(za.w, zb.w), t[e][3], cq[3]);
                }
            }
            const float dr = dRp[i];
            float out[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float2 h = unpack2(cq[c]);
                out[c] = dr + y[c] + (h.x + h.y);
            }
            *reinterpret_cast<float4 *>(Xs + i * AP_CH + 4 * lane) = make_float4(out[0], out[1], out[2], out[3]);
        }
        __syncthreads();
        // dX_c = U0 dZ, the mean over the rows out, scatter
        for (int j = warp; j < k; j += 8) {
            const float4 v = row_mix(Xs, k, lane, [&](int l) { return Us[j][l]; });
            *reinterpret_cast<float4 *>(Zs + j * AP_CH + 4 * lane) = v;
        }
        __syncthreads();
        if (tid < AP_CH) {
            float s = 0.f;
            for (int j = 0; j < k; ++j) s += Zs[j * AP_CH + tid];
            wa[tid] = s / (float)k;
        }
        __syncthreads();
        for (int j = warp; j < k; j += 8)
            for (int c = lane; c < AP_CH; c += 32)
                if (a0 + c < m) atomicAdd(dX + (int64_t)rows[j] * ldd + a0 + c, Zs[j * AP_CH + c] - wa[c]);
        __syncthreads();
    }
}

cudaError_t launch_adjoint(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld, const int32_t *idx,
                           int k, int64_t np, int variant, float rank_eps, const float *rot, const float *sigma,
                           const float *U, const float *M, const float *R, const float *Q, const float *gk, float *dG,
                           float *dR, float *dQ, float *C, float *dMbuf, float *dX, int64_t ldd, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    if (k > 64) return cudaErrorInvalidValue;
    const size_t smem = bw_smem_bytes(k);
    auto kspace = [&](auto kern, int nt) -> cudaError_t {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (r != cudaSuccess) return r;
        kern<<<(unsigned)np, nt, smem, s>>>(sigma, U, M, R, Q, gk, k, m, variant, rank_eps, dG, dR, dQ, C, dMbuf);
        return cudaGetLastError();
    };
    // one thread per 4 x 4 block: 64 threads to k = 32, 128 to 44, else 256
    cudaError_t e = k <= 32   ? kspace(adjoint_kspace_kernel<64, 8>, 64)
                    : k <= 44 ? kspace(adjoint_kspace_kernel<128, 4>, 128)
                              : kspace(adjoint_kspace_kernel<256, 2>, 256);
    if (e != cudaSuccess) return e;
    const size_t psmem = adjoint_patch_smem(k);
    if (dt == MECUCO_BF16) {
        e = cudaFuncSetAttribute(adjoint_patch_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)psmem);
        if (e != cudaSuccess) return e;
        adjoint_patch_kernel<<<(unsigned)np, 256, psmem, s>>>((const __nv_bfloat16 *)X, N, m, ld, idx, k, variant, rot,
                                                              dG, dR, dQ, C, dX, ldd);
    } else {
        e = cudaFuncSetAttribute(adjoint_patch_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem);
        if (e != cudaSuccess) return e;
        adjoint_patch_kernel<<<(unsigned)np, 256, psmem, s>>>((const float *)X, N, m, ld, idx, k, variant, rot, dG, dR,
                                                              dQ, C, dX, ldd);
    }
    return cudaGetLastError();
}

}  // namespace mecuco
