// fast_terms.cuh - the Fast estimator's sums of one point from its third moments
// in the rotated basis (the tensor-core and the FP32 third-moment kernels).
#pragma once

#include "common.cuh"

namespace mecuco {

// Two-term sums and products whose overflow gives an infinity (the plain forms
// give NaN: the error term of an infinite sum is inf - inf).
__device__ __forceinline__ float finite_err(float hi, float err) { return fabsf(hi) <= 3.402823466e+38f ? err : 0.f; }
__device__ __forceinline__ ff sum_add(ff a, ff b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e = finite_err(s, e + (a.lo + b.lo));
    const float h = s + e;
    return ff{h, finite_err(h, e - (h - s))};
}
__device__ __forceinline__ ff sum_mul(float a, float b) {
    const float h = __fmul_rn(a, b);
    return ff{h, finite_err(h, __fmaf_rn(a, b, -h))};
}
__device__ __forceinline__ ff sum_warp(ff v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = sum_add(v, ff_shfl_xor(v, o));
    return v;
}

// Numerical rank p of a point: eigenvalues above rank_eps * s_0 (the rounding
// scale of the Gram that was solved), at most min(k - 1, m); counts a point below
// that.  Called by one warp, the result in every lane.
__device__ __forceinline__ int fast_rank(const float *__restrict__ sg, int k, int64_t m, float rank_eps,
                                         DevCounters *ctr) {
    const int lane = threadIdx.x & 31;
    const float a = lane < k ? sg[lane] : 0.f, b = lane + 32 < k ? sg[lane + 32] : 0.f;
    const float lim = rank_eps * fmaxf(__shfl_sync(0xffffffffu, a, 0), 0.f);
    const int rank = __popc(__ballot_sync(0xffffffffu, a > lim && a > 0.f)) +
                     __popc(__ballot_sync(0xffffffffu, b > lim && b > 0.f));
    const int pmax = (int64_t)(k - 1) > m ? (int)m : k - 1;
    if (lane == 0 && rank < pmax) atomicAdd(&ctr->rank_deficient, 1ull);
    return rank < pmax ? rank : pmax;
}

// kappa of one point.  gsum: the thread's part of |G_tens|^2; diag[r * ldd + l] =
// T^[(r,r), l] (r < p, l < k); Us, Qs: U and Q of the point in shared memory (Q for
// the Haar variant only), R and the eigenvalues sg in global memory; c_s (64) and
// red (a row per warp): scratch in shared memory.  Called by all THREADS threads (k <=
// 64 <= THREADS), Us, Qs and diag visible to all.
// The sums of squares, the quadratic forms' sums over the rows of Q and tau are
// two-term FP32 (2^-44 and better); c_l, the entries of U c and the products Q u are
// FP32 chains of at most 64 terms.  FP64 runs at 1/64 of the FP32 rate.  A CTA has nothing else to do meanwhile, so what counts is the length of
// the dependent chains: the sums of squares and the k quadratic forms of Q are
// spread over all threads, eight lanes to a form, and the two reciprocals in FP64
// are computed beside them (one thread per form: 44,000 of the 95,000 cycles that a
// point of 301 columns took at k = 37, Haar; 30,000 points 5.0 -> 3.8 ms).
template <int THREADS>
__device__ __forceinline__ void fast_kappa(int k, int p, int64_t m, int variant, ff gsum,
                                           const float *__restrict__ sg, const float *__restrict__ R,
                                           const float *diag, int ldd, const float *Us, int ldu, const float *Qs,
                                           int ldq, float *c_s, float2 (*red)[5], float *__restrict__ kappa) {
    constexpr int NW = THREADS / 32;
    __shared__ double recip[2];  // 1 / (k - 1); 1 / q, or 1 / (q + 2) for the Haar variant (0 for q = 0)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t q = m - p;
    if (tid == THREADS - 1) {
        recip[0] = 1.0 / (double)(k - 1);
        recip[1] = q > 0 ? 1.0 / (double)(variant == MECUCO_FAST_HAAR ? q + 2 : q) : 0.0;
    }
    ff dsum{0.f, 0.f}, xa2{0.f, 0.f}, hsum{0.f, 0.f}, tsum{0.f, 0.f};
    if (tid < k) {
        // c_l = sum_{r<p} T^[(r,r), l], r ascending
        const int l = tid;
        float cl = 0.f;
#pragma unroll 8
        for (int r = 0; r < p; ++r) cl += diag[r * ldd + l];
        c_s[l] = cl;
        if (l < p) tsum.hi = sg[l];
    }
    // t_range's sum: rows of T^[(r,r), .] by warp
    for (int r = warp; r < p; r += NW)
        for (int l = lane; l < k; l += 32) {
            const float v = diag[r * ldd + l];
            dsum = sum_add(dsum, sum_mul(v, v));
        }
    if (variant == MECUCO_FAST_HAAR) {
        // u_l^T Q u_l / s_l^2: eight lanes per l, lane g rows g, g + 8, ... of Q
        const int g = lane & 7;
        for (int l0 = 0; l0 < p; l0 += THREADS / 8) {
            const int l = l0 + (tid >> 3), lc = l < p ? l : 0;
            float qu[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) qu[i] = 0.f;
            const int na = (k + 7) / 8;
            for (int b = 0; b < k; ++b) {
                const float u = Us[b * ldu + lc];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i < na) qu[i] = fmaf(Qs[min(g + 8 * i, k - 1) * ldq + b], u, qu[i]);
            }
            ff acc{0.f, 0.f};
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (g + 8 * i < k) acc = sum_add(acc, sum_mul(Us[(g + 8 * i) * ldu + lc], qu[i]));
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) acc = sum_add(acc, ff_shfl_xor(acc, o));
            if (g == 0 && l < p) {
                const float s = sg[l], q1 = acc.hi / s;
                hsum = sum_add(hsum, ff{q1, finite_err(q1, (fmaf(-q1, s, acc.hi) + acc.lo) / s)});
            }
        }
    }
    __syncthreads();
    if (tid < k) {
        // X_c d_P = R - U c
        const int j = tid;
        float uc = 0.f;
#pragma unroll 8
        for (int l = 0; l < k; ++l) uc = fmaf(Us[j * ldu + l], c_s[l], uc);
        float h, e;
        two_sum(R[j], -uc, h, e);
        xa2 = sum_mul(h, h);
        xa2.lo = finite_err(xa2.hi, xa2.lo + 2.f * h * e);
    }
    gsum = sum_warp(gsum);
    dsum = sum_warp(dsum);
    if (variant == MECUCO_FAST_HAAR) hsum = sum_warp(hsum);
    if (warp < 2) {  // the threads that hold any of these
        xa2 = sum_warp(xa2);
        tsum = sum_warp(tsum);
    }
    if (lane == 0) {
        red[warp][0] = make_float2(gsum.hi, gsum.lo);
        red[warp][1] = make_float2(dsum.hi, dsum.lo);
        red[warp][2] = make_float2(xa2.hi, xa2.lo);
        red[warp][3] = make_float2(hsum.hi, hsum.lo);
        red[warp][4] = make_float2(tsum.hi, tsum.lo);
    }
    __syncthreads();
    if (tid < 32) {
        // warp w's terms in lane w
        ff t[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const float2 v = lane < NW ? red[lane][c] : make_float2(0.f, 0.f);
            t[c] = sum_warp(ff{v.x, v.y});
        }
        if (lane == 0) {
            const double ik = recip[0];
            const double gt2 = (double)t[0].hi + (double)t[0].lo, d2 = (double)t[1].hi + (double)t[1].lo;
            const double a2 = (double)t[2].hi + (double)t[2].lo, h = (double)t[3].hi + (double)t[3].lo;
            const double tau = ((double)t[4].hi + (double)t[4].lo) * ik;
            const double t_range = d2 * ik, t_A = a2 * ik;
            double t_null = 0.0;
            if (q > 0) {
                // |X_c V_r|_F^2 / (k-1) = tau in the literal form
                const double tB = variant == MECUCO_FAST_HAAR ? tau + (gt2 - 2.0 * h) * ik : gt2 * ik - tau;
                t_null = (t_A + 2.0 * tB) * recip[1];
            }
            *kappa = (float)fabs(0.5 * (t_range + t_null) + 0.5 * tau);
        }
    }
}

}  // namespace mecuco
