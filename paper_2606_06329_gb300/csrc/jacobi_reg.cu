// jacobi_reg.cu - Step 3 (eq. svd_cov; Alg. 1 SVD_p): the eigenvectors of each
// k x k patch Gram G = X_c X_c^T to the accuracy a refinement step needs
// (jacobi_refine_res_kernel follows), as a register-resident one-sided Jacobi.
//
// With a diagonally pivoted Cholesky factor G = L L^T, plane rotations of L's
// columns until they are mutually orthogonal give L V = U diag(s) (Veselic &
// Hari, Numer. Math. 56, 1989): the normalised columns are the eigenvectors
// and the squared column norms the eigenvalues, so neither G nor V is updated.
//
// Layout.  R = 8 ceil(k / 8) columns (zero past the k-th) of R rows;
// a group of R / 2 lanes holds one patch, lane i two whole columns x_i, y_i in
// registers (two rows per 64-bit register, packed FP32 FMAs).  A warp holds
// 32 / (R / 2) patches, and a patch never leaves its warp: no block barrier.
// A round rotates every lane's own pair - the inner product needs no
// shuffles - and then passes the y columns to the next lane of the ring.  In
// every second round one lane (the seam) exchanges its two columns instead of
// rotating them, and the seam moves back by one lane: R rounds meet each of
// the R (R - 1) / 2 pairs exactly once (the odd-even transposition order on a
// ring), with one column per lane moving per round.
// Rounds come in twos: the first applies the unscaled rotation x - t y,
// y + t x (two FMAs per row) and leaves the common factor c to the second,
// whose four coefficients absorb it.  Squared norms follow the rotations'
// exact updates and are recomputed every sweep.  The solve ends after a sweep whose
// largest |cos(x, y)| stayed below 2^-17.  Where all gaps are wide the next sweep would
// square that, but inside a cluster of eigenvalues a tiny inner product still turns
// two columns by any angle, which undoes earlier rotations to the size of the bound:
// with a bound of 2^-10, 64 eigenvalues 2^-12 apart kept residuals of 1e-3 lambda_1.
// (2^-17 costs a sweep on many patches: 30,000 of 301 columns at k = 37 11.1 to 11.3
// ms in all, a batch of 12 sets 54.2 to 55.3.)
//
// The factor is that of G + eps I, eps = 2^-13 of the largest diagonal entry,
// which has the same eigenvectors: the Gram of a centred patch is singular (its
// rows sum to zero) and in FP32 its smallest eigenvalue is rounding noise of
// either sign, on which a Cholesky of G itself would break down - dropping the
// last pivot moved the small eigenvectors by up to 50x the Gram's own noise.
// With the shift every pivot is above eps - noise (and clamped at eps / 4), so
// U always comes out as a full orthonormal basis, rank-deficient patches
// included.  The shift costs no accuracy: the rotations resolve inner products
// to 2^-24 of the column norms, i.e. G to 2^-24 (lambda + eps), and G carries
// noise of 2^-24 lambda_1 anyway.
//
// Measured (GB300, 2.07 GHz, per 100k patches of the curved-patch spectrum at 1,024
// columns, with the refinement): k = 64 42.2 ms, k = 50 31.2, k = 37 14.9, k = 32 5.4, k =
// 24 3.8 (37.7, 27.7, 13.5, 5.0 and 3.4 with the bound 2^-10 and the refinement of first
// order alone; the fused two-sided sweeps alone 127, 68, 40, 31 and 20); after the
// refinement U^T U - I is at most 1e-6, against 4e-5 to 2e-4.
// What bounds it: latency at the warps that fit (254 registers a thread at R = 64, no
// spills, two warps per scheduler, 150k warp instructions per patch; three warps at 168
// registers spill more than they hide and take 10% longer).  R <= 56 runs three warps
// per scheduler at 168 registers and spills 480 bytes a thread, R <= 32 four.  The floor
// per round and warp at R = 64 is 64 shuffles (one warp instruction per clock per SM)
// and 32 + 96 packed FMAs: about 8 warp instructions per rotation, against about 96 and
// 8 to 16 shared-memory words per row pair in jacobi_warp_kernel.
#include <math.h>

#include "common.cuh"
#include "kernels.h"

namespace mecuco {
namespace {

typedef unsigned long long f2;  // two FP32 rows of a column

__device__ __forceinline__ f2 pack2(float lo, float hi) {
    f2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void unpack2(f2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

constexpr float JR_SHIFT = 1.220703125e-04f;  // 2^-13: the shift eps, on the scaled Gram
constexpr float JR_STOP2 = 5.820766091346741e-11f;  // 2^-34: the last sweep's squared cosines stay below it

__host__ __device__ constexpr int jr_rows(int k) { return k <= 16 ? 16 : (k + 7) / 8 * 8; }
// patches per warp
__host__ __device__ constexpr int jr_ppw(int k) { return 32 / (jr_rows(k) / 2); }
// shared floats of a warp: its patches' R columns of R + 4
__host__ __device__ constexpr int jr_floats_r(int R) { return 32 / (R / 2) * R * (R + 4); }

// warps per block and blocks per SM of the instantiation for R <= RMAX
constexpr int jr_warps(int RMAX) { return RMAX > 56 ? 2 : 4; }
constexpr int jr_blocks(int RMAX) { return RMAX > 56 ? 4 : (RMAX > 32 ? 3 : 4); }

template <int NP>
__device__ __forceinline__ float dot_cols(const f2 (&a)[NP], const f2 (&b)[NP]) {
    f2 s0 = 0, s1 = 0, s2 = 0, s3 = 0;
#pragma unroll
    for (int q = 0; q < NP; q += 4) {
        s0 = fma2(a[q], b[q], s0);
        s1 = fma2(a[q + 1], b[q + 1], s1);
        s2 = fma2(a[q + 2], b[q + 2], s2);
        s3 = fma2(a[q + 3], b[q + 3], s3);
    }
    float l0, h0, l1, h1, l2, h2, l3, h3;
    unpack2(s0, l0, h0);
    unpack2(s1, l1, h1);
    unpack2(s2, l2, h2);
    unpack2(s3, l3, h3);
    return ((l0 + h0) + (l1 + h1)) + ((l2 + h2) + (l3 + h3));
}

// The rotation that makes columns of squared norms al, be and inner product ga
// orthogonal: x' = c (x - t y), y' = c (y + t x); t = 0 for orthogonal or zero
// columns.  cos2 is the squared cosine before.
__device__ __forceinline__ void rotation(float al, float be, float ga, float &t, float &c, float &cos2) {
    const float ab = al * be, g2 = ga * ga;
    t = 0.f;
    c = 1.f;
    cos2 = 0.f;
    if (g2 > 1e-14f * ab) {
        cos2 = __fdividef(g2, ab);
        const float z = __fdividef(be - al, 2.f * ga);
        const float w = fmaf(z, z, 1.f);
        t = copysignf(__fdividef(1.f, fabsf(z) + w * rsqrtf(w)), z);
        const float v = fmaf(t, t, 1.f);
        c = rsqrtf(v);
        c = c * fmaf(-0.5f * v * c, c, 1.5f);
    }
}

// The counters of a warp's solve of np patches, H lanes each; above: lanes above the
// bound in the last sweep.  A patch counts as not converged for itself, not for its
// warp.  Out of line: inlined, it made the R <= 56 kernel spill three times as much.
__device__ __noinline__ void report(unsigned long long rotations, unsigned above, int np, int H, int sweep,
                                    DevCounters *ctr) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, g = lane / H;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rotations += __shfl_xor_sync(FULL, rotations, o);
    const unsigned missed =
        __ballot_sync(FULL, g < np && lane == g * H && ((above >> lane) & (FULL >> (32 - H))) != 0u);
    if (lane == 0) {
        atomicMax(&ctr->jacobi_max_sweeps, (unsigned long long)sweep);
        atomicAdd(&ctr->jacobi_rotations, rotations);
        if (missed) {
            atomicAdd(&ctr->jacobi_not_converged, (unsigned long long)__popc(missed));
            atomicOr(&ctr->status, (unsigned)DEV_NOT_CONVERGED);
        }
    }
}

// Eigenvectors of up to 32 / (R / 2) patches of one warp, starting at `patch`
// (np of them); sm: the warp's jr_floats_r(R) shared floats.
template <int R>
__device__ __forceinline__ void solve(const PatchSeg &seg, int64_t patch, int np, float *sm, int max_sweeps,
                                      DevCounters *ctr) {
    constexpr int H = R / 2, PPW = 32 / H, NP = R / 2, LD = R + 4, LDU = R + 1;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool live = lane < PPW * H;  // lanes past the last group hold zeros
    const int g = live ? lane / H : PPW - 1;
    const int li = live ? lane - g * H : 0;
    const int gb = g * H;
    const bool mine = live && g < np;
    const int k = seg.k;
    const int c0 = 2 * li, c1 = 2 * li + 1;
    float *S = sm + g * (R * LD);
    // ---- G, row-major with stride LD, zero past k
    const float *gm = seg.G + (patch + (g < np ? g : 0)) * (int64_t)k * k;
    if (live) {
#pragma unroll 8
        for (int r = 0; r < R; ++r) {
            const bool in = mine && r < k;
            S[r * LD + li] = in && li < k ? gm[r * k + li] : 0.f;
            S[r * LD + li + H] = in && li + H < k ? gm[r * k + li + H] : 0.f;
        }
    }
    __syncwarp();
    f2 X[NP], Y[NP];
    auto load = [&]() {
#pragma unroll
        for (int q = 0; q < NP / 2; ++q) {
            float4 a = reinterpret_cast<const float4 *>(S + c0 * LD)[q];
            float4 b = reinterpret_cast<const float4 *>(S + c1 * LD)[q];
            if (!live) a = b = make_float4(0.f, 0.f, 0.f, 0.f);
            X[2 * q] = pack2(a.x, a.y);
            X[2 * q + 1] = pack2(a.z, a.w);
            Y[2 * q] = pack2(b.x, b.y);
            Y[2 * q + 1] = pack2(b.z, b.w);
        }
    };
    float dX = live ? S[c0 * LD + c0] : 0.f, dY = live ? S[c1 * LD + c1] : 0.f;
    // largest value over the group's lanes, in all of them
    auto group_max = [&](unsigned v) {
#pragma unroll
        for (int o = (H > 16 ? 16 : 8); o > 0; o >>= 1) {
            const unsigned w = __shfl_down_sync(FULL, v, o);
            if (li + o < H && live) v = max(v, w);
        }
        return __shfl_sync(FULL, v, gb);
    };
    auto bits = [](float d) { return d > 0.f ? __float_as_uint(d) : 0u; };
    // scaled by a power of two so that the largest diagonal entry lies in [1, 2),
    // and shifted by eps I
    const unsigned emax = max(1u, group_max(max(bits(dX), bits(dY))) >> 23);
    const float sc = __uint_as_float(max(1, 254 - (int)emax) << 23), inv_sc = 1.f / sc;
    bool alive0 = live && c0 < k, alive1 = live && c1 < k;
    if (alive0) S[c0 * LD + c0] = fmaf(JR_SHIFT, inv_sc, dX);
    if (alive1) S[c1 * LD + c1] = fmaf(JR_SHIFT, inv_sc, dY);
    __syncwarp();
    load();
    {
        const f2 s2 = pack2(sc, sc);
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            X[q] = mul2(X[q], s2);
            Y[q] = mul2(Y[q], s2);
        }
        dX = fmaf(dX, sc, JR_SHIFT);
        dY = fmaf(dY, sc, JR_SHIFT);
    }
    __syncwarp();
    // ---- pivoted Cholesky: column j of L to S[j * LD ..]; the columns left in
    // registers are those of the Schur complement
    for (int j = 0; j < k; ++j) {
        // largest remaining diagonal entry (to 2^-17), lowest column on ties
        const unsigned kx = alive0 ? (__float_as_uint(fmaxf(dX, 0.25f * JR_SHIFT)) & ~63u) | (63u - c0) : 0u;
        const unsigned ky = alive1 ? (__float_as_uint(fmaxf(dY, 0.25f * JR_SHIFT)) & ~63u) | (63u - c1) : 0u;
        const int p = 63 - (int)(group_max(max(kx, ky)) & 63u);
        const bool odd = p & 1;
        if (live && li == (p >> 1)) {
            const float dp = fmaxf(odd ? dY : dX, 0.25f * JR_SHIFT);
            float rs = rsqrtf(dp);
            rs = rs * fmaf(-0.5f * dp * rs, rs, 1.5f);
            const f2 r2 = pack2(rs, rs);
            float4 *dst = reinterpret_cast<float4 *>(S + j * LD);
            if (odd) {
#pragma unroll
                for (int q = 0; q < NP / 2; ++q) {
                    float4 v;
                    unpack2(mul2(Y[2 * q], r2), v.x, v.y);
                    unpack2(mul2(Y[2 * q + 1], r2), v.z, v.w);
                    dst[q] = v;
                }
                alive1 = false;
            } else {
#pragma unroll
                for (int q = 0; q < NP / 2; ++q) {
                    float4 v;
                    unpack2(mul2(X[2 * q], r2), v.x, v.y);
                    unpack2(mul2(X[2 * q + 1], r2), v.z, v.w);
                    dst[q] = v;
                }
                alive0 = false;
            }
        }
        __syncwarp();
        const float2 l = *reinterpret_cast<const float2 *>(S + j * LD + c0);
        const f2 nx = pack2(-l.x, -l.x), ny = pack2(-l.y, -l.y);
        dX = fmaf(-l.x, l.x, dX);
        dY = fmaf(-l.y, l.y, dY);
        const float4 *src = reinterpret_cast<const float4 *>(S + j * LD);
#pragma unroll
        for (int q = 0; q < NP / 2; ++q) {
            const float4 v = src[q];
            const f2 a = pack2(v.x, v.y), b = pack2(v.z, v.w);
            X[2 * q] = fma2(nx, a, X[2 * q]);
            X[2 * q + 1] = fma2(nx, b, X[2 * q + 1]);
            Y[2 * q] = fma2(ny, a, Y[2 * q]);
            Y[2 * q + 1] = fma2(ny, b, Y[2 * q + 1]);
        }
        __syncwarp();
    }
    // columns past the k-th are zero
    if (live)
        for (int j = k; j < R; ++j) {
            S[j * LD + li] = 0.f;
            S[j * LD + li + H] = 0.f;
        }
    __syncwarp();
    load();
    // ---- sweeps
    const int nxt = live ? gb + (li + 1 == H ? 0 : li + 1) : lane;
    auto pass_y = [&]() {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            float lo, hi;
            unpack2(Y[q], lo, hi);
            Y[q] = pack2(__shfl_sync(FULL, lo, nxt), __shfl_sync(FULL, hi, nxt));
        }
    };
    int sweep = 0, seam = H - 1;
    unsigned long long rotations = 0;
    unsigned above = FULL;  // lanes whose patch was above the bound in the last sweep
    while (sweep < max_sweeps) {
        float al = dot_cols<NP>(X, X), be = dot_cols<NP>(Y, Y);
        float mx = 0.f;
        unsigned nrot = 0;
        for (int rr = 0; rr < H; ++rr) {
            float t, c, cos2, ga;
            // every lane rotates: x - t y, y + t x, the factor c left over
            ga = dot_cols<NP>(X, Y);
            rotation(al, be, ga, t, c, cos2);
            mx = fmaxf(mx, cos2);
            nrot += t != 0.f;
            {
                const f2 tp = pack2(t, t), tn = pack2(-t, -t);
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const f2 x = X[q];
                    X[q] = fma2(tn, Y[q], x);
                    Y[q] = fma2(tp, x, Y[q]);
                }
            }
            al = fmaf(-t, ga, al);
            be = fmaf(t, ga, be);
            pass_y();
            const float dx = c, dy = __shfl_sync(FULL, c, nxt);
            be = __shfl_sync(FULL, be, nxt);
            // every lane but the seam rotates; the seam exchanges its columns
            const bool at_seam = li == seam;
            ga = dx * dy * dot_cols<NP>(X, Y);
            rotation(al, be, ga, t, c, cos2);
            float px = c * dx, py = -c * t * dy, qy = c * dy, qx = c * t * dx;
            if (at_seam) {
                px = qy = 0.f;
                py = dy;
                qx = dx;
                const float a = al;
                al = be;
                be = a;
            } else {
                mx = fmaxf(mx, cos2);
                nrot += t != 0.f;
                al = fmaf(-t, ga, al);
                be = fmaf(t, ga, be);
            }
            {
                const f2 p2 = pack2(px, px), r2 = pack2(py, py), q2 = pack2(qy, qy), u2 = pack2(qx, qx);
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const f2 x = X[q], y = Y[q];
                    X[q] = fma2(p2, x, mul2(r2, y));
                    Y[q] = fma2(q2, y, mul2(u2, x));
                }
            }
            pass_y();
            be = __shfl_sync(FULL, be, nxt);
            seam = seam == 0 ? H - 1 : seam - 1;
        }
        ++sweep;
        rotations += nrot;
        if (__all_sync(FULL, !(mx >= JR_STOP2))) {
            above = 0u;
            break;
        }
        if (sweep == max_sweeps) above = __ballot_sync(FULL, mx >= JR_STOP2);
    }
    // ---- eigenpairs sorted descending
    const float al = dot_cols<NP>(X, X), be = dot_cols<NP>(Y, Y);
    float *nu = S + R * LDU;
    __syncwarp();
    if (live) {
        nu[c0] = al;
        nu[c1] = be;
    }
    __syncwarp();
    int rx = 0, ry = 0;
    for (int c = 0; c < R; ++c) {
        const float v = nu[c];
        rx += pair_before(v, c, al, c0);
        ry += pair_before(v, c, be, c1);
    }
    if (mine) {
        float *sg = seg.sig + (patch + g) * (int64_t)k;
        if (rx < k) sg[rx] = (al - JR_SHIFT) * inv_sc;
        if (ry < k) sg[ry] = (be - JR_SHIFT) * inv_sc;
    }
    if (live) {
        const float ix = al > 0.f ? 1.f / sqrtf(al) : 0.f, iy = be > 0.f ? 1.f / sqrtf(be) : 0.f;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            float lo, hi;
            if (rx < R) {
                unpack2(X[q], lo, hi);
                S[rx * LDU + 2 * q] = lo * ix;
                S[rx * LDU + 2 * q + 1] = hi * ix;
            }
            if (ry < R) {
                unpack2(Y[q], lo, hi);
                S[ry * LDU + 2 * q] = lo * iy;
                S[ry * LDU + 2 * q + 1] = hi * iy;
            }
        }
    }
    __syncwarp();
    if (mine) {
        float *u = seg.U + (patch + g) * (int64_t)k * k;
        for (int r = 0; r < k; ++r)
            for (int c = li; c < k; c += H) u[r * k + c] = S[c * LDU + r];
    }
    report(rotations, above, np, H, sweep, ctr);
}

// One warp per group of patches; RMAX bounds every patch's R.  The bodies with
// R <= 32 need half the registers, so launches of k <= 32 get more warps.
template <int RMAX>
__global__ void __launch_bounds__(jr_warps(RMAX) * 32, jr_blocks(RMAX))
jacobi_reg_kernel(const __grid_constant__ PatchSeg one, const PatchSeg *__restrict__ tab, int ntab, int64_t nwarps,
                  int smem_floats, int max_sweeps, DevCounters *ctr) {
    extern __shared__ __align__(16) float jr_sm[];
    const int64_t w = (int64_t)blockIdx.x * jr_warps(RMAX) + (threadIdx.x >> 5);
    if (w >= nwarps) return;
    // the segment of this warp: a warp's patches belong to one segment
    const PatchSeg *sp = &one;
    if (ntab) {
        int lo = 0, hi = ntab - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tab[mid].jfirst <= w) lo = mid;
            else hi = mid - 1;
        }
        sp = tab + lo;
    }
    const PatchSeg &seg = *sp;
    const int R = jr_rows(seg.k), ppw = jr_ppw(seg.k);
    const int64_t patch = (w - seg.jfirst) * ppw;
    const int np = (int)min((int64_t)ppw, (int64_t)seg.npts - patch);
    float *sm = jr_sm + (threadIdx.x >> 5) * smem_floats;
    if (np <= 0) return;
    switch (R) {
        case 16: solve<16>(seg, patch, np, sm, max_sweeps, ctr); break;
        case 24: solve<24>(seg, patch, np, sm, max_sweeps, ctr); break;
        case 32: solve<32>(seg, patch, np, sm, max_sweeps, ctr); break;
        default:
            if constexpr (RMAX > 32) {
                if (R == 40) solve<40>(seg, patch, np, sm, max_sweeps, ctr);
                else if (R == 48) solve<48>(seg, patch, np, sm, max_sweeps, ctr);
                else if (RMAX == 56 || R == 56) solve<56>(seg, patch, np, sm, max_sweeps, ctr);
                else if constexpr (RMAX > 56) solve<64>(seg, patch, np, sm, max_sweeps, ctr);
            }
    }
}

template <int RMAX>
cudaError_t launch(const PatchSeg &one, const PatchSeg *tab, int ntab, int kmax, int64_t nwarps, int max_sweeps,
                   DevCounters *ctr, cudaStream_t s) {
    int fl = 0;
    for (int R = 16; R <= jr_rows(kmax); R += 8) fl = fl > jr_floats_r(R) ? fl : jr_floats_r(R);
    constexpr int W = jr_warps(RMAX);
    const size_t smem = (size_t)W * fl * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(jacobi_reg_kernel<RMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    jacobi_reg_kernel<RMAX><<<(unsigned)((nwarps + W - 1) / W), W * 32, smem, s>>>(
        one, tab, ntab, nwarps, fl, max_sweeps, ctr);
    return cudaGetLastError();
}
}  // namespace

int64_t jacobi_reg_warps(int k, int64_t np) { return (np + jr_ppw(k) - 1) / jr_ppw(k); }

cudaError_t launch_jacobi_reg(const PatchSeg &one, const PatchSeg *tab, int ntab, int kmax, int64_t nwarps,
                              int max_sweeps, DevCounters *ctr, cudaStream_t s) {
    if (nwarps <= 0) return cudaSuccess;
    if (kmax > 64 || kmax < 1) return cudaErrorInvalidValue;
    if (kmax <= 32) return launch<32>(one, tab, ntab, kmax, nwarps, max_sweeps, ctr, s);
    if (kmax <= 56) return launch<56>(one, tab, ntab, kmax, nwarps, max_sweeps, ctr, s);
    return launch<64>(one, tab, ntab, kmax, nwarps, max_sweeps, ctr, s);
}

}  // namespace mecuco
