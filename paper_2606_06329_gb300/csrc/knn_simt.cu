// knn_simt.cu - Step 1 (Sec. 3 Step 1, eq. knn; Alg. 1 kNN-Graph): candidate
// search with FP32 arithmetic on the CUDA cores, the exact re-rank with its
// certification test, and the exact full-scan fallback.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace mecuco {

// The table entry of batch row `row` (entries sorted by row_begin).
__device__ __forceinline__ const KnnSet &find_set_row(const KnnSet *sets, int nsets, int64_t row) {
    int lo = 0, hi = nsets - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sets[mid].row_begin <= row) lo = mid;
        else hi = mid - 1;
    }
    return sets[lo];
}

// One warp, one read of a row: |x|^2 as a compensated sum (hi + lo rounded once,
// so within a few FP32 units of the exact value), the BF16 operand rows of the
// tensor-core search (ya, and yb for the three-term split; NULL: none), and, for
// quant != NONE, the norms of the row's BF16 rounding terms (rounded up) into
// resid[0..1]: single rounding h = bf16(x): |x - h| and 0; three-term split,
// l = bf16(x - h): |l| and |x - h - l| (both differences exact in FP32).  The
// dataset's largest |x|^2 and terms go to maxima[0..2] (non-negative floats, so
// their bit patterns order as integers).
// Operand rows (leading dimension ldb, zero past the data): one rounding, y = h;
// the three-term split, in segments of ms columns, query copy [h | h | l] and
// candidate copy [h | l | h], so that one GEMM over K = 3 ms gives h.h' + h.l' +
// l.h', the FP32 product up to l.l' and the remainders past two terms.
template <typename T, int COPIES>
__device__ __forceinline__ void row_prep_copies(const T *__restrict__ x, int64_t m, int lane, float *norm_out,
                                              float *resid_out, float *maxima, int quant,
                                              __nv_bfloat16 *__restrict__ ya, __nv_bfloat16 *__restrict__ yb,
                                              int64_t ms, int64_t ldb) {
    ff acc{0.f, 0.f};
    float a1 = 0.f, a2 = 0.f;
    for (int64_t a = lane; a < m; a += 32) {
        const float v = load_elem(x + a);
        ff_acc_sqdiff(acc, v, 0.f);
        if constexpr (COPIES > 0 || sizeof(T) == 4) {
            const __nv_bfloat16 h = __float2bfloat16_rn(v);
            const float r = v - __bfloat162float(h);
            const __nv_bfloat16 lb = __float2bfloat16_rn(r);
            if (quant == KNN_QUANT_SINGLE) {
                a1 = fmaf(r, r, a1);
            } else if (quant == KNN_QUANT_SPLIT) {
                const float l = __bfloat162float(lb);
                const float r2 = r - l;
                a1 = fmaf(l, l, a1);
                a2 = fmaf(r2, r2, a2);
            }
            if constexpr (COPIES == 2) {
                ya[a] = h;
                ya[ms + a] = h;
                ya[2 * ms + a] = lb;
                yb[a] = h;
                yb[ms + a] = lb;
                yb[2 * ms + a] = h;
            } else if constexpr (COPIES == 1) {
                ya[a] = h;
            }
        }
    }
    const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
    if constexpr (COPIES == 2) {
        for (int64_t a = m + lane; a < ms; a += 32)
            ya[a] = ya[ms + a] = ya[2 * ms + a] = yb[a] = yb[ms + a] = yb[2 * ms + a] = zero;
        for (int64_t a = 3 * ms + lane; a < ldb; a += 32) ya[a] = yb[a] = zero;
    } else if constexpr (COPIES == 1) {
        for (int64_t a = m + lane; a < ldb; a += 32) ya[a] = zero;
    }
    acc = ff_warp_sum(acc);
    const float n = acc.hi + acc.lo;
    if (quant != KNN_QUANT_NONE) {
        a1 = warp_sum(a1);
        a2 = warp_sum(a2);
    }
    if (lane == 0) {
        *norm_out = n;
        if (quant != KNN_QUANT_NONE) {
            // the FP32 sums of m squares are within m 2^-24 of their values: 2^-10 covers it
            const float t1 = sqrtf(a1) * (1.f + 9.765625e-04f), t2 = sqrtf(a2) * (1.f + 9.765625e-04f);
            resid_out[0] = t1;
            resid_out[1] = t2;
            atomicMax(reinterpret_cast<int *>(maxima), __float_as_int(n));
            atomicMax(reinterpret_cast<int *>(maxima) + 1, __float_as_int(t1));
            atomicMax(reinterpret_cast<int *>(maxima) + 2, __float_as_int(t2));
        }
    }
}

template <typename T>
__device__ __forceinline__ void row_prep_warp(const T *x, int64_t m, int lane, float *norm_out, float *resid_out,
                                              float *maxima, int quant, __nv_bfloat16 *ya, __nv_bfloat16 *yb,
                                              int64_t ms, int64_t ldb) {
    if (yb) row_prep_copies<T, 2>(x, m, lane, norm_out, resid_out, maxima, quant, ya, yb, ms, ldb);
    else if (ya) row_prep_copies<T, 1>(x, m, lane, norm_out, resid_out, maxima, quant, ya, yb, ms, ldb);
    else row_prep_copies<T, 0>(x, m, lane, norm_out, resid_out, maxima, quant, ya, yb, ms, ldb);
}

template <typename T>
__global__ void row_prep_kernel(const T *__restrict__ X, int64_t N, int64_t m, int64_t ld, float *__restrict__ out,
                                float *__restrict__ resid, float *__restrict__ maxima, int quant,
                                __nv_bfloat16 *__restrict__ ya, __nv_bfloat16 *__restrict__ yb, int64_t ms,
                                int64_t ldb) {
    int64_t row = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    int lane = threadIdx.x & 31;
    if (row >= N) return;
    row_prep_warp(X + row * ld, m, lane, out + row, quant ? resid + 2 * row : nullptr, maxima, quant,
                  ya ? ya + row * ldb : nullptr, yb ? yb + row * ldb : nullptr, ms, ldb);
}

cudaError_t launch_row_prep(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld, float *norms,
                            cudaStream_t s, float *resid, float *maxima, int quant, void *ya, void *yb, int64_t ms,
                            int64_t ldb) {
    if (N <= 0) return cudaSuccess;
    if (dt == MECUCO_BF16 || !resid || !maxima) quant = KNN_QUANT_NONE;
    dim3 block(256), grid((unsigned)((N + 7) / 8));
    __nv_bfloat16 *a = (__nv_bfloat16 *)ya, *b = (__nv_bfloat16 *)yb;
    if (dt == MECUCO_BF16)
        row_prep_kernel<<<grid, block, 0, s>>>((const __nv_bfloat16 *)X, N, m, ld, norms, nullptr, nullptr, quant, a,
                                               b, ms, ldb);
    else
        row_prep_kernel<<<grid, block, 0, s>>>((const float *)X, N, m, ld, norms, resid, maxima, quant, a, b, ms, ldb);
    return cudaGetLastError();
}

// The same for every row of a batch: one warp per row, each row's dataset from
// the table (xb, xb2 its operand rows where it has them).
template <typename T>
__global__ void row_prep_batch_kernel(const KnnSet *__restrict__ sets, int nsets, int64_t nrows) {
    const int64_t gr = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    const int lane = threadIdx.x & 31;
    if (gr >= nrows) return;
    const KnnSet &d = find_set_row(sets, nsets, gr);
    const int64_t row = gr - d.row_begin;
    __nv_bfloat16 *ya = static_cast<__nv_bfloat16 *>(d.xb), *yb = static_cast<__nv_bfloat16 *>(d.xb2);
    row_prep_warp(static_cast<const T *>(d.X) + row * d.ld, d.m, lane, d.norms + row,
                  d.quant ? d.resid + 2 * row : nullptr, d.maxima, d.quant, ya ? ya + row * d.ldb : nullptr,
                  yb ? yb + row * d.ldb : nullptr, d.mk / 3, d.ldb);
}

cudaError_t launch_row_prep_batch(const KnnSet *sets, int nsets, int64_t nrows, mecuco_dtype dt, cudaStream_t s) {
    if (nrows <= 0) return cudaSuccess;
    dim3 block(256), grid((unsigned)((nrows + 7) / 8));
    if (dt == MECUCO_BF16) row_prep_batch_kernel<__nv_bfloat16><<<grid, block, 0, s>>>(sets, nsets, nrows);
    else row_prep_batch_kernel<float><<<grid, block, 0, s>>>(sets, nsets, nrows);
    return cudaGetLastError();
}

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

// ---------------------------------------------------------------------------
// Candidate search, plain FP32.  A block of 256 threads owns 128 query rows and
// sweeps its split of the candidate rows in tiles of 256; thread (tx, ty) of a
// 16 x 16 grid accumulates rows 8 ty .. + 7 against columns 64 g + 4 tx .. + 3
// (g < 4) as packed FP32 pairs (two columns per FMA), over K slices of 16 that are
// double-buffered through registers.  A 16-byte shared load takes the banks four
// cycles whatever its lanes share, so the tile is as large as the registers
// allow: 6 loads feed 64 packed FMAs, 192 of 256 cycles.
// Selection: every row keeps its kc smallest d~ = |x|^2 + |y|^2 - 2 x.y as a
// max-heap in shared memory.  A thread reserves room for its admitted entries
// (below the heap's root) in the row's pending buffer with one shared atomic per
// row, and 128 threads, one per row, fold the buffers into the heaps together
// once any holds more than SP_HIGH; a tile that does not fit (the first ones,
// which admit everything) is taken in eight parts of 32 columns.
// Measured per search: 50,000 x 256, k = 32 81 -> 27 ms (47 TFLOP/s; FP32-issue
// bound with one block per SM; 33 with 128-wide tiles and the query slice stored
// twice, 28.5 with it stored once); 20,000 x 24, k = 32 10.8 -> 1.7 ms (selection
// bound).  Before, 8 scalar loads per operand and K step and one thread per row
// walking all 128 distances of a tile.
// ---------------------------------------------------------------------------
constexpr int SBM = 128, SBN = 256, SBK = 16, STHREADS = 256;
constexpr int SLDA = SBM + 4, SLDB = SBN + 4;  // row strides of the operand slices (floats)
constexpr int NG = SBN / 64, NC = 4 * NG;      // groups of 4 columns, and columns, of a thread
constexpr int SPEND = 32;    // pending candidates per row
constexpr int SP_HIGH = 16;  // above this, a row asks for an update

__host__ __device__ inline size_t simt_smem_bytes(int kc) {
    return sizeof(float) * (size_t)(2 * SBK * (SLDA + SLDB) + 2 * SPEND * SBM + 2 * kc * SBM + 2 * SBM + SBN) +
           sizeof(int) * (size_t)(2 * SBM + 4);
}

// Four consecutive elements of a row from column a (zero past m).
__device__ __forceinline__ float4 load4(const float *row, int64_t a, int64_t m, bool vec) {
    if (vec && a + 4 <= m) return __ldg(reinterpret_cast<const float4 *>(row + a));
    float4 v;
    v.x = a < m ? __ldg(row + a) : 0.f;
    v.y = a + 1 < m ? __ldg(row + a + 1) : 0.f;
    v.z = a + 2 < m ? __ldg(row + a + 2) : 0.f;
    v.w = a + 3 < m ? __ldg(row + a + 3) : 0.f;
    return v;
}
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *row, int64_t a, int64_t m, bool vec) {
    if (vec && a + 4 <= m) {
        const uint2 w = __ldg(reinterpret_cast<const uint2 *>(row + a));
        return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                           __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
    }
    float4 v;
    v.x = a < m ? load_elem(row + a) : 0.f;
    v.y = a + 1 < m ? load_elem(row + a + 1) : 0.f;
    v.z = a + 2 < m ? load_elem(row + a + 2) : 0.f;
    v.w = a + 3 < m ? load_elem(row + a + 3) : 0.f;
    return v;
}

// One entry into a row's max-heap of capacity kc (position p at Hd[p * SBM],
// children 4 p + 1 .. 4 p + 4: the four loads of a level are independent, so a
// full heap of 64 costs three dependent steps instead of six).
__device__ __forceinline__ void heap_insert(float *Hd, int *Hi, int &cnt, float d, int c, int kc) {
    if (cnt < kc) {
        int pos = cnt++;
        while (pos > 0) {
            const int par = (pos - 1) >> 2;
            const float pd = Hd[par * SBM];
            const int pi = Hi[par * SBM];
            if (pd >= d) break;
            Hd[pos * SBM] = pd;
            Hi[pos * SBM] = pi;
            pos = par;
        }
        Hd[pos * SBM] = d;
        Hi[pos * SBM] = c;
        return;
    }
    int pos = 0;
    for (;;) {
        const int l = 4 * pos + 1;
        if (l >= kc) break;
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = l + e < kc ? Hd[(l + e) * SBM] : -INFINITY;
        const float m01 = fmaxf(v[0], v[1]), m23 = fmaxf(v[2], v[3]);
        const int b01 = v[1] > v[0] ? 1 : 0, b23 = v[3] > v[2] ? 3 : 2;
        const float dc = fmaxf(m01, m23);
        const int ch = l + (m23 > m01 ? b23 : b01);
        if (dc <= d) break;
        Hd[pos * SBM] = dc;
        Hi[pos * SBM] = Hi[ch * SBM];
        pos = ch;
    }
    Hd[pos * SBM] = d;
    Hi[pos * SBM] = c;
}
}  // namespace

template <typename T>
__global__ void __launch_bounds__(STHREADS, 1)
knn_simt_kernel(const T *__restrict__ X, int64_t N, int64_t m, int64_t ld,
                const float *__restrict__ norms, int64_t q0, int64_t nq, int kc, int nsplit,
                int include_self, float *__restrict__ cand_d, int32_t *__restrict__ cand_i) {
    extern __shared__ __align__(16) float smem[];
    float *As = smem;                          // [2][SBK][SLDA] query slice
    float *Bs = As + 2 * SBK * SLDA;           // [2][SBK][SLDB]
    float *Pd = Bs + 2 * SBK * SLDB;           // [SPEND][SBM] pending distances
    int *Pc = reinterpret_cast<int *>(Pd + SPEND * SBM);
    float *Hd = reinterpret_cast<float *>(Pc + SPEND * SBM);  // [kc][SBM] heaps
    int *Hi = reinterpret_cast<int *>(Hd + kc * SBM);
    float *thr = reinterpret_cast<float *>(Hi + kc * SBM);  // [SBM] admission thresholds
    float *qns = thr + SBM;                    // [SBM]
    float *cns = qns + SBM;                    // [SBN]
    int *pcnt = reinterpret_cast<int *>(cns + SBN);  // [SBM] pending entries
    int *pold = pcnt + SBM;                    // [SBM] and before the current tile
    int *flags = pold + SBM;                   // overflow, update wanted

    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t qb = q0 + (int64_t)blockIdx.x * SBM;
    const int64_t qend = q0 + nq;
    const int split = blockIdx.y;
    const int64_t per = (N + nsplit - 1) / nsplit;
    const int64_t cbeg = (int64_t)split * per;
    const int64_t cend = min(N, cbeg + per);
    const bool vec = (ld % 4 == 0) && (reinterpret_cast<uintptr_t>(X) & (4 * sizeof(T) - 1)) == 0;

    if (tid < SBM) {
        qns[tid] = (qb + tid < qend) ? norms[qb + tid] : 0.f;
        thr[tid] = (qb + tid < qend) ? INFINITY : -INFINITY;
        pcnt[tid] = pold[tid] = 0;
    }
    if (tid < 2) flags[tid] = 0;
    int cnt = 0;  // entries of row tid's heap (tid < SBM)
    // rows of this thread's loads: lr, lr + 64; columns 4 lq .. + 3 of a slice
    const int lr = tid >> 2, lq = tid & 3;
    const T *qrow[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) qrow[h] = X + min(qb + lr + 64 * h, N - 1) * ld;
    const int nslice = (int)((m + SBK - 1) / SBK);
    // every row's pending entries into its heap (128 threads; the rest wait)
    auto update = [&]() {
        if (tid < SBM) {
            const int n = pcnt[tid];
            float t = thr[tid], dn = Pd[tid];
            int cn = Pc[tid];
            for (int i = 0; i < n; ++i) {
                const float d = dn;
                const int c = cn;
                const int nx = min(i + 1, SPEND - 1);
                dn = Pd[nx * SBM + tid];
                cn = Pc[nx * SBM + tid];
                if (d < t) {
                    heap_insert(Hd + tid, Hi + tid, cnt, d, c, kc);
                    if (cnt == kc) t = Hd[tid];
                }
            }
            thr[tid] = t;
            pcnt[tid] = pold[tid] = 0;
        }
        __syncthreads();
    };
    bool filling = true;  // some list of the block may still be short
    for (int64_t c0 = cbeg; c0 < cend; c0 += SBN) {
        f2 acc[8][NC / 2];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < NC / 2; ++j) acc[i][j] = 0ull;
        const T *crow[NG];
#pragma unroll
        for (int h = 0; h < NG; ++h) crow[h] = X + min(c0 + lr + 64 * h, N - 1) * ld;
        float4 ra[2], rb[NG];
        auto fetch = [&](int sl) {
            const int64_t a = (int64_t)sl * SBK + 4 * lq;
#pragma unroll
            for (int h = 0; h < 2; ++h) ra[h] = load4(qrow[h], a, m, vec);
#pragma unroll
            for (int h = 0; h < NG; ++h) rb[h] = load4(crow[h], a, m, vec);
        };
        auto stage = [&](int buf) {
            float *A = As + buf * SBK * SLDA, *B = Bs + buf * SBK * SLDB;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float av[4] = {ra[h].x, ra[h].y, ra[h].z, ra[h].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) A[(4 * lq + e) * SLDA + lr + 64 * h] = av[e];
            }
#pragma unroll
            for (int h = 0; h < NG; ++h) {
                const float bv[4] = {rb[h].x, rb[h].y, rb[h].z, rb[h].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) B[(4 * lq + e) * SLDB + lr + 64 * h] = bv[e];
            }
        };
        fetch(0);
        cns[tid] = (c0 + tid < cend) ? norms[c0 + tid] : INFINITY;
        stage(0);
        __syncthreads();
        for (int sl = 0; sl < nslice; ++sl) {
            if (sl + 1 < nslice) fetch(sl + 1);
            const float *A = As + (sl & 1) * SBK * SLDA + 8 * ty, *B = Bs + (sl & 1) * SBK * SLDB + 4 * tx;
#pragma unroll
            for (int kk = 0; kk < SBK; ++kk) {
                const float4 a0 = *reinterpret_cast<const float4 *>(A + kk * SLDA);
                const float4 a1 = *reinterpret_cast<const float4 *>(A + kk * SLDA + 4);
                f2 b[NC / 2];
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const ulonglong2 b2 = *reinterpret_cast<const ulonglong2 *>(B + kk * SLDB + 64 * g);
                    b[2 * g] = b2.x;
                    b[2 * g + 1] = b2.y;
                }
                const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const f2 a = pack2(av[i], av[i]);
#pragma unroll
                    for (int j = 0; j < NC / 2; ++j) acc[i][j] = fma2(a, b[j], acc[i][j]);
                }
            }
            if (sl + 1 < nslice) stage((sl + 1) & 1);
            __syncthreads();
        }
        // distances in place: column 2j of a pair and 2j + 1
        const bool selfs = !include_self && c0 < qb + SBM && qb < c0 + SBN;
        // append this thread's entries of its columns [J0, J1); flags[0] if a row's
        // buffer has no room for them
        auto append = [&](auto J0, auto J1) {
            constexpr int j0 = decltype(J0)::value, j1 = decltype(J1)::value;
            float cn[j1 - j0];
#pragma unroll
            for (int j = j0; j < j1; ++j) cn[j - j0] = cns[(j >> 2) * 64 + 4 * tx + (j & 3)];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = 8 * ty + i;
                const float q = qns[r], t = thr[r];
                float d[j1 - j0];
                unsigned adm = 0;
#pragma unroll
                for (int j = j0; j < j1; ++j) {
                    const float2 v = unpack2(acc[i][j >> 1]);
                    d[j - j0] = fmaf(-2.f, (j & 1) ? v.y : v.x, q + cn[j - j0]);
                    const int c = (j >> 2) * 64 + 4 * tx + (j & 3);
                    const bool in = d[j - j0] < t && !(selfs && c0 + c == qb + r);
                    adm |= (in ? 1u : 0u) << j;
                }
                if (adm) {
                    const int na = __popc(adm);
                    int pos = atomicAdd(&pcnt[r], na);
                    if (pos + na > SPEND) {
                        flags[0] = 1;
                    } else {
                        if (pos + na > SP_HIGH) flags[1] = 1;
#pragma unroll
                        for (int j = j0; j < j1; ++j)
                            if ((adm >> j) & 1u) {
                                Pd[pos * SBM + r] = d[j - j0];
                                Pc[pos * SBM + r] = (int)c0 + (j >> 2) * 64 + 4 * tx + (j & 3);
                                ++pos;
                            }
                    }
                }
            }
        };
        bool parts = filling;
        if (!parts) {
            append(std::integral_constant<int, 0>(), std::integral_constant<int, NC>());
            __syncthreads();
            parts = flags[0] != 0;
            if (parts) {
                // does not fit: forget this tile's entries
                __syncthreads();
                if (tid < SBM) pcnt[tid] = pold[tid];
                if (tid == 0) flags[0] = 0;
                __syncthreads();
            }
        }
        if (parts) {
            update();
#pragma unroll 1
            for (int p = 0; p < NC / 2; ++p) {  // two columns a thread: at most 32 entries a row
                using std::integral_constant;
                if (p == 0) append(integral_constant<int, 0>(), integral_constant<int, 2>());
                else if (p == 1) append(integral_constant<int, 2>(), integral_constant<int, 4>());
                else if (p == 2) append(integral_constant<int, 4>(), integral_constant<int, 6>());
                else if (p == 3) append(integral_constant<int, 6>(), integral_constant<int, 8>());
                else if (p == 4) append(integral_constant<int, 8>(), integral_constant<int, 10>());
                else if (p == 5) append(integral_constant<int, 10>(), integral_constant<int, 12>());
                else if (p == 6) append(integral_constant<int, 12>(), integral_constant<int, 14>());
                else append(integral_constant<int, 14>(), integral_constant<int, 16>());
                __syncthreads();
                update();
            }
            if (tid == 0) flags[1] = 0;
            filling = __syncthreads_or(tid < SBM && cnt < kc && thr[tid] == INFINITY);
        } else if (flags[1]) {
            __syncthreads();
            if (tid == 0) flags[1] = 0;
            update();
        } else {
            if (tid < SBM) pold[tid] = pcnt[tid];
        }
    }
    __syncthreads();
    update();
    if (tid < SBM && qb + tid < qend) {
        int64_t base = ((qb + tid - q0) * nsplit + split) * (int64_t)kc;
        for (int e = 0; e < kc; ++e) {
            const bool used = e < cnt;
            cand_d[base + e] = used ? Hd[e * SBM + tid] : INFINITY;
            cand_i[base + e] = used ? Hi[e * SBM + tid] : -1;
        }
    }
}

cudaError_t launch_knn_simt(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld,
                            const float *norms, int64_t q0, int64_t nq, int kc, int nsplit,
                            int include_self, float *cand_d, int32_t *cand_i, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const dim3 grid((unsigned)((nq + SBM - 1) / SBM), (unsigned)nsplit);
    const size_t smem = simt_smem_bytes(kc);
    auto run = [&](auto kern, const auto *Xp) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, STHREADS, smem, s>>>(Xp, N, m, ld, norms, q0, nq, kc, nsplit, include_self, cand_d, cand_i);
        return cudaGetLastError();
    };
    return dt == MECUCO_BF16 ? run(knn_simt_kernel<__nv_bfloat16>, (const __nv_bfloat16 *)X)
                             : run(knn_simt_kernel<float>, (const float *)X);
}

// ---------------------------------------------------------------------------
// Exact re-rank + certification.  One warp per query row.  An exact distance is
// sum_a (x_a - y_a)^2 as a float-float pair: the difference by TwoSum, its
// square added to a two-term sum by FMAs, whose offset is kept within 8 times the
// distance, so it carries ~2^-42 relative error: ranks agree with an FP64 brute force
// except at ties closer than that.
// Certification: a point left out - rejected by a list, or a candidate that is
// not evaluated here - has d~ >= some threshold thr, so its true distance is >=
// thr - e_hi, e_hi bounding the overestimate d~ - d; it cannot enter the top k
// when thr - e_hi exceeds the exact k-th distance theta.  The search's
// accumulation error has no useful worst-case bound and is dominated by a part that
// the near candidates of a row have in common (the FP32 accumulator's truncation of
// partial sums of similar size, in one order of the columns), so e_hi is estimated a
// posteriori from the row's own evaluated candidates: the largest observed d~ - d
// plus 3x the observed spread of d~ - d, plus 2^-21 (|x|^2 + |y|^2) (a few units in
// the last place of the norms, |y| the largest evaluated or that of a point at
// theta); FP32 rows searched in BF16 add the rounding's a-priori bound.
// The lists hold two to three times as many candidates as neighbours asked for,
// so a row first evaluates the k + RR_EXTRA smallest by d~ (a threshold found by
// bisection) and RR_SAMPLE others, and then only those with d~ <= theta + e_hi,
// usually none.  The others are taken at equal steps through the lists, whose order
// does not follow d~, with the largest d~ among them: the smallest d~ are those that
// the search underestimates most, and where they are copies of one point they show
// the error of that point alone (of 2,400 FP32 rows of 4,096 columns with 23 copies in
// each cluster, up to 16 came out certified and wrong without the sample).  Rows
// whose lists' own threshold (the smallest maximum of the full lists) does not
// pass the test are re-solved exactly by the full scan.
// Measured per 100k queries against the form that evaluated and ranked every
// candidate: 512 columns BF16, k = 32, 128 candidates 6.4 to 3.0 ms (2.6 without the
// sample); per 70k of 784 FP32 columns, k = 50 6.7 to 4.1 ms (3.7); 2,000 x 32 with
// several hundred candidates a row 2.98 to 0.03 ms.  Bound by the FP32 pipe (12
// operations a term, in packed pairs, 22 before) up to about 1,000 columns, then by
// the candidate rows' DRAM reads.
// ---------------------------------------------------------------------------
constexpr int RR_WARPS = 4;
constexpr int RR_MAXL = 1024;
constexpr int RR_EXTRA = 16;
constexpr int RR_SAMPLE = 16;
constexpr int RR_CAP = 128;  // evaluated candidates kept at a time (>= 64 + RR_EXTRA + RR_SAMPLE + slack, a multiple of 32)

namespace {
// 16 bytes of a row as packed FP32 pairs
template <typename T>
__device__ __forceinline__ void widen(uint4 v, f2 (&o)[8 / sizeof(T)]);
template <>
__device__ __forceinline__ void widen<float>(uint4 v, f2 (&o)[2]) {
    o[0] = pack2(__uint_as_float(v.x), __uint_as_float(v.y));
    o[1] = pack2(__uint_as_float(v.z), __uint_as_float(v.w));
}
template <>
__device__ __forceinline__ void widen<__nv_bfloat16>(uint4 v, f2 (&o)[4]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
        o[e] = pack2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));
}
// (hi, lo) += (x - y)^2 for two terms at once.  hi carries an offset 2^b above
// the sum, so that it stays in one binade: h = fma(d, d, hi) loses d^2 - (h - hi)
// exactly (h - hi is exact), which the next FMA rounds once.
struct PairAcc {
    f2 hi, lo;
};
__device__ __forceinline__ void acc_sqdiff2(PairAcc &a, f2 x, f2 y, f2 minus, f2 two) {
    const f2 d = fma2(y, minus, x);            // x - y, rounded
    const f2 bb = fma2(x, minus, d);           // its rounding error, by TwoSum
    const f2 t = fma2(fma2(bb, minus, d), minus, x);
    const f2 dl = fma2(add2(y, bb), minus, t);
    const f2 h = fma2(d, d, a.hi);
    const f2 er = fma2(d, d, fma2(h, minus, a.hi));
    a.hi = h;
    a.lo = fma2(dl, fma2(d, two, dl), add2(a.lo, er));
}
// order-preserving image of a float
__device__ __forceinline__ unsigned order_key(float v) {
    const unsigned b = __float_as_uint(v);
    return b & 0x80000000u ? ~b : b | 0x80000000u;
}
}  // namespace

// Exact distance of rows xq and y over the G lanes of a group, renormalising every
// term (no offset).  All groups of the warp together; not inlined, so that the usual
// case keeps its registers (a second pass with a better offset inside exact_dist4 made
// 100,000 x 512 take 16.5 ms instead of 15.3 without ever running).
template <typename T>
__device__ __noinline__ ff exact_dist_renorm(const T *__restrict__ xq, const T *__restrict__ y, int64_t m, int G) {
    ff s{0.f, 0.f};
    for (int64_t a = (threadIdx.x & 31) & (G - 1); a < m; a += G)
        ff_acc_sqdiff(s, load_elem(xq + a), load_elem(y + a));
    for (int o = G >> 1; o > 0; o >>= 1) s = ff_add(s, ff_shfl_xor(s, o));
    return s;
}

// Exact distances of the candidates j[u] (u < 4; -1: none) from row q, one per
// group of G lanes and u, returned in every lane of the group.  base[u]: the
// offset, a power of two above twice the search's distance.  Where it proves too
// small (a partial sum reaches it), or more than 8 times the distance (the low word
// would hold, rounded to FP32, what hi cannot: points far closer than the search
// resolves), the sum is formed again without an offset.
template <typename T>
__device__ __forceinline__ void exact_dist4(const T *__restrict__ X, int64_t m, int64_t ld, const T *__restrict__ xq,
                                            int64_t q, const int (&j)[4], const float (&base)[4], int G, bool vec,
                                            ff (&out)[4]) {
    constexpr int VEC = 16 / (int)sizeof(T), NP = VEC / 2;
    const int lane = threadIdx.x & 31, gl = lane & (G - 1);
    const f2 minus = pack2(-1.f, -1.f), two = pack2(2.f, 2.f);
    const T *xr[4];
    PairAcc acc[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        xr[u] = X + (int64_t)(j[u] >= 0 ? j[u] : q) * ld;  // an empty slot reads the query row, discarded
        acc[u].hi = pack2(base[u], base[u]);
        acc[u].lo = pack2(0.f, 0.f);
    }
    int64_t a0 = 0;
    if (vec) {
        const int64_t mv = m / VEC * VEC;  // vector part of the row; the tail is scalar
        for (int64_t a = (int64_t)gl * VEC; a < mv; a += G * VEC) {
            uint4 yv[4];
            const uint4 qv = __ldg(reinterpret_cast<const uint4 *>(xq + a));
#pragma unroll
            for (int u = 0; u < 4; ++u) yv[u] = __ldg(reinterpret_cast<const uint4 *>(xr[u] + a));
            f2 xe[NP];
            widen<T>(qv, xe);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                f2 ye[NP];
                widen<T>(yv[u], ye);
#pragma unroll
                for (int e = 0; e < NP; ++e) acc_sqdiff2(acc[u], xe[e], ye[e], minus, two);
            }
        }
        a0 = mv;
    }
    for (int64_t a = a0 + gl; a < m; a += G) {
        const float x = load_elem(xq + a);
#pragma unroll
        for (int u = 0; u < 4; ++u) acc_sqdiff2(acc[u], pack2(x, 0.f), pack2(load_elem(xr[u] + a), 0.f), minus, two);
    }
    unsigned bad = 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float2 h = unpack2(acc[u].hi), l = unpack2(acc[u].lo);
        if (!(h.x < 2.f * base[u]) || !(h.y < 2.f * base[u])) bad |= 1u << u;
        // two sums of a lane, then the group's: renormalised float-float additions
        ff s, e;
        two_sum(h.x - base[u], l.x, s.hi, s.lo);
        two_sum(h.y - base[u], l.y, e.hi, e.lo);
        out[u] = ff_add(s, e);
    }
    for (int o = G >> 1; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u) out[u] = ff_add(out[u], ff_shfl_xor(out[u], o));
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (8.f * out[u].hi < base[u] && out[u].hi != 0.f && j[u] >= 0) bad |= 1u << u;
    bad = __reduce_or_sync(0xffffffffu, bad);  // any group's: the renormalised form is never less accurate
    if (bad) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if ((bad >> u) & 1u) out[u] = exact_dist_renorm<T>(xq, xr[u], m, G);
    }
}

template <typename T, bool BATCH>
__global__ void __launch_bounds__(RR_WARPS * 32)
knn_rerank_kernel(const T *__restrict__ X_, int64_t N_, int64_t m_, int64_t ld_,
                  const float *__restrict__ norms_, int64_t q0_, int64_t nq, int kc_, int nsplit_, int k_,
                  const float *__restrict__ cand_d_, const int32_t *__restrict__ cand_i_,
                  int32_t *__restrict__ idx_out_, float *__restrict__ dist_out_,
                  int32_t *__restrict__ flags_, DevCounters *ctr, const KnnSet *__restrict__ sets, int nsets,
                  int lmax, const float *__restrict__ resid_, const float *__restrict__ maxima_, int quant_) {
    extern __shared__ float rsm[];
    constexpr unsigned FULL = 0xffffffffu;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t qi = (int64_t)blockIdx.x * RR_WARPS + w;  // the launch's row (the batch's row when batched)
    if (qi >= nq) return;
    // the row's dataset: the arguments, or its entry of a batch's table
    const T *X = X_;
    int64_t N = N_, m = m_, ld = ld_, q0 = q0_;
    const float *norms = norms_, *cand_d = cand_d_;
    const int32_t *cand_i = cand_i_;
    int32_t *idx_out = idx_out_, *flags = flags_;
    float *dist_out = dist_out_;
    const float *resid = resid_, *maxima = maxima_;
    int quant = quant_;
    int kc = kc_, nsplit = nsplit_, k = k_;
    if constexpr (BATCH) {
        const KnnSet &d = find_set_row(sets, nsets, qi);
        qi -= d.row_begin;
        X = static_cast<const T *>(d.X);
        N = d.N;
        m = d.m;
        ld = d.ld;
        q0 = 0;
        norms = d.norms;
        cand_d = d.cand_d;
        cand_i = d.cand_i;
        idx_out = d.idx;
        flags = d.flags;
        dist_out = nullptr;
        kc = d.kcl;
        nsplit = d.lists;
        k = d.k;
        resid = d.resid;
        maxima = d.maxima;
        quant = d.quant;
    }
    const int L = kc * nsplit;
    const int LS = BATCH ? lmax : L;  // per-warp shared-memory size in candidates
    // the row's candidates: d~ as ordered keys and indices; the evaluated ones
    unsigned *key = reinterpret_cast<unsigned *>(rsm + (size_t)w * (2 * LS + 4 * RR_CAP));
    int *ci = reinterpret_cast<int *>(key + LS);
    float *eh = reinterpret_cast<float *>(ci + LS), *el = eh + RR_CAP;
    int *ei = reinterpret_cast<int *>(el + RR_CAP), *ec = ei + RR_CAP;
    const int64_t q = q0 + qi;
    const float *cd = cand_d + qi * (int64_t)L;
    const int32_t *cidx = cand_i + qi * (int64_t)L;
    const T *xq = X + q * ld;
    const float nq_ = norms[q];

    // a complete search leaves -1 or a row of X in every slot; anything else
    // (slots a search that timed out never wrote) is skipped, never read
    bool bad = false;
    unsigned kmin = 0xffffffffu, kmax = 0u;
    int live = 0;
    float thr = INFINITY;
    for (int sp = 0; sp < nsplit; ++sp) {
        // a list that is full admitted only d~ < its maximum
        float mx = -INFINITY;
        bool full = true;
        for (int c = sp * kc + lane; c < (sp + 1) * kc; c += 32) {
            int j = cidx[c];
            if (j >= N) { bad = true; j = -1; }
            const float d = cd[c];
            const unsigned kk = order_key(d);
            key[c] = kk;
            ci[c] = j;
            mx = fmaxf(mx, d);
            full = full && j >= 0;
            if (j >= 0) {
                ++live;
                kmin = min(kmin, kk);
                kmax = max(kmax, kk);
            }
        }
        mx = warp_max(mx);
        if (__all_sync(FULL, full)) thr = fminf(thr, mx);
    }
    live = __reduce_add_sync(FULL, live);
    kmin = __reduce_min_sync(FULL, kmin);
    kmax = __reduce_max_sync(FULL, kmax);
    __syncwarp();

    constexpr int VEC = 16 / (int)sizeof(T);
    const bool vec = (ld % VEC == 0) && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    // lanes per candidate: a power of two that a narrow row still fills
    int G = 32;
    while (G > 4 && (vec ? (G / 2) * VEC : G / 2) >= m) G >>= 1;
    const int per = 32 / G, gid = lane / G;

    // the a-priori part of e_hi (FP32 rows searched in BF16): a bound on |x.y -
    // (the search's product)| for any candidate y, with the dataset's largest |y|
    // and rounding terms.
    //   single (x = h + d):      |h||d_y| + |d||h_y| + |d||d_y|
    //   split (x = h + l + r):   |l||l_y| + |h + l||r_y| + |r||h_y + l_y| + |r||r_y|
    // The tensor core's FP32 accumulation stays with the estimate.
    float e_apriori = -INFINITY;
    if (quant != KNN_QUANT_NONE) {
        const float t1 = resid[2 * q], t2 = resid[2 * q + 1], xn = sqrtf(nq_);
        const float ym = sqrtf(maxima[0]), m1 = maxima[1], m2 = maxima[2];
        const float b = quant == KNN_QUANT_SINGLE ? (xn + t1) * m1 + t1 * (ym + m1) + t1 * m1
                                                  : t1 * m1 + (xn + t2) * m2 + t2 * (ym + m2) + t2 * m2;
        e_apriori = 2.f * b * (1.f + 9.765625e-04f) + ldexpf(nq_ + maxima[0], -21);
    }

    float err_max = -INFINITY, err_min = INFINITY, nmax = 0.f;
    int n = 0;            // evaluated candidates held (eh, el, ei)
    float theta = INFINITY, e_hi = INFINITY;
    const unsigned kend = min(kmax, 0xfffffffeu) + 1u;  // past every key
    auto count_below = [&](unsigned t) {  // candidates not evaluated yet with key < t
        int c = 0;
        for (int i = lane; i < L; i += 32) c += ci[i] >= 0 && key[i] < t;
        return (int)__reduce_add_sync(FULL, c);
    };
    // first the k + RR_EXTRA smallest: a key with that many candidates below it (to a
    // few), by bisection; count_below(lo) < want <= count_below(hi)
    unsigned want_key = kend;
    if (const int want = min(live, k + RR_EXTRA); want > 0) {
        unsigned lo = kmin;
        while (want_key - lo > 1u) {
            const unsigned mid = lo + (want_key - lo) / 2u;
            const int c = count_below(mid);
            if (c >= want) {
                want_key = mid;
                if (c <= want + 4) break;
            } else {
                lo = mid;
            }
        }
    }
    // and, in the same pass, RR_SAMPLE candidates spread over the lists and the largest
    // d~ of all: the sample that the error estimate needs besides the nearest
    int every = (live + RR_SAMPLE - 1) / RR_SAMPLE;  // 0: no sample (the later passes)
    while (live > 0) {
        // ---- the next candidates: those below want_key, as many as there is room for
        // (the rest, equal keys for instance, in the passes that follow); an evaluated
        // one leaves the list
        const int room = RR_CAP - n;
        int nb = 0, seen = 0;
        for (int i0 = 0; i0 < L && nb < room; i0 += 32) {
            const int i = i0 + lane;
            const bool in = i < L && ci[i] >= 0;
            bool take = in && key[i] < want_key;
            if (every) {
                const unsigned am = __ballot_sync(FULL, in);
                const int ord = seen + __popc(am & ((1u << lane) - 1u));
                take = take || (in && (ord % every == 0 || key[i] == kmax));
                seen += __popc(am);
            }
            const unsigned mk = __ballot_sync(FULL, take);
            const int pos = nb + __popc(mk & ((1u << lane) - 1u));
            if (take && pos < room) {
                ec[n + pos] = i;
                ei[n + pos] = ci[i];
                ci[i] = -1;
            }
            nb += __popc(mk);
        }
        nb = min(nb, room);
        every = 0;
        __syncwarp();
        // ---- their exact distances
        for (int c0 = n; c0 < n + nb; c0 += 4 * per) {
            int cc[4], j[4];
            float base[4], dt[4];
            ff d[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                cc[u] = c0 + u * per + gid;
                const bool in = cc[u] < n + nb;
                j[u] = in ? ei[cc[u]] : -1;
                dt[u] = in ? cd[ec[cc[u]]] : 0.f;
                // 2^b above twice the search's distance
                base[u] = __uint_as_float(min((__float_as_uint(fabsf(dt[u])) & 0x7f800000u) + (2u << 23), 0x7e800000u));
            }
            exact_dist4<T>(X, m, ld, xq, q, j, base, G, vec, d);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j[u] >= 0) {
                    const float e = dt[u] - d[u].hi;  // overestimate of the search's distance
                    err_max = fmaxf(err_max, e);
                    err_min = fminf(err_min, e);
                    nmax = fmaxf(nmax, norms[j[u]]);
                    if ((lane & (G - 1)) == 0) {
                        eh[cc[u]] = d[u].hi;
                        el[cc[u]] = d[u].lo;
                    }
                }
        }
        n += nb;
        __syncwarp();
        err_max = warp_max(err_max);
        err_min = -warp_max(-err_min);
        nmax = warp_max(nmax);
        // ---- the k best of the evaluated ones, in order, to the front
        float vh[RR_CAP / 32], vl[RR_CAP / 32];
        int vi[RR_CAP / 32], vr[RR_CAP / 32];
#pragma unroll
        for (int t = 0; t < RR_CAP / 32; ++t) {
            const int c = t * 32 + lane;
            vr[t] = RR_CAP;
            if (c < n) {
                vh[t] = eh[c];
                vl[t] = el[c];
                vi[t] = ei[c];
                int rank = 0;
                for (int o = 0; o < n; ++o) rank += ff_less(ff{eh[o], el[o]}, ei[o], ff{vh[t], vl[t]}, vi[t]);
                vr[t] = rank;
            }
        }
        __syncwarp();
#pragma unroll
        for (int t = 0; t < RR_CAP / 32; ++t)
            if (vr[t] < k) {
                eh[vr[t]] = vh[t];
                el[vr[t]] = vl[t];
                ei[vr[t]] = vi[t];
            }
        __syncwarp();
        n = min(n, k);
        theta = n == k ? eh[k - 1] : INFINITY;
        // a point within theta has a norm of at most |x| + sqrt(theta)
        const float yn = sqrtf(nq_) + sqrtf(fmaxf(theta, 0.f));
        e_hi = fmaxf(fmaxf(err_max, 0.f) + 3.f * (err_max - err_min) + ldexpf(nq_ + fmaxf(nmax, yn * yn), -21),
                     e_apriori);
        // ---- candidates left that could still enter: d~ <= theta + e_hi
        const float lim = theta + e_hi;
        want_key = lim < INFINITY ? min(order_key(lim) + 1u, kend) : kend;
        if (count_below(want_key) == 0) break;
    }
    for (int c = lane; c < n; c += 32) {
        idx_out[qi * k + c] = ei[c];
        if (dist_out) dist_out[qi * k + c] = eh[c] + el[c];
    }
    if (lane == 0 && bad) atomicOr(&ctr->status, (unsigned)DEV_INVALID);
    if (lane == 0) {
        // theta as before when fewer than k candidates exist: certified by thr = +inf
        const int ok = (thr == INFINITY) || (n == k && thr - e_hi > theta);
        flags[qi] = ok ? 0 : 1;
        if (!ok) atomicAdd(&ctr->knn_uncertified, 1ull);
    }
}

size_t knn_rerank_smem(int L) { return (size_t)RR_WARPS * (2 * L + 4 * RR_CAP) * sizeof(float); }

cudaError_t launch_knn_rerank(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld,
                              const float *norms, int64_t q0, int64_t nq, int kc, int nsplit, int k,
                              const float *cand_d, const int32_t *cand_i, int32_t *idx_out,
                              float *dist_out, int32_t *flags, DevCounters *ctr, cudaStream_t s,
                              const float *resid, const float *maxima, int quant) {
    if (!resid || !maxima) quant = KNN_QUANT_NONE;
    if (nq <= 0) return cudaSuccess;
    int L = kc * nsplit;
    if (L > RR_MAXL) return cudaErrorInvalidValue;
    size_t smem = knn_rerank_smem(L);
    dim3 grid((unsigned)((nq + RR_WARPS - 1) / RR_WARPS)), block(RR_WARPS * 32);
    cudaError_t e;
    if (dt == MECUCO_BF16) {
        e = cudaFuncSetAttribute(knn_rerank_kernel<__nv_bfloat16, false>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        knn_rerank_kernel<__nv_bfloat16, false><<<grid, block, smem, s>>>((const __nv_bfloat16 *)X, N, m, ld, norms,
                                                                          q0, nq, kc, nsplit, k, cand_d, cand_i,
                                                                          idx_out, dist_out, flags, ctr, nullptr, 0, 0,
                                                                          resid, maxima, quant);
    } else {
        e = cudaFuncSetAttribute(knn_rerank_kernel<float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return e;
        knn_rerank_kernel<float, false><<<grid, block, smem, s>>>((const float *)X, N, m, ld, norms, q0, nq, kc,
                                                                  nsplit, k, cand_d, cand_i, idx_out, dist_out, flags,
                                                                  ctr, nullptr, 0, 0, resid, maxima, quant);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Exact full scan for flagged rows: one CTA of 8 warps per query; warp w takes
// candidates j = w, w + 8, ...; each distance is a warp-cooperative compensated
// sum; lane 0 keeps the warp's k best in shared memory (sorted insertion);
// finally the 8 lists are merged by rank.
// ---------------------------------------------------------------------------
constexpr int FB_WARPS = 8;

template <typename T, bool BATCH>
__global__ void __launch_bounds__(FB_WARPS * 32)
knn_fallback_kernel(const T *__restrict__ X_, int64_t N_, int64_t m_, int64_t ld_, int64_t q0_,
                    int64_t nq, int k_, int include_self_, const int32_t *__restrict__ flags_,
                    int32_t *__restrict__ idx_out_, float *__restrict__ dist_out_, DevCounters *ctr,
                    const KnnSet *__restrict__ sets, int nsets, int kmax) {
    extern __shared__ float fsm[];
    const int KS = BATCH ? kmax : k_;      // shared-memory stride of one warp's list
    float *bh = fsm;                       // [FB_WARPS][KS]
    float *bl = bh + FB_WARPS * KS;        // [FB_WARPS][KS]
    int *bi = reinterpret_cast<int *>(bl + FB_WARPS * KS);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int64_t gi = blockIdx.x; gi < nq; gi += gridDim.x) {
        // the row's dataset: the arguments, or its entry of a batch's table
        const T *X = X_;
        int64_t N = N_, m = m_, ld = ld_, q0 = q0_, qi = gi;
        const int32_t *flags = flags_;
        int32_t *idx_out = idx_out_;
        float *dist_out = dist_out_;
        int k = k_, include_self = include_self_;
        if constexpr (BATCH) {
            const KnnSet &d = find_set_row(sets, nsets, gi);
            qi = gi - d.row_begin;
            X = static_cast<const T *>(d.X);
            N = d.N;
            m = d.m;
            ld = d.ld;
            q0 = 0;
            flags = d.flags;
            idx_out = d.idx;
            dist_out = nullptr;
            k = d.k;
            include_self = d.include_self;
        }
        if (flags[qi] == 0) continue;  // uniform across the CTA
        const int64_t q = q0 + qi;
        const T *xq = X + q * ld;
        float *mh = bh + w * KS, *ml = bl + w * KS;
        int *mi = bi + w * KS;
        if (lane == 0)
            for (int s = 0; s < k; ++s) { mh[s] = INFINITY; ml[s] = 0.f; mi[s] = 0x7fffffff; }
        __syncwarp();
        for (int64_t j = w; j < N; j += FB_WARPS) {
            if (!include_self && j == q) continue;
            const T *xj = X + j * ld;
            ff acc{0.f, 0.f};
            for (int64_t a = lane; a < m; a += 32) ff_acc_sqdiff(acc, load_elem(xq + a), load_elem(xj + a));
            acc = ff_warp_sum(acc);
            if (lane == 0 && ff_less(acc, (int)j, ff{mh[k - 1], ml[k - 1]}, mi[k - 1])) {
                int pos = k - 1;
                while (pos > 0 && ff_less(acc, (int)j, ff{mh[pos - 1], ml[pos - 1]}, mi[pos - 1])) {
                    mh[pos] = mh[pos - 1]; ml[pos] = ml[pos - 1]; mi[pos] = mi[pos - 1];
                    --pos;
                }
                mh[pos] = acc.hi; ml[pos] = acc.lo; mi[pos] = (int)j;
            }
            __syncwarp();
        }
        __syncthreads();
        // merge: rank every entry among all FB_WARPS * k entries
        for (int e = threadIdx.x; e < FB_WARPS * KS; e += blockDim.x) {
            if (e % KS >= k || bi[e] == 0x7fffffff) continue;
            ff me{bh[e], bl[e]};
            int rank = 0;
            for (int o = 0; o < FB_WARPS * KS; ++o)
                if (o % KS < k && bi[o] != 0x7fffffff && ff_less(ff{bh[o], bl[o]}, bi[o], me, bi[e])) ++rank;
            if (rank < k) {
                idx_out[qi * k + rank] = bi[e];
                if (dist_out) dist_out[qi * k + rank] = me.hi + me.lo;
            }
        }
        if (threadIdx.x == 0) atomicAdd(&ctr->knn_fallback_rows, 1ull);
        __syncthreads();
    }
}

cudaError_t launch_knn_fallback(const void *X, mecuco_dtype dt, int64_t N, int64_t m, int64_t ld,
                                int64_t q0, int64_t nq, int k, int include_self, const int32_t *flags,
                                int32_t *idx_out, float *dist_out, DevCounters *ctr, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    size_t smem = (size_t)FB_WARPS * k * 3 * sizeof(float);
    unsigned grid = (unsigned)(nq < 4096 ? nq : 4096);
    if (dt == MECUCO_BF16)
        knn_fallback_kernel<__nv_bfloat16, false><<<grid, FB_WARPS * 32, smem, s>>>(
            (const __nv_bfloat16 *)X, N, m, ld, q0, nq, k, include_self, flags, idx_out, dist_out, ctr, nullptr, 0, 0);
    else
        knn_fallback_kernel<float, false><<<grid, FB_WARPS * 32, smem, s>>>(
            (const float *)X, N, m, ld, q0, nq, k, include_self, flags, idx_out, dist_out, ctr, nullptr, 0, 0);
    return cudaGetLastError();
}

// Batched forms: the rows of every dataset of a table, one launch.
cudaError_t launch_knn_rerank_batch(const KnnSet *sets, int nsets, int64_t nrows, int lmax, mecuco_dtype dt,
                                    DevCounters *ctr, cudaStream_t s) {
    if (nrows <= 0) return cudaSuccess;
    if (lmax > RR_MAXL) return cudaErrorInvalidValue;
    size_t smem = knn_rerank_smem(lmax);
    dim3 grid((unsigned)((nrows + RR_WARPS - 1) / RR_WARPS)), block(RR_WARPS * 32);
    cudaError_t e;
    if (dt == MECUCO_BF16) {
        e = cudaFuncSetAttribute(knn_rerank_kernel<__nv_bfloat16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return e;
        knn_rerank_kernel<__nv_bfloat16, true><<<grid, block, smem, s>>>(nullptr, 0, 0, 0, nullptr, 0, nrows, 0, 0, 0,
                                                                         nullptr, nullptr, nullptr, nullptr, nullptr,
                                                                         ctr, sets, nsets, lmax, nullptr, nullptr, 0);
    } else {
        e = cudaFuncSetAttribute(knn_rerank_kernel<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return e;
        knn_rerank_kernel<float, true><<<grid, block, smem, s>>>(nullptr, 0, 0, 0, nullptr, 0, nrows, 0, 0, 0, nullptr,
                                                                 nullptr, nullptr, nullptr, nullptr, ctr, sets, nsets,
                                                                 lmax, nullptr, nullptr, 0);
    }
    return cudaGetLastError();
}

cudaError_t launch_knn_fallback_batch(const KnnSet *sets, int nsets, int64_t nrows, int kmax, mecuco_dtype dt,
                                      DevCounters *ctr, cudaStream_t s) {
    if (nrows <= 0) return cudaSuccess;
    size_t smem = (size_t)FB_WARPS * kmax * 3 * sizeof(float);
    unsigned grid = (unsigned)(nrows < 4096 ? nrows : 4096);
    if (dt == MECUCO_BF16)
        knn_fallback_kernel<__nv_bfloat16, true><<<grid, FB_WARPS * 32, smem, s>>>(
            nullptr, 0, 0, 0, 0, nrows, 0, 0, nullptr, nullptr, nullptr, ctr, sets, nsets, kmax);
    else
        knn_fallback_kernel<float, true><<<grid, FB_WARPS * 32, smem, s>>>(
            nullptr, 0, 0, 0, 0, nrows, 0, 0, nullptr, nullptr, nullptr, ctr, sets, nsets, kmax);
    return cudaGetLastError();
}

}  // namespace mecuco
