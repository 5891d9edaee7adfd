// Dense linear algebra and grouping kernels of the index build and the query
// prologue:
//   * rotation o' = P^T (o_r - c) with FP64 accumulation (index time) -- the
//     Section 3.3 workflow step "apply P^{-1} to the data vectors";
//   * FP32 SGEMM (query rotation q' = P^T q_r, centroid distances for the IVF
//     probe of Section 4.1, the P-multiply of the backward pass);
//   * cluster means (Section 5.1 local centring) and a stable counting sort
//     that groups rows by cluster (IVF lists, Section 4.1);
//   * per-row selection of the p smallest entries (probe lists, k-means).
#include <cuda_runtime.h>
#include <stdint.h>

#include "erq_kernels.cuh"
#include "warp_sort.cuh"

namespace erq {

// ---------------------------------------------------------------------------
// Rotation with FP64 accumulation.
//   out[r][j] = fl32( sum_{k=0..D-1, ascending} (double)res_k * (double)P[k][j] )
//   res_k     = fl32(X[src][k] - C[cl][k])  (or X[src][k] when C == nullptr)
// Products of two FP32 values are exact in FP64, so fma(res, p, acc) equals the
// sequential "acc += res * p" of a plain FP64 loop: the result is bit-identical
// to any implementation that sums in ascending k.
// Tile 64 rows x 64 columns, 256 threads, 4x4 outputs per thread, BK = 16.
// The FP64 pipe bounds it (0.75 TFLOP/s).  launch_rotate_fp64 therefore takes
// the sliced tensor-core form of the same sums (k_rotate_tc.cu: 100,000 x 768
// in 3 ms instead of 156) wherever it can allocate its digits; this kernel runs
// inside a stream capture and, with `flag`, for a block that the sliced form
// gave up on.
// ---------------------------------------------------------------------------
constexpr int R64_BM = 64, R64_BN = 64, R64_BK = 16;

__global__ void __launch_bounds__(256) rotate_fp64_kernel(const float* __restrict__ X,
                                                          const int64_t* __restrict__ gather,
                                                          const float* __restrict__ C,
                                                          const int32_t* __restrict__ cl,
                                                          const float* __restrict__ P, float* __restrict__ out,
                                                          int64_t n, int D, const uint32_t* __restrict__ flag) {
    if (flag && *flag == 0u) return;
    __shared__ float As[R64_BK][R64_BM + 4];
    __shared__ float Bs[R64_BK][R64_BN + 4];
    const int tid = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.y * R64_BM;
    const int col0 = blockIdx.x * R64_BN;
    const int tr = tid / 16, tc = tid % 16;
    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;

    // loader mapping: A tile 64 rows x 16 k = 1024 floats, 4 per thread
    const int a_row = tid / 4, a_k = (tid % 4) * 4;
    const int64_t grow = row0 + a_row;
    const float* xrow = nullptr;
    const float* crow = nullptr;
    if (grow < n) {
        const int64_t src = gather ? gather[grow] : grow;
        xrow = X + src * (int64_t)D;
        if (C) crow = C + (int64_t)(cl ? cl[grow] : 0) * D;
    }
    // B tile 16 k x 64 cols = 1024 floats, 4 per thread
    const int b_k = tid / 16, b_c = (tid % 16) * 4;

    for (int k0 = 0; k0 < D; k0 += R64_BK) {
        float4 av = make_float4(0.f, 0.f, 0.f, 0.f);
        if (xrow) {
            av = *reinterpret_cast<const float4*>(xrow + k0 + a_k);
            if (crow) {
                const float4 cv = *reinterpret_cast<const float4*>(crow + k0 + a_k);
                av.x = __fsub_rn(av.x, cv.x);
                av.y = __fsub_rn(av.y, cv.y);
                av.z = __fsub_rn(av.z, cv.z);
                av.w = __fsub_rn(av.w, cv.w);
            }
        }
        As[a_k + 0][a_row] = av.x;
        As[a_k + 1][a_row] = av.y;
        As[a_k + 2][a_row] = av.z;
        As[a_k + 3][a_row] = av.w;
        const float4 bv = *reinterpret_cast<const float4*>(P + (int64_t)(k0 + b_k) * D + col0 + b_c);
        *reinterpret_cast<float4*>(&Bs[b_k][b_c]) = bv;
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < R64_BK; ++kk) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = (double)As[kk][tr * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = (double)Bs[kk][tc * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = __fma_rn(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t r = row0 + tr * 4 + i;
        if (r >= n) continue;
        float4 o;
        o.x = __double2float_rn(acc[i][0]);
        o.y = __double2float_rn(acc[i][1]);
        o.z = __double2float_rn(acc[i][2]);
        o.w = __double2float_rn(acc[i][3]);
        *reinterpret_cast<float4*>(out + r * D + col0 + tc * 4) = o;
    }
}

cudaError_t launch_rotate_fp64(const float* X, const int64_t* gather, const float* C, const int32_t* cl,
                               const float* P, float* out, int64_t n, int D, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const cudaError_t e = launch_rotate_tc(X, gather, C, cl, P, out, n, D, s);
    return e != cudaErrorNotSupported ? e : launch_rotate_fp64_if(nullptr, X, gather, C, cl, P, out, n, D, s);
}

cudaError_t launch_rotate_fp64_if(const uint32_t* flag, const float* X, const int64_t* gather, const float* C,
                                  const int32_t* cl, const float* P, float* out, int64_t n, int D, cudaStream_t s) {
    const int64_t slab = 65535ll * R64_BM;
    for (int64_t r0 = 0; r0 < n; r0 += slab) {
        const int64_t m = n - r0 < slab ? n - r0 : slab;
        dim3 grid(D / R64_BN, (unsigned)ceil_div(m, R64_BM));
        // rows are addressed through `gather` when given, else directly
        count_launch();
        rotate_fp64_kernel<<<grid, 256, 0, s>>>(gather ? X : X + r0 * D, gather ? gather + r0 : nullptr, C,
                                                cl ? cl + r0 : nullptr, P, out + r0 * D, m, D, flag);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP32 SGEMM  C[M][N] = A[M][K] * op(B), op(B) = B[K][N] (NN) or B[N][K]^T (NT).
// 128x128 tile, BK = 8, 256 threads, 8x8 outputs per thread (split 4+4 in both
// dimensions), register prefetch of the next tile.  K % 8 == 0; for NN N % 4 == 0.
// Epilogues:
//   EPI_PLAIN : C = alpha * acc + (addend ? addend[m][n] : 0)
//   EPI_DIST  : C = rown[m] + coln[n] - 2 * acc      (squared L2 distances)
// ---------------------------------------------------------------------------
enum { EPI_PLAIN = 0, EPI_DIST = 1 };

// Two FP32 multiply-adds in one instruction, each rounded as fmaf (the 64 FMAs of
// a k step are 32 issue slots: 100,000 x 256 x 768, 0.916 -> 0.887 ms).
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t pack2(float x, float y) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// LIST: row i of the product is row list[i] of A, for the *count listed rows.
template <bool NT, int EPI, bool LIST = false>
__global__ void __launch_bounds__(256) sgemm_kernel(const float* __restrict__ A, const float* __restrict__ Bm,
                                                    float* __restrict__ Cm, int64_t M, int N, int K, float alpha,
                                                    const float* __restrict__ addend,
                                                    const float* __restrict__ rown,
                                                    const float* __restrict__ coln, int64_t ldc,
                                                    const int32_t* __restrict__ list = nullptr,
                                                    const int32_t* __restrict__ count = nullptr) {
    if (LIST) {
        M = *count;
        if ((int64_t)blockIdx.y * 128 >= M) return;
    }
    __shared__ __align__(16) float As[2][8][128];
    __shared__ __align__(16) float Bs[2][8][128];
    const int tid = threadIdx.x;
    const int64_t m0 = (int64_t)blockIdx.y * 128;
    const int n0 = blockIdx.x * 128;
    // A loader: row tid/2, k offset (tid%2)*4
    const int la_r = tid >> 1, la_k = (tid & 1) * 4;
    const bool a_ok = (m0 + la_r) < M;
    const float* a_ptr = A + (a_ok ? (LIST ? (int64_t)list[m0 + la_r] : m0 + la_r) : 0) * (int64_t)K + la_k;
    // B loader
    int lb_k, lb_n;
    bool b_ok;
    const float* b_ptr;
    if (NT) {
        lb_n = tid >> 1;
        lb_k = (tid & 1) * 4;
        b_ok = (n0 + lb_n) < N;
        b_ptr = Bm + (int64_t)(b_ok ? (n0 + lb_n) : 0) * K + lb_k;
    } else {
        lb_k = tid >> 5;
        lb_n = (tid & 31) * 4;
        b_ok = (n0 + lb_n) < N;
        b_ptr = Bm + (int64_t)lb_k * N + (b_ok ? n0 + lb_n : 0);
    }
    float4 ra, rb;
    auto load_regs = [&](int k0) {
        ra = a_ok ? *reinterpret_cast<const float4*>(a_ptr + k0) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (NT)
            rb = b_ok ? *reinterpret_cast<const float4*>(b_ptr + k0) : make_float4(0.f, 0.f, 0.f, 0.f);
        else
            rb = b_ok ? *reinterpret_cast<const float4*>(b_ptr + (int64_t)k0 * N) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto store_smem = [&](int buf) {
        As[buf][la_k + 0][la_r] = ra.x;
        As[buf][la_k + 1][la_r] = ra.y;
        As[buf][la_k + 2][la_r] = ra.z;
        As[buf][la_k + 3][la_r] = ra.w;
        if (NT) {
            Bs[buf][lb_k + 0][lb_n] = rb.x;
            Bs[buf][lb_k + 1][lb_n] = rb.y;
            Bs[buf][lb_k + 2][lb_n] = rb.z;
            Bs[buf][lb_k + 3][lb_n] = rb.w;
        } else {
            *reinterpret_cast<float4*>(&Bs[buf][lb_k][lb_n]) = rb;
        }
    };
    uint64_t acc2[8][4];                     // columns 2 j, 2 j + 1 of the thread's eight
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc2[i][j] = 0ull;
    const int ty = tid / 16, tx = tid % 16;
    load_regs(0);
    store_smem(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += 8) {
        const bool more = (k0 + 8) < K;
        if (more) load_regs(k0 + 8);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][64 + ty * 4]);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][tx * 4]);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][64 + tx * 4]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const uint64_t b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint64_t aa = pack2(a[i], a[i]);
#pragma unroll
                for (int j = 0; j < 4; ++j) fma2(acc2[i][j], aa, b[j]);
            }
        }
        if (more) {
            store_smem(buf ^ 1);
            __syncthreads();
            buf ^= 1;
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t m = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4));
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int nn = n0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + (j - 4));
            if (nn >= N) continue;
            const float2 pr = unpack2(acc2[i][j >> 1]);
            const float ac = (j & 1) ? pr.y : pr.x;
            float v;
            if (EPI == EPI_DIST) {
                v = rown[LIST ? (int64_t)list[m] : m] + coln[nn] - 2.f * ac;
            } else {
                v = alpha * ac;
                if (addend) v += addend[m * ldc + nn];
            }
            Cm[m * ldc + nn] = v;
        }
    }
}

constexpr int64_t kMaxSlabRows = 65535ll * 128;  // gridDim.y limit x tile rows

cudaError_t launch_sgemm(bool nt, const float* A, const float* B, float* C, int64_t M, int N, int K, float alpha,
                         const float* addend, cudaStream_t s) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    for (int64_t m0 = 0; m0 < M; m0 += kMaxSlabRows) {
        const int64_t m = M - m0 < kMaxSlabRows ? M - m0 : kMaxSlabRows;
        dim3 grid((unsigned)ceil_div(N, 128), (unsigned)ceil_div(m, 128));
        const float* add = addend ? addend + m0 * N : nullptr;
        count_launch();
        if (nt)
            sgemm_kernel<true, EPI_PLAIN><<<grid, 256, 0, s>>>(A + m0 * K, B, C + m0 * N, m, N, K, alpha, add, nullptr,
                                                               nullptr, N);
        else
            sgemm_kernel<false, EPI_PLAIN><<<grid, 256, 0, s>>>(A + m0 * K, B, C + m0 * N, m, N, K, alpha, add,
                                                                nullptr, nullptr, N);
    }
    return cudaGetLastError();
}

cudaError_t launch_sqdist(const float* Q, const float* qn, const float* C, const float* cn, float* out, int64_t nq,
                          int nc, int D, cudaStream_t s) {
    if (nq <= 0 || nc <= 0) return cudaSuccess;
    for (int64_t m0 = 0; m0 < nq; m0 += kMaxSlabRows) {
        const int64_t m = nq - m0 < kMaxSlabRows ? nq - m0 : kMaxSlabRows;
        dim3 grid((unsigned)ceil_div(nc, 128), (unsigned)ceil_div(m, 128));
        count_launch();
        sgemm_kernel<true, EPI_DIST><<<grid, 256, 0, s>>>(Q + m0 * D, C, out + m0 * nc, m, nc, D, 1.f, nullptr,
                                                          qn + m0, cn, nc);
    }
    return cudaGetLastError();
}

// Squared norms of rows (FP32, one warp per row).
__global__ void row_sqnorm_kernel(const float* __restrict__ X, int64_t n, int D, float* __restrict__ out) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n) return;
    const float* x = X + w * D;
    float s = 0.f;
    for (int k = lane * 4; k < D; k += 128) {
        const float4 v = *reinterpret_cast<const float4*>(x + k);
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
    }
    s = warp_sum(s);
    if (lane == 0) out[w] = s;
}

// Rows scaled to unit length (cosine similarity as the inner product of unit
// vectors): y = fl32(x / sqrt(sum x^2)) with the sum in FP64, one warp per
// row; a zero row stays zero.  X and Y may be the same array (each thread
// rewrites only the elements it read).
//
// The FP64 pipe does two lanes a clock, and a division is some twenty of its
// instructions: dividing every element took 184 us for 4,000 x 1,536, 43 us
// with the division done in FP32 pairs.  1 / norm is split as r + t (one
// FP64 division a row); x r is formed as a product and its exact remainder, x t
// is added to the remainder, and the pair (product, remainder) is x / norm to
// 2^-45.  Its rounding to FP32 is x / norm's unless the part dropped lies within
// 2^-45 of a rounding boundary; those elements (2^-18 of them), those of a power
// of two and those too small for an exact remainder are divided in FP64.
__device__ __forceinline__ float div_by_norm(float x, double nrm, float r, float t) {
    if (x == 0.f) return x;
    const float y = x * r;
    const float e = fmaf(x, t, fmaf(x, r, -y));
    const float s = y + e, d = e - (s - y);                     // y + e = s + d exactly (|e| << |y|)
    const uint32_t b = __float_as_uint(s) & 0x7fffffffu;
    const float half = __uint_as_float(b & 0x7f800000u) * 5.9604644775390625e-8f;   // half the spacing at s: 2^-24
    if (fabsf(y) >= 1.2621774e-29f && fabsf(y) <= 1e30f && (b & 0x7fffffu) != 0u &&
        fabsf(d) <= half * 0.999998f)
        return s;
    return (float)((double)x / nrm);
}

__global__ void __launch_bounds__(256) normalize_rows_kernel(const float* X, int64_t n, int D, float* Y) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const float* x = X + r * D;
    double s = 0.0;
    int k = lane;
    for (; k + 224 < D; k += 256) {                             // eight loads in flight
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = x[k + 32 * u];
#pragma unroll
        for (int u = 0; u < 8; ++u) s += (double)v[u] * (double)v[u];
    }
    for (; k < D; k += 32) s += (double)x[k] * (double)x[k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const double nrm = sqrt(s);
    float* y = Y + r * D;
    if (!(nrm > 0.0)) {
        for (k = lane; k < D; k += 32) y[k] = 0.f;
        return;
    }
    const double inv = 1.0 / nrm;
    if (!(inv > 1e-30 && inv < 1e30)) {                         // (r and t would leave FP32's normal range)
        for (k = lane; k < D; k += 32) y[k] = (float)((double)x[k] / nrm);
        return;
    }
    const float ir = (float)inv, it = (float)(inv - (double)ir);
    for (k = lane; k + 224 < D; k += 256) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = x[k + 32 * u];
#pragma unroll
        for (int u = 0; u < 8; ++u) y[k + 32 * u] = div_by_norm(v[u], nrm, ir, it);
    }
    for (; k < D; k += 32) y[k] = div_by_norm(x[k], nrm, ir, it);
}

cudaError_t launch_normalize_rows(const float* X, int64_t n, int D, float* Y, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    normalize_rows_kernel<<<(unsigned)ceil_div(n * 32, 256), 256, 0, s>>>(X, n, D, Y);
    return cudaGetLastError();
}

cudaError_t launch_row_sqnorm(const float* X, int64_t n, int D, float* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    row_sqnorm_kernel<<<(unsigned)ceil_div(n * 32, 256), 256, 0, s>>>(X, n, D, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Cluster means (reading of Section 5.1 "local centroid"): per (cluster,
// coordinate) the FP64 sum over the cluster's rows in stored order (ascending
// original id), one division and one rounding to FP32.  Empty clusters keep
// `keep_empty ? old value : 0`.
//
// The FP64 sum in order is a chain of additions on a pipe of two lanes a clock
// (100,000 x 768 in 256 lists: 630 us).  It is formed as pairs of FP32 numbers
// instead (Knuth's two-sum: a running sum and the sum of its exact remainders),
// in segments of 32 rows that are added up in FP64, a sixteenth of the rows per
// thread.  The mean's rounding to FP32 is that of the sum in order unless it lies
// within the two sums' error bounds of a rounding boundary (a segment's remainders
// round within 32^2 2^-48 of its magnitudes, a sum in order within n 2^-53); those
// elements, about one in a thousand, are listed and summed in order.  240 us,
// half of them those few sums' chains; the rows' bytes take 45.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum_add(float x, float& s, float& c, float& m) {
    const float t = s + x, z = t - s;
    c += (s - (t - z)) + (x - z);
    s = t;
    m += fabsf(x);
}

constexpr int CW = 16;             // row slots of a block: 16 threads of four coordinates each
__global__ void __launch_bounds__(256) centroid_kernel(const float* __restrict__ X, const int64_t* __restrict__ list_off,
                                                       const int64_t* __restrict__ list_ids, int D,
                                                       float* __restrict__ C, int keep_empty,
                                                       int32_t* __restrict__ redo, int32_t* __restrict__ n_redo) {
    __shared__ double sh[2][CW][64];
    const int j = blockIdx.x, l = threadIdx.x & 15, w = threadIdx.x >> 4;
    const int k0 = blockIdx.y * 64;                                 // (D % 64 == 0)
    const int64_t b = list_off[j], e = list_off[j + 1];
    if (b == e) {
        if (!keep_empty && threadIdx.x < 64) C[(int64_t)j * D + k0 + threadIdx.x] = 0.f;
        return;
    }
    double S[4] = {0.0, 0.0, 0.0, 0.0}, G[4] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t r = b + w; r < e; r += 32 * CW) {
        float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f}, m[4] = {0.f, 0.f, 0.f, 0.f};
        for (int g = 0; g < 32 && r + g * CW < e; g += 4) {
            float4 x[4];                                            // four loads in flight
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t rr = r + (g + u) * CW;
                x[u] = rr < e ? *reinterpret_cast<const float4*>(X + list_ids[rr] * D + k0 + 4 * l)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                two_sum_add(x[u].x, s[0], c[0], m[0]);
                two_sum_add(x[u].y, s[1], c[1], m[1]);
                two_sum_add(x[u].z, s[2], c[2], m[2]);
                two_sum_add(x[u].w, s[3], c[3], m[3]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            S[i] += (double)s[i] + (double)c[i];
            G[i] += (double)m[i];
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        sh[0][w][4 * l + i] = S[i];
        sh[1][w][4 * l + i] = G[i];
    }
    __syncthreads();
    if (threadIdx.x >= 64) return;
    const int k = threadIdx.x;
    double sum = 0.0, mag = 0.0;
#pragma unroll
    for (int u = 0; u < CW; ++u) {
        sum += sh[0][u][k];
        mag += sh[1][u][k];
    }
    const double inv = 1.0 / (double)(e - b), mean = sum * inv;
    const double err = mag * inv * (0x1p-38 + ((double)(e - b) + 64.0) * 0x1p-52) * 1.01;
    const float lo = (float)(mean - err), hi = (float)(mean + err);
    float* out = C + (int64_t)j * D + k0 + k;
    // (not decided here: both sides of the interval round differently, sums that may have overflowed or underflowed)
    if (mag == 0.0) *out = 0.f;
    else if (lo == hi && mag < 1e37 && fabsf(lo) > 1e-25f) *out = lo;
    else redo[atomicAdd(n_redo, 1)] = (int32_t)((int64_t)j * D + k0 + k);
}

// (cluster, coordinate) pairs in FP64, in stored order: the listed ones, or all.
// Eight lanes per pair fetch 32 rows, the next 32 while these are added.
__global__ void __launch_bounds__(128) centroid_ordered_kernel(const float* __restrict__ X,
                                                               const int64_t* __restrict__ list_off,
                                                               const int64_t* __restrict__ list_ids, int64_t total,
                                                               int D, float* __restrict__ C, int keep_empty,
                                                               const int32_t* __restrict__ redo,
                                                               const int32_t* __restrict__ n_redo) {
    const int64_t n = redo ? (int64_t)*n_redo : total;
    const int lane = threadIdx.x & 31, l = lane & 7;
    const int64_t groups = (int64_t)gridDim.x * blockDim.x / 8;
    // (the groups of a warp take the same number of rounds: a warp's lanes stay together in the exchanges)
    for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32 * 4; i0 < n; i0 += groups) {
        const int64_t i = i0 + lane / 8;
        const int64_t t = i < n ? (redo ? (int64_t)redo[i] : i) : -1;
        const int j = t >= 0 ? (int)(t / D) : 0, k = t >= 0 ? (int)(t % D) : 0;
        const int64_t b = t >= 0 ? list_off[j] : 0, e = t >= 0 ? list_off[j + 1] : 0;
        int64_t rounds = (e - b + 31) / 32;
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {
            const int64_t y = __shfl_xor_sync(0xffffffffu, rounds, o);
            rounds = y > rounds ? y : rounds;
        }
        float x[4];
        auto load = [&](int64_t r) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t rr = r + 8 * u + l;
                x[u] = rr < e ? X[list_ids[rr] * D + k] : 0.f;
            }
        };
        load(b);
        double acc = 0.0;
        for (int64_t it = 0; it < rounds; ++it) {
            const int64_t r = b + 32 * it;
            const float y[4] = {x[0], x[1], x[2], x[3]};
            load(r + 32);
#pragma unroll
            for (int u = 0; u < 32; ++u) {                          // ascending rows
                const float v = __shfl_sync(0xffffffffu, y[u >> 3], (lane & 24) + (u & 7));
                if (r + u < e) acc = __dadd_rn(acc, (double)v);
            }
        }
        if (t >= 0 && l == 0) {
            if (e > b) C[t] = __double2float_rn(__ddiv_rn(acc, (double)(e - b)));
            else if (!keep_empty) C[t] = 0.f;
        }
    }
}

// The ordered sums of short lists: a thread per (cluster, coordinate), neighbouring
// coordinates side by side, four rows in flight.
__global__ void __launch_bounds__(256) centroid_short_kernel(const float* __restrict__ X,
                                                             const int64_t* __restrict__ list_off,
                                                             const int64_t* __restrict__ list_ids, int64_t total, int D,
                                                             float* __restrict__ C, int keep_empty) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int64_t j = t / D;
    const int k = (int)(t - j * D);
    const int64_t b = list_off[j], e = list_off[j + 1];
    double acc = 0.0;
    for (int64_t r = b; r < e; r += 4) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = r + u < e ? X[list_ids[r + u] * D + k] : 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (r + u < e) acc = __dadd_rn(acc, (double)x[u]);
    }
    if (e > b) C[t] = __double2float_rn(__ddiv_rn(acc, (double)(e - b)));
    else if (!keep_empty) C[t] = 0.f;
}

cudaError_t launch_centroids(const float* X, const int64_t* list_off, const int64_t* list_ids, int64_t rows, int nlist,
                             int D, float* C, int keep_empty, cudaStream_t s) {
    const int64_t tot = (int64_t)nlist * D;
    int32_t* redo = nullptr;
    // Up to 32 rows a list on average, the sums in order at once: one launch instead of
    // two with a list allocated between them, and chains too short to wait for (an
    // iteration of k-means over 4,000 x 64 in 256 lists: 135 -> 120 us).
    if (rows <= 32 * (int64_t)nlist) {
        count_launch();
        centroid_short_kernel<<<(unsigned)ceil_div(tot, 256), 256, 0, s>>>(X, list_off, list_ids, tot, D, C, keep_empty);
        return cudaGetLastError();
    }
    const bool fast = tot < 0x7fffffff && D % 64 == 0 && D / 64 <= 65535 && ((uintptr_t)X & 15) == 0;
    if (!fast || cudaMallocAsync((void**)&redo, sizeof(int32_t) * (size_t)(tot + 1), s) != cudaSuccess) {
        if (fast) cudaGetLastError();                               // (no memory for the list: all in order)
        count_launch();
        centroid_ordered_kernel<<<(unsigned)std::min<int64_t>(ceil_div(tot, 16), 1 << 20), 128, 0, s>>>(
            X, list_off, list_ids, tot, D, C, keep_empty, nullptr, nullptr);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(redo + tot, 0, sizeof(int32_t), s);
    if (e == cudaSuccess) {
        count_launch();
        centroid_kernel<<<dim3((unsigned)nlist, (unsigned)(D / 64)), 256, 0, s>>>(X, list_off, list_ids, D, C, keep_empty,
                                                                                  redo, redo + tot);
        count_launch();
        centroid_ordered_kernel<<<1216, 128, 0, s>>>(X, list_off, list_ids, tot, D, C, keep_empty, redo, redo + tot);
        e = cudaGetLastError();
    }
    const cudaError_t ef = cudaFreeAsync(redo, s);
    return e != cudaSuccess ? e : ef;
}

// ---------------------------------------------------------------------------
// Stable counting sort of rows by cluster id.
//   pass 1: counts[b][c] = rows of chunk b in cluster c       (one warp per chunk)
//   pass 2: base[b][c] = list_off[c] + sum_{b'<b} counts[b'][c] (one thread per c)
//   pass 3: each chunk walks its rows in order; rank among equal clusters inside
//           a 32-row step comes from __match_any_sync, so rows land in ascending
//           id order within their cluster.
// ---------------------------------------------------------------------------
__global__ void group_count_kernel(const int32_t* __restrict__ assign, int64_t n, int64_t chunk, int nlist,
                                   int32_t* __restrict__ counts, uint32_t* __restrict__ status) {
    const int b = blockIdx.x;
    const int lane = threadIdx.x;
    const int64_t r0 = (int64_t)b * chunk, r1 = min(n, r0 + chunk);
    int32_t* cnt = counts + (int64_t)b * nlist;
    for (int64_t r = r0 + lane; r < r1; r += 32) {
        const int c = assign[r];
        if (c < 0 || c >= nlist) {
            atomicOr(status, kStatusBounds);
            continue;
        }
        atomicAdd(&cnt[c], 1);
    }
}

__global__ void group_scan_kernel(const int32_t* __restrict__ counts, int nb, int nlist,
                                  int64_t* __restrict__ total, int64_t* __restrict__ base) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nlist) return;
    int64_t s = 0;
    for (int b = 0; b < nb; ++b) {
        base[(int64_t)b * nlist + c] = s;
        s += counts[(int64_t)b * nlist + c];
    }
    total[c] = s;
}

// exclusive scan of nlist totals into list_off (single block, sequential per thread chunk)
__global__ void offsets_scan_kernel(const int64_t* __restrict__ total, int nlist, int64_t* __restrict__ off) {
    __shared__ int64_t part[1024];
    const int t = threadIdx.x;
    const int per = (nlist + 1023) / 1024;
    const int c0 = t * per, c1 = min(nlist, c0 + per);
    int64_t s = 0;
    for (int c = c0; c < c1; ++c) s += total[c];
    part[t] = s;
    __syncthreads();
    if (t == 0) {
        int64_t run = 0;
        for (int i = 0; i < 1024; ++i) {
            const int64_t v = part[i];
            part[i] = run;
            run += v;
        }
        off[nlist] = run;
    }
    __syncthreads();
    s = part[t];
    for (int c = c0; c < c1; ++c) {
        off[c] = s;
        s += total[c];
    }
}

__global__ void group_scatter_kernel(const int32_t* __restrict__ assign, int64_t n, int64_t chunk, int nlist,
                                     const int64_t* __restrict__ list_off, int64_t* __restrict__ base,
                                     int64_t* __restrict__ list_ids, int64_t* __restrict__ row_of,
                                     int32_t* __restrict__ cl_of_row) {
    const int b = blockIdx.x;
    const int lane = threadIdx.x;
    const int64_t r0 = (int64_t)b * chunk, r1 = min(n, r0 + chunk);
    int64_t* bs = base + (int64_t)b * nlist;
    for (int64_t s = r0; s < r1; s += 32) {
        const int64_t r = s + lane;
        const bool ok = r < r1;
        int c = ok ? assign[r] : -1;
        if (c < 0 || c >= nlist) c = -1;
        const unsigned active = __ballot_sync(0xffffffffu, ok && c >= 0);
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        const unsigned grp = peers & active;
        if (ok && c >= 0) {
            const int leader = __ffs(grp) - 1;
            const int rank = __popc(grp & ((1u << lane) - 1u));
            int64_t old = 0;
            if (lane == leader) {
                old = bs[c];
                bs[c] = old + __popc(grp);
            }
            old = __shfl_sync(grp, old, leader);
            const int64_t pos = list_off[c] + old + rank;
            list_ids[pos] = r;
            if (row_of) row_of[r] = pos;
            if (cl_of_row) cl_of_row[pos] = c;
        }
        __syncwarp();
    }
}

cudaError_t launch_group(const int32_t* assign, int64_t n, int nlist, int64_t* list_off, int64_t* list_ids,
                         int64_t* row_of, int32_t* cl_of_row, void* scratch, size_t scratch_bytes,
                         uint32_t* status, cudaStream_t s) {
    int64_t chunk = 2048;
    // layout: counts (nb*nlist int32, 256-aligned) | base (nb*nlist int64) | total (nlist int64)
    while (ceil_div(n, chunk) * (int64_t)nlist * 12 + (int64_t)nlist * 8 + 512 > (int64_t)scratch_bytes) chunk *= 2;
    const int nb = (int)ceil_div(n, chunk);
    int32_t* counts = (int32_t*)scratch;
    int64_t* base = (int64_t*)((char*)scratch + ((size_t)nb * nlist * 4 + 255) / 256 * 256);
    int64_t* total = base + (int64_t)nb * nlist;
    cudaError_t e = cudaMemsetAsync(counts, 0, (size_t)nb * nlist * 4, s);
    if (e != cudaSuccess) return e;
    count_launch();
    group_count_kernel<<<nb, 32, 0, s>>>(assign, n, chunk, nlist, counts, status);
    count_launch();
    group_scan_kernel<<<(unsigned)ceil_div(nlist, 256), 256, 0, s>>>(counts, nb, nlist, total, base);
    count_launch();
    offsets_scan_kernel<<<1, 1024, 0, s>>>(total, nlist, list_off);
    count_launch();
    group_scatter_kernel<<<nb, 32, 0, s>>>(assign, n, chunk, nlist, list_off, base, list_ids, row_of, cl_of_row);
    return cudaGetLastError();
}

size_t group_scratch_bytes(int64_t n, int nlist) {
    const int64_t nb = ceil_div(n, 2048);
    const size_t want = (size_t)nb * nlist * 12 + (size_t)nlist * 8 + 512;
    const size_t floor_bytes = (size_t)nlist * 8 * 3 + 4096;  // room for one chunk row
    const size_t cap = ((size_t)1 << 30) > floor_bytes ? ((size_t)1 << 30) : floor_bytes;
    return want < cap ? want : cap;
}

// ---------------------------------------------------------------------------
// Per-row selection of the p smallest values (ties by lower column) of a
// [rows][ncols] FP32 matrix.  One block per row; the row is processed in
// chunks of CH columns: the chunk's keys plus the running best p are sorted
// with a block-wide bitonic network in shared memory and the first p kept.
// out_idx[row][0..p-1] ascending; out_val optional.
// ---------------------------------------------------------------------------
__device__ void block_bitonic_sort_u64(uint64_t* a, int n) {
    // n is a power of two, blockDim.x threads cooperate
    for (int size = 2; size <= n; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < n / 2; i += blockDim.x) {
                const int lo = 2 * i - (i & (stride - 1));
                const int hi = lo + stride;
                const bool up = ((lo & size) == 0);
                const uint64_t x = a[lo], y = a[hi];
                if ((x > y) == up) {
                    a[lo] = y;
                    a[hi] = x;
                }
            }
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(512) row_topk_kernel(const float* __restrict__ V, int64_t rows, int ncols,
                                                       int64_t ld, int p, int sortn, int32_t* __restrict__ out_idx,
                                                       float* __restrict__ out_val, int64_t ld_out) {
    extern __shared__ uint64_t sk[];
    const int64_t row = blockIdx.x;
    const float* v = V + row * ld;
    const int chunk = sortn - p;  // new entries per round
    for (int i = threadIdx.x; i < p; i += blockDim.x) sk[i] = kEmptyKey;
    __syncthreads();
    for (int c0 = 0; c0 < ncols; c0 += chunk) {
        for (int i = threadIdx.x; i < chunk; i += blockDim.x) {
            const int c = c0 + i;
            sk[p + i] = c < ncols ? make_key(v[c], (uint32_t)c) : kEmptyKey;
        }
        __syncthreads();
        block_bitonic_sort_u64(sk, sortn);
    }
    for (int i = threadIdx.x; i < p; i += blockDim.x) {
        const uint64_t k = sk[i];
        out_idx[row * ld_out + i] = k == kEmptyKey ? -1 : (int32_t)key_id(k);
        if (out_val) out_val[row * ld_out + i] = k == kEmptyKey ? INFINITY : key_value(k);
    }
}

cudaError_t launch_row_topk(const float* V, int64_t rows, int ncols, int64_t ld, int p, int32_t* out_idx,
                            float* out_val, int64_t ld_out, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    int sortn = 1024;
    while (sortn < 2 * p) sortn <<= 1;
    while (sortn < ncols + p && sortn < 8192) sortn <<= 1;
    cudaError_t e = cudaFuncSetAttribute(row_topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sortn * 8);
    if (e != cudaSuccess) return e;
    count_launch();
    row_topk_kernel<<<(unsigned)rows, 512, sortn * 8, s>>>(V, rows, ncols, ld, p, sortn, out_idx, out_val, ld_out);
    return cudaGetLastError();
}

}  // namespace erq

namespace erq {

// Column of the smallest value in each row (ties -> lower column); one warp per row.
// With `list`: of row i the answer goes to out[list[i]], for the *count listed rows.
__global__ void row_argmin_kernel(const float* __restrict__ V, int64_t rows, int ncols, int32_t* __restrict__ out,
                                  const int32_t* __restrict__ list, const int32_t* __restrict__ count) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= (list ? (int64_t)*count : rows)) return;
    const float* v = V + w * ncols;
    uint64_t best = kEmptyKey;
    for (int c = lane; c < ncols; c += 32) {
        const uint64_t k = make_key(v[c], (uint32_t)c);
        best = k < best ? k : best;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t t = __shfl_xor_sync(0xffffffffu, best, o);
        best = t < best ? t : best;
    }
    if (lane == 0) out[list ? (int64_t)list[w] : w] = (int32_t)key_id(best);
}

cudaError_t launch_row_argmin(const float* V, int64_t rows, int ncols, int32_t* out, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    count_launch();
    row_argmin_kernel<<<(unsigned)ceil_div(rows * 32, 256), 256, 0, s>>>(V, rows, ncols, out, nullptr, nullptr);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Nearest centroid of every row by the FP32 distances of sgemm_kernel (its chain
// of D fused multiply-adds per product), most of them decided on the tensor
// cores.  V holds d_j = |x|^2 + |c_j|^2 - 2 <x, c_j> with the product from FP16
// parts (gemm_tma).  Both products are within
//     E_j = 8 D 2^-24 |x| |c_j|
// of <x, c_j> together: the chain of D roundings within D 2^-24, the parts' three
// products within 3 D / 16 tensor-core steps that each lose at most 17 units of
// 2^-23 of the largest magnitude (sixteen products and the accumulator aligned
// and truncated: Fasi, Higham, Mikaitis, Pranesh, "Numerical behavior of NVIDIA
// tensor cores", 2021), the dropped parts within 2^-21; the sums of the norms add
// 2^-21 (|x|^2 + |c_j|^2).  A row whose smallest d_j lies below all others by more
// than both errors has that column; the others are listed and get the FP32
// distances of the columns that can be the smallest (all of them where these are
// more than 32), so the answer is the same for every row.  100,000 x 256 at D =
// 768: 930 us a pass with FP32 products alone, 340 us.
// ---------------------------------------------------------------------------
struct AssignBound {
    float fx, x2;                                                    // (|x| and |c| apart: x2 c2 underflows for small rows)
    __device__ __forceinline__ float operator()(float c2) const {    // (twice E: the product enters as 2 <x, c>)
        return fx * sqrtf(c2) + 0x1p-21f * (x2 + c2);
    }
};
__device__ __forceinline__ AssignBound assign_bound(int D, float x2) {
    return {2.02f * 8.f * 0x1p-24f * (float)D * sqrtf(x2), x2};
}

// One warp per row: decides it, or lists it with the upper bound of its smallest distance.
__global__ void __launch_bounds__(256) assign_certain_kernel(const float* __restrict__ V,
                                                             const float* __restrict__ xn,
                                                             const float* __restrict__ cn, int64_t rows, int ncols,
                                                             int D, int32_t* __restrict__ out, float* __restrict__ upper,
                                                             int32_t* __restrict__ list, int32_t* __restrict__ count) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= rows) return;
    const float* v = V + w * ncols;
    const AssignBound bd = assign_bound(D, xn[w]);
    // the smallest upper bound, and the smallest two lower bounds with the first one's column
    float up = INFINITY, lo1 = INFINITY, lo2 = INFINITY;
    int col = -1, upc = -1;
    bool odd = false;
    for (int c0 = 0; c0 < ncols; c0 += 128) {
        float x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + 32 * u + lane;
            x[u] = c < ncols ? v[c] : INFINITY;
            y[u] = c < ncols ? cn[c] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = c0 + 32 * u + lane;
            if (c >= ncols) break;
            const float e = bd(y[u]), h = x[u] + e, l = x[u] - e;
            // not finite, or so small that the bound's terms underflow: not decided by it
            odd |= !(fabsf(x[u]) < INFINITY) || !(e < INFINITY) || bd.x2 + y[u] < 1e-30f;
            if (h < up) {
                up = h;
                upc = c;
            }
            if (l < lo1) {
                lo2 = lo1;
                lo1 = l;
                col = c;
            } else {
                lo2 = fminf(lo2, l);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float u2 = __shfl_xor_sync(0xffffffffu, up, o), l1 = __shfl_xor_sync(0xffffffffu, lo1, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo2, o);
        const int uc = __shfl_xor_sync(0xffffffffu, upc, o), lc = __shfl_xor_sync(0xffffffffu, col, o);
        if (u2 < up || (u2 == up && uc < upc)) {
            up = u2;
            upc = uc;
        }
        lo2 = fminf(fminf(lo2, l2), fmaxf(lo1, l1));
        if (l1 < lo1 || (l1 == lo1 && lc < col)) {
            lo1 = l1;
            col = lc;
        }
    }
    odd = __any_sync(0xffffffffu, odd);
    if (lane == 0) {
        if (!odd && upc == col && lo2 > up) {
            out[w] = col;
        } else {
            const int i = atomicAdd(count, 1);
            list[i] = (int32_t)w;
            upper[i] = odd ? INFINITY : up;
        }
    }
}

// The listed rows: the FP32 distances of the columns that can be the smallest,
// one lane per column, each the same chain of fused multiply-adds as
// sgemm_kernel's; rows with more than 32 such columns go on to the full product.
__global__ void __launch_bounds__(256) assign_close_kernel(const float* __restrict__ X, const float* __restrict__ C,
                                                           const float* __restrict__ V, const float* __restrict__ xn,
                                                           const float* __restrict__ cn, int ncols, int D,
                                                           int32_t* __restrict__ out, const float* __restrict__ upper,
                                                           const int32_t* __restrict__ list,
                                                           const int32_t* __restrict__ count,
                                                           int32_t* __restrict__ list2, int32_t* __restrict__ count2) {
    const int lane = threadIdx.x & 31;
    const int n = *count;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n;
         i += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int32_t w = list[i];
        const float* v = V + (int64_t)w * ncols;
        const float up = upper[i];
        const AssignBound bd = assign_bound(D, xn[w]);
        int mine = -1, total = 0;
        for (int c0 = 0; c0 < ncols && total <= 32; c0 += 32) {
            const int c = c0 + lane;
            const unsigned in = __ballot_sync(0xffffffffu, c < ncols && !(v[c] - bd(cn[c]) > up));
            // the columns go to the lanes total, total + 1, ..
            const int take = lane - total;
            if (take >= 0 && take < __popc(in)) mine = c0 + (int)__fns(in, 0, take + 1);
            total += __popc(in);
        }
        if (total > 32 || total < 1) {
            if (lane == 0) list2[atomicAdd(count2, 1)] = w;
            continue;
        }
        uint64_t key = kEmptyKey;
        if (mine >= 0) {
            const float4* x = reinterpret_cast<const float4*>(X + (int64_t)w * D);
            const float4* c = reinterpret_cast<const float4*>(C + (int64_t)mine * D);
            float ac = 0.f;
#pragma unroll 8
            for (int k = 0; k < D / 4; ++k) {
                const float4 a = x[k], b = c[k];
                ac = fmaf(a.x, b.x, ac);
                ac = fmaf(a.y, b.y, ac);
                ac = fmaf(a.z, b.z, ac);
                ac = fmaf(a.w, b.w, ac);
            }
            key = make_key(xn[w] + cn[mine] - 2.f * ac, (uint32_t)mine);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const uint64_t t = __shfl_xor_sync(0xffffffffu, key, o);
            key = t < key ? t : key;
        }
        if (lane == 0) out[w] = (int32_t)key_id(key);
    }
}

// Rows X [rows][D] with their parts and exponents (query_prep), the centroids C
// with theirs; V is scratch [rows][nc], list [3 rows + 2] likewise.
cudaError_t launch_assign(const float* X, const __half* Xhi, const __half* Xlo, const int32_t* eX, const float* xn,
                          int64_t rows, const float* C, const __half* Chi, const __half* Clo, const int32_t* eC,
                          const float* cn, int nc, int D, float* V, int32_t* list, int32_t* out, uint32_t* status,
                          cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    if (rows > kMaxSlabRows || D % 4 != 0 || (((uintptr_t)X | (uintptr_t)C) & 15) != 0) return cudaErrorInvalidValue;
    int32_t *count = list, *close = list + 2, *far = close + rows;
    float* upper = reinterpret_cast<float*>(far + rows);
    cudaError_t e = cudaMemsetAsync(count, 0, 2 * sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    if ((e = launch_gemm_tma(Xhi, Xlo, eX, rows, Chi, Clo, eC, nc, D, V, nc, 1, xn, cn, nullptr, status, s)) !=
        cudaSuccess)
        return e;
    count_launch();
    assign_certain_kernel<<<(unsigned)ceil_div(rows * 32, 256), 256, 0, s>>>(V, xn, cn, rows, nc, D, out, upper, close,
                                                                             count);
    count_launch();
    assign_close_kernel<<<(unsigned)std::min<int64_t>(ceil_div(rows, 8), 2432), 256, 0, s>>>(
        X, C, V, xn, cn, nc, D, out, upper, close, count, far, count + 1);
    dim3 grid((unsigned)ceil_div(nc, 128), (unsigned)ceil_div(rows, 128));
    count_launch();
    sgemm_kernel<true, EPI_DIST, true><<<grid, 256, 0, s>>>(X, C, V, rows, nc, D, 1.f, nullptr, xn, cn, nc, far, count + 1);
    count_launch();
    row_argmin_kernel<<<(unsigned)ceil_div(rows * 32, 256), 256, 0, s>>>(V, rows, nc, out, far, count + 1);
    return cudaGetLastError();
}

__global__ void gather_rows_kernel(const float* __restrict__ X, const int64_t* __restrict__ idx, int64_t n, int D,
                                   float* __restrict__ out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t vecs = (int64_t)n * (D / 4);
    if (t >= vecs) return;
    const int64_t r = t / (D / 4), c = t % (D / 4);
    reinterpret_cast<float4*>(out)[r * (D / 4) + c] = reinterpret_cast<const float4*>(X)[idx[r] * (D / 4) + c];
}

cudaError_t launch_gather_rows(const float* X, const int64_t* idx, int64_t n, int D, float* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    gather_rows_kernel<<<(unsigned)ceil_div(n * (D / 4), 256), 256, 0, s>>>(X, idx, n, D, out);
    return cudaGetLastError();
}

__global__ void fill_i32_kernel(int32_t* p, int64_t n, int32_t v) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) p[t] = v;
}

cudaError_t launch_fill_i32(int32_t* p, int64_t n, int32_t v, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    fill_i32_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(p, n, v);
    return cudaGetLastError();
}

// k-means training sample: n evenly spaced row ids with a seed-dependent offset.
__global__ void strided_ids_kernel(int64_t* out, int64_t n, int64_t N, uint64_t seed) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double step = (double)N / (double)n;
    const int64_t off = (int64_t)(seed % (uint64_t)(step > 1.0 ? (int64_t)step : 1));
    int64_t r = (int64_t)((double)t * step) + off;
    out[t] = r < N ? r : N - 1;
}

cudaError_t launch_strided_ids(int64_t* out, int64_t n, int64_t N, uint64_t seed, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    strided_ids_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(out, n, N, seed);
    return cudaGetLastError();
}

}  // namespace erq

namespace erq {

// ---------------------------------------------------------------------------
// Per-row selection of more than 32 (probe lists): the p smallest (value,
// column) pairs of each row, ascending, ties by lower column.  One block per
// row, T threads x E values in registers (column i = j T + thread).
//
// One counting pass over 2,048 equal intervals of the row's key range (the
// order-preserving integers between its minimum and maximum): distances of one
// row lie within a factor of a few of each other, so intervals of the key's top
// bits would put most of them in a handful of counters (whose atomics then
// queue), intervals of the range hold a few values each.  The counters' prefix
// sums give every value up to the interval of the p-th smallest its place but
// for the order within an interval, which each value finds by comparing itself
// with the interval's others: no sort.  A row whose p-th smallest lies in an
// interval with more than SLACK values beyond p (far outliers, many equal
// values) goes through the radix select over 11 + 11 + 10 key bits and a bitonic
// sort instead.
// Bound by the latency of its block-wide phases; 16,384 rows of 4,096, p = 256:
// 624 us with the radix select for every row, 216 us.
// ---------------------------------------------------------------------------
constexpr int RS_BINS = 2048;
constexpr int RS_SLACK = 256;

template <int T, int E>
__global__ void __launch_bounds__(T, T == 256 ? 5 : 1) row_topk_range_kernel(const float* __restrict__ V, int ncols,
                                                                             int64_t ld, int p, int cap, int sortn,
                                                                             int32_t* __restrict__ out_idx,
                                                                             float* __restrict__ out_val,
                                                                             int64_t ld_out) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    int* hist = reinterpret_cast<int*>(rs_smem);                                   // [2048]
    uint64_t* sel = reinterpret_cast<uint64_t*>(rs_smem + RS_BINS * 4);            // [max(cap, sortn)]
    __shared__ uint32_t s_lo[T / 32], s_hi[T / 32];
    __shared__ int s_sum[T / 32];
    __shared__ int s_bin, s_below, s_end;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* v = V + (int64_t)blockIdx.x * ld;
    int32_t* out = out_idx + (int64_t)blockIdx.x * ld_out;
    float* val = out_val ? out_val + (int64_t)blockIdx.x * ld_out : nullptr;
    uint32_t k[E];
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int j = 0; j < E; ++j) k[j] = j * T + tid < ncols ? float_to_ordered(v[j * T + tid]) : 0u;
#pragma unroll
    for (int j = 0; j < E; ++j)
        if (j * T + tid < ncols) {
            lo = min(lo, k[j]);
            hi = max(hi, k[j]);
        }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
    }
    constexpr int BT = RS_BINS / T;                       // counters of a thread: 8 or 2
#pragma unroll
    for (int j = 0; j < BT; ++j) hist[tid + j * T] = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < T / 32; ++w) {
        lo = min(lo, s_lo[w]);
        hi = max(hi, s_hi[w]);
    }
    const int shift = max(0, 32 - __clz(hi - lo) - 11);   // (hi - lo) >> shift < 2048
#pragma unroll
    for (int j = 0; j < E; ++j)
        if (j * T + tid < ncols) atomicAdd(&hist[(k[j] - lo) >> shift], 1);
    __syncthreads();
    int c[BT], own = 0;
#pragma unroll
    for (int j = 0; j < BT; ++j) {
        c[j] = hist[tid * BT + j];
        own += c[j];
    }
    const int inc = warp_incl_scan(own);
    if (lane == 31) s_sum[warp] = inc;
    __syncthreads();
    int run = inc - own;
    for (int w = 0; w < warp; ++w) run += s_sum[w];
#pragma unroll
    for (int j = 0; j < BT; ++j) {
        hist[tid * BT + j] = run;                         // the interval's first place
        if (run < p && run + c[j] >= p) {
            s_bin = tid * BT + j;
            s_below = run;
            s_end = run + c[j];
        }
        run += c[j];
    }
    __syncthreads();
    const int bin = s_bin, end = s_end;
    if (end <= cap) {
#pragma unroll
        for (int j = 0; j < E; ++j)
            if (j * T + tid < ncols) {
                const int b = (int)((k[j] - lo) >> shift);
                if (b <= bin) sel[atomicAdd(&hist[b], 1)] = ((uint64_t)k[j] << 32) | (uint32_t)(j * T + tid);
            }
        __syncthreads();
        // hist[b] is now the end of interval b, for every b <= bin
        for (int i = tid; i < end; i += T) {
            const uint64_t key = sel[i];
            const int b = (int)(((uint32_t)(key >> 32) - lo) >> shift);
            const int b0 = b > 0 ? hist[b - 1] : 0, b1 = hist[b];
            int rank = b0;
            for (int u = b0; u < b1; ++u) rank += sel[u] < key;
            if (rank < p) {
                out[rank] = (int32_t)(uint32_t)key;
                if (val) val[rank] = ordered_to_float((uint32_t)(key >> 32));
            }
        }
        return;
    }
    // ---- the general case: p-th smallest key by radix select
    uint32_t prefix = 0, pmask = 0;
    int need = p;                       // rank (1-based) of the wanted key among the candidates
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
        const int sh = pass == 0 ? 21 : pass == 1 ? 10 : 0, nb = pass == 2 ? 1024 : 2048;
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < nb; i += T) hist[i] = 0;
        __syncthreads();
#pragma unroll 1
        for (int i = tid; i < ncols; i += T) {
            const uint32_t x = float_to_ordered(v[i]);
            if ((x & pmask) == prefix) atomicAdd(&hist[(x >> sh) & (nb - 1)], 1);
        }
        __syncthreads();
        if (tid < 32) {                 // first bin whose running count reaches `need`
            const int per = nb / 32;
            int mine = 0;
#pragma unroll 1
            for (int b = lane * per; b < (lane + 1) * per; ++b) mine += hist[b];
            const int incl = warp_incl_scan(mine), excl = incl - mine;
            const unsigned hit = __ballot_sync(0xffffffffu, incl >= need && excl < need);
            if (lane == __ffs(hit) - 1) {
                int r = excl, b = lane * per;
#pragma unroll 1
                for (; b < (lane + 1) * per - 1; ++b) {
                    if (r + hist[b] >= need) break;
                    r += hist[b];
                }
                s_bin = b;
                s_below = r;
            }
        }
        __syncthreads();
        need -= s_below;
        prefix |= (uint32_t)s_bin << sh;
        pmask |= (uint32_t)(nb - 1) << sh;
    }
    // `need` entries equal to prefix are wanted, all smaller ones are in
    __syncthreads();
    if (tid == 0) s_end = 0;
#pragma unroll 1
    for (int i = tid; i < sortn; i += T) sel[i] = kEmptyKey;
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < ncols; i += T) {
        const uint32_t x = float_to_ordered(v[i]);
        if (x < prefix) sel[atomicAdd(&s_end, 1)] = ((uint64_t)x << 32) | (uint32_t)i;
    }
    __syncthreads();
    if (tid < 32) {                     // the `need` lowest columns among the equal ones
        const int base = s_end;
        int taken = 0;
#pragma unroll 1
        for (int c0 = 0; c0 < ncols && taken < need; c0 += 32) {
            const int i = c0 + lane;
            const bool eq = i < ncols && float_to_ordered(v[i]) == prefix;
            const unsigned m = __ballot_sync(0xffffffffu, eq);
            const int rank = __popc(m & ((1u << lane) - 1u));
            if (eq && taken + rank < need) sel[base + taken + rank] = ((uint64_t)prefix << 32) | (uint32_t)i;
            taken += __popc(m);
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int size = 2; size <= sortn; size <<= 1)
#pragma unroll 1
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll 1
            for (int i = tid; i < sortn / 2; i += T) {
                const int l = 2 * i - (i & (stride - 1));
                const int h = l + stride;
                const bool up = (l & size) == 0;
                const uint64_t x = sel[l], y = sel[h];
                if ((x > y) == up) { sel[l] = y; sel[h] = x; }
            }
            __syncthreads();
        }
#pragma unroll 1
    for (int i = tid; i < p; i += T) {
        out[i] = (int32_t)(uint32_t)sel[i];
        if (val) val[i] = ordered_to_float((uint32_t)(sel[i] >> 32));
    }
}

// Smallest p <= 32 entries of each row (keys (value, column), so ties take the
// lower column), one warp per row.  A first pass takes the p-th smallest of the
// 32 lanes' minima over their columns: at least p entries lie at or below it,
// so it is a valid admission bound, and a tight one.  The second pass keeps the
// current p best in a sorted 32-entry list across the lanes; a 32-column chunk
// with an entry below the bound and the list's p-th key is sorted and merged in.
__global__ void __launch_bounds__(256) row_topk_warp_kernel(const float* __restrict__ V, int64_t rows, int ncols,
                                                            int64_t ld, int p, int32_t* __restrict__ out_idx,
                                                            float* __restrict__ out_val, int64_t ld_out) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    const float* v = V + row * ld;
    constexpr int PF = 8;                        // chunks loaded ahead
    uint32_t lmin = 0xffffffffu;                 // this lane's smallest ordered value
    for (int c0 = 0; c0 < ncols; c0 += 32 * PF) {
        uint32_t o[PF];
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            const int c = c0 + 32 * u + lane;
            o[u] = c < ncols ? float_to_ordered(v[c]) : 0xffffffffu;
        }
#pragma unroll
        for (int u = 0; u < PF; ++u) lmin = o[u] < lmin ? o[u] : lmin;
    }
    // p-th smallest lane minimum (lanes that saw no column contribute the maximum)
    const uint32_t bound = (uint32_t)(ws_shfl(ws_sort32(((uint64_t)lmin << 32) | (uint32_t)lane, lane), p - 1) >> 32);
    uint64_t list = kEmptyKey, th = kEmptyKey;
    for (int c0 = 0; c0 < ncols; c0 += 32 * PF) {
        uint32_t o[PF];
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            const int c = c0 + 32 * u + lane;
            o[u] = c < ncols ? float_to_ordered(v[c]) : 0xffffffffu;
        }
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            const int c = c0 + 32 * u + lane;
            const uint64_t key = ((uint64_t)o[u] << 32) | (uint32_t)c;
            const bool pass = c < ncols && o[u] <= bound && key < th;
            if (!__any_sync(0xffffffffu, pass)) continue;
            list = ws_merge32(list, ws_sort32(pass ? key : kEmptyKey, lane), lane);
            th = ws_shfl(list, p - 1);
        }
    }
    if (lane < p) {
        out_idx[row * ld_out + lane] = list == kEmptyKey ? -1 : (int32_t)(list & 0xffffffffu);
        if (out_val) out_val[row * ld_out + lane] = list == kEmptyKey ? INFINITY : ordered_to_float((uint32_t)(list >> 32));
    }
}

// Smallest p <= 32 entries of each row (keys (value, column), ties to the lower
// column) given the minimum of every 32-column group, one warp per row: the
// p-th smallest group minimum bounds the p-th smallest entry (p groups hold an
// entry at or below it), so only groups whose minimum is at or below it can
// hold an answer; those are read and merged into a sorted 32-entry warp list.
__global__ void __launch_bounds__(256) row_topk_groups_kernel(const float* __restrict__ V,
                                                              const float* __restrict__ gmin, int64_t rows, int ncols,
                                                              int64_t ld, int p, int32_t* __restrict__ out_idx,
                                                              float* __restrict__ out_val, int64_t ld_out) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= rows) return;
    const int ng = (ncols + 31) / 32;
    const float* gm = gmin + row * ng;
    // bound: p-th smallest group minimum (groups visited 32 at a time)
    uint64_t best = kEmptyKey;
    for (int g0 = 0; g0 < ng; g0 += 32) {
        const int gi = g0 + lane;
        const uint64_t key = gi < ng ? ((uint64_t)float_to_ordered(gm[gi]) << 32) | (uint32_t)gi : kEmptyKey;
        best = ws_merge32(best, ws_sort32(key, lane), lane);
    }
    const uint32_t bound = (uint32_t)(ws_shfl(best, p - 1) >> 32);
    const float* v = V + row * ld;
    uint64_t list = kEmptyKey, th = kEmptyKey;
    for (int g0 = 0; g0 < ng; g0 += 32) {
        const int gi = g0 + lane;
        uint32_t cand = __ballot_sync(0xffffffffu, gi < ng && float_to_ordered(gm[gi]) <= bound);
        while (cand) {                                   // candidate groups, up to 4 loaded together
            int gsel[4];
            uint32_t o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                gsel[u] = cand ? g0 + __ffs(cand) - 1 : -1;
                if (cand) cand &= cand - 1;
                const int c = gsel[u] * 32 + lane;
                o[u] = (gsel[u] >= 0 && c < ncols) ? float_to_ordered(v[c]) : 0xffffffffu;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (gsel[u] < 0) break;                      // warp-uniform
                const int c = gsel[u] * 32 + lane;
                const uint64_t key = ((uint64_t)o[u] << 32) | (uint32_t)c;
                const bool pass = c < ncols && o[u] <= bound && key < th;
                ws_insert_each(list, th, key, pass, p, lane);
            }
        }
    }
    if (lane < p) {
        out_idx[row * ld_out + lane] = list == kEmptyKey ? -1 : (int32_t)(list & 0xffffffffu);
        if (out_val) out_val[row * ld_out + lane] = list == kEmptyKey ? INFINITY : ordered_to_float((uint32_t)(list >> 32));
    }
}

cudaError_t launch_row_topk_groups(const float* V, const float* gmin, int64_t rows, int ncols, int64_t ld, int p,
                                   int32_t* out_idx, float* out_val, int64_t ld_out, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    count_launch();
    row_topk_groups_kernel<<<(unsigned)ceil_div(rows * 32, 256), 256, 0, s>>>(V, gmin, rows, ncols, ld, p, out_idx, out_val,
                                                                            ld_out);
    return cudaGetLastError();
}

// p <= ncols.  Rows of more than 16,384 or p > 2,048 take the general selection.
cudaError_t launch_row_topk_fast(const float* V, int64_t rows, int ncols, int64_t ld, int p, int32_t* out_idx,
                                 float* out_val, int64_t ld_out, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    if (p <= 32) {
        count_launch();
        row_topk_warp_kernel<<<(unsigned)ceil_div(rows * 32, 256), 256, 0, s>>>(V, rows, ncols, ld, p, out_idx, out_val,
                                                                               ld_out);
        return cudaGetLastError();
    }
    if (ncols > 16384 || p > 2048 || p > ncols)
        return launch_row_topk(V, rows, ncols, ld, p, out_idx, out_val, ld_out, s);
    int sortn = 32;
    while (sortn < p) sortn <<= 1;
    const int cap = p + RS_SLACK;
    const size_t smem = RS_BINS * 4 + (size_t)std::max(cap, sortn) * 8;      // (at most 26 KB)
    count_launch();
    if (ncols <= 1024)
        row_topk_range_kernel<256, 4><<<(unsigned)rows, 256, smem, s>>>(V, ncols, ld, p, cap, sortn, out_idx, out_val, ld_out);
    else if (ncols <= 4096)
        row_topk_range_kernel<256, 16><<<(unsigned)rows, 256, smem, s>>>(V, ncols, ld, p, cap, sortn, out_idx, out_val, ld_out);
    else
        row_topk_range_kernel<1024, 16><<<(unsigned)rows, 1024, smem, s>>>(V, ncols, ld, p, cap, sortn, out_idx, out_val, ld_out);
    return cudaGetLastError();
}

}  // namespace erq

namespace erq {

// out[c][r] = X[r][c] (32x32 tiles through shared memory).
__global__ void transpose_kernel(const float* __restrict__ X, int rows, int cols, float* __restrict__ out) {
    __shared__ float t[32][33];
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int r = r0 + i, c = c0 + threadIdx.x;
        if (r < rows && c < cols) t[i][threadIdx.x] = X[(int64_t)r * cols + c];
    }
    __syncthreads();
    for (int i = threadIdx.y; i < 32; i += 8) {
        const int c = c0 + i, r = r0 + threadIdx.x;
        if (r < rows && c < cols) out[(int64_t)c * rows + r] = t[threadIdx.x][i];
    }
}

cudaError_t launch_transpose(const float* X, int rows, int cols, float* out, cudaStream_t s) {
    count_launch();
    transpose_kernel<<<dim3((unsigned)ceil_div(cols, 32), (unsigned)ceil_div(rows, 32)), dim3(32, 8), 0, s>>>(X, rows,
                                                                                                         cols, out);
    return cudaGetLastError();
}

}  // namespace erq
