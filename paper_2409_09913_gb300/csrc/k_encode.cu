// Encoder: Algorithm 1 (Quantize) of Section 3.1, one warp per vector.
//
// The algorithm walks the rescaling factor t upward through the critical
// values at which the rounding of t*o' changes, keeps <y_cur, o'> and
// ||y_cur||^2 up to date in O(1) per step and records the state of largest
// cosine <y_cur/||y_cur||, o'>.  With |y_i| = m_i + 1/2 the critical values of
// coordinate i are t = (m+1)/|o'_i|, m = 0 .. 2^(B-1)-2.
//
// GPU formulation (bit-identical to a sequential FP64 walk with a min-heap).
// The state at a given t needs no walk: m_i = min(floor(t |o'_i|), 2^(B-1)-1).
// So the walk is bounded first and only the events that can hold its maximum
// are put in order:
//  * Bounds.  An event at t adds |o'_i| to S = <y, o'> and 8 t |o'_i| to
//    N = 4 ||y||^2.  For states between E0 (at t0) and E1, N >= N0 + 8 t0
//    (S - S0); S^2 over a line is quasi-convex, so 4 S^2 / N <= max(v0^2,
//    4 S1^2 / (N0 + 8 t0 (S1 - S0))).  A range whose bound is below the cosine
//    of some known state cannot hold the maximum (the walk's maximum is the
//    maximum over all grid points, so any grid point is a lower bound).
//    Level 1 evaluates 32 values of t at once (lane = t, the row broadcast from
//    shared memory); the following levels drop the events of the remaining
//    range into NBK buckets (sums by shared-memory atomics) and prefix-sum
//    them.  Sums are fixed-point with a known error, which is added to every
//    bound.  About 20 events a coordinate pass through the buckets instead of
//    through a sort, whatever B.
//  * Jump.  The FP64 running sum at the range's start is the exact sum wherever
//    no FP64 addition on the way rounds (below), formed in parallel; otherwise
//    the way is shortened until the events that do round fit a window, which is
//    walked (about once per binade that the sum crosses).
//  * Windows of at most W events of the remaining range, sorted by (FP32 key
//    RN((m+1)/|o'_i|), i) with a warp bitonic network; every run of equal FP32
//    keys is then re-sorted (one lane per run) by the exact rational
//    comparison (m+1)*|o'_j| vs (m'+1)*|o'_i| (exact FP64 products).  Ties of
//    the exact value go to the lower coordinate.  A single key value with more
//    than W events is sorted by that comparison alone, as 16-bit coordinates.
//  * <y_cur, o'> is the FP64 sum of the |o'_i| in that order.  When the running
//    sum and all of a range's addends are multiples of 2^g and the range's final
//    sum is below 2^(53+g), no addition of the range rounds: its partial sums
//    are the exact int64 prefix sums in units of 2^g, formed in parallel.
//    Windows that fail the test are walked serially in FP64 by one lane,
//    rounding at every step.  ||y_cur||^2 is an exact integer multiple of 1/4.
//  * All lanes bound each state's cosine in FP32 and only states within 4e-6
//    of the window's best are re-evaluated with correctly rounded FP64 sqrt and
//    division; the first state of strictly largest cosine wins.
//  * The recorded event (i*, m*) defines the final state: m_i = number of
//    events of coordinate i that precede or equal (i*, m*) in the exact order.
//  * sum |o'_i| and ||o'||^2 are sequential FP64 sums by definition.  The first
//    is formed in parallel where the test above shows it exact; the
//    second in parallel FP64, and serially only when the difference (at most
//    D 2^-53 relative) could change the FP32 factors derived from it.
#include <cuda_runtime.h>
#include <stdint.h>

#include "erq_kernels.cuh"

namespace erq {

namespace {

// event word: the FP32 key in the high half, then the coordinate i (22 bits)
// and the level m (10 bits: m <= 2^(B-1) - 2 = 510 at B = 10)
constexpr int EV_MBITS = 10;
constexpr uint64_t EV_MMASK = (1u << EV_MBITS) - 1, EV_IMASK = (1u << (32 - EV_MBITS)) - 1;
__device__ __forceinline__ int ev_i(uint64_t x) { return (int)((x >> EV_MBITS) & EV_IMASK); }
__device__ __forceinline__ int ev_m(uint64_t x) { return (int)(x & EV_MMASK); }

constexpr int ENC_W = 512;       // events of a sorted window
constexpr int NBK = 512;         // buckets of a bounding level

// Exponent of the lowest set bit of a positive FP32 / FP64 value.
__device__ __forceinline__ int low_exp(float a) {
    const uint32_t b = __float_as_uint(a), e = (b >> 23) & 0xffu;
    const uint32_t mant = e == 0 ? (b & 0x7fffffu) : ((b & 0x7fffffu) | 0x800000u);
    return (e == 0 ? -149 : (int)e - 150) + __ffs(mant) - 1;
}
__device__ __forceinline__ int low_exp(double a) {
    const uint64_t b = (uint64_t)__double_as_longlong(a), e = (b >> 52) & 0x7ffu;
    const uint64_t mant = (b & 0xfffffffffffffull) | 0x10000000000000ull;   // (the sums are normal numbers)
    return (int)e - 1075 + __ffsll((long long)mant) - 1;
}
// A positive FP32 value as an integer multiple of 2^g (g <= low_exp(a), and the
// result below 2^62 by the caller's range check).
__device__ __forceinline__ int64_t units_of(float a, int g) {
    const uint32_t b = __float_as_uint(a), e = (b >> 23) & 0xffu;
    const uint64_t mant = e == 0 ? (b & 0x7fffffu) : ((b & 0x7fffffu) | 0x800000u);
    const int sh = (e == 0 ? -149 : (int)e - 150) - g;
    return (int64_t)(sh >= 0 ? mant << sh : mant >> -sh);
}
__device__ __forceinline__ int64_t warp_excl_scan_i64(int64_t v, int64_t& total) {
    const int lane = threadIdx.x & 31;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    total = __shfl_sync(0xffffffffu, x, 31);
    return x - v;
}
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max_f64(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// The row is held scaled by a power of two so that its largest magnitude lies
// in [1, 2); the k-th event (0-based) of a coordinate has key RN((k+1) / a),
// a correctly rounded division, so keys are a monotone function of the exact
// critical value t = (k+1)/a.
__device__ __forceinline__ float ev_key(int k, float a) { return __fdiv_rn((float)(k + 1), a); }

// Number of events of a coordinate with key <= T (a > 0), in [0, M]: floor(T a)
// unless the product is so near an integer that the rounding of T a (2^-24) or
// of the key (2^-24) could decide, which the keys themselves then do.
__device__ __forceinline__ int events_upto(float T, float a, int M) {
    if (!(a > 0.f)) return 0;
    const float x = __fmul_rn(T, a);                 // (T = inf: inf)
    if (x > 1.001f * (float)M + 1.f) return M;
    const float fl = floorf(x), d = x - fl, eps = x * 0x1p-20f;
    int j = min(M, (int)fl);
    if (d > eps && d < 1.f - eps) return j;
    while (j < M && ev_key(j, a) <= T) ++j;
    while (j > 0 && ev_key(j - 1, a) > T) --j;
    return j;
}

// Exact order of events: true if (ia, ma) precedes (ib, mb).
__device__ __forceinline__ bool ev_before(const float* a, int ia, int ma, int ib, int mb) {
    const double lhs = (double)(ma + 1) * (double)a[ib];
    const double rhs = (double)(mb + 1) * (double)a[ia];
    if (lhs != rhs) return lhs < rhs;
    return ia < ib;
}

// Events of the whole row with key <= T.
__device__ int count_upto(const float* a, int D, int M, float T) {
    int c = 0;
    for (int i = threadIdx.x & 31; i < D; i += 32) c += events_upto(T, a[i], M);
    return warp_sum_int(c);
}

// Bucket of a key of the range (Tlo, ...]; monotone in the key.
__device__ __forceinline__ int bucket_of(float key, float Tlo, float scale) {
    return min(NBK - 1, (int)((key - Tlo) * scale));
}

// The range (Tlo, Thi] of keys that can hold the walk's maximum (every event
// outside it ends in a state of smaller cosine).  a: the scaled row; sum_a its
// sum up to FP64 rounding; amin the smallest non-zero magnitude; buf: 4 NBK words.
__device__ void find_range(const float* a, int D, int M, double sum_a, float amin, float amax, uint32_t* buf, float& Tlo_out,
                           float& Thi_out) {
    const int lane = threadIdx.x & 31;
    const double dD = (double)D;
    double best2 = sum_a * sum_a / dD * (1.0 - 1e-12);           // 4 S^2 / N of the initial state
    // ---- level 1: 32 values of t.  The state at U is taken with floor(U a), so a
    // visited state whose last key lies in (U_{j-1} (1 + 2^-21), U_{j+1} (1 -
    // 2^-21)] lies between the states j-1 and j+1; those pairs overlap and cover
    // the range.  The first pass puts 24 values where rows of Gaussian-like
    // coordinates have their maximum (t max|a| within 0.25 .. 2.5 of M) and the
    // rest towards the ends; later passes are geometric over what remains.
    float U0 = 0.5f;                                              // below the first event (a < 2)
    float U1 = fminf(1.001f * (float)M / amin, 1e38f);            // past the last one
    float Tlo = U0, Thi = U1;
    const double e1 = dD * (double)(M + 1) * 0x1p-22;             // error of S: 2^-23 a unit, doubled
    const float mid0 = fminf(fmaxf(0.25f * (float)M / amax, U0), U1), mid1 = fminf(10.f * mid0, U1);
    for (int pass = 0; pass < 3; ++pass) {
        const float ratio = U1 / U0;
        float U;
        if (pass > 0) U = U0 * exp2f((float)lane * (1.f / 31.f) * log2f(ratio));
        else if (lane < 4) U = U0 * exp2f((float)lane * 0.25f * log2f(mid0 / U0));
        else if (lane < 28) U = mid0 * exp2f((float)(lane - 4) * (1.f / 23.f) * log2f(mid1 / mid0));
        else U = mid1 * exp2f((float)(lane - 27) * 0.25f * log2f(U1 / mid1));
        U = lane == 0 ? U0 : (lane == 31 ? U1 : fminf(fmaxf(U, U0), U1));
        const float top = 8388608.f + (float)M;
        uint64_t Sa = 0;
        uint32_t Na = 0;
        for (int i = 0; i < D; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(a + i);
            const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t c = __float_as_uint(fminf(__fmaf_rd(U, x[q], 8388608.f), top)) & 0x7fffffu;
                const uint32_t f = __float_as_uint(x[q] + 2.f) - 0x40000000u; // a in units of 2^-22
                Sa += (uint64_t)f * c;
                Na += c * (c + 1u);
            }
        }
        const double S = (double)Sa * 0x1p-22 + 0.5 * sum_a;
        const double N = dD + 4.0 * (double)Na;
        const double v2 = 4.0 * S * S / N, rel = 2.0 * e1 / S;
        best2 = fmax(best2, warp_max_f64(v2 * (1.0 - rel - 1e-9)));
        const double Sp = __shfl_down_sync(0xffffffffu, S, 1);
        const double Sm = __shfl_up_sync(0xffffffffu, S, 1), Nm = __shfl_up_sync(0xffffffffu, N, 1);
        const double vm = __shfl_up_sync(0xffffffffu, v2 * (1.0 + rel), 1);
        const double tm = (double)__shfl_up_sync(0xffffffffu, U, 1) * (1.0 - 0x1p-20);
        const double den = Nm + 8.0 * tm * fmax(0.0, Sp - Sm - 2.0 * e1);
        const bool keep = lane >= 1 && lane <= 30 &&
                          (4.0 * (Sp + e1) * (Sp + e1) * (1.0 + 1e-9) >= best2 * den || vm >= best2);
        const uint32_t mask = __ballot_sync(0xffffffffu, keep);
        if (mask == 0u) break;                                    // (cannot happen: the best state is covered)
        const int jmin = __ffs(mask) - 1, jmax = 31 - __clz(mask);
        Tlo = jmin == 1 ? U0 : __shfl_sync(0xffffffffu, U, jmin) * (1.f - 0x1p-19f);
        Thi = jmax == 30 ? U1 : __shfl_sync(0xffffffffu, U, jmax) * (1.f + 0x1p-19f);
        U0 = Tlo * (1.f - 0x1p-18f);
        U1 = fminf(Thi * (1.f + 0x1p-18f), 1e38f);
        if (U1 < 6.f * U0 || U1 > 0.6f * ratio * U0) break;       // narrow enough, or no longer shrinking
    }
    // ---- bucket levels
    const double e2 = dD * (double)(M + 1) * 0x1p-30;             // error of S: 2^-31 a unit, doubled
    // (at most 4096 * 511 < 2^21 events: 11-bit parts of a never overflow a word)
    uint32_t* b_n = buf + 3 * NBK;
    auto bucket_sum = [&](int b) {
        return (int64_t)buf[b] + ((int64_t)buf[NBK + b] << 11) + ((int64_t)buf[2 * NBK + b] << 22);
    };
    int prev = 0x7fffffff;
    for (int level = 0; level < 8; ++level) {
        int64_t S0 = 0;
        uint32_t N0 = 0;
        int ev = 0;
        for (int i = lane; i < D; i += 32) {
            const float x = a[i];
            const uint32_t c = (uint32_t)events_upto(Tlo, x, M);
            ev += events_upto(Thi, x, M) - (int)c;
            S0 += (int64_t)((uint64_t)__float2uint_rn(x * 0x1p30f) * c);
            N0 += c * (c + 1u);
        }
        ev = warp_sum_int(ev);
        if (ev <= ENC_W || ev > prev - (prev >> 2)) break;
        prev = ev;
        const float width = Thi - Tlo;
        const float scale = __fdividef((float)NBK, width) * (1.f - 0x1p-18f);
        if (!(scale > 0.f) || !(scale < 1e30f)) break;
        S0 = warp_sum_i64(S0);
        N0 = (uint32_t)warp_sum_int((int)N0);
        __syncwarp();
        for (int i = lane; i < 4 * NBK; i += 32) buf[i] = 0u;
        __syncwarp();
        auto drop = [&](int k, float x, uint32_t f) {              // event k of a coordinate (f: x in units of 2^-30)
            const int b = bucket_of(ev_key(k, x), Tlo, scale);
            atomicAdd(buf + b, f & 0x7ffu);
            atomicAdd(buf + NBK + b, (f >> 11) & 0x7ffu);
            atomicAdd(buf + 2 * NBK + b, f >> 22);
            atomicAdd(b_n + b, (uint32_t)(k + 1));
        };
        for (int i0 = 0; i0 < D; i0 += 32) {
            const float x = a[i0 + lane];
            const uint32_t f = __float2uint_rn(x * 0x1p30f);
            const int k0 = events_upto(Tlo, x, M), k1 = events_upto(Thi, x, M);
            if (ev >= 12 * D) {                                    // many events a coordinate: the warp takes one at a time
                for (int src = 0; src < 32; ++src) {
                    const int ka = __shfl_sync(0xffffffffu, k0, src), kb = __shfl_sync(0xffffffffu, k1, src);
                    const float xs = __shfl_sync(0xffffffffu, x, src);
                    const uint32_t fs = __shfl_sync(0xffffffffu, f, src);
                    for (int k = ka + lane; k < kb; k += 32) drop(k, xs, fs);
                }
            } else {
                for (int k = k0; k < k1; ++k) drop(k, x, f);
            }
        }
        __syncwarp();
        constexpr int PER = NBK / 32;
        int64_t sl = 0;
        uint32_t nl = 0;
        for (int b = lane * PER; b < (lane + 1) * PER; ++b) {
            sl += bucket_sum(b);
            nl += b_n[b];
        }
        int64_t tot;
        const int64_t sb = S0 + warp_excl_scan_i64(sl, tot);
        const uint32_t nb = (uint32_t)(warp_incl_scan((int)nl) - (int)nl);
        // prefix sums (after each bucket) back to shared memory: S in 64 bits, N in 32
        uint64_t ps[PER];
        {
            int64_t s = sb;
            uint32_t nn = nb;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                s += bucket_sum(lane * PER + j);
                ps[j] = (uint64_t)s;
            }
            __syncwarp();
            uint64_t* P = reinterpret_cast<uint64_t*>(buf);
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int b = lane * PER + j;
                nn += b_n[b];
                P[b] = ps[j];
                buf[2 * NBK + b] = nn;
            }
            __syncwarp();
        }
        const uint64_t* P = reinterpret_cast<const uint64_t*>(buf);
        const uint32_t* Q = buf + 2 * NBK;                         // (b_n keeps the buckets' own sums)
        const double hs = 0.5 * sum_a, Nb = dD + 4.0 * (double)N0;
        const float hsf = (float)hs, Nbf = (float)Nb;
        // FP32 cosines (within 1e-6) choose the buckets worth the FP64 test
        float v2f[PER], mf = (float)best2;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int b = lane + 32 * j;
            const float S = (float)P[b] * 0x1p-30f + hsf;
            v2f[j] = __fdividef(4.f * S * S, Nbf + 8.f * (float)Q[b]);
            mf = fmaxf(mf, v2f[j]);
        }
        mf = warp_max(mf) * (1.f - 1e-5f);
        double m2 = 0.0;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (!__any_sync(0xffffffffu, v2f[j] >= mf)) continue;
            const int b = lane + 32 * j;
            const double S = (double)P[b] * 0x1p-30 + hs - e2;
            m2 = fmax(m2, 4.0 * S * S / (Nb + 8.0 * (double)Q[b]));
        }
        best2 = fmax(best2, warp_max_f64(m2) * (1.0 - 1e-12));
        int bmin = NBK, bmax = -1;
        const double iscale = 1.0 / (double)scale;
        const float b2f = (float)best2 * (1.f - 1e-5f), tlof = Tlo * (1.f - 1e-6f), isf = (float)iscale;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int b = lane + 32 * j;
            const uint32_t dn = b_n[b];
            const uint64_t s1 = P[b], s0 = b > 0 ? P[b - 1] : (uint64_t)S0;
            const uint32_t n0 = b > 0 ? Q[b - 1] : 0u;
            bool maybe = false;
            if (dn != 0u) {
                const float Sp = (float)s1 * 0x1p-30f + hsf, Sm = (float)s0 * 0x1p-30f + hsf;
                const float N = Nbf + 8.f * (float)n0;
                const float dS = fmaxf(0.f, (float)(s1 - s0) * (0x1p-30f * (1.f - 1e-6f)) - (float)dn * 0x1p-30f);
                maybe = 4.f * Sp * Sp >= b2f * (N + 8.f * (tlof + (float)b * isf * (1.f - 1e-6f)) * dS) ||
                        4.f * Sm * Sm >= b2f * N;
            }
            if (!__any_sync(0xffffffffu, maybe)) continue;
            if (maybe) {
                const double dd = (double)(s1 - s0) * 0x1p-30, de = (double)dn * 0x1p-30;
                const double Sm = (double)s0 * 0x1p-30 + hs + e2, Sp = (double)s1 * 0x1p-30 + hs + e2;
                const double N = Nb + 8.0 * (double)n0;
                const double t0 = ((double)Tlo + (double)b * iscale * (1.0 - 0x1p-20)) * (1.0 - 0x1p-22);
                if (4.0 * Sp * Sp * (1.0 + 1e-12) >= best2 * (N + 8.0 * t0 * fmax(0.0, dd - de)) ||
                    4.0 * Sm * Sm * (1.0 + 1e-12) >= best2 * N) {
                    bmin = min(bmin, b);
                    bmax = max(bmax, b);
                }
            }
        }
        bmin = __reduce_min_sync(0xffffffffu, bmin);
        bmax = __reduce_max_sync(0xffffffffu, bmax);
        if (bmax < bmin) break;                                   // (cannot happen)
        // largest keys below bucket bmin and in bucket bmax
        float lo = Tlo, hi = Thi;
        if (bmin > 0) {
            lo = fminf(fmaxf((float)((double)Tlo + (double)bmin / (double)scale), Tlo), Thi);
            while (lo > Tlo && bucket_of(lo, Tlo, scale) >= bmin) lo = __uint_as_float(__float_as_uint(lo) - 1u);
        }
        if (bmax < NBK - 1) {
            hi = fminf(fmaxf((float)((double)Tlo + (double)(bmax + 1) / (double)scale), Tlo), Thi);
            while (hi < Thi && bucket_of(hi, Tlo, scale) <= bmax) hi = __uint_as_float(__float_as_uint(hi) + 1u);
        }
        __syncwarp();
        Tlo = lo;
        Thi = hi;
    }
    __syncwarp();
    Tlo_out = Tlo;
    Thi_out = Thi;
}

}  // namespace

// bytes of one warp: the scaled row, and the window (event words; bucket sums;
// 16-bit coordinates of an oversized run)
__host__ __device__ inline int enc_run_cap(int D) {
    int n = ENC_W;
    while (n < D) n <<= 1;
    return n;
}
__host__ __device__ inline size_t enc_win_bytes(int D) {
    const size_t b = (size_t)4 * NBK * 4 > (size_t)ENC_W * 8 ? (size_t)4 * NBK * 4 : (size_t)ENC_W * 8;
    const size_t r = (size_t)enc_run_cap(D) * 2;
    return b > r ? b : r;
}

__global__ void __launch_bounds__(256) encode_kernel(const float* __restrict__ Rrot, int64_t n, int D, int B,
                                                     uint8_t* __restrict__ codes, float* __restrict__ f_add,
                                                     float* __restrict__ f_res, double* __restrict__ stats,
                                                     uint32_t* __restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nwarps = blockDim.x >> 5;
    const size_t win_bytes = enc_win_bytes(D);
    unsigned char* base = smem_raw + (size_t)warp * (win_bytes + (size_t)D * 4);
    uint64_t* keys = reinterpret_cast<uint64_t*>(base);
    uint16_t* run16 = reinterpret_cast<uint16_t*>(base);
    float* sa = reinterpret_cast<float*>(base + win_bytes);

    const int M = (1 << (B - 1)) - 1;
    const int half = 1 << (B - 1);
    const int64_t gw = (int64_t)blockIdx.x * nwarps + warp;
    const int64_t stride_w = (int64_t)gridDim.x * nwarps;

    for (int64_t v = gw; v < n; v += stride_w) {
        const float* r = Rrot + v * D;
        int nz = 0;
        float amax = 0.f, amin = INFINITY;
        bool bad = false;
        for (int i = lane; i < D; i += 32) {
            const float x = fabsf(r[i]);
            sa[i] = x;
            nz += (x != 0.f);
            bad |= !(x < INFINITY);
            amax = fmaxf(amax, x);
            if (x > 0.f) amin = fminf(amin, x);
        }
        nz = warp_sum_int(nz);
        amax = warp_max(amax);
        amin = -warp_max(-amin);
        int e2 = 1;
        if (amax > 0.f) frexpf(amax, &e2);       // amax in [2^(e2-1), 2^e2)
        const int es = e2 - 1;                   // the row is scaled by 2^-es
        // keys stay finite when every non-zero magnitude is >= 2^-118 * amax
        // (k + 1 <= 2^9 bounds every key by 2^127); non-finite rows have no events
        const bool small = nz > 0 && amin < ldexpf(amax, -118);
        if (small || (M > 0 && __any_sync(0xffffffffu, bad))) {
            if (lane == 0) atomicOr(status, small ? kStatusRange : kStatusBounds);
            continue;
        }
        double p2 = 0.0;
        float pf = 0.f;
        int g = 1 << 30;
        for (int i = lane; i < D; i += 32) {
            const float x = ldexpf(sa[i], -es);  // exact
            sa[i] = x;
            pf += x;
            p2 = __fma_rn((double)x, (double)x, p2);
            if (x > 0.f) g = min(g, low_exp(x));
        }
        amin = ldexpf(amin, -es);
        amax = ldexpf(amax, -es);
        pf = warp_sum(pf);
        const double nr2p = warp_sum_f64(p2);    // ||o'||^2 / 4^es up to rounding
        g = __reduce_min_sync(0xffffffffu, g);
        __syncwarp();
        // sum a_i in ascending i in FP64: exact when all are multiples of 2^g and
        // the sum is below 2^(53+g)
        double sum_a = 0.0;
        bool sum_exact = nz == 0;
        if (nz > 0 && (double)pf < ldexp(1.01, 53 + g)) {
            int64_t A = 0;
            for (int i = lane; i < D; i += 32)
                if (sa[i] > 0.f) A += units_of(sa[i], g);
            A = warp_sum_i64(A);
            if (A < (1ll << 53)) {
                sum_exact = true;
                sum_a = ldexp(__ll2double_rn(A), g);
            }
        }
        if (!sum_exact) {
            if (lane == 0)
                for (int i = 0; i < D; ++i) sum_a = __dadd_rn(sum_a, (double)sa[i]);
            sum_a = __shfl_sync(0xffffffffu, sum_a, 0);
        }

        // initial state: all |y_i| = 1/2
        double ip_run = __dmul_rn(0.5, sum_a);    // exact scaling
        uint32_t n2q_run = D;                      // 4 ||y||^2 <= D (2^B - 1)^2 < 2^32 (B <= 10, D <= 4096)
        double vmax = __ddiv_rn(ip_run, __dsqrt_rn(0.25 * (double)D));
        double ip_best = ip_run;
        uint32_t n2q_best = D;
        int best_i = -1, best_m = -1;
        const int total = nz * M;                  // <= 4096 * 511
        float T_cur = 0.f;                         // events with key <= T_cur are in the running state
        int n_cur = 0;                             // their number
        float Tlo = 0.f, Thi = INFINITY;
        if (total > ENC_W) find_range(sa, D, M, sum_a, amin, amax, reinterpret_cast<uint32_t*>(base), Tlo, Thi);
        const int n_lo = Tlo > 0.f ? count_upto(sa, D, M, Tlo) : 0;
        const int n_hi = Thi == INFINITY ? total : count_upto(sa, D, M, Thi);

        while (n_cur < n_hi) {
            // ---- the next threshold: the start of the range by jumps, or a window
            float T = Thi;
            int n_T = n_hi;
            if (n_cur < n_lo) {                    // still before the range
                T = Tlo;
                n_T = n_lo;
                float T_f = Tlo;                   // nearest threshold that a jump did not reach
                int n_f = n_lo;
                for (int tries = 0; tries < 200; ++tries) {
                    int gx = 1 << 30;
                    float dF = 0.f;
                    for (int i = lane; i < D; i += 32) {
                        const float x = sa[i];
                        const int d = events_upto(T, x, M) - events_upto(T_cur, x, M);
                        if (d == 0) continue;
                        dF = fmaf(x, (float)d, dF);
                        gx = min(gx, low_exp(x));
                    }
                    dF = warp_sum(dF);
                    gx = min(__reduce_min_sync(0xffffffffu, gx), low_exp(ip_run));
                    const double lim = ldexp(1.0, 53 + gx);
                    bool ok = ip_run + (double)dF * (1.0 - 1e-4) < lim;
                    if (ok) {
                        int64_t dA = 0;
                        uint32_t dN = 0;
                        for (int i = lane; i < D; i += 32) {
                            const float x = sa[i];
                            const int c0 = events_upto(T_cur, x, M), c1 = events_upto(T, x, M);
                            if (c1 == c0) continue;
                            dA += units_of(x, gx) * (c1 - c0);
                            dN += 4u * (uint32_t)(c1 * (c1 + 1) - c0 * (c0 + 1));
                        }
                        const int64_t S1 = __double2ll_rn(ldexp(ip_run, -gx)) + warp_sum_i64(dA);
                        dN = (uint32_t)warp_sum_int((int)dN);
                        ok = S1 < (1ll << 53);     // no addition on the way rounds
                        if (ok) {
                            ip_run = ldexp(__ll2double_rn(S1), gx);
                            n2q_run += dN;
                            T_cur = T;
                            n_cur = n_T;
                        }
                    }
                    if (!ok) {
                        T_f = T;
                        n_f = n_T;
                    }
                    if (n_cur >= n_lo || n_f - n_cur <= ENC_W) break;
                    // towards the sum that is still exact, or half way
                    float h = T_cur + 0.5f * (T_f - T_cur);
                    if (!(tries & 1) && !ok) {
                        const float fr = fmaxf(0.98f * (float)((lim - ip_run) / (double)dF), 0.4f * (float)ENC_W / (float)(n_f - n_cur));
                        h = T_cur + fminf(fr, 0.9f) * (T_f - T_cur);
                    }
                    if (!(h > T_cur && h < T_f)) break;            // one key value
                    T = h;
                    n_T = count_upto(sa, D, M, T);
                }
                if (n_cur >= n_lo) continue;
                T = T_f;                           // walk the events that round
                n_T = n_f;
            }
            int cnt = n_T - n_cur;
            if (cnt > ENC_W) {
                // a threshold with at most ENC_W events after T_cur: bisection on the
                // float bits, after guesses from the event rate
                float lo = T_cur, hi = T;
                int clo = 0, chi = cnt;
                bool found = false;
                for (int it = 0; it < 64; ++it) {
                    const uint32_t ul = __float_as_uint(lo);
                    const uint32_t uh = hi == INFINITY ? 0x7f800000u : __float_as_uint(hi);
                    if (uh <= ul + 1u) break;
                    float guess = hi == INFINITY ? 0.f : lo + (hi - lo) * (0.75f * (float)ENC_W - (float)clo) / (float)(chi - clo);
                    if ((it & 1) || !(guess > lo && guess < hi)) guess = __uint_as_float(ul + (uh - ul) / 2u);
                    const int c = count_upto(sa, D, M, guess) - n_cur;
                    if (c <= ENC_W && c >= ENC_W / 4) {
                        T = guess;
                        cnt = c;
                        found = true;
                        break;
                    }
                    if (c > ENC_W) { hi = guess; chi = c; }
                    else { lo = guess; clo = c; }
                }
                if (!found) {                       // lo and hi are neighbours: a short window, or one key value
                    T = clo > 0 ? lo : hi;
                    cnt = clo > 0 ? clo : chi;
                }
                if (cnt <= 0 || cnt > enc_run_cap(D)) {            // cannot happen for finite rows
                    if (lane == 0) atomicOr(status, kStatusBounds);
                    break;
                }
            }
            const bool over = cnt > ENC_W;          // one key value with more events than a window holds
            __syncwarp();
            if (!over) {
                // ---- gather the window's events
                int mine = 0;
                for (int i = lane; i < D; i += 32) mine += events_upto(T, sa[i], M) - events_upto(T_cur, sa[i], M);
                int pos = warp_incl_scan(mine) - mine;
                for (int i = lane; i < D; i += 32) {
                    const float ai = sa[i];
                    const int c1 = events_upto(T, ai, M);
                    for (int k = events_upto(T_cur, ai, M); k < c1; ++k) {
                        const uint32_t kb = __float_as_uint(ev_key(k, ai));
                        keys[pos++] = ((uint64_t)kb << 32) | ((uint64_t)i << EV_MBITS) | (uint64_t)k;
                    }
                }
                int np2 = 32;
                while (np2 < cnt) np2 <<= 1;
                for (int j = cnt + lane; j < np2; j += 32) keys[j] = ~0ull;
                __syncwarp();
                // ---- warp bitonic sort of np2 keys
                for (int size = 2; size <= np2; size <<= 1) {
                    for (int stride = size >> 1; stride > 0; stride >>= 1) {
                        for (int p = lane; p < np2 / 2; p += 32) {
                            const int lo_i = 2 * p - (p & (stride - 1));
                            const int hi_i = lo_i + stride;
                            const bool up = (lo_i & size) == 0;
                            const uint64_t x = keys[lo_i], y = keys[hi_i];
                            if ((x > y) == up) { keys[lo_i] = y; keys[hi_i] = x; }
                        }
                        __syncwarp();
                    }
                }
                // ---- exact order inside runs of equal FP32 keys: the lane at a run's
                // first position insertion-sorts the run (runs are disjoint, and the
                // FP32 key of every position is unchanged by sorting inside runs)
                for (int j = lane; j + 1 < cnt; j += 32) {
                    const uint32_t kj = (uint32_t)(keys[j] >> 32);
                    if ((uint32_t)(keys[j + 1] >> 32) != kj || (j > 0 && (uint32_t)(keys[j - 1] >> 32) == kj))
                        continue;
                    int e = j + 2;
                    while (e < cnt && (uint32_t)(keys[e] >> 32) == kj) ++e;
                    for (int h = j + 1; h < e; ++h) {
                        const uint64_t x = keys[h];
                        const int ix = ev_i(x), mx = ev_m(x);
                        int g = h - 1;
                        while (g >= j) {
                            const uint64_t y = keys[g];
                            const int iy = ev_i(y), my = ev_m(y);
                            if (!ev_before(sa, ix, mx, iy, my)) break;
                            keys[g + 1] = y;
                            --g;
                        }
                        keys[g + 1] = x;
                    }
                }
            } else {
                // ---- one key value: at most one event per coordinate (its level is
                // the coordinate's event count at T_cur), sorted by the exact order
                int mine = 0;
                for (int i = lane; i < D; i += 32) mine += events_upto(T, sa[i], M) - events_upto(T_cur, sa[i], M);
                int pos = warp_incl_scan(mine) - mine;
                for (int i = lane; i < D; i += 32)
                    if (events_upto(T, sa[i], M) > events_upto(T_cur, sa[i], M)) run16[pos++] = (uint16_t)i;
                int np2 = 32;
                while (np2 < cnt) np2 <<= 1;
                for (int j = cnt + lane; j < np2; j += 32) run16[j] = 0xffffu;
                __syncwarp();
                for (int size = 2; size <= np2; size <<= 1) {
                    for (int stride = size >> 1; stride > 0; stride >>= 1) {
                        for (int p = lane; p < np2 / 2; p += 32) {
                            const int lo_i = 2 * p - (p & (stride - 1));
                            const int hi_i = lo_i + stride;
                            const bool up = (lo_i & size) == 0;
                            const int x = run16[lo_i], y = run16[hi_i];
                            const bool gt = x == 0xffff ? y != 0xffff
                                                        : (y != 0xffff && ev_before(sa, y, events_upto(T_cur, sa[y], M), x,
                                                                                    events_upto(T_cur, sa[x], M)));
                            const bool lt = y == 0xffff ? x != 0xffff : !gt && x != y;
                            if (up ? gt : lt) { run16[lo_i] = (uint16_t)y; run16[hi_i] = (uint16_t)x; }
                        }
                        __syncwarp();
                    }
                }
            }
            __syncwarp();
            auto event = [&](int j, int& i, int& m) {
                if (!over) {
                    const uint64_t x = keys[j];
                    i = ev_i(x);
                    m = ev_m(x);
                } else {
                    i = run16[j];
                    m = events_upto(T_cur, sa[i], M);
                }
            };
            // ---- the window's states: <y, o'> after each event, 4 ||y||^2, and
            // the state of largest cosine (first one on ties)
            const int C = (cnt + 31) >> 5;                     // events per lane (contiguous chunk)
            const int c0 = min(cnt, lane * C), c1 = min(cnt, c0 + C);
            int sumN = 0, gx = 1 << 30;
            float sumF = 0.f;
            for (int j = c0; j < c1; ++j) {
                int i, m;
                event(j, i, m);
                sumN += 8 * (m + 1);                            // 4 * ((m + 3/2)^2 - (m + 1/2)^2)
                sumF += sa[i];
                gx = min(gx, low_exp(sa[i]));
            }
            const int baseN = warp_incl_scan(sumN) - sumN;
            const int totN = __shfl_sync(0xffffffffu, baseN + sumN, 31);
            // no addition of the window rounds when the running sum and all addends
            // are multiples of 2^g and the final sum is below 2^(53+g)
            gx = min(__reduce_min_sync(0xffffffffu, gx), low_exp(ip_run));
            int64_t S_int = 0, baseA = 0, totA = 0;
            bool fast = ip_run + (double)warp_sum(sumF) * (1.0 - 1e-4) < ldexp(1.0, 53 + gx);
            if (fast) {
                int64_t sumA = 0;
                for (int j = c0; j < c1; ++j) {
                    int i, m;
                    event(j, i, m);
                    sumA += units_of(sa[i], gx);
                }
                baseA = warp_excl_scan_i64(sumA, totA);
                S_int = __double2ll_rn(ldexp(ip_run, -gx));
                fast = S_int + totA < (1ll << 53);
            }
            // FP32 cosine bounds are within 4e-7 (a rounded sum and count, rsqrtf
            // within 2 ulp, one product); states within 4e-6 of the best are exact
            constexpr float kNear = 1.0f - 4e-6f;
            double bv = -1.0, bip = 0.0;                        // best cosine and its exact <y, o'>
            int bj = 0x7fffffff;
            uint32_t bn = 0;
            if (fast) {
                const float vmax_u = (float)ldexp(vmax, -gx);  // cosine bounds in units of 2^gx (scale-free)
                float lmax = 0.f;
                int64_t P = S_int + baseA;
                uint32_t N = n2q_run + (uint32_t)baseN;
                for (int j = c0; j < c1; ++j) {
                    int i, m;
                    event(j, i, m);
                    P += units_of(sa[i], gx);
                    N += 8 * (m + 1);
                    lmax = fmaxf(lmax, (float)P * rsqrtf(0.25f * (float)N));
                }
                const float thr = fmaxf(warp_max(lmax), vmax_u) * kNear;
                P = S_int + baseA;
                N = n2q_run + baseN;
                for (int j = c0; j < c1; ++j) {
                    int i, m;
                    event(j, i, m);
                    P += units_of(sa[i], gx);
                    N += 8 * (m + 1);
                    if ((float)P * rsqrtf(0.25f * (float)N) >= thr) {
                        const double ipj = ldexp(__ll2double_rn(P), gx);   // exact: P < 2^53
                        const double ve = __ddiv_rn(ipj, __dsqrt_rn(0.25 * (double)N));
                        if (ve > bv) { bv = ve; bip = ipj; bj = j; bn = N; }   // j ascending per lane: first max kept
                    }
                }
            } else if (lane == 0) {
                // serial FP64 walk, every addition rounded (two passes: bound, then exact check)
                float lmax = 0.f;
                double ip = ip_run;
                uint32_t N = n2q_run;
                for (int j = 0; j < cnt; ++j) {
                    int i, m;
                    event(j, i, m);
                    ip = __dadd_rn(ip, (double)sa[i]);
                    N += 8 * (m + 1);
                    lmax = fmaxf(lmax, (float)ip * rsqrtf(0.25f * (float)N));
                }
                const float thr = fmaxf(lmax, (float)vmax) * kNear;
                ip = ip_run;
                N = n2q_run;
                for (int j = 0; j < cnt; ++j) {
                    int i, m;
                    event(j, i, m);
                    ip = __dadd_rn(ip, (double)sa[i]);
                    N += 8 * (m + 1);
                    if ((float)ip * rsqrtf(0.25f * (float)N) >= thr) {
                        const double ve = __ddiv_rn(ip, __dsqrt_rn(0.25 * (double)N));
                        if (ve > bv) { bv = ve; bip = ip; bj = j; bn = N; }
                    }
                }
                ip_run = ip;   // lane 0 only; broadcast below
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
                const double oip = __shfl_xor_sync(0xffffffffu, bip, o);
                const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                const uint32_t on = __shfl_xor_sync(0xffffffffu, bn, o);
                if (ov > bv || (ov == bv && oj < bj)) { bv = ov; bip = oip; bj = oj; bn = on; }
            }
            if (bv > vmax) {
                vmax = bv;
                event(bj, best_i, best_m);
                ip_best = bip;
                n2q_best = bn;
            }
            // advance the running state
            if (fast) ip_run = ldexp(__ll2double_rn(S_int + totA), gx);
            else ip_run = __shfl_sync(0xffffffffu, ip_run, 0);
            n2q_run += totN;
            n_cur += cnt;
            T_cur = T;
            __syncwarp();
        }

        // ---- final state and code
        uint8_t* code = codes + v * D * code_bytes(B);
        const double abest = best_i >= 0 ? (double)sa[best_i] : 0.0;
        for (int i = lane; i < D; i += 32) {
            int mi = 0;
            const float ai = sa[i];
            if (best_i >= 0 && ai > 0.f) {
                const double rhs = (double)(best_m + 1) * (double)ai;
                auto qual = [&](int m) {  // event (i, m) precedes or equals (best_i, best_m)
                    const double lhs = (double)(m + 1) * abest;
                    return lhs < rhs || (lhs == rhs && i <= best_i);
                };
                const float q = __fdividef((float)(best_m + 1) * ai, (float)abest);
                const float fl = floorf(q), d = q - fl, eps = q * 1e-5f;
                int j = fl > (float)M ? M : (int)fl;
                if (!(d > eps && d < 1.f - eps)) {             // near an event: the exact comparison decides
                    while (j < M && qual(j)) ++j;
                    while (j > 0 && !qual(j - 1)) --j;
                }
                mi = j;
            }
            const float x = r[i];
            const int u = x >= 0.f ? half + mi : half - 1 - mi;
            if (B > 8) reinterpret_cast<uint16_t*>(code)[i] = (uint16_t)u;
            else code[i] = (uint8_t)u;
        }
        // ---- factors.  ||o'||^2 is the FP64 sum of the squares in ascending i;
        // the parallel sum differs by at most `rel`, which matters only when it
        // could change an FP32 result
        const double ipo = ldexp(ip_best, es);
        double nr2 = ldexp(nr2p, 2 * es);
        const double rel = (1.25 * (double)D + 32.0) * 0x1p-53;
        const double nlo = nr2 * (1.0 - rel), nhi = nr2 * (1.0 + rel);
        if (nr2 > 0.0 && (__double2float_rn(nlo) != __double2float_rn(nhi) ||
                          __double2float_rn(__ddiv_rn(-2.0 * nlo, ipo)) != __double2float_rn(__ddiv_rn(-2.0 * nhi, ipo)))) {
            nr2 = 0.0;
            if (lane == 0)
                for (int i = 0; i < D; ++i) {
                    const double x = (double)r[i];
                    nr2 = __fma_rn(x, x, nr2);
                }
        }
        if (lane == 0) {
            f_add[v] = __double2float_rn(nr2);
            f_res[v] = nr2 > 0.0 ? __double2float_rn(__ddiv_rn(-2.0 * nr2, ipo)) : 0.f;
            if (stats) {
                stats[2 * v] = ipo;
                stats[2 * v + 1] = 0.25 * (double)n2q_best;
            }
        }
        __syncwarp();
    }
}

cudaError_t launch_encode(const float* Rrot, int64_t n, int D, int B, uint8_t* codes, float* f_add, float* f_res,
                          double* stats, uint32_t* status, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const size_t per_warp = enc_win_bytes(D) + (size_t)D * 4;
    int warps = (int)((220 * 1024) / per_warp / 2);      // two blocks an SM and at most 8 warps a block
    warps = warps < 1 ? 1 : (warps > 8 ? 8 : warps);
    const size_t smem = per_warp * warps;
    cudaError_t e = cudaFuncSetAttribute(encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = ceil_div(n, warps);
    const int64_t cap = (int64_t)sms * 16;
    if (blocks > cap) blocks = cap;
    count_launch();
    encode_kernel<<<(unsigned)blocks, warps * 32, smem, s>>>(Rrot, n, D, B, codes, f_add, f_res, stats, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// g = f_add - f_res * <ybar, c'> per stored row (FP64 accumulation in ascending
// index, one rounding).  With it the estimate of Eq. 3.3 + Eq. (eq:dis to ip)
// against the *global* rotated query q' = P^T q_r becomes
//   est = ||q_r - c||^2 + g + f_res * <ybar, q'>,
// because P^T (q_r - c) = q' - c'.  One warp per row.  The products are exact
// in FP64; the sum is taken in parallel, and again serially in ascending order
// only when the two orders (each within D 2^-53 of sum |product|) could round
// to different FP32 results.
// ---------------------------------------------------------------------------
__global__ void gconst_kernel(const uint8_t* __restrict__ codes, const float* __restrict__ f_add,
                              const float* __restrict__ f_res, const float* __restrict__ Cp,
                              const int32_t* __restrict__ cl_of_row, int64_t n, int D, int B,
                              float* __restrict__ g_out) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n) return;
    const float* c = Cp + (int64_t)cl_of_row[w] * D;
    const double off = 0.5 * (double)((1 << B) - 1);
    const float off_f = (float)off;                  // at most 255.5, and code - off is exact in FP32
    double acc = 0.0;
    float mag = 0.f;
    for (int k = lane; k < D; k += 32) {
        const float y = (float)load_code(codes, B, w * D + k) - off_f, x = c[k];
        acc = __fma_rn((double)y, (double)x, acc);
        mag += fabsf(y * x);
    }
    acc = warp_sum_f64(acc);
    mag = warp_sum(mag);
    const double fa = (double)f_add[w], fr = (double)f_res[w];
    // both sums are within D 2^-53 sum|product| of the exact one
    const double tol = fabs(fr) * (double)mag * (2.2 * (double)D + 64.0) * 0x1p-53;
    double g = __dsub_rn(fa, __dmul_rn(fr, acc));
    const double slack = tol + (fabs(fa) + fabs(g)) * 0x1p-50;
    if (!(__double2float_rn(g - slack) == __double2float_rn(g + slack))) {
        acc = 0.0;
        if (lane == 0) {
            for (int k = 0; k < D; ++k)
                acc = __dadd_rn(acc, __dmul_rn((double)load_code(codes, B, w * D + k) - off, (double)c[k]));
            g = __dsub_rn(fa, __dmul_rn(fr, acc));
        }
    }
    if (lane == 0) g_out[w] = __double2float_rn(g);
}

cudaError_t launch_gconst(const uint8_t* codes, const float* f_add, const float* f_res, const float* Cp,
                          const int32_t* cl_of_row, int64_t n, int D, int B, float* g_out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    gconst_kernel<<<(unsigned)ceil_div(n * 32, 256), 256, 0, s>>>(codes, f_add, f_res, Cp, cl_of_row, n, D, B, g_out);
    return cudaGetLastError();
}

}  // namespace erq
