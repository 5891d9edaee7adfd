// The exact rotation on the tcgen05 tensor cores:
//   out[r][j] = fl32( sum_{k ascending} res_k * P[k][j] ),  res_k = fl32(X[r][k] - C[k]),
// the FP64 sum of rotate_fp64_kernel rounded once to FP32, bit for bit, without
// its FP64 multiply-adds (GB300's FP64 pipe holds that kernel to 0.75 TFLOP/s:
// 156 ms for 100,000 x 768; this path 3 ms).
//
// Error-free slicing (Ozaki, Ogita, Oishi, Rump 2012; on FP16 tensor cores
// Mukunoki et al. 2020): every row of residuals and every column of P is scaled
// by a power of two into (-1/2, 1/2) and written as seven signed 7-bit digits,
// x = sum_s d_s 2^-7s + tail, |d_s| <= 64, |tail| <= 2^-50.  A product of two
// digits is an integer of at most 2^12, exact in FP16 operands, and FP32
// accumulators hold the sums exactly while they stay below 2^24.  The 28 digit
// pairs with s + t <= 8 go to seven accumulators, one per weight s + t (at most
// 7 pairs x 512 coordinates x 2^12 < 2^24), which the epilogue warps add into
// one int64 per output every 512 coordinates.  The int64 value I (units
// 2^(e_row + e_col - 49)) is within
//   delta = 2.5 D + 16 + D/16 ||x|| ||p||
// of the sequential FP64 sum: dropped pairs and tails (2.1 D), the floor of the
// last accumulator, and the FP64 sum's own rounding (D 2^-53 sum |x p|, Cauchy-
// Schwarz).  Where I - delta and I + delta round to the same FP32 value, that is
// the result; the other elements (1 in 480 at D = 768, 1 in 115 at D = 4096) go to a
// list and are summed in FP64 in order by rotate_fix_kernel.  A list that overflows, a row that is
// not finite or a wait that runs out sets a flag, and rotate_fp64_kernel then
// computes the whole block.
//
// Tile 128 rows x 64 columns (7 x 64 TMEM columns of accumulators).  A stage is
// a K block of 32 coordinates, all 7 + 7 digit tiles (84 KB, 64-byte swizzled
// rows), so every digit is fetched once per tile and its 28 pairs read it from
// shared memory; two stages.  Bound by the MMA's shared-memory reads (6 KB per
// 128 x 64 x 16 instruction).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "erq_kernels.cuh"
#include "tc_common.cuh"

namespace erq {

namespace rot {
constexpr int BM = 128, BN = 64, BK = 32, ND = 7, WMAX = 8, STAGES = 2, THREADS = 320;
constexpr int W_TMA = 8, W_MMA = 9;                   // warps 0-7: epilogue, TMEM lanes 32 (w % 4), columns 32 (w / 4)
constexpr int KCHUNK = 512;                            // coordinates between drains of the accumulators
constexpr int TILE_A = BM * BK * 2, TILE_B = BN * BK * 2;
constexpr int STAGE = ND * (TILE_A + TILE_B);
constexpr int OFF_BARS = STAGES * STAGE;
constexpr int NBARS = 2 * STAGES + 3;
constexpr int OFF_TMEM = OFF_BARS + NBARS * 8;
constexpr int OFF_ABORT = OFF_TMEM + 4;
constexpr int SMEM = OFF_ABORT + 4 + 1024;
static_assert(SMEM <= 227 * 1024, "rotation shared memory");
static_assert((WMAX - 1) * KCHUNK * 4096 <= (1 << 24), "exact FP32 accumulation");

struct Args {
    const int32_t* ea;       // [n] row exponents
    const float* na;         // [n] row norms (scaled), < 0: a zero row
    const int32_t* eb;       // [D] column exponents
    const float* nb;         // [D] column norms (scaled)
    float* out;              // [n][D]
    int64_t n;
    int D;
    uint2* list;             // elements to sum in FP64
    uint32_t cap;
    uint32_t* ctr;           // [0] list entries, [1] whole-block fallback
};
}  // namespace rot

using namespace tc;

// Descriptor of a K-major tile with 64-byte swizzled rows (8-row groups of 512 bytes).
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t addr) {
    return (uint64_t)((addr >> 4) & 0x3fff) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)4 << 61);
}

__global__ void __launch_bounds__(rot::THREADS, 1)
    rotate_tc_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, rot::Args a) {
    using namespace rot;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t bars = smem_u32(sm + OFF_BARS);
    const uint32_t full0 = bars, empty0 = bars + 8 * STAGES, tfull = bars + 16 * STAGES, tempty = tfull + 8,
                   done_bar = tfull + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + OFF_TMEM);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + OFF_ABORT);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nkb = a.D / BK;
    const int64_t ntm = (a.n + BM - 1) / BM;
    const int ntn = a.D / BN;
    const int64_t ntiles = ntm * ntn;

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(tfull, 1);
        mbar_init(tempty, 256);
        mbar_init(done_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == W_TMA) {
        // ---------------------------------------------------------------- TMA
        uint32_t it = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
            const int m0 = (int)((tile / ntn) * BM), n0 = (int)(tile % ntn) * BN;
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int s = it % STAGES;
                if (!mbar_wait_warp(empty0 + 8 * s, ((it / STAGES) & 1) ^ 1, abort_flag)) { ok = false; break; }
                if (lane == 0) {
                    const uint32_t st = smem_u32(sm + s * STAGE), bar = full0 + 8 * s;
                    mbar_arrive_expect_tx(bar, STAGE);
#pragma unroll
                    for (int d = 0; d < ND; ++d) {             // (rows past n are another digit's, or zero: never stored)
                        tma_load_2d(st + d * TILE_A, &map_a, kb * BK, d * (int)a.n + m0, bar);
                        tma_load_2d(st + ND * TILE_A + d * TILE_B, &map_b, kb * BK, d * a.D + n0, bar);
                    }
                }
                __syncwarp();
            }
        }
        for (uint32_t k = 0; k < STAGES && k < it; ++k) {
            const uint32_t g = it - 1 - k;
            mbar_wait_drain(full0 + 8 * (g % STAGES), (g / STAGES) & 1);
        }
        __syncwarp();
    } else if (warp == W_MMA) {
        // ---------------------------------------------------------------- MMA issuer
        uint32_t it = 0, ch = 0;
        bool ok = true;
        const uint32_t idesc = idesc_f16(BM, BN);
        for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const bool first = kb % (KCHUNK / BK) == 0, last = kb + 1 == nkb || (kb + 1) % (KCHUNK / BK) == 0;
                if (first && !mbar_wait_warp(tempty, (ch & 1) ^ 1, abort_flag)) { ok = false; break; }
                const int s = it % STAGES;
                if (!mbar_wait_warp(full0 + 8 * s, (it / STAGES) & 1, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t st = smem_u32(sm + s * STAGE);
                const uint64_t da = sdesc_sw64(st), db = sdesc_sw64(st + ND * TILE_A);
                if (elect_one()) {
#pragma unroll
                    for (int x = 1; x <= ND; ++x)
#pragma unroll
                        for (int y = 1; y <= ND; ++y) {
                            if (x + y > WMAX) continue;
#pragma unroll
                            for (int k = 0; k < BK / 16; ++k)
                                mma_f16(tmem + (x + y - 2) * BN, da + (uint64_t)(((x - 1) * TILE_A + k * 32) >> 4),
                                        db + (uint64_t)(((y - 1) * TILE_B + k * 32) >> 4), idesc,
                                        !(first && x == 1 && k == 0));   // x = 1 comes first for every weight
                        }
                    mma_commit(empty0 + 8 * s);
                    if (last) mma_commit(tfull);
                }
                __syncwarp();
                if (last) ++ch;
            }
        }
        if (elect_one()) mma_commit(done_bar);
        __syncwarp();
        mbar_wait_drain(done_bar, 0);
        __syncwarp();
    } else {
        // ---------------------------------------------------------------- epilogue
        constexpr int NC = BN / 2;                          // columns of this warp
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const int col0 = (warp >> 2) * NC;
        const int nch = (a.D + KCHUNK - 1) / KCHUNK;
        uint32_t ch = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
            const int64_t m = (tile / ntn) * BM + (warp & 3) * 32 + lane;
            const int n0 = (int)(tile % ntn) * BN + col0;
            int64_t I[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) I[j] = 0;
            for (int c = 0; c < nch; ++c, ++ch) {
                if (!mbar_wait_warp(tfull, ch & 1, abort_flag)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int w = 2; w <= WMAX; ++w) {
                    uint32_t v[NC];
                    ERQ_TMEM_LD32(tmem + lane_base + (w - 2) * BN + col0, v);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        const int x = __float2int_rn(__uint_as_float(v[j]));
                        I[j] += w < WMAX ? (int64_t)x * (1ll << (7 * (WMAX - 1 - w))) : (int64_t)(x >> 7);
                    }
                }
                tc_fence_before();
                mbar_arrive(tempty);
            }
            if (!ok) break;
            if (m < a.n) {
                const float nx = a.na[m];
                const int ex = a.ea[m];
                const float dx = nx * (float)a.D * (1.05f / 16.f), d0 = 2.5f * (float)a.D + 16.f;
                float* o = a.out + m * a.D + n0;
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    const int64_t delta = (int64_t)fmaf(dx, a.nb[n0 + j], d0);
                    const float f = __ll2float_rn(I[j]);
                    const int e = ex + a.eb[n0 + j] - 49;
                    const float r = nx < 0.f ? 0.f : ldexpf(f, e);
                    // the two ends round differently, or the result is not a normal number
                    if (nx >= 0.f && (__ll2float_rn(I[j] - delta) != __ll2float_rn(I[j] + delta) || !(fabsf(r) >= 0x1p-125f))) {
                        const uint32_t at = atomicAdd(a.ctr, 1u);
                        if (at < a.cap) a.list[at] = make_uint2((uint32_t)m, (uint32_t)(n0 + j));
                        else a.ctr[1] = 1u;
                    }
                    o[j] = r;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag && tid == 0) a.ctr[1] = 1u;
    if (warp == W_MMA) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
    }
}

// Rows (or, for P, the rows of its transpose) -> seven 7-bit digits in FP16,
// the scale exponent E (|x| 2^-E < 1/2) and the scaled row's norm (-1: all
// zeros).  One warp per row, eight coordinates a lane.  A row that is not
// finite raises the whole-block fallback.
__global__ void __launch_bounds__(256) rotate_split_kernel(const float* __restrict__ X, const int64_t* __restrict__ gather,
                                                           const float* __restrict__ C, const int32_t* __restrict__ cl,
                                                           int64_t n, int D, __half* __restrict__ dig,
                                                           int32_t* __restrict__ ex, float* __restrict__ norm,
                                                           uint32_t* __restrict__ ctr) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const float* x = X + (gather ? gather[r] : r) * D;
    const float* c = C ? C + (int64_t)(cl ? cl[r] : 0) * D : nullptr;
    auto load8 = [&](int k, float (&v)[8]) {
        const float4 p = *reinterpret_cast<const float4*>(x + k), q = *reinterpret_cast<const float4*>(x + k + 4);
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w; v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
        if (c) {
            const float4 s = *reinterpret_cast<const float4*>(c + k), t = *reinterpret_cast<const float4*>(c + k + 4);
            const float w[8] = {s.x, s.y, s.z, s.w, t.x, t.y, t.z, t.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __fsub_rn(v[i], w[i]);
        }
    };
    float mx = 0.f;
    bool bad = false;
    for (int k = lane * 8; k < D; k += 256) {
        float v[8];
        load8(k, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            mx = fmaxf(mx, fabsf(v[i]));
            bad |= !(fabsf(v[i]) < INFINITY);
        }
    }
    mx = warp_max(mx);
    bad = __any_sync(0xffffffffu, bad);
    int E = 0;
    if (mx > 0.f && !bad) {
        frexpf(mx, &E);                                 // mx in [2^(E-1), 2^E)
        ++E;
    }
    float ss = 0.f;
    for (int k = lane * 8; k < D; k += 256) {
        float v[8];
        load8(k, v);
        uint32_t h[rot::ND][4];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            float t0 = bad ? 0.f : ldexpf(v[i], -E), t1 = bad ? 0.f : ldexpf(v[i + 1], -E);
            ss = fmaf(t0, t0, fmaf(t1, t1, ss));
#pragma unroll
            for (int d = 0; d < rot::ND; ++d) {
                t0 *= 128.f;
                t1 *= 128.f;
                const float i0 = rintf(t0), i1 = rintf(t1);
                t0 -= i0;                               // exact
                t1 -= i1;
                const __half2 hh = __floats2half2_rn(i0, i1);
                h[d][i / 2] = *reinterpret_cast<const uint32_t*>(&hh);
            }
        }
#pragma unroll
        for (int d = 0; d < rot::ND; ++d)
            *reinterpret_cast<uint4*>(dig + ((int64_t)d * n + r) * D + k) = make_uint4(h[d][0], h[d][1], h[d][2], h[d][3]);
    }
    ss = warp_sum(ss);
    if (lane == 0) {
        ex[r] = E;
        norm[r] = mx > 0.f ? sqrtf(ss) * 1.001f : -1.f;
        if (bad) ctr[1] = 1u;
    }
}

// The listed elements by the sequential FP64 sum, one thread each.
__global__ void __launch_bounds__(128) rotate_fix_kernel(const float* __restrict__ X, const int64_t* __restrict__ gather,
                                                         const float* __restrict__ C, const int32_t* __restrict__ cl,
                                                         const float* __restrict__ P, float* __restrict__ out, int D,
                                                         const uint2* __restrict__ list, uint32_t cap,
                                                         const uint32_t* __restrict__ ctr) {
    if (ctr[1]) return;                                 // the whole block is computed instead
    const uint32_t cnt = min(ctr[0], cap);
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += gridDim.x * blockDim.x) {
        const uint2 e = list[t];
        const float* x = X + (gather ? gather[e.x] : (int64_t)e.x) * D;
        const float* c = C ? C + (int64_t)(cl ? cl[e.x] : 0) * D : nullptr;
        const float* p = P + e.y;
        double acc = 0.0;
        for (int k = 0; k < D; k += 32) {                // 32 coordinates in flight: the loads' latency bounds this kernel
            float xv[32], pv[32];
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(x + k + i);
                xv[i] = v.x; xv[i + 1] = v.y; xv[i + 2] = v.z; xv[i + 3] = v.w;
                if (c) {
                    const float4 w = *reinterpret_cast<const float4*>(c + k + i);
                    xv[i] = __fsub_rn(v.x, w.x); xv[i + 1] = __fsub_rn(v.y, w.y);
                    xv[i + 2] = __fsub_rn(v.z, w.z); xv[i + 3] = __fsub_rn(v.w, w.w);
                }
            }
#pragma unroll
            for (int i = 0; i < 32; ++i) pv[i] = p[(int64_t)(k + i) * D];
#pragma unroll
            for (int i = 0; i < 32; ++i) acc = __fma_rn((double)xv[i], (double)pv[i], acc);
        }
        out[(int64_t)e.x * D + e.y] = __double2float_rn(acc);
    }
}

static bool make_digit_map(CUtensorMap* map, const __half* base, int64_t rows, int D, int box_rows) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void* fn = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return false;
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    const cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)D * 2};
    const cuuint32_t box[2] = {(cuuint32_t)rot::BK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (void*)base, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The sliced rotation of n rows (in blocks of rows whose digits take 256 MB at
// most).  Returns cudaErrorNotSupported, with nothing launched, where the caller
// has to use the FP64 kernel alone: inside a stream capture and without memory.
cudaError_t launch_rotate_tc(const float* X, const int64_t* gather, const float* C, const int32_t* cl, const float* P,
                             float* out, int64_t n, int D, cudaStream_t s) {
    using namespace rot;
    cudaStreamCaptureStatus cap_st = cudaStreamCaptureStatusNone;
    if (D % BN != 0 || ((uintptr_t)X & 15) || ((uintptr_t)P & 15) || ((uintptr_t)C & 15) ||
        cudaStreamIsCapturing(s, &cap_st) != cudaSuccess || cap_st != cudaStreamCaptureStatusNone)
        return cudaErrorNotSupported;
    const int64_t block = std::min<int64_t>(n, std::max<int64_t>(2048, ((256ll << 20) / (ND * 2 * (int64_t)D)) / BM * BM));
    // doubtful elements of ordinary rows: 1 in 480 at D = 768, 1 in 180 at 2,048, 1 in 115
    // at 3,072 and 4,096; a list that is too short costs the whole block again in FP64
    // (65,536 x 3,072 with room for 1 in 128: 1,600 ms, 62 with room for 1 in 32)
    const size_t cap = (size_t)(block * D / 32 + 8192);
    size_t off = 0;
    auto part = [&](size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_da = part((size_t)ND * block * D * 2), o_db = part((size_t)ND * D * D * 2), o_pt = part((size_t)D * D * 4),
                 o_ea = part(4 * (size_t)block), o_na = part(4 * (size_t)block), o_eb = part(4 * (size_t)D),
                 o_nb = part(4 * (size_t)D), o_list = part(8 * cap), o_ctr = part(16);
    char* ws = nullptr;
    if (cudaMallocAsync((void**)&ws, off, s) != cudaSuccess) {
        cudaGetLastError();
        return cudaErrorNotSupported;
    }
    CUtensorMap map_a, map_b;
    __half* da = (__half*)(ws + o_da);
    __half* db = (__half*)(ws + o_db);
    uint32_t* ctr = (uint32_t*)(ws + o_ctr);
    cudaError_t e = cudaFuncSetAttribute(rotate_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e == cudaSuccess && !make_digit_map(&map_b, db, (int64_t)ND * D, D, BN)) e = cudaErrorInvalidValue;
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int64_t r0 = 0; r0 < n && e == cudaSuccess; r0 += block) {
        const int64_t m = std::min(block, n - r0);
        const float* Xb = gather ? X : X + r0 * D;
        const int64_t* gb = gather ? gather + r0 : nullptr;
        const int32_t* cb = cl ? cl + r0 : nullptr;
        float* ob = out + r0 * D;
        if ((e = cudaMemsetAsync(ctr, 0, 8, s)) != cudaSuccess) break;
        if (r0 == 0 && (e = launch_transpose(P, D, D, (float*)(ws + o_pt), s)) != cudaSuccess) break;
        count_launch();                                 // (again for every block: a P that is not finite raises each one's flag)
        rotate_split_kernel<<<(unsigned)ceil_div(D, 8), 256, 0, s>>>((const float*)(ws + o_pt), nullptr, nullptr, nullptr, D, D,
                                                                    db, (int32_t*)(ws + o_eb), (float*)(ws + o_nb), ctr);
        count_launch();
        rotate_split_kernel<<<(unsigned)ceil_div(m, 8), 256, 0, s>>>(Xb, gb, C, cb, m, D, da, (int32_t*)(ws + o_ea),
                                                                    (float*)(ws + o_na), ctr);
        if (!make_digit_map(&map_a, da, (int64_t)ND * m, D, BM)) {
            e = cudaErrorInvalidValue;
            break;
        }
        Args a;
        a.ea = (const int32_t*)(ws + o_ea); a.na = (const float*)(ws + o_na); a.eb = (const int32_t*)(ws + o_eb);
        a.nb = (const float*)(ws + o_nb); a.out = ob; a.n = m; a.D = D; a.list = (uint2*)(ws + o_list); a.cap = (uint32_t)cap;
        a.ctr = ctr;
        const int64_t tiles = ceil_div(m, BM) * (D / BN);
        count_launch();
        rotate_tc_kernel<<<(unsigned)std::min<int64_t>(tiles, sms), THREADS, SMEM, s>>>(map_a, map_b, a);
        count_launch();
        rotate_fix_kernel<<<(unsigned)(sms * 4), 128, 0, s>>>(Xb, gb, C, cb, P, ob, D, a.list, a.cap, ctr);
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        e = launch_rotate_fp64_if(ctr + 1, Xb, gb, C, cb, P, ob, m, D, s);
    }
    const cudaError_t ef = cudaFreeAsync(ws, s);
    return e != cudaSuccess ? e : ef;
}

}  // namespace erq
