// Search path kernels (Section 4.1 IVF search with the Section 3.2 estimator):
//   dqc      ||q_r - c||^2 for every probed (query, cluster) pair
//   plan     invert probe lists into the scan's work items
//   scan     estimate every (query, candidate) pair of an item and keep the
//            item's top-k' per query (FP32 CUDA-core path)
//   merge    per query, the k' smallest estimates over all of its items
//   rerank   exact squared distances of the k' candidates, top-k
//   estimate estimates of explicit (query, id) pairs
//   backward gather of sum_j g_j f_res,j ybar_j and sum_j g_j c_j per query
//
// Estimator used by every GPU path (algebraically Eq. 3.3 + Eq. eq:dis to ip):
//   est = ||q_r - c||^2 + g + (f_res / 2) * <2 ybar, q'>,
//   q'  = P^T q_r (rotated once per query),  2 ybar = 2 ybar_u - (2^B - 1),
//   g   = f_add - f_res <ybar, c'>  (per row, index time),
// because P^T (q_r - c) = q' - c' and <ybar_u, x> - (2^B-1)/2 sum x = <ybar, x>.
#include <cuda_runtime.h>
#include <stdint.h>

#include "erq_kernels.cuh"
#include "erq_search.cuh"
#include "tc_common.cuh"
#include "warp_sort.cuh"

namespace erq {

// ---------------------------------------------------------------------------
// ||q_r - c||^2 (or, for the inner-product metric, -<q_r, c>) for every probed
// (query, cluster): one block per query, the query row in shared memory, one
// warp per probed cluster (looping when the query probes more clusters than
// the block has warps).  Each lane keeps up to eight 16-byte loads of the
// centroid row in flight (D <= 4096).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512) dqc_kernel(const float* __restrict__ Q, const float* __restrict__ C,
                                                  const int32_t* __restrict__ probe, const int32_t* __restrict__ npr,
                                                  int64_t nq, int maxp, int D, int ip, float* __restrict__ dqc) {
    extern __shared__ float qs[];
    const int64_t q = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int np = npr ? min(max(npr[q], 0), maxp) : maxp;
    // the first centroid row's loads are issued before the query row is waited for
    constexpr int RU = 8;
    int slot = warp;
    float4 a[RU];
    auto issue = [&](int sl) {
        const int c = sl < np ? probe[q * maxp + sl] : -1;
        const float* y = C + (int64_t)(c < 0 ? 0 : c) * D;
#pragma unroll
        for (int u = 0; u < RU; ++u) {
            const int t = 128 * u + lane * 4;
            if (t < D) a[u] = *reinterpret_cast<const float4*>(y + t);
        }
        return c;
    };
    int c = slot < np ? issue(slot) : -1;
    for (int k = threadIdx.x * 4; k < D; k += blockDim.x * 4)
        *reinterpret_cast<float4*>(qs + k) = *reinterpret_cast<const float4*>(Q + q * D + k);
    __syncthreads();
    for (; slot < np; slot += nw) {
        if (slot != warp) c = issue(slot);
        float s = 0.f;
        for (int t0 = 0; t0 < D; t0 += 128 * RU) {
            if (t0 > 0) {
                const float* y = C + (int64_t)(c < 0 ? 0 : c) * D;
#pragma unroll
                for (int u = 0; u < RU; ++u) {
                    const int t = t0 + 128 * u + lane * 4;
                    if (t < D) a[u] = *reinterpret_cast<const float4*>(y + t);
                }
            }
#pragma unroll
            for (int u = 0; u < RU; ++u) {
                const int t = t0 + 128 * u + lane * 4;
                if (t < D) {
                    const float4 b = *reinterpret_cast<const float4*>(qs + t);
                    if (ip) {
                        s = fmaf(b.x, a[u].x, s);
                        s = fmaf(b.y, a[u].y, s);
                        s = fmaf(b.z, a[u].z, s);
                        s = fmaf(b.w, a[u].w, s);
                    } else {
                        const float d0 = b.x - a[u].x, d1 = b.y - a[u].y, d2 = b.z - a[u].z, d3 = b.w - a[u].w;
                        s = fmaf(d0, d0, s);
                        s = fmaf(d1, d1, s);
                        s = fmaf(d2, d2, s);
                        s = fmaf(d3, d3, s);
                    }
                }
            }
        }
        s = warp_sum(s);
        // invalid probe ids are reported through the status word
        if (lane == 0 && c >= 0) dqc[q * maxp + slot] = ip ? -s : s;
    }
}

// ---------------------------------------------------------------------------
// Planning: probe lists -> work items.  A work item is (cluster, up to QT of its
// probing queries, up to RR of its rows).  Every (query, slot) pair takes its
// place among its cluster's queries with one atomic (plan_count); with the
// candidate lists numbered per query (plan_query, qbase) and the items numbered
// per cluster in order of decreasing size (item_first), the pair writes its own
// query slots of its cluster's items (plan_fill), so no query list is sorted or
// scattered in between.  16,384 queries x 256 slots over 4,096 lists: 0.40 ms in
// eight launches before, 0.15 ms in four now.  Up to kSmallPairs pairs run all of it in
// one block (plan_small_kernel), which is bound by the latency of its five
// phases instead of by launches.
// ---------------------------------------------------------------------------
struct PlanPair {
    int64_t q;
    int slot, c, nr;            // validated cluster (-1: none) and its row ranges
};
__device__ __forceinline__ PlanPair plan_pair(const PlanArgs& p, int64_t t) {
    PlanPair r;
    r.q = t / p.maxp;
    r.slot = (int)(t % p.maxp);
    int np = p.npr_in ? p.npr_in[r.q] : p.npr_uniform;
    if (np < 1 || np > p.maxp) {
        if (r.slot == 0) atomicOr(p.status, kStatusBounds);
        np = np < 1 ? 0 : p.maxp;
    }
    if (r.slot == 0) p.npr[r.q] = np;
    r.c = -1;
    r.nr = 0;
    if (r.slot < np) {
        r.c = p.probe[r.q * p.probe_stride + r.slot];
        if (r.c < 0 || r.c >= p.nlist) {
            atomicOr(p.status, kStatusBounds);
            r.c = -1;
        }
    }
    return r;
}

// One pair: validation and its place in its cluster.
__device__ __forceinline__ void plan_count_one(const PlanArgs& p, int64_t t, unsigned long long& pairs,
                                               unsigned long long& rows) {
    PlanPair r = plan_pair(p, t);
    if (r.c >= 0) {
        const int64_t size = p.list_off[r.c + 1] - p.list_off[r.c];
        r.nr = (int)((size + p.RR - 1) / p.RR);
        const int pos = atomicAdd(&p.cnt_c[r.c], 1);
        p.slot_pos[t] = pos;
        if (pos == 0) rows += (unsigned long long)size;
        pairs += (unsigned long long)size;
    }
    p.probe_c[t] = r.c;
    if (p.slot_off) p.slot_off[t] = r.nr;                       // (offsets after plan_query)
}
// The block's sums, one atomic a block: a sum's one address takes an atomic a clock.
__device__ __forceinline__ void plan_add_stats(const PlanArgs& p, unsigned long long pairs, unsigned long long rows) {
    __shared__ unsigned long long sum[2];
    if (threadIdx.x < 2) sum[threadIdx.x] = 0ull;
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        rows += __shfl_xor_sync(0xffffffffu, rows, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (pairs) atomicAdd(&sum[0], pairs);
        if (rows) atomicAdd(&sum[1], rows);
    }
    __syncthreads();
    if (threadIdx.x < 2 && sum[threadIdx.x]) atomicAdd(&p.stats[threadIdx.x], sum[threadIdx.x]);
}
__global__ void __launch_bounds__(256) plan_count_kernel(PlanArgs p) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long pairs = 0, rows = 0;
    if (t < p.nq * p.maxp) plan_count_one(p, t, pairs, rows);
    plan_add_stats(p, pairs, rows);
}

// One warp: offsets of a query's (slot, range) candidate lists, and their total.
__device__ __forceinline__ void plan_query_one(const PlanArgs& p, int64_t q, int lane) {
    int run = 0;
    for (int s0 = 0; s0 < p.maxp; s0 += 32) {
        const int sl = s0 + lane;
        const int nr = sl < p.maxp ? p.slot_off[q * p.maxp + sl] : 0;
        const int inc = warp_incl_scan(nr);
        if (sl < p.maxp) p.slot_off[q * p.maxp + sl] = run + inc - nr;
        run += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) {
        p.qtot[q] = run;
        if (p.tq) p.tq[q] = kEmptyKey;
    }
}
__global__ void __launch_bounds__(256) plan_query_kernel(PlanArgs p) {
    const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (q < p.nq) plan_query_one(p, q, threadIdx.x & 31);
}

// Exclusive prefix sums over n values get(i) by one block of 1,024 threads, four
// consecutive values a thread; put(i, prefix) for every i, the total returned.
template <class Get, class Put>
__device__ int64_t block_excl_scan(int64_t n, Get get, Put put, int64_t* wsum, int64_t* carry_s) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int64_t carry = 0;
    for (int64_t base = 0; base < n; base += 4096) {
        const int64_t i0 = base + 4 * t;
        int64_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = i0 + j < n ? get(i0 + j) : 0;
        const int64_t own = v[0] + v[1] + v[2] + v[3];
        int64_t inc = own;                      // inclusive warp scan of the per-thread sums
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const int64_t w = wsum[lane];
            int64_t wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            wsum[lane] = wi - w;                // exclusive prefix of the warp totals
            if (lane == 31) *carry_s = wi;      // chunk total
        }
        __syncthreads();
        int64_t run = carry + wsum[warp] + inc - own;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (i0 + j < n) put(i0 + j, run);
            run += v[j];
        }
        carry += *carry_s;
        __syncthreads();                        // wsum / carry_s are rewritten by the next chunk
    }
    return carry;
}

__device__ __forceinline__ int64_t plan_items_of(const PlanArgs& p, int c) {
    const int64_t size = p.list_off[c + 1] - p.list_off[c];
    const int64_t n = p.cnt_c[c];
    return n > 0 && size > 0 ? ((n + p.QT - 1) / p.QT) * ((size + p.RR - 1) / p.RR) : 0;
}
__device__ void plan_scan_queries(const PlanArgs& p, int64_t* wsum, int64_t* carry) {
    const int64_t tot = block_excl_scan(p.nq, [&](int64_t i) { return p.qtot[i]; },
                                        [&](int64_t i, int64_t v) { p.qbase[i] = v; }, wsum, carry);
    if (threadIdx.x == 0) {
        p.qbase[p.nq] = tot;
        p.stats[4] = (unsigned long long)tot;
    }
}
// items in order of decreasing cluster size, so that long items start first
__device__ void plan_scan_items(const PlanArgs& p, int64_t* wsum, int64_t* carry) {
    const int64_t tot = block_excl_scan(p.nlist, [&](int64_t i) { return plan_items_of(p, p.corder[i]); },
                                        [&](int64_t i, int64_t v) { p.item_first[p.corder[i]] = (int32_t)v; }, wsum, carry);
    if (threadIdx.x == 0) {
        *p.n_items = tot;
        *p.work_ctr = 0u;
        p.stats[5] = (unsigned long long)tot;
    }
}
__global__ void __launch_bounds__(1024) plan_scan_kernel(PlanArgs p) {
    __shared__ int64_t wsum[32], carry;
    if (blockIdx.x == 0) plan_scan_queries(p, wsum, &carry);
    else plan_scan_items(p, wsum, &carry);
}

// One pair: its query slot in its cluster's items, for every row range; the pair
// in a chunk's first slot also writes the items themselves.
__device__ __forceinline__ void plan_fill_one(const PlanArgs& p, int64_t t) {
    const int c = p.probe_c[t];
    if (c < 0) return;
    const int64_t size = p.list_off[c + 1] - p.list_off[c];
    const int nr = (int)((size + p.RR - 1) / p.RR);
    if (nr == 0) return;
    const int pos = p.slot_pos[t], ch = pos / p.QT, slot = pos - ch * p.QT;
    const int nch = (p.cnt_c[c] + p.QT - 1) / p.QT, nqi = min(p.QT, p.cnt_c[c] - ch * p.QT);
    const int64_t q = t / p.maxp;
    const int64_t L0 = p.qbase[q] + p.slot_off[t];
    const int dq = __float_as_int(p.dqc[t]);
    for (int r = 0; r < nr; ++r) {
        const int64_t it = (int64_t)p.item_first[c] + (int64_t)r * nch + ch;    // row range first: a range's chunks run together
        if (!ERQ_DCHECK(it >= 0 && it < p.ck.items, p.ck.status, 9)) return;
        const int64_t L = L0 + r;
        p.itemq[it * p.QT + slot] = make_int4((int)q, dq, (int)(uint32_t)L, (int)(L >> 32));
        if (slot == 0) {
            const int64_t r0 = (int64_t)r * p.RR, rb0 = p.poff[c] + r0;
            const int nrows = (int)(imin64(size, r0 + p.RR) - r0);
            p.itemd[it] = make_int4((int)(uint32_t)rb0, (int)(rb0 >> 32), nrows, nqi);
            if (p.items) p.items[it] = make_int4(c, nqi, r, 0);
            if (p.count_blocks) {
                const unsigned long long nblk = (unsigned long long)((nrows + 127) / 128);
                atomicAdd(&p.stats[2], nblk);
                atomicAdd(&p.stats[3], nblk * (unsigned long long)(nqi <= 16 ? 16 : (nqi + 15) & ~15));
            }
        }
    }
}
__global__ void __launch_bounds__(256) plan_fill_kernel(PlanArgs p) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < p.nq * p.maxp) plan_fill_one(p, t);
}

// All of the above for few pairs, one block.
__global__ void __launch_bounds__(1024) plan_small_kernel(PlanArgs p, int32_t* inter_cnt, int64_t nlists) {
    __shared__ int64_t wsum[32], carry;
    const int64_t pairs = p.nq * p.maxp;
    for (int64_t i = threadIdx.x; i < p.nlist; i += 1024) p.cnt_c[i] = 0;
    for (int64_t i = threadIdx.x; i < nlists; i += 1024) inter_cnt[i] = 0;
    if (threadIdx.x < 8) p.stats[threadIdx.x] = 0ull;
    __syncthreads();
    unsigned long long np = 0, nr = 0;
    for (int64_t t = threadIdx.x; t < pairs; t += 1024) plan_count_one(p, t, np, nr);
    plan_add_stats(p, np, nr);
    __syncthreads();
    for (int64_t q = threadIdx.x >> 5; q < p.nq; q += 32) plan_query_one(p, q, threadIdx.x & 31);
    plan_scan_items(p, wsum, &carry);          // (reads the counts only)
    __syncthreads();
    plan_scan_queries(p, wsum, &carry);
    __syncthreads();
    for (int64_t t = threadIdx.x; t < pairs; t += 1024) plan_fill_one(p, t);
}

// Exclusive scan of n int64 (out has n + 1 entries, out[n] = total).
__global__ void __launch_bounds__(1024) excl_scan_i64_kernel(const int64_t* __restrict__ in, int64_t* __restrict__ out,
                                                             int64_t n) {
    __shared__ int64_t wsum[32], carry;
    const int64_t tot = block_excl_scan(n, [&](int64_t i) { return in[i]; }, [&](int64_t i, int64_t v) { out[i] = v; },
                                        wsum, &carry);
    if (threadIdx.x == 0) out[n] = tot;
}

// ---------------------------------------------------------------------------
// FP32 CUDA-core scan: Eq. 3.3's <2 ybar - (2^B - 1), q'> by FFMA.
// Item = (cluster c, query chunk, row range).  Tile: 64 queries x 128 rows,
// 128 threads with 8 x 8 outputs each (queries 4 tq .. 4 tq + 3 and 32 + 4 tq
// .. + 3, rows 4 tr .. + 3 and 64 + 4 tr .. + 3: four 16-byte shared loads per
// 64 FFMA; an item of at most 32 queries skips the upper half), K step 32.  The operands of step k + 1 are loaded from global
// memory into registers while step k is multiplied out of the other shared
// buffer (one barrier per step); codes are widened to 2 ybar - (2^B - 1) as
// they are stored.  After a tile the estimates go to shared memory (over the
// operand buffers) and 64 threads (one per query) push those that beat their
// heap's root through the query's max-heap of the k' best (estimate, id) keys.
// ---------------------------------------------------------------------------
constexpr int SC_QT = 64, SC_RB = 128, SC_BK = 32, SC_THREADS = 128;
constexpr int SC_QS = SC_QT + 4, SC_CS = SC_RB + 4;      // padded rows of the transposed operand tiles
constexpr int SC_OPS = 2 * SC_BK * (SC_QS + SC_CS) * 4;  // two buffers of both operands, bytes
constexpr int SC_EST = SC_QT * (SC_RB + 1) * 4;          // estimate tile (aliases the operand buffers)
static_assert(SC_EST <= SC_OPS, "estimate tile fits the operand buffers");

struct ScanArgs {
    const float* Qrot;          // [nq][D]
    const uint8_t* codes;       // [N][D]
    const float* g_const;       // [N]
    const float* f_res;         // [N]
    const int64_t* list_off;    // [nlist+1]
    const int64_t* list_ids;    // [N]
    const int4* items;          // {cluster, queries, row range, 0}
    const int4* itemq;          // [items][64] {query row, dqc bits, output list lo, hi}
    const int64_t* n_items;     // device scalar
    uint64_t* inter;            // [L][kp]
    int32_t* inter_cnt;         // [L]
    int64_t nq, N;              // extents of Qrot and of the stored rows (device-side checks)
    unsigned int* work_ctr;     // items taken after the first grid-size ones (zero at launch)
    int maxp, D, B, kp, RR, nlist;
    int ip;                     // inner-product metric: est = -<c, q_r> + (f_res / 4) <2 ybar, q'>
    DevChecks ck;
};

// Register-staged operands of one K step: 16 query values of query (tid & 63)
// at k0 + 16 (tid >> 6), and the 32 codes of row tid at k0 (CB bytes each:
// 1 for B <= 8, 2 for B = 9).
template <int CB>
struct Fp32Stage {
    float4 q[4];
    uint4 c[2 * CB];
};

template <int CB>
__device__ __forceinline__ void fp32_load(Fp32Stage<CB>& st, const float* qrow, const uint8_t* crow, int k0, int tid) {
    const int kq = (tid >> 6) * 16;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        st.q[j] = qrow ? __ldg(reinterpret_cast<const float4*>(qrow + k0 + kq) + j) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 2 * CB; ++j)
        st.c[j] = crow ? __ldg(reinterpret_cast<const uint4*>(crow + (int64_t)k0 * CB) + j) : make_uint4(0u, 0u, 0u, 0u);
}

template <int CB>
__device__ __forceinline__ void fp32_store(const Fp32Stage<CB>& st, float* qs, float* cs, int tid, float off) {
    const int qi = tid & 63, kq = (tid >> 6) * 16;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        qs[(kq + 4 * j + 0) * SC_QS + qi] = st.q[j].x;
        qs[(kq + 4 * j + 1) * SC_QS + qi] = st.q[j].y;
        qs[(kq + 4 * j + 2) * SC_QS + qi] = st.q[j].z;
        qs[(kq + 4 * j + 3) * SC_QS + qi] = st.q[j].w;
    }
    if constexpr (CB == 1) {
        const uint32_t w[8] = {st.c[0].x, st.c[0].y, st.c[0].z, st.c[0].w, st.c[1].x, st.c[1].y, st.c[1].z, st.c[1].w};
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int b = 0; b < 4; ++b) cs[(4 * j + b) * SC_CS + tid] = fmaf(2.f, (float)((w[j] >> (8 * b)) & 0xffu), -off);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t w[4] = {st.c[j].x, st.c[j].y, st.c[j].z, st.c[j].w};
#pragma unroll
            for (int h = 0; h < 4; ++h)
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    cs[(8 * j + 2 * h + b) * SC_CS + tid] = fmaf(2.f, (float)((w[h] >> (16 * b)) & 0xffffu), -off);
        }
    }
}

// The next work item of a block: the first grid-size items go to the blocks
// in order, the rest to whichever block asks first (items come by decreasing
// list size, so this balances the tail).
__device__ __forceinline__ int64_t fp32_next_item(unsigned int* ctr, int64_t* s_next) {
    __syncthreads();                              // every thread has read the previous value
    if (threadIdx.x == 0) *s_next = (int64_t)gridDim.x + atomicAdd(ctr, 1u);
    __syncthreads();
    return *s_next;
}

template <int CB>
__global__ void __launch_bounds__(SC_THREADS) scan_fp32_kernel(ScanArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    float* ops = reinterpret_cast<float*>(smem);     // buffer b: queries at b * BK * (QS + CS), codes after them
    float (*E)[SC_RB + 1] = reinterpret_cast<float (*)[SC_RB + 1]>(smem);
    uint64_t* heap = reinterpret_cast<uint64_t*>(smem + SC_OPS + 16);                      // [kp][QT]
    __shared__ int64_t s_q[SC_QT];
    __shared__ int64_t s_list[SC_QT];
    __shared__ float s_dqc[SC_QT];
    __shared__ int s_hsize[SC_QT];
    __shared__ float s_g[SC_RB], s_fh[SC_RB];
    __shared__ uint32_t s_id[SC_RB];
    __shared__ int64_t s_next;

    const int tid = threadIdx.x;
    const int tq = tid & 7, tr = tid >> 3;
    const int D = a.D;
    const float off = (float)((1 << a.B) - 1);
    int64_t nitems = *a.n_items;
    if (!ERQ_DCHECK(nitems >= 0 && nitems <= a.ck.items, a.ck.status, 5)) nitems = 0;

    for (int64_t it = blockIdx.x; it < nitems; it = fp32_next_item(a.work_ctr, &s_next)) {
        const int4 item = a.items[it];
        if (!ERQ_DCHECK(item.x >= 0 && item.x < a.nlist, a.ck.status, 5)) continue;   // block-uniform
        const int c = item.x, nqi = item.y;
        const int64_t rb0 = a.list_off[c] + (int64_t)item.z * a.RR;
        const int64_t rb1 = imin64(a.list_off[c + 1], rb0 + a.RR);
        if (tid < SC_QT) {
            s_q[tid] = -1;
            if (tid < nqi) {
                const int4 e = a.itemq[it * SC_QT + tid];
                if (ERQ_DCHECK(e.x >= 0 && e.x < a.nq, a.ck.status, 5)) {
                    s_q[tid] = e.x;
                    s_dqc[tid] = __int_as_float(e.y);
                    s_list[tid] = (int64_t)(uint32_t)e.z | ((int64_t)e.w << 32);
                }
            }
            s_hsize[tid] = 0;
        }
        __syncthreads();
        const int64_t qsel = s_q[tid & 63];
        const float* qrow = qsel >= 0 ? a.Qrot + qsel * D : nullptr;
        for (int64_t r0 = rb0; r0 < rb1; r0 += SC_RB) {
            const int nr = (int)imin64(SC_RB, rb1 - r0);
            const bool row_ok = tid < nr && ERQ_DCHECK(r0 + tid >= 0 && r0 + tid < a.N, a.ck.status, 5);
            if (row_ok) {
                s_g[tid] = a.ip ? 0.f : a.g_const[r0 + tid];
                s_fh[tid] = (a.ip ? 0.25f : 0.5f) * a.f_res[r0 + tid];
                s_id[tid] = (uint32_t)a.list_ids[r0 + tid];
            }
            const uint8_t* crow = row_ok ? a.codes + (r0 + tid) * D * CB : nullptr;
            float acc[8][8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
            Fp32Stage<CB> st;
            fp32_load(st, qrow, crow, 0, tid);
            fp32_store(st, ops, ops + SC_BK * SC_QS, tid, off);
            __syncthreads();
            int buf = 0;
            for (int k0 = 0; k0 < D; k0 += SC_BK, buf ^= 1) {
                const bool more = k0 + SC_BK < D;
                if (more) fp32_load(st, qrow, crow, k0 + SC_BK, tid);
                const float* qs = ops + buf * SC_BK * (SC_QS + SC_CS);
                const float* cs = qs + SC_BK * SC_QS;
                if (nqi > 32) {
#pragma unroll 4
                    for (int kk = 0; kk < SC_BK; ++kk) {
                        const float4 q0 = *reinterpret_cast<const float4*>(qs + kk * SC_QS + tq * 4);
                        const float4 q1 = *reinterpret_cast<const float4*>(qs + kk * SC_QS + 32 + tq * 4);
                        const float4 c0 = *reinterpret_cast<const float4*>(cs + kk * SC_CS + tr * 4);
                        const float4 c1 = *reinterpret_cast<const float4*>(cs + kk * SC_CS + 64 + tr * 4);
                        const float qa[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
                        const float ca[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                        for (int i = 0; i < 8; ++i)
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(qa[i], ca[j], acc[i][j]);
                    }
                } else {                                   // queries 32..63 are padding: half the FMAs
#pragma unroll 4
                    for (int kk = 0; kk < SC_BK; ++kk) {
                        const float4 q0 = *reinterpret_cast<const float4*>(qs + kk * SC_QS + tq * 4);
                        const float4 c0 = *reinterpret_cast<const float4*>(cs + kk * SC_CS + tr * 4);
                        const float4 c1 = *reinterpret_cast<const float4*>(cs + kk * SC_CS + 64 + tr * 4);
                        const float qa[4] = {q0.x, q0.y, q0.z, q0.w};
                        const float ca[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(qa[i], ca[j], acc[i][j]);
                    }
                }
                if (more) {
                    float* nq = ops + (buf ^ 1) * SC_BK * (SC_QS + SC_CS);
                    fp32_store(st, nq, nq + SC_BK * SC_QS, tid, off);
                }
                __syncthreads();
            }
            // estimates to shared memory (the operand buffers are free: the
            // last step ended with a barrier)
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int qi = (i < 4 ? 0 : 32) + tq * 4 + (i & 3), ri = (j < 4 ? 0 : 64) + tr * 4 + (j & 3);
                    float e = INFINITY;
                    if (qi < nqi && ri < nr) e = s_dqc[qi] + s_g[ri] + s_fh[ri] * acc[i][j];
                    E[qi][ri] = e;
                }
            __syncthreads();
            // heap update, one thread per query
            if (tid < nqi && s_q[tid] >= 0) {
                const int q = tid;
                int hs = s_hsize[q];
                const int kp = a.kp;
                uint64_t root = hs > 0 ? heap[q] : 0ull;
                for (int r = 0; r < nr; ++r) {
                    const uint64_t key = make_key(E[q][r], s_id[r]);
                    if (hs < kp) {  // sift up into a max-heap
                        int j = hs++;
                        while (j > 0) {
                            const int p = (j - 1) >> 1;
                            const uint64_t pk = heap[p * SC_QT + q];
                            if (pk >= key) break;
                            heap[j * SC_QT + q] = pk;
                            j = p;
                        }
                        heap[j * SC_QT + q] = key;
                        root = heap[q];
                    } else if (key < root) {  // replace the root, sift down
                        int j = 0;
                        for (;;) {
                            const int l = 2 * j + 1;
                            if (l >= kp) break;
                            int m = l;
                            uint64_t mk = heap[l * SC_QT + q];
                            if (l + 1 < kp) {
                                const uint64_t rk = heap[(l + 1) * SC_QT + q];
                                if (rk > mk) { m = l + 1; mk = rk; }
                            }
                            if (mk <= key) break;
                            heap[j * SC_QT + q] = mk;
                            j = m;
                        }
                        heap[j * SC_QT + q] = key;
                        root = heap[q];
                    }
                }
                s_hsize[q] = hs;
            }
            __syncthreads();
        }
        // write the item's lists
        if (tid < nqi && s_q[tid] >= 0 && ERQ_DCHECK(s_list[tid] >= 0 && s_list[tid] < a.ck.lists, a.ck.status, 4)) {
            const int hs = s_hsize[tid];
            const int64_t L = s_list[tid];
            uint64_t* dst = a.inter + L * a.kp;
            for (int j = 0; j < hs; ++j) dst[j] = heap[j * SC_QT + tid];
            a.inter_cnt[L] = hs;
        }
        __syncthreads();
    }
}

size_t scan_fp32_smem(int kp) { return (size_t)SC_OPS + 16 + (size_t)kp * SC_QT * 8; }

template <int CB>
static int fp32_blocks_per_sm(int kp) {
    int n = 1;
    const size_t smem = scan_fp32_smem(kp);
    if (cudaFuncSetAttribute(scan_fp32_kernel<CB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, scan_fp32_kernel<CB>, SC_THREADS, smem) != cudaSuccess ||
        n < 1)
        return 1;
    return n;
}

int scan_fp32_blocks_per_sm(int kp, int B) { return B > 8 ? fp32_blocks_per_sm<2>(kp) : fp32_blocks_per_sm<1>(kp); }

// ---------------------------------------------------------------------------
// Merge for k' > 32: per query the k' smallest keys over its lists, ascending, by
// one block.  Keys above the query's published threshold (tq, optional: never
// below its k'-th key) do not count.  Where the others fit the sort buffer they
// are sorted; where they do not, one pass counts their values in 2,048 equal
// intervals of their range and only the keys up to the interval of the k'-th are
// sorted; where even these do not fit (many equal values), a running best k' and
// a chunk at a time are.  Bound by the latency of the passes over the lists, a
// warp per list: 100 queries x 79 lists, k' = 100, 79 us with the chunks alone,
// 20 us.  1,024 threads or 256 (launch_merge).
// ---------------------------------------------------------------------------
__device__ void block_bitonic_u64(uint64_t* v, int n) {
    for (int size = 2; size <= n; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = threadIdx.x; i < n / 2; i += blockDim.x) {
                const int lo = 2 * i - (i & (stride - 1));
                const int hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint64_t x = v[lo], y = v[hi];
                if ((x > y) == up) { v[lo] = y; v[hi] = x; }
            }
            __syncthreads();
        }
}

__global__ void __launch_bounds__(1024) merge_kernel(const uint64_t* __restrict__ inter,
                                                     const int32_t* __restrict__ inter_cnt,
                                                     const int64_t* __restrict__ qbase, int kp, int lstride,
                                                     int sortn, const unsigned long long* __restrict__ tq,
                                                     uint64_t* __restrict__ cand, DevChecks ck) {
    extern __shared__ uint64_t buf[];  // [sortn]
    constexpr int BINS = 2048;
    __shared__ int hist[BINS];
    __shared__ uint32_t s_lo[32], s_hi[32];
    __shared__ int s_n[32];
    __shared__ int s_bin, s_end;
    __shared__ int s_fill;
    __shared__ uint64_t s_tau;         // entries >= s_tau cannot enter the top k'
    const int64_t q = blockIdx.x;
    const int64_t L0 = qbase[q], L1 = qbase[q + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const uint64_t top = tq ? (uint64_t)tq[q] : kEmptyKey;
    // every key that counts: a warp per list, the block for long lists
    auto each = [&](auto f) {
        const bool wide = lstride > 512;
        for (int64_t L = L0 + (wide ? 0 : warp); L < L1; L += wide ? 1 : nw) {
            if (!ERQ_DCHECK(L >= 0 && L < ck.lists, ck.status, 0)) break;
            int n = inter_cnt[L];
            if (!ERQ_DCHECK(n >= 0 && n <= lstride, ck.status, 0)) n = 0;
            for (int j = wide ? tid : lane; j < n; j += wide ? blockDim.x : 32) {
                const uint64_t key = inter[L * lstride + j];
                if (key <= top && key != kEmptyKey) f(key);
            }
        }
    };
    for (int i = tid; i < sortn; i += blockDim.x) buf[i] = kEmptyKey;
    for (int i = tid; i < BINS; i += blockDim.x) hist[i] = 0;
    if (tid == 0) s_fill = 0;
    uint32_t lo = 0xffffffffu, hi = 0u;
    int cnt = 0;
    each([&](uint64_t key) {
        lo = min(lo, (uint32_t)(key >> 32));
        hi = max(hi, (uint32_t)(key >> 32));
        ++cnt;
    });
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
        s_n[warp] = cnt;
    }
    __syncthreads();
    int total = 0;
    for (int w = 0; w < nw; ++w) {
        lo = min(lo, s_lo[w]);
        hi = max(hi, s_hi[w]);
        total += s_n[w];
    }
    int take = total, bin = BINS - 1;
    const int shift = hi > lo ? max(0, 21 - __clz(hi - lo)) : 0;   // (hi - lo) >> shift < 2048
    if (total > sortn) {
        each([&](uint64_t key) { atomicAdd(&hist[((uint32_t)(key >> 32) - lo) >> shift], 1); });
        __syncthreads();
        const int per = BINS / blockDim.x;
        int own = 0;
        for (int i = 0; i < per; ++i) own += hist[tid * per + i];
        const int inc = warp_incl_scan(own);
        if (lane == 31) s_n[warp] = inc;                           // (read above before the barrier)
        __syncthreads();
        int run = inc - own;
        for (int w = 0; w < warp; ++w) run += s_n[w];
        for (int i = 0; i < per; ++i) {
            const int c = hist[tid * per + i];
            if (run < kp && run + c >= kp) {
                s_bin = tid * per + i;
                s_end = run + c;
            }
            run += c;
        }
        __syncthreads();
        bin = s_bin;
        take = s_end;
    }
    if (take <= sortn) {
        each([&](uint64_t key) {
            if ((int)(((uint32_t)(key >> 32) - lo) >> shift) <= bin) buf[atomicAdd(&s_fill, 1)] = key;
        });
        __syncthreads();
        int n = 2;
        while (n < take || n < kp) n <<= 1;
        block_bitonic_u64(buf, n);
        for (int j = tid; j < kp; j += blockDim.x) cand[q * kp + j] = buf[j];
        return;
    }
    __syncthreads();
    if (threadIdx.x == 0) { s_fill = kp; s_tau = kEmptyKey; }
    __syncthreads();
    for (int64_t L = L0; L < L1; ++L) {
        if (!ERQ_DCHECK(L >= 0 && L < ck.lists, ck.status, 0)) break;
        int n = inter_cnt[L];
        if (!ERQ_DCHECK(n >= 0 && n <= lstride, ck.status, 0)) n = 0;
        const bool full = s_fill + n > sortn;
        __syncthreads();                   // every thread has read s_fill before any appends to it,
        if (full) {                        // so `full` is uniform
            block_bitonic_u64(buf, sortn);
            for (int i = kp + threadIdx.x; i < sortn; i += blockDim.x) buf[i] = kEmptyKey;
            __syncthreads();
            if (threadIdx.x == 0) { s_fill = kp; s_tau = buf[kp - 1]; }
            __syncthreads();
        }
        const uint64_t tau = s_tau;
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
            const uint64_t key = inter[L * lstride + j];
            if (key < tau) buf[atomicAdd(&s_fill, 1)] = key;
        }
        __syncthreads();
    }
    block_bitonic_u64(buf, sortn);
    for (int j = threadIdx.x; j < kp; j += blockDim.x) cand[q * kp + j] = buf[j];
}

// Merge for k' <= 32: W warps per query (1, 8 or 32), each keeping the k'
// smallest keys it has seen in a sorted 32-entry list across its lanes.  A warp
// takes an equal share of the query's lists, up to 32 at a time, numbers their
// entries through (a scan of the counts) and reads 128 entries at once whatever
// list they are in; entries above the query's published threshold (tq, optional:
// never below its k'-th key) or the warp's k'-th key are dropped before the sort.
// Bound by the latency of its loads and sorts: one query over 313 lists took one
// warp 170 us, 8 warps 26 us, 32 warps 7 us.
template <int W>
__global__ void __launch_bounds__(W == 32 ? 1024 : 256) merge32_kernel(
    const uint64_t* __restrict__ inter, const int32_t* __restrict__ inter_cnt, const int64_t* __restrict__ qbase,
    int64_t nq, int kp, int lstride, const unsigned long long* __restrict__ tq, uint64_t* __restrict__ cand,
    DevChecks ck) {
    __shared__ uint64_t part[W > 1 ? W * 32 : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t q = W > 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * 8 + warp;
    if (W == 1 && q >= nq) return;
    const int64_t L0 = qbase[q], L1 = qbase[q + 1];
    const int per = W > 1 ? (int)imin64(32, (L1 - L0 + W - 1) / W) : 32;       // (0 without lists)
    const uint64_t top = tq ? (uint64_t)tq[q] : kEmptyKey;
    uint64_t list = kEmptyKey, th = kEmptyKey;
    for (int64_t Lb = L0 + (W > 1 ? per * warp : 0); Lb < L1; Lb += per * W) {
        if (!ERQ_DCHECK(Lb >= 0 && L1 <= ck.lists, ck.status, 1)) break;
        const int nl = (int)imin64(per, L1 - Lb);
        int n = lane < nl ? inter_cnt[Lb + lane] : 0;
        if (!ERQ_DCHECK(n >= 0 && n <= lstride, ck.status, 1)) n = 0;
        const int incl = warp_incl_scan(n), total = __shfl_sync(0xffffffffu, incl, 31);
        for (int e0 = 0; e0 < total; e0 += 128) {
            uint64_t key[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                key[u] = kEmptyKey;
                if (e0 + 32 * u >= total) continue;
                const int e = e0 + 32 * u + lane;
                int j = 0, before = 0;                                 // lists that end at or before entry e
                if (nl > 1) {                                          // (one list: nothing to number)
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        if (__shfl_sync(0xffffffffu, incl, j + o - 1) <= e) j += o;
                    j = min(j, 31);                                    // (entries past the last)
                    const int prev = __shfl_sync(0xffffffffu, incl, max(j - 1, 0));
                    before = j > 0 ? prev : 0;
                }
                if (e < total) key[u] = inter[(Lb + j) * lstride + (e - before)];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e0 + 32 * u >= total) break;
                const bool pass = key[u] <= top && key[u] < th;
                if (!__any_sync(0xffffffffu, pass)) continue;
                list = ws_merge32(list, ws_sort32(pass ? key[u] : kEmptyKey, lane), lane);
                th = ws_shfl(list, kp - 1);
            }
        }
    }
    if (W > 1) {
        part[warp * 32 + lane] = list;
#pragma unroll 1
        for (int h = W / 2; h > 0; h >>= 1) {
            __syncthreads();
            if (warp < h) {
                list = ws_merge32(list, part[(warp + h) * 32 + lane], lane);
                part[warp * 32 + lane] = list;
            }
        }
        if (warp != 0) return;
    }
    if (lane < kp) cand[q * kp + lane] = list;
}

// ---------------------------------------------------------------------------
// Re-rank: exact squared distances (or inner products, ranked by -<o, q>) of
// the k' candidates (FP32), top-k; inner products are reported with their sign.
// Also writes cand_ids / cand_est when requested.  One block per query.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) rerank_kernel(const uint64_t* __restrict__ cand, int kp, const float* __restrict__ X,
                                                     const float* __restrict__ Q, int D, int k, int do_rerank,
                                                     int ip, int sortn, int64_t* __restrict__ ids,
                                                     float* __restrict__ dists, int64_t* __restrict__ cand_ids,
                                                     float* __restrict__ cand_est, DevChecks ck) {
    const float sgn = ip ? -1.f : 1.f;       // keys hold -<o, q> for the inner-product metric
    extern __shared__ uint64_t keys[];  // [sortn]
    const int64_t q = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t* cq = cand + q * kp;
    if (cand_ids)
        for (int j = threadIdx.x; j < kp; j += blockDim.x) {
            const uint64_t kk = cq[j];
            cand_ids[q * kp + j] = kk == kEmptyKey ? -1 : (int64_t)key_id(kk);
            cand_est[q * kp + j] = sgn * (kk == kEmptyKey ? INFINITY : key_value(kk));
        }
    if (!do_rerank) {
        for (int j = threadIdx.x; j < k; j += blockDim.x) {
            const uint64_t kk = j < kp ? cq[j] : kEmptyKey;
            ids[q * k + j] = kk == kEmptyKey ? -1 : (int64_t)key_id(kk);
            dists[q * k + j] = sgn * (kk == kEmptyKey ? INFINITY : key_value(kk));
        }
        return;
    }
    for (int i = threadIdx.x; i < sortn; i += blockDim.x) keys[i] = kEmptyKey;
    __syncthreads();
    const float* qr = Q + q * D;
    for (int j = warp; j < kp; j += blockDim.x / 32) {
        const uint64_t kk = cq[j];
        if (kk == kEmptyKey) continue;
        const uint32_t id = key_id(kk);
        if (!ERQ_DCHECK((int64_t)id < ck.rows, ck.status, 2)) continue;
        const float* x = X + (int64_t)id * D;
        float s = 0.f;
        constexpr int RU = 8;                 // float4 loads per lane in flight
        for (int t0 = 0; t0 < D; t0 += 128 * RU) {
            float4 a[RU], b[RU];
#pragma unroll
            for (int u = 0; u < RU; ++u) {
                const int t = t0 + 128 * u + lane * 4;
                if (t < D) {
                    a[u] = *reinterpret_cast<const float4*>(x + t);
                    b[u] = *reinterpret_cast<const float4*>(qr + t);
                }
            }
#pragma unroll
            for (int u = 0; u < RU; ++u) {
                if (t0 + 128 * u + lane * 4 < D) {
                    if (ip) {
                        s = fmaf(a[u].x, b[u].x, s);
                        s = fmaf(a[u].y, b[u].y, s);
                        s = fmaf(a[u].z, b[u].z, s);
                        s = fmaf(a[u].w, b[u].w, s);
                    } else {
                        const float d0 = a[u].x - b[u].x, d1 = a[u].y - b[u].y, d2 = a[u].z - b[u].z,
                                    d3 = a[u].w - b[u].w;
                        s = fmaf(d0, d0, s);
                        s = fmaf(d1, d1, s);
                        s = fmaf(d2, d2, s);
                        s = fmaf(d3, d3, s);
                    }
                }
            }
        }
        s = warp_sum(s);
        if (lane == 0) keys[j] = make_key(sgn * s, id);
    }
    __syncthreads();
    block_bitonic_u64(keys, sortn);
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        const uint64_t kk = keys[j];
        ids[q * k + j] = kk == kEmptyKey ? -1 : (int64_t)key_id(kk);
        dists[q * k + j] = sgn * (kk == kEmptyKey ? INFINITY : key_value(kk));
    }
}

// ---------------------------------------------------------------------------
// Estimates of explicit pairs (FP32), in two forms of the same sums in the same
// order (launch_estimate).  estimate_kernel: a block takes up to 128 of a query's ids:
// q_r and P^T q_r stay in shared memory, the ids' rows and clusters are looked
// up once, and each warp streams its pairs' centroid and code rows through two
// shared-memory slots of its own with bulk copies (16-byte aligned: D is a
// multiple of 64), so that loads run ahead of the arithmetic without holding
// registers.  Bound by the L2 reads of the gathered rows (4 D + D bytes a pair;
// 4,096 x 100 pairs at D = 1024 are 2.1 GB): 0.71 -> 0.29 ms
// (7.3 TB/s) against one warp per pair reading both query rows as well; the same
// loads held in registers, eight in flight per lane, took 0.83.
// ---------------------------------------------------------------------------
constexpr int EST_PAIRS = 128;

// 2 ybar_u - (2^B - 1) of four consecutive coordinates; a code is made a float by
// placing it in the mantissa of 2^23.
template <int CB>
__device__ __forceinline__ float4 codes4(const uint8_t* p, float off) {
    uint32_t u[4];
    if constexpr (CB == 1) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = __byte_perm(w, 0x4B000000u, 0x7440u + (uint32_t)i);
    } else {
        const uint2 w = *reinterpret_cast<const uint2*>(p);
        u[0] = __byte_perm(w.x, 0x4B000000u, 0x7410u); u[1] = __byte_perm(w.x, 0x4B000000u, 0x7432u);
        u[2] = __byte_perm(w.y, 0x4B000000u, 0x7410u); u[3] = __byte_perm(w.y, 0x4B000000u, 0x7432u);
    }
    float f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = fmaf(2.f, __uint_as_float(u[i]) - 8388608.f, -off);
    return make_float4(f[0], f[1], f[2], f[3]);
}

// Four coordinates of a pair: into ||q_r - c||^2 (or <c, q_r>) and <2 ybar, q'>.
__device__ __forceinline__ void estimate_add(const float4 cv, const float4 yv, const float4 x, const float4 xr, int ipm,
                                             float4& dq, float4& ip) {
    if (ipm) {
        dq.x = fmaf(cv.x, x.x, dq.x);
        dq.y = fmaf(cv.y, x.y, dq.y);
        dq.z = fmaf(cv.z, x.z, dq.z);
        dq.w = fmaf(cv.w, x.w, dq.w);
    } else {
        const float d0 = x.x - cv.x, d1 = x.y - cv.y, d2 = x.z - cv.z, d3 = x.w - cv.w;
        dq.x = fmaf(d0, d0, dq.x);
        dq.y = fmaf(d1, d1, dq.y);
        dq.z = fmaf(d2, d2, dq.z);
        dq.w = fmaf(d3, d3, dq.w);
    }
    ip.x = fmaf(yv.x, xr.x, ip.x);
    ip.y = fmaf(yv.y, xr.y, ip.y);
    ip.z = fmaf(yv.z, xr.z, ip.z);
    ip.w = fmaf(yv.w, xr.w, ip.w);
}
// Squared distance ||q_r - c||^2 + g + (f_res/2) <2 ybar, q'>, or inner product
// <c, q_r> - (f_res/4) <2 ybar, q'>.
__device__ __forceinline__ float estimate_of(float dq, float ip, int64_t row, const float* __restrict__ g_const,
                                             const float* __restrict__ f_res, int ipm) {
    return ipm ? dq - 0.25f * f_res[row] * ip : dq + g_const[row] + 0.5f * f_res[row] * ip;
}

template <int CB>
__global__ void __launch_bounds__(256) estimate_kernel(const float* __restrict__ Q, const float* __restrict__ Qrot,
                                                       const int64_t* __restrict__ ids, int64_t nq, int nc, int64_t N,
                                                       const int64_t* __restrict__ row_of,
                                                       const int32_t* __restrict__ cl_of_row,
                                                       const float* __restrict__ C, const uint8_t* __restrict__ codes,
                                                       const float* __restrict__ g_const,
                                                       const float* __restrict__ f_res, int D, int B, int ipm,
                                                       float* __restrict__ est, uint32_t* __restrict__ status,
                                                       int jbase) {
    extern __shared__ __align__(16) float es[];       // q_r [D], P^T q_r [D], then two row slots per warp
    __shared__ int64_t s_row[EST_PAIRS];               // stored row, -1: absent id
    __shared__ int32_t s_cl[EST_PAIRS];
    __shared__ uint64_t s_bar[16];
    __shared__ int s_abort;
    const int64_t q = blockIdx.x;
    const int j0 = jbase + blockIdx.y * EST_PAIRS, nj = min(EST_PAIRS, nc - j0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const uint32_t slot_bytes = (uint32_t)D * (4 + CB);
    unsigned char* ring = reinterpret_cast<unsigned char*>(es + 2 * D) + (size_t)warp * 2 * slot_bytes;
    if (threadIdx.x < 2 * nw) tc::mbar_init(tc::smem_u32(s_bar + threadIdx.x), 1);
    if (threadIdx.x == 0) s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int k = threadIdx.x * 4; k < D; k += blockDim.x * 4) {
        *reinterpret_cast<float4*>(es + k) = *reinterpret_cast<const float4*>(Q + q * D + k);
        *reinterpret_cast<float4*>(es + D + k) = *reinterpret_cast<const float4*>(Qrot + q * D + k);
    }
    for (int j = threadIdx.x; j < nj; j += blockDim.x) {
        const int64_t id = ids[q * nc + j0 + j];
        if (id >= N) atomicOr(status, kStatusBounds);
        const int64_t row = id < 0 || id >= N ? -1 : row_of[id];
        s_row[j] = row;
        s_cl[j] = row >= 0 ? cl_of_row[row] : 0;
    }
    __syncthreads();
    const uint32_t bar0 = tc::smem_u32(s_bar + 2 * warp);
    auto issue = [&](int j, int slot) {                // (an absent id fetches row 0 and ignores it)
        const int64_t row = s_row[j] < 0 ? 0 : s_row[j];
        const uint32_t dst = tc::smem_u32(ring + slot * slot_bytes), bar = bar0 + 8 * slot;
        tc::mbar_arrive_expect_tx(bar, slot_bytes);
        tc::bulk_load(dst, C + (int64_t)s_cl[j] * D, (uint32_t)D * 4, bar);
        tc::bulk_load(dst + D * 4, codes + row * D * CB, (uint32_t)D * CB, bar);
    };
    if (lane == 0) {
        if (warp < nj) issue(warp, 0);
        if (warp + nw < nj) issue(warp + nw, 1);
    }
    const float off = (float)((1 << B) - 1);
    for (int i = 0, j = warp; j < nj; ++i, j += nw) {
        const int slot = i & 1;
        if (!tc::mbar_wait_warp(bar0 + 8 * slot, (i >> 1) & 1, &s_abort)) {
            if (lane == 0) atomicOr(status, kStatusTimeout);
            tc::mbar_wait_drain(bar0 + 8 * slot, (i >> 1) & 1);     // (bounded) the copies in flight land first
            if (j + nw < nj) tc::mbar_wait_drain(bar0 + 8 * (slot ^ 1), ((i + 1) >> 1) & 1);
            break;
        }
        const float* c = reinterpret_cast<const float*>(ring + slot * slot_bytes);
        const uint8_t* code = ring + slot * slot_bytes + D * 4;
        float4 dq = make_float4(0.f, 0.f, 0.f, 0.f), ip = dq;
#pragma unroll 4
        for (int k = lane * 4; k < D; k += 128) {
            estimate_add(*reinterpret_cast<const float4*>(c + k), codes4<CB>(code + k * CB, off),
                         *reinterpret_cast<const float4*>(es + k), *reinterpret_cast<const float4*>(es + D + k), ipm, dq, ip);
        }
        __syncwarp();                                  // the slot has been read
        if (lane == 0 && j + 2 * nw < nj) issue(j + 2 * nw, slot);
        const float dqs = warp_sum((dq.x + dq.y) + (dq.z + dq.w)), ips = warp_sum((ip.x + ip.y) + (ip.z + ip.w));
        if (lane == 0) {
            const int64_t row = s_row[j];
            est[q * nc + j0 + j] = row < 0 ? NAN : estimate_of(dqs, ips, row, g_const, f_res, ipm);
        }
    }
}

// W lanes per pair (16 for D = 64, one coordinate group a lane; else a warp), both
// rows and both query rows read as they are: the form for few pairs a query, where
// staging costs more than it saves, and for long rows.
template <int CB, int W>
__global__ void __launch_bounds__(256) estimate_pair_kernel(const float* __restrict__ Q, const float* __restrict__ Qrot,
                                                            const int64_t* __restrict__ ids, int64_t nq, int nc, int64_t N,
                                                            const int64_t* __restrict__ row_of,
                                                            const int32_t* __restrict__ cl_of_row,
                                                            const float* __restrict__ C,
                                                            const uint8_t* __restrict__ codes,
                                                            const float* __restrict__ g_const,
                                                            const float* __restrict__ f_res, int D, int B, int ipm,
                                                            float* __restrict__ est, uint32_t* __restrict__ status) {
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / W;
    const int lane = threadIdx.x & (W - 1);
    if (w >= nq * nc) return;
    const int64_t q = w / nc, id = ids[w];
    if (id < 0 || id >= N) {
        if (lane == 0) {
            est[w] = NAN;
            if (id >= N) atomicOr(status, kStatusBounds);
        }
        return;
    }
    const int64_t row = row_of[id];
    const float* c = C + (int64_t)cl_of_row[row] * D;
    const uint8_t* code = codes + row * D * CB;
    const float *x = Q + q * D, *xr = Qrot + q * D;
    const float off = (float)((1 << B) - 1);
    float4 dq = make_float4(0.f, 0.f, 0.f, 0.f), ip = dq;
#pragma unroll 4
    for (int k = lane * 4; k < D; k += 4 * W)
        estimate_add(*reinterpret_cast<const float4*>(c + k), codes4<CB>(code + k * CB, off),
                     *reinterpret_cast<const float4*>(x + k), *reinterpret_cast<const float4*>(xr + k), ipm, dq, ip);
    float dqs = (dq.x + dq.y) + (dq.z + dq.w), ips = (ip.x + ip.y) + (ip.z + ip.w);
    const unsigned group = W == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);   // (the other half may have left)
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
        dqs += __shfl_xor_sync(group, dqs, o);
        ips += __shfl_xor_sync(group, ips, o);
    }
    if (lane == 0) est[w] = estimate_of(dqs, ips, row, g_const, f_res, ipm);
}

// ---------------------------------------------------------------------------
// Backward gather: per query
//   V[q]  = sum_j g_j f_res,j ybar_j          (rotated space)
//   Wv[q] = 2 (G q_r - sum_j g_j c_j),  G = sum_j g_j
// then grad_Q = V P^T + Wv (one GEMM).  A block takes one query and up to 1,024
// coordinates, four a thread; the candidates' rows, clusters and weights are
// looked up once, a producer warp streams their centroid and code rows through
// BG_RING shared-memory stages with bulk copies, and the threads add them in
// order.  Bound by the same gathered L2 reads as the estimates: 4,096 x 100
// at D = 1024, 1.05 -> 0.28 ms (7.4 TB/s) against a walk that chased id -> row ->
// codes for every coordinate.
// ---------------------------------------------------------------------------
constexpr int BG_STAGE = 128, BG_RING = 8, BG_COLS = 1024;

template <int CB>
__global__ void __launch_bounds__(288) backward_gather_kernel(const float* __restrict__ Q,
                                                              const int64_t* __restrict__ ids,
                                                              const float* __restrict__ gs, int nc, int64_t N,
                                                              const int64_t* __restrict__ row_of,
                                                              const int32_t* __restrict__ cl_of_row,
                                                              const float* __restrict__ C,
                                                              const uint8_t* __restrict__ codes,
                                                              const float* __restrict__ f_res, int D, int B,
                                                              int ipm, float* __restrict__ V, float* __restrict__ Wv,
                                                              uint32_t* __restrict__ status) {
    // squared distance: d est / d q_r = 2 (q_r - c) + f_res P ybar;
    // inner product:    d est / d q_r = c - (f_res / 2) P ybar
    extern __shared__ __align__(16) unsigned char bg_ring[];   // BG_RING x {cols floats, cols codes}
    __shared__ int64_t s_row[BG_STAGE];
    __shared__ int32_t s_cl[BG_STAGE];
    __shared__ float2 s_w[BG_STAGE];                   // {g_j f_res,j (or -g_j f_res,j / 2), g_j}; 0 for absent ids
    __shared__ uint64_t s_bar[2 * BG_RING];            // full, empty
    __shared__ int s_abort;
    const int64_t q = blockIdx.x;
    const int k0 = blockIdx.y * BG_COLS, cols = min(BG_COLS, D - k0);   // (multiples of 64)
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x >> 5) - 1;   // warp nw: producer
    const int t = threadIdx.x * 4;                     // this thread's coordinates k0 + t ..
    const bool on = warp < nw && t < cols;
    const uint32_t st_bytes = (uint32_t)cols * (4 + CB);
    const uint32_t full0 = tc::smem_u32(s_bar), empty0 = tc::smem_u32(s_bar + BG_RING);
    if (threadIdx.x < BG_RING) {
        tc::mbar_init(full0 + 8 * threadIdx.x, 1);
        tc::mbar_init(empty0 + 8 * threadIdx.x, nw);
    }
    if (threadIdx.x == 0) s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    const float off = (float)((1 << B) - 1);
    const float fs = ipm ? -0.5f : 1.f;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f), wc = v;
    float G = 0.f;
    uint32_t it = 0;                                   // candidates before this staging pass
    bool ok = true;
    for (int j0 = 0; j0 < nc; j0 += BG_STAGE) {
        const int nj = min(BG_STAGE, nc - j0);
        __syncthreads();
        for (int j = threadIdx.x; j < nj; j += blockDim.x) {
            const int64_t id = ids[q * nc + j0 + j];
            const bool in = id >= 0 && id < N;
            if (id >= N && blockIdx.y == 0) atomicOr(status, kStatusBounds);
            const int64_t row = in ? row_of[id] : 0;
            const float g = in ? gs[q * nc + j0 + j] : 0.f;
            s_row[j] = row;
            s_cl[j] = in ? cl_of_row[row] : 0;
            s_w[j] = make_float2(in ? g * (fs * f_res[row]) : 0.f, g);
        }
        __syncthreads();
        if (warp == nw) {
            for (int j = 0; j < nj && ok; ++j) {
                const uint32_t n = it + j, s = n % BG_RING;
                ok = tc::mbar_wait_warp(empty0 + 8 * s, ((n / BG_RING) & 1) ^ 1, &s_abort);
                if (ok && tc::elect_one()) {
                    const uint32_t dst = tc::smem_u32(bg_ring + s * st_bytes), bar = full0 + 8 * s;
                    tc::mbar_arrive_expect_tx(bar, st_bytes);
                    tc::bulk_load(dst, C + (int64_t)s_cl[j] * D + k0, (uint32_t)cols * 4, bar);
                    tc::bulk_load(dst + cols * 4, codes + (s_row[j] * D + k0) * CB, (uint32_t)cols * CB, bar);
                }
                __syncwarp();
            }
        } else {
            for (int j = 0; j < nj && ok; ++j) {
                const uint32_t n = it + j, s = n % BG_RING;
                ok = tc::mbar_wait_warp(full0 + 8 * s, (n / BG_RING) & 1, &s_abort);
                if (!ok) break;
                if (on) {
                    const unsigned char* st = bg_ring + s * st_bytes;
                    const float4 cv = *reinterpret_cast<const float4*>(st + t * 4);
                    const float4 yv = codes4<CB>(st + cols * 4 + t * CB, off);   // 2 ybar
                    const float2 w = s_w[j];
                    v.x = fmaf(w.x, 0.5f * yv.x, v.x);
                    v.y = fmaf(w.x, 0.5f * yv.y, v.y);
                    v.z = fmaf(w.x, 0.5f * yv.z, v.z);
                    v.w = fmaf(w.x, 0.5f * yv.w, v.w);
                    wc.x = fmaf(w.y, cv.x, wc.x);
                    wc.y = fmaf(w.y, cv.y, wc.y);
                    wc.z = fmaf(w.y, cv.z, wc.z);
                    wc.w = fmaf(w.y, cv.w, wc.w);
                    G += w.y;
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(empty0 + 8 * s);
            }
        }
        it += nj;
    }
    if (!ok && lane == 0) atomicOr(status, kStatusTimeout);
    // every copy has landed before the block exits
    if (warp == nw)
        for (uint32_t k = 0; k < BG_RING && k < it; ++k) {
            const uint32_t n = it - 1 - k;
            tc::mbar_wait_drain(full0 + 8 * (n % BG_RING), (n / BG_RING) & 1);
        }
    if (!on) return;
    const int k = k0 + t;
    *reinterpret_cast<float4*>(V + q * D + k) = v;
    if (!ipm) {
        const float* x_ = Q + q * D + k;                // (the caller's rows need no 16-byte alignment here)
        const float4 x = make_float4(x_[0], x_[1], x_[2], x_[3]);
        wc = make_float4(2.f * (G * x.x - wc.x), 2.f * (G * x.y - wc.y), 2.f * (G * x.z - wc.z), 2.f * (G * x.w - wc.w));
    }
    *reinterpret_cast<float4*>(Wv + q * D + k) = wc;
}

// ---------------------------------------------------------------------------
// Host-side launch helpers
// ---------------------------------------------------------------------------
cudaError_t launch_dqc(const float* Q, const float* C, const int32_t* probe, const int32_t* npr, int64_t nq, int maxp,
                       int D, int ip, float* dqc, cudaStream_t s) {
    if (nq <= 0 || maxp <= 0) return cudaSuccess;
    const size_t smem = (size_t)D * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(dqc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    count_launch();
    dqc_kernel<<<(unsigned)nq, 32 * std::min(maxp, 16), smem, s>>>(Q, C, probe, npr, nq, maxp, D, ip, dqc);
    return cudaGetLastError();
}

// The pairs' validation and places (all that the two-stage search needs).
cudaError_t launch_plan_count(const PlanArgs& p, cudaStream_t s) {
    const int64_t pairs = p.nq * p.maxp;
    cudaError_t e;
    if ((e = cudaMemsetAsync(p.cnt_c, 0, sizeof(int32_t) * p.nlist, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(p.stats, 0, 8 * sizeof(unsigned long long), s)) != cudaSuccess) return e;
    count_launch();
    plan_count_kernel<<<(unsigned)ceil_div(pairs, 256), 256, 0, s>>>(p);
    return cudaGetLastError();
}

// Candidate-list offsets, item numbers and their totals.
cudaError_t launch_plan_offsets(const PlanArgs& p, cudaStream_t s) {
    count_launch();
    plan_query_kernel<<<(unsigned)ceil_div(p.nq, 8), 256, 0, s>>>(p);
    count_launch();
    plan_scan_kernel<<<2, 1024, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_plan_fill(const PlanArgs& p, cudaStream_t s) {
    count_launch();
    plan_fill_kernel<<<(unsigned)ceil_div(p.nq * p.maxp, 256), 256, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_plan_small(const PlanArgs& p, int32_t* inter_cnt, int64_t nlists, cudaStream_t s) {
    count_launch();
    plan_small_kernel<<<1, 1024, 0, s>>>(p, inter_cnt, nlists);
    return cudaGetLastError();
}

cudaError_t launch_excl_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s) {
    count_launch();
    excl_scan_i64_kernel<<<1, 1024, 0, s>>>(in, out, n);
    return cudaGetLastError();
}

cudaError_t launch_scan_fp32(const ScanLaunch& L, cudaStream_t s) {
    ScanArgs a;
    a.ck = L.ck;
    a.Qrot = L.Qrot; a.codes = L.codes; a.g_const = L.g_const; a.f_res = L.f_res; a.list_off = L.list_off;
    a.list_ids = L.list_ids; a.items = L.items; a.itemq = L.itemq; a.n_items = L.n_items;
    a.inter = L.inter; a.inter_cnt = L.inter_cnt;
    a.maxp = L.maxp; a.D = L.D; a.B = L.B; a.kp = L.kp; a.RR = L.RR; a.ip = L.ip; a.nlist = L.nlist;
    a.nq = L.nq; a.N = L.N; a.work_ctr = L.work_ctr;
    if (!a.work_ctr) return cudaErrorInvalidValue;
    const size_t smem = scan_fp32_smem(L.kp);
    const bool wide = L.B > 8;                    // 16-bit codes
    cudaError_t e = wide ? cudaFuncSetAttribute(scan_fp32_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                         : cudaFuncSetAttribute(scan_fp32_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (L.grid <= 0) return cudaSuccess;
    if (L.D % SC_BK != 0) return cudaErrorInvalidValue;
    count_launch();
    if (wide) scan_fp32_kernel<2><<<L.grid, SC_THREADS, smem, s>>>(a);
    else scan_fp32_kernel<1><<<L.grid, SC_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// (id, value) pairs <-> candidate keys, for merging and re-ranking candidate
// lists given by the caller (e.g. the lists of several index shards).
// ---------------------------------------------------------------------------
// Empty key for ids < 0 or >= id_limit (id_limit > 0); the inner-product
// metric ranks by -value.  vals may be null (value 0: re-rank by id only).
__global__ void make_keys_kernel(const int64_t* __restrict__ ids, const float* __restrict__ vals, int64_t n,
                                 int64_t id_limit, int neg, uint64_t* __restrict__ keys) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const int64_t id = ids[t];
    const bool empty = id < 0 || id > 0xfffffffell || (id_limit > 0 && id >= id_limit);
    const float v = vals ? (neg ? -vals[t] : vals[t]) : 0.f;
    keys[t] = empty ? kEmptyKey : make_key(v, (uint32_t)id);
}

// Keys -> (id, value): empty keys give -1 and +inf (-inf for the inner-product metric).
__global__ void keys_to_pairs_kernel(const uint64_t* __restrict__ keys, int64_t n, int neg, int64_t* __restrict__ ids,
                                     float* __restrict__ vals) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const uint64_t k = keys[t];
    const float sgn = neg ? -1.f : 1.f;
    ids[t] = k == kEmptyKey ? -1 : (int64_t)key_id(k);
    vals[t] = sgn * (k == kEmptyKey ? INFINITY : key_value(k));
}

// One list per query: counts[q] = m, offsets[q] = q.
__global__ void one_list_per_query_kernel(int64_t nq, int m, int32_t* __restrict__ counts, int64_t* __restrict__ off) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t <= nq) off[t] = t;
    if (t < nq) counts[t] = m;
}

cudaError_t launch_make_keys(const int64_t* ids, const float* vals, int64_t n, int64_t id_limit, int neg,
                             uint64_t* keys, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    make_keys_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(ids, vals, n, id_limit, neg, keys);
    return cudaGetLastError();
}

cudaError_t launch_keys_to_pairs(const uint64_t* keys, int64_t n, int neg, int64_t* ids, float* vals, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    keys_to_pairs_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(keys, n, neg, ids, vals);
    return cudaGetLastError();
}

cudaError_t launch_one_list_per_query(int64_t nq, int m, int32_t* counts, int64_t* off, cudaStream_t s) {
    count_launch();
    one_list_per_query_kernel<<<(unsigned)ceil_div(nq + 1, 256), 256, 0, s>>>(nq, m, counts, off);
    return cudaGetLastError();
}

static int sm_count() {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

int merge_sortn(int kp, int lstride) {
    int sortn = 128;
    while (sortn < 4 * kp || sortn < kp + lstride + 32) sortn <<= 1;
    return sortn;
}

cudaError_t launch_merge(const uint64_t* inter, const int32_t* inter_cnt, const int64_t* qbase, int64_t nq, int kp,
                         int lstride, const unsigned long long* tq, uint64_t* cand, const DevChecks& ck,
                         cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int sms = sm_count();
    if (kp <= 32) {
        count_launch();
        // Eight warps per query where there are lists for them (more than 32 a query)
        // or too few queries to fill the chip with one warp each (1,000 queries x 8 lists:
        // 10.7 us with eight, 12.0 with one; 1,500: 14.1 and 14.2; 2,000: 17.4 and 13.9);
        // a whole block's 32 while each query can have an SM to itself (128 queries x 64
        // lists: 9.7 us with 32, 12.7 with eight; 200: 16.6 and 14.4).
        if (nq <= sms && ck.lists > 32 * nq)
            merge32_kernel<32><<<(unsigned)nq, 1024, 0, s>>>(inter, inter_cnt, qbase, nq, kp, lstride, tq, cand, ck);
        else if (ck.lists > 32 * nq || nq < 10 * sms)
            merge32_kernel<8><<<(unsigned)nq, 256, 0, s>>>(inter, inter_cnt, qbase, nq, kp, lstride, tq, cand, ck);
        else
            merge32_kernel<1><<<(unsigned)ceil_div(nq, 8), 256, 0, s>>>(inter, inter_cnt, qbase, nq, kp, lstride, tq, cand,
                                                                       ck);
        return cudaGetLastError();
    }
    const int sortn = merge_sortn(kp, lstride);
    cudaError_t e = cudaFuncSetAttribute(merge_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sortn * 8);
    if (e != cudaSuccess) return e;
    count_launch();
    // (k' = 100, 64 lists: 300 queries 18.5 us with 1,024 threads, 23.1 with 256; 400: 26.9 and 29.6; 608: 34.0 and 31.4)
    merge_kernel<<<(unsigned)nq, nq <= 3 * sms ? 1024 : 256, sortn * 8, s>>>(inter, inter_cnt, qbase, kp, lstride, sortn, tq, cand, ck);
    return cudaGetLastError();
}

// Exact re-rank for k' <= 32: one block of NW warps per query (eight; 32 while each
// query can have an SM to itself, so that all candidates' rows are fetched at once:
// 128 queries, k' = 20, D = 960: 4.9 -> 3.6 us; 200: 5.2 and 5.9), the query row in
// shared memory; warp
// w computes ||x - q||^2 for candidates w, w + NW, ...
// with each lane keeping up to eight 16-byte loads of the row in flight (the
// first row's loads are issued before the query row is waited for), then warp
// 0 sorts the k' keys (distance, id) and writes the top k.
template <int NW>
__global__ void __launch_bounds__(32 * NW, NW == 8 ? 4 : 1) rerank32_kernel(const uint64_t* __restrict__ cand, int kp,
                                                          const float* __restrict__ X, const float* __restrict__ Q,
                                                          int D, int k, int ip, int64_t* __restrict__ ids,
                                                          float* __restrict__ dists, int64_t* __restrict__ cand_ids,
                                                          float* __restrict__ cand_est, DevChecks ck) {
    const float sgn = ip ? -1.f : 1.f;       // keys hold -<o, q> for the inner-product metric
    extern __shared__ float qrow[];           // [D]
    __shared__ uint64_t keys[32];
    const int64_t q = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t* cq = cand + q * kp;
    constexpr int RU = 8;
    float4 a[RU];
    auto issue = [&](int j, int t0) {
        uint64_t kk = cq[j];
        if (kk != kEmptyKey && !ERQ_DCHECK((int64_t)key_id(kk) < ck.rows, ck.status, 3)) kk = kEmptyKey;
        const float* x = X + (int64_t)(kk == kEmptyKey ? 0u : key_id(kk)) * D;
#pragma unroll
        for (int u = 0; u < RU; ++u) {
            const int t = t0 + 128 * u + lane * 4;
            if (t < D) a[u] = *reinterpret_cast<const float4*>(x + t);
        }
        return kk;
    };
    uint64_t kk = warp < kp ? issue(warp, 0) : kEmptyKey;
    for (int t = threadIdx.x * 4; t < D; t += blockDim.x * 4)
        *reinterpret_cast<float4*>(qrow + t) = *reinterpret_cast<const float4*>(Q + q * D + t);
    if (cand_ids && threadIdx.x < kp) {
        const uint64_t c = cq[threadIdx.x];
        cand_ids[q * kp + threadIdx.x] = c == kEmptyKey ? -1 : (int64_t)key_id(c);
        cand_est[q * kp + threadIdx.x] = sgn * (c == kEmptyKey ? INFINITY : key_value(c));
    }
    __syncthreads();
    for (int j = warp; j < kp; j += NW) {
        if (j != warp) kk = issue(j, 0);
        float s = 0.f;
        for (int t0 = 0; t0 < D; t0 += 128 * RU) {
            if (t0 > 0) issue(j, t0);
#pragma unroll
            for (int u = 0; u < RU; ++u) {
                const int t = t0 + 128 * u + lane * 4;
                if (t < D) {
                    const float4 b = *reinterpret_cast<const float4*>(qrow + t);
                    if (ip) {
                        s = fmaf(a[u].x, b.x, s);
                        s = fmaf(a[u].y, b.y, s);
                        s = fmaf(a[u].z, b.z, s);
                        s = fmaf(a[u].w, b.w, s);
                    } else {
                        const float d0 = a[u].x - b.x, d1 = a[u].y - b.y, d2 = a[u].z - b.z, d3 = a[u].w - b.w;
                        s = fmaf(d0, d0, s);
                        s = fmaf(d1, d1, s);
                        s = fmaf(d2, d2, s);
                        s = fmaf(d3, d3, s);
                    }
                }
            }
        }
        s = warp_sum(s);
        if (lane == 0) keys[j] = kk == kEmptyKey ? kEmptyKey : make_key(sgn * s, key_id(kk));
    }
    __syncthreads();
    if (warp == 0) {
        const uint64_t v = ws_sort32(lane < kp ? keys[lane] : kEmptyKey, lane);
        if (lane < k) {
            ids[q * k + lane] = v == kEmptyKey ? -1 : (int64_t)key_id(v);
            dists[q * k + lane] = sgn * (v == kEmptyKey ? INFINITY : key_value(v));
        }
    }
}

cudaError_t launch_rerank(const uint64_t* cand, int64_t nq, int kp, const float* X, const float* Q, int D, int k,
                          int do_rerank, int ip, int64_t* ids, float* dists, int64_t* cand_ids, float* cand_est,
                          const DevChecks& ck, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    if (do_rerank && kp <= 32) {
        const size_t smem = (size_t)D * sizeof(float);
        // (at most 16 KB of shared memory)
        count_launch();
        if (nq <= sm_count())
            rerank32_kernel<32><<<(unsigned)nq, 1024, smem, s>>>(cand, kp, X, Q, D, k, ip, ids, dists, cand_ids, cand_est, ck);
        else
            rerank32_kernel<8><<<(unsigned)nq, 256, smem, s>>>(cand, kp, X, Q, D, k, ip, ids, dists, cand_ids, cand_est, ck);
        return cudaGetLastError();
    }
    int sortn = 32;
    while (sortn < kp) sortn <<= 1;
    cudaError_t e = cudaFuncSetAttribute(rerank_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sortn * 8);
    if (e != cudaSuccess) return e;
    count_launch();
    rerank_kernel<<<(unsigned)nq, 256, sortn * 8, s>>>(cand, kp, X, Q, D, k, do_rerank, ip, sortn, ids, dists,
                                                       cand_ids, cand_est, ck);
    return cudaGetLastError();
}

cudaError_t launch_estimate(const float* Q, const float* Qrot, const int64_t* ids, int64_t nq, int nc,
                            const erq_index* ix, int ipm, float* est, cudaStream_t s) {
    if (nq <= 0 || nc <= 0) return cudaSuccess;
    // The staged form from 32 ids a query and 65,536 pairs on (262,144 above D = 512),
    // for D = 128 .. 1024: the lanes of a pair take 1.00 to 1.50 of its time there (8,192
    // x 100 at D = 256: 280 and 215 us; at D = 1024: 633 and 546), 0.14 to 1.0 of it for
    // fewer ids or pairs (2,048 x 10 at D = 128: 8 and 13 us), for longer rows (2,048 x
    // 100 at D = 4096: 490 and 775) and at D = 64 (8,192 x 100: 124 and 190), where a
    // block's staging is not shared by enough pairs or leaves too few warps on the SM.
    if (nc < 32 || ix->D == 64 || ix->D > 1024 || nq * nc < (ix->D > 512 ? 262144 : 65536)) {
        count_launch();
        const int w = ix->D == 64 ? 16 : 32;
        const auto kern = ix->B > 8 ? (w == 16 ? estimate_pair_kernel<2, 16> : estimate_pair_kernel<2, 32>)
                                    : (w == 16 ? estimate_pair_kernel<1, 16> : estimate_pair_kernel<1, 32>);
        kern<<<(unsigned)ceil_div(nq * nc * w, 256), 256, 0, s>>>(Q, Qrot, ids, nq, nc, ix->N, ix->row_of, ix->cl_of_row, ix->C,
                                                            ix->codes, ix->g_const, ix->f_res, ix->D, ix->B, ipm, est,
                                                            ix->status);
        return cudaGetLastError();
    }
    constexpr int warps = 8;
    const size_t row = (size_t)ix->D * (4 + code_bytes(ix->B));
    const size_t smem = (size_t)ix->D * 8 + 2 * warps * row;    // (at most 106 KB: two blocks an SM)
    const auto kern = ix->B > 8 ? estimate_kernel<2> : estimate_kernel<1>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int slab = 65535 * EST_PAIRS;               // blockIdx.y holds at most 65,535 groups of pairs
    for (int jb = 0; jb < nc; jb = nc - jb > slab ? jb + slab : nc) {
        count_launch();
        kern<<<dim3((unsigned)nq, (unsigned)ceil_div(std::min(slab, nc - jb), EST_PAIRS)), warps * 32, smem, s>>>(
            Q, Qrot, ids, nq, nc, ix->N, ix->row_of, ix->cl_of_row, ix->C, ix->codes, ix->g_const, ix->f_res, ix->D, ix->B,
            ipm, est, ix->status, jb);
    }
    return cudaGetLastError();
}

cudaError_t launch_backward_gather(const float* Q, const int64_t* ids, const float* gs, int64_t nq, int nc,
                                   const erq_index* ix, int ipm, float* V, float* Wv, cudaStream_t s) {
    if (nq <= 0) return cudaSuccess;
    const int cols = std::min(BG_COLS, ix->D);
    const int threads = (int)ceil_div(cols / 4, 32) * 32 + 32;          // consumers and the producer warp
    const size_t smem = (size_t)BG_RING * cols * (4 + code_bytes(ix->B));
    const auto kern = ix->B > 8 ? backward_gather_kernel<2> : backward_gather_kernel<1>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    count_launch();
    kern<<<dim3((unsigned)nq, (unsigned)ceil_div(ix->D, BG_COLS)), threads, smem, s>>>(
        Q, ids, gs, nc, ix->N, ix->row_of, ix->cl_of_row, ix->C, ix->codes, ix->f_res, ix->D, ix->B, ipm, V, Wv,
        ix->status);
    return cudaGetLastError();
}

}  // namespace erq
