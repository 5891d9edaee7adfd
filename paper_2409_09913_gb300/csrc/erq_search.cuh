// Launch descriptors of the search kernels (k_search.cu, k_scan_tc.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "erq_internal.cuh"

namespace erq {

// Inputs/outputs of the planning kernels (probe lists -> work items).
struct PlanArgs {
    const int32_t* probe;       // [nq][probe_stride]
    int64_t probe_stride;
    const int32_t* npr_in;      // optional [nq]
    int npr_uniform;
    int64_t nq;
    int maxp, nlist, QT, RR;
    const int64_t* list_off;
    const int64_t* poff;        // [nlist+1] padded list offsets
    const int32_t* corder;      // [nlist] clusters by decreasing size
    int32_t* npr;               // [nq] effective nprobe
    int32_t* probe_c;           // [nq][maxp] validated cluster or -1
    int32_t* cnt_c;             // [nlist] queries per cluster
    int32_t* slot_pos;          // [nq][maxp] the pair's place among its cluster's queries
    int32_t* slot_off;          // [nq][maxp] row ranges of the slot's cluster, then its first list within the query
    int64_t* qtot;              // [nq] candidate lists of the query
    int64_t* qbase;             // [nq+1] its first list
    int32_t* item_first;        // [nlist] first work item of the cluster
    int64_t* n_items;           // device scalar
    unsigned int* work_ctr;     // the scan's item counter (zeroed)
    unsigned long long* tq;     // optional [nq] the scan's thresholds (set to all ones)
    int4* itemd;                // [items] {first padded row lo, hi, rows, queries}
    int4* itemq;                // [items][QT] {query row, ||q_r - c||^2 bits, output list lo, hi}
    int4* items;                // optional [items] {cluster, queries, row range, 0} (CUDA-core scan)
    uint32_t* status;
    const float* dqc;           // [nq][maxp] ||q_r - c||^2, or -<q_r, c>, of the pairs
    int count_blocks;           // accumulate stats[2], stats[3]
    DevChecks ck;
    unsigned long long* stats;  // [8]: (query, candidate) pairs, rows of distinct probed clusters, tensor-core row
                                //      blocks, row blocks x padded queries, candidate lists, work items
};
constexpr int64_t kSmallPairs = 2048;   // pairs that plan_small_kernel takes

struct ScanLaunch {
    const float* Qrot;
    const void* Qh;             // FP16 rotated queries (tensor-core path; FP32 precision: their whole-number parts)
    const void* Ql;             // FP32 precision: remainders (scaled by 1 / qscale, as Qh then is)
    const void* Q8;             // e4m3 rotated queries, rows of Dq bytes (kind::f8f6f4 path)
    const float* qscale;        // per-query power-of-two scales of Q8, or of Qh + Ql
    int64_t Dq;
    uint32_t* status;
    int64_t N;
    const uint8_t* codes;
    const float* g_const;
    const float* f_res;
    const int64_t* list_off;
    const int64_t* list_ids;
    const int4* items;
    const int64_t* n_items;
    uint64_t* inter;
    int32_t* inter_cnt;
    uint64_t* spill;            // tensor-core path: continuation of the CTAs' candidate lists
    const int4* itemd;          // tensor-core path: per-item {rb0 lo, rb0 hi, rows, queries}
    const int4* itemq;          // tensor-core path: per-item query slots
    const float4* rowmeta;      // tensor-core path: per padded row {g, f_res/2, id, 0}
    const uint64_t* codes_p;    // tensor-core path: packed B-bit codes, tiled and padded
    int64_t Np;                 // tensor-core path: padded rows
    unsigned long long* tq;     // tensor-core path: [nq] query-wide thresholds (all ones at the start)
    int maxp, D, B, kp, RR, nlist;
    int qn;                     // tensor-core path: queries per work item (32, 64 or 128)
    int64_t nq;                 // tensor-core path: query rows (extent of the gathered query matrix)
    unsigned int* work_ctr;     // tensor-core path: dynamic work-item counter, zero at launch
    unsigned long long wait_ns; // tensor-core path: limit of every bounded device-side wait (0 = default)
    long long stall_stage = -1; // tensor-core path: test stall of the bounded-wait path (-1 = none)
    int grid;
    int ip;                     // inner-product metric (per-row factor f_res / 4, no g; dqc holds -<c, q_r>)
    DevChecks ck;
};

// Two-stage (MSB-first) search, k_two_stage.cu.
struct TwoStageLaunch {
    const int32_t* probe_c;     // [nq][maxp] validated probes (-1: none)
    const float* dqc;           // [nq][maxp] ||q_r - c||^2
    const int64_t* list_off;
    const int64_t* poff;
    const uint64_t* codes_p;
    const float4* rowmeta;      // [Np] {g, f_res / 2, id, 0}
    const float4* meta1;        // [Np] {g1, f1 / 2, err1, 0} (stage-1 factors)
    const float* Qrot;          // [nq][D]
    float* T;                   // [nq][D / 4][16] workspace: plane-word nibble tables
    const int32_t* rbase;       // [nq][maxp] first row of each probe within its query
    const int64_t* qoffr;       // [nq + 1] first row slot of each query
    float* ub;                  // [rows] workspace
    float* lb;                  // [rows] workspace
    float* s1;                  // [rows] workspace
    float* tau;                 // [nq] out: pruning thresholds
    int32_t* scnt;              // [nq] out: survivors
    uint64_t* skey;             // [rows] workspace (also the threshold selection's scratch)
    uint32_t* scratch;          // [rows] u32 scratch (may alias skey)
    uint64_t* cand;             // [nq][kp] out: the k' best survivors' keys, ascending
    int64_t nq;
    int maxp, D, B, kp;
    int64_t max_list;           // rows of the largest list
    float eps0;
};
cudaError_t launch_stage1_factors(const float* R, int64_t r0, int64_t m, int D, int B, const uint8_t* codes,
                                  const float* f_add, const float* Cp, const int32_t* cl_of_row,
                                  const int64_t* list_off, const int64_t* poff, float4* meta1, cudaStream_t s);
cudaError_t launch_two_stage_rows(const int32_t* probe_c, int64_t nq, int maxp, const int64_t* list_off,
                                  int32_t* rbase, int64_t* qrows, cudaStream_t s);
cudaError_t launch_two_stage(const TwoStageLaunch& L, cudaStream_t s);
cudaError_t launch_excl_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s);

cudaError_t launch_dqc(const float* Q, const float* C, const int32_t* probe, const int32_t* npr, int64_t nq, int maxp,
                       int D, int ip, float* dqc, cudaStream_t s);
cudaError_t launch_plan_count(const PlanArgs& p, cudaStream_t s);
cudaError_t launch_plan_offsets(const PlanArgs& p, cudaStream_t s);
cudaError_t launch_plan_fill(const PlanArgs& p, cudaStream_t s);
cudaError_t launch_plan_small(const PlanArgs& p, int32_t* inter_cnt, int64_t nlists, cudaStream_t s);
cudaError_t launch_scan_fp32(const ScanLaunch& L, cudaStream_t s);
size_t scan_fp32_smem(int kp);
int scan_fp32_blocks_per_sm(int kp, int B);   // resident FP32-scan blocks per SM at this k' and code width
int merge_sortn(int kp, int lstride);
cudaError_t launch_make_keys(const int64_t* ids, const float* vals, int64_t n, int64_t id_limit, int neg,
                             uint64_t* keys, cudaStream_t s);
cudaError_t launch_keys_to_pairs(const uint64_t* keys, int64_t n, int neg, int64_t* ids, float* vals, cudaStream_t s);
cudaError_t launch_one_list_per_query(int64_t nq, int m, int32_t* counts, int64_t* off, cudaStream_t s);
cudaError_t launch_merge(const uint64_t* inter, const int32_t* inter_cnt, const int64_t* qbase, int64_t nq, int kp,
                         int lstride, const unsigned long long* tq, uint64_t* cand, const DevChecks& ck,
                         cudaStream_t s);
int scan_list_stride(int precision, int kp, int qn);
int64_t scan_spill_entries(int qn, int grid);
bool scan_tc_shape_ok(int qn, int kp);
cudaError_t launch_scan_layout(const uint8_t* codes, const float* g, const float* f_res, const int64_t* ids,
                               const int64_t* list_off, const int64_t* poff, int nlist, int64_t Np, int D, int B,
                               uint64_t* codes_p, float4* rowmeta, cudaStream_t s);
cudaError_t launch_query_parts(const float* x, int64_t n, int D, int B, __half* hi, __half* lo, float* scale,
                               cudaStream_t s);
cudaError_t launch_quant_e4m3(const float* x, int64_t n, int D, int Dq, int dup, unsigned char* y, float* scale,
                              cudaStream_t s);
cudaError_t launch_rerank(const uint64_t* cand, int64_t nq, int kp, const float* X, const float* Q, int D, int k,
                          int do_rerank, int ip, int64_t* ids, float* dists, int64_t* cand_ids, float* cand_est,
                          const DevChecks& ck, cudaStream_t s);
cudaError_t launch_estimate(const float* Q, const float* Qrot, const int64_t* ids, int64_t nq, int nc,
                            const erq_index* ix, int ipm, float* est, cudaStream_t s);
cudaError_t launch_backward_gather(const float* Q, const int64_t* ids, const float* gs, int64_t nq, int nc,
                                   const erq_index* ix, int ipm, float* V, float* Wv, cudaStream_t s);

}  // namespace erq
