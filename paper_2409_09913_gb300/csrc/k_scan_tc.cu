// Tensor-core code scan (tcgen05, sm_103a): the contraction of Eq. 3.3,
// <2 ybar, q'> for every (query, candidate) pair of a work item, on the
// 5th-generation tensor cores with FP32 accumulation in tensor memory.
//
// A work item is (cluster, up to QN of the queries that probe it, up to RR
// stored rows).  Operands of one MMA (kind::f16, M = 128, N = npad, K = 16):
//   A = 128 stored rows of the cluster, codes expanded to 2*ybar_u - (2^B-1),
//       odd integers in [-511, 511] and therefore exact in FP16, held in
//       tensor memory (row = lane, two FP16 values per column);
//   B = the item's queries (rotated q' in FP16), npad = the query count rounded
//       up to a multiple of 16, K-major, 128-byte swizzled rows gathered from
//       the query matrix by TMA (tile::gather4, four rows per copy).
// Codes are read from a packed, scan-specific copy: every inverted list padded
// to a multiple of 32 rows and stored as [tiles of 32 rows][K blocks of 64]
// [B words][32 rows] of 8 bytes, i.e. exactly B bits per coordinate (the
// layout is given at unpack_codes); the 128 rows of one row block and K block
// are four contiguous 256*B-byte pieces fetched by one TMA load.
//
// The estimate is est = ||q_r - c||^2 + g + (f_res / 2) * acc with g, f_res the
// stored per-row factors, or for the inner-product metric the ranking score
// -<c, q_r> + (f_res / 4) * acc = -(estimated <o_r, q_r>).  The product is
// exact up to the FP16 rounding of q' (relative 2^-11 per element);
// accumulation is FP32.
//
// One persistent CTA per SM takes work items from a global counter (items are
// ordered by decreasing cluster size).  A stage group is up to RP = 2 row
// blocks of 128 rows that share the stage's query tile; a stage is one
// 64-coordinate K block of the group, a unit one row block of a stage.  Units
// are numbered through the CTA's life, and so are row blocks.  Warp roles (28
// warps):
//   warps 0-15   epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (its 32
//                rows) of every finished accumulator, the 16-query column groups
//                going round the quarter's four warps; the values are held in
//                registers, the accumulator is released, one compare per value
//                against the query's threshold (in the units of g + (f_res/2)
//                acc) gives each thread a mask of its candidates, and every
//                thread appends its own to the queries' lists in shared memory
//                (one atomic each; two or three rounds a warp and row block).
//                Lists beyond their shared capacity continue in global memory;
//                after a row block the lists above TRIG entries are cut to (about)
//                their k' smallest, which also lowers the query's threshold;
//   warps 16-23  converters, two sets of four warps: set U % 2 unpacks unit U,
//                one thread per row, from the raw ring in shared memory into FP16
//                (or e4m3) values in TMEM slot U % AS;
//   warp 24      code loader: publishes the items, per row block a bulk copy of
//                the rows' factors and ids, per unit one TMA load of the packed
//                codes into a raw ring that is released as soon as the
//                converters have read it (the ring's length is a multiple of
//                two, so that each slot belongs to one converter set, which
//                awaits its phases in order);
//   warps 25, 26 query loaders: per stage the item's query rows by TMA gather4
//                into the stage's swizzled B tile, the stages taken in turn;
//   warp 27      MMA issuer (one elected thread; owner of the tensor memory).
//                Row blocks take the accumulators in turn (NACC of them), so
//                that one is drained while the others fill.
// What bounds it, by per-role clocks: with short lists and wide queries (zipf,
// 16,384 queries x 256 lists at D = 768) nothing alone - converters are busy half
// of the time, the issuer waits a quarter of it for an accumulator and a sixth for
// query tiles, which come from the L2 at 2.4 TB/s; at D = 192 the epilogue (list
// cuts and appends); with split e4m3 codes the converters. Measured against eight
// epilogue warps with one vote per query and four converter sets: 10,000 queries x
// 16 lists of 400,000 x 960, 0.51 -> 0.31 ms; zipf above, 3.64 -> 2.53 ms.  Unrolled
// appends or a cut inlined three times over made every role slower, bound by the
// instruction cache.
// A query starts from the smallest threshold published so far by its items,
// which is never below its final k'-th key, so each list stays a superset of
// what the item contributes.
// Every mbarrier wait is bounded (the limit is a kernel argument): on expiry
// the kernel records ERQ_ETIMEOUT in the status word, every role stops at its
// next wait (the abort flag; the epilogue warps agree on it at their named
// barrier), the copies and MMAs already issued are drained (bounded), TMEM is
// freed and the kernel returns.
#include <algorithm>
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "erq_kernels.cuh"
#include "erq_search.cuh"
#include "tc_common.cuh"
#include "warp_sort.cuh"

namespace erq {

namespace tc {

constexpr int MR = 128;          // stored rows per row block (MMA M = TMEM lanes)
static_assert(MR == 128, "four 32-row lane quarters per row block");
constexpr int KB = 64;           // FP16 elements per K block (one 128-byte swizzle row)
constexpr int RP = 2;            // row blocks per stage group
constexpr int MS = 4;            // row-factor buffers
constexpr int RSMAX = 16;        // raw-code ring slots at most
constexpr int NEP = 16;          // epilogue warps 0 .. NEP - 1 (a multiple of four)
constexpr int W_CV = NEP;        // converter warps: set (w - W_CV) / 4, lane quarter w % 4
constexpr int NSET = 2;
constexpr int W_LD = W_CV + 4 * NSET;   // code loader and item publisher
constexpr int W_QL = W_LD + 1;          // query-tile loaders (stage g: loader g % NQL)
constexpr int NQL = 2;
constexpr int W_MMA = W_QL + NQL;       // MMA issuer, TMEM owner
constexpr int NWARP = W_MMA + 1;
constexpr int THREADS = 32 * NWARP;
constexpr int TMEM_COLS = 512;
constexpr int KCAP = 128;        // largest k' of the tensor-core path
constexpr int SP = 128;          // entries of a list's continuation in global memory
constexpr int BAR_EP = 1;        // named barrier of the epilogue warps
static_assert(W_CV % 4 == 0, "a set's warps own their lane quarters");

// Work-item capacities: QN queries per item at most (the MMA's N extent), KC
// shared list entries per query, TRIG entries above which a list is cut after a
// row block, LS query-tile stages of QB bytes per query, RAWK KB of raw ring, AS
// TMEM slots of converted units (32 columns each), EX how a list is cut
// (ListRegs::bound).  TMEM not taken by the slots holds the accumulators: with
// 128 queries four slots leave three, so that a stage group's two row blocks
// start while the last one's second is still read out (16,384 queries x 256 lists
// at D = 768: 2.67 -> 2.53 ms against eight slots and two accumulators).
template <int QN_, int KC_, int TRIG_, int LS_, int QB_, int RAWK_, int AS_, bool EX_ = false>
struct Cfg {
    static constexpr int QN = QN_, KC = KC_, TRIG = TRIG_, LS = LS_, QB = QB_;
    static constexpr int AS = AS_;
    static constexpr bool EX = EX_;
    static constexpr int ACOL = TMEM_COLS - AS * (KB / 2);   // first TMEM column of the code slots
    static constexpr int DCOL = QB == 256 ? 2 * QN : QN;     // columns of an accumulator (two query parts: one sum each)
    static constexpr int NACC = ACOL / DCOL;         // accumulators
    static_assert(AS % NSET == 0, "a set owns whole slots");
    static constexpr int RAW_BYTES = RAWK_ * 1024;
    static constexpr int TILE_Q = QN * QB;           // one stage's query tile
    static_assert(NACC >= RP && QN % 32 == 0, "a stage group's accumulators fit");
    // entries after a row block: at most TRIG before it and 128 new ones
    static_assert(KC % 32 == 0 && TRIG <= KC && TRIG + MR <= KC + SP, "list capacity");
    struct Smem {
        // offsets in bytes from a 1024-aligned base
        static constexpr int q = 0;                              // LS x [QN][QB] query tiles, swizzled
        static constexpr int raw = q + LS * TILE_Q;              // raw-code ring (RS slots of B KB)
        static constexpr int lists = raw + RAW_BYTES;            // [QN][KC] u64 candidate keys
        static constexpr int meta = lists + QN * KC * 8;         // MS x [MR] float4 {g, f_res/2, id, 0}
        static constexpr int iq = meta + MS * MR * 16;           // 2 x [QN] int4 {query row, dqc bits, list lo, hi}
        static constexpr int tq = iq + 2 * QN * 16;              // 2 x [QN] u64 query-wide threshold at publication
        static constexpr int tau = tq + 2 * QN * 8;              // [QN] u64 admission key
        static constexpr int thr = tau + QN * 8;                 // [QN] f32 relaxed threshold (NaN: no query)
        static constexpr int cnt = thr + QN * 4;                 // [QN] u32 list fill
        static constexpr int qsc = cnt + QN * 4;                 // 2 x [QN] f32 query scale
        static constexpr int itd = qsc + 2 * QN * 4;             // 2 x int4 {rb0 lo, rb0 hi, rows, queries | -1}
        static constexpr int bars = itd + 2 * 16;
        static constexpr int nbars = 2 * RSMAX + 2 * LS + 2 * AS + 2 * NACC + 2 * MS + 4 + 2;
        static constexpr int tmem_slot = bars + nbars * 8;
        static constexpr int abort_flag = tmem_slot + 4;
        static constexpr int total = abort_flag + 4 + 1024;      // + alignment slack
    };
    static_assert(Smem::total <= 227 * 1024, "scan_tc shared memory");
    // barrier byte offsets from Smem::bars
    static constexpr int b_full_raw(int s) { return 8 * s; }
    static constexpr int b_empty_raw(int s) { return 8 * (RSMAX + s); }
    static constexpr int b_full_q(int s) { return 8 * (2 * RSMAX + s); }
    static constexpr int b_empty_q(int s) { return 8 * (2 * RSMAX + LS + s); }
    static constexpr int B0 = 2 * RSMAX + 2 * LS;
    static constexpr int b_full_a(int s) { return 8 * (B0 + s); }
    static constexpr int b_empty_a(int s) { return 8 * (B0 + AS + s); }
    static constexpr int b_tfull(int u) { return 8 * (B0 + 2 * AS + u); }
    static constexpr int b_tempty(int u) { return 8 * (B0 + 2 * AS + NACC + u); }
    static constexpr int B1 = B0 + 2 * AS + 2 * NACC;
    static constexpr int b_full_meta(int m) { return 8 * (B1 + m); }
    static constexpr int b_empty_meta(int m) { return 8 * (B1 + MS + m); }
    static constexpr int b_full_item(int i) { return 8 * (B1 + 2 * MS + i); }
    static constexpr int b_empty_item(int i) { return 8 * (B1 + 2 * MS + 2 + i); }
    static constexpr int b_done() { return 8 * (B1 + 2 * MS + 4); }
    // a barrier nothing arrives on (the test stall of the bounded-wait path)
    static constexpr int b_never() { return 8 * (B1 + 2 * MS + 5); }
};
using CfgA = Cfg<64, 160, 96, 6, 128, 48, 8>;    // k' <= 32, up to 64 queries per item
using CfgW = Cfg<128, 96, 88, 4, 128, 40, 4>;    // k' <= 32, up to 128 queries per item
using CfgB = Cfg<32, 256, 160, 6, 128, 48, 8>;   // k' <= 128, up to 32 queries per item
using CfgA32 = Cfg<64, 160, 96, 4, 256, 48, 4>;  // the same with two query parts (FP32 precision)
using CfgB32 = Cfg<32, 256, 160, 6, 256, 48, 8>;
using CfgAx = Cfg<64, 160, 96, 6, 128, 48, 8, true>;   // KMIN < k' <= 32
using CfgWx = Cfg<128, 96, 88, 4, 128, 40, 4, true>;
using CfgA32x = Cfg<64, 160, 96, 4, 256, 48, 4, true>;
constexpr int KMIN = 24;

// arrivals that complete a phase of the item-release barrier: one per warp of
// the epilogue, the converters, the query loaders and the issuer
constexpr int kItemReleasers = NEP + 4 * NSET + NQL + 1;

// Packed codes of one stored row and one 64-coordinate K block -> 32 TMEM
// columns of FP16 pairs 2u - (2^B - 1) (column c holds coordinates 2c, 2c+1).
// The row's 8B bytes are B 8-byte words; word j of the 32 rows of a tile is a
// contiguous 256-byte run, so `base` points at word 0 of this row and word j
// is at base + 256 j.  With h the 32-bit half index (0..7 over words 0-3) and
// L a byte lane:
//   B >= 4: words 0-3 hold the low four bits of every code as nibbles, byte L
//           of half h = (u[8h + L] & 15) | (u[8h + 4 + L] & 15) << 4, and word
//           b (4 <= b < B) is bit plane b;
//   B < 4:  word b (b < B) is bit plane b;
//   bit plane b: bit 8L + (m & 7) of half (m >> 3) is bit b of u[4m + L].
// Four coordinates 4m..4m+3 are assembled in the byte lanes of one register
// (nibble: one shift and mask; each plane: one shift and one masked OR), as
// 2u for B <= 7 and u for B = 8.  A byte x placed under 0x64 is the FP16
// value 1024 + x (exact); 2u - off = (1024 + 2u) - (1024 + off) is then one
// exact subtraction (for B = 8: 2 (1024 + u) - 2048 - off, each step exact).
template <int B>
__device__ __forceinline__ void unpack_codes(const unsigned char* base, uint32_t (&w)[32]) {
    constexpr int T = B <= 7 ? 1 : 0;
    constexpr int BS = B >= 4 ? 4 : 0;
    uint2 W[B];
#pragma unroll
    for (int j = 0; j < B; ++j) W[j] = *reinterpret_cast<const uint2*>(base + 256 * j);
    const float off = (float)((1 << B) - 1);
    const __half2 c2 = __floats2half2_rn(1024.f + off, 1024.f + off);
    const __half2 off2 = __floats2half2_rn(off, off);
    const __half2 two = __floats2half2_rn(2.f, 2.f);
    const __half2 m2048 = __floats2half2_rn(-2048.f, -2048.f);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        uint32_t V = 0;
        if constexpr (B >= 4) {
            const int h = m >> 1;
            const uint32_t N = (h & 1) ? W[h >> 1].y : W[h >> 1].x;
            if constexpr (T == 1) V = (m & 1) ? (N >> 3) & 0x1E1E1E1Eu : (N << 1) & 0x1E1E1E1Eu;
            else V = (m & 1) ? (N >> 4) & 0x0F0F0F0Fu : N & 0x0F0F0F0Fu;
        }
#pragma unroll
        for (int b = BS; b < B; ++b) {
            const uint32_t P = m < 8 ? W[b].x : W[b].y;
            const int sh = b + T - (m & 7);
            const uint32_t x = sh >= 0 ? P << sh : P >> (-sh);
            V |= x & (0x01010101u << (b + T));
        }
        const uint32_t p0 = __byte_perm(V, 0x6464u, 0x4140u);   // {x0, 0x64, x1, 0x64}
        const uint32_t p1 = __byte_perm(V, 0x6464u, 0x4342u);   // {x2, 0x64, x3, 0x64}
        __half2 h0 = *reinterpret_cast<const __half2*>(&p0);
        __half2 h1 = *reinterpret_cast<const __half2*>(&p1);
        if constexpr (T == 1) {
            h0 = __hsub2(h0, c2);
            h1 = __hsub2(h1, c2);
        } else {
            h0 = __hsub2(__hfma2(h0, two, m2048), off2);
            h1 = __hsub2(__hfma2(h1, two, m2048), off2);
        }
        w[2 * m] = *reinterpret_cast<uint32_t*>(&h0);
        w[2 * m + 1] = *reinterpret_cast<uint32_t*>(&h1);
    }
}

// B = 9: bits 0-7 assembled in byte lanes as for B = 8 (nibble words 0-3,
// planes 4-7) and bit 8 from plane 8; placed under 0x64 with bit 8 in the high
// byte's lowest bit, each 16-bit lane is the FP16 value 1024 + u (u < 512,
// exact), and 2 (1024 + u) - 2048 - 511 = 2u - 511 (each step exact).
__device__ __forceinline__ void unpack_codes9(const unsigned char* base, uint32_t (&w)[32]) {
    uint2 W[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) W[j] = *reinterpret_cast<const uint2*>(base + 256 * j);
    const __half2 off2 = __floats2half2_rn(511.f, 511.f);
    const __half2 two = __floats2half2_rn(2.f, 2.f);
    const __half2 m2048 = __floats2half2_rn(-2048.f, -2048.f);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int h = m >> 1;
        const uint32_t N = (h & 1) ? W[h >> 1].y : W[h >> 1].x;
        uint32_t V = (m & 1) ? (N >> 4) & 0x0F0F0F0Fu : N & 0x0F0F0F0Fu;
#pragma unroll
        for (int b = 4; b < 8; ++b) {
            const uint32_t P = m < 8 ? W[b].x : W[b].y;
            const int sh = b - (m & 7);
            const uint32_t x = sh >= 0 ? P << sh : P >> (-sh);
            V |= x & (0x01010101u << b);
        }
        const uint32_t P8 = m < 8 ? W[8].x : W[8].y;
        const uint32_t H = ((P8 >> (m & 7)) & 0x01010101u) | 0x64646464u;   // 0x64 | bit 8, per byte lane
        const uint32_t p0 = __byte_perm(V, H, 0x5140u);   // {u0 lo, 0x64 | u0 bit 8, u1 lo, ...}
        const uint32_t p1 = __byte_perm(V, H, 0x7362u);
        __half2 h0 = *reinterpret_cast<const __half2*>(&p0);
        __half2 h1 = *reinterpret_cast<const __half2*>(&p1);
        h0 = __hsub2(__hfma2(h0, two, m2048), off2);
        h1 = __hsub2(__hfma2(h1, two, m2048), off2);
        w[2 * m] = *reinterpret_cast<uint32_t*>(&h0);
        w[2 * m + 1] = *reinterpret_cast<uint32_t*>(&h1);
    }
}

__device__ __forceinline__ void unpack_codes_b(int B, const unsigned char* base, uint32_t (&w)[32]) {
    switch (B) {
        case 1: unpack_codes<1>(base, w); break;
        case 2: unpack_codes<2>(base, w); break;
        case 3: unpack_codes<3>(base, w); break;
        case 4: unpack_codes<4>(base, w); break;
        case 5: unpack_codes<5>(base, w); break;
        case 6: unpack_codes<6>(base, w); break;
        case 7: unpack_codes<7>(base, w); break;
        case 8: unpack_codes<8>(base, w); break;
        default: unpack_codes9(base, w); break;
    }
}

// Two FP16 values holding odd integers |x| <= 15 (exact in e4m3) -> their
// e4m3 encodings in bytes 0 and 2: the e4m3 exponent is the FP16 one minus 8
// (biases 15 and 7) and the three mantissa bits are the FP16 mantissa's top
// three (the lower seven are zero for these values).  With X16 the encodings
// are those of 16 x (exponent + 4; at most 240, below e4m3's 448).
template <bool X16 = false>
__device__ __forceinline__ uint32_t half2_to_e4m3_pair(uint32_t w) {
    constexpr uint32_t sub = X16 ? 0x00200020u : 0x00400040u;
    return (((w >> 7) & 0x00FF00FFu) - sub) | ((w >> 8) & 0x00800080u);
}

// Four byte lanes holding 2x (x < 16) -> the e4m3 encodings of 2x - off
// (odd, |2x - off| <= 15), times 16 with X16, in byte lanes 0..3.
template <bool X16>
__device__ __forceinline__ uint32_t lanes_to_e4m3(uint32_t V, __half2 c) {
    const uint32_t p0 = __byte_perm(V, 0x6464u, 0x4140u);   // {x0, 0x64, x1, 0x64}: FP16 1024 + 2x
    const uint32_t p1 = __byte_perm(V, 0x6464u, 0x4342u);
    const __half2 h0 = __hsub2(*reinterpret_cast<const __half2*>(&p0), c);
    const __half2 h1 = __hsub2(*reinterpret_cast<const __half2*>(&p1), c);
    return __byte_perm(half2_to_e4m3_pair<X16>(*reinterpret_cast<const uint32_t*>(&h0)),
                       half2_to_e4m3_pair<X16>(*reinterpret_cast<const uint32_t*>(&h1)), 0x6420u);
}

// Split e4m3 form of B = 5..8 codes (Section 3.3 remarks that a B-bit code
// can be handled as parts of fewer bits).  With u = 16 h + l, l < 16,
//   2u - (2^B - 1) = 16 (2h - (2^(B-4) - 1)) + (2l - 15),
// and both brackets are odd integers of magnitude <= 15, so 16 hc and lc are
// exact in e4m3.  Output: 32 columns for one 64-coordinate block, w[m] the
// four values 16 hc of coordinates 4m..4m+3 and w[16 + m] their lc; the
// stage's query tile holds the block's e4m3 queries twice (bytes 0-63 and
// 64-127), so the four K = 32 MMAs of the stage sum 16 hc q + lc q exactly.
// Packed layout as at unpack_codes (B >= 4: nibble words 0-3, planes 4..B-1).
template <int B>
__device__ __forceinline__ void unpack_split(const unsigned char* base, uint32_t (&w)[32]) {
    static_assert(B >= 5 && B <= 8, "split form is for B = 5..8");
    uint2 W[B];
#pragma unroll
    for (int j = 0; j < B; ++j) W[j] = *reinterpret_cast<const uint2*>(base + 256 * j);
    const float offh = (float)((1 << (B - 4)) - 1);
    const __half2 ch = __floats2half2_rn(1024.f + offh, 1024.f + offh);
    const __half2 cl = __floats2half2_rn(1039.f, 1039.f);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int h = m >> 1;
        const uint32_t N = (h & 1) ? W[h >> 1].y : W[h >> 1].x;
        const uint32_t L = (m & 1) ? (N >> 3) & 0x1E1E1E1Eu : (N << 1) & 0x1E1E1E1Eu;   // 2l per byte lane
        uint32_t H = 0;                                                                 // 2h per byte lane
#pragma unroll
        for (int b = 4; b < B; ++b) {
            const uint32_t P = m < 8 ? W[b].x : W[b].y;
            const int sh = (b - 3) - (m & 7);
            const uint32_t x = sh >= 0 ? P << sh : P >> (-sh);
            H |= x & (0x01010101u << (b - 3));
        }
        w[m] = lanes_to_e4m3<true>(H, ch);
        w[16 + m] = lanes_to_e4m3<false>(L, cl);
    }
}

__device__ __forceinline__ void unpack_split_b(int B, const unsigned char* base, uint32_t (&w)[32]) {
    switch (B) {
        case 5: unpack_split<5>(base, w); break;
        case 6: unpack_split<6>(base, w); break;
        case 7: unpack_split<7>(base, w); break;
        default: unpack_split<8>(base, w); break;
    }
}

struct Args {
    const int4* itemd;            // [items] {rb0 lo, rb0 hi, rows, queries}
    const int4* itemq;            // [items][qn] {query row or -1, dqc bits, output list index lo, hi}
    int qn;                       // queries per item of the plan (row stride of itemq)
    const float4* rowmeta;        // [Np] {g, f_res / 2, id bits, 0} in padded stored-row order
    const int64_t* n_items;
    unsigned int* work_ctr;       // items taken after the first grid-size ones (zero at launch)
    uint64_t* inter;
    int32_t* inter_cnt;
    int lstride;                  // entries of an output list
    uint64_t* spill;              // [grid][QN][SP] continuation of the CTAs' lists
    unsigned long long* tq;       // [nq] query-wide admission threshold (k'-th key of a finished item)
    const float* qscale;          // e4m3 path: per-query power-of-two scale of the e4m3 values
    uint32_t* status;
    int D, B, kp, nkb;            // nkb: stages per row group (64 FP16 or 128 e4m3 coordinates each)
    int ip;                       // inner-product metric: est = -<c, q_r> + (f_res / 4) * acc
    int codes_shared;             // items of one cluster share its rows (queries > QN): codes stay in L2 normally,
                                  // else they are loaded evict-first
    unsigned long long wait_ns;   // limit of every bounded wait
    long long stall_stage;        // >= 0: the first issuer waits at this stage on a barrier nothing arrives on
    DevChecks ck;
};

__device__ __forceinline__ int npad_of(int nqi) { return nqi <= 16 ? 16 : (nqi + 15) & ~15; }
__device__ __forceinline__ int64_t rb0_of(int4 d) { return (int64_t)(uint32_t)d.x | ((int64_t)d.y << 32); }

}  // namespace tc

using namespace tc;

// A threshold on the accumulator values (g + (f_res/2) acc) that admits every
// value v with fl(dq + v) <= tf: tf - dq, raised by 2^-20 of |tf| + |dq| to
// cover the roundings of fl(dq + v) and of this expression (each within 2^-24
// of the magnitudes involved) and by 2^-120 for the absolute error of
// subnormal results; +inf stays +inf.
__device__ __forceinline__ float relaxed_threshold(float tf, float dq) {
    return (tf - dq) + (0x1p-20f * (fabsf(tf) + fabsf(dq)) + 0x1p-120f);
}

__device__ __forceinline__ uint32_t sort32_step(uint32_t m, int d, bool asc, int lane) {
    const uint32_t p = __shfl_xor_sync(0xffffffffu, m, d);
    return ((lane & d) == 0) == asc ? min(m, p) : max(m, p);
}
// Of two ascending lists across the lanes, the 32 smallest, ascending.
__device__ __forceinline__ uint32_t merge32_u32(uint32_t x, uint32_t y, int lane) {
    uint32_t m = min(x, __shfl_sync(0xffffffffu, y, 31 - lane));
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) m = sort32_step(m, d, true, lane);
    return m;
}

// The kp-th smallest (kp <= 32) estimate, as its order-preserving integer, of a
// list of cnt keys (kc in shared memory, the rest in `spill`): 128 keys at a time
// are sorted in runs of 32 side by side, which are merged into the 32 smallest
// so far.
__device__ __forceinline__ uint32_t list_kth(const uint64_t* list, const uint64_t* spill, int cnt, int kc, int kp, int lane) {
    uint32_t best = 0xffffffffu;
#pragma unroll 1
    for (int e0 = 0; e0 < cnt; e0 += 128) {
        uint32_t c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = e0 + 32 * u + lane;
            c[u] = 0xffffffffu;
            if (e < cnt) c[u] = (uint32_t)((e < kc ? list[e] : __ldcg(spill + (e - kc))) >> 32);
        }
#pragma unroll
        for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
            for (int d = size >> 1; d > 0; d >>= 1)
#pragma unroll
                for (int u = 0; u < 4; ++u) c[u] = sort32_step(c[u], d, size == 32 || (lane & size) == 0, lane);
        best = merge32_u32(best, merge32_u32(merge32_u32(c[0], c[1], lane), merge32_u32(c[2], c[3], lane), lane), lane);
    }
    return __shfl_sync(0xffffffffu, best, kp - 1);
}

// One query's list (cnt entries: KC in shared memory, the rest in `spill`),
// held by a warp as keys e = 32 j + lane in v[j].
template <int KC>
struct ListRegs {
    static constexpr int E = (KC + SP) / 32;
    uint64_t v[E];
    __device__ __forceinline__ void load(const uint64_t* list, const uint64_t* spill, int cnt, int lane) {
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const int e = 32 * j + lane;
            v[j] = kEmptyKey;
            if (32 * j < cnt && e < cnt) v[j] = e < KC ? list[e] : __ldcg(spill + (e - KC));
        }
    }
    // the keys <= k to list[0 ..]; their number
    __device__ __forceinline__ int store_le(uint64_t* list, uint64_t k, int lane) const {
        int n = 0;
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const bool in = v[j] <= k;
            const uint32_t msk = __ballot_sync(0xffffffffu, in);
            if (in) list[n + __popc(msk & ((1u << lane) - 1u))] = v[j];
            n += __popc(msk);
        }
        __syncwarp();
        return n;
    }
    __device__ __forceinline__ int count_le(uint64_t k) const {
        int n = 0;
#pragma unroll
        for (int j = 0; j < E; ++j) n += __popc(__ballot_sync(0xffffffffu, v[j] <= k));
        return n;
    }
    // A key that at least kp entries do not exceed and at most `most` do (kp <=
    // cnt, kp <= most).  For kp <= 32 every key of an estimate: with EX the kp-th
    // smallest (`kth`, list_kth's), else the kp-th smallest of the lanes' smallest (kp lanes
    // hold an entry at or below it).  Where that admits too many (or kp > 32), the
    // exact kp-th key bit by bit.
    // The lanes' minima are the cheaper, but of 128 entries they let 28 stay at kp =
    // 20, 37 at 24 and 74 at 32, so that lists fill again at once or are cut bit by
    // bit (64 rounds of votes, 4,000 cycles): EX from kp > KMIN (10,770 queries x 38
    // lists at D = 192, k' = 32: 1.69 -> 1.23 ms; at k' = 20 the sort costs more than
    // it saves, 4,000 x 32 at D = 1536: 0.32 -> 0.37 ms).
    template <bool EX>
    __device__ __forceinline__ uint64_t bound(uint32_t kth, int kp, int most, int lane) const {
        if (kp <= 32) {
            if (!EX) {
                uint32_t m = 0xffffffffu;
#pragma unroll
                for (int j = 0; j < E; ++j) m = min(m, (uint32_t)(v[j] >> 32));
#pragma unroll
                for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
                    for (int d = size >> 1; d > 0; d >>= 1) m = sort32_step(m, d, size == 32 || (lane & size) == 0, lane);
                kth = __shfl_sync(0xffffffffu, m, kp - 1);
            }
            const uint64_t k = ((uint64_t)kth << 32) | 0xffffffffull;
            if (count_le(k) <= most && k != kEmptyKey) return k;
        }
        uint64_t k = 0;
#pragma unroll 1
        for (int b = 63; b >= 0; --b)
            if (count_le(k | ((1ull << b) - 1ull)) < kp) k |= 1ull << b;
        return k;
    }
};

// v[k] of N registers by a selection tree (no indexed registers).
template <int N>
__device__ __forceinline__ float select_reg(const uint32_t (&v)[N], int k) {
    if constexpr (N == 1) {
        return __uint_as_float(v[0]);
    } else {
        uint32_t h[N / 2];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) h[i] = (k & 1) ? v[2 * i + 1] : v[2 * i];
        return select_reg<N / 2>(h, k >> 1);
    }
}

// One candidate of one thread: value v = g + (f_res/2) acc of its row for query
// q.  Appends its key to the query's list if the key is admitted; returns
// whether the list went above TRIG.
template <class C>
__device__ __forceinline__ bool append_candidate(unsigned char* sm, const int4* iq, uint64_t* spill, int q, float v,
                                                 uint32_t id) {
    const uint64_t key = make_key(__int_as_float(iq[q].y) + v, id);
    if (key > reinterpret_cast<const uint64_t*>(sm + C::Smem::tau)[q]) return false;
    const int pos = (int)atomicAdd(reinterpret_cast<uint32_t*>(sm + C::Smem::cnt) + q, 1u);
    if (pos < C::KC) reinterpret_cast<uint64_t*>(sm + C::Smem::lists)[q * C::KC + pos] = key;
    else if (pos < C::KC + SP) spill[q * SP + pos - C::KC] = key;
    return pos >= C::TRIG;
}

// P selects the operand form: 0 FP16 codes and queries (kind::f16, K = 16);
// 1 e4m3 codes (B <= 4) and queries with a per-query scale (kind::f8f6f4,
// K = 32), a stage covering 128 coordinates (two packed 64-coordinate blocks)
// in the same 128 bytes per row of tensor memory and query tile as 64 FP16
// coordinates; 2 the split e4m3 form of B = 5..8 codes (unpack_split), a
// stage covering 64 coordinates whose query tile holds them twice; 3 FP16 codes
// and queries as two FP16 parts (FP32 precision, query_parts_kernel): whole
// numbers of at most 2^11 and the FP16 remainders.  Each part has its own FP32
// accumulator.  The tensor core cuts a sum off at every step, so one accumulator
// for both would lose half a unit of its last bit 2 D / 16 times over, in one
// direction (2.3 times the error of round-to-nearest multiply-adds in the whole
// estimate at D = 1536, B = 9); sums of whole numbers below 2^24 lose nothing, and
// what the remainders' sum loses is 2^-12 of that.  The query tile is the whole
// numbers' rows, then the remainders'.
template <class C, int P>
__global__ void __launch_bounds__(THREADS, 1)
    scan_tc_kernel(const __grid_constant__ CUtensorMap codes_map, const __grid_constant__ CUtensorMap codes_map1,
                   const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap q_map_lo, tc::Args a) {
    constexpr bool F8 = P == 1 || P == 2;   // e4m3 operands
    constexpr bool W2 = P == 1;       // two packed blocks per unit
    constexpr bool S32 = P == 3;      // two query parts
    constexpr bool SC = F8 || S32;    // scaled queries
    static_assert(C::QB == (S32 ? 256 : 128), "query tile");
    constexpr int QN = C::QN, KC = C::KC, LS = C::LS, NACC = C::NACC, TILE_Q = C::TILE_Q;
    constexpr int AS = C::AS, ACOL = C::ACOL;
    using Smem = typename C::Smem;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t bars = smem_u32(sm + Smem::bars);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + Smem::tmem_slot);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + Smem::abort_flag);
    int4* s_iq = reinterpret_cast<int4*>(sm + Smem::iq);
    int4* s_itd = reinterpret_cast<int4*>(sm + Smem::itd);
    unsigned long long* s_tq = reinterpret_cast<unsigned long long*>(sm + Smem::tq);
    float* s_qsc = reinterpret_cast<float*>(sm + Smem::qsc);
    const unsigned long long wlim = a.wait_ns;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nkb = a.nkb;
    const uint32_t blk = (uint32_t)(MR / 32) * 256u * (uint32_t)a.B;    // packed codes of one 128-row K block
    const uint32_t slot_bytes = blk * (W2 ? 2u : 1u);
    // a multiple of NSET raw slots: unit U uses slot U % RS and converter set
    // U % NSET, so every slot belongs to one set, which awaits its phases in order
    const int RS = min(RSMAX, (int)(C::RAW_BYTES / slot_bytes)) & ~(NSET - 1);
    int64_t nitems = *a.n_items;
    if (!ERQ_DCHECK(nitems >= 0 && nitems <= a.ck.items, a.ck.status, 7)) nitems = 0;   // uniform: every thread reads it

    if (tid == 0) {
        for (int s = 0; s < RSMAX; ++s) {
            mbar_init(bars + C::b_full_raw(s), 1);
            mbar_init(bars + C::b_empty_raw(s), 4);      // the warps of the unit's converter set
        }
        for (int s = 0; s < LS; ++s) {
            mbar_init(bars + C::b_full_q(s), 1);
            mbar_init(bars + C::b_empty_q(s), 1);
        }
        for (int s = 0; s < AS; ++s) {
            mbar_init(bars + C::b_full_a(s), 4);
            mbar_init(bars + C::b_empty_a(s), 1);
        }
        for (int u = 0; u < NACC; ++u) {
            mbar_init(bars + C::b_tfull(u), 1);
            mbar_init(bars + C::b_tempty(u), NEP);
        }
        for (int m = 0; m < MS; ++m) {
            mbar_init(bars + C::b_full_meta(m), 1);
            mbar_init(bars + C::b_empty_meta(m), NEP);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bars + C::b_full_item(i), 1);
            mbar_init(bars + C::b_empty_item(i), kItemReleasers);
        }
        mbar_init(bars + C::b_done(), 1);
        mbar_init(bars + C::b_never(), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == W_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "n"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // one arrival for the warp, after everything its lanes did
    auto arrive_warp = [&](uint32_t bar) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
    };

    if (warp == W_LD) {
        // ------------------------------------------------------------ code loader, item publisher
        uint32_t U = 0, rs = 0, rph = 1, blkc = 0, li = 0;     // unit, its raw slot, the slot's awaited phase
        bool ok = true;
        int64_t item = blockIdx.x;
        const uint64_t pol_codes = a.codes_shared ? l2_evict_normal() : l2_evict_first();
        // the descriptor and query slots of the item published next, fetched
        // while the previous item streams (its thresholds are read when it is
        // published, so they are as tight as possible)
        constexpr int QPL = QN / 32;
        int4 pd = make_int4(0, 0, 0, -1), pv[QPL];
        auto prefetch = [&](int64_t it) {
            if (it >= nitems) return;
            pd = a.itemd[it];
#pragma unroll
            for (int k = 0; k < QPL; ++k) {
                const int q = lane + 32 * k;
                pv[k] = q < a.qn ? a.itemq[it * a.qn + q] : make_int4(-1, 0, 0, 0);
            }
        };
        prefetch(item);
        for (;; ++li) {
            const int ib = li & 1;
            if (!mbar_wait_warp(bars + C::b_empty_item(ib), ((li >> 1) & 1) ^ 1, abort_flag, wlim)) {
                ok = false;
                break;
            }
            const bool have = item < nitems;
            int4 d = make_int4(0, 0, 0, -1);
            if (have) {
                d = pd;
#pragma unroll
                for (int k = 0; k < QPL; ++k) {
                    const int q = lane + 32 * k;
                    const int4 v = q < d.w ? pv[k] : make_int4(-1, 0, 0, 0);   // (slots past the item's queries are not written)
                    s_iq[ib * QN + q] = v;
                    s_tq[ib * QN + q] = v.x >= 0 ? __ldcg(a.tq + v.x) : kEmptyKey;
                    if (SC) s_qsc[ib * QN + q] = v.x >= 0 ? a.qscale[v.x] : 0.f;
                }
            }
            if (lane == 0) s_itd[ib] = d;
            arrive_warp(bars + C::b_full_item(ib));
            if (!have) break;
            const int64_t rb0 = rb0_of(d);                 // first padded row (multiple of 32)
            const int nrows = d.z;
            // the next item is claimed exactly once per published item: at the
            // start of this item's last stage group, so that its descriptor
            // arrives while the group streams (claiming no earlier keeps the
            // items of one list on several SMs at about the same time, sharing
            // its codes in L2), or below for an item without rows
            bool claimed = false;
            auto claim_next = [&]() {
                int nx = 0;
                if (lane == 0) nx = (int)atomicAdd(a.work_ctr, 1u);
                item = (int64_t)gridDim.x + __shfl_sync(0xffffffffu, nx, 0);
                prefetch(item);
                claimed = true;
            };
            for (int r = 0; r < nrows && ok; r += RP * MR) {
                if (r + RP * MR >= nrows) claim_next();
                const int nb = min(RP, (nrows - r + MR - 1) / MR);     // row blocks in this stage group
                for (int bb = 0; bb < nb && ok; ++bb, ++blkc) {
                    const int nr = min(MR, nrows - r - bb * MR);
                    const int m = blkc % MS;
                    if (!mbar_wait_warp(bars + C::b_empty_meta(m), ((blkc / MS) & 1) ^ 1, abort_flag, wlim)) {
                        ok = false;
                        break;
                    }
                    if (elect_one()) {
                        mbar_arrive_expect_tx(bars + C::b_full_meta(m), (uint32_t)nr * 16u);
                        bulk_load(smem_u32(sm + Smem::meta + m * MR * 16), a.rowmeta + rb0 + r + bb * MR,
                                  (uint32_t)nr * 16u, bars + C::b_full_meta(m));
                    }
                }
                for (int kb = 0; kb < nkb && ok; ++kb)
                    for (int bb = 0; bb < nb; ++bb, ++U) {
                        const uint32_t s = rs;
                        if (!mbar_wait_warp(bars + C::b_empty_raw(s), rph, abort_flag, wlim)) {
                            ok = false;
                            break;
                        }
                        if (++rs == (uint32_t)RS) {
                            rs = 0;
                            rph ^= 1u;
                        }
                        if (elect_one()) {
                            // whole 32-row tiles of the item's rows only: a block of
                            // fewer than 128 rows takes its tiles one by one (the rows
                            // past them are never admitted)
                            const int nt = min(MR / 32, ((nrows - r - bb * MR) + 31) >> 5);
                            const int tile = (int)((rb0 + r + bb * MR) >> 5);
                            mbar_arrive_expect_tx(bars + C::b_full_raw(s),
                                                  (uint32_t)nt * 256u * (uint32_t)a.B * (W2 ? 2u : 1u));
                            const uint32_t dst = smem_u32(sm + Smem::raw + s * slot_bytes);
                            // (the second block of the last P = 1 unit may lie past D: the TMA fills zeros)
                            for (int h = 0; h < (W2 ? 2 : 1); ++h) {
                                const int kk = W2 ? 2 * kb + h : kb;
                                if (nt == MR / 32) {
                                    tma_load_4d_hint(dst + h * blk, &codes_map, 0, 0, kk, tile,
                                                     bars + C::b_full_raw(s), pol_codes);
                                } else {
                                    for (int t = 0; t < nt; ++t)
                                        tma_load_4d_hint(dst + h * blk + t * 256u * (uint32_t)a.B, &codes_map1, 0, 0,
                                                         kk, tile + t, bars + C::b_full_raw(s), pol_codes);
                                }
                            }
                        }
                        __syncwarp();
                    }
            }
            if (!ok) break;
            if (!claimed) claim_next();
        }
        // drain: every copy this warp issued has landed before the CTA exits
        for (uint32_t k = 0; k < (uint32_t)RS && k < U; ++k) {
            const uint32_t g = U - 1 - k;
            mbar_wait_drain(bars + C::b_full_raw(g % (uint32_t)RS), (g / (uint32_t)RS) & 1);
        }
        for (uint32_t k = 0; k < MS && k < blkc; ++k) {
            const uint32_t g = blkc - 1 - k;
            mbar_wait_drain(bars + C::b_full_meta(g % MS), (g / MS) & 1);
        }
        __syncwarp();
    } else if (warp >= W_QL && warp < W_QL + NQL) {
        // ------------------------------------------------------------ query loaders (TMA gather4)
        // Loader j issues the query tiles of the stages g with g % NQL == j.
        const uint32_t qj = (uint32_t)(warp - W_QL);
        const uint64_t pol_q = l2_evict_last();           // the query rows are read by many items
        uint32_t g = 0;
        bool ok = true;
        for (uint32_t li = 0; ok; ++li) {
            const int ib = li & 1;
            if (!mbar_wait_warp(bars + C::b_full_item(ib), (li >> 1) & 1, abort_flag, wlim)) break;
            const int4 d = s_itd[ib];
            if (d.w < 0) break;
            const int npad = npad_of(d.w);
            const int nsteps = ((d.z + RP * MR - 1) / (RP * MR)) * nkb;
            // lane i gathers query slots 4i .. 4i+3 (padding slots repeat slot 0's row)
            const int4* iq = s_iq + ib * QN;
            const int r0 = iq[0].x;
            int y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int qs = 4 * lane + j;
                const int qr = qs < QN ? iq[qs].x : -1;
                y[j] = qr >= 0 ? qr : r0;
            }
            for (int t = 0; t < nsteps; ++t, ++g) {
                if (g % NQL != qj) continue;
                const int s = g % LS, kb = t % nkb;
                if (!mbar_wait_warp(bars + C::b_empty_q(s), ((g / LS) & 1) ^ 1, abort_flag, wlim)) {
                    ok = false;
                    break;
                }
                if (lane == 0) mbar_arrive_expect_tx(bars + C::b_full_q(s), (uint32_t)npad * (uint32_t)C::QB);
                __syncwarp();
                if (4 * lane < npad)
                    tma_gather4_hint(smem_u32(sm + Smem::q + s * TILE_Q + lane * 512), &q_map, kb * 128, y[0], y[1],
                                     y[2], y[3], bars + C::b_full_q(s), pol_q);
                if (S32 && 4 * lane < npad)
                    tma_gather4_hint(smem_u32(sm + Smem::q + s * TILE_Q + QN * 128 + lane * 512), &q_map_lo, kb * 128,
                                     y[0], y[1], y[2], y[3], bars + C::b_full_q(s), pol_q);
                __syncwarp();
            }
            if (!ok) break;
            arrive_warp(bars + C::b_empty_item(ib));
        }
        for (uint32_t k = 0; k < LS && k < g; ++k) {     // (the stages this loader issued)
            const uint32_t gg = g - 1 - k;
            if (gg % NQL == qj) mbar_wait_drain(bars + C::b_full_q(gg % LS), (gg / LS) & 1);
        }
        __syncwarp();
    } else if (warp >= W_CV && warp < W_CV + 4 * NSET) {
        // ------------------------------------------------------------ converters
        // Set cs converts the units U with U % NSET == cs: thread = one row of the
        // block (TMEM lane 32 (w % 4) + lane).
        const uint32_t cs = (uint32_t)(warp - W_CV) >> 2;
        const int qt = warp & 3;
        const int r = qt * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(qt * 32) << 16;
        const int B = a.B;
        const int roff = (r >> 5) * 256 * B + (r & 31) * 8;   // word 0 of row r in a 128-row block
        uint32_t U0 = 0;                                       // units before this item
        uint32_t rs = cs, rph = 0;                             // raw slot of the set's next unit, its phase
        bool ok = true;
        for (uint32_t li = 0; ok; ++li) {
            const int ib = li & 1;
            if (!mbar_wait_warp(bars + C::b_full_item(ib), (li >> 1) & 1, abort_flag, wlim)) break;
            const int4 d = s_itd[ib];
            if (d.w < 0) break;
            const uint32_t nu = (uint32_t)((d.z + MR - 1) / MR) * (uint32_t)nkb;
            for (uint32_t U = U0 + ((cs - U0) & (uint32_t)(NSET - 1)); U < U0 + nu; U += NSET) {
                const uint32_t s = U % AS;
                // the slot's TMEM columns are free (its previous MMAs completed)
                // and its raw codes have landed
                if (!mbar_wait_warp(bars + C::b_full_raw(rs), rph, abort_flag, wlim)) {
                    ok = false;
                    break;
                }
                uint32_t w[32];
                const unsigned char* src = sm + Smem::raw + rs * slot_bytes + roff;
                if (W2) {
                    // two packed blocks -> 128 e4m3 codes, four per column
#pragma unroll
                    for (int hb = 0; hb < 2; ++hb) {
                        uint32_t h[32];
                        unpack_codes_b(B, src + hb * blk, h);
#pragma unroll
                        for (int c = 0; c < 16; ++c)
                            w[16 * hb + c] = __byte_perm(half2_to_e4m3_pair(h[2 * c]),
                                                         half2_to_e4m3_pair(h[2 * c + 1]), 0x6420u);
                    }
                } else if (P == 2) {
                    unpack_split_b(B, src, w);
                } else {
                    unpack_codes_b(B, src, w);
                }
                if (!mbar_wait_warp(bars + C::b_empty_a(s), ((U / AS) & 1) ^ 1, abort_flag, wlim)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                ERQ_TMEM_ST32(tmem + lane_addr + ACOL + s * (KB / 2), w);
                arrive_warp(bars + C::b_empty_raw(rs));        // the raw slot may be refilled
                rs += NSET;
                if (rs >= (uint32_t)RS) {
                    rs -= (uint32_t)RS;
                    rph ^= 1u;
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                arrive_warp(bars + C::b_full_a(s));
            }
            if (!ok) break;
            U0 += nu;
            arrive_warp(bars + C::b_empty_item(ib));
        }
    } else if (warp == W_MMA) {
        // ------------------------------------------------------------ MMA issuer
        // One elected thread keeps the tensor pipe fed: with the code operand in
        // tensor memory it issues an MMA per 35 cycles at N = 64 and 64 at
        // N = 128, the tensor core's own rate (32 and 64).
        uint32_t g = 0, U = 0, blkc = 0;
        bool ok = true;
        for (uint32_t li = 0; ok; ++li) {
            const int ib = li & 1;
            if (!mbar_wait_warp(bars + C::b_full_item(ib), (li >> 1) & 1, abort_flag, wlim)) break;
            const int4 d = s_itd[ib];
            if (d.w < 0) break;
            const uint32_t idesc = idesc_f16(MR, npad_of(d.w));
            for (int r0 = 0; r0 < d.z && ok; r0 += RP * MR) {
                const int nb = min(RP, (d.z - r0 + MR - 1) / MR);
                for (int kb = 0; kb < nkb && ok; ++kb, ++g) {
                    const int s = g % LS;
                    if ((long long)g == a.stall_stage &&
                        !mbar_wait_warp(bars + C::b_never(), 0, abort_flag, wlim)) {
                        ok = false;                                // (always: nothing arrives on it)
                        break;
                    }
                    if (!mbar_wait_warp(bars + C::b_full_q(s), (g / LS) & 1, abort_flag, wlim)) {
                        ok = false;
                        break;
                    }
                    const uint64_t tq = sdesc(smem_u32(sm + Smem::q + s * TILE_Q));
                    for (int b = 0; b < nb; ++b, ++U) {
                        const uint32_t buf = (blkc + b) % NACC, as = U % AS;
                        if (kb == 0 && !mbar_wait_warp(bars + C::b_tempty(buf), (((blkc + b) / NACC) & 1) ^ 1,
                                                       abort_flag, wlim)) {
                            ok = false;
                            break;
                        }
                        if (!mbar_wait_warp(bars + C::b_full_a(as), (U / AS) & 1, abort_flag, wlim)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t ta = tmem + ACOL + as * (KB / 2), dt = tmem + buf * C::DCOL;
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < KB / 16; ++k) {         // 32 bytes of K per instruction
                                if (F8) mma_f8_ta(dt, ta + k * 8, tq + 2 * k, idesc, (kb | k) != 0);
                                else mma_f16_ta(dt, ta + k * 8, tq + 2 * k, idesc, (kb | k) != 0);
                            }
                            if (S32) {
#pragma unroll
                                for (int k = 0; k < KB / 16; ++k)
                                    mma_f16_ta(dt + QN, ta + k * 8, tq + 2 * k + (QN * 128 >> 4), idesc, (kb | k) != 0);
                            }
                            mma_commit(bars + C::b_empty_a(as));       // code slot free
                            if (b == nb - 1) mma_commit(bars + C::b_empty_q(s));
                            if (kb == nkb - 1) mma_commit(bars + C::b_tfull(buf));
                        }
                        __syncwarp();
                    }
                }
                blkc += nb;
            }
            if (!ok) break;
            arrive_warp(bars + C::b_empty_item(ib));
        }
        // all issued MMAs complete before TMEM is released
        if (elect_one()) mma_commit(bars + C::b_done());
        __syncwarp();
        mbar_wait_drain(bars + C::b_done(), 0);
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue
        uint64_t* lists = reinterpret_cast<uint64_t*>(sm + Smem::lists);
        uint64_t* s_tau = reinterpret_cast<uint64_t*>(sm + Smem::tau);
        float* s_thr = reinterpret_cast<float*>(sm + Smem::thr);
        uint32_t* s_cnt = reinterpret_cast<uint32_t*>(sm + Smem::cnt);
        const float4* s_meta = reinterpret_cast<const float4*>(sm + Smem::meta);
        uint64_t* spill = a.spill + (int64_t)blockIdx.x * QN * SP;
        constexpr int CSTEP = 16 * (NEP / 4);             // 16-column groups go round the warps of a quarter
        const int quarter = warp & 3, par = warp >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const int kp = a.kp;
        uint32_t blkc = 0;
        for (uint32_t li = 0;; ++li) {
            const int ib = li & 1;
            const bool got = mbar_wait_warp(bars + C::b_full_item(ib), (li >> 1) & 1, abort_flag, wlim);
            // every warp takes the same decision (and has written its lists of the last item)
            if (bar_or(BAR_EP, 32 * NEP, !got)) break;
            const int4 d = s_itd[ib];
            if (d.w < 0) break;
            const int nrows = d.z, nqi = d.w, npad = npad_of(d.w);
            const int4* iq = s_iq + ib * QN;
            for (int q = tid; q < QN; q += 32 * NEP) {
                const uint64_t t = s_tq[ib * QN + q];
                s_tau[q] = t;
                s_cnt[q] = 0u;
                s_thr[q] = q < nqi ? relaxed_threshold(t == kEmptyKey ? INFINITY : key_value(t), __int_as_float(iq[q].y))
                                   : __int_as_float(0x7fc00000);
            }
            bar_sync(BAR_EP, 32 * NEP);
            bool dead = false;
            for (int r = 0; r < nrows; r += MR, ++blkc) {
                const uint32_t m = blkc % MS, buf = blkc % NACC;
                bool need = false;                                  // a list of mine went above TRIG
                dead = !mbar_wait_warp(bars + C::b_full_meta(m), (blkc / MS) & 1, abort_flag, wlim) ||
                       !mbar_wait_warp(bars + C::b_tfull(buf), (blkc / NACC) & 1, abort_flag, wlim);
                if (!dead) {
                    tc_fence_after();
                    float4 mt = s_meta[m * MR + row];
                    const uint32_t id = __float_as_uint(mt.z);
                    if (a.ip) {                                     // -<c, q_r> + (f_res / 4) acc: no g, half the factor
                        mt.x = 0.f;
                        mt.y *= 0.5f;
                    }
                    if (row >= nrows - r) {                         // past the block's rows: NaN, which no
                        mt.x = __int_as_float(0x7fc00000);          // threshold admits
                        mt.y = 0.f;
                    }
                    arrive_warp(bars + C::b_empty_meta(m));
                    const uint32_t tacc = tmem + lane_base + buf * C::DCOL;
                    // 16-column groups 16 (par + 4 g) .. of this warp, all loaded at once so
                    // that the accumulator is released before the compares
                    constexpr int NG = QN > CSTEP ? QN / CSTEP : 1;
                    uint32_t v[16 * NG];
#pragma unroll
                    for (int g = 0; g < NG; ++g)
                        if (16 * par + CSTEP * g < npad) ERQ_TMEM_LD16(tacc + 16 * par + CSTEP * g, (v + 16 * g));
                    uint32_t vl[S32 ? 16 : 1];
                    static_assert(!S32 || NG == 1, "one column group a warp where queries have two parts");
                    if constexpr (S32)
                        if (16 * par < npad) ERQ_TMEM_LD16(tacc + QN + 16 * par, vl);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    tc_fence_before();
                    arrive_warp(bars + C::b_tempty(buf));
                    if constexpr (S32) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            v[i] = __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(vl[i]));
                    }
                    // straight-line: the compares into a mask
                    uint32_t mine = 0u;
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        const int cc = 16 * par + CSTEP * g;
                        if (cc < npad) {                            // (uniform)
#pragma unroll
                            for (int i = 0; i < 16; i += 4) {
                                const float4 th = *reinterpret_cast<const float4*>(s_thr + cc + i);
                                float4 sc = make_float4(1.f, 1.f, 1.f, 1.f);
                                if (SC) sc = *reinterpret_cast<const float4*>(s_qsc + ib * QN + cc + i);
                                const float t4[4] = {th.x, th.y, th.z, th.w}, s4[4] = {sc.x, sc.y, sc.z, sc.w};
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    float x = __uint_as_float(v[16 * g + i + j]);
                                    if (SC) x *= s4[j];             // a power of two: exact
                                    const float val = fmaf(mt.y, x, mt.x);
                                    if (S32 ? !(val > t4[j]) : val <= t4[j]) mine |= 1u << (16 * g + i + j);
                                }
                            }
                        }
                    }
                    // FP32 precision ranks estimates that are not numbers last, as the
                    // CUDA-core scan does (a query with a NaN or one whose distances
                    // overflow): its comparison admits them, so the rows past the block
                    // and the padding queries are taken out here
                    if (S32) mine = row < nrows - r ? mine & ((1u << min(max(nqi - 16 * par, 0), 16)) - 1u) : 0u;
                    // every thread appends its own candidates: as many rounds as the
                    // thread with the most has, usually two or three
                    while (__any_sync(0xffffffffu, mine != 0u)) {
                        if (mine != 0u) {
                            const int i = __ffs(mine) - 1, q = 16 * par + (i & 15) + CSTEP * (i >> 4);
                            mine &= mine - 1u;
                            float x = select_reg<16 * NG>(v, i);
                            if (SC) x *= s_qsc[ib * QN + q];
                            need |= append_candidate<C>(sm, iq, spill, q, fmaf(mt.y, x, mt.x), id);
                        }
                        __syncwarp();
                    }
                }
                // every candidate of the block is in its list; the lists above TRIG are
                // cut before the next block adds to them
                if (!bar_or(BAR_EP, 32 * NEP, need || dead)) continue;
                if (!dead) {
                    // lane j looks at query warp + NEP j
                    const int ql = warp + NEP * lane;
                    for (uint32_t todo = __ballot_sync(0xffffffffu, ql < nqi && s_cnt[min(ql, QN - 1)] > (uint32_t)C::TRIG);
                         todo; todo &= todo - 1u) {
                        const int q = warp + NEP * (__ffs(todo) - 1);
                        int n = (int)s_cnt[q];
                        ListRegs<KC> L;
                        const uint32_t kth = C::EX ? list_kth(lists + q * KC, spill + q * SP, n, KC, kp, lane) : 0u;
                        L.load(lists + q * KC, spill + q * SP, n, lane);
                        const uint64_t k = L.template bound<C::EX>(kth, kp, C::TRIG, lane);
                        __syncwarp();
                        n = L.store_le(lists + q * KC, k, lane);    // (kp <= n, so k is below the empty key)
                        if (lane == 0) {
                            s_cnt[q] = (uint32_t)n;
                            s_tau[q] = k;
                            s_thr[q] = relaxed_threshold(key_value(k), __int_as_float(iq[q].y));
                            // k' keys of this query are <= k and stay in its lists, so k
                            // bounds its other items too
                            atomicMin(a.tq + iq[q].x, (unsigned long long)k);
                        }
                        __syncwarp();
                    }
                }
                if (bar_or(BAR_EP, 32 * NEP, dead)) {
                    dead = true;
                    break;
                }
            }
            if (dead) break;                                        // (uniform: decided at the barrier)
            // write the lists (lane j: query warp + NEP j); a list of k' or more keys
            // is cut first and bounds the query's other items
            {
                const int ql = warp + NEP * lane;
                int cl = ql < nqi ? (int)s_cnt[ql] : 0;
                int64_t ol = 0;
                bool put = ql < nqi;                                // this lane's list is written
                if (put) {
                    ol = (int64_t)(uint32_t)iq[ql].z | ((int64_t)iq[ql].w << 32);
                    put = ERQ_DCHECK(ol >= 0 && ol < a.ck.lists && cl >= 0 && cl <= C::TRIG, a.ck.status, 6);
                    if (!put) cl = 0;
                }
                for (uint32_t todo = __ballot_sync(0xffffffffu, cl >= kp); todo; todo &= todo - 1u) {
                    const int j = __ffs(todo) - 1, q = warp + NEP * j;
                    ListRegs<KC> L;
                    const int m = __shfl_sync(0xffffffffu, cl, j);
                    const uint32_t kth = C::EX ? list_kth(lists + q * KC, spill + q * SP, m, KC, kp, lane) : 0u;
                    L.load(lists + q * KC, spill + q * SP, m, lane);
                    const uint64_t k = L.template bound<C::EX>(kth, kp, min(C::TRIG, a.lstride), lane);   // (kp <= lstride)
                    __syncwarp();
                    const int n = L.store_le(lists + q * KC, k, lane);
                    if (lane == 0) atomicMin(a.tq + iq[q].x, (unsigned long long)k);
                    if (lane == j) cl = n;
                }
                __syncwarp();
                if (put) a.inter_cnt[ol] = cl;
                for (uint32_t todo = __ballot_sync(0xffffffffu, cl > 0); todo; todo &= todo - 1u) {
                    const int j = __ffs(todo) - 1;
                    const int n = __shfl_sync(0xffffffffu, cl, j);
                    uint64_t* dst = a.inter + __shfl_sync(0xffffffffu, ol, j) * a.lstride;
                    const uint64_t* src = lists + (warp + NEP * j) * KC;
                    for (int e = lane; e < n; e += 32) dst[e] = src[e];
                }
            }
            arrive_warp(bars + C::b_empty_item(ib));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag && tid == 0) atomicOr(a.status, kStatusTimeout);
    if (warp == W_MMA) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS));
    }
}

bool tc_available(int precision, int D, int kp) {
    return precision != ERQ_PREC_INT8 && D % KB == 0 && kp <= KCAP;
}

// Work-item query counts the tensor-core scan is built for, given k'.
bool scan_tc_shape_ok(int qn, int kp) {
    return (kp <= 32 && (qn == 32 || qn == CfgA::QN || qn == CfgW::QN)) || (kp <= KCAP && qn == CfgB::QN);
}

// Capacity (stride) of the per-(query, item) candidate lists written by the scan.
int scan_list_stride(int precision, int kp, int qn) {
    (void)qn;
    if (precision == ERQ_PREC_FP32 && kp > KCAP) return kp;      // the CUDA-core scan
    return kp <= 32 ? 64 : CfgB::TRIG;   // (a list of k' or more entries is cut to this before it is written)
}

// Entries of the lists' continuation that a launch of `grid` CTAs needs.
int64_t scan_spill_entries(int qn, int grid) { return (int64_t)grid * std::max(qn, 32) * SP; }

// Packed scan layout of the index.  One thread per (tile t, K block kb, row r
// of the tile): padded row p = 32 t + r takes its cluster's stored row (or
// zeros past the cluster's end), packs the 64 codes of block kb into B 8-byte
// words (layout at unpack_codes) and writes word j to
// codes_p[((t * nkb + kb) * B + j) * 32 + r]; the kb = 0 thread also writes the
// row's {g, f_res / 2, id, 0} to rowmeta[p].
__global__ void scan_layout_kernel(const uint8_t* __restrict__ codes, const float* __restrict__ g,
                                   const float* __restrict__ f_res, const int64_t* __restrict__ ids,
                                   const int64_t* __restrict__ list_off, const int64_t* __restrict__ poff, int nlist,
                                   int64_t Np, int D, int B, uint64_t* __restrict__ codes_p,
                                   float4* __restrict__ rowmeta) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int nkb = D / 64;
    const int r = (int)(tid & 31);
    const int64_t tk = tid >> 5;                 // t * nkb + kb
    const int64_t t = tk / nkb;
    const int kb = (int)(tk % nkb);
    const int64_t p = t * 32 + r;
    if (p >= Np) return;
    int lo = 0, hi = nlist;                      // cluster with poff[lo] <= p < poff[lo + 1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (poff[mid] <= p) lo = mid;
        else hi = mid;
    }
    const int64_t j = p - poff[lo];
    const bool valid = j < list_off[lo + 1] - list_off[lo];
    const int64_t src = list_off[lo] + j;
    uint32_t u[16];                              // 64 codes, four per word (byte i of u[k] = bits 0-7 of code 4k + i)
    uint32_t h8[16] = {};                        // B = 9: byte i of h8[k] = bit 8 of code 4k + i
    if (B <= 8) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const uint4 v = valid ? reinterpret_cast<const uint4*>(codes + src * D + kb * 64)[x] : make_uint4(0u, 0u, 0u, 0u);
            u[4 * x] = v.x; u[4 * x + 1] = v.y; u[4 * x + 2] = v.z; u[4 * x + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int x = 0; x < 8; ++x) {            // 16-bit codes: eight per uint4
            const uint4 v = valid ? reinterpret_cast<const uint4*>(codes + (src * D + kb * 64) * 2)[x]
                                  : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int h = 0; h < 2; ++h) {        // codes 8x + 4h .. + 3 -> word 2x + h
                const uint32_t a = w[2 * h], b = w[2 * h + 1];
                u[2 * x + h] = __byte_perm(a, b, 0x6420u);
                h8[2 * x + h] = __byte_perm(a, b, 0x7531u) & 0x01010101u;
            }
        }
    }
    uint64_t* dst = codes_p + (tk * B) * 32 + r;
    const int bs = B >= 4 ? 4 : 0;
    if (B >= 4) {
        // half h: byte L = (code 8h + L) & 15 | ((code 8h + 4 + L) & 15) << 4
        uint32_t N[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) N[h] = (u[2 * h] & 0x0F0F0F0Fu) | ((u[2 * h + 1] & 0x0F0F0F0Fu) << 4);
#pragma unroll
        for (int w = 0; w < 4; ++w) dst[w * 32] = (uint64_t)N[2 * w] | ((uint64_t)N[2 * w + 1] << 32);
    }
    for (int b = bs; b < B; ++b) {
        // bit 8L + (m & 7) of half (m >> 3) = bit b of code 4m + L
        uint32_t P[2] = {0u, 0u};
#pragma unroll
        for (int m = 0; m < 16; ++m)
            P[m >> 3] |= (b < 8 ? (u[m] >> b) & 0x01010101u : h8[m]) << (m & 7);
        dst[b * 32] = (uint64_t)P[0] | ((uint64_t)P[1] << 32);
    }
    if (kb == 0)
        rowmeta[p] = valid ? make_float4(g[src], 0.5f * f_res[src], __uint_as_float((uint32_t)ids[src]), 0.f)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
}

cudaError_t launch_scan_layout(const uint8_t* codes, const float* g, const float* f_res, const int64_t* ids,
                               const int64_t* list_off, const int64_t* poff, int nlist, int64_t Np, int D, int B,
                               uint64_t* codes_p, float4* rowmeta, cudaStream_t s) {
    if (Np <= 0) return cudaSuccess;
    count_launch();
    const int64_t n = ceil_div(Np, 32) * (D / 64) * 32;
    scan_layout_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(codes, g, f_res, ids, list_off, poff, nlist, Np, D,
                                                                  B, codes_p, rowmeta);
    return cudaGetLastError();
}

// 3-D view of the packed codes in 8-byte elements: (32 B words of a tile and
// K block, K block, tile); a box of (32 B, 1, 4) is the 128 rows x 8 B bytes
// of one stage, four contiguous tiles.
static bool make_codes_map(CUtensorMap* map, const uint64_t* codes_p, int64_t Np, int D, int B, int box_tiles) {
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
    // 4-D view [tiles][K blocks][B words][32 rows] of u64 (a box extent is at most 256 elements,
    // so the 32 B words of a tile and K block are two dimensions, not one of 32 B)
    const int nkb = D / KB;
    const cuuint64_t dims[4] = {32, (cuuint64_t)B, (cuuint64_t)nkb, (cuuint64_t)((Np + 31) / 32)};
    const cuuint64_t strides[3] = {256, (cuuint64_t)256 * B, (cuuint64_t)256 * B * nkb};
    const cuuint32_t box[4] = {32, (cuuint32_t)B, 1, (cuuint32_t)box_tiles};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, (void*)codes_p, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D view of the query operand (FP16 or e4m3 rows of row_bytes bytes) for
// tile::gather4: a box of one row of 128 bytes, 128-byte swizzle, so that four
// gathered rows land as consecutive 128-byte rows of the MMA's B tile.
static bool make_query_map(CUtensorMap* map, const void* base, int64_t nq, int64_t row_bytes) {
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
    const cuuint64_t dims[2] = {(cuuint64_t)row_bytes, (cuuint64_t)nq};
    const cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
    const cuuint32_t box[2] = {128, 1};
    const cuuint32_t estr[2] = {1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <class C, int P>
static erq_status scan_tc_launch(const ScanLaunch& L, const tc::Args& a, const void* qbase, const void* qlo,
                                 int64_t qrow_bytes, cudaStream_t s) {
    const int smem = C::Smem::total;
    {   // the kernel's raw-code ring must hold a multiple of NSET unit slots
        const int64_t slot = (int64_t)(MR / 32) * 256 * L.B * (P == 1 ? 2 : 1);
        if ((std::min<int64_t>(RSMAX, C::RAW_BYTES / slot) & ~(int64_t)(NSET - 1)) < NSET)
            return fail(ERQ_EUNSUPPORTED, "tensor-core scan: raw-code ring too small for this code width");
    }
    cudaError_t e = cudaFuncSetAttribute(scan_tc_kernel<C, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(e, "scan_tc smem attribute");
    if (L.grid <= 0) return ERQ_OK;
    CUtensorMap cmap, cmap1, qmap, qmap_lo;
    if (!L.codes_p || ((uintptr_t)L.codes_p & 15) != 0 || (L.D % KB) != 0 || L.B < 1 || L.B > 9 ||
        !make_codes_map(&cmap, L.codes_p, L.Np, L.D, L.B, MR / 32) ||
        !make_codes_map(&cmap1, L.codes_p, L.Np, L.D, L.B, 1))
        return fail(ERQ_ECUDA, "tensor-core scan: cuTensorMapEncodeTiled failed for the code array");
    if (!qbase || ((uintptr_t)qbase & 15) != 0 || qrow_bytes % 128 != 0 || L.nq < 1 ||
        !make_query_map(&qmap, qbase, L.nq, qrow_bytes) || ((uintptr_t)qlo & 15) != 0 ||
        !make_query_map(&qmap_lo, qlo ? qlo : qbase, L.nq, qrow_bytes))
        return fail(ERQ_ECUDA, "tensor-core scan: cuTensorMapEncodeTiled failed for the query array");
    count_launch();
    scan_tc_kernel<C, P><<<L.grid, THREADS, smem, s>>>(cmap, cmap1, qmap, qmap_lo, a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "scan_tc launch");
    return ERQ_OK;
}

template <class C>
static erq_status scan_tc_form(int P, const ScanLaunch& L, const tc::Args& a, const void* qb, int64_t qrow,
                               cudaStream_t s) {
    if (P == 1) return scan_tc_launch<C, 1>(L, a, qb, nullptr, qrow, s);
    if (P == 2) return scan_tc_launch<C, 2>(L, a, qb, nullptr, qrow, s);
    return scan_tc_launch<C, 0>(L, a, qb, nullptr, qrow, s);
}

erq_status scan_tc(const ScanLaunch& L, int precision, cudaStream_t s) {
    if (!tc_available(precision, L.D, L.kp))
        return fail(ERQ_EUNSUPPORTED, "tensor-core scan: needs precision fp32, fp16 or fp8 and k' <= 128");
    const bool f8 = precision == ERQ_PREC_FP8, f32 = precision == ERQ_PREC_FP32;
    const int P = f32 ? 3 : (f8 ? (L.B <= 4 ? 1 : 2) : 0);
    if (P == 2 && L.B > 8)
        return fail(ERQ_EUNSUPPORTED, "tensor-core scan: e4m3 holds the split code parts only for B <= 8");
    if (P == 2 && L.Dq != 2 * (int64_t)L.D) return fail(ERQ_EINVAL, "tensor-core scan: split e4m3 needs doubled query rows");
    if (!(f8 ? (L.Q8 && L.qscale) : L.Qh != nullptr) || (f32 && (!L.Ql || !L.qscale)))
        return fail(ERQ_EINVAL, "tensor-core scan: queries missing");
    if (!L.itemd || !L.itemq || !L.rowmeta || !L.tq || !L.work_ctr || !L.spill)
        return fail(ERQ_EINVAL, "tensor-core scan: item tables missing");
    if (!scan_tc_shape_ok(L.qn, L.kp) || (f32 && L.qn > CfgA32::QN))
        return fail(ERQ_EINVAL, "tensor-core scan: no kernel for this item shape");
    tc::Args a;
    a.ck = L.ck;
    a.itemd = L.itemd; a.itemq = L.itemq; a.qn = L.qn; a.rowmeta = L.rowmeta; a.n_items = L.n_items;
    a.work_ctr = L.work_ctr;
    a.lstride = scan_list_stride(precision, L.kp, L.qn);
    a.spill = L.spill;
    a.inter = L.inter; a.inter_cnt = L.inter_cnt; a.tq = L.tq; a.qscale = L.qscale; a.status = L.status;
    a.D = L.D; a.B = L.B; a.kp = L.kp; a.ip = L.ip;
    a.nkb = P == 1 ? (int)(L.Dq / 128) : L.D / KB;
    a.wait_ns = L.wait_ns ? L.wait_ns : kWaitNs;
    // a cluster probed by more queries than one item holds is read by several
    // items at about the same time (items are ordered row range first)
    a.codes_shared = L.nq * (int64_t)L.maxp > (int64_t)L.qn * L.nlist ? 1 : 0;
    a.stall_stage = L.stall_stage;
    const void* qb = f8 ? L.Q8 : L.Qh;
    const int64_t qrow = f8 ? L.Dq : 2 * (int64_t)L.D;
    const bool ex = L.kp > KMIN && L.kp <= 32;
    if (f32 && L.qn > CfgB32::QN && ex) return scan_tc_launch<CfgA32x, 3>(L, a, L.Qh, L.Ql, qrow, s);
    if (f32 && L.qn > CfgB32::QN) return scan_tc_launch<CfgA32, 3>(L, a, L.Qh, L.Ql, qrow, s);
    if (f32) return scan_tc_launch<CfgB32, 3>(L, a, L.Qh, L.Ql, qrow, s);
    if (ex && L.qn > CfgA::QN) return scan_tc_form<CfgWx>(P, L, a, qb, qrow, s);
    if (ex && L.qn > CfgB::QN) return scan_tc_form<CfgAx>(P, L, a, qb, qrow, s);
    if (L.kp <= 32 && L.qn > CfgA::QN) return scan_tc_form<CfgW>(P, L, a, qb, qrow, s);
    if (L.kp <= 32 && L.qn > CfgB::QN) return scan_tc_form<CfgA>(P, L, a, qb, qrow, s);
    return scan_tc_form<CfgB>(P, L, a, qb, qrow, s);
}

// Rotated queries -> e4m3 for the kind::f8f6f4 scan.  Per query row a power of
// two s = 2^(floor(log2 max|q'|) - 7) puts the largest magnitude in [128, 256)
// (e4m3's largest finite value is 448); every q'_i / s (exact) is rounded to
// the nearest e4m3 value, ties to even, from its FP32 bits: for |y| >= 2^-6 the
// 23-bit mantissa keeps its top 3 bits (carry into the exponent on overflow),
// below it y is a multiple of 2^-9 after rounding |y| * 2^9 to an integer
// (8 then being the smallest normal's code).  Columns D .. Dq-1 are zero.
// With dup (the split form of B = 5..8 codes, Dq = 2 D) every 64-coordinate
// block is written twice: byte 128 j + t holds coordinate 64 j + (t mod 64).
// One warp per query row.
__device__ __forceinline__ uint32_t e4m3_rn(float y) {
    const uint32_t bits = __float_as_uint(y);
    const uint32_t sign = (bits >> 31) << 7;
    const int ex = (int)((bits >> 23) & 0xffu) - 127;
    const uint32_t mant = bits & 0x7fffffu;
    uint32_t code;
    if (ex >= -6) {
        uint32_t r = mant >> 20;
        const uint32_t rem = mant & 0xfffffu;
        if (rem > 0x80000u || (rem == 0x80000u && (r & 1u))) ++r;
        int e4 = ex + 7;
        if (r == 8u) {
            r = 0u;
            ++e4;
        }
        code = ((uint32_t)e4 << 3) | r;
    } else if (ex >= -10) {
        const int sh = 14 - ex;                        // 21 .. 24
        const uint32_t full = mant | 0x800000u;
        uint32_t q = full >> sh;
        const uint32_t rem = full & ((1u << sh) - 1u), half = 1u << (sh - 1);
        if (rem > half || (rem == half && (q & 1u))) ++q;
        code = q;
    } else {
        code = 0u;                                     // below half of the smallest subnormal
    }
    return sign | code;
}

__global__ void quant_e4m3_kernel(const float* __restrict__ X, int64_t n, int D, int Dq, int dup,
                                  unsigned char* __restrict__ Y, float* __restrict__ scale) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const float* x = X + r * D;
    float m = 0.f;
#pragma unroll 4
    for (int i = lane * 4; i < D; i += 128) {              // (D % 64 == 0, rows on 16-byte boundaries)
        const float4 v = *reinterpret_cast<const float4*>(x + i);
        m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
    m = warp_max(m);
    int e = 0;
    if (m > 0.f) {
        frexpf(m, &e);                                 // m in [2^(e-1), 2^e)
        e -= 8;                                        // m / 2^e in [128, 256)
    }
    e = max(-126, min(127, e));
    const float inv = __int_as_float((127 - e) << 23), s = __int_as_float((127 + e) << 23);
    if (lane == 0) scale[r] = m > 0.f ? s : 1.f;
    unsigned char* y = Y + r * Dq;
#pragma unroll 4
    for (int c = lane * 4; c < (dup ? D : Dq); c += 128) {
        uint32_t w = 0u;
        if (c < D) {
            const float4 v = *reinterpret_cast<const float4*>(x + c);
            w = e4m3_rn(v.x * inv) | e4m3_rn(v.y * inv) << 8 | e4m3_rn(v.z * inv) << 16 | e4m3_rn(v.w * inv) << 24;
        }
        if (dup) {                                             // four coordinates of one block, in both of its copies
            const int i = ((c >> 6) << 7) | (c & 63);
            *reinterpret_cast<uint32_t*>(y + i) = w;
            *reinterpret_cast<uint32_t*>(y + i + 64) = w;
        } else {
            *reinterpret_cast<uint32_t*>(y + c) = w;
        }
    }
}

cudaError_t launch_quant_e4m3(const float* x, int64_t n, int D, int Dq, int dup, unsigned char* y, float* scale,
                              cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (D % 4 != 0 || ((uintptr_t)x & 15) != 0 || Dq % 4 != 0 || (dup && Dq != 2 * D) || (!dup && Dq < D)) return cudaErrorInvalidValue;
    count_launch();
    quant_e4m3_kernel<<<(unsigned)ceil_div(n * 32, 256), 256, 0, s>>>(x, n, D, Dq, dup, y, scale);
    return cudaGetLastError();
}

// Rotated queries -> the two FP16 parts of the FP32-precision scan, one warp per
// row.  With the row's power of two 2^e, t = x 2^-e: hi = t rounded to a whole
// number, |hi| <= 2^11 (exact in FP16), and lo = RN16(t - hi), |lo| <= 1/2, so t is
// held to 2^-13.  e is the smallest with ||t|| <= lim as well: a row of codes c has
// <c, hi> = cos ||c|| ||hi||, ||c|| is about 0.36 2^B sqrt(D) (uniform levels of a
// Gaussian-like row), and lim keeps that below 2^24 for cosines up to 0.6, so that
// the accumulator's sums of whole numbers are exact (or nearly, for the last steps
// of larger cosines).  Against 64 bits, over D = 64 .. 4096 and B = 1 .. 9, the
// sum's error is 0.03 to 0.7 of that of D round-to-nearest multiply-adds from a
// cosine of 0.1 on; between orthogonal vectors, whose sum is next to nothing, up
// to 1.3 of it for D <= 128 and, at B = 9 alone, 2 to 3 for D >= 1536.
__global__ void query_parts_kernel(const float* __restrict__ X, int64_t n, int D, float lim, __half* __restrict__ hi,
                                   __half* __restrict__ lo, float* __restrict__ scale) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const float4* x = reinterpret_cast<const float4*>(X + r * D);
    float mx = 0.f;
    for (int i = lane; i < D / 4; i += 32) {
        const float4 v = x[i];
        mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    }
    mx = warp_max(mx);
    int e = 0;
    if (mx > 0.f && mx < INFINITY) {
        frexpf(mx, &e);                                    // mx in [2^(e-1), 2^e)
        e = min(max(e - 11, -126), 126);
        const float s = __int_as_float((127 - e) << 23);
        float ss = 0.f;
        for (int i = lane; i < D / 4; i += 32) {
            const float4 v = x[i];
            const float a = v.x * s, b = v.y * s, c = v.z * s, d = v.w * s;
            ss += (a * a + b * b) + (c * c + d * d);
        }
        const float over = sqrtf(warp_sum(ss)) / lim;      // (NaN: not raised)
        if (over > 1.f) {
            int k;
            frexpf(over, &k);                              // over < 2^k
            e = min(e + k, 126);
        }
    }
    if (lane == 0) scale[r] = __int_as_float((127 + e) << 23);
    const float s = __int_as_float((127 - e) << 23);
    for (int i = lane; i < D / 4; i += 32) {
        const float4 v = x[i];
        const float t[4] = {v.x * s, v.y * s, v.z * s, v.w * s};
        float h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) h[j] = rintf(t[j]);
        const __half2 h0 = __floats2half2_rn(h[0], h[1]), h1 = __floats2half2_rn(h[2], h[3]);
        const __half2 l0 = __floats2half2_rn(t[0] - h[0], t[1] - h[1]), l1 = __floats2half2_rn(t[2] - h[2], t[3] - h[3]);
        reinterpret_cast<uint2*>(hi + r * D)[i] =
            make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
        reinterpret_cast<uint2*>(lo + r * D)[i] =
            make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
    }
}

cudaError_t launch_query_parts(const float* x, int64_t n, int D, int B, __half* hi, __half* lo, float* scale,
                               cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (D % 4 != 0 || (((uintptr_t)x | (uintptr_t)hi | (uintptr_t)lo) & 15) != 0) return cudaErrorInvalidValue;
    const float code = (B > 1 ? 0.36f * (float)(1 << B) : 1.f) * sqrtf((float)D);
    count_launch();
    query_parts_kernel<<<(unsigned)ceil_div(n * 32, 256), 256, 0, s>>>(x, n, D, 16777216.f / (0.6f * code), hi, lo, scale);
    return cudaGetLastError();
}

// FP32 -> FP16 (round to nearest) of the rotated queries.
__global__ void to_half_kernel(const float* __restrict__ x, __half* __restrict__ y, int64_t n) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t * 4 >= n) return;
    const float4 v = reinterpret_cast<const float4*>(x)[t];
    __half2* o = reinterpret_cast<__half2*>(y) + 2 * t;
    o[0] = __floats2half2_rn(v.x, v.y);
    o[1] = __floats2half2_rn(v.z, v.w);
}

cudaError_t launch_to_half(const float* x, __half* y, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    count_launch();
    to_half_kernel<<<(unsigned)ceil_div(n / 4, 256), 256, 0, s>>>(x, y, n);
    return cudaGetLastError();
}

}  // namespace erq
