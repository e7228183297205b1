// Split-BF16 contractions: constants and device buffers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <climits>

#include <utility>
#include <vector>

#include "mma_schedule.h"
#include "ops.cuh"
#include "vfmm_internal.cuh"

namespace vfmm {

// contractions of the mixed form, in the order of vfmm_ops_set_slices
enum { kCtrNear = 0, kCtrS2M = 1, kCtrM2L = 2, kCtrS2L = 3, kCtrFar = 4, kNumCtr = 5 };
constexpr int kTileM = 128;  // target leaves per tile (TMEM lanes)
constexpr int kKBlock = 32;  // K values per pipeline stage (64-byte rows)
constexpr int kStages = 2;   // shared-memory stages
constexpr int kTileN = 80;   // table rows per tile
constexpr int kTileNSmall = 48;  // table rows per tile when 2p <= 48 (S2M, M2L, S2L at p <= 24)
constexpr int kTmemCols = 512;                  // allocation (power of two >= kNumAcc * kTileN)
constexpr int kEpilogueWarps = 8;
constexpr int kEpilogueThreads = 32 * kEpilogueWarps;
constexpr int kProducerThreads = 96;
constexpr int kMmaWarp = kEpilogueWarps + kProducerThreads / 32;  // 11
constexpr int kThreads = 32 * (kMmaWarp + 1);                     // 384: 3 warps per SM sub-partition
constexpr int kMaxSplit = 16;  // largest split-K factor (partial sums held for small contractions only)
static_assert(kNumAcc * kTileN <= kTmemCols, "TMEM budget");

// Table rows per tile (the MMA's N, TMEM columns per accumulator) of a gathered contraction whose tables have
// Rp rows: 80, or 48 for the 48-row tables of small expansions. The targets are its M side, 128 per group.
__host__ __device__ constexpr int table_rows_per_tile(int Rp) { return Rp % kTileN == 0 ? kTileN : kTileNSmall; }

// Splits v / 2^E (|v| < 2^E) into kSlices balanced base-128 digits, out[(i - 1) * stride] =
// d_i 2^(-7 i), with v / 2^E = sum_i d_i 2^(-7 i) + (|v| 2^(56 - E) - floor(|v| 2^(56 - E))) 2^-56:
// q = floor(|v| 2^(56 - E)) is written in base 128 from its low end, a digit of 64 or more becoming
// d - 128 with a carry into the next higher one, so d_2..d_8 lie in [-64, 63] and d_1 in [0, 128] (up to
// 256 for the tables in reflection classes, whose scale may be half of that);
// a negative v negates every digit. Each is an integer of at most 8 significant bits (exact in
// BF16), the products of two are below 2^14, and the first S digits are v / 2^E rounded to the
// nearest multiple of 2^(-7 S) (error at most 2^(-7 S - 1) of the scale 2^E). Integer work on the
// bits of v (its significand shifted to 56 fractional bits).
__device__ __forceinline__ void slice_fixed(double v, int E, __nv_bfloat16* out, int stride) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    int ev = (int)((bits >> 52) & 0x7FF);
    unsigned long long mant = bits & ((1ull << 52) - 1);
    if (ev) mant |= 1ull << 52;
    else ev = 1;
    // |v| 2^(56 - E) = mant 2^(ev - 1075 + 56 - E): a right shift by 1019 - ev + E (>= -4)
    const int shift = 1019 - ev + E;
    const unsigned long long q = shift >= 64 ? 0ull : (shift >= 0 ? mant >> shift : mant << (-shift));
    const bool neg = (bits >> 63) != 0;
    int carry = 0;
#pragma unroll
    for (int i = kSlices; i >= 1; --i) {
        int d = (int)((q >> (7 * (kSlices - i))) & (i > 1 ? 127ull : 511ull)) + carry;
        carry = (i > 1 && d >= 64) ? 1 : 0;
        d -= carry << 7;
        const float s = (float)(neg ? -d : d) * __int_as_float((127 - 7 * i) << 23);
        out[(i - 1) * stride] = __float2bfloat16_rn(s);
    }
}

// (double)x * 2^e for a float x from the bits, with integer operations only (the FP64 units are
// the scarce ones): sign and mantissa move over, the exponent is rebiased and shifted by e. A zero
// or subnormal x gives (signed) zero: the (hi, lo) outputs of the split contractions are
// normalised, so a part below 2^-126 is far below the rounding of the sum it belongs to. The
// result must lie in the normal double range.
__device__ __forceinline__ double f2d_scaled(float x, int e) {
    const unsigned int u = __float_as_uint(x);
    const int ex = (int)((u >> 23) & 0xFF);
    const unsigned long long sign = (unsigned long long)(u >> 31) << 63;
    const unsigned long long mag = ((unsigned long long)(ex - 127 + 1023 + e) << 52) |
                                   ((unsigned long long)(u & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)(sign | (ex == 0 ? 0ull : mag)));
}

// f2d_scaled(v.x, e) + f2d_scaled(v.y, e), rounded as that sum, by integer operations: lo in units of the
// last place of hi's double (half of it just below a power of two) is added to the bits. A pair whose lo
// is not below half an ulp of hi takes the FP64 addition; the contractions' outputs are normalised.
__device__ __forceinline__ double f2d_pair(float2 v, int e) {
    const unsigned u = __float_as_uint(v.x), l = __float_as_uint(v.y);
    const int ex = (int)((u >> 23) & 0xFF), lx = (int)((l >> 23) & 0xFF), d = ex - lx;
    if (lx != 0 && d < 24) return f2d_scaled(v.x, e) + f2d_scaled(v.y, e);
    const bool minus = (int)(u ^ l) < 0;
    const int unit = 150 + 29 + (minus && (u & 0x7FFFFFu) == 0 ? 1 : 0) - d;  // biased exponent of lo in units
    const int n = lx ? __float2int_rn(__uint_as_float(((unsigned)max(unit, 1) << 23 | (l & 0x7FFFFFu)))) : 0;
    const long long mag = ex ? (((long long)(ex - 127 + 1023 + e) << 52) | ((long long)(u & 0x7FFFFFu) << 29)) +
                                   (minus ? -n : n)
                             : 0ll;
    return __longlong_as_double(mag | ((long long)(u >> 31) << 63));
}

// Binary exponent e with |m| < 2^e (frexp convention), from the bits; 0 for m = 0.
__device__ __forceinline__ int exp_bound(double m) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(m);
    if ((bits << 1) == 0) return 0;
    const int ev = (int)((bits >> 52) & 0x7FF);
    return (ev ? ev : 1) - 1022;
}

// Offset of (row, slice 0, k) in a sliced operand [row][K block of 32][slice][32 values].
__device__ __forceinline__ size_t slice_at(size_t row, int Kp, int k) {
    return ((row * (Kp / kKBlock) + k / kKBlock) * kSlices) * kKBlock + (k % kKBlock);
}

// Level exponents of the M2L operand: G(l, r) = max over the boxes b of level l and the parts k
// (Re, Im of coefficient k / 2) of multipole row b of part_exp(value, k), kept as G + kGexpBias in
// an unsigned array that starts at zero, so that every producer of a multipole can take the maximum
// with atomicMax as it writes (order-independent, hence deterministic; skipped where the slot already holds
// as much, since the atomics of a level meet at one address).
constexpr unsigned kGexpBias = 1u << 20;

// frexp exponent of |v| (from the bits, integer work) plus floor(k / 4); INT_MIN for +-0.
__device__ __forceinline__ int part_exp(double v, int k) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    if ((bits << 1) == 0) return INT_MIN;
    const int ev = (int)((bits >> 52) & 0x7FF);
    return (ev ? ev : 1) - 1022 + (k >> 2);
}

// Warp-wide maximum of e, then one atomicMax into the biased level exponent (lanes with INT_MIN
// contribute nothing).
__device__ __forceinline__ void level_exp_max(int e, unsigned* slot) {
    for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if ((threadIdx.x & 31) == 0 && e != INT_MIN && (unsigned)(e + (int)kGexpBias) > __ldcg(slot))
        atomicMax(slot, (unsigned)(e + (int)kGexpBias));
}

// Block-wide maximum of e, then one atomicMax by thread 0 (every thread of the block must call it;
// at most 32 warps).
__device__ __forceinline__ void level_exp_max_block(int e, unsigned* slot) {
    __shared__ int wmax[32];
    for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)((blockDim.x + 31) >> 5); ++w) e = max(e, wmax[w]);
        if (e != INT_MIN && (unsigned)(e + (int)kGexpBias) > __ldcg(slot)) atomicMax(slot, (unsigned)(e + (int)kGexpBias));
    }
}

// Level exponent from its biased form.
__device__ __forceinline__ int level_exp_value(unsigned g) { return g ? (int)g - (int)kGexpBias : 0; }

// slice_fixed of 8 consecutive values (one exponent bound E) with each slice's 8 BF16 written
// by one 16-byte store: out + i * stride for slice i (16-byte aligned).
__device__ __forceinline__ void slice8_fixed(const double* v, int E, __nv_bfloat16* out, int stride) {
    __align__(16) __nv_bfloat16 tmp[kSlices][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) slice_fixed(v[j], E, &tmp[0][j], 8);
#pragma unroll
    for (int i = 0; i < kSlices; ++i) *reinterpret_cast<uint4*>(out + (size_t)i * stride) = *reinterpret_cast<uint4*>(tmp[i]);
}

// Sliced tables are stored tile by tile in the shared-memory image of a stage: [table][row tile][K block]
// [slice][tile row][64 bytes], each 64-byte row (32 values) in the 64-byte swizzle of the MMA operand
// (16-byte chunk c of row m at c ^ (m / 2 mod 4)). The slices that a contraction takes of one K block are
// one contiguous piece, fetched by one bulk copy. Offset (elements) of (table, slice 0, row, k) for
// tables of Rp rows in tiles of `tile` rows and Kp columns; slice i lies i * tile * kKBlock further on.
__host__ __device__ inline size_t table_at(size_t table, int Rp, int tile, int Kp, int row, int k) {
    const int rt = row / tile, m = row - rt * tile, kb = k / kKBlock, kk = k - kb * kKBlock;
    return ((((table * (Rp / tile) + rt) * (Kp / kKBlock) + kb) * kSlices * tile) + m) * kKBlock +
           ((((kk >> 3) ^ (m >> 1)) & 3) << 3) + (kk & 7);
}

// Shape of a contraction in reflection classes. Output rows [4][nch * N]: class c's rows (u, u_x, u_y of
// its quadrant nodes) from c * nch * N on, in nch tiles of N rows, the rest padding.
struct ClassTab {
    int norb = 0, k = 0, N = 0, nch = 0;
    int seg[13] = {};                                    // first row of (class, field) at 3 * class + field
    uint8_t fold[12] = {};                               // reflections that fix the orbit's representative
    int16_t K[12][4] = {}, nkb[12][4] = {};              // columns, K blocks
    int32_t toff[12][4] = {};                            // first table tile of (orbit, class), in K blocks
};

// Near field in reflection classes (mixed_sym.cu), or one gathered row per list entry (split_gemm) where a
// table is a single tile and K block: k <= 5. There a class has as many K blocks as a table and its rows
// fill a quarter of a tile (us per solve, classes / entries, 1,024 uniform and 900 graded leaves: k = 4
// 134 / 129 and 148 / 139, k = 5 131 / 133 and 150 / 139, k = 6 129 / 141 and 146 / 171).
__host__ __device__ constexpr bool near_by_classes(int k) { return 3 * k * k > kTileN || k * k > kKBlock; }

struct MixedOps {
    int N = kTileN; // table rows per tile
    int Rp = 0;     // 3k^2 rounded up to N
    int Kp = 0;     // k^2 rounded up to kKBlock
    // near field in reflection classes (mixed_sym.cu): tables of every (orbit, class), exponents of the
    // output rows
    ClassTab near;
    void* near_tab = nullptr;
    int* near_E = nullptr;
    // leaf far field the same way: orbit 0 L2T, 1..5 M2T
    ClassTab leaf;
    void* leaf_tab = nullptr;
    int* leaf_E = nullptr;
    // near field by entries: bf16 tables (table_at), 33, and their row exponents [Rp]
    void* tsl = nullptr;
    int* Er = nullptr;
    // far field: expansion coefficients as reals (Re, Im of 0..p), Kx = 2(p+1) padded
    int Kx = 0;           // 2(p+1) rounded up to kKBlock
    int Rx = 0;           // 2p rounded up to 48 (2p <= 48) or to kTileN (rows of S2M and M2L without coefficient 0)
    void* s2m_sl = nullptr;   // bf16 table: S2M rows 2..2p+1
    int* s2m_E = nullptr;     // [Rx]
    // M2L rows 2..2p+1 over input columns 0..2p+1, column k scaled by 2^-floor(k/4) (the decay
    // bound of multipole coefficient k/2), then per row by 2^-m2l_E[r]
    void* m2l_sl = nullptr;   // bf16 tables, 40
    int* m2l_E = nullptr;     // [Rx]
    void* far_sl = nullptr;   // bf16 tables, 21: L2T (0) and M2T per W configuration
    int* far_E = nullptr;     // [Rp]
    void* s2l_sl = nullptr;   // bf16 tables, 20: S2L rows of coefficients 1..p
    int* s2l_E = nullptr;     // [Rx]
    double* s2l_r0 = nullptr; // [20][kk] FP64: Re of S2L row 0
    double* m2l_r0 = nullptr; // [40][p+1] complex FP64: M2L row 0 (output coefficient 0) per offset
    // slices taken per contraction (kCtr*): the first S of the 8 stored slices of each operand and
    // the S(S+1)/2 products i + j <= S + 1. Default 6 for all (42 bits, 21 products): the error
    // against the FP64 form is then at most 6e-12 on the 20-Gaussian, kinked and uniform k = 16
    // workloads, 17x below 1e-10 (7 for all: 6e-14)
    int slices[kNumCtr] = {6, 6, 6, 6, 6};
};

// s + e = a + b exactly (FP32, round to nearest).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (hi, lo) += v in double-float with exact two-sums; df_final renormalises.
__device__ __forceinline__ void df_add(float& hi, float& lo, float2 v) {
    float s1, e1, s2, e2;
    two_sum(hi, v.x, s1, e1);
    two_sum(s1, v.y, s2, e2);
    hi = s2;
    lo = __fadd_rn(lo, __fadd_rn(e1, e2));
}

__device__ __forceinline__ float2 df_final(float hi, float lo) {
    const float h = __fadd_rn(hi, lo);
    return make_float2(h, __fsub_rn(lo, __fsub_rn(h, hi)));
}

struct MixedWork {
    void* fsl = nullptr;                  // bf16 [n_leaves][kSlices][Kp]
    float2* out = nullptr;                // near field (hi, lo): class rows [n_leaves][4 nch N], scaled by
                                          // 2^-(E_f + 1 + E_r), or node rows [n_leaves][Rp], by 2^-(E_f + E_r)
    long long* ffix = nullptr;            // [R][n_leaves][k^2] f 2^(59 - E_f), truncated (near field)
    void* near_opnd = nullptr;            // near field's operand tiles, a chunk at a time
    size_t near_opnd_bytes = 0;
    int near_split = 1, leaf_split = 1;   // partial sums in out and far_out, one row set after another (by classes)
    unsigned long long* fmax = nullptr;   // [R] max |f| per right-hand side (bits)
    int* Ef = nullptr;                    // [R] exponent of f per right-hand side
    int* err = nullptr;                   // non-zero after a bounded wait expired
    // far field
    float2* s2m_out = nullptr;            // [n_leaves][Rx]
    unsigned* glev = nullptr;             // [(depth + 1) * R] G(l, r) + kGexpBias (0: level all zero):
                                          // |multipole part k| 2^floor(k/4) < 2^G for parts k = 0 .. 2p+1
    void* msl = nullptr;                  // bf16 [n_boxes][kSlices][Kx]
    float2* m2l_out = nullptr;            // [n_boxes][Rx]
    double* m2l_c0 = nullptr;             // [n_boxes] Re local coefficient 0 from the V and X lists
    float2* s2l_out = nullptr;            // [n_boxes][Rx]
    void* aprep = nullptr;                // bf16 [n_far_slots][kSlices][Kx], or the classes' operand tiles, a chunk at a time
    size_t aprep_bytes = 0;
    int* bexp = nullptr;                  // [n_boxes] exponent bounds of the multipoles (far field by classes)
    int* Et = nullptr;                    // [n_leaves]
    float2* far_out = nullptr;            // [n_leaves][Rp], or class rows [n_leaves][4 nch N]
    float2* part = nullptr;               // partial sums or slab of S2M, M2L and the leaf far field
    float2* part_side = nullptr;          // partial sums or slab of the near field by entries
    float2* part_s2l = nullptr;           // partial sums or slab of S2L
    cudaEvent_t* cev = nullptr;           // optional (start, stop) pairs: near, S2M, M2L, S2L, far
};

// Host staging of the index arrays of one plan set: put() appends an array and returns its offset
// (int32 elements; pieces start on 256-byte boundaries); commit_plan_arena() makes one device
// allocation, copies everything once and points every plan of the set (and its alternative form)
// into it.
struct PlanArena {
    std::vector<int32_t> data;
    int64_t put(const std::vector<int32_t>& v) {
        const int64_t off = (int64_t)data.size();
        const size_t len = std::max<size_t>(64, (v.size() + 63) / 64 * 64);
        data.resize(off + len, 0);
        std::copy(v.begin(), v.end(), data.begin() + off);
        return off;
    }
};
int commit_plan_arena(PlanArena& A, PlanSet* PS, cudaStream_t st);

// Targets of one split contraction in flat form: target t (output row tgt[t]) holds the items
// (tab[e], src[e]) = (table, gathered operand row), e in [ptr[t], ptr[t + 1]), and sorts by key[t].
struct PlanItems {
    std::vector<int32_t> tgt, ptr{0}, tab, src;
    std::vector<std::pair<uint64_t, uint64_t>> key;
    void add(int32_t table, int32_t row) {
        tab.push_back(table);
        src.push_back(row);
    }
    void close(int32_t id, uint64_t k0, uint64_t k1) {  // ends the target whose items were just added
        tgt.push_back(id);
        ptr.push_back((int32_t)tab.size());
        key.push_back({k0, k1});
    }
};
// Groups of 128 targets taken in the given order; per group the tables present
// and, per table, the gathered row of each target (-1 when the target has no entry for that table).
int build_split_plan(const PlanItems& I, const std::vector<int32_t>& order, int n_tables, int n_chunks, int R,
                     int nkb, PlanArena& A, SplitPlan* P);
// build_split_plan, or its entry-major form when that executes enough fewer columns: chosen when
// (entry-major columns) x (1 + slab_overhead) < 0.85 x (grouped columns, padding included) and the
// slab (entries x R x slab_row_bytes) stays within 256 MB. slab_overhead = the slab's write and read
// time per column relative to its tensor time. A small contraction (fewer CTAs than two per SM)
// whose slab fits keeps the form not chosen in P->alt.
int build_contraction_plan(const PlanItems& I, int n_tables, int n_chunks, int R, int nkb,
                           double slab_overhead, size_t slab_row_bytes, PlanArena& A, SplitPlan* P);
// ev (optional): a (start, stop) event pair recorded around the contraction and its reduction.
int split_gemm(const SplitPlan& P, const void* asl, const void* tables, int Kp, int Rp, float2* out, int* err,
               float2* part, size_t n_out_rows, int slices, cudaStream_t st, cudaEvent_t* ev = nullptr,
               int defer = 0);
// split_gemm's `defer` bits: the consumer of the output sums the entry-major slab rows of each
// target (kDeferSegments) or the split-K partial sums (kDeferSplits) itself, in the same order and
// arithmetic as the reduction kernels, which are then not launched
constexpr int kDeferSegments = 1;
constexpr int kDeferSplits = 2;
// Partial-sum elements (float2) of the three buffers whose contractions may run at the same time:
// [0] S2M, M2L and the leaf far field (one after another), [1] S2L, [2] the near field by entries.
void split_part_elems(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, size_t elems[3]);
int build_mixed_plan(DeviceTree* T, cudaStream_t st);
// Host copies of the tree arrays the plan builders read (fetched once per plan set).
struct HostLists {
    std::vector<int32_t> bol, lob, ptr[4], idx[4], cfg[4];
};
int fetch_host_lists(const DeviceTree& T, HostLists* H);
int build_far_slots(DeviceTree* T, const HostLists& H, cudaStream_t st);
// Plan of one far-field contraction (kCtrS2M, kCtrM2L, kCtrS2L or kCtrFar) into PS.
int build_far_plan(int which, const DeviceTree& T, int R, const HostLists& H, PlanArena& A, PlanSet* PS);
// max |f| and the f slices (operand of S2M and S2L).
int near_slices(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, const MixedWork& w,
                cudaStream_t st);
// Near field (by classes or by entries).
int near_contract(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, const MixedWork& w,
                  cudaStream_t st);
// Reflection classes (mixed_sym.cu): tables, plans, operand buffers, contractions and the kernels they launch.
int near_classes_prepare(vfmm_ops* o, cudaStream_t st);
int leaf_classes_prepare(vfmm_ops* o, const std::vector<double>& F, cudaStream_t st);
int build_near_classes(const DeviceTree& T, int R, const HostLists& H, PlanArena& A, ClassPlan* P);
int build_leaf_classes(const DeviceTree& T, int R, const HostLists& H, PlanArena& A, ClassPlan* P);
size_t class_operand_bytes(const ClassTab& ct, const ClassPlan& P, size_t room);
double class_tiles(const ClassTab& ct, const ClassPlan& P);  // operand tiles of all pieces
int near_class_contract(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, const MixedWork& w,
                        cudaStream_t st);
// exponent bounds of the multipoles, before leaf_class_contract (trees of depth 2 and more)
int leaf_class_bounds(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* Mexp, const MixedWork& w,
                      cudaStream_t st);
int leaf_class_contract(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* Mexp, const double* Lexp,
                        const MixedWork& w, cudaStream_t st);
// Slices that the leaf far field takes in reflection classes: one more than set. A node's images share the
// rounding of the largest of them. On 1,219 leaves its error is 2.3e-12 of the largest u_x at 6 slices
// (gathered form: 3.0e-12) and 2.4e-14 at 7, on 200,104 leaves 4.2e-12 (5.2e-12) and 4.1e-14, for 3 % of a solve.
inline int leaf_class_slices(const MixedOps& mo) { return mo.slices[kCtrFar] < kSlices ? mo.slices[kCtrFar] + 1 : kSlices; }
int class_launches(const ClassTab& ct, const ClassPlan& P, int S, size_t opnd_bytes);
int far_prepare(vfmm_ops* o, cudaStream_t st);
void far_free(MixedOps* mo);
// Stages of the split-precision far field (see mixed_far.cu). Multipoles and locals are stored per
// virtual box (box * R + r); f is [R][n_leaves][k^2].
int s2m_mixed(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, double* Mexp,
              const MixedWork& w, cudaStream_t st);
int m2l_mixed(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* Mexp, const MixedWork& w,
              cudaStream_t st);
int s2l_mixed(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const MixedWork& w, cudaStream_t st);
int far_leaf_mixed(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* Mexp, const double* Lexp,
                   const MixedWork& w, cudaStream_t st);

}  // namespace vfmm
