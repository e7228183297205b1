// Split-BF16 near field and leaf far field (L2T, M2T) in the reflection classes of sym.cuh (VFMM_MIXED).
//
// The arithmetic is that of mixed.cu (power-of-two scales, balanced base-128 digits, slice products by
// diagonal, exact drains into double-FP32). What differs is the contraction:
//  * targets are leaves (128 per group, leaves with the same set of orbits together), the MMA's M side;
//    the table rows of one class (a quarter of the leaf's 3k^2) are its N side;
//  * the operand of (leaf, orbit, class) is g = sum_s chi(s) f_{sR}(s y), summed from fixed-point values
//    (integers; FP64 additions are the scarce ones) and written by class_operand_kernel as the digits of
//    a tile in the order and swizzle in which the MMA reads it. A stage of the pipeline is then two bulk
//    copies of contiguous memory by one thread.
//  * |f| < 2^E makes |g| < 2^(E+2); E + 1 is the scale all the same: the top digit of a tile may be as
//    large as 256, which BF16 holds. What this costs an orbit with a single member, its last slice makes up
//    for: not a whole digit but all that is left, rounded to BF16 (at most 1/8 of the digit's unit).
//  * a table row's scale is half its largest entry's power of two (top digits up to 256) wherever the entries of
//    a K block are on average no larger than that scale (755 of the near field's 768 rows at k = 16): half the
//    weight of the slice products left out. Per K value diagonals 0 to 4 then sum to at most 36,864 units, 448 of
//    them below 2^24: diagonal 0 to 256 x 128 (the table's average), diagonal 4 to 256 x 64 + 3 x 64^2
//    + 64 x 128. The sixth accumulator (diagonals from 5 on, 40,960 units at S = 6) may round by 2^-49 of
//    the scales' product where its sum is past 2^24 units, 1/400 of what the products left out may weigh.
//  * the outputs of a class are put together at the nodes by the leaf kernel (double-FP32).
// The leaf far field does the same with the leaf's local (one K block per class) and its W orbits, scaled
// per leaf: with E_t the exponent of its largest coefficient and m the most boxes in one of its orbits,
// by 2^(E_t - 1 + ceil(log2 m)), which the top digit's range covers. The local goes in once with tables
// four times as large (not as the sum of its four reflections), so that its rows keep their bits.
// Operand tiles are made and consumed in chunks that fit the workspace's buffer.
//
// What bounds it: a K block of 128 x 64 outputs moves 207 KB through shared memory (72 KB written, the A
// tiles once, the B tiles once per product), 1,620 cycles; the MMAs take 1,700 of the 2,220 cycles measured,
// 300 go to operands not yet there and 220 to drains. The operand is bound by HBM writes and integer work.
// Against gathered rows and plain tables (ms): 200,104 graded leaves 13.3 -> 8.1, 16,384 uniform leaves
// k = 16 1.32 -> 0.39, 1,378 graded leaves 0.18 -> 0.11, 4,096 rows of k = 8 0.081 -> 0.034; the far field of
// the 200,104 leaves 4.1 -> 1.9. Error against the FP64 form at 6 slices, largest of u_x: near field on 1,219
// graded leaves 3.5e-12 -> 1.7e-12, far field (7 slices here) 3.0e-12 -> 2.4e-14.
// k <= 5 keeps the gathered rows: its class rows fill half a tile of 48.
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <vector>

#include "mixed.cuh"
#include "mma_issue.cuh"
#include "ops.cuh"
#include "sym.cuh"
#include "tc_ptx.cuh"
#include "vfmm_internal.cuh"

namespace vfmm {

using bf16 = __nv_bfloat16;

constexpr int kClsEpilogueWarps = 8;
constexpr int kClsEpilogueThreads = 32 * kClsEpilogueWarps;
constexpr int kClsThreads = kClsEpilogueThreads + 64;  // + producer warp + MMA warp
constexpr int kClsMaxStages = 4;
constexpr int kClsDrain = 14;  // K blocks summed in TMEM between two drains (448 K values)
constexpr size_t kClsSmem = 224 * 1024;
constexpr size_t kClsUnit = kTileM * 64;  // bytes of one slice of an operand tile

// ---------------------------------------------------------------- tables
// E[output row] = scale of that row over the orbits (0: padding). A class has its own: for the smooth
// potential tables the odd ones are far smaller than the even one. With e the exponent of the row's largest
// entry it is e - 1 if no K block's entries sum to more than 31.8 2^(e - 1) (32 top digits then sum to at
// most 31.8 x 128 and 32 carries, below 32 x 128), else e.
__global__ void __launch_bounds__(256) class_row_exp_kernel(SymOp op, ClassTab ct, int* __restrict__ E) {
    __shared__ double red[8], reds[8];
    const int c = blockIdx.x / (ct.nch * ct.N), r = blockIdx.x - c * (ct.nch * ct.N);
    double m = 0.0, ms = 0.0;
    if (r < op.M[c])
        for (int o = 0; o < op.norb; ++o) {
            const double* A = op.A + op.off[o][c] + r;
            const int Kp = ct.nkb[o][c] * kKBlock;  // a warp takes whole K blocks
            for (int col = threadIdx.x; col < Kp; col += blockDim.x) {
                const double v = col < op.K[o][c] ? fabs(A[(size_t)col * op.M[c]]) : 0.0;
                double s = v;
                for (int x = 16; x > 0; x >>= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
                m = fmax(m, v);
                ms = fmax(ms, s);
            }
        }
    for (int x = 16; x > 0; x >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, x));
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = m;
        reds[threadIdx.x >> 5] = ms;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            m = fmax(m, red[w]);
            ms = fmax(ms, reds[w]);
        }
        const int e = m > 0.0 ? exp_bound(m) : 0;
        E[blockIdx.x] = m > 0.0 && ms <= ldexp(31.8, e - 1) ? e - 1 : e;
    }
}
static_assert(kKBlock == 32, "a K block per warp");

// Digits of every table, tile by tile (table_at with one orbit's class as a table of nch * N rows).
__global__ void class_table_kernel(SymOp op, ClassTab ct, const int* __restrict__ E, bf16* __restrict__ out) {
    const int o = blockIdx.y >> 2, c = blockIdx.y & 3, r = blockIdx.x;  // padded row of the class
    const int K = op.K[o][c], Kp = ct.nkb[o][c] * kKBlock, e = E[c * ct.nch * ct.N + r];
    bf16* base = out + (size_t)ct.toff[o][c] * kSlices * ct.N * kKBlock;
    for (int col = threadIdx.x; col < Kp; col += blockDim.x) {
        const double v = r < op.M[c] && col < K ? op.A[op.off[o][c] + (size_t)col * op.M[c] + r] : 0.0;
        slice_fixed(v, e, base + table_at(0, ct.nch * ct.N, ct.N, Kp, r, col), ct.N * kKBlock);
    }
}

// Row tiles of a class: width N and number, the fewest cycles per K block (measured per MMA at the tensor
// pipe's rate, with 16 for the tile's loads).
static void class_tile_rows(int k, int* N, int* nch) {
    int mmax = 0;
    for (int c = 0; c < 4; ++c) {
        int m = 0;
        for (int q = 0; q < 3; ++q) m += sym_half(k, sym_pa(c, q)) * sym_half(k, sym_pb(c, q));
        mmax = std::max(mmax, m);
    }
    const int width[3] = {48, 64, 80};
    const double cycles[3] = {29.5 + 16, 35.6 + 16, 41.6 + 16};
    double best = 1e300;
    for (int i = 0; i < 3; ++i) {
        const int n = (mmax + width[i] - 1) / width[i];
        if (n * cycles[i] < best) {
            best = n * cycles[i];
            *N = width[i];
            *nch = n;
        }
    }
}

// CTAs that share a piece's K blocks where the pieces alone leave SMs idle: their partial sums are added by
// the leaf kernel, so a share is at least six K blocks (184 leaves, k = 16: 66 K blocks on 24 CTAs took 75
// us, half the solve).
static int class_split(int n_groups, int nch, double units) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int items = std::max(1, 4 * n_groups * nch);
    return std::max(1, std::min({8, sms / items, (int)(units / (4.0 * std::max(1, n_groups)) / 6.0)}));
}

static int class_prepare(SymOp& op, ClassTab& ct, void** tab, int** E, cudaStream_t st) {
    const int k = op.k;
    class_tile_rows(k, &ct.N, &ct.nch);
    ct.norb = op.norb;
    ct.k = k;
    int64_t tiles = 0;
    for (int x = 0; x < op.norb; ++x) {
        ct.fold[x] = (op.fx[x] ? 1 : 0) | (op.fy[x] ? 2 : 0);
        for (int c = 0; c < 4; ++c) {
            ct.K[x][c] = op.K[x][c];
            ct.nkb[x][c] = (op.K[x][c] + kKBlock - 1) / kKBlock;
            ct.toff[x][c] = (int)tiles;
            tiles += (int64_t)ct.nkb[x][c] * ct.nch;
        }
    }
    for (int i = 0; i < 13; ++i) {
        // node rows of class c start at c * nch * N of an output row
        const int c = std::min(3, i / 3);
        ct.seg[i] = i < 12 ? op.seg[i] - op.roff[c] + c * ct.nch * ct.N : 4 * ct.nch * ct.N;
    }
    const int rows = 4 * ct.nch * ct.N;
    VFMM_CUDA(cudaMalloc(E, rows * sizeof(int)));
    VFMM_CUDA(cudaMalloc(tab, (size_t)tiles * kSlices * ct.N * kKBlock * sizeof(bf16)));
    class_row_exp_kernel<<<rows, 256, 0, st>>>(op, ct, *E);
    class_table_kernel<<<dim3(ct.nch * ct.N, 4 * op.norb), 128, 0, st>>>(op, ct, *E, (bf16*)*tab);
    VFMM_CUDA(cudaGetLastError());
    VFMM_CUDA(cudaStreamSynchronize(st));
    return VFMM_OK;
}

int near_classes_prepare(vfmm_ops* o, cudaStream_t st) {
    MixedOps* mo = (MixedOps*)o->mixed;
    SymOp op;
    int rc = sym_near_op(o, &op, st);
    if (rc == VFMM_OK) rc = class_prepare(op, mo->near, &mo->near_tab, &mo->near_E, st);
    if (op.A) cudaFree(op.A);
    return rc;
}

// F0: L2T without coefficient 0 and the M2T tables [21][3 k^2][2(p+1)].
int leaf_classes_prepare(vfmm_ops* o, const std::vector<double>& F0, cudaStream_t st) {
    MixedOps* mo = (MixedOps*)o->mixed;
    std::vector<double> F = F0;
    for (size_t i = 0; i < F.size() / (1 + kFarCfg); ++i) F[i] *= 4.0;  // the local is no sum of four
    double* dF = nullptr;
    VFMM_CUDA(cudaMalloc(&dF, F.size() * sizeof(double)));
    SymOp op;
    cudaError_t e = cudaMemcpyAsync(dF, F.data(), F.size() * sizeof(double), cudaMemcpyHostToDevice, st);
    int rc = e == cudaSuccess ? sym_far_op(o, dF, &op, st) : cuda_fail(e, "cudaMemcpyAsync");
    if (rc == VFMM_OK) rc = class_prepare(op, mo->leaf, &mo->leaf_tab, &mo->leaf_E, st);
    cudaStreamSynchronize(st);
    cudaFree(dF);
    if (op.A) cudaFree(op.A);
    return rc;
}

// ---------------------------------------------------------------- plan
// K blocks of class c over the orbits of a group's mask, from the node counts alone.
static int class_units(int k, uint32_t mask, int c) {
    int u = 0;
    for (int o = 0; o < kNearOrb; ++o) {
        if (!((mask >> o) & 1u)) continue;
        const int fx = o == 0 || o == 2, fy = o == 0 || o == 1;  // (0, 0), (0, 1): mx; (0, 0), (1, 0): my
        const int K = (fx ? sym_half(k, c & 1) : k) * (fy ? sym_half(k, c >> 1) : k);
        u += (K + kKBlock - 1) / kKBlock;
    }
    return u;
}

// Leaves in the order of their masks (n_masks of them), groups of 128 virtual leaves and their masks.
static int class_groups(const DeviceTree& T, int R, const std::vector<uint16_t>& mask, int n_masks, PlanArena& A,
                        ClassPlan* P, std::vector<int32_t>& gmask) {
    const int nl = T.n_leaves;
    const int64_t nv = (int64_t)nl * R;
    if (nv > (int64_t)INT32_MAX / 2) return fail(VFMM_ERR_INVALID_ARG, "too many rows for one split contraction");
    std::vector<int32_t> start(n_masks + 1, 0), order(nl);
    for (int t = 0; t < nl; ++t) ++start[mask[t] + 1];
    for (int m = 0; m < n_masks; ++m) start[m + 1] += start[m];
    for (int t = 0; t < nl; ++t) order[start[mask[t]]++] = t;
    P->n_groups = (int32_t)((nv + kTileM - 1) / kTileM);
    gmask.assign(P->n_groups, 0);
    for (int g = 0; g < P->n_groups; ++g) {
        const int64_t t0 = (int64_t)g * kTileM / R, t1 = (std::min<int64_t>((int64_t)(g + 1) * kTileM, nv) - 1) / R;
        for (int64_t t = t0; t <= t1; ++t) gmask[g] |= mask[order[t]];
    }
    P->off[0] = A.put(order);
    P->off[1] = A.put(gmask);
    return VFMM_OK;
}

int build_near_classes(const DeviceTree& T, int R, const HostLists& H, PlanArena& A, ClassPlan* P) {
    const std::vector<int32_t>&ptr = H.ptr[VFMM_LIST_U], &cfg = H.cfg[VFMM_LIST_U];
    uint16_t bit[kNearCfg];
    for (int c = 0; c < kNearCfg; ++c) {
        int slots;
        bit[c] = (uint16_t)(1u << sym_orbit(VFMM_LIST_U, c, &slots));
    }
    std::vector<uint16_t> mask(T.n_leaves, 0);
    for (int t = 0; t < T.n_leaves; ++t)
        for (int e = ptr[H.bol[t]]; e < ptr[H.bol[t] + 1]; ++e) mask[t] |= bit[cfg[e]];
    std::vector<int32_t> gmask;
    VFMM_CHECK(class_groups(T, R, mask, 1 << kNearOrb, A, P, gmask));
    P->first.assign(4 * (size_t)P->n_groups + 1, 0);
    int64_t units = 0;
    for (int p = 0; p < 4 * P->n_groups; ++p) {
        const int u = class_units(T.k, (uint32_t)gmask[p >> 2], p & 3);
        P->max_units = std::max(P->max_units, u);
        units += u;
        if (units > INT32_MAX) return fail(VFMM_ERR_INVALID_ARG, "too many operand tiles");
        P->first[p + 1] = (int32_t)units;
    }
    int N, nch;
    class_tile_rows(T.k, &N, &nch);
    P->split = class_split(P->n_groups, nch, (double)units);
    P->off[2] = A.put(P->first);
    return VFMM_OK;
}

// Orbit 0 (the leaf's own local) in every group, then the W orbits.
int build_leaf_classes(const DeviceTree& T, int R, const HostLists& H, PlanArena& A, ClassPlan* P) {
    const std::vector<int32_t>&ptr = H.ptr[VFMM_LIST_W], &cfg = H.cfg[VFMM_LIST_W];
    uint16_t bit[kFarCfg];
    for (int c = 0; c < kFarCfg; ++c) {
        int slots;
        bit[c] = (uint16_t)(2u << sym_orbit(VFMM_LIST_W, c, &slots));
    }
    std::vector<uint16_t> mask(T.n_leaves, 1);
    for (int t = 0; t < T.n_leaves; ++t)
        for (int e = ptr[H.bol[t]]; e < ptr[H.bol[t] + 1]; ++e) mask[t] |= bit[cfg[e]];
    std::vector<int32_t> gmask;
    VFMM_CHECK(class_groups(T, R, mask, 2 << kFarOrb, A, P, gmask));
    P->orbits.assign((size_t)P->n_groups + 1, 0);
    for (int g = 0; g < P->n_groups; ++g) {
        int n = 0;
        for (int o = 1; o <= kFarOrb; ++o) n += (gmask[g] >> o) & 1;
        P->max_units = std::max(P->max_units, n);
        P->orbits[g + 1] = P->orbits[g] + n;
    }
    int N, nch;
    class_tile_rows(T.k, &N, &nch);
    // three K blocks per W orbit (p up to 47; only this choice depends on it)
    P->split = class_split(P->n_groups, nch, 4.0 * (P->n_groups + 3.0 * P->orbits.back()));
    P->off[2] = A.put(P->orbits);
    return VFMM_OK;
}

// Operand tiles before a piece, host and device; U: the piece's own.
struct ClassSpans {
    const int32_t* first;   // near field, or null
    const int32_t* orbits;  // leaf far field
    int nkb;                // its K blocks per W orbit (one for the local)
};
__host__ __device__ inline long long class_span(const ClassSpans& s, int p, int* U) {
    if (s.first) {
        if (U) *U = s.first[p + 1] - s.first[p];
        return s.first[p];
    }
    const int g = p >> 2, c = p & 3;
    const int u = c || U ? 1 + s.nkb * (s.orbits[g + 1] - s.orbits[g]) : 0;
    if (U) *U = u;
    return 4 * ((long long)g + (long long)s.nkb * s.orbits[g]) + (long long)c * u;
}
static ClassSpans host_spans(const ClassTab& ct, const ClassPlan& P) {
    return ClassSpans{P.first.empty() ? nullptr : P.first.data(), P.orbits.empty() ? nullptr : P.orbits.data(),
                      ct.norb > 1 ? ct.nkb[1][0] : 0};
}
static ClassSpans device_spans(const ClassTab& ct, const ClassPlan& P) {
    return ClassSpans{P.first.empty() ? nullptr : P.first_dev, P.first.empty() ? P.first_dev : nullptr,
                      ct.norb > 1 ? ct.nkb[1][0] : 0};
}

double class_tiles(const ClassTab& ct, const ClassPlan& P) {
    return P.n_groups ? (double)class_span(host_spans(ct, P), 4 * P.n_groups, nullptr) : 0.0;
}

// Bytes of the operand buffer: all tiles at once, up to 768 MB; more take turns in it. room (not 0): as many
// as fit in it. At least the largest piece's.
size_t class_operand_bytes(const ClassTab& ct, const ClassPlan& P, size_t room) {
    if (P.n_groups == 0) return 0;
    const size_t all = (size_t)class_tiles(ct, P) * kSlices * kClsUnit;
    const size_t most = P.first.empty() ? 1 + (size_t)P.max_units * ct.nkb[1][0] : (size_t)P.max_units;
    return std::max(std::min(all, room ? room : size_t(768) << 20), most * kSlices * kClsUnit);
}

// Chunks of pieces [p0, p1) whose tiles fit the buffer.
template <class Chunk>
static int class_chunks(const ClassTab& ct, const ClassPlan& P, int S, size_t bytes, Chunk&& chunk) {
    const ClassSpans sp = host_spans(ct, P);
    const int64_t room = (int64_t)(bytes / (S * kClsUnit));
    for (int p0 = 0; p0 < 4 * P.n_groups;) {
        const int64_t at = class_span(sp, p0, nullptr);
        int p1 = p0 + 1;
        while (p1 < 4 * P.n_groups && class_span(sp, p1 + 1, nullptr) - at <= room) ++p1;
        if (class_span(sp, p1, nullptr) - at > room) return fail(VFMM_ERR_INTERNAL, "operand buffer too small");
        VFMM_CHECK(chunk(p0, p1));
        p0 = p1;
    }
    return VFMM_OK;
}

int class_launches(const ClassTab& ct, const ClassPlan& P, int S, size_t opnd_bytes) {
    int n = 0;
    class_chunks(ct, P, S, opnd_bytes, [&](int, int) {
        n += 2;
        return (int)VFMM_OK;
    });
    return n;
}

// ---------------------------------------------------------------- operand
struct ClassOperandArgs {
    ClassTab ct;
    int S, R, nleaf, nv;
    long long bias;      // class_bias(S)
    int p0, p1;          // pieces (4 * group + class) of this chunk
    const int32_t* order;
    const int32_t* gmask;
    ClassSpans spans;
    const int32_t* box_of_leaf;
    const int32_t* inst_ptr;
    const int4* inst_src;
    const uint32_t* inst_mask;
    const long long* f;  // fixed-point leaf values (class_fixed_kernel)
    // leaf far field: expansions of the virtual boxes, exponent bounds, the leaves' scales (written)
    const double *Mexp, *Lexp;
    const int* bexp;
    const int32_t *wptr, *widx;
    int* Et;
    unsigned char* out;  // chunk's tiles: K block u of piece p at (span(p) - span(p0) + u) * S * kClsUnit
};

// floor(|v| 2^(60 - E)) with v's sign (|v| < 2^(E + 1)), integer work.
__device__ __forceinline__ long long fixed60(double v, int E) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    int ev = (int)((bits >> 52) & 0x7FF);
    unsigned long long mant = bits & ((1ull << 52) - 1);
    if (ev) mant |= 1ull << 52;
    else ev = 1;
    const int shift = 1015 - ev + E;
    const long long q = (long long)(shift >= 64 ? 0ull : (shift >= 0 ? mant >> shift : mant << (-shift)));
    return (bits >> 63) ? -q : q;
}

// q[r][i] = f[r][i] 2^(59 - E_f[r]), truncated: the fixed-point values that the operand sums.
__global__ void __launch_bounds__(256) class_fixed_kernel(const double* __restrict__ f, int64_t n,
                                                          const int* __restrict__ Ef, long long* __restrict__ q) {
    const int E = Ef[blockIdx.y] + 1;
    const size_t base = (size_t)blockIdx.y * n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        q[base + i] = fixed60(f[base + i], E);
}

// S slices of 4 values q 2^-60 (|q| < 2^61): slices 1 .. S - 1 balanced base-128 digits, d_i = digit i of
// q + bias less 64 (the top one as it is), bias = 64 of each later digit's unit; the last slice what is left,
// less than 64 units of 2^(-7 S), rounded to BF16. 8-byte stores, slice i at out + i * kClsUnit.
__device__ __forceinline__ void class_digits4(const long long* q, int S, long long bias, unsigned char* out) {
    constexpr float kMagic = 12582912.0f;  // 1.5 2^23: an integer below 2^22 added to its bits is added to it
    long long b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = q[e] + bias;
    auto store = [&](int i, const float* v) {
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
        *reinterpret_cast<uint2*>(out + (size_t)i * kClsUnit) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    };
    float v[4];
#pragma unroll
    for (int i = 0; i < kSlices - 1; ++i) {
        if (i >= S - 1) break;
        const int shift = 53 - 7 * i;
        const float sc = __int_as_float((127 - 7 * (i + 1)) << 23);
        const float zero = (i == 0 ? kMagic : kMagic + 64.0f) * sc;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int d = (int)(b[e] >> shift);
            v[e] = fmaf(__int_as_float(0x4B400000 + (i == 0 ? d : d & 127)), sc, -zero);
        }
        store(i, v);
    }
    const int low = 67 - 7 * S;  // bits below digit S - 1 (25 at S = 6); exact in FP32
#pragma unroll
    for (int e = 0; e < 4; ++e)
        v[e] = (float)(((int)b[e] & ((1 << low) - 1)) - (1 << (low - 1))) * __int_as_float((127 - 60) << 23);
    store(S - 1, v);
}
static long long class_bias(int S) {
    long long b = 0;
    for (int i = 1; i < S; ++i) b += 64ll << (53 - 7 * i);
    return b;
}

// One CTA per (group, orbit) and share of its K blocks, thread = (target row, 4 columns of a 64-byte row), so that
// the sources of a row are looked up once for all its columns. The four classes share their loads and
// sums wherever a column is the same node for all (every orbit off the axes, every orbit for even k).
__global__ void __launch_bounds__(1024) class_operand_kernel(const __grid_constant__ ClassOperandArgs a) {
    __shared__ int4 s_src[kTileM];
    __shared__ int s_r[kTileM];
    const int g = a.p0 / 4 + blockIdx.x, o = blockIdx.y, k = a.ct.k, kk = k * k;
    const uint32_t gm = (uint32_t)a.gmask[g];
    if (!((gm >> o) & 1u)) return;
    if (threadIdx.x < kTileM) {
        const int64_t v = (int64_t)g * kTileM + threadIdx.x;
        int4 s = make_int4(-1, -1, -1, -1);
        int r = 0;
        if (v < a.nv) {
            const int leaf = a.order[v / a.R], b = a.box_of_leaf[leaf];
            r = (int)(v % a.R);
            const uint32_t mk = a.inst_mask[b];
            if ((mk >> o) & 1u) s = a.inst_src[a.inst_ptr[b] + __popc(mk & ((1u << o) - 1u))];
        }
        s_src[threadIdx.x] = s;
        s_r[threadIdx.x] = r;
    }
    int before[4] = {0, 0, 0, 0}, nkb = 0;  // K blocks of the orbits before this one
    for (int x = 0; x < o; ++x)
        if ((gm >> x) & 1u)
            for (int c = 0; c < 4; ++c) before[c] += a.ct.nkb[x][c];
    for (int c = 0; c < 4; ++c) nkb = max(nkb, (int)a.ct.nkb[o][c]);
    __syncthreads();
    const int m = threadIdx.x >> 3, c4 = threadIdx.x & 7;
    const int4 src = s_src[m];
    const int fold = a.ct.fold[o];
    const long long* f = a.f + (size_t)s_r[m] * a.nleaf * kk;
    const long long* f0 = f + (size_t)max(src.x, 0) * kk;
    const long long* f1 = f + (size_t)max(src.y, 0) * kk;
    const long long* f2 = f + (size_t)max(src.z, 0) * kk;
    const long long* f3 = f + (size_t)max(src.w, 0) * kk;
    const size_t row = (size_t)m * 64 + ((((c4 >> 1) ^ (m >> 1)) & 3) << 4) + ((c4 & 1) << 3);
    const bool shared = fold == 0 || (k & 1) == 0;
    const long long at0 = class_span(a.spans, a.p0, nullptr);
    for (int kb = blockIdx.z; kb < nkb; kb += gridDim.z) {
        const int col0 = kb * kKBlock + c4 * 4;
        auto tile = [&](int c) {
            return a.out + (size_t)(class_span(a.spans, 4 * g + c, nullptr) - at0 + before[c] + kb) * a.S * kClsUnit + row;
        };
        auto mine = [&](int c) { return 4 * g + c >= a.p0 && 4 * g + c < a.p1 && kb < a.ct.nkb[o][c]; };
        for (int c0 = 0; c0 < (shared ? 1 : 4); ++c0) {
            if (!shared && !mine(c0)) continue;
            const int nx = (fold & 1) ? sym_half(k, c0 & 1) : k, K = a.ct.K[o][c0];
            int j = col0 / nx, i = col0 - j * nx;
            long long s0[4], s1[4], s2[4], s3[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool in = col0 + e < K;
                const int up = j * k, dn = (k - 1 - j) * k;
                s0[e] = in && src.x >= 0 ? __ldg(f0 + up + i) : 0;
                s1[e] = in && src.y >= 0 ? __ldg(f1 + up + k - 1 - i) : 0;
                s2[e] = in && src.z >= 0 ? __ldg(f2 + dn + i) : 0;
                s3[e] = in && src.w >= 0 ? __ldg(f3 + dn + k - 1 - i) : 0;
                if (++i == nx) {
                    i = 0;
                    ++j;
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const long long x = s0[e] + s1[e], y = s0[e] - s1[e], z = s2[e] + s3[e], w = s2[e] - s3[e];
                s0[e] = x + z;
                s1[e] = y + w;
                s2[e] = x - z;
                s3[e] = y - w;
            }
            if (shared ? mine(0) : c0 == 0) class_digits4(s0, a.S, a.bias, tile(0));
            if (shared ? mine(1) : c0 == 1) class_digits4(s1, a.S, a.bias, tile(1));
            if (shared ? mine(2) : c0 == 2) class_digits4(s2, a.S, a.bias, tile(2));
            if (shared ? mine(3) : c0 == 3) class_digits4(s3, a.S, a.bias, tile(3));
        }
    }
}

// Exponent bound of every virtual box's multipole: a warp per box. Runs beside M2L, off the main chain.
__global__ void __launch_bounds__(256) box_bound_kernel(int64_t nvb, int P2, const double* __restrict__ Mexp,
                                                        int* __restrict__ bexp) {
    const int64_t vb = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (vb >= nvb) return;
    int m = INT_MIN;
    for (int q = lane; q < P2; q += 32) {
        const double x = Mexp[vb * P2 + q];
        if (x != 0.0) m = max(m, exp_bound(x));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) bexp[vb] = m;
}

// Operand of the leaf far field: as class_operand_kernel, orbit 0 the leaf's own local without coefficient 0
// (a class holds its parts), orbit 1 + o the sums of the W orbit's multipoles, whose parts the
// reflections multiply by +-1.
__global__ void __launch_bounds__(1024) class_far_operand_kernel(const __grid_constant__ ClassOperandArgs a) {
    __shared__ int4 s_src[kTileM];
    __shared__ int s_r[kTileM], s_E[kTileM];
    const int g = a.p0 / 4 + blockIdx.x, o = blockIdx.y;
    const int P2 = a.ct.K[1][0];
    const uint32_t gm = (uint32_t)a.gmask[g];
    if (!((gm >> o) & 1u)) return;
    const int m = threadIdx.x >> 3, c4 = threadIdx.x & 7;
    {
        // a row's eight threads take the bound of its local's parts, the first of them the rest
        const int64_t v = (int64_t)g * kTileM + m;
        const bool in = v < a.nv;
        const int leaf = in ? a.order[v / a.R] : 0, b = a.box_of_leaf[leaf], r = in ? (int)(v % a.R) : 0;
        int E = INT_MIN;
        const double* L = a.Lexp + ((size_t)b * a.R + r) * P2;
        for (int q = 2 + c4; in && q < P2; q += 8)
            if (L[q] != 0.0) E = max(E, exp_bound(L[q]));
        for (int q = 4; q > 0; q >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, q));
        if (c4 == 0) {
            int4 s = make_int4(-1, -1, -1, -1);
            if (in) {
                for (int e = a.wptr[b]; e < a.wptr[b + 1]; ++e) E = max(E, a.bexp[(size_t)a.widx[e] * a.R + r]);
                const uint32_t mk = (a.inst_mask[b] >> sym_first_row(VFMM_LIST_W)) & ((1u << kFarOrb) - 1u);
                const int4* inst = a.inst_src + a.inst_ptr[b];
                int most = 1;
                for (int i = 0; i < __popc(mk); ++i)
                    most = max(most, (inst[i].x >= 0) + (inst[i].y >= 0) + (inst[i].z >= 0) + (inst[i].w >= 0));
                E = E == INT_MIN ? 0 : E - 1 + (most > 2 ? 2 : most - 1);
                if (o == 0) {
                    s = make_int4(b, b, b, b);
                    if (blockIdx.z == 0) a.Et[(size_t)leaf * a.R + r] = E;
                } else if ((mk >> (o - 1)) & 1u) {
                    s = inst[__popc(mk & ((1u << (o - 1)) - 1u))];
                }
            }
            s_src[m] = s;
            s_r[m] = r;
            s_E[m] = in ? E : 0;
        }
    }
    const int nkb = a.ct.nkb[o][0];
    const int before = o == 0 ? 0 : 1 + a.ct.nkb[1][0] * __popc((gm >> 1) & ((1u << (o - 1)) - 1u));
    const long long at0 = class_span(a.spans, a.p0, nullptr);
    __syncthreads();
    const int4 src = s_src[m];
    const int r = s_r[m], E = s_E[m];
    const size_t row = (size_t)m * 64 + ((((c4 >> 1) ^ (m >> 1)) & 3) << 4) + ((c4 & 1) << 3);
    auto tile = [&](int c, int kb) {
        return a.out + (size_t)(class_span(a.spans, 4 * g + c, nullptr) - at0 + before + kb) * a.S * kClsUnit + row;
    };
    auto mine = [&](int c) { return 4 * g + c >= a.p0 && 4 * g + c < a.p1; };
    if (o == 0) {
        if (blockIdx.z != 0) return;
        const double* L = a.Lexp + ((size_t)max(src.x, 0) * a.R + r) * P2;
        for (int c = 0; c < 4; ++c) {
            if (!mine(c)) continue;
            long long q[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int part = sym_part(c, c4 * 4 + e);
                q[e] = src.x >= 0 && part >= 2 && part < P2 ? fixed60(L[part], E) : 0;
            }
            class_digits4(q, a.S, a.bias, tile(c, 0));
        }
        return;
    }
    const double* M0 = a.Mexp + ((size_t)max(src.x, 0) * a.R + r) * P2;
    const double* M1 = a.Mexp + ((size_t)max(src.y, 0) * a.R + r) * P2;
    const double* M2 = a.Mexp + ((size_t)max(src.z, 0) * a.R + r) * P2;
    const double* M3 = a.Mexp + ((size_t)max(src.w, 0) * a.R + r) * P2;
    for (int kb = blockIdx.z; kb < nkb; kb += gridDim.z) {
        const int col0 = kb * kKBlock + c4 * 4;
        long long q0[4], q1[4], q2[4], q3[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int part = col0 + e;
            const bool in = part < P2;
            long long s0 = in && src.x >= 0 ? fixed60(__ldg(M0 + part), E) : 0;
            long long s1 = in && src.y >= 0 ? fixed60(__ldg(M1 + part), E) : 0;
            long long s2 = in && src.z >= 0 ? fixed60(__ldg(M2 + part), E) : 0;
            long long s3 = in && src.w >= 0 ? fixed60(__ldg(M3 + part), E) : 0;
            if (sym_part_sign(part, 1)) s1 = -s1;
            if (sym_part_sign(part, 2)) s2 = -s2;
            if (sym_part_sign(part, 3)) s3 = -s3;
            const long long x = s0 + s1, y = s0 - s1, z = s2 + s3, w = s2 - s3;
            q0[e] = x + z;
            q1[e] = y + w;
            q2[e] = x - z;
            q3[e] = y - w;
        }
        if (mine(0)) class_digits4(q0, a.S, a.bias, tile(0, kb));
        if (mine(1)) class_digits4(q1, a.S, a.bias, tile(1, kb));
        if (mine(2)) class_digits4(q2, a.S, a.bias, tile(2, kb));
        if (mine(3)) class_digits4(q3, a.S, a.bias, tile(3, kb));
    }
}

// ---------------------------------------------------------------- contraction
struct ClassGemmArgs {
    ClassTab ct;
    int S, nst, R, nv, split;
    int p0, n_items;
    const bf16* tab;
    const unsigned char* opnd;
    const int32_t* order;
    const int32_t* gmask;
    ClassSpans spans;
    float2* out;  // [split][leaf * R + r][4 * nch * N]
    int* err;
};

// Item = (piece, share of its K blocks, row tile), the last pieces (the masks with most orbits) first; tiles of a piece next to
// each other, so that they read its operand from L2 together. Warps 0..7 epilogue, 8 producer, 9 MMA.
template <int N>
__global__ void __launch_bounds__(kClsThreads, 1) class_gemm_kernel(const __grid_constant__ ClassGemmArgs a) {
    extern __shared__ unsigned char cls_sm[];
    __shared__ __align__(8) uint64_t bars[2 * kClsMaxStages + 3];
    __shared__ uint32_t tmem_holder;
    __shared__ volatile int abort_flag;
    constexpr int HALF = N / 2;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int S = a.S, nst = a.nst;
    const uint32_t bytesA = S * kClsUnit, bytesB = S * N * 64, stage = bytesA + bytesB;
    const uint32_t sbase = (tc::smem_u32(cls_sm) + 1023u) & ~1023u;
    const uint32_t full0 = tc::smem_u32(&bars[0]), empty0 = tc::smem_u32(&bars[kClsMaxStages]);
    const uint32_t acc_full = tc::smem_u32(&bars[2 * kClsMaxStages]);
    const uint32_t acc_empty = acc_full + 8, mma_done = acc_full + 16;
    if (tid == 0) {
        for (int s = 0; s < nst; ++s) {
            tc::mbar_init(full0 + 8 * s, 1);
            tc::mbar_init(empty0 + 8 * s, 1);
        }
        tc::mbar_init(acc_full, 1);
        tc::mbar_init(acc_empty, kClsEpilogueThreads);
        tc::mbar_init(mma_done, 1);
        abort_flag = 0;
        tc::mbar_fence_init();
    }
    if (warp == kClsEpilogueWarps + 1) {
        tc::tmem_alloc(tc::smem_u32(&tmem_holder), kTmemCols);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_holder, 0);
    struct Item {
        int g, c, nt, sp, u0, U, du;  // K blocks u0 .. u0 + U of the piece; du of them per drain group
        long long at;                 // tiles before its piece
    };
    auto item = [&](int it) {
        Item x;
        const int qq = it / a.ct.nch, q = qq / a.split;
        x.nt = it - qq * a.ct.nch;
        x.sp = qq - q * a.split;
        const int p = a.p0 + a.n_items / (a.ct.nch * a.split) - 1 - q;
        x.g = p >> 2;
        x.c = p & 3;
        int all;
        x.at = class_span(a.spans, p, &all);
        x.u0 = all * x.sp / a.split;
        x.U = all * (x.sp + 1) / a.split - x.u0;
        const int nd = (x.U + kClsDrain - 1) / kClsDrain;
        x.du = nd ? (x.U + nd - 1) / nd : 1;
        return x;
    };
    int issued = 0;  // producer: units whose copies were started

    if (warp == kClsEpilogueWarps) {
        // ------------------------------------------------ producer
        if (lane == 0) {
            int gu = 0;
            bool ok = true;
            const long long at0 = class_span(a.spans, a.p0, nullptr);
            for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
                const Item x = item(it);
                const uint32_t gm = (uint32_t)a.gmask[x.g];
                const unsigned char* A = a.opnd + (size_t)(x.at - at0 + x.u0) * bytesA;
                int before = 0;  // K blocks of the orbits before
                for (int o = 0; o < a.ct.norb && ok; ++o) {
                    if (!((gm >> o) & 1u)) continue;
                    const int nkb = a.ct.nkb[o][x.c];
                    const unsigned char* B = reinterpret_cast<const unsigned char*>(a.tab) +
                                             (size_t)(a.ct.toff[o][x.c] + x.nt * nkb) * (kSlices * N * 64);
                    const int k0 = max(0, x.u0 - before), k1 = min(nkb, x.u0 + x.U - before);
                    before += nkb;
                    B += (size_t)k0 * (kSlices * N * 64);
                    for (int kb = k0; kb < k1; ++kb, ++gu, A += bytesA, B += kSlices * N * 64) {
                        const int s = gu % nst;
                        if (gu >= nst && !tc::mbar_wait(empty0 + 8 * s, (gu / nst - 1) & 1, &abort_flag)) {
                            abort_flag = 1;
                            atomicExch(a.err, 1);
                            ok = false;
                            break;
                        }
                        const uint32_t dst = sbase + s * stage, bar = full0 + 8 * s;
                        tc::mbar_arrive_expect_tx(bar, stage);
                        tc::bulk_copy_g2s(dst, A, bytesA, bar);
                        tc::bulk_copy_g2s(dst + bytesA, B, bytesB, bar);
                        issued = gu + 1;
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == kClsEpilogueWarps + 1) {
        // ------------------------------------------------ MMA issuer (the whole warp in step)
        const uint64_t desc0 = tc::smem_desc(sbase, 16, 512, tc::kLayoutSwizzle64B);
        int gu = 0, dg = 0;
        bool stop = false;
        auto wait = [&](uint32_t bar, uint32_t parity, int code) {
            if (__all_sync(0xffffffffu, tc::mbar_wait(bar, parity, &abort_flag))) return true;
            abort_flag = 1;
            if (lane == 0) atomicExch(a.err, code);
            return false;
        };
        for (int it = blockIdx.x; it < a.n_items && !stop; it += gridDim.x) {
            const Item x = item(it);
            for (int u = 0; u < x.U; ++u, ++gu) {
                const bool first = u % x.du == 0;
                if (first && dg > 0 && !wait(acc_empty, (dg - 1) & 1, 4)) {
                    stop = true;
                    break;
                }
                const int s = gu % nst;
                if (!wait(full0 + 8 * s, (gu / nst) & 1, 2)) {
                    stop = true;
                    break;
                }
                tc::tc_fence_after();
                const uint64_t ad0 = desc0 + ((s * stage) >> 4), bd0 = desc0 + ((s * stage + bytesA) >> 4);
                switch (S) {
                    case 6: first ? issue_unit<true, 6, N>(tmem, ad0, bd0) : issue_unit<false, 6, N>(tmem, ad0, bd0); break;
                    case 7: first ? issue_unit<true, 7, N>(tmem, ad0, bd0) : issue_unit<false, 7, N>(tmem, ad0, bd0); break;
                    default: first ? issue_unit<true, 8, N>(tmem, ad0, bd0) : issue_unit<false, 8, N>(tmem, ad0, bd0); break;
                }
                tc::umma_commit(empty0 + 8 * s);
                if (u % x.du == x.du - 1 || u == x.U - 1) {
                    tc::umma_commit(acc_full);
                    ++dg;
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue: drain each drain group, write each item
        const int quad = warp & 3, half = warp >> 2;
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + half * HALF;
        bool ok = true;
        int dg = 0;
        for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
            const Item x = item(it);
            float hi[HALF], lo[HALF];
#pragma unroll
            for (int j = 0; j < HALF; ++j) hi[j] = lo[j] = 0.0f;
            const int nd = (x.U + x.du - 1) / x.du;
            for (int d = 0; d < nd; ++d, ++dg) {
                ok = ok && tc::mbar_wait(acc_full, dg & 1, &abort_flag);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) {
                    if (lane == 0) atomicExch(a.err, 3);
                    abort_flag = 1;
                    break;
                }
                tc::tc_fence_after();
#pragma unroll
                for (int q = 0; q < HALF / 8; ++q) {
                    uint32_t r[kNumAcc][8];
#pragma unroll
                    for (int acc = 0; acc < kNumAcc; ++acc) tc::tmem_ld8_nowait(lane_base + acc * N + q * 8, r[acc]);
                    tc::tmem_wait_ld();
#pragma unroll
                    for (int acc = 0; acc < kNumAcc; ++acc)
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            float s2, e2;
                            two_sum(hi[q * 8 + j], __uint_as_float(r[acc][j]), s2, e2);
                            hi[q * 8 + j] = s2;
                            lo[q * 8 + j] = __fadd_rn(lo[q * 8 + j], e2);
                        }
                }
                tc::tc_fence_before();
                tc::mbar_arrive(acc_empty);
            }
            if (!ok) break;
            const int64_t v = (int64_t)x.g * kTileM + quad * 32 + lane;
            if (v < a.nv) {
                const size_t row = (size_t)a.order[v / a.R] * a.R + v % a.R;
                float4* o = reinterpret_cast<float4*>(a.out + ((size_t)x.sp * a.nv + row) * (4 * a.ct.nch * N) + (x.c * a.ct.nch + x.nt) * N +
                                                      half * HALF);
#pragma unroll
                for (int j = 0; j < HALF / 2; ++j) {
                    const float2 p = df_final(hi[2 * j], lo[2 * j]), q = df_final(hi[2 * j + 1], lo[2 * j + 1]);
                    o[j] = make_float4(p.x, p.y, q.x, q.y);
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (abort_flag) {
        // after an abort: wait, with a longer bound, for the copies and MMAs still in flight before the
        // shared memory and TMEM they use are released
        const volatile int never = 0;
        if (tid == kClsEpilogueThreads)
            for (int u = max(0, issued - nst); u < issued; ++u)
                tc::mbar_wait(full0 + 8 * (u % nst), (u / nst) & 1, &never, 1ll << 27);
        if (warp == kClsEpilogueWarps + 1) {
            tc::umma_commit(mma_done);
            tc::mbar_wait(mma_done, 0, &never, 1ll << 27);
            __syncwarp();
        }
        __syncthreads();
    }
    if (warp == kClsEpilogueWarps + 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, kTmemCols);
    }
}

template <int N>
static int launch_classes(const ClassGemmArgs& a, int grid, cudaStream_t st) {
    static thread_local int attr_dev = -1;
    int dev = 0;
    VFMM_CUDA(cudaGetDevice(&dev));
    if (attr_dev != dev) {
        VFMM_CUDA(cudaFuncSetAttribute(class_gemm_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClsSmem));
        attr_dev = dev;
    }
    const size_t smem = (size_t)a.nst * a.S * (kClsUnit + N * 64) + 1024;
    class_gemm_kernel<N><<<(unsigned)grid, kClsThreads, smem, st>>>(a);
    VFMM_CUDA(cudaGetLastError());
    return VFMM_OK;
}

// Makes the operand of a chunk (operand(p0, p1, grid)) and contracts it, chunk after chunk.
template <class Operand>
static int class_contract(const DeviceTree& T, const ClassTab& ct, const void* tab, const ClassPlan& P, int S, int R,
                          int split, void* opnd, size_t opnd_bytes, float2* out, int* err, cudaStream_t st,
                          Operand&& operand) {
    int dev = 0, sms = 0;
    VFMM_CUDA(cudaGetDevice(&dev));
    VFMM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    ClassGemmArgs ga;
    ga.ct = ct;
    ga.S = S;
    ga.nst = (int)std::min<size_t>(kClsMaxStages, (kClsSmem - 1024) / ((size_t)S * (kClsUnit + ct.N * 64)));
    ga.R = R;
    ga.split = split;
    ga.nv = T.n_leaves * R;
    ga.tab = (const bf16*)tab;
    ga.opnd = (const unsigned char*)opnd;
    ga.order = P.order;
    ga.gmask = P.gmask;
    ga.spans = device_spans(ct, P);
    ga.out = out;
    ga.err = err;
    return class_chunks(ct, P, S, opnd_bytes, [&](int p0, int p1) -> int {
        // K blocks of an orbit spread over CTAs while there are few groups
        const int groups = (p1 - 1) / 4 - p0 / 4 + 1, zs = std::max(1, std::min(8, 4 * sms / (groups * ct.norb)));
        operand(p0, p1, dim3((unsigned)groups, ct.norb, zs));
        VFMM_CUDA(cudaGetLastError());
        ga.p0 = p0;
        ga.n_items = (p1 - p0) * split * ct.nch;
        // persistent CTAs, one per SM unless capped: an item's first loads overlap the drain and the output
        // of the one before (a CTA per item: 0.32 ms, persistent 0.27 on 16,384 uniform leaves)
        const int grid = std::min(P.ctas > 0 ? P.ctas : sms, ga.n_items);
        switch (ct.N) {
            case 48: return launch_classes<48>(ga, grid, st);
            case 64: return launch_classes<64>(ga, grid, st);
            default: return launch_classes<80>(ga, grid, st);
        }
    });
}

static ClassOperandArgs operand_args(const DeviceTree& T, const ClassTab& ct, const ClassPlan& P, int S, int R, int list,
                                     void* opnd) {
    ClassOperandArgs oa = {};
    oa.ct = ct;
    oa.S = S;
    oa.bias = class_bias(S);
    oa.R = R;
    oa.nleaf = T.n_leaves;
    oa.nv = T.n_leaves * R;
    oa.order = P.order;
    oa.gmask = P.gmask;
    oa.spans = device_spans(ct, P);
    oa.box_of_leaf = T.box_of_leaf;
    oa.inst_ptr = T.inst_ptr[list];
    oa.inst_src = T.inst_src[list];
    oa.inst_mask = T.inst_mask;
    oa.out = (unsigned char*)opnd;
    return oa;
}

int near_class_contract(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, const MixedWork& w,
                        cudaStream_t st) {
    const MixedOps* mo = (const MixedOps*)o.mixed;
    if (w.cev) VFMM_CUDA(cudaEventRecord(w.cev[0], st));
    const int S = mo->slices[kCtrNear];
    const int64_t nv = (int64_t)T.n_leaves * o.k * o.k;
    class_fixed_kernel<<<dim3((unsigned)std::min<int64_t>((nv + 255) / 256, 8192), PS.R), 256, 0, st>>>(f, nv, w.Ef, w.ffix);
    VFMM_CUDA(cudaGetLastError());
    ClassOperandArgs oa = operand_args(T, mo->near, PS.near, S, PS.R, VFMM_LIST_U, w.near_opnd);
    oa.f = w.ffix;
    VFMM_CHECK(class_contract(T, mo->near, mo->near_tab, PS.near, S, PS.R, w.near_split, w.near_opnd, w.near_opnd_bytes, w.out, w.err, st,
                              [&](int p0, int p1, dim3 grid) {
                                  oa.p0 = p0;
                                  oa.p1 = p1;
                                  class_operand_kernel<<<grid, 1024, 0, st>>>(oa);
                              }));
    if (w.cev) VFMM_CUDA(cudaEventRecord(w.cev[1], st));
    return VFMM_OK;
}

int leaf_class_bounds(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* Mexp, const MixedWork& w,
                      cudaStream_t st) {
    const int64_t nvb = (int64_t)T.n_boxes * PS.R;
    box_bound_kernel<<<(unsigned)((nvb + 7) / 8), 256, 0, st>>>(nvb, 2 * (o.p + 1), Mexp, w.bexp);
    VFMM_CUDA(cudaGetLastError());
    return VFMM_OK;
}

int leaf_class_contract(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* Mexp, const double* Lexp,
                        const MixedWork& w, cudaStream_t st) {
    const MixedOps* mo = (const MixedOps*)o.mixed;
    if (w.cev) VFMM_CUDA(cudaEventRecord(w.cev[8], st));
    const int S = leaf_class_slices(*mo);
    ClassOperandArgs oa = operand_args(T, mo->leaf, PS.leaf, S, PS.R, VFMM_LIST_W, w.aprep);
    oa.Mexp = Mexp;
    oa.Lexp = Lexp;
    oa.bexp = w.bexp;
    oa.wptr = T.lptr[VFMM_LIST_W];
    oa.widx = T.lidx[VFMM_LIST_W];
    oa.Et = w.Et;
    VFMM_CHECK(class_contract(T, mo->leaf, mo->leaf_tab, PS.leaf, S, PS.R, w.leaf_split, w.aprep, w.aprep_bytes, w.far_out, w.err, st,
                              [&](int p0, int p1, dim3 grid) {
                                  oa.p0 = p0;
                                  oa.p1 = p1;
                                  class_far_operand_kernel<<<grid, 1024, 0, st>>>(oa);
                              }));
    if (w.cev) VFMM_CUDA(cudaEventRecord(w.cev[9], st));
    return VFMM_OK;
}

}  // namespace vfmm
