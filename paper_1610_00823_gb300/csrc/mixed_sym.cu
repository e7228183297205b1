// Split-BF16 near field in the reflection classes of sym.cuh (VFMM_MIXED).
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
//    large as 256, which BF16 holds, at the price of draining every 448 K values instead of 512
//    (36,864 units per K value on diagonal 4, 448 of them below 2^24).
//  * the outputs of a class are put together at the nodes by the leaf kernel (double-FP32).
// Operand tiles are made and consumed in chunks that fit the workspace's buffer.
//
// What bounds it: a K block of 128 x 64 outputs moves 207 KB through shared memory (72 KB written, the A
// tiles once, the B tiles once per product), 1,620 cycles; the MMAs take 1,700 of the 2,220 cycles measured,
// 300 go to operands not yet there and 220 to drains. The operand is bound by HBM writes and integer work.
// Against gathered rows and plain tables (ms): 200,104 graded leaves 13.3 -> 8.0, 16,384 uniform leaves
// k = 16 1.32 -> 0.39, 1,378 graded leaves 0.18 -> 0.11, 4,096 rows of k = 8 0.081 -> 0.034.
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
// E[field * h^2 + quadrant node] = exponent of the largest entry of that row over orbits and classes.
__global__ void class_row_exp_kernel(SymOp op, int* __restrict__ E) {
    __shared__ double red[256];
    const int k = op.k, hx = (k + 1) / 2, q = blockIdx.x / (hx * hx), e = blockIdx.x - q * hx * hx;
    const int j = e / hx, i = e - j * hx;
    double m = 0.0;
    for (int o = 0; o < op.norb; ++o)
        for (int c = 0; c < 4; ++c) {
            const int nx = sym_half(k, sym_pa(c, q));
            if (i >= nx || j >= sym_half(k, sym_pb(c, q))) continue;
            const int row = op.seg[3 * c + q] - op.roff[c] + j * nx + i;
            const double* A = op.A + op.off[o][c] + row;
            for (int col = threadIdx.x; col < op.K[o][c]; col += blockDim.x)
                m = fmax(m, fabs(A[(size_t)col * op.M[c]]));
        }
    red[threadIdx.x] = m;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
        __syncthreads();
    }
    if (threadIdx.x == 0) E[blockIdx.x] = red[0] > 0.0 ? exp_bound(red[0]) : 0;
}

// Digits of every table, tile by tile (table_at with one orbit's class as a table of nch * N rows).
__global__ void class_table_kernel(SymOp op, ClassTab ct, const int* __restrict__ E, bf16* __restrict__ out) {
    const int o = blockIdx.y >> 2, c = blockIdx.y & 3, r = blockIdx.x;  // padded row of the class
    const int k = op.k, hx = (k + 1) / 2, K = op.K[o][c], Kp = ct.nkb[o][c] * kKBlock;
    int e = 0, row = r;
    if (r < op.M[c]) {
        int q = 0;
        row += op.roff[c];
        while (row >= op.seg[3 * c + q + 1]) ++q;
        const int nx = sym_half(k, sym_pa(c, q)), rr = row - op.seg[3 * c + q];
        e = E[q * hx * hx + (rr / nx) * hx + rr % nx];
    }
    bf16* base = out + (size_t)ct.toff[o][c] * kSlices * ct.N * kKBlock;
    for (int col = threadIdx.x; col < Kp; col += blockDim.x) {
        const double v = r < op.M[c] && col < K ? op.A[op.off[o][c] + (size_t)col * op.M[c] + r] : 0.0;
        slice_fixed(v, e, base + table_at(0, ct.nch * ct.N, ct.N, Kp, r, col), ct.N * kKBlock);
    }
}

int near_classes_prepare(vfmm_ops* o, cudaStream_t st) {
    MixedOps* mo = (MixedOps*)o->mixed;
    const int k = o->k;
    SymOp op;
    int rc = sym_near_op(o, &op, st);
    ClassTab& ct = mo->near;
    // rows per tile: the fewest cycles per K block (measured per MMA, with 16 for the tile's loads)
    int mmax = 0;
    for (int c = 0; c < 4; ++c) mmax = std::max(mmax, op.M[c]);
    const int width[3] = {48, 64, 80};
    const double cycles[3] = {29.5 + 16, 35.6 + 16, 41.6 + 16};
    double best = 1e300;
    for (int i = 0; i < 3; ++i) {
        const int n = (mmax + width[i] - 1) / width[i];
        if (n * cycles[i] < best) {
            best = n * cycles[i];
            ct.N = width[i];
            ct.nch = n;
        }
    }
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
    const int hx = (k + 1) / 2;
    auto work = [&]() -> int {
        VFMM_CHECK(rc);
        VFMM_CUDA(cudaMalloc(&mo->near_E, 3 * hx * hx * sizeof(int)));
        VFMM_CUDA(cudaMalloc(&mo->near_tab, (size_t)tiles * kSlices * ct.N * kKBlock * sizeof(bf16)));
        class_row_exp_kernel<<<3 * hx * hx, 256, 0, st>>>(op, mo->near_E);
        class_table_kernel<<<dim3(ct.nch * ct.N, 4 * op.norb), 128, 0, st>>>(op, ct, mo->near_E, (bf16*)mo->near_tab);
        VFMM_CUDA(cudaGetLastError());
        VFMM_CUDA(cudaStreamSynchronize(st));
        return VFMM_OK;
    };
    rc = work();
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

int build_near_classes(const DeviceTree& T, int R, const HostLists& H, PlanArena& A, NearPlan* P) {
    const std::vector<int32_t>&ptr = H.ptr[VFMM_LIST_U], &cfg = H.cfg[VFMM_LIST_U];
    uint16_t bit[kNearCfg];
    for (int c = 0; c < kNearCfg; ++c) {
        int slots;
        bit[c] = (uint16_t)(1u << sym_orbit(VFMM_LIST_U, c, &slots));
    }
    const int nl = T.n_leaves;
    if ((int64_t)nl * R > (int64_t)INT32_MAX / 2) return fail(VFMM_ERR_INVALID_ARG, "too many rows for one split contraction");
    std::vector<uint16_t> mask(nl);
    std::vector<int32_t> start((1 << kNearOrb) + 1, 0), order(nl);
    for (int t = 0; t < nl; ++t) {
        const int b = H.bol[t];
        uint16_t m = 0;
        for (int e = ptr[b]; e < ptr[b + 1]; ++e) m |= bit[cfg[e]];
        mask[t] = m;
        ++start[m + 1];
    }
    for (int m = 0; m < (1 << kNearOrb); ++m) start[m + 1] += start[m];
    for (int t = 0; t < nl; ++t) order[start[mask[t]]++] = t;
    const int64_t nv = (int64_t)nl * R;
    P->n_groups = (int32_t)((nv + kTileM - 1) / kTileM);
    std::vector<int32_t> gmask(P->n_groups, 0), first(4 * (size_t)P->n_groups + 1, 0);
    int64_t units = 0;
    for (int g = 0; g < P->n_groups; ++g) {
        const int64_t t0 = (int64_t)g * kTileM / R, t1 = (std::min<int64_t>((int64_t)(g + 1) * kTileM, nv) - 1) / R;
        for (int64_t t = t0; t <= t1; ++t) gmask[g] |= mask[order[t]];
        for (int c = 0; c < 4; ++c) {
            const int u = class_units(T.k, (uint32_t)gmask[g], c);
            P->max_units = std::max(P->max_units, u);
            units += u;
            if (units > INT32_MAX) return fail(VFMM_ERR_INVALID_ARG, "too many operand tiles");
            first[4 * (size_t)g + c + 1] = (int32_t)units;
        }
    }
    P->first = first;
    P->off[0] = A.put(order);
    P->off[1] = A.put(gmask);
    P->off[2] = A.put(first);
    return VFMM_OK;
}

// Bytes of the operand buffer: all tiles at once, up to 16 rows of outputs per leaf (what the near field
// by entries kept for its partial sums), at least 8 MB and at most 768 MB; more tiles take turns in it.
size_t near_operand_bytes(const DeviceTree& T, const NearPlan& P, int R) {
    if (P.n_groups == 0) return 0;
    const size_t all = (size_t)P.first.back() * kSlices * kClsUnit;
    const size_t rows = (size_t)T.n_leaves * R * 16 * 3 * T.k * T.k * sizeof(float2);
    const size_t cap = std::min(std::max(rows, size_t(8) << 20), size_t(768) << 20);
    return std::max(std::min(all, cap), (size_t)P.max_units * kSlices * kClsUnit);
}

// ---------------------------------------------------------------- operand
struct ClassOperandArgs {
    ClassTab ct;
    int S, R, nleaf, nv;
    int p0, p1;          // pieces (4 * group + class) of this chunk
    const int32_t* order;
    const int32_t* gmask;
    const int32_t* first;
    const int32_t* box_of_leaf;
    const int32_t* inst_ptr;
    const int4* inst_src;
    const uint32_t* inst_mask;
    const long long* f;  // fixed-point leaf values (class_fixed_kernel)
    unsigned char* out;  // chunk's tiles: unit u of piece p at (first[p] - first[p0] + u) * S * kClsUnit
};

// floor(|v| 2^(56 - E)) with v's sign (|v| < 2^E), integer work.
__device__ __forceinline__ long long fixed56(double v, int E) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    int ev = (int)((bits >> 52) & 0x7FF);
    unsigned long long mant = bits & ((1ull << 52) - 1);
    if (ev) mant |= 1ull << 52;
    else ev = 1;
    const int shift = 1019 - ev + E;
    const long long q = (long long)(shift >= 64 ? 0ull : (shift >= 0 ? mant >> shift : mant << (-shift)));
    return (bits >> 63) ? -q : q;
}

// q[r][i] = f[r][i] 2^(55 - E_f[r]), truncated: the fixed-point values that the operand sums.
__global__ void __launch_bounds__(256) class_fixed_kernel(const double* __restrict__ f, int64_t n,
                                                          const int* __restrict__ Ef, long long* __restrict__ q) {
    const int E = Ef[blockIdx.y] + 1;
    const size_t base = (size_t)blockIdx.y * n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        q[base + i] = fixed56(f[base + i], E);
}

// Balanced base-128 digits of 4 values q 2^-56 (|q| < 2^57): d_i = digit 8 - i of q + 64 (128^6 + ... + 1),
// less 64, the top one the rest; S 8-byte stores, slice i at out + i * kClsUnit.
__device__ __forceinline__ void class_digits4(const long long* q, int S, unsigned char* out) {
    constexpr long long kBias = 64ll * (((1ll << 49) - 1) / 127);
    constexpr float kMagic = 12582912.0f;  // 1.5 2^23: an integer below 2^22 added to its bits is added to it
    long long b[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) b[e] = q[e] + kBias;
#pragma unroll
    for (int i = 0; i < kSlices; ++i) {
        if (i >= S) break;
        const int shift = 7 * (kSlices - 1 - i);
        const float sc = __int_as_float((127 - 7 * (i + 1)) << 23);
        const float zero = (i == 0 ? kMagic : kMagic + 64.0f) * sc;
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int d = (int)(b[e] >> shift);
            v[e] = fmaf(__int_as_float(0x4B400000 + (i == 0 ? d : d & 127)), sc, -zero);
        }
        const __nv_bfloat162 h0 = __floats2bfloat162_rn(v[0], v[1]), h1 = __floats2bfloat162_rn(v[2], v[3]);
        *reinterpret_cast<uint2*>(out + (size_t)i * kClsUnit) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
    }
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
    for (int kb = blockIdx.z; kb < nkb; kb += gridDim.z) {
        const int col0 = kb * kKBlock + c4 * 4;
        auto tile = [&](int c) {
            return a.out + (size_t)(a.first[4 * g + c] - a.first[a.p0] + before[c] + kb) * a.S * kClsUnit + row;
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
            if (shared ? mine(0) : c0 == 0) class_digits4(s0, a.S, tile(0));
            if (shared ? mine(1) : c0 == 1) class_digits4(s1, a.S, tile(1));
            if (shared ? mine(2) : c0 == 2) class_digits4(s2, a.S, tile(2));
            if (shared ? mine(3) : c0 == 3) class_digits4(s3, a.S, tile(3));
        }
    }
}

// ---------------------------------------------------------------- contraction
struct ClassGemmArgs {
    ClassTab ct;
    int S, nst, R, nv;
    int p0, n_items;
    const bf16* tab;
    const unsigned char* opnd;
    const int32_t* order;
    const int32_t* gmask;
    const int32_t* first;
    float2* out;  // [leaf * R + r][4 * nch * N]
    int* err;
};

// Item = (piece, row tile), the last pieces (the masks with most orbits) first; tiles of a piece next to
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
        int g, c, nt, U, du;  // du: K blocks per drain group
    };
    auto item = [&](int it) {
        Item x;
        const int q = it / a.ct.nch;
        x.nt = it - q * a.ct.nch;
        const int p = a.p0 + a.n_items / a.ct.nch - 1 - q;
        x.g = p >> 2;
        x.c = p & 3;
        x.U = a.first[p + 1] - a.first[p];
        const int nd = (x.U + kClsDrain - 1) / kClsDrain;
        x.du = (x.U + nd - 1) / nd;
        return x;
    };
    int issued = 0;  // producer: units whose copies were started

    if (warp == kClsEpilogueWarps) {
        // ------------------------------------------------ producer
        if (lane == 0) {
            int gu = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < a.n_items && ok; it += gridDim.x) {
                const Item x = item(it);
                const uint32_t gm = (uint32_t)a.gmask[x.g];
                const unsigned char* A = a.opnd + (size_t)(a.first[4 * x.g + x.c] - a.first[a.p0]) * bytesA;
                for (int o = 0; o < a.ct.norb && ok; ++o) {
                    if (!((gm >> o) & 1u)) continue;
                    const int nkb = a.ct.nkb[o][x.c];
                    const unsigned char* B = reinterpret_cast<const unsigned char*>(a.tab) +
                                             (size_t)(a.ct.toff[o][x.c] + x.nt * nkb) * (kSlices * N * 64);
                    for (int kb = 0; kb < nkb; ++kb, ++gu, A += bytesA, B += kSlices * N * 64) {
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
                float4* o = reinterpret_cast<float4*>(a.out + row * (4 * a.ct.nch * N) + (x.c * a.ct.nch + x.nt) * N +
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

int near_class_contract(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, const MixedWork& w,
                        cudaStream_t st) {
    const MixedOps* mo = (const MixedOps*)o.mixed;
    const NearPlan& P = PS.near;
    if (w.cev) VFMM_CUDA(cudaEventRecord(w.cev[0], st));
    const int S = mo->slices[kCtrNear], pieces = 4 * P.n_groups;
    const int64_t room = (int64_t)(w.near_opnd_bytes / (S * kClsUnit));  // tiles
    const int64_t nv = (int64_t)T.n_leaves * o.k * o.k;
    class_fixed_kernel<<<dim3((unsigned)std::min<int64_t>((nv + 255) / 256, 8192), PS.R), 256, 0, st>>>(f, nv, w.Ef, w.ffix);
    VFMM_CUDA(cudaGetLastError());
    ClassOperandArgs oa;
    oa.ct = mo->near;
    oa.S = S;
    oa.R = PS.R;
    oa.nleaf = T.n_leaves;
    oa.nv = T.n_leaves * PS.R;
    oa.order = P.order;
    oa.gmask = P.gmask;
    oa.first = P.first_dev;
    oa.box_of_leaf = T.box_of_leaf;
    oa.inst_ptr = T.inst_ptr[VFMM_LIST_U];
    oa.inst_src = T.inst_src[VFMM_LIST_U];
    oa.inst_mask = T.inst_mask;
    oa.f = w.ffix;
    oa.out = (unsigned char*)w.near_opnd;
    ClassGemmArgs ga;
    ga.ct = mo->near;
    ga.S = S;
    const size_t stage = (size_t)S * (kClsUnit + mo->near.N * 64);
    ga.nst = (int)std::min<size_t>(kClsMaxStages, (kClsSmem - 1024) / stage);
    ga.R = PS.R;
    ga.nv = oa.nv;
    ga.tab = (const bf16*)mo->near_tab;
    ga.opnd = oa.out;
    ga.order = P.order;
    ga.gmask = P.gmask;
    ga.first = P.first_dev;
    ga.out = w.out;
    ga.err = w.err;
    int dev = 0, sms = 0;
    VFMM_CUDA(cudaGetDevice(&dev));
    VFMM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    for (int p0 = 0; p0 < pieces;) {
        int p1 = p0 + 1;
        while (p1 < pieces && P.first[p1 + 1] - P.first[p0] <= room) ++p1;
        if (P.first[p1] - P.first[p0] > room) return fail(VFMM_ERR_INTERNAL, "near-field operand buffer too small");
        oa.p0 = p0;
        oa.p1 = p1;
        // K blocks of an orbit spread over CTAs while there are few groups
        const int groups = (p1 - 1) / 4 - p0 / 4 + 1, zs = std::max(1, std::min(8, 4 * sms / (groups * mo->near.norb)));
        class_operand_kernel<<<dim3((unsigned)groups, mo->near.norb, zs), 1024, 0, st>>>(oa);
        VFMM_CUDA(cudaGetLastError());
        ga.p0 = p0;
        ga.n_items = (p1 - p0) * mo->near.nch;
        // persistent CTAs, one per SM unless capped: an item's first loads overlap the drain and the output
        // of the one before (a CTA per item: 0.32 ms, persistent 0.27 on 16,384 uniform leaves)
        const int grid = std::min(P.ctas > 0 ? P.ctas : sms, ga.n_items);
        switch (mo->near.N) {
            case 48: VFMM_CHECK(launch_classes<48>(ga, grid, st)); break;
            case 64: VFMM_CHECK(launch_classes<64>(ga, grid, st)); break;
            default: VFMM_CHECK(launch_classes<80>(ga, grid, st)); break;
        }
        p0 = p1;
    }
    if (w.cev) VFMM_CUDA(cudaEventRecord(w.cev[1], st));
    return VFMM_OK;
}

// Kernels that near_class_contract launches.
int near_launches(const MixedOps& mo, const NearPlan& P, size_t opnd_bytes) {
    const int pieces = 4 * P.n_groups;
    const int64_t room = (int64_t)(opnd_bytes / (mo.slices[kCtrNear] * kClsUnit));
    int n = 1;
    for (int p0 = 0; p0 < pieces; n += 2) {
        int p1 = p0 + 1;
        while (p1 < pieces && P.first[p1 + 1] - P.first[p0] <= room) ++p1;
        p0 = p1;
    }
    return n;
}

}  // namespace vfmm
