// The FP64 form's table products in the reflection classes of sym.cuh: tables, instances, contraction.
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "sym.cuh"
#include "vfmm_internal.cuh"

namespace vfmm {

// ---------------------------------------------------------------- tables
struct RepCfg {
    int cfg[kSymMaxOrb];
};

// A[orbit][class][column][row] from the plain table T[cfg][trows][tcols]: for t in the quadrant
// 1/4 sum over the reflections that move R of chi c T_R(s t, y), plus the images of y under those
// that do not. One thread per entry.
__global__ void sym_table_kernel(SymOp op, RepCfg rep, const double* __restrict__ T, int trows, int tcols) {
    const int o = blockIdx.y >> 2, c = blockIdx.y & 3;
    const int M = op.M[c], K = op.K[o][c], k = op.k, kk = k * k;
    const int a = c & 1, b = c >> 1, fx = op.fx[o], fy = op.fy[o];
    const double* Tc = T + (size_t)rep.cfg[o] * trows * tcols;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < M * K; e += gridDim.x * blockDim.x) {
        const int col = e / M, r = e - col * M;
        int q = 0, ti = 0, tj = 0;
        if (op.node_rows) {
            while (r + op.roff[c] >= op.seg[3 * c + q + 1]) ++q;
            const int nx = sym_half(k, sym_pa(c, q)), rr = r + op.roff[c] - op.seg[3 * c + q];
            tj = rr / nx;
            ti = rr - tj * nx;
        }
        double v = 0.0;
        for (int s = 0; s < 4; ++s) {
            if (((s & 1) && fx) || ((s & 2) && fy)) continue;
            int row = sym_part(c, r);
            double sg = 1.0;
            if (op.node_rows) {
                row = q * kk + ((s & 2) ? k - 1 - tj : tj) * k + ((s & 1) ? k - 1 - ti : ti);
                if (((s & 1) & sym_pa(c, q)) ^ ((s >> 1) & sym_pb(c, q))) sg = -1.0;
            }
            const double* Tr = Tc + (size_t)row * tcols;
            if (!op.node_cols) {
                const int part = fx && fy ? sym_part(c, col) : (fx ? 2 * col + ((col & 1) ^ a) : (fy ? 2 * col + b : col));
                v += sg * Tr[part];
                continue;
            }
            const int nx = fx ? sym_half(k, a) : k;
            const int j = col / nx, i = col - j * nx;
            const bool ix = fx && k - 1 - i != i, iy = fy && k - 1 - j != j;  // distinct images
            double w = Tr[j * k + i];
            const double sa = a ? -1.0 : 1.0, sb = b ? -1.0 : 1.0;
            if (ix) w += sa * Tr[j * k + k - 1 - i];
            if (iy) w += sb * Tr[(k - 1 - j) * k + i];
            if (ix && iy) w += sa * sb * Tr[(k - 1 - j) * k + k - 1 - i];
            v += sg * w;
        }
        op.A[op.off[o][c] + e] = 0.25 * v;
    }
}

// Shape of an operator over list q's orbits (q < 0: the leaf itself; kLeafFar: the leaf itself, then the W
// list's) and its table.
constexpr int kLeafFar = 4;
static int make_op(SymOp* op, int q, int k, int P, bool node_rows, bool node_cols, const double* T, int trows, int tcols,
                   cudaStream_t st) {
    op->norb = q < 0 ? 1 : (q == kLeafFar ? 1 + kFarOrb : sym_orbits(q));
    op->k = k;
    op->P = P;
    op->node_rows = node_rows;
    op->node_cols = node_cols;
    RepCfg rep = {};
    if (q < 0) {
        op->fx[0] = op->fy[0] = 1;
    } else if (q == kLeafFar) {
        op->fx[0] = op->fy[0] = 1;
        for (int cfg = 0; cfg < kFarCfg; ++cfg) {
            int slots;
            const int o = sym_orbit(VFMM_LIST_W, cfg, &slots);
            if (slots & 1) rep.cfg[1 + o] = 1 + cfg;
        }
    } else {
        const int ncfg = q == VFMM_LIST_U ? kNearCfg : (q == VFMM_LIST_V ? kVCfg : kFarCfg);
        for (int cfg = 0; cfg < ncfg; ++cfg) {
            int slots, dx, dy;
            const int o = sym_orbit(q, cfg, &slots);
            if (!(slots & 1)) continue;  // the representative holds slot 0
            sym_offset(q, cfg, &dx, &dy);
            rep.cfg[o] = cfg;
            op->fx[o] = dx == 0;
            op->fy[o] = dy == 0;
        }
    }
    int row = 0;
    for (int c = 0; c < 4; ++c) {
        op->roff[c] = node_rows ? row : 0;
        if (node_rows) {
            for (int f = 0; f < 3; ++f) {
                op->seg[3 * c + f] = row;
                row += sym_half(k, sym_pa(c, f)) * sym_half(k, sym_pb(c, f));
            }
            op->M[c] = row - op->roff[c];
        } else {
            op->M[c] = sym_parts(c, P);
        }
    }
    op->seg[12] = row;
    int64_t total = 0;
    for (int o = 0; o < op->norb; ++o)
        for (int c = 0; c < 4; ++c) {
            const int fx = op->fx[o], fy = op->fy[o];
            if (node_cols) op->K[o][c] = (fx ? sym_half(k, c & 1) : k) * (fy ? sym_half(k, c >> 1) : k);
            else op->K[o][c] = fx && fy ? sym_parts(c, P) : (fx || fy ? P : 2 * P);
            op->off[o][c] = total;
            total += (int64_t)op->K[o][c] * op->M[c];
        }
    VFMM_CUDA(cudaMalloc(&op->A, std::max<int64_t>(1, total) * sizeof(double)));
    sym_table_kernel<<<dim3(32, 4 * op->norb), 256, 0, st>>>(*op, rep, T, trows, tcols);
    VFMM_CUDA(cudaGetLastError());
    return VFMM_OK;
}

// M2T of the five representatives, rows as l2t's (u, h u_x, h u_y), columns the source box's parts; the
// a_0 log h_w term is added by the leaf kernel. The column of Im a_0 (always zero) is left out.
static void m2t_tables(int k, int P, std::vector<double>& F) {
    typedef std::complex<double> cd;
    const int kk = k * k, P2 = 2 * P;
    const double pi = 3.14159265358979323846, c = 1.0 / (2.0 * pi);
    F.assign((size_t)kFarCfg * 3 * kk * P2, 0.0);
    for (int cfg = 0; cfg < kFarCfg; ++cfg) {
        int px, py;
        far_pattern(cfg, &px, &py);
        if (px < 0 || py < 0) continue;
        double* Fc = F.data() + (size_t)cfg * 3 * kk * P2;
        for (int t = 0; t < kk; ++t) {
            const double x = -std::cos(pi * (2.0 * (t % k) + 1.0) / (2.0 * k)) / 2.0;
            const double y = -std::cos(pi * (2.0 * (t / k) + 1.0) / (2.0 * k)) / 2.0;
            const cd zeta(2.0 * (x - px / 4.0), 2.0 * (y - py / 4.0)), zi = 1.0 / zeta;
            cd zp = 1.0;  // zeta^-n
            for (int n = 0; n < P; ++n) {
                const cd v = n == 0 ? cd(std::log(std::abs(zeta))) : zp;
                const cd d = 2.0 * (n == 0 ? zi : -(double)n * zp * zi);  // h times the derivative, h / h_w = 2
                Fc[(size_t)t * P2 + 2 * n] = -c * v.real();
                Fc[(size_t)(kk + t) * P2 + 2 * n] = -c * d.real();
                Fc[(size_t)(2 * kk + t) * P2 + 2 * n] = c * d.imag();
                if (n > 0) {
                    Fc[(size_t)t * P2 + 2 * n + 1] = c * v.imag();
                    Fc[(size_t)(kk + t) * P2 + 2 * n + 1] = c * d.imag();
                    Fc[(size_t)(2 * kk + t) * P2 + 2 * n + 1] = c * d.real();
                }
                zp *= zi;
            }
        }
    }
}

int sym_near_op(const vfmm_ops* o, SymOp* op, cudaStream_t st) {
    return make_op(op, VFMM_LIST_U, o->k, o->p + 1, true, true, o->near, 3 * o->k * o->k, o->k * o->k, st);
}

int sym_far_op(const vfmm_ops* o, const double* F, SymOp* op, cudaStream_t st) {
    return make_op(op, kLeafFar, o->k, o->p + 1, true, false, F, 3 * o->k * o->k, 2 * (o->p + 1), st);
}

int sym_prepare(vfmm_ops* o, const double* m2l, const double* s2l, cudaStream_t st) {
    const int k = o->k, kk = k * k, P = o->p + 1, P2 = 2 * P;
    SymTables* s = new SymTables();
    o->sym = s;
    VFMM_CHECK(sym_near_op(o, &s->near, st));
    VFMM_CHECK(make_op(&s->s2m, -1, k, P, false, true, o->s2m, P2, kk, st));
    VFMM_CHECK(make_op(&s->l2t, -1, k, P, true, false, o->l2t, 3 * kk, P2, st));
    VFMM_CHECK(make_op(&s->m2l, VFMM_LIST_V, k, P, false, false, m2l, P2, P2, st));
    VFMM_CHECK(make_op(&s->s2l, VFMM_LIST_X, k, P, false, true, s2l, P2, kk, st));
    std::vector<double> F;
    m2t_tables(k, P, F);
    double* dF = nullptr;
    VFMM_CUDA(cudaMalloc(&dF, F.size() * sizeof(double)));
    cudaError_t e = cudaMemcpyAsync(dF, F.data(), F.size() * sizeof(double), cudaMemcpyHostToDevice, st);
    int rc = e == cudaSuccess ? make_op(&s->m2t, VFMM_LIST_W, k, P, true, false, dF, 3 * kk, P2, st)
                              : cuda_fail(e, "cudaMemcpyAsync");
    cudaStreamSynchronize(st);
    cudaFree(dF);
    return rc;
}

void sym_free(vfmm_ops* o) {
    SymTables* s = (SymTables*)o->sym;
    if (!s) return;
    for (SymOp* op : {&s->near, &s->s2m, &s->m2l, &s->s2l, &s->l2t, &s->m2t})
        if (op->A) cudaFree(op->A);
    delete s;
    o->sym = nullptr;
}

// ---------------------------------------------------------------- instances
struct InstLists {
    const int32_t *ptr[4], *idx[4], *cfg[4];
    const int32_t* leaf_of_box;
};
struct InstOut {
    int32_t *ptr[4], *order[4];
    int4* src[4];
    int32_t* ostart;  // per list its orbits' first positions in `order` and the end: sym_first_row(q) + q on
};

// One warp per box: the mask of its (list, orbit) rows, the instances per list and one flag per row.
__global__ void __launch_bounds__(256) inst_count_kernel(InstLists L, int n, uint32_t* __restrict__ mask,
                                                         int32_t* __restrict__ cnt, int32_t* __restrict__ flags) {
    const int b = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (b >= n) return;
    uint32_t m = 0;
    for (int q = 0; q < 4; ++q)
        for (int e = L.ptr[q][b] + lane; e < L.ptr[q][b + 1]; e += 32) {
            int slots;
            m |= 1u << (sym_first_row(q) + sym_orbit(q, L.cfg[q][e], &slots));
        }
    m = __reduce_or_sync(0xffffffffu, m);
    if (lane == 0) mask[b] = m;
    if (lane < 4)
        cnt[(size_t)lane * n + b] = __popc((m >> sym_first_row(lane)) & ((1u << sym_orbits(lane)) - 1u));
    flags[(size_t)lane * n + b] = (m >> lane) & 1u;
}

// One warp per box: sources of its instances, and their places in orbit-major order. cnt and pos are
// the exclusive scans of the counts (list-major) and of the flags (row-major).
__global__ void __launch_bounds__(256) inst_fill_kernel(InstLists L, InstOut O, int n, const uint32_t* __restrict__ mask,
                                                        const int32_t* __restrict__ cnt,
                                                        const int32_t* __restrict__ pos, int total) {
    const int b = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (b >= n) return;
    const uint32_t m = mask[b];
    for (int q = 0; q < 4; ++q) {
        const int r0 = sym_first_row(q), first = cnt[(size_t)q * n + b] - cnt[(size_t)q * n];
        const uint32_t mq = (m >> r0) & ((1u << sym_orbits(q)) - 1u);
        if (lane == 0) {
            O.ptr[q][b] = first;
            if (b == n - 1) O.ptr[q][n] = first + __popc(mq);
        }
        for (int e = L.ptr[q][b] + lane; e < L.ptr[q][b + 1]; e += 32) {
            int slots;
            const int o = sym_orbit(q, L.cfg[q][e], &slots);
            const int s = L.idx[q][e];
            const int id = q == VFMM_LIST_U || q == VFMM_LIST_X ? L.leaf_of_box[s] : s;
            int* dst = reinterpret_cast<int*>(O.src[q] + first + __popc(mq & ((1u << o) - 1u)));
            for (int t = 0; t < 4; ++t)
                if ((slots >> t) & 1) dst[t] = id;
        }
        if (lane < sym_orbits(q) && ((mq >> lane) & 1u))
            O.order[q][pos[(size_t)(r0 + lane) * n + b] - pos[(size_t)r0 * n]] = first + __popc(mq & ((1u << lane) - 1u));
        if (b == 0 && lane <= sym_orbits(q)) {
            const int next = r0 + lane < kSymRows ? pos[(size_t)(r0 + lane) * n] : total;
            O.ostart[r0 + q + lane] = next - pos[(size_t)r0 * n];
        }
    }
}

int build_instances(DeviceTree* T, cudaStream_t st) {
    const int n = T->n_boxes;
    void* tmp = nullptr;  // [counts 4 n][flags 32 n]
    VFMM_CHECK(tree_malloc(reinterpret_cast<void**>(&T->inst_mask), (size_t)n * sizeof(uint32_t), st));
    VFMM_CHECK(tree_malloc(&tmp, (size_t)36 * n * sizeof(int32_t), st));
    uint32_t* mask = T->inst_mask;
    int32_t *cnt = (int32_t*)tmp, *flags = cnt + (size_t)4 * n;
    InstLists L;
    L.leaf_of_box = T->leaf_of_box;
    for (int q = 0; q < 4; ++q) {
        L.ptr[q] = T->lptr[q];
        L.idx[q] = T->lidx[q];
        L.cfg[q] = T->lcfg[q];
    }
    const unsigned grid = (unsigned)(((int64_t)n * 32 + 255) / 256);
    auto work = [&]() -> int {
        inst_count_kernel<<<grid, 256, 0, st>>>(L, n, mask, cnt, flags);
        VFMM_CUDA(cudaGetLastError());
        int64_t total = 0;
        VFMM_CHECK(exclusive_scan(flags, flags, (int64_t)kSymRows * n, nullptr, st));
        int32_t start[5] = {};
        VFMM_CHECK(exclusive_scan(cnt, cnt, (int64_t)4 * n, &total, st));
        for (int q = 1; q < 4; ++q)
            VFMM_CUDA(cudaMemcpyAsync(&start[q], cnt + (int64_t)q * n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
        VFMM_CUDA(cudaStreamSynchronize(st));
        start[4] = (int32_t)total;
        // one allocation: sources, then per list the box pointers and the orbit-major order, orbit starts
        size_t words = 4 * (size_t)total + total + 4 * ((size_t)n + 1) + kSymRows + 4;
        void* base = nullptr;
        VFMM_CHECK(tree_malloc(&base, words * sizeof(int32_t), st));
        T->inst = base;
        int4* s = (int4*)base;
        int32_t* w = (int32_t*)(s + total);
        VFMM_CUDA(cudaMemsetAsync(s, 0xFF, (size_t)total * sizeof(int4), st));
        InstOut O;
        for (int q = 0; q < 4; ++q) {
            T->n_inst[q] = start[q + 1] - start[q];
            O.src[q] = s + start[q];
            O.order[q] = w;
            w += T->n_inst[q];
            O.ptr[q] = w;
            w += n + 1;
            T->inst_src[q] = O.src[q];
            T->inst_order[q] = O.order[q];
            T->inst_ptr[q] = O.ptr[q];
        }
        O.ostart = w;
        for (int q = 0; q < 4; ++q) T->inst_ostart[q] = w + sym_first_row(q) + q;
        inst_fill_kernel<<<grid, 256, 0, st>>>(L, O, n, mask, cnt, flags, (int)total);
        VFMM_CUDA(cudaGetLastError());
        return VFMM_OK;
    };
    const int rc = work();
    cudaFreeAsync(tmp, st);
    return rc;
}

// ---------------------------------------------------------------- contraction
// What bounds it: the FP64 pipe (2 FMAs per clock and SM, one warp instruction in 64 clocks of a
// scheduler; one that its predicate switches off takes as long), so a tile is chosen to hold little
// padding: lanes hold columns (instances), warps rows, and the row tile is the smallest of 24, 48 and 96
// that fits a class (21 parts at p = 40, 48 node rows at k = 8, half of the 192 at k = 16). More rows
// spread the sums that form g (three additions per column value and row tile).
// Before, with plain tables, one column per list entry and 64 x 64 tiles -> now, us: near field 3850 ->
// 2127 (1,378 graded leaves, k = 16: many orbits hold one entry), 11498 -> 3193 (4,096 uniform leaves,
// the FP64 rate), 75 -> 17 (64 leaves, k = 8); graded tree S2M 279 -> 29, M2L 684 -> 253, S2L 277 -> 206,
// L2T 204 -> 49, M2T 252 (a series per node in the leaf kernel: 1500).
constexpr int kSymBK = 16, kSymThreads = 128;
constexpr int kSymMaxK = 256;

struct SymArgs {
    SymOp op;
    SymRun r;
    int n;  // q < 0: leaves
    const int32_t* ostart;
    const int32_t* order;
    const int4* src4;
};

template <int BN, int BM>
__global__ void __launch_bounds__(kSymThreads) sym_gemm_kernel(const __grid_constant__ SymArgs a) {
    constexpr int NSUB = 32 / BN, SLOTS = 4 * NSUB, NI = (BM + SLOTS - 1) / SLOTS;
    constexpr int NA = BM * kSymBK / kSymThreads, NB = BN * kSymBK / kSymThreads;
    static_assert(BM * kSymBK % kSymThreads == 0, "whole loads");
    __shared__ double As[kSymBK][NI * SLOTS];
    __shared__ double Bs[kSymBK][BN + 1];
    __shared__ const double* sp[4][BN];
    __shared__ int lut[4][kSymMaxK];  // offset of column k under reflection s, sign in the top bit
    const SymOp& op = a.op;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int c = blockIdx.z, row0 = blockIdx.y * BM;
    // the last orbits, which have the most columns, first
    int o = op.norb - 1, t = blockIdx.x, beg = 0, end = 0;
    for (; o >= 0; --o) {
        beg = a.ostart ? a.ostart[o] : 0;
        end = a.ostart ? a.ostart[o + 1] : a.n;
        const int nt = (end - beg + BN - 1) / BN;
        if (t < nt) break;
        t -= nt;
    }
    const int M = op.M[c] - row0;
    if (o < 0 || M <= 0) return;
    beg += t * BN;
    const int ncol = min(BN, end - beg), K = op.K[o][c];
    if (tid < BN) {
        int4 s = make_int4(-1, -1, -1, -1);
        if (tid < ncol) {
            if (a.src4) {
                s = a.src4[a.order[beg + tid]];
            } else {
                const int id = a.r.src_map ? a.r.src_map[beg + tid] : beg + tid;
                s = make_int4(id, id, id, id);
            }
        }
        sp[0][tid] = s.x >= 0 ? a.r.src + (size_t)s.x * a.r.src_stride : nullptr;
        sp[1][tid] = s.y >= 0 ? a.r.src + (size_t)s.y * a.r.src_stride : nullptr;
        sp[2][tid] = s.z >= 0 ? a.r.src + (size_t)s.z * a.r.src_stride : nullptr;
        sp[3][tid] = s.w >= 0 ? a.r.src + (size_t)s.w * a.r.src_stride : nullptr;
    }
    const int k = op.k, fx = op.fx[o], fy = op.fy[o], ca = c & 1, cb = c >> 1;
    const int nx = fx ? sym_half(k, ca) : k;
    for (int col = tid; col < K; col += kSymThreads)
        for (int s = 0; s < 4; ++s) {
            int at, neg = ((s & 1) & ca) ^ ((s >> 1) & cb);
            if (op.node_cols) {
                const int j = col / nx, i = col - j * nx;
                at = ((s & 2) ? k - 1 - j : j) * k + ((s & 1) ? k - 1 - i : i);
            } else {
                at = fx && fy ? sym_part(c, col) : (fx ? 2 * col + ((col & 1) ^ ca) : (fy ? 2 * col + cb : col));
                neg ^= sym_part_sign(at, s);
            }
            lut[s][col] = at | (neg << 31);
        }
    const double* A = op.A + op.off[o][c] + row0;
    const int ld = op.M[c], Mt = min(M, BM);
    __syncthreads();
    double ra[NA], rb[NB][4], acc[NI];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int e = tid + i * kSymThreads, kq = k0 + e / BM, r = e % BM;
            ra[i] = (kq < K && r < Mt) ? __ldg(A + (size_t)kq * ld + r) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = tid + i * kSymThreads, kq = k0 + (e & (kSymBK - 1)), col = e / kSymBK;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const double* p = sp[s][col];
                double v = 0.0;
                if (p && kq < K) {
                    const int at = lut[s][kq];
                    v = __ldg(p + (at & 0x7fffffff));
                    v = __hiloint2double(__double2hiint(v) ^ (at & 0x80000000), __double2loint(v));
                }
                rb[i][s] = v;
            }
        }
    };
    const int slot = warp * NSUB + lane / BN, bcol = lane & (BN - 1);
#pragma unroll
    for (int i = 0; i < NI; ++i) acc[i] = 0.0;
    load(0);
    for (int k0 = 0; k0 < K; k0 += kSymBK) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const int e = tid + i * kSymThreads;
            As[e / BM][e % BM] = ra[i];
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = tid + i * kSymThreads;
            Bs[e & (kSymBK - 1)][e / kSymBK] = (rb[i][0] + rb[i][1]) + (rb[i][2] + rb[i][3]);
        }
        __syncthreads();
        if (k0 + kSymBK < K) load(k0 + kSymBK);
        const int kn = min(kSymBK, K - k0);
        for (int kq = 0; kq < kn; ++kq) {
            const double b = Bs[kq][bcol];
#pragma unroll
            for (int i = 0; i < NI; ++i)
                acc[i] = fma(As[kq][slot + i * SLOTS], b, acc[i]);
        }
    }
    if (bcol >= ncol) return;
    int id = beg + bcol;
    double scale = 1.0;
    if (a.order) id = a.order[id];
    else if (a.r.out_map) id = a.r.out_map[id];
    if (a.r.level) {
        const double h = ldexp(a.r.width, -a.r.level[id]);
        scale = h * h;
    }
    double* out = a.r.out + (size_t)id * a.r.out_stride;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int r = slot + i * SLOTS;
        if (r < Mt) out[op.node_rows ? op.roff[c] + row0 + r : sym_part(c, row0 + r)] = scale * acc[i];
    }
}

template <int BM>
static void launch_sym(int bn, int64_t n, const SymArgs& a, int rows, cudaStream_t st) {
    const dim3 grid((unsigned)(n / bn + a.op.norb), rows, 4);
    if (bn == 32) sym_gemm_kernel<32, BM><<<grid, kSymThreads, 0, st>>>(a);
    else if (bn == 16) sym_gemm_kernel<16, BM><<<grid, kSymThreads, 0, st>>>(a);
    else sym_gemm_kernel<8, BM><<<grid, kSymThreads, 0, st>>>(a);
}

int sym_gemm(const DeviceTree& T, const SymOp& op, const SymRun& r, cudaStream_t st) {
    const int64_t n = r.q < 0 ? T.n_leaves : T.n_inst[r.q];
    if (n == 0) return VFMM_OK;
    SymArgs a;
    a.op = op;
    a.r = r;
    a.n = T.n_leaves;
    a.ostart = r.q < 0 ? nullptr : T.inst_ostart[r.q];
    a.order = r.q < 0 ? nullptr : T.inst_order[r.q];
    a.src4 = r.q < 0 ? nullptr : T.inst_src[r.q];
    int mmax = 0;
    for (int c = 0; c < 4; ++c) mmax = std::max(mmax, op.M[c]);
    const int bm = mmax <= 24 ? 24 : (mmax <= 48 ? 48 : 96), rows = (mmax + bm - 1) / bm;
    int dev = 0, sms = 0;
    VFMM_CUDA(cudaGetDevice(&dev));
    VFMM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // columns per CTA: 32 with at least twelve CTAs per SM (the last wave then costs little), fewer
    // where the tree is small, so that every SM's FP64 pipe has work
    int bn = 32;
    while (bn > 8 && (n / bn + op.norb) * rows * 4 < 12ll * sms) bn /= 2;
    if (bm == 24) launch_sym<24>(bn, n, a, rows, st);
    else if (bm == 48) launch_sym<48>(bn, n, a, rows, st);
    else launch_sym<96>(bn, n, a, rows, st);
    VFMM_CUDA(cudaGetLastError());
    return VFMM_OK;
}

}  // namespace vfmm
