// The FMM passes of the box code (Section 3.1), with the gradient from differentiated tables and
// expansions (Section 3.2), and the solve driver of both forms (FP64 below; the split-BF16
// contractions of the mixed form are in mixed.cu, mixed_far.cu and mixed_sym.cu).
//
//   S2M      leaf multipoles  a = h^2 Q f
//   M2M      one cooperative persistent pass over all levels (position-DFT form, readiness counters)
//   M2L      dense per V list or plane-wave (planewave.cu); S2L over the X list
//   DOWN     a second persistent pass:
//            b = L2L(parent) + sum_V M2L a_c (+ a_0(c) log h) + sum_X (2h)^2 R f_c (+ a_0(c) log h)
//   NEAR     sum over the U list of the configurations' tables applied to f
//   L2T, M2T far-field values from the leaf's local expansion and the W list's multipoles
//   LEAF     one CTA per leaf: u = h^2 NEAR - (1/2pi) log(h) sum_U a_0(src) + L2T + M2T (+ its log terms),
//            gradient = h NEAR' + (L2T' + M2T')/h
// The FP64 form's products run in the reflection classes of sym.cuh.
//
// Workspace (caller-owned, from vfmm_workspace_size): status word, multipoles and locals
// [n_boxes][2(p+1)], the FP64 form's slabs (a row per instance) or the mixed form's operands and
// outputs (+ I/O copies); see layout().
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "mixed.cuh"
#include "ops.cuh"
#include "sym.cuh"
#include "tc_ptx.cuh"
#include "vfmm_internal.cuh"

namespace vfmm {

constexpr double kInv2Pi = 0.15915494309189533577;

// log(h) of every level: a logarithm per box on the device is some 50 FP64 instructions of a whole warp,
// as much as the rest of a leaf's scalar terms.
struct LevelLogs {
    double v[kMaxDepth + 1];
    double h2[kMaxDepth + 1];  // h^2
};
static LevelLogs level_logs(double width) {
    LevelLogs l;
    for (int i = 0; i <= kMaxDepth; ++i) {
        l.v[i] = std::log(std::ldexp(width, -i));
        l.h2[i] = std::ldexp(width, -i) * std::ldexp(width, -i);
    }
    return l;
}

// Re of local coefficient 0 from the V and X lists of each virtual box (box, r): sum over V of
// Re(row 0 of M2L_c . a_c) + a_0(c) log h, and over X of (2h)^2 Re(S2L row 0) . f_c + a_0(c) log h.
// FP64, which bounds it (two FMAs per term; as product, FMA and addition 1.54 ms, now 1.14, at 266,805
// boxes); the other coefficients come from the split-precision M2L and S2L. Persistent CTAs hold the
// row-0 tables in shared memory; one warp per virtual box, the (entry, coefficient) pairs of eight
// V entries at a time spread over the lanes.
__global__ void __launch_bounds__(256) m2l_c0_kernel(int begin, int end, int R, int P,
                                                     const __grid_constant__ LevelLogs logs,
                                                     const int32_t* __restrict__ level,
                                                     const int32_t* __restrict__ vptr, const int32_t* __restrict__ vidx,
                                                     const int32_t* __restrict__ vcfg, const double2* __restrict__ m2l_r0,
                                                     const double* __restrict__ Mexp, double* __restrict__ c0,
                                                     const int32_t* __restrict__ xptr, const int32_t* __restrict__ xidx,
                                                     const int32_t* __restrict__ xcfg,
                                                     const int32_t* __restrict__ leaf_of_box,
                                                     const double* __restrict__ s2l_r0, const double* __restrict__ f,
                                                     int nleaf, int kk) {
    extern __shared__ __align__(16) unsigned char c0_raw[];
    double2* sM = reinterpret_cast<double2*>(c0_raw);           // [40][P]
    double* sX = reinterpret_cast<double*>(sM + kVCfg * P);      // [20][kk]
    for (int q = threadIdx.x; q < kVCfg * P; q += blockDim.x) sM[q] = m2l_r0[q];
    for (int q = threadIdx.x; q < kFarCfg * kk; q += blockDim.x) sX[q] = s2l_r0[q];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t total = (int64_t)(end - begin) * R;
    for (int64_t vw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; vw < total;
         vw += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int b = begin + (int)(vw / R), r = (int)(vw % R);
        const double logh = logs.v[level[b]];
        // V list: the warp walks the entries; lane n takes coefficients n, n + 32 of the source
        // multipole (coalesced), partial sums stay per lane until one final reduction
        double acc = 0.0, acc2 = 0.0;  // two FMAs per term, in chains of their own
        const int e_end = vptr[b + 1];
        // V list in batches of 8 entries: the batch's (entry, coefficient) pairs spread over the lanes,
        // so all 32 lanes work whatever p is (coalesced within an entry's multipole)
        for (int e0 = vptr[b]; e0 < e_end; e0 += 8) {
            const int nb = min(8, e_end - e0);
            int j = 0, n = lane;
            while (n >= P) {
                n -= P;
                ++j;
            }
#pragma unroll 4
            for (int item = lane; item < nb * P; item += 32) {
                const int e = e0 + j;
                const double2 x = reinterpret_cast<const double2*>(Mexp + ((size_t)vidx[e] * R + r) * 2 * P)[n];
                const double2 m = sM[vcfg[e] * P + n];
                acc = fma(m.x, x.x, acc);
                acc2 = fma(-m.y, x.y, acc2);
                n += 32;
                while (n >= P) {
                    n -= P;
                    ++j;
                }
            }
        }
        // log(h) a_0(c) of every V entry: one lane per entry
        double a0 = 0.0;
        for (int e = vptr[b] + lane; e < e_end; e += 32) a0 += Mexp[((size_t)vidx[e] * R + r) * 2 * P];
        acc += acc2;
        acc = fma(a0, logh, acc);
        // X list: (2h)^2 [Re(S2L row 0) . f_c + log(h) W . f_c], with W . f_c = a_0(c) / (2h)^2
        for (int e = xptr[b]; e < xptr[b + 1]; ++e) {
            const double* fc = f + ((size_t)r * nleaf + leaf_of_box[xidx[e]]) * kk;
            const double* r0 = sX + xcfg[e] * kk;
            double part = 0.0;
            for (int s = lane; s < kk; s += 32) part += r0[s] * fc[s];
            acc += 4.0 * logs.h2[level[b]] * part;
            if (lane == 0) acc += logh * Mexp[((size_t)xidx[e] * R + r) * 2 * P];
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) c0[(size_t)b * R + r] = acc;
    }
}

static int sm_count() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

// ---------------------------------------------------------------- a box's own terms of the downward pass
struct DownArgs {
    int P, R;  // R right-hand sides folded into the box rows (virtual box = box * R + r)
    double width;
    LevelLogs logs;
    const int32_t *vptr, *vidx;
    const int32_t *xptr, *xidx;
    const double* Mexp;
    // split-precision M2L rows 2..2p+1 (null in the FP64 form): (hi, lo) scaled by 2^-E[level][r]
    const float2* m2l_out;
    // split-K M2L: its partial sums [split][n_boxes * R][Rx], summed here when m2l_split > 1 (the
    // reduction kernel's order and arithmetic; that kernel is then not launched)
    const float2* m2l_part;
    int m2l_split;
    size_t m2l_stride;
    const int* m2l_E;   // [Rx] row exponents of the M2L tables
    const unsigned* m2l_G;  // [(depth + 1) R] biased level exponents of the multipole operand
    const double* m2l_c0;  // Re of local coefficient 0 from the V and X lists, with the log(h) terms
    const double* vslab;   // FP64 form: M2L of every V instance, [2(p+1)]
    const double* xslab;   // FP64 form: S2L of every X instance, [2(p+1)]
    const int32_t *viptr, *xiptr;  // instances of each box
    const double* pwloc;   // FP64 form, plane-wave M2L: [n_boxes][2(p+1)] V-list locals (null: vslab)
    int lw;                 // root width = wm 2^lw, wm in [1, 2)
    double wm;
    const float2* s2l_out; // split-precision S2L rows 2..2p+1, scaled by 2^-(E_f + E_r)
    const int* s2l_E;
    const int* Ef;
    int Rx;
};

// M2L output (hi, lo) of virtual box vb, row q: from the split-K partials or the reduced output.
__device__ __forceinline__ float2 m2l_value(const DownArgs& d, size_t vb, int q) {
    if (d.m2l_split > 1) {
        float hi = 0.0f, lo = 0.0f;
        for (int s = 0; s < d.m2l_split; ++s) df_add(hi, lo, d.m2l_part[(size_t)s * d.m2l_stride + vb * d.Rx + q]);
        return df_final(hi, lo);
    }
    return d.m2l_out[vb * d.Rx + q];
}

// FP64 form: a box's own terms of local coefficients t = lane, lane + 32 (one warp per box): the V and X
// instances' rows, in order, and the log(h) a_0 terms of the scaling.
__device__ __forceinline__ void own_terms_fp64(const DownArgs& d, int level, int b, int lane, double2 own[2]) {
    const int P = d.P;
    const double h = ldexp(d.width, -level);
    double a0 = 0.0;
    for (int e = d.vptr[b] + lane; e < d.vptr[b + 1]; e += 32) a0 += d.Mexp[(size_t)d.vidx[e] * 2 * P];
    for (int e = d.xptr[b] + lane; e < d.xptr[b + 1]; e += 32) a0 += d.Mexp[(size_t)d.xidx[e] * 2 * P];
    for (int o = 16; o > 0; o >>= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int t = lane + 32 * i;
        double re = 0.0, im = 0.0;
        if (t < P) {
            if (d.xiptr[b + 1] > d.xiptr[b]) {
                for (int e = d.xiptr[b]; e < d.xiptr[b + 1]; ++e) {
                    const double2 v = reinterpret_cast<const double2*>(d.xslab)[(size_t)e * P + t];
                    re += v.x;
                    im += v.y;
                }
                re *= 4.0 * h * h;
                im *= 4.0 * h * h;
            }
            if (d.pwloc) {
                const double2 v = reinterpret_cast<const double2*>(d.pwloc)[(size_t)b * P + t];
                re += v.x;
                im += v.y;
            } else {
#pragma unroll 4
                for (int e = d.viptr[b]; e < d.viptr[b + 1]; ++e) {
                    const double2 v = reinterpret_cast<const double2*>(d.vslab)[(size_t)e * P + t];
                    re += v.x;
                    im += v.y;
                }
            }
        }
        own[i] = make_double2(re, im);
    }
    if (lane == 0) own[0].x += d.logs.v[level] * a0;
}

// Mixed form: coefficient t of the local expansion of virtual box (b, r) at `level` = the L2L
// value (re, im) plus the split-precision M2L and S2L outputs scaled back by their exponents and
// the FP64 coefficient 0 (V and X rows 0 with the log(h) terms).
__device__ __forceinline__ double2 combine_local(const DownArgs& d, int level, int b, int r, int t, double re,
                                                 double im) {
    // (hi, lo) outputs to FP64 with their power-of-two scales folded into the exponent bits; the
    // S2L factor (2h)^2 = wm^2 2^(2 + 2 (lw - level)) for a root width wm 2^lw
    const size_t vb = (size_t)b * d.R + r;
    const bool has_v = d.vptr[b + 1] > d.vptr[b], has_x = d.xptr[b + 1] > d.xptr[b];
    if (has_x && t >= 1) {
        const float2 vr = d.s2l_out[vb * d.Rx + 2 * (t - 1)];
        const float2 vi = d.s2l_out[vb * d.Rx + 2 * (t - 1) + 1];
        const int e = d.Ef[r] + 2 + 2 * (d.lw - level);
        const int er = e + d.s2l_E[2 * (t - 1)], ei = e + d.s2l_E[2 * (t - 1) + 1];
        double sr = f2d_pair(vr, er);
        double si = f2d_pair(vi, ei);
        if (d.wm != 1.0) {
            sr *= d.wm * d.wm;
            si *= d.wm * d.wm;
        }
        re += sr;
        im += si;
    }
    if (has_v || has_x) {
        if (t == 0) {
            re += d.m2l_c0[vb];
        } else if (has_v) {
            const float2 vr = m2l_value(d, vb, 2 * (t - 1));
            const float2 vi = m2l_value(d, vb, 2 * (t - 1) + 1);
            const int g = level_exp_value(d.m2l_G[(size_t)level * d.R + r]);
            const int er = g + d.m2l_E[2 * (t - 1)], ei = g + d.m2l_E[2 * (t - 1) + 1];
            re += f2d_pair(vr, er);
            im += f2d_pair(vi, ei);
        }
    }
    return make_double2(re, im);
}

// ---------------------------------------------------------------- persistent tree passes
// One cooperative launch walks all levels. A unit is one virtual box, taken by a group of
// kGroupThreads threads (one warp on each of the SM's four schedulers, synchronised by a named
// barrier), and the real triangular matrix of the translation sits in shared memory for the whole
// pass. There is no barrier between levels: a unit waits (bounded) only for the expansions it reads,
// through per-box readiness counters, so a box starts as soon as its children (M2M) or its parent
// (L2L) are done. Every unit's inputs are produced by work that comes earlier in the global order,
// and each group takes its units in that order, so the earliest unfinished unit can always proceed
// (all CTAs are resident: cooperative launch). Data written by other CTAs are read through L2
// (ld.global.cg).
//
// Position-DFT form of the translations (this part retires about 2 FP64 FMAs per clock per SM, so
// the FP64 operation count per box sets the time of a level). With the rotated real form (tables.cu)
// M2M is A_l = sum_pos sigma^pos_l sum_n Rm[n][l] rho^pos_n a^pos_n, and the four child shifts
// are the Gaussian integers g_pos = i^e g_0, g_0 = 1 + i, with e = 0, 1, 2, 3 for the children
// at (+,+), (-,+), (-,-), (+,-) (child slots 3, 2, 0, 1). Then sigma^pos_l = i^(e l) sigma0_l and
// rho^pos_n = i^(-e n) rho0_n with sigma0_l = i^floor(l/2) (1 + i)^(l mod 2), rho0_n = conj(sigma0_n), so
//   M2M:  A_l = sigma0_l sum_{n<=l} Rm[n][l] E^(l mod 4)_n,   E^(c)_n = rho0_n F^((c - n) mod 4)_n,
//         F^(k)_n = sum_e i^(e k) a^(e)_n (a 4-point DFT over the children);
//   L2L:  c^(e)_m = rho0_m sum_c i^(e c) S^(c)_m,   S^(c)_m = sum_{l>=m, l-m = c mod 4} Rl[l][m] sigma0_l b_l.
// One real matrix-vector product per box instead of four complex ones: about P^2 FMAs plus 16 adds
// per coefficient for the DFT, against 8 P^2 FMAs with the four complex position tables.
constexpr int kPassThreads = 512;
constexpr int kGroupThreads = 128;
constexpr int kPassGroups = kPassThreads / kGroupThreads;
constexpr int kPassWarps = kPassThreads / 32;
constexpr int kPassMaxCtas = 152;  // largest pass grid

// Readiness counters of the dataflow tree passes: a producer publishes with a release add after its
// writes, a consumer polls with acquire loads before reading the expansion through L2.
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add_u32(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Waits (bounded) until *flag >= need. Gives up, recording code 6 in the status word, when the
// bound runs out; gives up at once when another wait already did (the status word is set).
__device__ bool wait_ready(const unsigned* flag, unsigned need, int* err) {
    for (long long it = 0; it < (1ll << 22); ++it) {
        if (ld_acquire_u32(flag) >= need) return true;
        if ((it & 63) == 63 && *(volatile int*)err) return false;
        __nanosleep(32);
    }
    atomicExch(err, 6);
    return false;
}

// Barrier of the kGroupThreads threads of group `grp` (named barrier 1 + grp; 0 is __syncthreads).
__device__ __forceinline__ void group_sync(int grp) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(kGroupThreads) : "memory");
}

// v, or -v where `on` (bit 0): on the bits, since a negation kept in a register costs an FP64 instruction.
__device__ __forceinline__ double flip(double v, int on) {
    return __hiloint2double(__double2hiint(v) ^ (on << 31), __double2loint(v));
}
// v i^m (sign changes and swaps; exact).
__device__ __forceinline__ double2 mul_ipow(double2 v, int m) {
    const double x = m & 1 ? v.y : v.x, y = m & 1 ? v.x : v.y;
    return make_double2(flip(x, (m ^ (m >> 1)) & 1), flip(y, (m >> 1) & 1));
}
// v sigma0_l = v i^floor(l/2) (1 + i)^(l mod 2): one addition per component for odd l.
__device__ __forceinline__ double2 mul_sigma0(double2 v, int l) {
    if (l & 1) v = make_double2(v.x - v.y, v.x + v.y);
    return mul_ipow(v, l >> 1);
}
// v rho0_n = v (-i)^floor(n/2) (1 - i)^(n mod 2).
__device__ __forceinline__ double2 mul_rho0(double2 v, int n) {
    if (n & 1) v = make_double2(v.x + v.y, v.y - v.x);
    return mul_ipow(v, -(n >> 1));
}
// sum_e i^(e k) x_e (one output of a 4-point DFT): (x0 +- x2) + i^k (x1 +- x3).
__device__ __forceinline__ double2 dft4(double2 x0, double2 x1, double2 x2, double2 x3, int k) {
    const int o = k & 1;  // one addition per component whichever k, not one for each parity in a mixed warp
    const double2 u = make_double2(x0.x + flip(x2.x, o), x0.y + flip(x2.y, o));
    const double2 w = mul_ipow(make_double2(x1.x + flip(x3.x, o), x1.y + flip(x3.y, o)), k);
    return make_double2(u.x + w.x, u.y + w.y);
}
// Child slot of DFT index e (g_pos = i^e (1 + i)).
__device__ __forceinline__ int child_of_e(int e) { return (0x1023 >> (4 * e)) & 0xF; }

struct PassArgs {
    int depth, R, P;
    const int32_t* nonleaf;
    const int32_t* nonleaf_start;  // device, depth + 2
    const int32_t* level_start;    // device, depth + 2
    const int32_t* child0;
    const double* tab;     // the real triangular matrix of the rotated form, [in][out]
    double2* ex;           // Mexp (upward) or Lexp (downward), [n_boxes * R][P] complex
    unsigned int* ready;   // [n_boxes * R] readiness counters, zero at launch
    unsigned* glev;        // upward pass, mixed form: biased level exponents of the M2L operand (or null)
    const int32_t* level;
    int* err;
};

// Shared memory of a pass: the real matrix [P][P] (rounded up to 16 bytes), then per group the
// scratch of one unit: M2M E [4][P] and the partial sums [kGroupThreads][2]; L2L sigma0 b [P] and
// S [4][P] (complex).
__host__ __device__ inline size_t pass_table_bytes(int P) { return ((size_t)P * P * sizeof(double) + 15) & ~(size_t)15; }
__host__ __device__ inline size_t pass_group_bytes(int P) { return (size_t)(4 * P + 2 * kGroupThreads) * sizeof(double2); }
__host__ __device__ inline size_t pass_smem_bytes(int P) { return pass_table_bytes(P) + kPassGroups * pass_group_bytes(P); }

// The real matrix into shared memory (plain loads; P^2 doubles need not be a multiple of 16 bytes).
__device__ __forceinline__ void load_real_table(double* sR, const double* tab, int P) {
    for (int q = threadIdx.x; q < P * P; q += blockDim.x) sR[q] = __ldg(tab + q);
    __syncthreads();
}

// All M2M levels, finest parents first (the global unit order): unit = one virtual parent box.
__global__ void __launch_bounds__(kPassThreads, 1) upward_pass_kernel(PassArgs a) {
    extern __shared__ __align__(128) unsigned char pass_raw[];
    __shared__ int abort_grp[kPassGroups];
    const int P = a.P, R = a.R;
    double* sR = reinterpret_cast<double*>(pass_raw);
    const int grp = threadIdx.x / kGroupThreads, g = threadIdx.x % kGroupThreads;
    double2* sE = reinterpret_cast<double2*>(pass_raw + pass_table_bytes(P) + grp * pass_group_bytes(P));
    double2* sPart = sE + 4 * P;
    if (g == 0) abort_grp[grp] = 0;
    load_real_table(sR, a.tab, P);
    const int npair = (P + 1) / 2, ns = max(1, kGroupThreads / npair);  // row pairs x slices
    const int slot = grp * gridDim.x + blockIdx.x, nslots = gridDim.x * kPassGroups;
    int l = a.depth - 1, lbase = 0;
    int lunits = l >= 2 ? (a.nonleaf_start[l + 1] - a.nonleaf_start[l]) * R : 0;
    for (int u = slot;; u += nslots) {
        while (l >= 2 && u >= lbase + lunits) {
            lbase += lunits;
            if (--l >= 2) lunits = (a.nonleaf_start[l + 1] - a.nonleaf_start[l]) * R;
        }
        if (l < 2) break;
        const int vi = u - lbase, bi = vi / R, r = vi - bi * R;
        const int b = a.nonleaf[a.nonleaf_start[l] + bi], c0 = a.child0[b];
        // the non-leaf children's multipoles must be complete (leaf multipoles come from S2M)
        if (g < 4 && a.child0[c0 + g] >= 0 && !wait_ready(a.ready + (size_t)(c0 + g) * R + r, 1u, a.err))
            abort_grp[grp] = 1;
        group_sync(grp);
        if (abort_grp[grp]) return;
        // E^(c)_n over the (k, n) pairs, the four children read once per pair
        const double2* x = a.ex + ((size_t)c0 * R + r) * P;
        const size_t xs = (size_t)R * P;
        for (int q = g; q < 4 * P; q += kGroupThreads) {
            const int k = q / P, n = q - k * P;
            const double2 f = dft4(__ldcg(x + 3 * xs + n), __ldcg(x + 2 * xs + n), __ldcg(x + n),
                                   __ldcg(x + xs + n), k);
            sE[((k + n) & 3) * P + n] = mul_rho0(f, n);
        }
        group_sync(grp);
        // row pair (j, P-1-j), slice s of the fused loop over both rows' inputs (row oa takes n <= oa)
        if (g < npair * ns) {
            const int j = g / ns, s = g - j * ns;
            const int oa = j, ob = P - 1 - j;
            const int la = oa + 1, lb = ob != oa ? ob + 1 : 0;
            const double2* ea = sE + (oa & 3) * P;
            const double2* eb = sE + (ob & 3) * P;
            double ar = 0.0, ai = 0.0, br = 0.0, bi2 = 0.0;
            // one loop per row: in a common loop a warp whose lanes are in different rows issues both bodies
            int i = s;
            for (; i < la; i += ns) {
                const double m = sR[i * P + oa];
                const double2 e = ea[i];
                ar = fma(m, e.x, ar);
                ai = fma(m, e.y, ai);
            }
            for (i -= la; i < lb; i += ns) {
                const double m = sR[i * P + ob];
                const double2 e = eb[i];
                br = fma(m, e.x, br);
                bi2 = fma(m, e.y, bi2);
            }
            sPart[2 * g] = make_double2(ar, ai);
            sPart[2 * g + 1] = make_double2(br, bi2);
        }
        group_sync(grp);
        // row l: its slices summed in order, rotated by sigma0_l
        int e = INT_MIN;
        if (g < P) {
            const int j = min(g, P - 1 - g), w = g == j ? 0 : 1;
            double2 acc = sPart[2 * j * ns + w];
            for (int s = 1; s < ns; ++s) {
                const double2 t = sPart[2 * (j * ns + s) + w];
                acc = make_double2(acc.x + t.x, acc.y + t.y);
            }
            acc = mul_sigma0(acc, g);
            a.ex[((size_t)b * R + r) * P + g] = acc;
            e = max(part_exp(acc.x, 2 * g), part_exp(acc.y, 2 * g + 1));
            __threadfence();
        }
        // the M2L operand's level exponent (mixed form), taken as the coefficients are written
        if (a.glev && g < ((P + 31) & ~31)) level_exp_max(e, a.glev + (size_t)l * R + r);
        group_sync(grp);
        if (g == 0) red_release_add_u32(a.ready + (size_t)b * R + r, 1u);
    }
}

// All downward levels. First every box of level >= 2 gets its own terms (the M2L and S2L outputs and
// coefficient 0) in one warp unit per virtual box, counted 1 on its readiness word
// (level 2 boxes are then complete). Then, level by level, each non-leaf parent's local is shifted
// to its 4 children (L2L) and added to their own terms, counted 1 more (complete at 2).
template <bool kMixed>
__global__ void __launch_bounds__(kPassThreads, 1) downward_pass_kernel(PassArgs a, DownArgs d) {
    extern __shared__ __align__(128) unsigned char pass_raw[];
    __shared__ int abort_grp[kPassGroups];
    const int P = a.P, R = a.R;
    double* sR = reinterpret_cast<double*>(pass_raw);
    const int grp = threadIdx.x / kGroupThreads, g = threadIdx.x % kGroupThreads;
    double2* sG = reinterpret_cast<double2*>(pass_raw + pass_table_bytes(P) + grp * pass_group_bytes(P));
    double2* sS = sG + P;
    if (g == 0) abort_grp[grp] = 0;
    load_real_table(sR, a.tab, P);
    // own terms: one warp per virtual box
    {
        const int lane = threadIdx.x & 31;
        const int wslot = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nw = gridDim.x * kPassWarps;
        const int64_t vb0 = (int64_t)a.level_start[2] * R, vb1 = (int64_t)a.level_start[a.depth + 1] * R;
        for (int64_t vb = vb0 + wslot; vb < vb1; vb += nw) {
            const int b = (int)(vb / R), r = (int)(vb % R), lv = a.level[b];
            if constexpr (kMixed) {
                for (int t = lane; t < P; t += 32) a.ex[(size_t)vb * P + t] = combine_local(d, lv, b, r, t, 0.0, 0.0);
            } else {
                double2 own[2];
                own_terms_fp64(d, lv, b, lane, own);
                if (lane < P) a.ex[(size_t)vb * P + lane] = own[0];
                if (lane + 32 < P) a.ex[(size_t)vb * P + lane + 32] = own[1];
            }
            __threadfence();
            __syncwarp();
            if (lane == 0) red_release_add_u32(a.ready + vb, 1u);
        }
    }
    const int npair = (P + 1) / 2;
    const int slot = grp * gridDim.x + blockIdx.x, nslots = gridDim.x * kPassGroups;
    int l = 3, lbase = 0;  // l: the children's level
    int lunits = l <= a.depth ? (a.nonleaf_start[l] - a.nonleaf_start[l - 1]) * R : 0;
    for (int u = slot;; u += nslots) {
        while (l <= a.depth && u >= lbase + lunits) {
            lbase += lunits;
            if (++l <= a.depth) lunits = (a.nonleaf_start[l] - a.nonleaf_start[l - 1]) * R;
        }
        if (l > a.depth) break;
        const int vi = u - lbase, bi = vi / R, r = vi - bi * R;
        const int b = a.nonleaf[a.nonleaf_start[l - 1] + bi], c0 = a.child0[b];
        // the parent's local must be complete, the children's own terms written
        bool ok = true;
        if (g == 4) ok = wait_ready(a.ready + (size_t)b * R + r, l - 1 == 2 ? 1u : 2u, a.err);
        else if (g < 4) ok = wait_ready(a.ready + (size_t)(c0 + g) * R + r, 1u, a.err);
        if (!ok) abort_grp[grp] = 1;
        group_sync(grp);
        if (abort_grp[grp]) return;
        const double2* bl = a.ex + ((size_t)b * R + r) * P;
        for (int t = g; t < P; t += kGroupThreads) sG[t] = mul_sigma0(__ldcg(bl + t), t);
        group_sync(grp);
        // S^(c) of the row pair (oa, ob): thread (j, c)
        for (int q = g; q < 4 * npair; q += kGroupThreads) {
            const int j = q >> 2, c = q & 3;
            const int oa = j, ob = P - 1 - j;
            double ar = 0.0, ai = 0.0;
            for (int li = oa + c; li < P; li += 4) {
                const double m = sR[li * P + oa];
                ar = fma(m, sG[li].x, ar);
                ai = fma(m, sG[li].y, ai);
            }
            sS[c * P + oa] = make_double2(ar, ai);
            if (ob != oa) {
                double br = 0.0, bi2 = 0.0;
                for (int li = ob + c; li < P; li += 4) {
                    const double m = sR[li * P + ob];
                    br = fma(m, sG[li].x, br);
                    bi2 = fma(m, sG[li].y, bi2);
                }
                sS[c * P + ob] = make_double2(br, bi2);
            }
        }
        group_sync(grp);
        // child e, coefficient m: own terms + rho0_m sum_c i^(e c) S^(c)_m
        for (int q = g; q < 4 * P; q += kGroupThreads) {
            const int e = q / P, m = q - e * P;
            const double2 h = mul_rho0(dft4(sS[m], sS[P + m], sS[2 * P + m], sS[3 * P + m], e), m);
            double2* out = a.ex + ((size_t)(c0 + child_of_e(e)) * R + r) * P + m;
            const double2 own = __ldcg(out);
            *out = make_double2(own.x + h.x, own.y + h.y);
        }
        __threadfence();
        group_sync(grp);
        if (g < 4) red_release_add_u32(a.ready + (size_t)(c0 + g) * R + r, 1u);
    }
}

// Mixed form, one CTA per virtual leaf (leaf, r), one thread per node: u, u_x, u_y = near + far +
// scalar, the split contraction outputs (hi, lo) scaled back by their power-of-two exponents. The
// scalar part, the same at every node of the leaf, is FP64:
// -(1/2pi) [log(h) sum_U a_0 + Re b_0 + sum_W a_0 (log h_w)], h_w = h / 2 (first warp, fixed-order sums).
// q / d for q below 1024 and d up to 64: (q m) >> 16, m = floor(65535 / d) + 1.
struct SmallDiv {
    unsigned m;
    __device__ __forceinline__ int operator()(int q) const { return (int)(((unsigned)q * m) >> 16); }
};
static SmallDiv small_div(int d) { return SmallDiv{65535u / (unsigned)d + 1u}; }

struct LeafMixedArgs {
    int nleaf, R, k, kk, Rp, P, lw;
    double wm;
    bool scaled;  // wm != 1 (a comparison in FP64 costs what an addition does)
    LevelLogs logs;
    const int32_t* box_of_leaf;
    const int32_t* level;
    const int32_t *uptr, *uidx, *wptr, *widx;
    const double* Mexp;
    const double* Lexp;
    SmallDiv by_hh, by_h, by_k;
    int near_split, far_split;  // partial sums by classes
    ClassTab ct, ft;        // near field, far field (N = 0: by entries)
    const float2* nearmix;  // class rows (ct.N > 0) or node rows
    const int* Er;          // exponents of these rows
    const int* Ef;
    const float2* farmix;
    const int* farE;
    const int* Et;
    // entry-major leaf far field: the slab rows of every leaf's entries, summed here in entry order (the
    // arithmetic of the separate segmented sum, which the contraction then skips); null: farmix holds the sums
    const float2* far_slab;
    const int32_t* far_seg;
    double *u, *ux, *uy;
};

// Sum of the slab rows of entries [e0, e1), right-hand side r, row `row` (double-float, entry order).
__device__ __forceinline__ float2 slab_sum(const float2* __restrict__ slab, int e0, int e1, int R, int r, int Rp,
                                           int row) {
    float hi = 0.0f, lo = 0.0f;
#pragma unroll 4
    for (int e = e0; e < e1; ++e) df_add(hi, lo, slab[((size_t)e * R + r) * Rp + row]);
    return df_final(hi, lo);
}

__device__ __forceinline__ float2 df_sum(float2 a, float2 b, float sgn) {
    float hi = a.x, lo = a.y;
    df_add(hi, lo, make_float2(sgn * b.x, sgn * b.y));
    return df_final(hi, lo);
}

// Node values s [3][kk] from class rows: the four classes of a quadrant node, brought to the largest of their
// exponents, put together at its images (double-FP32: the FP64 pipe is what bounds the kernel), and
// that exponent, se [3][quadrant nodes].
__device__ __forceinline__ void class_nodes(const ClassTab& ct, const float2* __restrict__ rows,
                                            int split, size_t stride, const int* __restrict__ E, int k, SmallDiv by_hh,
                                            SmallDiv by_h, float2* s, int* se) {
    const int hx = (k + 1) / 2, kk = k * k;
    for (int q = threadIdx.x; q < 3 * hx * hx; q += blockDim.x) {
        const int fl = by_hh(q), e = q - fl * hx * hx, j = by_h(e), i = e - j * hx;
        float2 w[4];  // by the field's parity in x and y
        int ew[4], emax = -1000;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int pa = u & 1, pb = u >> 1, c = (pa ^ (fl == 1)) | ((pb ^ (fl == 2)) << 1), nx = sym_half(k, pa);
            const bool in = i < nx && j < sym_half(k, pb);
            const int row = ct.seg[3 * c + fl] + j * nx + i;
            w[u] = in ? rows[row] : make_float2(0.0f, 0.0f);
            for (int sp = 1; in && sp < split; ++sp) w[u] = df_sum(w[u], rows[sp * stride + row], 1.0f);
            ew[u] = in ? E[row] : -1000;
            emax = max(emax, ew[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            // 2^(ew - emax); an exponent 100 below the largest is far beneath its last bit
            const float sc = ew[u] > emax - 100 ? __int_as_float((127 + ew[u] - emax) << 23) : 0.0f;
            w[u] = make_float2(w[u].x * sc, w[u].y * sc);
        }
        se[q] = emax;
        const float2 x = df_sum(w[0], w[1], 1.0f), y = df_sum(w[0], w[1], -1.0f);
        const float2 z = df_sum(w[2], w[3], 1.0f), v = df_sum(w[2], w[3], -1.0f);
        float2* o = s + fl * kk;
        const int i1 = k - 1 - i, j1 = k - 1 - j;
        o[j * k + i] = df_sum(x, z, 1.0f);
        if (i1 != i) o[j * k + i1] = df_sum(y, v, 1.0f);
        if (j1 != j) o[j1 * k + i] = df_sum(x, z, -1.0f);
        if (i1 != i && j1 != j) o[j1 * k + i1] = df_sum(y, v, -1.0f);
    }
}

__global__ void leaf_mixed_kernel(const __grid_constant__ LeafMixedArgs a) {
    // width = wm 2^lw with wm in [1, 2): h = wm 2^(lw - lv), so every power-of-two scale is folded
    // into the exponents (f2d_scaled), times wm^(2, 1, -1) when wm is not one
    // near field and far field at the nodes, [3][kk] each; by classes, their exponents [3][h][h]
    extern __shared__ float2 s_near[];
    __shared__ int s_ne[3 * 64], s_fe[3 * 64];
    __shared__ double s_scal;
    const int nleaf = a.nleaf, R = a.R, kk = a.kk, Rp = a.Rp, lw = a.lw, k = a.k, hx = (k + 1) / 2;
    const double wm = a.wm;
    const unsigned vl = blockIdx.x;
    const int t = threadIdx.x;
    const unsigned leaf = vl / (unsigned)R, r = vl - leaf * (unsigned)R;
    const int b = a.box_of_leaf[leaf];
    const int lv = a.level[b];
    float2* s_far = s_near + 3 * kk;
    if (a.ct.N == 0) {  // by entries: node rows
        const float2* nm = a.nearmix + (size_t)vl * Rp;
        for (int q = t; q < 3 * kk; q += blockDim.x) s_near[q] = nm[q];
    } else {
        const size_t nrow = 4 * a.ct.nch * a.ct.N, frow = 4 * a.ft.nch * a.ft.N, nv = (size_t)nleaf * R;
        class_nodes(a.ct, a.nearmix + vl * nrow, a.near_split, nv * nrow, a.Er, k, a.by_hh, a.by_h, s_near, s_ne);
        class_nodes(a.ft, a.farmix + vl * frow, a.far_split, nv * frow, a.farE, k, a.by_hh, a.by_h, s_far, s_fe);
    }
    __syncthreads();
    double n0 = 0.0, n1 = 0.0, n2 = 0.0, f0 = 0.0, f1 = 0.0, f2 = 0.0;
    if (t < kk) {
        const float2* __restrict__ farmix = a.farmix;
        const int* Er = a.ct.N ? s_ne : a.Er;
        const int* farE = a.ct.N ? s_fe : a.farE;
        const int* __restrict__ Et = a.Et;
        const int* __restrict__ Ef = a.Ef;
        const float2* fm = farmix + (size_t)vl * Rp;
        const int en = Ef[r] + (a.ct.N ? 1 : 0) + lw - lv, et = Et[vl], ef = et + lv - lw;  // near scale h 2^(E_f + 0, 1), far scale 2^E_t / h
        const float2 v0 = s_near[t], v1 = s_near[kk + t], v2 = s_near[2 * kk + t];
        float2 w0, w1, w2;
        if (a.ft.N) {
            w0 = s_far[t];
            w1 = s_far[kk + t];
            w2 = s_far[2 * kk + t];
        } else if (a.far_slab) {
            const int s0 = a.far_seg[leaf], s1 = a.far_seg[leaf + 1];
            w0 = slab_sum(a.far_slab, s0, s1, R, r, Rp, t);
            w1 = slab_sum(a.far_slab, s0, s1, R, r, Rp, kk + t);
            w2 = slab_sum(a.far_slab, s0, s1, R, r, Rp, 2 * kk + t);
        } else {
            w0 = fm[t];
            w1 = fm[kk + t];
            w2 = fm[2 * kk + t];
        }
        const int tj = a.by_k(t), ti = t - tj * k;
        const int qn = a.ct.N ? min(tj, k - 1 - tj) * hx + min(ti, k - 1 - ti) : t, qs = a.ct.N ? hx * hx : kk;
        const int e0 = en + lw - lv + Er[qn], e1 = en + Er[qs + qn], e2 = en + Er[2 * qs + qn];
        n0 = f2d_pair(v0, e0);  // h^2 x near u
        n1 = f2d_pair(v1, e1);  // h x near u_x
        n2 = f2d_pair(v2, e2);
        const int g0 = et + farE[qn], g1 = ef + farE[qs + qn], g2 = ef + farE[2 * qs + qn];
        f0 = f2d_pair(w0, g0);
        f1 = f2d_pair(w1, g1);  // far u_x / h
        f2 = f2d_pair(w2, g2);
        if (a.scaled) {
            n0 *= wm * wm;
            n1 *= wm;
            n2 *= wm;
            f1 /= wm;
            f2 /= wm;
        }
    }
    if (t < 32) {
        const size_t P2 = 2 * (size_t)a.P;
        const double logh = a.logs.v[lv];
        double m = 0.0, w0 = 0.0;
        for (int e = a.uptr[b] + t; e < a.uptr[b + 1]; e += 32) m += a.Mexp[((size_t)a.uidx[e] * R + r) * P2];
        for (int e = a.wptr[b] + t; e < a.wptr[b + 1]; e += 32) w0 += a.Mexp[((size_t)a.widx[e] * R + r) * P2];
        m = fma(logh, m, (logh - 0.6931471805599453) * w0);
        for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
        if (t == 0) s_scal = -kInv2Pi * (m + a.Lexp[((size_t)b * R + r) * P2]);
    }
    __syncthreads();
    if (t >= kk) return;
    const size_t o = ((size_t)r * nleaf + leaf) * kk + t;
    a.u[o] = n0 + s_scal + f0;
    a.ux[o] = n1 + f1;
    a.uy[o] = n2 + f2;
}

// ---------------------------------------------------------------- leaf pass (one CTA per leaf)
struct LeafArgs {
    SymOp op;  // rows of the classes
    int nleaf, kk, k, P;
    double width;
    LevelLogs logs;
    const int32_t* box_of_leaf;
    const int32_t* level;
    const int32_t *uptr, *uidx, *wptr, *widx;
    const int32_t *uiptr, *wiptr;  // instances of each box
    const double* slab;            // near field of every U instance, [3kk]
    const double* wslab;           // M2T of every W instance, [3kk]
    const double* far;             // L2T of every leaf, [3kk]
    const double* Mexp;
    const double* Lexp;
    double* u;
    double* ux;
    double* uy;
};

// FP64 form: one CTA per leaf sums its instances' rows and the far values class by class, in order,
// then each node puts its four classes together and adds the scalar log terms
// -(1/2pi) (log(h) sum_U a_0 + log(h_w) sum_W a_0), h_w = h / 2 (first warp).
__global__ void __launch_bounds__(256) leaf_kernel(const __grid_constant__ LeafArgs a) {
    extern __shared__ double rows[];  // [3kk] class rows of u, u_x, u_y
    __shared__ double s_scal;
    const int leaf = blockIdx.x, t = threadIdx.x, kk = a.kk, k = a.k;
    const int b = a.box_of_leaf[leaf];
    const double h = ldexp(a.width, -a.level[b]), ih = 1.0 / h;
    for (int r = t; r < 3 * kk; r += blockDim.x) {
        int s = 0;
        while (r >= a.op.seg[s + 1]) ++s;
        double n = 0.0, f = a.far[(size_t)leaf * 3 * kk + r];
        for (int e = a.uiptr[b]; e < a.uiptr[b + 1]; ++e) n += a.slab[(size_t)e * 3 * kk + r];
        for (int e = a.wiptr[b]; e < a.wiptr[b + 1]; ++e) f += a.wslab[(size_t)e * 3 * kk + r];
        rows[r] = s % 3 == 0 ? fma(h * h, n, f) : fma(h, n, f * ih);
    }
    if (t < 32) {
        const int P2 = 2 * a.P;
        double m = 0.0, w0 = 0.0;
        for (int e = a.uptr[b] + t; e < a.uptr[b + 1]; e += 32) m += a.Mexp[(size_t)a.uidx[e] * P2];
        for (int e = a.wptr[b] + t; e < a.wptr[b + 1]; e += 32) w0 += a.Mexp[(size_t)a.widx[e] * P2];
        for (int o = 16; o > 0; o >>= 1) {
            m += __shfl_xor_sync(0xffffffffu, m, o);
            w0 += __shfl_xor_sync(0xffffffffu, w0, o);
        }
        if (t == 0) {
            const double logh = a.logs.v[a.level[b]];
            s_scal = -kInv2Pi * (logh * m + (logh - 0.6931471805599453) * w0);
        }
    }
    __syncthreads();
    if (t >= kk) return;
    const int j = t / k, i = t - j * k;
    const int i0 = min(i, k - 1 - i), j0 = min(j, k - 1 - j), s = (i > i0 ? 1 : 0) | (j > j0 ? 2 : 0);
    double v[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int pa = sym_pa(c, q), pb = sym_pb(c, q), nx = sym_half(k, pa);
            if (i0 >= nx || j0 >= sym_half(k, pb)) continue;  // an odd field's middle line
            const double x = rows[a.op.seg[3 * c + q] + j0 * nx + i0];
            v[q] += ((s & pa) ^ ((s >> 1) & pb)) & 1 ? -x : x;
        }
    const size_t o = (size_t)leaf * kk + t;
    a.u[o] = v[0] + s_scal;
    a.ux[o] = v[1];
    a.uy[o] = v[2];
}

// ---------------------------------------------------------------- host side
struct Workspace {
    bool fork = false;  // mixed form: run the near field and S2L on the thread's second stream
    double* vslab;      // FP64 form: per V instance M2L rows
    double* xslab;      // FP64 form: per X instance S2L rows
    double* wslab;      // FP64 form: per W instance M2T rows
    double* pwX;        // FP64 form, plane-wave M2L: [n_boxes][4][s] outgoing coefficients (null: dense)
    double* pwL;        // FP64 form, plane-wave M2L: [n_boxes][2(p+1)] V-list local coefficients
    const PlanSet* ps;  // split-contraction plans for the folded right-hand sides (mixed form)
    unsigned int* ready; // [2][n_boxes * R] readiness counters of the persistent tree passes, then
                         // [(depth + 1) R] biased level exponents (mixed form)
    size_t ready_words;
    double* Mexp;
    double* Lexp;
    double* slab;
    double* far;
    double* io;  // f, u, ux, uy copies for the host entry point
    MixedWork mix;
    size_t bytes;
};

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Workspace carving. The mixed form folds all nrhs right-hand sides into one solve (every per-box and
// per-leaf buffer has nrhs rows per box); the FP64 form solves them one at a time. room (not 0): bytes of a
// scratch of fixed size, for a solve on one stream; its near field and leaf far field then take no split sums
// and, one after the other, the same operand buffer, which gets what the rest leaves.
static int layout(const DeviceTree& T, const vfmm_ops& o, int nrhs, bool io, Workspace* w, char* base,
                  size_t* bytes, size_t room = 0) {
    const size_t P2 = 2 * (size_t)(o.p + 1), kk = (size_t)o.k * o.k;
    size_t off = 0;
    auto take = [&](double** p, size_t n) {
        if (w) *p = (double*)(base + off);
        off += align256(std::max<size_t>(1, n) * sizeof(double));
    };
    double* dummy;
    const bool mixed = o.precision == VFMM_MIXED;
    const size_t R = mixed ? (size_t)nrhs : 1;
    // the status word comes first in both forms, so that it can be read back knowing only the
    // workspace address (vfmm_workspace_status)
    int* err = nullptr;
    {
        double* e = nullptr;
        take(&e, 1);
        err = reinterpret_cast<int*>(e);
    }
    take(w ? &w->Mexp : &dummy, (size_t)T.n_boxes * R * P2);
    take(w ? &w->Lexp : &dummy, (size_t)T.n_boxes * R * P2);
    {
        // readiness counters of the persistent passes, then the mixed form's biased level exponents:
        // one zeroing at the start of a solve covers both
        double* g = nullptr;
        const size_t words = 2 * (size_t)T.n_boxes * R + (size_t)(T.depth + 1) * R;
        take(&g, (words + 1) / 2);
        if (w) {
            w->ready = reinterpret_cast<unsigned int*>(g);
            w->ready_words = words;
        }
    }
    const bool pw = !mixed && o.m2l_form == VFMM_M2L_PLANEWAVE;
    if (w) w->slab = w->far = w->vslab = w->xslab = w->wslab = w->pwX = w->pwL = nullptr;
    if (!mixed) {
        take(w ? &w->slab : &dummy, (size_t)T.n_inst[VFMM_LIST_U] * 3 * kk);
        // the M2L and S2L rows (or plane waves) are read before the leaf far field is written: one region
        const size_t shared = off;
        if (pw) {
            take(w ? &w->pwX : &dummy, planewave_work_doubles(T.n_boxes, o));
            take(w ? &w->pwL : &dummy, (size_t)T.n_boxes * P2);
        } else {
            take(w ? &w->vslab : &dummy, (size_t)T.n_inst[VFMM_LIST_V] * P2);
        }
        take(w ? &w->xslab : &dummy, (size_t)T.n_inst[VFMM_LIST_X] * P2);
        const size_t down_end = off;
        off = shared;
        take(w ? &w->far : &dummy, (size_t)T.n_leaves * 3 * kk);
        take(w ? &w->wslab : &dummy, (size_t)T.n_inst[VFMM_LIST_W] * 3 * kk);
        off = std::max(off, down_end);
    }
    if (mixed) {
        const MixedOps* mo = (const MixedOps*)o.mixed;
        const PlanSet* PS = nullptr;
        VFMM_CHECK(plans_for(T, (int)R, &PS));
        if (w) w->ps = PS;
        const size_t nl = (size_t)T.n_leaves * R, nb = (size_t)T.n_boxes * R;
        double* p = nullptr;
        take(&p, (nl * kSlices * mo->Kp * 2 + 7) / 8);
        if (w) w->mix.fsl = (void*)p;
        const bool cls = near_by_classes(o.k);
        const int ns = cls && !room ? PS->near.split : 1, fs = cls && !room ? PS->leaf.split : 1;  // partial sums
        if (w) {
            w->mix.near_split = ns;
            w->mix.leaf_split = fs;
        }
        take(&p, nl * ns * (cls ? 4 * mo->near.nch * mo->near.N : mo->Rp));
        if (w) w->mix.out = (float2*)p;
        take(&p, R);
        if (w) w->mix.fmax = (unsigned long long*)p;
        take(&p, (R + 1) / 2);
        if (w) w->mix.Ef = (int*)p;
        take(&p, nl * mo->Rx);
        if (w) w->mix.s2m_out = (float2*)p;
        if (w) w->mix.glev = w->ready + 2 * (size_t)T.n_boxes * R;
        take(&p, (nb * kSlices * mo->Kx * 2 + 7) / 8);
        if (w) w->mix.msl = (void*)p;
        take(&p, nb * mo->Rx);
        if (w) w->mix.m2l_out = (float2*)p;
        take(&p, nb);
        if (w) w->mix.m2l_c0 = p;
        take(&p, nb * mo->Rx);
        if (w) w->mix.s2l_out = (float2*)p;
        const size_t ab = !cls ? (size_t)T.n_far_slots * R * kSlices * mo->Kx * 2
                               : (room ? 0 : class_operand_bytes(mo->leaf, PS->leaf, 0));
        take(&p, (ab + 7) / 8);
        if (w) {
            w->mix.aprep = (void*)p;
            w->mix.aprep_bytes = ab;
        }
        take(&p, cls ? (nb + 1) / 2 : 1);
        if (w) w->mix.bexp = (int*)p;
        take(&p, (nl + 1) / 2);
        if (w) w->mix.Et = (int*)p;
        take(&p, nl * fs * (cls ? 4 * mo->leaf.nch * mo->leaf.N : mo->Rp));
        if (w) w->mix.far_out = (float2*)p;
        size_t np[3] = {0, 0, 0};
        split_part_elems(T, *PS, o, np);
        float2** bufs[3] = {w ? &w->mix.part : nullptr, w ? &w->mix.part_s2l : nullptr,
                            w ? &w->mix.part_side : nullptr};
        for (int i = 0; i < 3; ++i) {
            take(&p, std::max<size_t>(np[i], 1));  // one float2 per double
            if (w) *bufs[i] = np[i] ? (float2*)p : nullptr;
        }
        take(&p, cls ? nl * kk : 1);
        if (w) w->mix.ffix = (long long*)p;
        const size_t left = room > off ? (room - off) & ~(size_t)255 : size_t(1);
        size_t ob = class_operand_bytes(mo->near, PS->near, room ? left : 0);
        if (room && cls) ob = std::max(ob, class_operand_bytes(mo->leaf, PS->leaf, left));
        take(&p, (ob + 7) / 8);
        if (w) {
            w->mix.near_opnd = p;
            w->mix.near_opnd_bytes = ob;
            if (room && cls) {
                w->mix.aprep = p;
                w->mix.aprep_bytes = ob;
            }
        }
    } else if (w) {
        w->mix = MixedWork();
        w->ps = &T.plans;
    }
    if (w) w->mix.err = err;
    if (io) take(w ? &w->io : &dummy, (size_t)4 * nrhs * T.n_leaves * kk);
    else if (w) w->io = nullptr;
    if (w) w->bytes = off;
    *bytes = off;
    return VFMM_OK;
}

// Optional stage timing: a start and a stop event around every stage.
struct StageEvents {
    cudaEvent_t ev[2 * VFMM_N_STAGES];
    int launches = 0;
};

enum { ST_S2M = 0, ST_M2M = 1, ST_DOWN = 2, ST_NEAR = 3, ST_L2T = 4, ST_LEAF = 5, ST_CONTRACTIONS = 6 };

static inline void mark(StageEvents* se, int stage, bool stop, cudaStream_t st) {
    if (se) cudaEventRecord(se->ev[2 * stage + (stop ? 1 : 0)], st);
}

static void fill_down_args(DownArgs& d, const DeviceTree& T, const vfmm_ops& o, const Workspace& w, int R) {
    const MixedOps* mo = (const MixedOps*)o.mixed;
    d.R = R;
    d.wm = 2.0 * std::frexp(T.width, &d.lw);
    d.lw -= 1;
    d.P = o.p + 1;
    d.width = T.width;
    d.logs = level_logs(T.width);
    d.vptr = T.lptr[VFMM_LIST_V];
    d.vidx = T.lidx[VFMM_LIST_V];
    d.xptr = T.lptr[VFMM_LIST_X];
    d.xidx = T.lidx[VFMM_LIST_X];
    d.Mexp = w.Mexp;
    d.vslab = w.vslab;
    d.xslab = w.xslab;
    d.viptr = T.inst_ptr[VFMM_LIST_V];
    d.xiptr = T.inst_ptr[VFMM_LIST_X];
    d.pwloc = w.pwL;
    d.m2l_out = mo ? w.mix.m2l_out : nullptr;
    // a grouped split-K M2L leaves its partial sums to the downward kernels (m2l_mixed defers them)
    const bool m2l_parts = mo && !w.ps->m2l.entry && w.ps->m2l.split > 1 && w.mix.part;
    d.m2l_part = m2l_parts ? w.mix.part : nullptr;
    d.m2l_split = m2l_parts ? w.ps->m2l.split : 1;
    d.m2l_stride = (size_t)T.n_boxes * R * (mo ? mo->Rx : 0);
    d.m2l_E = mo ? mo->m2l_E : nullptr;
    d.m2l_G = mo ? w.mix.glev : nullptr;
    d.m2l_c0 = mo ? w.mix.m2l_c0 : nullptr;
    d.s2l_out = mo ? w.mix.s2l_out : nullptr;
    d.s2l_E = mo ? mo->s2l_E : nullptr;
    d.Ef = mo ? w.mix.Ef : nullptr;
    d.Rx = mo ? mo->Rx : 0;
}

// One cooperative launch per pass, whatever the tree's size: one real matrix-vector product per box, and
// no launch per level. On 266,805 boxes the upward levels took 2.17 ms as one launch each, 1.21 as a pass,
// the downward ones 2.32 and 1.60; with one FP64 addition per term of the DFTs whatever the lane's index and
// one loop per row 0.89 and 1.43. Bound by FP64 (2 FMA a clock and SM) and its latency at one CTA per SM;
// small trees by the levels' latency.
template <typename... Args>
static int launch_pass(void (*kernel)(Args...), int R, int P, int widest_items, int cap, cudaStream_t st,
                       Args... args) {
    const size_t smem = pass_smem_bytes(P);
    static thread_local int attr_dev[3] = {-1, -1, -1};
    const int slot = (void*)kernel == (void*)upward_pass_kernel ? 0
                     : (void*)kernel == (void*)downward_pass_kernel<true> ? 1 : 2;
    int dev = 0;
    cudaGetDevice(&dev);
    if (attr_dev[slot] != dev) {
        VFMM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr_dev[slot] = dev;
    }
    int per_sm = 0;
    VFMM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kPassThreads, smem));
    if (per_sm < 1) return fail(VFMM_ERR_INTERNAL, "tree pass kernel does not fit on an SM");
    // A cooperative launch: a unit may wait for units held by any other CTA, so all CTAs must be
    // resident. One CTA per box of the widest level (the first group of each CTA takes a level's
    // first boxes, so that they run on different SMs), at most one per SM and at most kPassMaxCtas:
    // a smaller grid starts sooner when another stream's kernels still hold SMs (the launch waits
    // until the whole grid fits).
    int grid = std::max(1, std::min(std::min(per_sm * sm_count(), kPassMaxCtas), widest_items));
    if (cap > 0) grid = std::min(grid, cap);  // any grid works: units wait only on lower-numbered units
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kPassThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    VFMM_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
    return VFMM_OK;
}

// Second stream of the calling host thread on the current device, with its fork and join events:
// a split-precision solve runs its S2L and near-field contractions there, beside S2M, M2M and M2L.
// Created by the first call outside stream capture (a call under capture before that runs on one
// stream) and kept for the life of the process. One per thread, so that the event sequence of a
// solve cannot interleave with another thread's.
struct SideStream {
    cudaStream_t s = nullptr;    // S2L and the near field, lowest priority
    cudaStream_t hp = nullptr;   // everything else, highest priority: first to get SMs that free up
    cudaStream_t aux = nullptr;  // coefficient 0 beside M2L, highest priority
    // f sliced; S2L done; near field done; solve start; solve end; M2M done; coefficient 0 done
    cudaEvent_t ev[7] = {};
};

static SideStream* side_stream(cudaStream_t st) {
    constexpr int kMaxDevices = 16;
    thread_local SideStream slots[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    SideStream& ss = slots[dev];
    if (ss.s) return &ss;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) return nullptr;
    SideStream n;
    int least = 0, greatest = 0;
    bool ok = cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess;
    ok = ok && cudaStreamCreateWithPriority(&n.s, cudaStreamNonBlocking, least) == cudaSuccess;
    ok = ok && cudaStreamCreateWithPriority(&n.hp, cudaStreamNonBlocking, greatest) == cudaSuccess;
    ok = ok && cudaStreamCreateWithPriority(&n.aux, cudaStreamNonBlocking, greatest) == cudaSuccess;
    for (int i = 0; i < 7 && ok; ++i) ok = cudaEventCreateWithFlags(&n.ev[i], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
        for (cudaEvent_t e : n.ev)
            if (e) cudaEventDestroy(e);
        if (n.s) cudaStreamDestroy(n.s);
        if (n.hp) cudaStreamDestroy(n.hp);
        if (n.aux) cudaStreamDestroy(n.aux);
        cudaGetLastError();
        return nullptr;
    }
    ss = n;
    return &ss;
}

// Kernels one split contraction launches: the contraction, and its split-K or segmented reduction
// unless the consumer takes that sum over (split_gemm's defer bits).
static int gemm_launches(const SplitPlan& P, int defer = 0) {
    const bool reduce = P.entry ? !(defer & kDeferSegments) : (P.split > 1 && !(defer & kDeferSplits));
    return P.n_groups > 0 ? 1 + (reduce ? 1 : 0) : 0;
}

// One solve of R right-hand sides (f: [R][n_leaves][k^2]). The mixed form folds them into the
// rows of every contraction (PS holds plans for R); the FP64 form takes R = 1.
static int solve_steps(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, double* u,
                       double* ux, double* uy, const Workspace& w, cudaStream_t st, StageEvents* se,
                       SideStream* side);

static int solve_one(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, double* u,
                     double* ux, double* uy, const Workspace& w, cudaStream_t st, StageEvents* se = nullptr) {
    // Mixed form with side streams: once f is sliced, S2L and then the near field run on a
    // low-priority stream while a high-priority stream takes every other step; the latter waits
    // for S2L before the downward combine and for the near field before the leaf kernels, and the
    // caller's stream waits for it at the end. Timed calls keep to the caller's stream.
    SideStream* side = (o.precision == VFMM_MIXED && w.fork && !se && !w.mix.cev) ? side_stream(st) : nullptr;
    if (!side) return solve_steps(T, PS, o, f, u, ux, uy, w, st, se, nullptr);
    VFMM_CUDA(cudaEventRecord(side->ev[3], st));
    VFMM_CUDA(cudaStreamWaitEvent(side->hp, side->ev[3], 0));
    VFMM_CHECK(solve_steps(T, PS, o, f, u, ux, uy, w, side->hp, se, side));
    VFMM_CUDA(cudaEventRecord(side->ev[4], side->hp));
    VFMM_CUDA(cudaStreamWaitEvent(st, side->ev[4], 0));
    return VFMM_OK;
}

static int solve_steps(const DeviceTree& T, const PlanSet& PS, const vfmm_ops& o, const double* f, double* u,
                       double* ux, double* uy, const Workspace& w, cudaStream_t st, StageEvents* se,
                       SideStream* side) {
    const int P = o.p + 1, P2 = 2 * P, kk = o.k * o.k;
    const int nleaf = T.n_leaves;
    const bool mixed = o.precision == VFMM_MIXED;
    const int R = PS.R;
    if (!mixed && R != 1) return fail(VFMM_ERR_INTERNAL, "the FP64 form solves one right-hand side at a time");
    const MixedOps* mo = (const MixedOps*)o.mixed;
    const SymTables* sy = (const SymTables*)o.sym;
    int launches = 0;
    // readiness counters (persistent passes) and level exponents (mixed form) start at zero
    VFMM_CUDA(cudaMemsetAsync(w.ready, 0, w.ready_words * sizeof(unsigned int), st));
    if (mixed) {
        // near field first: its f slices also feed S2M and S2L
        mark(se, ST_NEAR, false, st);
        VFMM_CHECK(near_slices(T, PS, o, f, w.mix, st));
        launches += 2;
        if (side) {
            VFMM_CUDA(cudaEventRecord(side->ev[0], st));
            VFMM_CUDA(cudaStreamWaitEvent(side->s, side->ev[0], 0));
            if (T.depth >= 2) {
                VFMM_CHECK(s2l_mixed(T, PS, o, w.mix, side->s));
                launches += gemm_launches(PS.s2l);
            }
            VFMM_CUDA(cudaEventRecord(side->ev[1], side->s));
            VFMM_CHECK(near_contract(T, PS, o, f, w.mix, side->s));
            VFMM_CUDA(cudaEventRecord(side->ev[2], side->s));
        } else {
            VFMM_CHECK(near_contract(T, PS, o, f, w.mix, st));
        }
        launches += near_by_classes(o.k)
                        ? 1 + class_launches(mo->near, PS.near, mo->slices[kCtrNear], w.mix.near_opnd_bytes)
                        : gemm_launches(PS.entries);
        mark(se, ST_NEAR, true, st);
    }
    // S2M
    mark(se, ST_S2M, false, st);
    if (mixed) {
        VFMM_CHECK(s2m_mixed(T, PS, o, f, w.Mexp, w.mix, st));
        launches += 1 + gemm_launches(PS.s2m, kDeferSplits);
    } else {
        ++launches;
        SymRun r;
        r.src = f;
        r.src_stride = kk;
        r.out = w.Mexp;
        r.out_stride = P2;
        r.out_map = T.box_of_leaf;
        r.level = T.level;
        r.width = T.width;
        VFMM_CHECK(sym_gemm(T, sy->s2m, r, st));
    }
    mark(se, ST_S2M, true, st);
    // M2M, finest parents first (levels >= 2 are the ones the lists read)
    mark(se, ST_M2M, false, st);
    int widest = 0;
    for (int l = 1; l <= T.depth; ++l) widest = std::max(widest, T.nonleaf_start[l + 1] - T.nonleaf_start[l]);
    if (T.depth >= 3) {
        PassArgs pa;
        pa.depth = T.depth;
        pa.R = R;
        pa.P = P;
        pa.nonleaf = T.nonleaf;
        pa.nonleaf_start = T.nonleaf_start_dev;
        pa.level_start = T.level_start_dev;
        pa.child0 = T.child0;
        pa.tab = o.m2m_r;
        pa.ex = reinterpret_cast<double2*>(w.Mexp);
        pa.ready = w.ready;
        pa.glev = mixed ? w.mix.glev : nullptr;
        pa.level = T.level;
        pa.err = w.mix.err;
        VFMM_CHECK(launch_pass(upward_pass_kernel, R, P, widest * R, mixed ? PS.pass_ctas : 0, st, pa));
        ++launches;
    }
    mark(se, ST_M2M, true, st);
    // downward pass
    mark(se, ST_DOWN, false, st);
    if (mixed && T.depth >= 2) {
        // coefficient 0 (FP64) needs only the multipoles: beside M2L when forked
        cudaStream_t c0s = st;
        if (side) {
            VFMM_CUDA(cudaEventRecord(side->ev[5], st));
            VFMM_CUDA(cudaStreamWaitEvent(side->aux, side->ev[5], 0));
            c0s = side->aux;
        }
        VFMM_CHECK(m2l_mixed(T, PS, o, w.Mexp, w.mix, st));
        if (PS.m2l.n_groups > 0) launches += 2 + gemm_launches(PS.m2l, kDeferSplits);
        if (near_by_classes(o.k)) {
            VFMM_CHECK(leaf_class_bounds(T, PS, o, w.Mexp, w.mix, c0s));
            ++launches;
        }
        const int begin = T.level_start[2], end = T.level_start[T.depth + 1];
        const int64_t warps = (int64_t)(end - begin) * R;
        const size_t c0_smem = (size_t)kVCfg * P * sizeof(double2) + (size_t)kFarCfg * kk * sizeof(double);
        static thread_local int c0_attr_dev = -1;
        int dev = 0;
        cudaGetDevice(&dev);
        if (c0_attr_dev != dev) {
            cudaFuncSetAttribute(m2l_c0_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
            c0_attr_dev = dev;
        }
        const unsigned c0_grid = (unsigned)std::min<int64_t>((warps + 7) / 8, 3ll * sm_count());
        m2l_c0_kernel<<<c0_grid, 256, c0_smem, c0s>>>(
            begin, end, R, P, level_logs(T.width), T.level, T.lptr[VFMM_LIST_V], T.lidx[VFMM_LIST_V], T.lcfg[VFMM_LIST_V],
            reinterpret_cast<const double2*>(mo->m2l_r0), w.Mexp, w.mix.m2l_c0, T.lptr[VFMM_LIST_X],
            T.lidx[VFMM_LIST_X], T.lcfg[VFMM_LIST_X], T.leaf_of_box, mo->s2l_r0, f, nleaf, kk);
        ++launches;
        if (side) {
            VFMM_CUDA(cudaEventRecord(side->ev[6], side->aux));
            VFMM_CUDA(cudaStreamWaitEvent(st, side->ev[6], 0));
        }
        if (!side) {
            VFMM_CHECK(s2l_mixed(T, PS, o, w.mix, st));
            launches += gemm_launches(PS.s2l);
        }
    }
    if (side) VFMM_CUDA(cudaStreamWaitEvent(st, side->ev[1], 0));
    if (!mixed) {
        // FP64 form: M2L (V list) and S2L (X list) in reflection classes, one slab row per instance; the
        // downward kernels below sum them
        if (w.pwX) {
            // plane-wave form: outgoing waves of every box, then diagonal translations and the
            // incoming conversion per target box
            if (T.depth >= 2) {
                launches += 2;
                VFMM_CHECK(planewave_m2l(o, T.level_start[2], T.n_boxes, T.lptr[VFMM_LIST_V],
                                         T.lidx[VFMM_LIST_V], T.lcfg[VFMM_LIST_V], w.Mexp, w.pwX, w.pwL, st));
            }
        } else if (T.n_inst[VFMM_LIST_V] > 0) {
            ++launches;
            SymRun r;
            r.q = VFMM_LIST_V;
            r.src = w.Mexp;
            r.src_stride = P2;
            r.out = w.vslab;
            r.out_stride = P2;
            VFMM_CHECK(sym_gemm(T, sy->m2l, r, st));
        }
        if (T.n_inst[VFMM_LIST_X] > 0) {
            ++launches;
            SymRun r;
            r.q = VFMM_LIST_X;
            r.src = f;
            r.src_stride = kk;
            r.out = w.xslab;
            r.out_stride = P2;
            VFMM_CHECK(sym_gemm(T, sy->s2l, r, st));
        }
    }
    if (T.depth >= 2) {
        DownArgs d;
        fill_down_args(d, T, o, w, R);
        PassArgs pa;
        pa.depth = T.depth;
        pa.R = R;
        pa.P = P;
        pa.nonleaf = T.nonleaf;
        pa.nonleaf_start = T.nonleaf_start_dev;
        pa.level_start = T.level_start_dev;
        pa.child0 = T.child0;
        pa.tab = o.l2l_r;
        pa.ex = reinterpret_cast<double2*>(w.Lexp);
        pa.ready = w.ready + (size_t)T.n_boxes * R;
        pa.glev = nullptr;
        pa.level = T.level;
        pa.err = w.mix.err;
        const int items = std::max(widest * R, 16 * R);
        if (mixed) VFMM_CHECK(launch_pass(downward_pass_kernel<true>, R, P, items, PS.pass_ctas, st, pa, d));
        else VFMM_CHECK(launch_pass(downward_pass_kernel<false>, R, P, items, 0, st, pa, d));
        ++launches;
    }
    if (T.depth < 2) VFMM_CUDA(cudaMemsetAsync(w.Lexp, 0, (size_t)T.n_boxes * R * P2 * sizeof(double), st));
    else VFMM_CUDA(cudaMemsetAsync(w.Lexp, 0, (size_t)T.level_start[2] * R * P2 * sizeof(double), st));
    mark(se, ST_DOWN, true, st);
    if (!mixed) {
        mark(se, ST_NEAR, false, st);
        ++launches;
        SymRun r;
        r.q = VFMM_LIST_U;
        r.src = f;
        r.src_stride = kk;
        r.out = w.slab;
        r.out_stride = 3 * kk;
        VFMM_CHECK(sym_gemm(T, sy->near, r, st));
        mark(se, ST_NEAR, true, st);
    }
    // far field at the leaves
    mark(se, ST_L2T, false, st);
    if (mixed) {
        VFMM_CHECK(far_leaf_mixed(T, PS, o, w.Mexp, w.Lexp, w.mix, st));
        launches += near_by_classes(o.k) ? class_launches(mo->leaf, PS.leaf, leaf_class_slices(*mo), w.mix.aprep_bytes)
                                         : 1 + gemm_launches(PS.far, kDeferSegments);
    } else {
        launches += T.n_inst[VFMM_LIST_W] > 0 ? 2 : 1;
        SymRun r;
        r.src = w.Lexp;
        r.src_stride = P2;
        r.src_map = T.box_of_leaf;
        r.out = w.far;
        r.out_stride = 3 * kk;
        VFMM_CHECK(sym_gemm(T, sy->l2t, r, st));
        r.q = VFMM_LIST_W;
        r.src = w.Mexp;
        r.src_map = nullptr;
        r.out = w.wslab;
        VFMM_CHECK(sym_gemm(T, sy->m2t, r, st));
    }
    mark(se, ST_L2T, true, st);
    mark(se, ST_LEAF, false, st);
    if (mixed) {
        const int64_t nv = (int64_t)nleaf * R;
        int lw = 0;
        const double wm = 2.0 * std::frexp(T.width, &lw);  // width = wm 2^lw, wm in [1, 2)
        lw -= 1;
        if (side) VFMM_CUDA(cudaStreamWaitEvent(st, side->ev[2], 0));  // the near-field output
        LeafMixedArgs la;
        la.nleaf = nleaf;
        la.R = R;
        la.k = o.k;
        la.kk = kk;
        la.Rp = mo->Rp;
        la.P = P;
        la.lw = lw;
        la.wm = wm;
        la.scaled = wm != 1.0;
        la.logs = level_logs(T.width);
        la.box_of_leaf = T.box_of_leaf;
        la.level = T.level;
        la.uptr = T.lptr[VFMM_LIST_U];
        la.uidx = T.lidx[VFMM_LIST_U];
        la.wptr = T.lptr[VFMM_LIST_W];
        la.widx = T.lidx[VFMM_LIST_W];
        la.Mexp = w.Mexp;
        la.Lexp = w.Lexp;
        la.nearmix = w.mix.out;
        const int hx = (o.k + 1) / 2;
        la.by_hh = small_div(hx * hx);
        la.by_h = small_div(hx);
        la.by_k = small_div(o.k);
        la.near_split = w.mix.near_split;
        la.far_split = w.mix.leaf_split;
        la.ct = mo->near;
        la.ft = mo->leaf;
        la.Er = near_by_classes(o.k) ? mo->near_E : mo->Er;
        la.Ef = w.mix.Ef;
        la.farmix = w.mix.far_out;
        la.farE = near_by_classes(o.k) ? mo->leaf_E : mo->far_E;
        la.Et = w.mix.Et;
        // an entry-major leaf far field leaves its per-leaf sums (a few entries per leaf) to this kernel
        la.far_slab = PS.far.entry ? w.mix.part : nullptr;
        la.far_seg = PS.far.entry ? PS.far.seg : nullptr;
        la.u = u;
        la.ux = ux;
        la.uy = uy;
        leaf_mixed_kernel<<<(unsigned)nv, std::max(32, ((kk + 31) / 32) * 32), (size_t)6 * kk * sizeof(float2), st>>>(la);
        ++launches;
    } else {
        LeafArgs a;
        a.op = sy->near;
        a.nleaf = nleaf;
        a.kk = kk;
        a.k = o.k;
        a.P = P;
        a.width = T.width;
        a.logs = level_logs(T.width);
        a.box_of_leaf = T.box_of_leaf;
        a.level = T.level;
        a.uptr = T.lptr[VFMM_LIST_U];
        a.uidx = T.lidx[VFMM_LIST_U];
        a.wptr = T.lptr[VFMM_LIST_W];
        a.widx = T.lidx[VFMM_LIST_W];
        a.uiptr = T.inst_ptr[VFMM_LIST_U];
        a.wiptr = T.inst_ptr[VFMM_LIST_W];
        a.slab = w.slab;
        a.wslab = w.wslab;
        a.far = w.far;
        a.Mexp = w.Mexp;
        a.Lexp = w.Lexp;
        a.u = u;
        a.ux = ux;
        a.uy = uy;
        leaf_kernel<<<(unsigned)nleaf, ((kk + 31) / 32) * 32, (size_t)3 * kk * sizeof(double), st>>>(a);
        ++launches;
    }
    mark(se, ST_LEAF, true, st);
    VFMM_CUDA(cudaGetLastError());
    if (se) se->launches += launches;
    return VFMM_OK;
}

}  // namespace vfmm

using namespace vfmm;

static int check_solve_args(const vfmm_tree* tree, const vfmm_ops* ops, int32_t nrhs) {
    if (!tree || !ops) return fail(VFMM_ERR_INVALID_ARG, "null tree or ops");
    if (tree->t.k != ops->k) return fail(VFMM_ERR_INVALID_ARG, "tree and ops differ in k");
    if (nrhs < 1) return fail(VFMM_ERR_INVALID_ARG, "nrhs must be >= 1");
    if (ops->p + 1 > 64) return fail(VFMM_ERR_INVALID_ARG, "p too large for the solve kernels");
    return VFMM_OK;
}

int vfmm::scratch_bytes(const vfmm_tree* tree, const vfmm_ops* ops, size_t room, size_t* bytes) {
    VFMM_CHECK(check_solve_args(tree, ops, 1));
    return layout(tree->t, *ops, 1, false, nullptr, nullptr, bytes, room);
}

extern "C" int vfmm_workspace_size(const vfmm_tree* tree, const vfmm_ops* ops, int32_t nrhs, int32_t with_io,
                                   size_t* bytes) {
    VFMM_CHECK(check_solve_args(tree, ops, nrhs));
    if (!bytes) return fail(VFMM_ERR_INVALID_ARG, "null bytes");
    return layout(tree->t, *ops, nrhs, with_io != 0, nullptr, nullptr, bytes);
}

// All right-hand sides: one folded solve in the mixed form, one solve per right-hand side in FP64.
static int solve_all(const DeviceTree& T, const vfmm_ops& o, const double* f, int nrhs, double* u, double* ux,
                     double* uy, const Workspace& w, cudaStream_t st, StageEvents* se = nullptr) {
    if (o.precision == VFMM_MIXED) return solve_one(T, *w.ps, o, f, u, ux, uy, w, st, se);
    const size_t n = (size_t)T.n_leaves * o.k * o.k;
    for (int r = 0; r < nrhs; ++r) VFMM_CHECK(solve_one(T, T.plans, o, f + r * n, u + r * n, ux + r * n, uy + r * n, w, st, se));
    return VFMM_OK;
}

static int reset_status(const Workspace& w, cudaStream_t st) {
    if (w.mix.err) VFMM_CUDA(cudaMemsetAsync(w.mix.err, 0, sizeof(int), st));
    return VFMM_OK;
}

// What a non-zero status word means: where the first bounded device wait that ran out was.
static const char* status_site(int code) {
    switch (code) {
        case 1: return "a tensor-core producer waiting for a free stage";
        case 2: return "the tensor-core MMA issuer waiting for operands";
        case 3: return "a tensor-core epilogue waiting for its accumulators";
        case 4: return "the tensor-core MMA issuer waiting for drained accumulators";
        case 6: return "a persistent tree pass waiting for an expansion another unit writes";
        case 7: return "the failure-path self-test's wait on an mbarrier nothing arrives on (expected)";
        default: return "an unknown site";
    }
}

// Reads the status word at `word` (device) after the solve that wrote it has finished.
int vfmm::read_status_word(const int* word) {
    if (!word) return VFMM_OK;
    int h = 0;
    VFMM_CUDA(cudaMemcpy(&h, word, sizeof(int), cudaMemcpyDeviceToHost));
    if (h) return fail(VFMM_ERR_TIMEOUT, std::string("a bounded wait ran out: ") + status_site(h) +
                                             " (code " + std::to_string(h) + ")");
    return VFMM_OK;
}

// After a synchronised solve: a bounded device wait that expired shows up here.
static int read_status(const Workspace& w) { return read_status_word(w.mix.err); }

int vfmm::volume_potential(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_dev, int32_t nrhs,
                           double* u_dev, double* ux_dev, double* uy_dev, void* workspace_dev, size_t workspace_bytes,
                           cudaStream_t st, bool fork, bool reset, bool fixed) {
    VFMM_CHECK(check_solve_args(tree, ops, nrhs));
    if (!f_dev || !u_dev || !ux_dev || !uy_dev || !workspace_dev) return fail(VFMM_ERR_INVALID_ARG, "null buffer");
    Workspace w;
    size_t need = 0;
    VFMM_CHECK(layout(tree->t, *ops, nrhs, false, &w, (char*)workspace_dev, &need, fixed ? workspace_bytes : 0));
    if (workspace_bytes < need) return fail(VFMM_ERR_WORKSPACE, "workspace too small");
    w.fork = fork && !fixed;
    if (reset) VFMM_CHECK(reset_status(w, st));
    return solve_all(tree->t, *ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, w, st);
}

int vfmm::solve_expansions(const vfmm_tree* tree, const vfmm_ops* ops, const void* workspace_dev,
                           size_t workspace_bytes, const double** Mexp, const double** Lexp, int* R) {
    Workspace w;
    size_t need = 0;
    VFMM_CHECK(layout(tree->t, *ops, 1, false, &w, (char*)const_cast<void*>(workspace_dev), &need));
    if (workspace_bytes < need) return fail(VFMM_ERR_WORKSPACE, "workspace smaller than a one-right-hand-side solve's");
    *Mexp = w.Mexp;
    *Lexp = w.Lexp;
    *R = 1;
    return VFMM_OK;
}

extern "C" int vfmm_workspace_status(const void* workspace_dev) {
    if (!workspace_dev) {
        // the allocation-free entry point's scratch on the current device
        const int* word = nullptr;
        VFMM_CHECK(noalloc_status_word(&word));
        return read_status_word(word);
    }
    return read_status_word(static_cast<const int*>(workspace_dev));
}

extern "C" int vfmm_volume_potential(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_dev, int32_t nrhs,
                                     double* u_dev, double* ux_dev, double* uy_dev, void* workspace_dev,
                                     size_t workspace_bytes, void* stream) {
    return volume_potential(tree, ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, workspace_dev, workspace_bytes,
                            (cudaStream_t)stream, true);
}

extern "C" int vfmm_volume_potential_host(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_host,
                                          int32_t nrhs, double* u_host, double* ux_host, double* uy_host,
                                          void* workspace_dev, size_t workspace_bytes, void* stream) {
    VFMM_CHECK(check_solve_args(tree, ops, nrhs));
    if (!f_host || !u_host || !ux_host || !uy_host || !workspace_dev) return fail(VFMM_ERR_INVALID_ARG, "null buffer");
    Workspace w;
    size_t need = 0;
    VFMM_CHECK(layout(tree->t, *ops, nrhs, true, &w, (char*)workspace_dev, &need));
    if (workspace_bytes < need) return fail(VFMM_ERR_WORKSPACE, "workspace too small (with_io = 1 required)");
    w.fork = true;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t n = (size_t)tree->t.n_leaves * ops->k * ops->k * nrhs;
    double* f = w.io;
    double* u = w.io + n;
    double* ux = w.io + 2 * n;
    double* uy = w.io + 3 * n;
    VFMM_CHECK(reset_status(w, st));
    VFMM_CUDA(cudaMemcpyAsync(f, f_host, n * sizeof(double), cudaMemcpyHostToDevice, st));
    VFMM_CHECK(solve_all(tree->t, *ops, f, nrhs, u, ux, uy, w, st));
    VFMM_CUDA(cudaMemcpyAsync(u_host, u, n * sizeof(double), cudaMemcpyDeviceToHost, st));
    VFMM_CUDA(cudaMemcpyAsync(ux_host, ux, n * sizeof(double), cudaMemcpyDeviceToHost, st));
    VFMM_CUDA(cudaMemcpyAsync(uy_host, uy, n * sizeof(double), cudaMemcpyDeviceToHost, st));
    VFMM_CUDA(cudaStreamSynchronize(st));
    return read_status(w);
}

extern "C" int vfmm_volume_potential_profiled(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_dev,
                                              int32_t nrhs, double* u_dev, double* ux_dev, double* uy_dev,
                                              void* workspace_dev, size_t workspace_bytes, void* stream,
                                              float* stage_ms, int32_t* launches) {
    VFMM_CHECK(check_solve_args(tree, ops, nrhs));
    if (!f_dev || !u_dev || !ux_dev || !uy_dev || !workspace_dev || !stage_ms || !launches)
        return fail(VFMM_ERR_INVALID_ARG, "null buffer");
    Workspace w;
    size_t need = 0;
    VFMM_CHECK(layout(tree->t, *ops, nrhs, false, &w, (char*)workspace_dev, &need));
    if (workspace_bytes < need) return fail(VFMM_ERR_WORKSPACE, "workspace too small");
    cudaStream_t st = (cudaStream_t)stream;
    VFMM_CHECK(reset_status(w, st));
    StageEvents se;
    for (int i = 0; i < 2 * VFMM_N_STAGES; ++i) VFMM_CUDA(cudaEventCreate(&se.ev[i]));
    for (int i = 0; i < VFMM_N_STAGES; ++i) stage_ms[i] = 0.0f;
    if (ops->precision == VFMM_MIXED) {
        // contraction timers: recorded once here so that a contraction the tree lacks reads 0
        w.mix.cev = se.ev + 2 * ST_CONTRACTIONS;
        for (int i = 2 * ST_CONTRACTIONS; i < 2 * VFMM_N_STAGES; ++i) VFMM_CUDA(cudaEventRecord(se.ev[i], st));
    }
    const size_t n = (size_t)tree->t.n_leaves * ops->k * ops->k;
    const bool folded = ops->precision == VFMM_MIXED;
    int rc = VFMM_OK;
    for (int r = 0; r < (folded ? 1 : nrhs) && rc == VFMM_OK; ++r) {
        rc = folded ? solve_one(tree->t, *w.ps, *ops, f_dev, u_dev, ux_dev, uy_dev, w, st, &se)
                    : solve_one(tree->t, tree->t.plans, *ops, f_dev + r * n, u_dev + r * n, ux_dev + r * n,
                                uy_dev + r * n, w, st, &se);
        if (rc != VFMM_OK) break;
        cudaError_t e = cudaEventSynchronize(se.ev[2 * ST_LEAF + 1]);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "cudaEventSynchronize");
            break;
        }
        const int n_timed = ops->precision == VFMM_MIXED ? VFMM_N_STAGES : ST_CONTRACTIONS;
        for (int i = 0; i < n_timed; ++i) {
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, se.ev[2 * i], se.ev[2 * i + 1]);
            stage_ms[i] += ms;
        }
    }
    for (int i = 0; i < 2 * VFMM_N_STAGES; ++i) cudaEventDestroy(se.ev[i]);
    *launches = se.launches;
    if (rc == VFMM_OK) rc = read_status(w);
    return rc;
}

extern "C" int vfmm_graph_create(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_dev, int32_t nrhs,
                                 double* u_dev, double* ux_dev, double* uy_dev, void* workspace_dev,
                                 size_t workspace_bytes, void* stream, vfmm_graph** out) {
    if (!out) return fail(VFMM_ERR_INVALID_ARG, "null out");
    *out = nullptr;
    cudaStream_t st = (cudaStream_t)stream;
    if (st == nullptr) return fail(VFMM_ERR_INVALID_ARG, "graph capture needs a non-default stream");
    VFMM_CHECK(vfmm_volume_potential(tree, ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, workspace_dev, workspace_bytes,
                                     stream));
    VFMM_CUDA(cudaStreamSynchronize(st));
    vfmm_graph* g = new vfmm_graph();
    cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) {
        delete g;
        return cuda_fail(e, "cudaStreamBeginCapture");
    }
    int rc = vfmm_volume_potential(tree, ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, workspace_dev, workspace_bytes,
                                   stream);
    e = cudaStreamEndCapture(st, &g->graph);
    if (rc != VFMM_OK || e != cudaSuccess) {
        if (g->graph) cudaGraphDestroy(g->graph);
        delete g;
        return rc != VFMM_OK ? rc : cuda_fail(e, "cudaStreamEndCapture");
    }
    // kernels keep the priority of the stream they were captured on
    e = cudaGraphInstantiate(&g->exec, g->graph, cudaGraphInstantiateFlagUseNodePriority);
    if (e != cudaSuccess) {
        cudaGraphDestroy(g->graph);
        delete g;
        return cuda_fail(e, "cudaGraphInstantiate");
    }
    *out = g;
    return VFMM_OK;
}

extern "C" int vfmm_graph_launch(const vfmm_graph* g, void* stream) {
    if (!g) return fail(VFMM_ERR_INVALID_ARG, "null graph");
    VFMM_CUDA(cudaGraphLaunch(g->exec, (cudaStream_t)stream));
    return VFMM_OK;
}

extern "C" int vfmm_graph_destroy(vfmm_graph* g) {
    if (!g) return VFMM_OK;
    if (g->exec) cudaGraphExecDestroy(g->exec);
    if (g->graph) cudaGraphDestroy(g->graph);
    delete g;
    return VFMM_OK;
}

// ---------------------------------------------------------------- schedule autotuner
extern "C" int vfmm_tune(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_dev, int32_t nrhs, double* u_dev,
                         double* ux_dev, double* uy_dev, void* workspace_dev, size_t workspace_bytes, void* stream,
                         int32_t* splits) {
    VFMM_CHECK(check_solve_args(tree, ops, nrhs));
    if (!f_dev || !u_dev || !ux_dev || !uy_dev || !workspace_dev) return fail(VFMM_ERR_INVALID_ARG, "null buffer");
    cudaStream_t st = (cudaStream_t)stream;
    Workspace w;
    size_t need = 0;
    VFMM_CHECK(layout(tree->t, *ops, nrhs, false, &w, (char*)workspace_dev, &need));
    if (workspace_bytes < need) return fail(VFMM_ERR_WORKSPACE, "workspace too small");
    if (splits)
        for (int i = 0; i < 4; ++i) splits[i] = 1;
    if (ops->precision != VFMM_MIXED) return VFMM_OK;
    const DeviceTree& T = tree->t;
    const MixedOps* mo = (const MixedOps*)ops->mixed;
    // one solve leaves every contraction's operands in the workspace
    VFMM_CHECK(reset_status(w, st));
    VFMM_CHECK(solve_all(T, *ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, w, st));
    VFMM_CUDA(cudaStreamSynchronize(st));
    PlanSet* PS = const_cast<PlanSet*>(w.ps);
    const size_t R = (size_t)PS->R;
    struct Job {
        SplitPlan* P;
        const void* a;
        const void* map;
        int Kp, Rp;
        float2* out;
        size_t rows;
        int slices;
    } jobs[4] = {{&PS->entries, w.mix.fsl, mo->tsl, mo->Kp, mo->Rp, w.mix.out, T.n_leaves * R, mo->slices[kCtrNear]},
                 {&PS->m2l, w.mix.msl, mo->m2l_sl, mo->Kx, mo->Rx, w.mix.m2l_out, T.n_boxes * R, mo->slices[kCtrM2L]},
                 {&PS->s2l, w.mix.fsl, mo->s2l_sl, mo->Kp, mo->Rx, w.mix.s2l_out, T.n_boxes * R, mo->slices[kCtrS2L]},
                 {&PS->far, w.mix.aprep, mo->far_sl, mo->Kx, mo->Rp, w.mix.far_out, T.n_leaves * R,
                  mo->slices[kCtrFar]}};
    cudaEvent_t e0, e1;
    VFMM_CUDA(cudaEventCreate(&e0));
    VFMM_CUDA(cudaEventCreate(&e1));
    int rc = VFMM_OK;
    const bool cls = near_by_classes(ops->k);
    int32_t& near_ctas = cls ? PS->near.ctas : PS->entries.ctas;
    auto use_form = [](SplitPlan* P, bool entry) {
        if (P->entry == entry || !P->alt) return;
        SplitPlan* alt = P->alt;
        P->alt = nullptr;
        std::swap(*P, *alt);
        P->alt = alt;
    };
    // the schedule as it stands, to go back to where its step is the faster one
    struct Form {
        bool entry;
        int32_t split, ctas;
    } forms0[4];
    for (int j = 0; j < 4; ++j) forms0[j] = Form{jobs[j].P->entry, jobs[j].P->split, jobs[j].P->ctas};
    const int near0 = near_ctas, pass0 = PS->pass_ctas;
    // fastest of a few forked solves (the step as vfmm_volume_potential and its graphs run it)
    auto time_step = [&]() -> float {
        Workspace wf = w;
        wf.fork = true;
        float best = 1e30f;
        for (int rep = 0; rep < 6 && rc == VFMM_OK; ++rep) {
            cudaEventRecord(e0, st);
            rc = solve_all(T, *ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, wf, st);
            cudaEventRecord(e1, st);
            if (rc != VFMM_OK) break;
            cudaError_t e = cudaEventSynchronize(e1);
            float ms = 0.0f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e != cudaSuccess) rc = cuda_fail(e, "timing a forked solve");
            if (rep > 0) best = std::min(best, ms);  // the first run warms up
        }
        return best;
    };
    // fastest split-K factor of one form of a contraction (its current factor when it cannot split)
    auto time_form = [&](const Job& jb, SplitPlan* P, float2* part, int* best_sp, float* best_ms) {
        const double avg_units = (double)P->entries * (jb.Kp / kKBlock) / std::max(1, P->n_groups);
        const int max_sp = P->may_split ? kMaxSplit : 1;
        const int keep = P->split;
        *best_sp = keep;
        *best_ms = -1.0f;
        for (int sp = P->may_split ? 1 : keep; sp <= std::max(max_sp, keep) && rc == VFMM_OK; sp *= 2) {
            if (P->may_split && sp > std::max(1.0, avg_units)) break;
            P->split = sp;
            float total = 1e30f;  // the fastest of a few runs
            for (int rep = 0; rep < 4 && rc == VFMM_OK; ++rep) {
                cudaEventRecord(e0, st);
                rc = split_gemm(*P, jb.a, jb.map, jb.Kp, jb.Rp, jb.out, w.mix.err, part, jb.rows, jb.slices, st);
                cudaEventRecord(e1, st);
                if (rc != VFMM_OK) break;
                cudaError_t e = cudaEventSynchronize(e1);
                float ms = 0.0f;
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                if (e != cudaSuccess) rc = cuda_fail(e, "timing a split contraction");
                if (rep > 0) total = std::min(total, ms);  // the first run warms up
            }
            if (rc == VFMM_OK && (*best_ms < 0.0f || total < *best_ms)) {
                *best_ms = total;
                *best_sp = sp;
            }
            if (!P->may_split) break;
        }
        P->split = *best_sp;
    };
    // persistent CTAs (one per SM, each walking several work items) against one CTA per item, for a
    // contraction with more items than SMs; the faster is kept
    auto time_ctas = [&](const Job& jb, SplitPlan* P, float2* part) {
        const int nchunks = jb.Rp / table_rows_per_tile(jb.Rp);
        const long long items = (long long)P->n_groups * (P->entry ? 1 : P->split) * nchunks;
        const int sms = sm_count();
        if (items <= sms) return;
        float best = -1.0f;
        int best_c = P->ctas;
        for (int c : {0, sms}) {
            P->ctas = c;
            float total = 1e30f;  // the fastest of a few runs
            for (int rep = 0; rep < 4 && rc == VFMM_OK; ++rep) {
                cudaEventRecord(e0, st);
                rc = split_gemm(*P, jb.a, jb.map, jb.Kp, jb.Rp, jb.out, w.mix.err, part, jb.rows, jb.slices, st);
                cudaEventRecord(e1, st);
                if (rc != VFMM_OK) break;
                cudaError_t e = cudaEventSynchronize(e1);
                float ms = 0.0f;
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                if (e != cudaSuccess) rc = cuda_fail(e, "timing a split contraction");
                if (rep > 0) total = std::min(total, ms);
            }
            if (rc == VFMM_OK && (best < 0.0f || total < best)) {
                best = total;
                best_c = c;
            }
        }
        P->ctas = best_c;
    };
    for (int j = 0; j < 4 && rc == VFMM_OK; ++j) {
        Job& jb = jobs[j];
        if (jb.P->n_groups == 0 || (!jb.P->may_split && !jb.P->alt)) continue;
        float2* part = j == 0 ? w.mix.part_side : j == 2 ? w.mix.part_s2l : w.mix.part;
        int sp = 1;
        float ms = -1.0f;
        time_form(jb, jb.P, part, &sp, &ms);
        if (rc == VFMM_OK && jb.P->alt && jb.P->alt->n_groups > 0) {
            // the other form (grouped or entry-major): kept if faster
            int sp_alt = 1;
            float ms_alt = -1.0f;
            time_form(jb, jb.P->alt, part, &sp_alt, &ms_alt);
            if (rc == VFMM_OK && ms_alt >= 0.0f && ms_alt < ms) use_form(jb.P, !jb.P->entry);
        }
        if (rc == VFMM_OK) time_ctas(jb, jb.P, part);
    }
    // Co-scheduling of the whole step: in a forked solve the near field (low-priority stream) and the
    // main chain share the SMs, and a near-field CTA leaves no room for anything else on its SM.
    // Timed on the forked solve itself: one near-field CTA per item, persistent ones on every SM, or on
    // 7/8 ... 4/8 of them with the cooperative tree passes capped to the SMs they leave free (they can
    // start only when their whole grid fits); the fastest is kept. A near field with fewer items than
    // half the SMs leaves the chain room as it is.
    const int sms = sm_count();
    const bool wide = cls ? 8 * PS->near.n_groups * mo->near.nch > sms : PS->entries.ctas > 0;
    float best = 1e30f;
    if (rc == VFMM_OK && wide && T.depth >= 3) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, upward_pass_kernel, kPassThreads, pass_smem_bytes(ops->p + 1));
        int best_near = near0, best_pass = pass0;
        const int fracs[6] = {0, 8, 7, 6, 5, 4};  // eighths of the SMs; 0: uncapped
        for (int c = 0; c < 6 && rc == VFMM_OK; ++c) {
            const int ncta = fracs[c] == 0 ? 0 : std::max(1, sms * fracs[c] / 8);
            near_ctas = ncta;
            PS->pass_ctas = fracs[c] == 0 || fracs[c] == 8 ? 0 : std::max(1, per_sm * (sms - ncta));
            const float ms = time_step();
            if (rc == VFMM_OK && ms < best) {
                best = ms;
                best_near = near_ctas;
                best_pass = PS->pass_ctas;
            }
        }
        near_ctas = best_near;
        PS->pass_ctas = best_pass;
    } else if (rc == VFMM_OK) {
        best = time_step();
    }
    // The contractions were timed alone; beside each other their fastest forms need not make the fastest
    // step (1,378 leaves: 353 us as planned, 365 with the forms picked alone)
    if (rc == VFMM_OK) {
        const int near1 = near_ctas, pass1 = PS->pass_ctas;
        Form forms1[4];
        for (int j = 0; j < 4; ++j) forms1[j] = Form{jobs[j].P->entry, jobs[j].P->split, jobs[j].P->ctas};
        auto set = [&](const Form* f, int nc, int pc) {
            for (int j = 0; j < 4; ++j) {
                use_form(jobs[j].P, f[j].entry);
                jobs[j].P->split = f[j].split;
                jobs[j].P->ctas = f[j].ctas;
            }
            near_ctas = nc;
            PS->pass_ctas = pc;
        };
        set(forms0, near0, pass0);
        const float ms = time_step();
        if (rc == VFMM_OK && ms > best) set(forms1, near1, pass1);
    }
    if (splits)
        for (int j = 0; j < 4; ++j) splits[j] = jobs[j].P->split;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    VFMM_CHECK(rc);
    // leave the outputs of an ordinary solve with the chosen schedule
    VFMM_CHECK(solve_all(T, *ops, f_dev, nrhs, u_dev, ux_dev, uy_dev, w, st));
    VFMM_CUDA(cudaStreamSynchronize(st));
    return read_status(w);
}

extern "C" int vfmm_schedule_get(const vfmm_tree* tree, int32_t nrhs, int32_t* near_ctas, int32_t* pass_ctas) {
    if (!tree || !near_ctas || !pass_ctas || nrhs < 1) return fail(VFMM_ERR_INVALID_ARG, "bad schedule query");
    const PlanSet* PS = nullptr;
    VFMM_CHECK(plans_for(tree->t, nrhs, &PS));
    *near_ctas = near_by_classes(tree->t.k) ? PS->near.ctas : PS->entries.ctas;
    *pass_ctas = PS->pass_ctas;
    return VFMM_OK;
}

extern "C" int vfmm_schedule_set(vfmm_tree* tree, int32_t nrhs, int32_t near_ctas, int32_t pass_ctas) {
    if (!tree || nrhs < 1 || near_ctas < 0 || pass_ctas < 0) return fail(VFMM_ERR_INVALID_ARG, "bad schedule");
    const PlanSet* PS = nullptr;
    VFMM_CHECK(plans_for(tree->t, nrhs, &PS));
    PlanSet* ps = const_cast<PlanSet*>(PS);
    (near_by_classes(tree->t.k) ? ps->near.ctas : ps->entries.ctas) = near_ctas;
    ps->pass_ctas = pass_ctas;
    return VFMM_OK;
}
