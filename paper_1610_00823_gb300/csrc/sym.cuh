// Reflections of the square in the FP64 form's tables.
//
// The kernels log|x - y| and its gradient, the leaf nodes and the expansions all map onto themselves
// under the reflections mx: x -> -x and my: y -> -y (the group G = {1, mx, my, mx my}, numbered
// s = 0..3, bit 0 for mx, bit 1 for my). So every operator T_D of a list configuration D (source box at
// offset D from the target box) satisfies T_{sD}(s t, s y) = c(s) T_D(t, y), c(s) = -1 for u_x under mx
// and u_y under my. Configurations fall into orbits {sR} of a representative R with non-negative
// components, and values split into four classes chi = (a, b), chi(mx) = (-1)^a, chi(my) = (-1)^b:
//   out^chi(t) = sum_s chi(s) c(s) out(s t)                 for t in a quadrant of the target nodes
//              = sum_R sum_y A^chi_R(t, y) g^chi_R(y),      g^chi_R(y) = sum_s chi(s) f_{sR}(s y),
//   out(s t)   = c(s) sum_chi chi(s) out^chi(t)             (the 1/4 of this sum sits in A)
// One instance (target, R) takes the place of up to four list entries, with a quarter of one entry's
// rows in each class; where R lies on an axis, g is even or odd under the reflection that fixes R and
// half (both axes: a quarter) of its columns are enough. A box with all its neighbours does 1/4 of the
// products of the plain tables (1/2.7 for M2L, whose offsets are not all mirrored), an instance with
// one entry never more.
//
// Rows and columns are leaf nodes (fields u, u_x, u_y; f) or expansion parts (Re, Im of coefficient n,
// part 2n, 2n + 1), which the reflections map to (-1)^n conj (mx) and conj (my): one sign per part.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ops.cuh"
#include "vfmm_internal.cuh"

namespace vfmm {

// Orbits of the four lists; row = first row of the list + orbit numbers them in a 32-bit mask.
constexpr int kNearOrb = 10, kVOrb = 12, kFarOrb = 5, kSymMaxOrb = 12;
constexpr int kSymRows = kNearOrb + kVOrb + 2 * kFarOrb;
static_assert(kSymRows == 32, "one bit per (list, orbit)");
__host__ __device__ constexpr int sym_first_row(int q) {
    return q == 0 ? 0 : (q == 1 ? kNearOrb : (q == 2 ? kNearOrb + kVOrb : kNearOrb + kVOrb + kFarOrb));
}
__host__ __device__ constexpr int sym_orbits(int q) { return q == 0 ? kNearOrb : (q == 1 ? kVOrb : kFarOrb); }

// Offset of configuration cfg of list q, in the units of its pattern.
__host__ __device__ inline void sym_offset(int q, int cfg, int* dx, int* dy) {
    if (q == VFMM_LIST_V) return v_offset(cfg, dx, dy);
    if (q != VFMM_LIST_U) return far_pattern(cfg, dx, dy);
    if (cfg >= 9) return near_pattern(cfg >= 21 ? cfg - 21 : cfg - 9, dx, dy);
    *dx = cfg % 3 - 1;
    *dy = cfg / 3 - 1;
}
// Orbit of configuration cfg, and the reflections s (bit mask) with sR = its offset.
__host__ __device__ inline int sym_orbit(int q, int cfg, int* slots) {
    int dx, dy;
    sym_offset(q, cfg, &dx, &dy);
    const int mx = dx < 0 ? 0xA : (dx > 0 ? 0x5 : 0xF), my = dy < 0 ? 0xC : (dy > 0 ? 0x3 : 0xF);
    *slots = mx & my;
    const int ax = dx < 0 ? -dx : dx, ay = dy < 0 ? -dy : dy;
    if (q == VFMM_LIST_V) {  // (2,0) (3,0) (0,2) (0,3) (1,2) (1,3) (2,1..3) (3,1..3)
        if (ay == 0) return ax - 2;
        if (ax == 0) return ay;
        return ax == 1 ? 2 + ay : 3 * ax + ay - 1;
    }
    if (q != VFMM_LIST_U) return ax == 5 ? (ay == 5 ? 4 : ay - 1) : ax;  // (5,1) (1,5) (5,3) (3,5) (5,5)
    if (cfg < 9) return ax + 2 * ay;                                     // (0,0) (1,0) (0,1) (1,1)
    return (cfg < 21 ? 4 : 7) + (ax == 1 ? 1 : (ay == 1 ? 0 : 2));       // (3,1) (1,3) (3,3)
}

// One operator in symmetrised form: A[orbit][class] is [K][M], columns (the contraction) by rows.
struct SymOp {
    int norb = 0, k = 0, P = 0;
    bool node_rows = false, node_cols = false;  // leaf nodes, else expansion parts
    double* A = nullptr;
    int M[4] = {}, roff[4] = {};         // rows of a class and its first one in an output row (nodes)
    int seg[13] = {};                    // node rows: first row of (class, field) at 3 * class + field
    int K[kSymMaxOrb][4] = {};
    int64_t off[kSymMaxOrb][4] = {};
    uint8_t fx[kSymMaxOrb] = {}, fy[kSymMaxOrb] = {};  // R on the y axis (mx fixes it), on the x axis
};

// Nodes of one axis with parity par under its reflection: the lower half, the middle one if even.
__host__ __device__ inline int sym_half(int k, int par) { return par ? k / 2 : (k + 1) / 2; }
// Parities of field q (u, u_x, u_y) in class c.
__host__ __device__ inline int sym_pa(int c, int q) { return (c & 1) ^ (q == 1); }
__host__ __device__ inline int sym_pb(int c, int q) { return (c >> 1) ^ (q == 2); }
// Part r of class c (the parts that the reflections multiply by chi): coefficients of one parity.
__host__ __device__ inline int sym_part(int c, int r) {
    const int a = c & 1, b = c >> 1;
    return 2 * ((a ^ b) + 2 * r) + b;
}
__host__ __device__ inline int sym_parts(int c, int P) { return (P - ((c & 1) ^ (c >> 1)) + 1) / 2; }
// Sign (0 / 1: -1) that reflection s gives a part.
__host__ __device__ inline int sym_part_sign(int part, int s) {
    const int n = part >> 1, im = part & 1;
    return ((s & 1) & ((n & 1) ^ im)) ^ ((s >> 1) & im);
}

struct SymTables {
    SymOp near, s2m, m2l, s2l, l2t, m2t;
};
// m2l [40][2(p+1)][2(p+1)] and s2l [20][2(p+1)][kk]: the real forms, rows 2l (Re), 2l + 1 (Im) of output
// coefficient l (device). The tables are complete when st is.
int sym_prepare(::vfmm_ops* o, const double* m2l, const double* s2l, cudaStream_t st);
void sym_free(::vfmm_ops* o);
// Operator alone, its table the caller's to free: the near field; L2T (orbit 0, the leaf itself) and the five
// orbits of M2T from the plain tables F [21][3 k^2][2(p+1)] (L2T, then every W configuration; device).
int sym_far_op(const ::vfmm_ops* o, const double* F, SymOp* op, cudaStream_t st);
int sym_near_op(const ::vfmm_ops* o, SymOp* op, cudaStream_t st);

// Instances of the four lists (built with the tree).
int build_instances(DeviceTree* T, cudaStream_t st);

// out[id * stride + row] = scale * sum of A g for every instance of list q, or (q < 0) for every leaf
// with itself as source; src rows are indexed by the instances' sources, or by src_map[leaf].
struct SymRun {
    int q = -1;
    const double* src = nullptr;
    int64_t src_stride = 0;
    const int32_t* src_map = nullptr;
    double* out = nullptr;
    int64_t out_stride = 0;
    const int32_t* out_map = nullptr;   // q < 0: output row of a leaf (null: the leaf)
    const int32_t* level = nullptr;     // q < 0: scale h^2 of box out_map[leaf] (null: 1)
    double width = 0.0;
};
int sym_gemm(const DeviceTree& T, const SymOp& op, const SymRun& r, cudaStream_t st);

}  // namespace vfmm
