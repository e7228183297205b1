// The computed potential at arbitrary points from the stored expansions (Section 5.3: the FMM's
// multipole and local expansions are kept so that a new target costs O(p) for its far field
// instead of a new FMM; Section 3.1 for the split into near and far field).
//
// For a point t of leaf b (located as the leaf interpolant locates it):
//   V f~(t) = -(1/2 pi) Re [ sum_l b~_l ((t - z_b)/h)^l + sum over W(b) of the multipole at t ]
//           + sum over U(b) of -(1/2 pi) int_{B_s} log|t - y| f~_s(y) dy,
// with the gradient from the differentiated expansions and kernels (Section 3.2). The far part
// reads the expansions a solve left in its workspace.
//
// Near part: on a leaf (unit box) f~ is a polynomial, and so is a P with Laplace P = f~. Green's second
// identity and the Cauchy-Pompeiu formula then leave integrals over the four edges only,
//   int log|t - y| f~ dy  = sum_e int (log|t - y| dP/dn - P d log|t - y|/dn) ds  [+ 2 pi P(t) inside],
//   int f~ / (t - y) dy   = (i/2) sum_e int F/(y - t) dy  [+ pi F(t) inside],  F = 2 (P_x - i P_y),
// and with the traces as Legendre series on an edge (x in [-1, 1], z the point in its coordinate)
//   int P_n(x) / (x - z) dx = -2 Q_n(z),   int P_n(x) log|x - z| dx = 2 Re (Q_{n+1} - Q_{n-1})/(2n + 1),
// Q_n the Legendre functions of the second kind: closed forms at any distance from the edge, where a
// quadrature needs ever more nodes. Q_n comes from its three-term recurrence, upwards where z is near
// the edge, else downwards from a start high enough (Miller) and scaled to Q_0 = log((z+1)/(z-1))/2.
//
// P is the polynomial of total degree 2k of least weighted norm (prepared per k on the host, per
// reflection class: tensor Legendre coefficients c_mn, m + n <= 2k, from the k x k leaf values).
//
// What bounds it: FP64 (about 0.4 MFMA per point, most of it leaf values to coefficients; one CTA per
// point, two per SM). 1000 points of a 1,378-leaf tree, k = 16: 247 ms with tanh-sinh quadrature of the
// neighbours (up to 8 x 201^2 nodes of k^2 terms each) -> 1.15 ms, error against 64-bit
// sums unchanged (1.5e-15).
#include <algorithm>
#include <cmath>
#include <vector>

#include "ops.cuh"
#include "sym.cuh"
#include "vfmm_internal.cuh"

namespace vfmm {

constexpr int kOffThreads = 256;
constexpr int kOffMaxU = 13;      // a leaf, and at most 12 neighbours
constexpr int kOffMaxN = 33;      // 2k + 1 Legendre coefficients along an edge
constexpr int kOffTasks = 4 * kOffMaxU;
constexpr int kOffSteps = 288;    // recurrence constants: steps above kOffMaxN that Miller needs for
constexpr float kOffForward = 1.08f;  // rho >= kOffForward: 37 / (2 log 1.08) = 241

// Rows (m, n), m = a + 2i, n = b + 2j, m + n <= 2k of class (a, b), i outer.
__host__ __device__ inline int off_ni(int k, int c) { return k + 1 - ((c & 1) + (c >> 1) + 1) / 2; }
__host__ __device__ inline int off_rows(int k, int c) { return off_ni(k, c) * (off_ni(k, c) + 1) / 2; }
__host__ __device__ inline int off_first(int k, int c) {
    int r = 0;
    for (int d = 0; d < c; ++d) r += off_rows(k, d);
    return r;
}
__host__ __device__ inline int off_row0(int k, int c, int i) { return off_first(k, c) + i * off_ni(k, c) - i * (i - 1) / 2; }
// First value of class c in a leaf's symmetrised values (a quadrant of nodes per class, k^2 in all).
__host__ __device__ inline int off_val(int k, int c) {
    int r = 0;
    for (int d = 0; d < c; ++d) r += sym_half(k, d & 1) * sym_half(k, d >> 1);
    return r;
}

struct alignas(16) OffStep {
    double x, y, z, w;
};
struct OffTables {
    double* G = nullptr;   // per class [value][row]: coefficients of P from the symmetrised values
    int64_t g_off[4] = {};
    OffStep* C = nullptr;  // [kOffSteps]: (2n+1)/n, (n+1)/n (downwards), (2n+1)/(n+1), n/(n+1) (upwards)
};

// ---------------------------------------------------------------- host: values -> P
// Legendre coefficients of the k Lagrange polynomials of the nodes xi: A[j][i].
static void legendre_of_nodes(int k, const std::vector<double>& xi, std::vector<double>& A) {
    std::vector<double> V((size_t)k * k), inv((size_t)k * k, 0.0);
    // V[i][j] = P_j(xi_i); A = V^-1 by Gauss-Jordan with pivoting, in extended precision
    std::vector<long double> M((size_t)k * 2 * k, 0.0L);
    for (int i = 0; i < k; ++i) {
        long double p0 = 1.0L, p1 = xi[i];
        for (int j = 0; j < k; ++j) {
            M[(size_t)i * 2 * k + j] = p0;
            const long double p2 = ((2 * j + 3) * (long double)xi[i] * p1 - (j + 1) * p0) / (j + 2);
            p0 = p1;
            p1 = p2;
        }
        M[(size_t)i * 2 * k + k + i] = 1.0L;
    }
    for (int c = 0; c < k; ++c) {
        int pv = c;
        for (int r = c + 1; r < k; ++r)
            if (std::fabs(M[(size_t)r * 2 * k + c]) > std::fabs(M[(size_t)pv * 2 * k + c])) pv = r;
        for (int q = 0; q < 2 * k; ++q) std::swap(M[(size_t)c * 2 * k + q], M[(size_t)pv * 2 * k + q]);
        const long double d = 1.0L / M[(size_t)c * 2 * k + c];
        for (int q = 0; q < 2 * k; ++q) M[(size_t)c * 2 * k + q] *= d;
        for (int r = 0; r < k; ++r) {
            const long double f = M[(size_t)r * 2 * k + c];
            if (r == c || f == 0.0L) continue;
            for (int q = 0; q < 2 * k; ++q) M[(size_t)r * 2 * k + q] -= f * M[(size_t)c * 2 * k + q];
        }
    }
    A.resize((size_t)k * k);
    for (int j = 0; j < k; ++j)
        for (int i = 0; i < k; ++i) A[(size_t)j * k + i] = (double)M[(size_t)j * 2 * k + k + i];
}

// G of one class, [value][row]. Unknowns c_mn of P, equations: Legendre coefficients of Laplace P = those
// of f~ (j + l <= 2k - 2; zero beyond its degrees), least norm of (1 + m(m+1) + n(n+1)) c_mn: Householder QR
// of the transposed weighted system and one refinement step with the residual in extended precision.
static void class_table(int k, int c, const std::vector<double>& A, double* G) {
    const int a = c & 1, b = c >> 1, nu = off_rows(k, c), ni = off_ni(k, c), base = off_first(k, c);
    std::vector<int> eq_j, eq_l;
    for (int j = a; j <= 2 * k - 2; j += 2)
        for (int l = b; j + l <= 2 * k - 2; l += 2) {
            eq_j.push_back(j);
            eq_l.push_back(l);
        }
    const int ne = (int)eq_j.size();
    auto row = [&](int m, int n) { return off_row0(k, c, m >> 1) - base + (n >> 1); };
    std::vector<double> W(nu);
    for (int i = 0; i < ni; ++i)
        for (int j = 0; i + j < ni; ++j) {
            const int m = a + 2 * i, n = b + 2 * j;
            W[row(m, n)] = 1.0 + m * (m + 1) + n * (n + 1);
        }
    // d2(j, m): coefficient j of the second derivative of Legendre polynomial m in unit-box coordinates
    auto d2 = [](int j, int m) { return 4.0 * (j + 0.5) * (m * (m + 1.0) - j * (j + 1.0)); };
    // columns = equations, rows = unknowns (weighted): H = Q R
    std::vector<double> H((size_t)ne * nu, 0.0), M;
    for (int e = 0; e < ne; ++e) {
        for (int m = eq_j[e] + 2; m + eq_l[e] <= 2 * k; m += 2) H[(size_t)e * nu + row(m, eq_l[e])] += d2(eq_j[e], m);
        for (int n = eq_l[e] + 2; n + eq_j[e] <= 2 * k; n += 2) H[(size_t)e * nu + row(eq_j[e], n)] += d2(eq_l[e], n);
        for (int u = 0; u < nu; ++u) H[(size_t)e * nu + u] /= W[u];
    }
    M = H;
    std::vector<double> tau(ne);
    for (int e = 0; e < ne; ++e) {
        double* v = H.data() + (size_t)e * nu;
        double nrm = 0.0;
        for (int u = e; u < nu; ++u) nrm += v[u] * v[u];
        nrm = std::sqrt(nrm);
        const double alpha = v[e] > 0.0 ? -nrm : nrm;
        const double v0 = v[e] - alpha;
        tau[e] = -v0 / alpha;
        for (int u = e + 1; u < nu; ++u) v[u] /= v0;
        v[e] = alpha;  // R's diagonal; the reflector's leading 1 is implied
        for (int q = e + 1; q < ne; ++q) {
            double* x = H.data() + (size_t)q * nu;
            double s = x[e];
            for (int u = e + 1; u < nu; ++u) s += v[u] * x[u];
            s *= tau[e];
            x[e] -= s;
            for (int u = e + 1; u < nu; ++u) x[u] -= s * v[u];
        }
    }
    // x = Q R^-T s
    auto solve = [&](std::vector<double> y, std::vector<double>& x) {
        for (int e = 0; e < ne; ++e) {
            double s = y[e];
            for (int q = 0; q < e; ++q) s -= H[(size_t)e * nu + q] * y[q];  // R[q][e]
            y[e] = s / H[(size_t)e * nu + e];
        }
        x.assign(nu, 0.0);
        std::copy(y.begin(), y.end(), x.begin());
        for (int e = ne - 1; e >= 0; --e) {
            const double* v = H.data() + (size_t)e * nu;
            double s = x[e];
            for (int u = e + 1; u < nu; ++u) s += v[u] * x[u];
            s *= tau[e];
            x[e] -= s;
            for (int u = e + 1; u < nu; ++u) x[u] -= s * v[u];
        }
    };
    const int nx = sym_half(k, a), ny = sym_half(k, b);
    std::vector<double> s(ne), r(ne), x, dx;
    for (int jy = 0; jy < ny; ++jy)
        for (int ix = 0; ix < nx; ++ix) {
            const double w = (2 * ix == k - 1 ? 0.5 : 1.0) * (2 * jy == k - 1 ? 0.5 : 1.0);
            for (int e = 0; e < ne; ++e)
                s[e] = eq_j[e] < k && eq_l[e] < k ? w * A[(size_t)eq_j[e] * k + ix] * A[(size_t)eq_l[e] * k + jy] : 0.0;
            solve(s, x);
            for (int e = 0; e < ne; ++e) {
                long double t = s[e];
                for (int u = 0; u < nu; ++u)
                    if (M[(size_t)e * nu + u] != 0.0) t -= (long double)M[(size_t)e * nu + u] * x[u];
                r[e] = (double)t;
            }
            solve(r, dx);
            for (int u = 0; u < nu; ++u) G[((size_t)jy * nx + ix) * nu + u] = (x[u] + dx[u]) / W[u];
        }
}

int offnode_prepare(vfmm_ops* o, cudaStream_t st) {
    const int k = o->k;
    const double pi = 3.14159265358979323846;
    std::vector<double> xi(k), A, G;
    for (int i = 0; i < k; ++i) xi[i] = -std::cos(pi * (2.0 * i + 1.0) / (2.0 * k));
    legendre_of_nodes(k, xi, A);
    OffTables* t = new OffTables();
    o->off = t;
    for (int c = 0; c < 4; ++c) {
        t->g_off[c] = (int64_t)G.size();
        const size_t n = (size_t)sym_half(k, c & 1) * sym_half(k, c >> 1) * off_rows(k, c);
        G.resize(G.size() + n);
        class_table(k, c, A, G.data() + t->g_off[c]);
    }
    std::vector<OffStep> C(kOffSteps);
    for (int n = 0; n < kOffSteps; ++n)
        C[n] = OffStep{n ? (2.0 * n + 1.0) / n : 0.0, n ? (n + 1.0) / n : 0.0, (2.0 * n + 1.0) / (n + 1.0),
                            n / (n + 1.0)};
    VFMM_CUDA(cudaMalloc(&t->G, G.size() * sizeof(double)));
    VFMM_CUDA(cudaMalloc(&t->C, C.size() * sizeof(OffStep)));
    VFMM_CUDA(cudaMemcpyAsync(t->G, G.data(), G.size() * sizeof(double), cudaMemcpyHostToDevice, st));
    VFMM_CUDA(cudaMemcpyAsync(t->C, C.data(), C.size() * sizeof(OffStep), cudaMemcpyHostToDevice, st));
    VFMM_CUDA(cudaStreamSynchronize(st));
    return VFMM_OK;
}

void offnode_free(vfmm_ops* o) {
    OffTables* t = (OffTables*)o->off;
    if (!t) return;
    if (t->G) cudaFree(t->G);
    if (t->C) cudaFree(t->C);
    delete t;
    o->off = nullptr;
}

// ---------------------------------------------------------------- device
struct OffArgs {
    int k, P, depth, R;
    int64_t n;
    double lox, loy, width;
    const int32_t *child0, *level, *ix, *iy, *leaf_of_box;
    const int32_t *uptr, *uidx, *wptr, *widx, *wcfg;
    const double* f;     // [n_leaves][k*k] leaf values of right-hand side 0
    const double* Mexp;  // [n_boxes][R][2P] scaled multipoles of the solve
    const double* Lexp;  // [n_boxes][R][2P] scaled locals of the solve
    const double *x, *y;
    double *u, *ux, *uy;
    OffTables t;
};

// A U leaf as seen from the point, unit-box coordinates: distances to its sides (left, right, bottom,
// top), positive inwards. On a side (all >= 0, some 0) the point counts as inside, by an amount that the
// arithmetic of the edges cannot see. Distances below 2^-498 (1.2e-150) of the width count as 0 (kOffOnEdge): of
// a point that near to a corner from outside, the sum of the squares would underflow and its logarithm be
// infinite. Both lines are drawn by exponents: a comparison in FP64 takes a warp as long as an addition.
constexpr int kOffOnEdge = 1023 - 498;
constexpr int kOffCorner = 1023 - 10;  // within 2^-10 of the leaf's width; both edges' recurrences then run upwards
// -d where `on` (bit 0), on the bits.
__device__ __forceinline__ double off_flip(double d, int on) {
    return __hiloint2double(__double2hiint(d) ^ (on << 31), __double2loint(d));
}
__device__ __forceinline__ int off_exp(double d) { return (__double2hiint(d) >> 20) & 0x7FF; }
struct OffLeaf {
    double d[4];
    double h;
    int leaf, inside;
    int corner;  // c where edge c starts, if the point is next to it, or -1
};

// sum over this thread's values v of the table columns, for NU leaves: cf[row][u] = sum_v G[v][row] fs[v][u]
template <int NU>
__device__ __forceinline__ void off_coeffs(const double* __restrict__ G, int K, int ld, const double* fs, double* out) {
    double acc[NU];
#pragma unroll
    for (int u = 0; u < NU; ++u) acc[u] = 0.0;
#pragma unroll 4
    for (int v = 0; v < K; ++v) {
        const double g = __ldg(G + (size_t)v * ld);
#pragma unroll
        for (int u = 0; u < NU; ++u) acc[u] = fma(g, fs[v * kOffMaxU + u], acc[u]);
    }
#pragma unroll
    for (int u = 0; u < NU; ++u) out[u] = acc[u];
}
template <int NU>
__device__ __forceinline__ void off_coeffs_n(int nu, const double* G, int K, int ld, const double* fs, double* out) {
    if (nu == NU) off_coeffs<NU>(G, K, ld, fs, out);
    else if constexpr (NU > 1) off_coeffs_n<NU - 1>(nu, G, K, ld, fs, out);
}

// Q_0 = log((z + 1)/(z - 1))/2 of an edge, z the point (w1, w2, zi as in edge_terms); l1 = log|z - 1|, dl and ang
// twice its parts.
struct EdgeLog {
    double l1, dl, ang;
};
__device__ __forceinline__ EdgeLog edge_log(double w1, double w2, double zi) {
    const double zr = 0.5 * (w2 - w1), n1 = w1 * w1 + zi * zi, n2 = w2 * w2 + zi * zi;
    EdgeLog r;
    r.l1 = 0.5 * log(n1);
    r.dl = zr >= 0.0 ? 0.5 * log1p(4.0 * zr / n1) : -0.5 * log1p(-4.0 * zr / n2);  // log|z+1| - log|z-1|
    r.ang = atan2(-2.0 * zi, zi * zi - w1 * w2);                                   // arg(z+1) - arg(z-1)
    return r;
}

// (V, Re Phi', Im Phi') of one edge of a unit box at the point: w1, w2 the distances along the edge from
// the point to its end and from its start (edge coordinate, length 2), zi the one across (positive inside);
// p, g, T: Legendre coefficients of P, its outward and its tangential derivative, stride kOffTasks; logs is
// log(h / 2); (tr, ti) the conjugate of the edge's direction.
__device__ __forceinline__ void edge_terms(double w1, double w2, double zi, const double* p, const double* g,
                                           const double* T, int N, const OffStep* __restrict__ C, double logs,
                                           double tr, double ti, double* out) {
    const double zr = 0.5 * (w2 - w1), n1 = w1 * w1 + zi * zi, n2 = w2 * w2 + zi * zi;
    const EdgeLog lg = edge_log(w1, w2, zi);
    const double l1 = lg.l1, dl = lg.dl, ang = lg.ang;
    const double q0r = 0.5 * dl, q0i = 0.5 * ang;
    // rho = |z + sqrt(z^2 - 1)|, the growth of the recurrence
    const float s = 0.5f * (sqrtf((float)n1) + sqrtf((float)n2));
    const float rho = s + sqrtf(fmaxf(s * s - 1.0f, 0.0f));
    double Ar = 0.0, Ai = 0.0, Br = 0.0, Bi = 0.0, Sr = 0.0, Si = 0.0;
    // s_n = g_(n-1)/(2n - 1) - g_(n+1)/(2n + 3), g_0 apart
    auto add = [&](int n, double qr, double qi, double gm, double gn, double gp) {
        double sn = 0.0;
        if (n >= 2) sn = gm / (2 * n - 1);
        if (n + 1 < N) sn -= gp / (2 * n + 3);
        Sr = fma(sn, qr, Sr);
        Si = fma(sn, qi, Si);
        if (n < N) {
            const double pn = p[n * kOffTasks], tn = T[n * kOffTasks];
            Ar = fma(pn, qr, Ar);
            Ai = fma(pn, qi, Ai);
            Br = fma(tn, qr, fma(-gn, qi, Br));
            Bi = fma(tn, qi, fma(gn, qr, Bi));
        }
    };
    if (rho < kOffForward) {
        double qr = q0r, qi = q0i, rr = zr * q0r - zi * q0i - 1.0, ri = zr * q0i + zi * q0r;  // Q_n, Q_(n+1)
        double gm = 0.0, gn = g[0];
        for (int n = 0; n <= N; ++n) {
            const double gp = n + 1 < N ? g[(n + 1) * kOffTasks] : 0.0;
            add(n, qr, qi, gm, gn, gp);
            gm = gn;
            gn = gp;
            const OffStep c = C[n + 1];
            const double xr = c.z * (zr * rr - zi * ri) - c.w * qr, xi = c.z * (zr * ri + zi * rr) - c.w * qi;
            qr = rr;
            qi = ri;
            rr = xr;
            ri = xi;
        }
    } else {
        int n = N + 1 + (int)(18.5f / logf(rho));
        double qr = 1e-100, qi = 0.0, rr = 0.0, ri = 0.0;  // q_n, q_(n+1)
        for (; n > N; --n) {
            const OffStep c = C[n];
            const double xr = c.x * (zr * qr - zi * qi) - c.y * rr, xi = c.x * (zr * qi + zi * qr) - c.y * ri;
            rr = qr;
            ri = qi;
            qr = xr;
            qi = xi;
        }
        double gp = 0.0, gn = 0.0;
        for (; n >= 0; --n) {
            const double gm = n >= 1 ? g[(n - 1) * kOffTasks] : 0.0;
            add(n, qr, qi, gm, gn, gp);
            if (n == 0) break;
            gp = gn;
            gn = gm;
            const OffStep c = C[n];
            const double xr = c.x * (zr * qr - zi * qi) - c.y * rr, xi = c.x * (zr * qi + zi * qr) - c.y * ri;
            rr = qr;
            ri = qi;
            qr = xr;
            qi = xi;
        }
        // all sums times Q_0 / q_0
        const double m = 1.0 / (qr * qr + qi * qi);
        const double fr = m * (q0r * qr + q0i * qi), fi = m * (q0i * qr - q0r * qi);
        const double a = Ar * fi + Ai * fr;
        Ai = a;
        const double br = Br * fr - Bi * fi;
        Bi = Br * fi + Bi * fr;
        Br = br;
        Sr = Sr * fr - Si * fi;
    }
    const double L0 = w1 * l1 + w2 * (l1 + dl) - zi * ang - 2.0;  // int log|x - z| dx
    out[0] = fma(logs + 0.5 * L0, g[0], Sr + 2.0 * Ai);
    // -2 i conj(tau) B
    const double cr = tr * Br - ti * Bi, ci = tr * Bi + ti * Br;
    out[1] = 2.0 * ci;
    out[2] = -2.0 * cr;
}

// Next to a corner Q_n grows like -log(r)/2 on both its edges. The parts cancel, since the two series have one
// value there, but only to a rounding of each times the logarithm. So the conjugate gradient at the corner, C,
// is taken off all four edges, and its own integral around the leaf, -2 pi C inside and 0 outside, is put back
// (u_x of one leaf, k = 16, width 1/4, random values of size 1, against extended precision: 1e-13 -> 8e-15 at
// r = 1e-10, 3e-13 -> 8e-15 at 1e-100).
// An edge with the corner at its end sg = 1 or start sg = -1: sum over n of (T_n + i g_n)(Q_n - sg^n Q_0). With
// S_n = sg^n Q_n - Q_0, D_n = S_(n+1) - S_n and delta = 1 - sg z the three-term recurrence reads
//   D_n = (n D_(n-1) - (2n + 1) delta (S_n + Q_0)) / (n + 1),   D_0 = -sg - delta Q_0,
// in which z, whose last bit the derivative of P_n blows up by n^2, stands no more.
__device__ __forceinline__ double2 edge_corner(double w1, double w2, double zi, double sg, const double* g, const double* T,
                                            int N, const OffStep* __restrict__ C) {
    const EdgeLog lg = edge_log(w1, w2, zi);
    const double qr = 0.5 * lg.dl, qi = 0.5 * lg.ang;
    const double ar = sg > 0.0 ? w1 : w2, ai = -sg * zi;  // delta
    double sr = 0.0, si = 0.0, dr = -sg - (ar * qr - ai * qi), di = -(ar * qi + ai * qr);  // S_n, D_n
    double Br = 0.0, Bi = 0.0, sn = 1.0;                                                  // sg^n
    for (int n = 0; n < N; ++n) {
        const double tn = sn * T[n * kOffTasks], gn = sn * g[n * kOffTasks];
        Br = fma(tn, sr, fma(-gn, si, Br));
        Bi = fma(tn, si, fma(gn, sr, Bi));
        sn *= sg;
        sr += dr;
        si += di;
        const OffStep c = C[n + 1];
        const double xr = sr + qr, xi = si + qi;
        dr = c.w * dr - c.z * (ar * xr - ai * xi);
        di = c.w * di - c.z * (ar * xi + ai * xr);
    }
    return make_double2(Br, Bi);
}

// The warp's edges (lanes 4 u + s) with the corner taken off where their leaf has one next to the point (corner >= 0):
// (Re Phi', Im Phi') of this lane's edge, `own` without. A call of its own: rare, and the kernel keeps its registers.
__device__ __noinline__ double2 corner_edges(double w1, double w2, double zi, int s, int corner, bool inside, const double* g,
                                             const double* T, int N, const OffStep* __restrict__ C, double2 own) {
    const double tr = s == 0 ? 1.0 : (s == 2 ? -1.0 : 0.0), ti = s == 1 ? -1.0 : (s == 3 ? 1.0 : 0.0);
    double cr = 0.0, ci = 0.0;  // C, from the edge that starts there
    if (s == corner) {
        double fr = 0.0, fi = 0.0;
        for (int n = N - 1; n >= 0; --n) {  // T + i g at the start, P_n = (-1)^n there
            fr = T[n * kOffTasks] - fr;
            fi = g[n * kOffTasks] - fi;
        }
        cr = tr * fr - ti * fi;
        ci = tr * fi + ti * fr;
    }
    const int from = ((threadIdx.x & 31) & ~3) | max(corner, 0);
    cr = __shfl_sync(0xffffffffu, cr, from);
    ci = __shfl_sync(0xffffffffu, ci, from);
    if (corner < 0) return own;
    const bool start = s == corner, end = s == ((corner + 3) & 3);
    if (start || end) {
        const double2 B = edge_corner(w1, w2, zi, end ? 1.0 : -1.0, g, T, N, C);
        own = make_double2(2.0 * (tr * B.y + ti * B.x), -2.0 * (tr * B.x - ti * B.y));
    } else {  // -2 i (sum - C Q_0)
        const EdgeLog q = edge_log(w1, w2, zi);
        own.x -= cr * q.ang + ci * q.dl;
        own.y += cr * q.dl - ci * q.ang;
    }
    if (start && inside) {
        const double two_pi = 6.28318530717958647693;
        own.x -= two_pi * cr;
        own.y -= two_pi * ci;
    }
    return own;
}

__global__ void __launch_bounds__(kOffThreads, 2) offnode_kernel(const __grid_constant__ OffArgs a) {
    extern __shared__ double off_sm[];
    __shared__ OffLeaf lf[kOffMaxU];
    __shared__ double s_far[3], s_in[3], s_edge[2][3];
    __shared__ double leg[4][kOffMaxN];  // P_m(x), P_m'(x), P_n(y), P_n'(y) at the point in an inside leaf
    __shared__ int s_b;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, k = a.k, kk = k * k, N = 2 * k + 1;
    const int nrows = off_first(k, 4);
    double* cf = off_sm;                            // [nrows][kOffMaxU]
    double* fs = cf + nrows * kOffMaxU;             // [kk][kOffMaxU], then the traces
    double* tp = fs;                                // [3][N][kOffTasks]: P, normal, tangential derivative
    double *tg = tp + N * kOffTasks, *tt = tg + N * kOffTasks;
    const int64_t pt = blockIdx.x;
    const double px = a.x[pt], py = a.y[pt];
    if (tid == 0) {
        // the leaf holding the point: integer coordinates at the finest level, a descent from the root
        const double X = (px - a.lox) / a.width, Y = (py - a.loy) / a.width;
        int b = -1;
        if (X >= 0.0 && X <= 1.0 && Y >= 0.0 && Y <= 1.0) {
            const int D = a.depth;
            const double side = ldexp(1.0, D);
            const int ixd = (int)fmin(floor(X * side), side - 1.0), iyd = (int)fmin(floor(Y * side), side - 1.0);
            b = 0;
            int l = 0;
            while (a.child0[b] >= 0) {
                ++l;
                const int cx = (ixd >> (D - l)) & 1, cy = (iyd >> (D - l)) & 1;
                b = a.child0[b] + ((cy << 1) | cx);
            }
        }
        s_b = b;
    }
    __syncthreads();
    const int b = s_b;
    if (b < 0) {  // outside the closed root box, or a NaN coordinate
        if (tid == 0) a.u[pt] = a.ux[pt] = a.uy[pt] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const int u0 = a.uptr[b], nu = a.uptr[b + 1] - u0;
    if (tid < nu) {
        const int s = a.uidx[u0 + tid];
        const double h = ldexp(a.width, -a.level[s]);
        OffLeaf L;
        L.h = h;
        L.leaf = a.leaf_of_box[s];
        const double x0 = a.lox + a.ix[s] * h, y0 = a.loy + a.iy[s] * h;
        L.d[0] = (px - x0) / h;
        L.d[1] = (x0 + h - px) / h;
        L.d[2] = (py - y0) / h;
        L.d[3] = (y0 + h - py) / h;
        for (int i = 0; i < 4; ++i)
            if (off_exp(L.d[i]) < kOffOnEdge) L.d[i] = 0.0;
        L.inside = L.d[0] >= 0.0 && L.d[1] >= 0.0 && L.d[2] >= 0.0 && L.d[3] >= 0.0;
        if (L.inside)
            for (int i = 0; i < 4; ++i) L.d[i] = fmax(L.d[i], 1e-30);
        const int dl = off_exp(L.d[0]), dr = off_exp(L.d[1]), db = off_exp(L.d[2]), dt = off_exp(L.d[3]);
        L.corner = -1;
        if (min(dl, dr) < kOffCorner && min(db, dt) < kOffCorner) L.corner = db < dt ? (dl < dr ? 0 : 1) : (dl < dr ? 3 : 2);
        lf[tid] = L;
    }
    __syncthreads();
    // the leaves' values in the four classes: sums over the mirrored nodes
    {
        const int hx = (k + 1) / 2;
        for (int q = tid; q < nu * hx * hx; q += kOffThreads) {
            const int u = q / (hx * hx), e = q - u * hx * hx, j = e / hx, i = e - j * hx;
            const double* f = a.f + (size_t)lf[u].leaf * kk;
            const double v0 = f[j * k + i], v1 = f[j * k + k - 1 - i];
            const double v2 = f[(k - 1 - j) * k + i], v3 = f[(k - 1 - j) * k + k - 1 - i];
            const double s0 = v0 + v1, d0 = v0 - v1, s1 = v2 + v3, d1 = v2 - v3;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int nx = sym_half(k, c & 1);
                if (i >= nx || j >= sym_half(k, c >> 1)) continue;
                const double v = (c & 1) ? ((c >> 1) ? d0 - d1 : d0 + d1) : ((c >> 1) ? s0 - s1 : s0 + s1);
                fs[(off_val(k, c) + j * nx + i) * kOffMaxU + u] = v;
            }
        }
    }
    __syncthreads();
    for (int r = tid; r < nrows; r += kOffThreads) {
        int c = 0;
        while (c < 3 && r >= off_first(k, c + 1)) ++c;
        const int K = sym_half(k, c & 1) * sym_half(k, c >> 1);
        off_coeffs_n<kOffMaxU>(nu, a.t.G + a.t.g_off[c] + (r - off_first(k, c)), K, off_rows(k, c),
                               fs + off_val(k, c) * kOffMaxU, cf + r * kOffMaxU);
    }
    __syncthreads();
    // traces. Edges 0..3 = bottom, right, top, left, run around the leaf counterclockwise (top and left
    // against their coordinate: a factor (-1)^n). (leaf, axis, n): n along the edge, the sum across it
    for (int q = tid; q < nu * 2 * N; q += kOffThreads) {
        const int u = q % nu, e = q / nu, axis = e & 1, n = e >> 1;
        double sp[2] = {0.0, 0.0}, sg[2] = {0.0, 0.0};  // even and odd coefficients across
#pragma unroll
        for (int par = 0; par < 2; ++par) {
            const int c = axis == 0 ? (n & 1) | (par << 1) : par | ((n & 1) << 1);  // axis 0: bottom and top
            for (int m = par; m + n <= 2 * k; m += 2) {
                const int row = axis == 0 ? off_row0(k, c, n >> 1) + (m >> 1) : off_row0(k, c, m >> 1) + (n >> 1);
                const double v = cf[row * kOffMaxU + u];
                sp[par] += v;
                sg[par] = fma((double)(m * (m + 1)), v, sg[par]);
            }
        }
        const double sgn = (n & 1) ? -1.0 : 1.0;
        const int lo = 4 * u + (axis == 0 ? 0 : 3), hi = 4 * u + (axis == 0 ? 2 : 1);
        const double flo = axis == 0 ? 1.0 : sgn, fhi = axis == 0 ? sgn : 1.0;
        tp[n * kOffTasks + lo] = flo * (sp[0] - sp[1]);
        tg[n * kOffTasks + lo] = flo * (sg[0] - sg[1]);
        tp[n * kOffTasks + hi] = fhi * (sp[0] + sp[1]);
        tg[n * kOffTasks + hi] = fhi * (sg[0] + sg[1]);
    }
    __syncthreads();
    for (int q = tid; q < 4 * nu * N; q += kOffThreads) {
        const int e = q % (4 * nu), n = q / (4 * nu);
        double s = 0.0;
        for (int m = n + 1; m < N; m += 2) s += tp[m * kOffTasks + e];
        tt[n * kOffTasks + e] = (4 * n + 2) * s;
    }
    __syncthreads();
    const double h = ldexp(a.width, -a.level[b]);
    const double inv2pi = 0.15915494309189533577, pi = 3.14159265358979323846;
    if (warp < 2) {
        // one edge per lane
        const int e = tid;
        double v[3] = {0.0, 0.0, 0.0}, w1 = 0.0, w2 = 0.0, zi = 0.0, hl = 0.0, tr = 0.0, ti = 0.0;
        int corner = -1;
        const int s = e & 3;
        if (e < 4 * nu) {
            const OffLeaf L = lf[e >> 2];
            // (end - point, point - start) along the edge, distance inwards
            w1 = 2.0 * (s == 0 ? L.d[1] : (s == 1 ? L.d[3] : (s == 2 ? L.d[0] : L.d[2])));
            w2 = 2.0 * (s == 0 ? L.d[0] : (s == 1 ? L.d[2] : (s == 2 ? L.d[1] : L.d[3])));
            zi = 2.0 * (s == 0 ? L.d[2] : (s == 1 ? L.d[1] : (s == 2 ? L.d[3] : L.d[0])));
            hl = L.h;
            tr = s == 0 ? 1.0 : (s == 2 ? -1.0 : 0.0);
            ti = s == 1 ? -1.0 : (s == 3 ? 1.0 : 0.0);
            edge_terms(w1, w2, zi, tp + e, tg + e, tt + e, N, a.t.C, log(0.5 * hl), tr, ti, v);
            corner = L.corner;
        }
        if (__any_sync(0xffffffffu, corner >= 0)) {
            const double2 w = corner_edges(w1, w2, zi, s, corner, corner >= 0 && lf[e >> 2].inside, tg + e, tt + e, N,
                                           a.t.C, make_double2(v[1], v[2]));
            v[1] = w.x;
            v[2] = w.y;
        }
        v[0] *= hl * hl;
        v[1] *= hl;
        v[2] *= hl;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
            if (lane == 0) s_edge[warp][i] = v[i];
        }
    } else if (warp == 2) {
        // far part: b's local expansion at zeta = (t - z_b)/h (lanes split the coefficients), then the
        // W multipoles (lanes split the boxes); fixed-order shuffle sums
        const int P = a.P;
        const double cxb = a.lox + ((double)a.ix[b] + 0.5) * h, cyb = a.loy + ((double)a.iy[b] + 0.5) * h;
        const double zr = (px - cxb) / h, zi = (py - cyb) / h;
        double phr = 0.0, dr = 0.0, di = 0.0;
        const double* L = a.Lexp + (size_t)b * a.R * 2 * P;
        for (int l = lane; l < P; l += 32) {
            // zeta^l and l zeta^(l-1) by repeated multiplication (l <= 63)
            double pr = 1.0, pi_ = 0.0, qr = 0.0, qi = 0.0;  // zeta^l, zeta^(l-1)
            for (int e = 0; e < l; ++e) {
                qr = pr;
                qi = pi_;
                const double t = pr * zr - pi_ * zi;
                pi_ = pr * zi + pi_ * zr;
                pr = t;
            }
            const double br = L[2 * l], bi = L[2 * l + 1];
            phr += br * pr - bi * pi_;
            dr += l * (br * qr - bi * qi) / h;  // Phi' = (1/h) sum_l l b~_l zeta^(l-1)
            di += l * (br * qi + bi * qr) / h;
        }
        // W list: box c of width h/2 at offset (dx, dy) (units of h/4 in the pattern): zeta_w = 2 (zeta - D)
        for (int e = a.wptr[b] + lane; e < a.wptr[b + 1]; e += 32) {
            const int c = a.widx[e];
            const int cfg = a.wcfg[e];
            int qx, qy;
            far_pattern(cfg, &qx, &qy);
            const double wr = 2.0 * (zr - qx / 4.0), wi = 2.0 * (zi - qy / 4.0);
            const double hw = 0.5 * h;
            const double* M = a.Mexp + (size_t)c * a.R * 2 * P;
            const double a0 = M[0];
            // a_0 (log h_w + log zeta_w) + sum_n a_n zeta_w^-n, derivative a_0/zeta_w - sum n a_n zeta_w^(-n-1)
            const double m2 = wr * wr + wi * wi;
            const double ir = wr / m2, ii = -wi / m2;  // 1/zeta_w
            double sr = a0 * (log(hw) + 0.5 * log(m2));  // Re of a_0 (log h_w + log zeta_w)
            double gr = a0 * ir, gi = a0 * ii;
            double zr_n = 1.0, zi_n = 0.0;  // zeta_w^-n
            for (int n = 1; n < P; ++n) {
                // derivative term -n a_n zeta^(-n-1) = -n a_n zeta^-n / zeta
                const double ar = M[2 * n], ai = M[2 * n + 1];
                const double t1 = zr_n * ir - zi_n * ii, t2 = zr_n * ii + zi_n * ir;  // zeta^-(n) * 1/zeta
                zr_n = t1;
                zi_n = t2;  // now zeta^-n
                sr += ar * zr_n - ai * zi_n;
                const double u1 = zr_n * ir - zi_n * ii, u2 = zr_n * ii + zi_n * ir;  // zeta^-(n+1)
                gr -= n * (ar * u1 - ai * u2);
                gi -= n * (ar * u2 + ai * u1);
            }
            phr += sr;
            dr += gr / hw;  // d zeta_w / dz = 1 / h_w
            di += gi / hw;
        }
        for (int o = 16; o > 0; o >>= 1) {
            phr += __shfl_xor_sync(0xffffffffu, phr, o);
            dr += __shfl_xor_sync(0xffffffffu, dr, o);
            di += __shfl_xor_sync(0xffffffffu, di, o);
        }
        if (lane == 0) {
            s_far[0] = -inv2pi * phr;
            s_far[1] = -inv2pi * dr;
            s_far[2] = inv2pi * di;
        }
    } else if (warp == 3) {
        // 2 pi P and pi F in the leaves that hold the point (one, or those that share its edge or corner)
        double v[3] = {0.0, 0.0, 0.0};
        for (int u = 0; u < nu; ++u) {
            const OffLeaf L = lf[u];
            if (!L.inside) continue;
            __syncwarp();
            if (lane < 2) {
                // 2 x = sg (1 - delta) in [-1, 1]; P_m by its differences, as in edge_corner
                const double dl = L.d[2 * lane], dr = L.d[2 * lane + 1], delta = 2.0 * fmin(dl, dr);
                const int neg = dl < dr ? 1 : 0;
                double p0 = 1.0, dp = -delta, q0 = 0.0, q1 = 2.0;  // sg^m P_m, its difference, 2 P_m', 2 P_(m+1)'
                for (int m = 0; m < N; ++m) {
                    leg[2 * lane][m] = off_flip(p0, m & neg);
                    leg[2 * lane + 1][m] = q0;
                    const OffStep c = a.t.C[m + 1];
                    p0 += dp;
                    const double q2 = fma((double)(4 * m + 6), off_flip(p0, (m + 1) & neg), q0);
                    dp = fma(-(c.z * delta), p0, c.w * dp);  // two operations in the chain
                    q0 = q1;
                    q1 = q2;
                }
            }
            __syncwarp();
            double w[3] = {0.0, 0.0, 0.0};
            for (int m = lane; m < N; m += 32)
                for (int n = 0; m + n <= 2 * k; ++n) {
                    const double cmn = cf[(off_row0(k, (m & 1) | ((n & 1) << 1), m >> 1) + (n >> 1)) * kOffMaxU + u];
                    w[0] = fma(cmn, leg[0][m] * leg[2][n], w[0]);
                    w[1] = fma(cmn, leg[1][m] * leg[2][n], w[1]);
                    w[2] = fma(cmn, leg[0][m] * leg[3][n], w[2]);
                }
            v[0] = fma(L.h * L.h, w[0], v[0]);
            v[1] = fma(L.h, w[1], v[1]);
            v[2] = fma(L.h, w[2], v[2]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
            if (lane == 0) s_in[i] = 2.0 * pi * v[i];
        }
    }
    __syncthreads();
    if (tid == 0) {
        // gradient: (u_x, u_y) = -(1/2pi) (Re Phi', -Im Phi')
        a.u[pt] = s_far[0] - inv2pi * ((s_edge[0][0] + s_edge[1][0]) + s_in[0]);
        a.ux[pt] = s_far[1] - inv2pi * ((s_edge[0][1] + s_edge[1][1]) + s_in[1]);
        a.uy[pt] = s_far[2] - inv2pi * (s_in[2] - (s_edge[0][2] + s_edge[1][2]));
    }
}

static size_t off_smem(int k) {
    const size_t rows = (size_t)off_first(k, 4) * kOffMaxU;
    return (rows + std::max((size_t)k * k * kOffMaxU, (size_t)3 * (2 * k + 1) * kOffTasks)) * sizeof(double);
}

}  // namespace vfmm

using namespace vfmm;

extern "C" int vfmm_evaluate_points(const vfmm_tree* tree, const vfmm_ops* ops, const double* f_dev,
                                    const void* workspace_dev, size_t workspace_bytes, int64_t n_points,
                                    const double* x_dev, const double* y_dev, double* u_dev, double* ux_dev,
                                    double* uy_dev, void* stream) {
    if (!tree || !ops) return fail(VFMM_ERR_INVALID_ARG, "null tree or ops");
    if (tree->t.k != ops->k) return fail(VFMM_ERR_INVALID_ARG, "tree and ops differ in k");
    if (n_points < 0) return fail(VFMM_ERR_INVALID_ARG, "n_points < 0");
    if (n_points == 0) return VFMM_OK;
    if (!f_dev || !workspace_dev || !x_dev || !y_dev || !u_dev || !ux_dev || !uy_dev)
        return fail(VFMM_ERR_INVALID_ARG, "null buffer");
    if (n_points > (int64_t)INT32_MAX) return fail(VFMM_ERR_INVALID_ARG, "too many points for one call");
    const DeviceTree& T = tree->t;
    const double* Mexp = nullptr;
    const double* Lexp = nullptr;
    int R = 1;
    VFMM_CHECK(solve_expansions(tree, ops, workspace_dev, workspace_bytes, &Mexp, &Lexp, &R));
    OffArgs a;
    a.k = ops->k;
    a.P = ops->p + 1;
    a.depth = T.depth;
    a.R = R;
    a.n = n_points;
    a.lox = T.cx - T.width / 2.0;
    a.loy = T.cy - T.width / 2.0;
    a.width = T.width;
    a.child0 = T.child0;
    a.level = T.level;
    a.ix = T.ix;
    a.iy = T.iy;
    a.leaf_of_box = T.leaf_of_box;
    a.uptr = T.lptr[VFMM_LIST_U];
    a.uidx = T.lidx[VFMM_LIST_U];
    a.wptr = T.lptr[VFMM_LIST_W];
    a.widx = T.lidx[VFMM_LIST_W];
    a.wcfg = T.lcfg[VFMM_LIST_W];
    a.f = f_dev;
    a.Mexp = Mexp;
    a.Lexp = Lexp;
    a.x = x_dev;
    a.y = y_dev;
    a.u = u_dev;
    a.ux = ux_dev;
    a.uy = uy_dev;
    a.t = *(const OffTables*)ops->off;
    static thread_local int attr_dev = -1;
    int dev = 0;
    VFMM_CUDA(cudaGetDevice(&dev));
    if (attr_dev != dev) {
        VFMM_CUDA(cudaFuncSetAttribute(offnode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)off_smem(16)));
        attr_dev = dev;
    }
    offnode_kernel<<<(unsigned)n_points, kOffThreads, off_smem(ops->k), (cudaStream_t)stream>>>(a);
    VFMM_CUDA(cudaGetLastError());
    return VFMM_OK;
}
