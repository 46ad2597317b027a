// a2: FP64 near field. For every ordered pair of triangles sharing a vertex,
// the local 3x3 Galerkin blocks of V, K, D (Laplace and Yukawa) by a
// regularised [0,1]^4 rule (maps in the manner of Sauter and Schwab, with a
// Gauss-Legendre product rule), minus the same blocks by the far rule that the
// pair kernel applies to every pair, summed into the vertex-pair CSR. The full
// (regularised) diagonals are kept for the block-diagonal preconditioner.
//
// Operators (paper eq. layer_potentials, weak forms on P1):
//   V_ab = int int l_a(x) G(x,y) l_b(y)       K_ab = int int l_a(x) dG/dn_y l_b(y)
//   D_ab = int int G [curl l_a . curl l_b + kappa^2 n_x.n_y l_a l_b]  (hypersingular,
//          integrated by parts; curl l_a = -e_a / (2|tau|), e_a the edge opposite a)
// with G_int = 1/(4 pi r), G_ext = exp(-kappa r)/(4 pi r).
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "exp64.cuh"
#include "internal.h"

namespace pb {

struct Gauss {
    double x[12];
    double w[12];
    int n;
};

// Gauss-Legendre nodes on [0,1] by Newton's method on P_n (three-term
// recurrence for P_n, derivative from P_n and P_{n-1}).
static Gauss gauss01(int n) {
    Gauss g;
    g.n = n;
    for (int i = 0; i < n; ++i) {
        double x = cos(M_PI * (i + 0.75) / (n + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            if (n == 1) { p1 = x; p0 = 1.0; }
            dp = n * (x * p1 - p0) / (x * x - 1.0);
            double dx = p1 / dp;
            x -= dx;
            if (fabs(dx) < 1e-16) break;
        }
        // recompute the derivative at the converged node for the weight
        double p0 = 1.0, p1 = x;
        for (int k = 2; k <= n; ++k) {
            double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        if (n == 1) { p1 = x; p0 = 1.0; }
        dp = n * (x * p1 - p0) / (x * x - 1.0);
        double w = 2.0 / ((1.0 - x * x) * dp * dp);
        g.x[i] = 0.5 * (1.0 - x);  // ascending on [0,1]
        g.w[i] = 0.5 * w;
    }
    return g;
}

// One regularised cube point -> reference points (sx,tx) in tau and (sy,ty)
// in sigma on {0 <= t <= s <= 1}, returning the region Jacobian.
// kind 0: coincident (6 regions), 1: common edge t = 0 (6), 2: common vertex (0,0) (2).
__device__ __forceinline__ double ss_map(int kind, int reg, double xi, double e1, double e2, double e3,
                                         double& sx, double& tx, double& sy, double& ty) {
    double a0, a1, b0, b1, jac;
    int base = reg;
    bool swap = false;
    if (kind == 2) {
        swap = reg == 1;
        a0 = xi; a1 = xi * e1;
        b0 = xi * e2; b1 = xi * e2 * e3;
        jac = xi * xi * xi * e2;
    } else {
        if (reg >= 3) { base = reg - 3; swap = true; }
        if (kind == 0) {
            jac = xi * xi * xi * e1 * e1 * e2;
            if (base == 0) {
                a0 = xi; a1 = xi * (1.0 - e1 + e1 * e2);
                b0 = xi * (1.0 - e1 * e2 * e3); b1 = xi * (1.0 - e1);
            } else if (base == 1) {
                a0 = xi; a1 = xi * e1 * (1.0 - e2 + e2 * e3);
                b0 = xi * (1.0 - e1 * e2); b1 = xi * e1 * (1.0 - e2);
            } else {
                a0 = xi * (1.0 - e1 * e2 * e3); a1 = xi * e1 * (1.0 - e2 * e3);
                b0 = xi; b1 = xi * e1 * (1.0 - e2);
            }
        } else {
            // x^ = (s1, s1 w1), y^ = (s2, s2 w2), s1 = xi, s2 = xi (1 - h); the
            // largest of (h, w1, w2) is e1 and the other two are e1 times (e2, e3)
            double h, w1, w2;
            if (base == 0) { h = e1; w1 = e1 * e2; w2 = e1 * e3; }
            else if (base == 1) { w1 = e1; h = e1 * e2; w2 = e1 * e3; }
            else { w2 = e1; h = e1 * e2; w1 = e1 * e3; }
            double s2 = xi * (1.0 - h);
            a0 = xi; a1 = xi * w1;
            b0 = s2; b1 = s2 * w2;
            jac = xi * xi * xi * (1.0 - h) * e1 * e1;
        }
    }
    if (swap) { sx = b0; tx = b1; sy = a0; ty = a1; }
    else { sx = a0; tx = a1; sy = b0; ty = b1; }
    return jac;
}

// The regularised rule of the coincident pairs does not depend on the pair:
// every (region, Gauss index) point of regions 0..2 of the coincident map, its
// reference points in both copies of the triangle and its weight (Gauss
// weights times the region Jacobian), computed once per build. Structure of
// arrays over the entries.
struct SSTable {
    const double* sx;
    const double* tx;
    const double* sy;
    const double* ty;
    const double* w;
    // w times the monomials (s', t', s, s s', s t', t, t s', t t') of the
    // entry's frame coordinates: mono[c * n + e]
    const double* mono;
    int n;       // entries in all (3 n^4)
};
constexpr int SS_TABLE_ARRAYS = 13;  // sx, tx, sy, ty, w and the eight weighted monomials

__global__ void k_ss_table(Gauss gq, int n, double* __restrict__ tab) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int q = gq.n, n4 = q * q * q * q;
    const int reg = e / n4, r = e - reg * n4;
    const int i0 = r / (q * q * q), i1 = (r / (q * q)) % q, i2 = (r / q) % q, i3 = r % q;
    double sx, tx, sy, ty;
    const double jac = ss_map(0, reg, gq.x[i0], gq.x[i1], gq.x[i2], gq.x[i3], sx, tx, sy, ty);
    tab[e] = sx;
    tab[n + e] = tx;
    tab[2 * n + e] = sy;
    tab[3 * n + e] = ty;
    const double w = gq.w[i0] * gq.w[i1] * gq.w[i2] * gq.w[i3] * jac;
    tab[4 * n + e] = w;
    const double ws = w * sx, wt = w * tx;
    const double mono[8] = {w * sy, w * ty, ws, ws * sy, ws * ty, wt, wt * sy, wt * ty};
    for (int c = 0; c < 8; ++c) tab[(5 + c) * n + e] = mono[c];
}

// Points of the edge (kind 1, 6 regions) and vertex (kind 2, 2 regions) maps.
// Three properties of both maps carry the pair sums (k_adj_pairs):
//   - every frame coordinate is proportional to xi, so with both frames starting
//     at the shared vertex x - y = xi d(eta) and r = xi |d|: the geometry is
//     evaluated at xi = 1 only, once per (eta1, eta2, eta3);
//   - the Laplace kernels are homogeneous in xi (G ~ 1/xi, K ~ 1/xi^2), so their
//     xi sums are the constants mu_m = sum_i w_i xi_i^m; the Yukawa kernels need
//     E_m(z) = sum_i w_i xi_i^m e^{-z xi_i}, z = kappa |d|, m = 1..4 (Radial);
//   - eta3 enters a single coordinate, the second one (t) of one frame, and
//     linearly, while the region Jacobian does not involve it; so over the eta3
//     points of an entry d = D0 + eta3 D1 and every weighted monomial is affine
//     in eta3: two sums per kernel (sum w3 g, sum w3 eta3 g), expanded into the
//     nine moments once per entry.
// One entry per (region, eta1, eta2), at xi = 1 (array c at v[c * n + e]):
//   0..3  sa, ta, sa', ta': the frame coordinates at eta3 = 0 (x: s, t; y: s', t')
//   4, 5  tb, tb': the slopes of t and t' in eta3 (one of them is zero)
//   6..14 c0[3 alpha + beta] = W P_alpha Q_beta, P = (1, sa, ta), Q = (1, sa', ta'),
//         W = the Gauss weights of eta1, eta2 times the Jacobian
//   15..19 the eta3-slope coefficients of the moments that change with eta3:
//         (0,2) W tb', (1,2) W sa tb', (2,0) W tb, (2,1) W tb sa', (2,2) W (ta tb' + tb ta')
// One table per class (edge or vertex), each with its own Gauss rule.
struct SSOuter {
    const double* v;
    int n;        // entries (regions x nss^2)
    int nss;      // Gauss points per dimension
    int nreg;     // regions of the map: 6 (edge) or 2 (vertex)
};
constexpr int SS_OUTER_ARRAYS = 20;

__global__ void k_ss_outer(Gauss gq, int kind, int n, double* __restrict__ tab) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = gq.n, n2 = q * q;
    if (e >= n) return;
    const int reg = e / n2, r = e - reg * n2;
    const int i1 = r / q, i2 = r % q;
    double sx0, tx0, sy0, ty0, sx1, tx1, sy1, ty1;
    const double jac = ss_map(kind, reg, 1.0, gq.x[i1], gq.x[i2], 0.0, sx0, tx0, sy0, ty0);
    const double jac1 = ss_map(kind, reg, 1.0, gq.x[i1], gq.x[i2], 1.0, sx1, tx1, sy1, ty1);
    const double tb = tx1 - tx0, tb2 = ty1 - ty0;
    const double W = gq.w[i1] * gq.w[i2] * jac;
    // the structure the factorisation relies on: s, s' and the Jacobian free of eta3
    const bool ok = sx1 == sx0 && sy1 == sy0 && jac1 == jac;
    const double P[3] = {1.0, sx0, tx0}, Q[3] = {1.0, sy0, ty0};
    double v[SS_OUTER_ARRAYS] = {sx0, tx0, sy0, ty0, tb, tb2};
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) v[6 + 3 * a + b] = ok ? W * P[a] * Q[b] : __longlong_as_double(0x7ff8000000000000LL);
    v[15] = W * tb2;
    v[16] = W * sx0 * tb2;
    v[17] = W * tb;
    v[18] = W * tb * sy0;
    v[19] = W * (tx0 * tb2 + tb * ty0);
    for (int c = 0; c < SS_OUTER_ARRAYS; ++c) tab[c * n + e] = v[c];
}

// The xi rule of an adjacent pair's sums: mu_m and E_m(z), m = 1..4. For z up to
// zlim[RAD_DEG] E_m is its Taylor polynomial, sum_k (-1)^k mu_{m+k} z^k / k!, of the
// degree d whose first omitted term is below 2^-56 for z <= zlim[d] (its terms
// alternate and fall); beyond, the exponentials themselves are summed. Passed
// by value: the coefficients are then constant operands of the FMAs.
constexpr int RAD_DEG = 13;
struct Radial {
    double c[4][RAD_DEG + 1];  // c[m - 1][k]
    double mu[4];              // mu_1..mu_4
    double x[12], w[12];       // the Gauss rule (xi and eta3)
    double wx[4][12];          // w_i xi_i^m
    float zlim[RAD_DEG + 1];
    int n;
};

static Radial make_radial(const Gauss& g) {
    Radial r;
    r.n = g.n;
    for (int i = 0; i < 12; ++i) {
        r.x[i] = i < g.n ? g.x[i] : 0.0;
        r.w[i] = i < g.n ? g.w[i] : 0.0;
        double p = r.w[i];
        for (int m = 0; m < 4; ++m) r.wx[m][i] = p *= r.x[i];
    }
    for (int m = 1; m <= 4; ++m) {
        double f = 1.0;  // (-1)^k / k!
        for (int k = 0; k <= RAD_DEG; ++k) {
            double mu = 0.0;
            for (int i = 0; i < g.n; ++i) mu += g.w[i] * std::pow(g.x[i], m + k);
            r.c[m - 1][k] = f * mu;
            f *= -1.0 / (k + 1);
        }
        r.mu[m - 1] = r.c[m - 1][0];
    }
    double fact = 1.0;
    for (int d = 0; d <= RAD_DEG; ++d) {
        fact *= d + 1;
        r.zlim[d] = (float)std::pow(fact * std::ldexp(1.0, -56), 1.0 / (d + 1));
    }
    return r;
}

// Geometry of one triangle in the reordered frame of its singular map:
// Q0, E1 = Q1 - Q0, E2 = Q2 - Q1 (x(s,t) = Q0 + s E1 + t E2), the inverse
// permutation (original corner -> reordered), normal and area. Kept in shared
// memory per warp: the lanes read it by broadcast.
struct TriFrame {
    double q0[3], e1[3], e2[3];
    double n[3];
    double area;
    int inv[3];  // reordered index of original corner a
};

__device__ void make_frame(const double* verts, const int32_t* tris, const double* tgeo, int t, int perm,
                           TriFrame& f) {
    double p[3][3];
    for (int a = 0; a < 3; ++a)
        for (int k = 0; k < 3; ++k) p[a][k] = verts[3 * (int64_t)tris[3 * (int64_t)t + a] + k];
    int o[3] = {perm & 3, (perm >> 2) & 3, (perm >> 4) & 3};  // original corner of reordered k
    for (int k = 0; k < 3; ++k) {
        f.q0[k] = p[o[0]][k];
        f.e1[k] = p[o[1]][k] - p[o[0]][k];
        f.e2[k] = p[o[2]][k] - p[o[1]][k];
        f.n[k] = tgeo[16 * (int64_t)t + k];
    }
    f.area = tgeo[16 * (int64_t)t + 3];
    for (int k = 0; k < 3; ++k) f.inv[o[k]] = k;
}

// original corner a of the triangle
__device__ __forceinline__ double corner(const TriFrame& f, int a, int k) {
    int r = f.inv[a];
    return f.q0[k] + (r >= 1 ? f.e1[k] : 0.0) + (r >= 2 ? f.e2[k] : 0.0);
}

// e^x for x <= 0 (the Yukawa factor e^{-kappa r}) by the table-driven method
// of Tang (ACM Trans. Math. Software 15(2), 1989): x = (32 m + j) ln2/32 + r
// with |r| <= ln2/64, and e^x = 2^m 2^{j/32} e^r, with 2^{j/32} from a table
// (correctly rounded doubles) and e^r its Taylor polynomial of degree 6
// (remainder below 2e-18). The reduction subtracts n ln2/32 in two parts, the
// first with 37 significant bits so that n times it is exact for |n| < 2^15.
// Arguments below -700 give 0 (the exact value is below 1e-304).
__device__ const double g_exp2_32[32] = {
    0x1.0000000000000p+0, 0x1.059b0d3158574p+0, 0x1.0b5586cf9890fp+0, 0x1.11301d0125b51p+0,
    0x1.172b83c7d517bp+0, 0x1.1d4873168b9aap+0, 0x1.2387a6e756238p+0, 0x1.29e9df51fdee1p+0,
    0x1.306fe0a31b715p+0, 0x1.371a7373aa9cbp+0, 0x1.3dea64c123422p+0, 0x1.44e086061892dp+0,
    0x1.4bfdad5362a27p+0, 0x1.5342b569d4f82p+0, 0x1.5ab07dd485429p+0, 0x1.6247eb03a5585p+0,
    0x1.6a09e667f3bcdp+0, 0x1.71f75e8ec5f74p+0, 0x1.7a11473eb0187p+0, 0x1.82589994cce13p+0,
    0x1.8ace5422aa0dbp+0, 0x1.93737b0cdc5e5p+0, 0x1.9c49182a3f090p+0, 0x1.a5503b23e255dp+0,
    0x1.ae89f995ad3adp+0, 0x1.b7f76f2fb5e47p+0, 0x1.c199bdd85529cp+0, 0x1.cb720dcef9069p+0,
    0x1.d5818dcfba487p+0, 0x1.dfc97337b9b5fp+0, 0x1.ea4afa2a490dap+0, 0x1.f50765b6e4540p+0};

__device__ __forceinline__ double exp_nonpos(double x) {
    const double shifter = 0x1.8p52;  // adding it rounds to an integer held in the low mantissa bits
    const double tn = __fma_rn(x, 0x1.71547652b82fep+5, shifter);  // x 32/ln2, rounded
    const int n = __double2loint(tn);
    const double nd = __dsub_rn(tn, shifter);
    const double r = __fma_rn(-nd, 0x1.cf79abc9e3b3ap-45, __fma_rn(-nd, 0x1.62e42fefa0000p-6, x));
    double q = 1.0 / 720.0;
    q = __fma_rn(q, r, 1.0 / 120.0);
    q = __fma_rn(q, r, 1.0 / 24.0);
    q = __fma_rn(q, r, 1.0 / 6.0);
    q = __fma_rn(q, r, 0.5);
    q = __fma_rn(q, r, 1.0);
    q = __fma_rn(q, r, 1.0);
    const double v = __ldg(g_exp2_32 + (n & 31)) * q;
    const long long bits = __double_as_longlong(v) + ((long long)(n >> 5) << 52);  // times 2^m
    return x < -700.0 ? 0.0 : __longlong_as_double(bits);
}

// Accumulators of a pair: SL[9], SY[9], KL[9], KY[9], sum w G_L, sum w G_Y, and
// KTL[9], KTY[9]: the double-layer kernel with the normal of the first triangle,
// which is the K block of the reversed pair.
#define NACC_SYM 56

// Regularised rules in the frames' own coordinates. A point of a frame is
// q0 + s e1 + t e2 and its corner basis values are mu = (1 - s, s - t, t) in the
// frame's corner order; so the quadrature sums are taken as moments in the
// monomial bases (1, s, t) x (1, s', t') and turned into the corner blocks once
// per pair (frame_to_corner). For an adjacent pair both frames start at the
// shared vertex, and d = x - y is formed from the frame vectors directly.

// The vectors of an adjacent pair that its lanes read by broadcast: the frames'
// edges and the normals. (d . n_B is the height of x over the second triangle's plane
// and needs no y, but only for a normal without rounding: see band_pass.)
struct AdjGeo {
    double e1a[3], e2a[3], e1b[3], e2b[3];
    double na[3], nb[3];
};

// One entry (region, eta1, eta2) of an adjacent pair: the eta3 points' sums, then
// the moments mom[9 k + 3 alpha + beta], k = G_L, G_Y, K_L, K_Y, K^T_L, K^T_Y (the
// reversed pair's double layers), without the factor 1/(4 pi) and, for the Laplace
// kernels, without the xi sums (mu). A moment of degree deg = [alpha > 0] +
// [beta > 0] carries xi^deg: the Yukawa sums are kept per degree.
template <int NSS>
__device__ __forceinline__ void accum_entry(double* mom, const SSOuter& tab, const Radial& rad, int e,
                                            const AdjGeo& P, double kappa, int deg) {
    const int n = tab.n;
    const double ta = tab.v[n + e], ta2 = tab.v[3 * n + e], tb = tab.v[4 * n + e], tb2 = tab.v[5 * n + e];
    double D0[3], D1[3], hb0, hb1, ha0, ha1;
    {
        const double sa = tab.v[e], sa2 = tab.v[2 * n + e];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            D0[k] = __fma_rn(-ta2, P.e2b[k], __fma_rn(-sa2, P.e1b[k], __fma_rn(ta, P.e2a[k], sa * P.e1a[k])));
            D1[k] = __fma_rn(tb, P.e2a[k], -tb2 * P.e2b[k]);
        }
    }
    hb0 = D0[0] * P.nb[0] + D0[1] * P.nb[1] + D0[2] * P.nb[2];  // d . n_B and -d . n_A
    hb1 = D1[0] * P.nb[0] + D1[1] * P.nb[1] + D1[2] * P.nb[2];
    ha0 = -(D0[0] * P.na[0] + D0[1] * P.na[1] + D0[2] * P.na[2]);
    ha1 = -(D1[0] * P.na[0] + D1[1] * P.na[1] + D1[2] * P.na[2]);
    // Laplace: sums with w3 and w3 eta3; Yukawa: with w3 for degrees 0..2, with w3 eta3 for 1, 2
    double l0[3] = {0, 0, 0}, l1[3] = {0, 0, 0}, y0[3][3], y1[3][2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int c = 0; c < 3; ++c) y0[k][c] = 0.0;
        y1[k][0] = y1[k][1] = 0.0;
    }
    const int nss = NSS > 0 ? NSS : rad.n;
#pragma unroll 1
    for (int j = 0; j < nss; ++j) {
        const double x3 = rad.x[j], w3 = rad.w[j];
        double r2;
        {
            const double d0 = __fma_rn(x3, D1[0], D0[0]), d1 = __fma_rn(x3, D1[1], D0[1]),
                         d2 = __fma_rn(x3, D1[2], D0[2]);
            r2 = __fma_rn(d2, d2, __fma_rn(d1, d1, d0 * d0));
        }
        const double rinv = rsqrt(r2);
        const double z = kappa * (r2 * rinv);
        double E[4] = {0, 0, 0, 0};
        if (deg <= RAD_DEG) {
#pragma unroll
            for (int k = RAD_DEG; k >= 0; --k)
                if (k <= deg) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) E[m] = __fma_rn(E[m], z, rad.c[m][k]);
                }
        } else {
            for (int i = 0; i < nss; ++i) {
                const double ex = exp_nonpos(-z * rad.x[i]);
#pragma unroll
                for (int m = 0; m < 4; ++m) E[m] = __fma_rn(rad.wx[m][i], ex, E[m]);
            }
        }
        const double wr = w3 * rinv, fl = wr * (rinv * rinv);
        // (1 + z xi) e^{-z xi}: the double layers' xi sums per degree
        const double F[3] = {__fma_rn(z, E[1], E[0]), __fma_rn(z, E[2], E[1]), __fma_rn(z, E[3], E[2])};
        const double g[3] = {wr, fl * __fma_rn(x3, hb1, hb0), fl * __fma_rn(x3, ha1, ha0)};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double gx = g[k] * x3;
            const double* W = k == 0 ? E + 1 : F;
            l0[k] += g[k];
            l1[k] += gx;
#pragma unroll
            for (int c = 0; c < 3; ++c) y0[k][c] = __fma_rn(g[k], W[c], y0[k][c]);
            y1[k][0] = __fma_rn(gx, W[1], y1[k][0]);
            y1[k][1] = __fma_rn(gx, W[2], y1[k][1]);
        }
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        const double c0 = tab.v[(6 + c) * n + e];
        const int dg = (c >= 3) + (c % 3 > 0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            mom[18 * k + c] = __fma_rn(c0, l0[k], mom[18 * k + c]);
            mom[18 * k + 9 + c] = __fma_rn(c0, y0[k][dg], mom[18 * k + 9 + c]);
        }
    }
    constexpr int slot[5] = {2, 5, 6, 7, 8}, sdeg[5] = {1, 2, 1, 2, 2};
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double c1 = tab.v[(15 + q) * n + e];
        const int c = slot[q];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            mom[18 * k + c] = __fma_rn(c1, l1[k], mom[18 * k + c]);
            mom[18 * k + 9 + c] = __fma_rn(c1, y1[k][sdeg[q] - 1], mom[18 * k + 9 + c]);
        }
    }
}

// coincident pair: one frame, d = (s - s') e1 + (t - t') e2; k = G_L, G_Y
__device__ __forceinline__ void accum_coin_frame(double* mom, const SSTable& tab, int e, const TriFrame& A,
                                                 double kappa) {
    const double ds = tab.sx[e] - tab.sy[e], dt = tab.tx[e] - tab.ty[e];
    double d[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = __fma_rn(dt, A.e2[k], ds * A.e1[k]);
    const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const double rinv = rsqrt(r2);
    const double gl = rinv * 0.07957747154594767;  // 1 / (4 pi r)
    const double gy = exp_nonpos(-kappa * (r2 * rinv)) * gl;
    double m[9];
    m[0] = tab.w[e];
#pragma unroll
    for (int c = 0; c < 8; ++c) m[1 + c] = tab.mono[c * tab.n + e];
#pragma unroll
    for (int c = 0; c < 9; ++c) {
        mom[c] += gl * m[c];
        mom[9 + c] += gy * m[c];
    }
}

// moments of one kernel (mom[3 alpha + beta] over (1, s, t) x (1, s', t')) into
// its corner block out[3 a + b] = sum w g l_a(x) l_b(y)
__device__ __forceinline__ void frame_to_corner(const double* mom, const TriFrame& A, const TriFrame& B,
                                                double* out) {
    double R[3][3], U[3][3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {  // mu_0 = 1 - s, mu_1 = s - t, mu_2 = t on the first frame
        R[0][b] = mom[b] - mom[3 + b];
        R[1][b] = mom[3 + b] - mom[6 + b];
        R[2][b] = mom[6 + b];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // and on the second
        U[a][0] = R[a][0] - R[a][1];
        U[a][1] = R[a][1] - R[a][2];
        U[a][2] = R[a][2];
    }
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) out[3 * a + b] = U[A.inv[a]][B.inv[b]];
}

// One level of a warp reduce-scatter: a lane keeps half of its first 2H
// entries (the upper half when its bit o is set) and adds its partner's copy.
template <int H>
__device__ __forceinline__ void rs_level(double* v, int lane, int o) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const double lo = v[i], hi = v[i + H];
        v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
    }
}

// Warp sums of v[0..NV) into every lane's v. A reduce-scatter over the five
// lane bits (offsets 16 .. 1, N the power of two with NV <= N <= 2 NV, entries
// past NV being zero) leaves lane L with the totals of entries [L N/32,
// (L + 1) N/32) after N/2 + N/4 + ... + N/32 additions, against 5 NV for a
// butterfly on every entry; the totals go through the warp's shared buffer
// (N doubles) back to all lanes. Fixed order: deterministic.
template <int NV, int N>
__device__ __forceinline__ void warp_allsum(double* v, int lane, double* buf) {
    static_assert(N >= 32 && (N & (N - 1)) == 0 && NV <= N && 2 * NV >= N, "reduce-scatter size");
    {
        constexpr int h = N / 2;
        const bool up = lane & 16;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double lo = v[i], hi = i + h < NV ? v[i + h] : 0.0;
            v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, 16);
        }
    }
    rs_level<N / 4>(v, lane, 8);
    rs_level<N / 8>(v, lane, 4);
    rs_level<N / 16>(v, lane, 2);
    rs_level<N / 32>(v, lane, 1);
    constexpr int K = N / 32;
#pragma unroll
    for (int j = 0; j < K; ++j) buf[lane * K + j] = v[j];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = buf[k];
    __syncwarp();  // the buffer is free again
}

// Sums of v[0..NV) over the groups of G lanes of a warp: a reduce-scatter over
// the group's lane bits (N >= NV entries, those past NV being zero), after which lane
// L of a group holds the totals of entries [L N/G, (L + 1) N/G) in v[0..N/G): N (1 -
// 1/G) additions a lane, against NV log2(G) for a butterfly on every entry. Fixed
// order: deterministic.
template <int NV, int N, int G>
__device__ __forceinline__ void group_sums(double* v, int lane) {
    static_assert(N % G == 0 && NV <= N && 2 * NV >= N && (G == 4 || G == 8 || G == 32), "reduce-scatter size");
    {
        constexpr int h = N / 2;
        const bool up = lane & (G / 2);
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double lo = v[i], hi = i + h < NV ? v[i + h] : 0.0;
            v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, G / 2);
        }
    }
    rs_level<N / 4>(v, lane, G / 4);
    if (G >= 8) rs_level<N / 8>(v, lane, G / 8);
    if (G >= 32) {
        rs_level<N / 16>(v, lane, 2);
        rs_level<N / 32>(v, lane, 1);
    }
}

// Six 3x3 blocks (V_L, K_L, D_L, V_Y, K_Y, D_Y) of the pair (tau, sigma), or with
// rev = true of the reversed pair (sigma, tau): every block transposed and the
// double layer taken from the KT accumulators. Layout: out[6 (3a + b) + k] for
// corner a of the test triangle, corner b of the trial one and operator k, so
// that the six values one row-assembly lane reads are 48 contiguous bytes.
__device__ __forceinline__ void expand_blocks(const double* acc, const double* tgeoA, const double* tgeoB, double kappa,
                                              bool rev, double* out) {
    const double nn = tgeoA[0] * tgeoB[0] + tgeoA[1] * tgeoB[1] + tgeoA[2] * tgeoB[2];
    const double f = 1.0 / (4.0 * tgeoA[3] * tgeoB[3]);
    const int kL = rev ? 38 : 18, kY = rev ? 47 : 27;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
            const double* ea = tgeoA + 4 + 3 * a;
            const double* eb = tgeoB + 4 + 3 * b;
            double cc = f * (ea[0] * eb[0] + ea[1] * eb[1] + ea[2] * eb[2]);
            const int ab = 3 * a + b;
            const int o = rev ? 3 * b + a : ab;
            double* e = out + 6 * o;
            e[0] = acc[ab];
            e[1] = acc[kL + ab];
            e[2] = cc * acc[36];
            e[3] = acc[9 + ab];
            e[4] = acc[kY + ab];
            e[5] = cc * acc[37] + kappa * kappa * nn * acc[9 + ab];
        }
}

constexpr int NEAR_THREADS = 128;

// FP64 flops by formula count (a fused multiply-add counted as two). An adjacent
// pair's (eta1, eta2, eta3) point (k_adj_pairs): d and r^2 (6 FMA), rsqrt, r, z (3),
// the four E_m at degree 10 (40 FMA), w rinv, w/r^3 (3), F (3 FMA), the heights and
// kernels (2 FMA, 2), eta3 products (3), sums (6 + 15 FMA): 155; an entry: D0, D1 and
// their products with the normals (20 FMA, 10), the moments (6 x 14 FMA): 218. A coincident pair's point
// (moments from the rule's table of weighted monomials): d from (s - s', t - t') (11),
// r^2 to the Yukawa single layer (11), 2 x 2 x 9 (36); by the polynomials (k_coin_poly), per
// direction: v and r^2 (24), rsqrt, r, z (3), the Yukawa moments (18 a degree), both kernels' (36).
constexpr double NEAR_FLOPS_ADJ_POINT = 155;
constexpr double NEAR_FLOPS_ADJ_ENTRY = 218;
constexpr double NEAR_FLOPS_COIN = 22 + 36;
static double coin_dir_flops(int deg) { return 63.0 + 18.0 * deg; }

// Regularised blocks of the adjacent pairs of one class: G lanes per listed pair
// (one of each two reversed ones) over the entries of the class's map, their
// moments summed over the group by a reduce-scatter, turned into corner blocks in
// shared memory by the group's lanes (a kernel each) and written for the pair and
// for its reverse rev[p] (V and D transposed, K from the K^T moments).
// Bound by the FP64 pipe (a warp instruction every 16 cycles of an SM). One xi
// evaluation instead of n (the Laplace kernels' xi sums are constants, the Yukawa
// kernels' polynomials of z) takes an (eta1, eta2, eta3) point from 4 x 59
// instructions to about 95 at n = 4; small groups keep the per-pair work (sums over
// lanes, corner blocks) to a few per cent: 8 lanes hold 12 of an edge pair's 96
// entries each, 4 lanes 8 of a vertex pair's 32; G = 32 for few pairs (adj_group).
// 38,720 triangles, n = 4: edge and vertex launches 34.0 -> 10.2 ms (with the far
// rule in the former); 2,000 triangles 1.91 -> 0.58 ms.
template <int NSS, int G>
__global__ void __launch_bounds__(NEAR_THREADS, 2)
k_adj_pairs(const double* __restrict__ verts, const int32_t* __restrict__ tris, const double* __restrict__ tgeo,
            const int4* __restrict__ pairs, const int32_t* __restrict__ list, int64_t nlist,
            const int32_t* __restrict__ rev, SSOuter tab, const __grid_constant__ Radial rad, double kappa,
            double* __restrict__ ss_out) {
    constexpr int N = G == 32 ? 64 : 56, K = N / G;  // moments after padding, and of one lane after the reduction
    struct Shared {
        AdjGeo geo;
        double mom[N];  // moments, then the corner blocks 9 k + 3 a + b
        double cc[9];   // curl products of the corners
        double sum[2];  // sums of w G_L and w G_Y
        int inv[2][3];  // frame index of original corner a
    };
    __shared__ Shared sh[NEAR_THREADS / G];
    const int lane = threadIdx.x & 31, gl = threadIdx.x % G;
    const int64_t li = (blockIdx.x * (int64_t)NEAR_THREADS + threadIdx.x) / G;
    const bool live = li < nlist;  // the last block's spare groups repeat the last pair and write nothing
    const int64_t p = list[live ? li : nlist - 1];
    const int4 pr = pairs[p];
    Shared& S = sh[threadIdx.x / G];
    const double* gA = tgeo + 16 * (int64_t)pr.x;
    const double* gB = tgeo + 16 * (int64_t)pr.y;
    const double areaA = gA[3], areaB = gB[3];
    if (gl < 3) {  // component gl of the frames' edges
        const int k = gl;
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const int perm = pr.w >> (6 * f);
            const int32_t* t = tris + 3 * (int64_t)(f ? pr.y : pr.x);
            const double q0 = verts[3 * (int64_t)t[perm & 3] + k], q1 = verts[3 * (int64_t)t[(perm >> 2) & 3] + k],
                         q2 = verts[3 * (int64_t)t[(perm >> 4) & 3] + k];
            (f ? S.geo.e1b : S.geo.e1a)[k] = q1 - q0;
            (f ? S.geo.e2b : S.geo.e2a)[k] = q2 - q1;
            S.inv[f][(perm >> (2 * k)) & 3] = k;
        }
        S.geo.na[k] = gA[k];
        S.geo.nb[k] = gB[k];
    }
    const double fc = 1.0 / (4.0 * areaA * areaB);
    for (int ab = gl; ab < 9; ab += G) {
        const double *ea = gA + 4 + 3 * (ab / 3), *eb = gB + 4 + 3 * (ab % 3);
        S.cc[ab] = fc * (ea[0] * eb[0] + ea[1] * eb[1] + ea[2] * eb[2]);
    }
    __syncwarp();
    int deg = RAD_DEG + 1;
    {   // |x - y| at xi = 1 is at most the sum of the triangles' longest distances from the shared vertex
        float z = 0.f;
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const double *e1 = f ? S.geo.e1b : S.geo.e1a, *e2 = f ? S.geo.e2b : S.geo.e2a;
            float u = 0.f, v = 0.f;
            for (int k = 0; k < 3; ++k) {
                const float c1 = (float)e1[k], c2 = (float)(e1[k] + e2[k]);
                u = fmaf(c1, c1, u);
                v = fmaf(c2, c2, v);
            }
            z += sqrtf(fmaxf(u, v));
        }
        z *= 1.0001f * (float)kappa;
        for (int d = RAD_DEG; d >= 0; --d)
            if (z <= rad.zlim[d]) deg = d;
    }
    deg = __reduce_max_sync(0xffffffffu, deg);
    double mom[54];
#pragma unroll
    for (int k = 0; k < 54; ++k) mom[k] = 0.0;
    for (int e = gl; e < tab.n; e += G) accum_entry<NSS>(mom, tab, rad, e, S.geo, kappa, deg);
    __syncwarp();
    group_sums<54, N, G>(mom, lane);
#pragma unroll
    for (int j = 0; j < K; ++j) S.mom[gl * K + j] = mom[j];
    __syncwarp();
    // the pair's Jacobian, 1/(4 pi) and the Laplace kernels' xi sums; frame moments -> corner blocks
    const double scale = (2.0 * areaA) * (2.0 * areaB) * 0.07957747154594767;
    for (int k = gl; k < 6; k += G) {
        double m[9], R[3][3], U[3][3];
        const int m0 = k == 0 ? 1 : 0;  // mu index of degree 0: G_L mu_2, K_L and K^T_L mu_1
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            const int dg = (c >= 3) + (c % 3 > 0);
            m[c] = S.mom[9 * k + c] * (k & 1 ? scale : scale * rad.mu[m0 + dg]);
        }
        if (k < 2) S.sum[k] = m[0];  // the (1, 1) moment
#pragma unroll
        for (int b = 0; b < 3; ++b) {  // mu_0 = 1 - s, mu_1 = s - t, mu_2 = t on the first frame
            R[0][b] = m[b] - m[3 + b];
            R[1][b] = m[3 + b] - m[6 + b];
            R[2][b] = m[6 + b];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {  // and on the second
            U[a][0] = R[a][0] - R[a][1];
            U[a][1] = R[a][1] - R[a][2];
            U[a][2] = R[a][2];
        }
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) S.mom[9 * k + 3 * a + b] = U[a][b];
    }
    __syncwarp();
    if (!live) return;
    const double knn = kappa * kappa * (gA[0] * gB[0] + gA[1] * gB[1] + gA[2] * gB[2]);
    const int64_t pv = rev[p];
    for (int idx = gl; idx < 108; idx += G) {
        const bool r = idx >= 54;
        const int i = r ? idx - 54 : idx, o = i / 6, k = i - 6 * o;
        const int a = r ? o % 3 : o / 3, b = r ? o / 3 : o % 3;  // corners of the first and the second triangle
        const int at = 3 * S.inv[0][a] + S.inv[1][b];
        // kernels 0..5: G_L, G_Y, K_L, K_Y, K^T_L, K^T_Y; values V_L, K_L, D_L, V_Y, K_Y, D_Y
        const int blk = (k >= 3) + (k % 3 == 1 ? (r ? 4 : 2) : 0);
        double v = S.mom[9 * blk + at];
        if (k == 2) v = S.cc[3 * a + b] * S.sum[0];
        if (k == 5) v = __fma_rn(S.cc[3 * a + b], S.sum[1], knn * v);
        ss_out[54 * (r ? pv : p) + i] = v;
    }
}

// Coincident pairs (tau, tau). The double layer vanishes (x - y lies in the
// plane of tau), and the single-layer integrand is symmetric in x and y, so
// the three regions of the coincident map whose roles are exchanged (regions
// 3..5) give the transposes of regions 0..2: integrate those and symmetrise.
// Accumulators: S_L[9], S_Y[9], sum w G_L, sum w G_Y. The far rule likewise
// over its point pairs i < j (identical points are skipped by the pair kernel).
__device__ __forceinline__ void accum_v(double* acc, double w, const double* x, const double* y, const double* lx,
                                        const double* ly, double kappa) {
    const double d0 = x[0] - y[0], d1 = x[1] - y[1], d2 = x[2] - y[2];
    const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
    const double rinv = rsqrt(r2);
    const double gl = rinv * 0.07957747154594767;  // 1 / (4 pi r)
    const double gy = exp_nonpos(-kappa * (r2 * rinv)) * gl;
    for (int a = 0; a < 3; ++a) {
        const double wa = w * lx[a];
        for (int b = 0; b < 3; ++b) {
            const double ll = wa * ly[b];
            acc[3 * a + b] += gl * ll;
            acc[9 + 3 * a + b] += gy * ll;
        }
    }
    acc[18] += w * gl;
    acc[19] += w * gy;
}

__device__ __forceinline__ void expand_coin(const double* acc, const double* tgeoA, double kappa, double* out) {
    const double nn = tgeoA[0] * tgeoA[0] + tgeoA[1] * tgeoA[1] + tgeoA[2] * tgeoA[2];
    const double f = 1.0 / (4.0 * tgeoA[3] * tgeoA[3]);
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b) {
            const double* ea = tgeoA + 4 + 3 * a;
            const double* eb = tgeoA + 4 + 3 * b;
            const double cc = f * (ea[0] * eb[0] + ea[1] * eb[1] + ea[2] * eb[2]);
            const int ab = 3 * a + b, ba = 3 * b + a;
            const double vl = acc[ab] + acc[ba], vy = acc[9 + ab] + acc[9 + ba];
            double* e = out + 6 * ab;  // the layout of expand_blocks
            e[0] = vl;
            e[1] = 0.0;
            e[2] = cc * (2.0 * acc[18]);
            e[3] = vy;
            e[4] = 0.0;
            e[5] = cc * (2.0 * acc[19]) + kappa * kappa * nn * vy;
        }
}

__global__ void __launch_bounds__(NEAR_THREADS, 4)
k_coin_pairs(const double* __restrict__ verts, const int32_t* __restrict__ tris, const double* __restrict__ tgeo,
             const int4* __restrict__ pairs, const int32_t* __restrict__ list, int64_t nlist, SSTable tab, int n4,
             Rule rule, double kappa, double* __restrict__ ss_out, double* __restrict__ far_out) {
    __shared__ TriFrame frames[NEAR_THREADS / 32];
    __shared__ double red[NEAR_THREADS / 32][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t li = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (li >= nlist) return;  // whole warps leave together
    const int64_t p = list[li];
    const int4 pr = pairs[p];
    TriFrame& A = frames[wid];
    if (lane == 0) make_frame(verts, tris, tgeo, pr.x, pr.w & 63, A);
    __syncwarp();
    const int e0 = 0;
    const double jac_ab = (2.0 * A.area) * (2.0 * A.area);
    double acc[20];
    {
        double mom[18];
        for (int k = 0; k < 18; ++k) mom[k] = 0.0;
        for (int idx = lane; idx < 3 * n4; idx += 32) accum_coin_frame(mom, tab, e0 + idx, A, kappa);
        warp_allsum<18, 32>(mom, lane, red[wid]);
        for (int k = 0; k < 18; ++k) mom[k] *= jac_ab;
        frame_to_corner(mom, A, A, acc);
        frame_to_corner(mom + 9, A, A, acc + 9);
        acc[18] = mom[0];
        acc[19] = mom[9];
    }
    const double* gA = tgeo + 16 * (int64_t)pr.x;
    if (lane == 0) expand_coin(acc, gA, kappa, ss_out + 54 * p);
    for (int k = 0; k < 20; ++k) acc[k] = 0.0;
    const int Q = rule.Q;
    for (int idx = lane; idx < Q * Q; idx += 32) {
        const int i = idx / Q, j = idx % Q;
        if (j <= i) continue;
        double x[3], y[3];
        for (int k = 0; k < 3; ++k) {
            x[k] = rule.l[i][0] * corner(A, 0, k) + rule.l[i][1] * corner(A, 1, k) + rule.l[i][2] * corner(A, 2, k);
            y[k] = rule.l[j][0] * corner(A, 0, k) + rule.l[j][1] * corner(A, 1, k) + rule.l[j][2] * corner(A, 2, k);
        }
        const double w = rule.w[i] * A.area * rule.w[j] * A.area;
        accum_v(acc, w, x, y, rule.l[i], rule.l[j], kappa);
    }
    warp_allsum<20, 32>(acc, lane, red[wid]);
    if (lane == 0) expand_coin(acc, gA, kappa, far_out + 54 * p);
}

// The same by the structure of the coincident map: in regions 0..2 x - y = rho v(eta3) with
// rho = xi eta1 eta2, so r = rho |v| takes 3 n directions per triangle, the Laplace moments
// over (xi, eta1, eta2) are constants over |v|, and the Yukawa ones polynomials of z =
// kappa |v| (as the adjacent pairs' E_m, RAD_DEG). Four lanes per triangle share the
// directions and the far rule's point pairs. Table entry
// (direction q = region n + j, moment c, k), at tab[(q (RAD_DEG + 1) + k) 9 + c]: the rule's sum
// of w mono_c rho^{k - 1} (-1)^k / k!; then 3 n pairs (s - s', t - t') of v.
// n = 4, 38,720 triangles: 1.70 -> 0.23 ms; 2,000: 223 -> 72 us. Used while kappa times the
// longest edge is within the polynomials' range; beyond, k_coin_pairs.
constexpr int COIN_STRIDE = 9 * (RAD_DEG + 1);
static_assert(sizeof(double) * 36 * (COIN_STRIDE + 2) <= (48u << 10), "the table at n = 12 in shared memory");

// a warp per (direction, moment), its lanes over the points (xi, eta1, eta2)
__global__ void k_coin_table(Gauss gq, double* __restrict__ tab) {
    const int n = gq.n, e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (e >= 3 * n * 9) return;  // whole warps
    const int q = e / 9, c = e % 9, reg = q / n, j = q % n;
    double v[RAD_DEG + 1], sx, tx, sy, ty;
#pragma unroll
    for (int k = 0; k <= RAD_DEG; ++k) v[k] = 0.0;
    for (int i = lane; i < n * n * n; i += 32) {
        const int i0 = i / (n * n), i1 = (i / n) % n, i2 = i % n;
        const double jac = ss_map(0, reg, gq.x[i0], gq.x[i1], gq.x[i2], gq.x[j], sx, tx, sy, ty);
        const double rho = gq.x[i0] * gq.x[i1] * gq.x[i2];
        const double px = c < 3 ? 1.0 : c < 6 ? sx : tx, py = c % 3 == 0 ? 1.0 : c % 3 == 1 ? sy : ty;
        double t = gq.w[i0] * gq.w[i1] * gq.w[i2] * gq.w[j] * jac * px * py / rho;
#pragma unroll
        for (int k = 0; k <= RAD_DEG; ++k) {
            v[k] += t;
            t *= rho * (-1.0 / (k + 1));
        }
    }
#pragma unroll
    for (int k = 0; k <= RAD_DEG; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane > 0) return;
#pragma unroll
    for (int k = 0; k <= RAD_DEG; ++k) tab[q * COIN_STRIDE + 9 * k + c] = v[k];
    if (c == 0) {
        ss_map(0, reg, 1.0, 1.0, 1.0, gq.x[j], sx, tx, sy, ty);
        tab[3 * n * COIN_STRIDE + 2 * q] = sx - sy;
        tab[3 * n * COIN_STRIDE + 2 * q + 1] = tx - ty;
    }
}

constexpr int COIN_THREADS = 128;
constexpr int COIN_LANES = 4;  // per triangle

__global__ void __launch_bounds__(COIN_THREADS)
k_coin_poly(const double* __restrict__ verts, const int32_t* __restrict__ tris, const double* __restrict__ tgeo,
            const int4* __restrict__ pairs, const int32_t* __restrict__ list, int64_t nlist, int n, int deg,
            const double* __restrict__ table, Rule rule, double kappa, double* __restrict__ ss_out,
            double* __restrict__ far_out) {
    extern __shared__ double tab[];
    for (int k = threadIdx.x; k < 3 * n * (COIN_STRIDE + 2); k += COIN_THREADS) tab[k] = table[k];
    __syncthreads();
    const int gl = threadIdx.x % COIN_LANES;
    const int64_t li = (blockIdx.x * (int64_t)COIN_THREADS + threadIdx.x) / COIN_LANES;
    const bool live = li < nlist;  // the last block's spare lanes repeat the last triangle and write nothing
    const int64_t p = list[live ? li : nlist - 1];
    const int32_t t = pairs[p].x;
    const double* g = tgeo + 16 * (int64_t)t;
    double c[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) c[a][k] = verts[3 * (int64_t)tris[3 * (int64_t)t + a] + k];
    double mom[18];
#pragma unroll
    for (int k = 0; k < 18; ++k) mom[k] = 0.0;
    const double* dir = tab + 3 * n * COIN_STRIDE;
    for (int q = gl; q < 3 * n; q += COIN_LANES) {
        const double ds = dir[2 * q], dt = dir[2 * q + 1];
        double r2 = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {  // v = ds e1 + dt e2, e1 = c1 - c0, e2 = c2 - c1
            const double v = __fma_rn(dt, c[2][k] - c[1][k], ds * (c[1][k] - c[0][k]));
            r2 = __fma_rn(v, v, r2);
        }
        const double rinv = rsqrt(r2), z = kappa * (r2 * rinv);
        const double* tq = tab + q * COIN_STRIDE;
        double y[9];
#pragma unroll
        for (int m = 0; m < 9; ++m) y[m] = tq[9 * deg + m];
        for (int k = deg - 1; k >= 0; --k)
#pragma unroll
            for (int m = 0; m < 9; ++m) y[m] = __fma_rn(y[m], z, tq[9 * k + m]);
#pragma unroll
        for (int m = 0; m < 9; ++m) {
            mom[m] = __fma_rn(rinv, tq[m], mom[m]);
            mom[9 + m] = __fma_rn(rinv, y[m], mom[9 + m]);
        }
    }
#pragma unroll
    for (int k = 0; k < 18; ++k)
        for (int o = COIN_LANES / 2; o > 0; o >>= 1) mom[k] += __shfl_xor_sync(0xffffffffu, mom[k], o);
    double acc[20];  // the far rule's point pairs i < j
#pragma unroll
    for (int k = 0; k < 20; ++k) acc[k] = 0.0;
    int ij = 0;
    for (int i = 0; i < rule.Q; ++i)
        for (int j = i + 1; j < rule.Q; ++j, ++ij) {
            if (ij % COIN_LANES != gl) continue;
            double x[3], y[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                x[k] = rule.l[i][0] * c[0][k] + rule.l[i][1] * c[1][k] + rule.l[i][2] * c[2][k];
                y[k] = rule.l[j][0] * c[0][k] + rule.l[j][1] * c[1][k] + rule.l[j][2] * c[2][k];
            }
            accum_v(acc, rule.w[i] * g[3] * rule.w[j] * g[3], x, y, rule.l[i], rule.l[j], kappa);
        }
#pragma unroll
    for (int k = 0; k < 20; ++k)
        for (int o = COIN_LANES / 2; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    // lane 0 writes the regularised blocks, lane 1 the far rule's
    const double scale = 4.0 * g[3] * g[3] * 0.07957747154594767;  // the Jacobians and 1/(4 pi)
    if (gl == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            double R[3][3];
            const double* mh = mom + 9 * h;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                R[0][b] = mh[b] - mh[3 + b];
                R[1][b] = mh[3 + b] - mh[6 + b];
                R[2][b] = mh[6 + b];
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                acc[9 * h + 3 * a] = scale * (R[a][0] - R[a][1]);
                acc[9 * h + 3 * a + 1] = scale * (R[a][1] - R[a][2]);
                acc[9 * h + 3 * a + 2] = scale * R[a][2];
            }
            acc[18 + h] = scale * mh[0];
        }
    }
    if (live && gl < 2) expand_coin(acc, g, kappa, (gl ? far_out : ss_out) + 54 * p);
}

// Band pairs (share no vertex, closer than the plan's band): the blocks of the
// band rule minus those of the far rule, for the pair and its reverse, one
// thread per band pair (t, s) with t < s. Points are the rules' barycentric
// combinations of the corners, in the corners' original order. Band pair q is
// stored at n_adj + q.
//
// Bound by the FP64 pipe, so by the instructions of a point pair:
//   - both rules are products of one triangle rule on each triangle, so every block
//     entry factors as sum_i w_i l_a(x_i) [sum_j w_j l_b(y_j) g(x_i, y_j)]: for each x
//     point the kernels are first summed over the y points, then added into the blocks;
//   - the points come in orbits of three with l_b(y_j) = a + (1 - 3 a) [b = j mod 3], so
//     the inner sums take two FMAs per kernel: one sum over the orbit and one per corner;
//   - (x - y) . n_y is the height of x over the plane of y's triangle, whatever y: it
//     multiplies the inner sums; (y - x) . n_x, the height of y, goes into y's weights.
//     The band rule only. The far rule, whose blocks are to cancel what the pair kernel
//     adds for the pair, takes the products d . n as the pair kernel does: y's own
//     height is the rounding of the normal, the same for all points of a triangle, so
//     that leaving it out of one side only does not average out (errors of K and T, 500
//     triangles, against 80-bit sums: 1.1e-15, with the products 1.5e-16; of the adjacent
//     pairs, by the same in k_adj_pairs and k_adj_far, 4.0 and 1.5e-16).
// 39 instructions a point pair (27 the kernels; 49 of the far rule's) and 92 an x point; 60 and
// 95 with the normal products per point pair and three FMAs per kernel. 38,720 triangles, band of 3
// radii, 6- and 3-point rules: 17.7 -> 10.0 ms (with full lanes, below). The y points of both rules are staged in
// shared memory, per thread.
constexpr int BAND_THREADS = 128;
constexpr int ADJ_FAR_THREADS = 64;
// doubles staged per y point: position and, for heights, a w and (1 - 3 a) w times its height
__host__ __device__ constexpr int staged(bool heights) { return heights ? 5 : 3; }

// FP64 flops of one band pair under a Q-point rule by formula count: per point
// pair the kernels (d 3, r^2 5, rsqrt, r, exp and its argument 17, 1/r^2, the four
// kernels 6: 33) and the sums (12 FMA); per point of either triangle its position (15) and
// height (5); per x point its weights (6), the sums' ends (18) and the block updates (54 FMA).
// Without heights 14 more a point pair (d . n twice, 5 each, and 4 products), 13 fewer an x point.
__host__ __device__ constexpr double band_flops(int Q, bool heights) {
    return Q * Q * (33.0 + 24.0 + (heights ? 0.0 : 14.0)) + Q * (40.0 + 24.0 + 108.0 - (heights ? 0.0 : 13.0));
}

// the Q points of a triangle with corners pb into ys (staged() x Q slots, NT apart), with
// HEIGHTS their heights over the plane through a0 with normal n
template <int Q, int NT, bool HEIGHTS>
__device__ __forceinline__ void stage_points(double* ys, const double (&pb)[3][3], const Rule& R, const double* a0,
                                             const double* n) {
    constexpr int YW = staged(HEIGHTS);
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        double y[3], h = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            y[k] = R.l[j][0] * pb[0][k] + R.l[j][1] * pb[1][k] + R.l[j][2] * pb[2][k];
            h += (y[k] - a0[k]) * n[k];
            ys[(YW * j + k) * NT] = y[k];
        }
        if (HEIGHTS) {
            const double a = R.l[j][Q == 1 ? 0 : (j + 1) % 3];
            ys[(YW * j + 3) * NT] = R.w[j] * a * h;
            ys[(YW * j + 4) * NT] = R.w[j] * (1.0 - 3.0 * a) * h;
        }
    }
}

// blocks: V_L, V_Y, K_L, K_Y at 0, 9, 18, 27; the reversed pair's K_L, K_Y at 38, 47 (without 1/(4 pi))
template <int Q, int NT, bool HEIGHTS>
__device__ __forceinline__ void band_pass(double* acc, const double (&pa)[3][3], const double* ys, const Rule& R,
                                          double wscale, const double* b0, const double* na, const double* nb,
                                          double kappa, double t64) {
    constexpr int ORB = Q == 1 ? 1 : 3, YW = staged(HEIGHTS);
#pragma unroll 1
    for (int i = 0; i < Q; ++i) {
        double x[3], hx = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x[k] = R.l[i][0] * pa[0][k] + R.l[i][1] * pa[1][k] + R.l[i][2] * pa[2][k];
            hx += (x[k] - b0[k]) * nb[k];
        }
        double T[6], U[6][3];
#pragma unroll
        for (int k = 0; k < 6; ++k) T[k] = U[k][0] = U[k][1] = U[k][2] = 0.0;
#pragma unroll 1
        for (int o = 0; o < Q; o += ORB) {
            const double a = R.l[o][Q == 1 ? 0 : 1], al = R.w[o] * a, be = R.w[o] * (1.0 - 3.0 * a);
            const double* yo = ys + YW * o * NT;
#pragma unroll
            for (int c = 0; c < ORB; ++c) {  // the orbit's point whose own corner is c
                const double* y = yo + YW * c * NT;
                const double d0 = x[0] - y[0], d1 = x[1] - y[NT], d2 = x[2] - y[2 * NT];
                const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
                const double rinv = rsqrt(r2);
                const double e = exp2_64th((r2 * rinv) * t64);
                const double ri2 = rinv * rinv, g = e * rinv;
                double v[6] = {rinv, g, rinv * ri2, __fma_rn(kappa, e, g) * ri2};
                double ah = al, bh = be;  // weights of the reversed pair's
                if (HEIGHTS) {
                    ah = y[3 * NT];
                    bh = y[4 * NT];
                    v[4] = v[2];
                    v[5] = v[3];
                } else {
                    const double dny = d0 * nb[0] + d1 * nb[1] + d2 * nb[2], dnx = -(d0 * na[0] + d1 * na[1] + d2 * na[2]);
                    v[4] = v[2] * dnx;
                    v[5] = v[3] * dnx;
                    v[2] *= dny;
                    v[3] *= dny;
                }
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    T[k] = __fma_rn(k < 4 ? al : ah, v[k], T[k]);
                    U[k][c] = __fma_rn(k < 4 ? be : bh, v[k], U[k][c]);
                }
            }
        }
        const double wi = wscale * R.w[i];
#pragma unroll
        for (int k = 0; k < 6; ++k)
#pragma unroll
            for (int c = 0; c < 3; ++c) U[k][c] += T[k];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double wa = wi * R.l[i][a], wh = HEIGHTS ? wa * hx : wa;
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int base = k < 4 ? 9 * k : 38 + 9 * (k - 4);
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    acc[base + 3 * a + c] = __fma_rn(k == 2 || k == 3 ? wh : wa, U[k][c], acc[base + 3 * a + c]);
            }
        }
    }
}

// the pair's blocks and its reverse's from the accumulators, the sums of w G_L and
// w G_Y following from the single-layer blocks
__device__ __forceinline__ void write_blocks(double* acc, const double* gA, const double* gB, double kappa,
                                             double* out, double* out_rev) {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        s0 += acc[k];
        s1 += acc[9 + k];
    }
    acc[36] = s0;
    acc[37] = s1;
    expand_blocks(acc, gA, gB, kappa, false, out);
    expand_blocks(acc, gA, gB, kappa, true, out_rev);
}

template <int QF, int QC>
__device__ __forceinline__ void band_pair(int64_t q, double* ys, const double* __restrict__ verts,
                                          const int32_t* __restrict__ tris, const double* __restrict__ tgeo,
                                          const int32_t* __restrict__ band_ptr, const int32_t* __restrict__ band_s,
                                          const int32_t* __restrict__ band_t, int64_t n_adj, const Rule& fine,
                                          const Rule& coarse, double kappa, double* __restrict__ ss_out,
                                          int* __restrict__ status) {
    const int32_t pt = band_t[q], ps = band_s[q];
    // the reversed pair: t among the partners of s (sorted)
    int32_t lo = band_ptr[ps], hi = band_ptr[ps + 1];
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (band_s[mid] < pt) lo = mid + 1;
        else hi = mid;
    }
    if (lo >= band_ptr[ps + 1] || band_s[lo] != pt) {  // the band lists are symmetric by construction
        atomicExch(status, PB_EMESH);
        return;
    }
    const int64_t p = n_adj + q, pr_rev = n_adj + lo;
    double* ysc = ys + staged(true) * QF * BAND_THREADS;  // the far rule's points
    const double* gA = tgeo + 16 * (int64_t)pt;
    const double* gB = tgeo + 16 * (int64_t)ps;
    const double na[3] = {gA[0], gA[1], gA[2]};
    double pa[3][3], b0[3];
    {
        double pb[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                pa[a][k] = verts[3 * (int64_t)tris[3 * (int64_t)pt + a] + k];
                pb[a][k] = verts[3 * (int64_t)tris[3 * (int64_t)ps + a] + k];
            }
        stage_points<QF, BAND_THREADS, true>(ys, pb, fine, pa[0], na);
        stage_points<QC, BAND_THREADS, false>(ysc, pb, coarse, pa[0], na);
#pragma unroll
        for (int k = 0; k < 3; ++k) b0[k] = pb[0][k];
    }
    const double nb[3] = {gB[0], gB[1], gB[2]};
    double acc[NACC_SYM];
#pragma unroll
    for (int k = 0; k < NACC_SYM; ++k) acc[k] = 0.0;
    const double area2 = gA[3] * gB[3] * 0.07957747154594767, t64 = -kappa * EXP64_PER_UNIT;  // 1 / (4 pi)
    band_pass<QF, BAND_THREADS, true>(acc, pa, ys, fine, area2, b0, na, nb, kappa, t64);
    band_pass<QC, BAND_THREADS, false>(acc, pa, ysc, coarse, -area2, b0, na, nb, kappa, t64);
    write_blocks(acc, gA, gB, kappa, ss_out + 54 * p, ss_out + 54 * pr_rev);
}

// A block takes `span` consecutive entries of the band list, of which those with t < s are
// integrated: it lists them first, so that its lanes stay full (with a thread per entry
// about a third of the lanes of an active warp had nothing to do).
constexpr int BAND_SPAN = 1024;
template <int QF, int QC>
__global__ void __launch_bounds__(BAND_THREADS, 2)
k_band_pairs(const double* __restrict__ verts, const int32_t* __restrict__ tris, const double* __restrict__ tgeo,
             const int32_t* __restrict__ band_ptr, const int32_t* __restrict__ band_s,
             const int32_t* __restrict__ band_t, int64_t n_band, int span, int64_t n_adj, Rule fine, Rule coarse,
             double kappa, double* __restrict__ ss_out, int* __restrict__ status) {
    __shared__ double ysm[(staged(true) * QF + staged(false) * QC) * BAND_THREADS];
    __shared__ uint16_t todo[BAND_SPAN];  // the block's entries with t < s, in order
    __shared__ int wcnt[BAND_THREADS / 32];
    const int64_t q0 = blockIdx.x * (int64_t)span;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int total = 0;
    for (int k0 = 0; k0 < span; k0 += BAND_THREADS) {
        const int64_t q = q0 + k0 + threadIdx.x;
        const bool mine = q < n_band && band_t[q] < band_s[q];
        const unsigned m = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) wcnt[wid] = __popc(m);
        __syncthreads();
        int at = total + __popc(m & ((1u << lane) - 1u));
        for (int w = 0; w < BAND_THREADS / 32; ++w) {
            if (w < wid) at += wcnt[w];
            total += wcnt[w];
        }
        if (mine) todo[at] = (uint16_t)(k0 + threadIdx.x);
        __syncthreads();
    }
    for (int k = threadIdx.x; k < total; k += BAND_THREADS)
        band_pair<QF, QC>(q0 + todo[k], ysm + threadIdx.x, verts, tris, tgeo, band_ptr, band_s, band_t, n_adj, fine,
                          coarse, kappa, ss_out, status);
}

// The far rule's blocks of the adjacent pairs (what the pair kernel adds for them):
// one thread per pair and its reverse, by the band pairs' sums. (As a lane's share of
// a warp per pair, 9 or 36 point pairs left most lanes idle: 260 FP64 instructions of
// a warp per pair, against 25 or 85 here. 3-point rule, 38,720 triangles: 0.44 ms.)
template <int Q>
__global__ void __launch_bounds__(ADJ_FAR_THREADS)
k_adj_far(const double* __restrict__ verts, const int32_t* __restrict__ tris, const double* __restrict__ tgeo,
          const int4* __restrict__ pairs, const int32_t* __restrict__ list, int64_t nlist,
          const int32_t* __restrict__ rev, Rule rule, double kappa, double* __restrict__ far_out) {
    __shared__ double ysm[Q * staged(false) * ADJ_FAR_THREADS];
    const int64_t li = blockIdx.x * (int64_t)ADJ_FAR_THREADS + threadIdx.x;
    if (li >= nlist) return;
    const int64_t p = list[li];
    const int4 pr = pairs[p];
    double pa[3][3], pb[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            pa[a][k] = verts[3 * (int64_t)tris[3 * (int64_t)pr.x + a] + k];
            pb[a][k] = verts[3 * (int64_t)tris[3 * (int64_t)pr.y + a] + k];
        }
    const double* gA = tgeo + 16 * (int64_t)pr.x;
    const double* gB = tgeo + 16 * (int64_t)pr.y;
    const double na[3] = {gA[0], gA[1], gA[2]}, nb[3] = {gB[0], gB[1], gB[2]};
    stage_points<Q, ADJ_FAR_THREADS, false>(ysm + threadIdx.x, pb, rule, pa[0], na);
    double acc[NACC_SYM];
#pragma unroll
    for (int k = 0; k < NACC_SYM; ++k) acc[k] = 0.0;
    band_pass<Q, ADJ_FAR_THREADS, false>(acc, pa, ysm + threadIdx.x, rule, gA[3] * gB[3] * 0.07957747154594767, pb[0], na,
                                         nb, kappa, -kappa * EXP64_PER_UNIT);
    write_blocks(acc, gA, gB, kappa, far_out + 54 * p, far_out + 54 * (int64_t)rev[p]);
}

// One warp per row i. The warp walks the contributions of the row in a fixed
// order (the triangles t of i; each one's adjacent pairs, then its band pairs;
// the trial corner b), BATCH (128) at a time: each lane finds its contributions'
// column positions (binary search in the row's sorted columns) and stages their
// six values; then the two lanes that own a position (position mod 16; three
// operators each) add the staged values for it in slot order. Every entry
// therefore sums its contributions in the walk's order, whatever the scheduling.
// Adjacent pairs (p < n_adj) hold the regularised blocks in ss and the far rule's in
// far; band pairs hold the difference in ss. The row's accumulators (6 operators and
// M) live in shared memory, maxrow entries per warp. Bound by the FP64 additions of
// the busiest lane of a batch: with 32 slots a batch, seven values and a lane per
// position, its busiest lane had nearly four times the average (38,720 triangles, band
// of 3 radii: 3.28 -> 2.00 ms).
// Batches of 32 are for rows so long that a warp's shared memory holds no more.
constexpr int ROW_OWNERS = 16;

__device__ __forceinline__ int row_lower_bound(const int32_t* c, int n, int32_t v) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (c[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// shared memory of one warp, in doubles: the staged values, positions and adjacent pairs of
// a batch; seven accumulators and the column of every entry (even: values are staged by
// 16-byte stores)
__host__ __device__ inline size_t row_warp_doubles(int batch, int maxrow) {
    return (7 * (size_t)batch + 7 * (size_t)maxrow + ((size_t)maxrow + 1) / 2 + 1) / 2 * 2;
}

template <int BATCH>
__global__ void k_near_rows(int64_t nv, int64_t nnz, int maxrow, int warps, const int32_t* __restrict__ row_ptr,
                            const int32_t* __restrict__ col, const int32_t* __restrict__ v2t_ptr,
                            const int32_t* __restrict__ v2t, const int32_t* __restrict__ tris,
                            const int32_t* __restrict__ adj_ptr, const int4* __restrict__ pairs,
                            const int32_t* __restrict__ band_ptr, const int32_t* __restrict__ band_s, int64_t n_adj,
                            const double* __restrict__ tgeo, const double* __restrict__ ss,
                            const double* __restrict__ far, double* __restrict__ val, double* __restrict__ diag) {
    static_assert(BATCH == 32 || BATCH == 128, "the owned slots are kept in two 64-bit words");
    extern __shared__ __align__(16) double rsm[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * warps + w;
    if (i >= nv) return;  // whole warps
    double* stage = rsm + (size_t)w * row_warp_doubles(BATCH, maxrow);
    int32_t* spos = (int32_t*)(stage + BATCH * 6);  // BATCH positions
    int32_t* sadj = spos + BATCH;                   // the adjacent pair of a slot on the diagonal, or -1
    double* acc = stage + BATCH * 7;
    double* accm = acc + 6 * (size_t)maxrow;
    int32_t* scol = (int32_t*)(accm + maxrow);
    const int32_t r0 = row_ptr[i];
    const int n = row_ptr[i + 1] - r0;  // <= maxrow
    for (int k = lane; k < n; k += 32) {
        scol[k] = col[r0 + k];
        accm[k] = 0.0;
    }
    for (int k = lane; k < 6 * n; k += 32) acc[k] = 0.0;
    __syncwarp();
    const int diag_pos = row_lower_bound(scol, n, (int32_t)i);
    const int owner = lane & (ROW_OWNERS - 1), half = lane / ROW_OWNERS;
    double dfull[3] = {0, 0, 0};  // the diagonal entry's full values (kept by its owner lanes)
    for (int32_t k = v2t_ptr[i]; k < v2t_ptr[i + 1]; ++k) {
        const int32_t t = v2t[k] / 3, a = v2t[k] % 3;
        const int32_t p0 = adj_ptr[t], L1 = adj_ptr[t + 1] - p0;
        const int32_t q0 = band_ptr ? band_ptr[t] : 0, L2 = band_ptr ? band_ptr[t + 1] - q0 : 0;
        const int total = 3 * (L1 + L2);
        // the triangle's own mass entries
        if (lane < 3) {
            const int pos = row_lower_bound(scol, n, tris[3 * (int64_t)t + lane]);
            accm[pos] += tgeo[16 * (int64_t)t + 3] / 12.0 * (lane == a ? 2.0 : 1.0);
        }
        for (int c0 = 0; c0 < total; c0 += BATCH) {
            const int m = min(BATCH, total - c0);
            unsigned own[BATCH / 32];
#pragma unroll
            for (int g = 0; g < BATCH / 32; ++g) {
                const int sl = 32 * g + lane, c = c0 + sl;
                int pos = -1;
                if (sl < m) {
                    double2* my = reinterpret_cast<double2*>(stage + 6 * sl);
                    const int idx = c / 3, b = c - 3 * idx, ab = 3 * a + b;
                    int at = -1;
                    if (idx < L1) {
                        const int64_t pp = p0 + idx;
                        const int32_t j = tris[3 * (int64_t)pairs[pp].y + b];
                        pos = row_lower_bound(scol, n, j);
                        if (pos == diag_pos) at = (int32_t)pp;
                        const double2* s2 = reinterpret_cast<const double2*>(ss + 54 * pp + 6 * ab);
                        const double2* f2 = reinterpret_cast<const double2*>(far + 54 * pp + 6 * ab);
#pragma unroll
                        for (int h = 0; h < 3; ++h) {
                            const double2 sv = s2[h], fv = f2[h];
                            my[h] = make_double2(sv.x - fv.x, sv.y - fv.y);
                        }
                    } else {
                        const int32_t q = q0 + idx - L1;
                        const double2* s2 = reinterpret_cast<const double2*>(ss + 54 * (n_adj + q) + 6 * ab);
                        const double2 v0 = s2[0], v1 = s2[1], v2 = s2[2];
                        pos = row_lower_bound(scol, n, tris[3 * (int64_t)band_s[q] + b]);
                        my[0] = v0;
                        my[1] = v1;
                        my[2] = v2;
                    }
                    spos[sl] = pos;
                    sadj[sl] = at;
                }
                // the slots whose position this lane owns
                const int o = pos < 0 ? -1 : pos & (ROW_OWNERS - 1);
                own[g] = 0;
#pragma unroll
                for (int q = 0; q < ROW_OWNERS; ++q) {
                    const unsigned b = __ballot_sync(0xffffffffu, o == q);
                    if (q == owner) own[g] = b;
                }
            }
            __syncwarp();
            unsigned long long lo = own[0], hi = 0;
            if (BATCH == 128) {
                lo |= (unsigned long long)own[BATCH / 32 > 1 ? 1 : 0] << 32;
                hi = own[BATCH / 32 > 2 ? 2 : 0] | (unsigned long long)own[BATCH / 32 > 3 ? 3 : 0] << 32;
            }
            while (lo | hi) {  // in slot order
                int sl;
                if (lo) {
                    sl = __ffsll((long long)lo) - 1;
                    lo &= lo - 1;
                } else {
                    sl = 63 + __ffsll((long long)hi);
                    hi &= hi - 1;
                }
                const double* st = stage + 6 * sl + 3 * half;
                double* e = acc + 6 * (size_t)spos[sl] + 3 * half;
                const int32_t at = sadj[sl];
#pragma unroll
                for (int o = 0; o < 3; ++o) e[o] += st[o];
                if (at >= 0)
#pragma unroll
                    for (int o = 0; o < 3; ++o)
                        dfull[o] += ss[54 * (int64_t)at + 6 * (3 * a + (c0 + sl) % 3) + 3 * half + o];
            }
            __syncwarp();
        }
    }
    const int map[6] = {N_VL, N_KL, N_DL, N_VY, N_KY, N_DY};
#pragma unroll
    for (int o = 0; o < 6; ++o)
        for (int k = lane; k < n; k += 32) val[map[o] * nnz + r0 + k] = acc[6 * (size_t)k + o];
    for (int k = lane; k < n; k += 32) val[N_M * nnz + r0 + k] = accm[k];
    if (owner == (diag_pos & (ROW_OWNERS - 1)))
#pragma unroll
        for (int o = 0; o < 3; ++o) diag[(half ? map[3 + o] : map[o]) * nv + i] = dfull[o];
    if (lane == 0) diag[N_M * nv + i] = accm[diag_pos];
}

// The mass matrix on its own pattern: the entries of each row whose mass value
// is not zero (exactly the vertices sharing a triangle with the row's).
__global__ void k_mass_rows(int64_t nv, int64_t nnz, int pass, const int32_t* __restrict__ row_ptr,
                            const int32_t* __restrict__ col, const double* __restrict__ val,
                            int32_t* __restrict__ cnt, const int32_t* __restrict__ mrow_ptr,
                            int32_t* __restrict__ mcol, double* __restrict__ mval) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= nv) return;
    const double* mv = val + N_M * nnz;
    int n = 0;
    for (int32_t k = row_ptr[i]; k < row_ptr[i + 1]; ++k) {
        if (mv[k] == 0.0) continue;
        if (pass) {
            mcol[mrow_ptr[i] + n] = col[k];
            mval[mrow_ptr[i] + n] = mv[k];
        }
        ++n;
    }
    if (!pass) cnt[i] = n;
}

static void free_near(pb_near* nf) {
    if (nf->val) cudaFree(nf->val);  // diag and the mass matrix are parts of it
    nf->val = nf->diag = nullptr;
    nf->mrow_ptr = nullptr;
}

// Lanes per adjacent pair: 8 for edge pairs and 4 for vertex pairs, or a whole warp for
// few pairs, where small groups leave the last of one or two waves of CTAs nearly empty
// and a pair's entries in sequence set the time. Edge and vertex launches together, us,
// small groups | whole warps, by triangles: 320: 385 | 142, 1,280: 523 | 459, 2,000: 721 |
// 628 (582 with whole warps for the edge pairs alone), 5,120: 1,558 | 1,574 (1,449),
// 8,000: 2,192 | 2,436. Lines: 16 warps per SM for edge pairs, 6 for vertex pairs.
static int adj_group(int64_t nlist, int cls, int num_sms) {
    const int g = cls == 0 ? 8 : 4, warps_per_sm = cls == 0 ? 16 : 6;
    return nlist * g < (int64_t)32 * warps_per_sm * num_sms ? 32 : g;
}

template <int G>
static void launch_adj_g(const pb_mesh* m, const int32_t* list, int64_t nlist, const SSOuter& ot, const Radial& rad,
                         double kappa, double* ss, cudaStream_t s) {
    const unsigned b = (unsigned)((nlist * G + NEAR_THREADS - 1) / NEAR_THREADS);
    if (ot.nss == 4)
        k_adj_pairs<4, G><<<b, NEAR_THREADS, 0, s>>>(m->verts, m->tris, m->tgeo, m->pairs, list, nlist, m->pair_rev, ot,
                                                     rad, kappa, ss);
    else
        k_adj_pairs<0, G><<<b, NEAR_THREADS, 0, s>>>(m->verts, m->tris, m->tgeo, m->pairs, list, nlist, m->pair_rev, ot,
                                                     rad, kappa, ss);
}

static void launch_adj(int group, const pb_mesh* m, const int32_t* list, int64_t nlist, const SSOuter& ot,
                       const Radial& rad, double kappa, double* ss, cudaStream_t s) {
    if (group == 32) launch_adj_g<32>(m, list, nlist, ot, rad, kappa, ss, s);
    else if (group == 8) launch_adj_g<8>(m, list, nlist, ot, rad, kappa, ss, s);
    else launch_adj_g<4>(m, list, nlist, ot, rad, kappa, ss, s);
}

static int build(pb_ctx* ctx, const pb_mesh* m, double kappa, pb_near* nf, cudaStream_t s, bool pooled) {
    nf->mesh = m;
    nf->kappa = kappa;
    // one allocation for what stays (values, diagonals, mass matrix on its own pattern: pointers,
    // counts, columns, total, values), one for what the build needs itself: with six, and the frees
    // of the last three, a build of 2,000 triangles with its first application took 1,480 us, now 1,270
    auto part = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
    const size_t val_bytes = part(sizeof(double) * N_VALS * m->nnz), diag_bytes = part(sizeof(double) * N_VALS * m->nv);
    const size_t mass_bytes = sizeof(int32_t) * (2 * (m->nv + 1) + m->nnz) + sizeof(double) * (m->nnz + 2) + 64;
    PB_TRY(dev_alloc((void**)&nf->val, val_bytes + diag_bytes + mass_bytes));
    nf->diag = (double*)((char*)nf->val + val_bytes);
    nf->mrow_ptr = (int32_t*)((char*)nf->diag + diag_bytes);
    int rc = PB_OK;
    {
        // coincident pairs: the table of their regularised rule
        const int nc = m->n_ss_cls[0], ne = m->n_ss_cls[1], nvx = m->n_ss_cls[2];
        const Gauss gq = gauss01(nc);
        const int n4i = nc * nc * nc * nc, ntab = 3 * n4i;
        // edge and vertex pairs: the outer entries of their maps, each with its own rule
        const int nout_e = 6 * ne * ne, nout_v = 2 * nvx * nvx;
        // the coincident pairs' polynomials, where kappa times the longest edge is within their range
        int coin_deg = RAD_DEG + 1;
        {
            const Radial lim = make_radial(gq);
            const float z = 1.0001f * (float)(kappa * m->max_edge);
            for (int d = RAD_DEG; d >= 0; --d)
                if (z <= lim.zlim[d]) coin_deg = d;
        }
        const bool poly = coin_deg <= RAD_DEG;
        const size_t coin_bytes = sizeof(double) * 3 * nc * (COIN_STRIDE + 2);
        const size_t bt = poly ? coin_bytes : sizeof(double) * SS_TABLE_ARRAYS * ntab;
        const size_t be = sizeof(double) * (size_t)SS_OUTER_ARRAYS * nout_e;
        const size_t bv = sizeof(double) * (size_t)SS_OUTER_ARRAYS * nout_v;
        const size_t ss_bytes = part(sizeof(double) * 54 * m->npairs), far_bytes = part(sizeof(double) * 54 * m->n_adj);
        CallScratch scratch;
        PB_TRY(scratch.take(ctx, ss_bytes + far_bytes + bt + be + bv, s, pooled));
        double* const ss = (double*)scratch.ptr;
        double* const far = (double*)((char*)scratch.ptr + ss_bytes);
        double* const tabm = (double*)((char*)far + far_bytes);
        double* tabe = tabm + bt / sizeof(double);
        double* tabv = tabe + be / sizeof(double);
        if (poly) k_coin_table<<<(27 * nc + 3) / 4, 128, 0, s>>>(gq, tabm);
        else k_ss_table<<<(ntab + 127) / 128, 128, 0, s>>>(gq, ntab, tabm);
        const Gauss gauss_e = gauss01(ne), gauss_v = gauss01(nvx);
        k_ss_outer<<<(nout_e + 127) / 128, 128, 0, s>>>(gauss_e, 1, nout_e, tabe);
        k_ss_outer<<<(nout_v + 127) / 128, 128, 0, s>>>(gauss_v, 2, nout_v, tabv);
        ::pb::count_launch(3);
        SSTable tab = {tabm, tabm + ntab, tabm + 2 * ntab, tabm + 3 * ntab, tabm + 4 * ntab, tabm + 5 * ntab, ntab};
        const SSOuter outer_e = {tabe, nout_e, ne, 6}, outer_v = {tabv, nout_v, nvx, 2};
        int threads = NEAR_THREADS;  // one warp per pair
        // coincident pairs, then one of each pair of reversed pairs (which also writes the other)
        unsigned bc = (unsigned)((m->n_coin * 32 + threads - 1) / threads);
        // quadrature point pairs of each kernel's rule, for the profile (formula flop counts in
        // NEAR_FLOPS_*: kernel evaluation and accumulation, a fused multiply-add counted as two)
        const double n4 = (double)n4i, Q = m->Q, Qb = m->Qr;
        if (bc && poly) {
            const double rule_pairs = 3.0 * n4 + Q * (Q - 1) / 2;
            Timer tm(ctx, PB_KERNEL_NEAR_COIN, s, m->n_coin * rule_pairs,
                     (3.0 * nc * coin_dir_flops(coin_deg) + Q * (Q - 1) / 2 * NEAR_FLOPS_COIN) / rule_pairs);
            k_coin_poly<<<(unsigned)((m->n_coin * COIN_LANES + COIN_THREADS - 1) / COIN_THREADS), COIN_THREADS, coin_bytes, s>>>(
                m->verts, m->tris, m->tgeo, m->pairs, m->pair_coin, m->n_coin, nc, coin_deg, tabm, mesh_rule(m), kappa,
                ss, far);
            tm.stop();
        } else if (bc) {
            Timer tm(ctx, PB_KERNEL_NEAR_COIN, s, m->n_coin * (3.0 * n4 + Q * (Q - 1) / 2), NEAR_FLOPS_COIN);
            k_coin_pairs<<<bc, threads, 0, s>>>(m->verts, m->tris, m->tgeo, m->pairs, m->pair_coin, m->n_coin, tab,
                                                n4i, mesh_rule(m), kappa, ss, far);
            tm.stop();
        }
        ::pb::count_launch();
        // edge-adjacent pairs (the first n_prim_edge of the primary list), then vertex-adjacent ones
        for (int cls = 0; cls < 2; ++cls) {
            const int64_t nlist = cls == 0 ? m->n_prim_edge : m->n_prim - m->n_prim_edge;
            if (nlist == 0) continue;
            const int32_t* list = m->pair_prim + (cls == 0 ? 0 : m->n_prim_edge);
            const SSOuter& ot = cls == 0 ? outer_e : outer_v;
            const Radial rad = make_radial(cls == 0 ? gauss_e : gauss_v);
            const double entries = (double)nlist * ot.n, points = entries * ot.nss;
            {
                const double rule_pairs = points * ot.nss;  // the xi points are not evaluated one by one
                Timer tm(ctx, PB_KERNEL_NEAR_ADJ, s, rule_pairs,
                         (points * NEAR_FLOPS_ADJ_POINT + entries * NEAR_FLOPS_ADJ_ENTRY) / rule_pairs);
                launch_adj(adj_group(nlist, cls, ctx->num_sms), m, list, nlist, ot, rad, kappa, ss, s);
                ::pb::count_launch();
                tm.stop();
            }
        }
        if (m->n_prim) {
            const Rule rule = mesh_rule(m);
            const unsigned gf = (unsigned)((m->n_prim + ADJ_FAR_THREADS - 1) / ADJ_FAR_THREADS);
#define PB_FAR_ARGS m->verts, m->tris, m->tgeo, m->pairs, m->pair_prim, m->n_prim, m->pair_rev, rule, kappa, far
            if (m->Q == 6) k_adj_far<6><<<gf, ADJ_FAR_THREADS, 0, s>>>(PB_FAR_ARGS);
            else if (m->Q == 3) k_adj_far<3><<<gf, ADJ_FAR_THREADS, 0, s>>>(PB_FAR_ARGS);
            else k_adj_far<1><<<gf, ADJ_FAR_THREADS, 0, s>>>(PB_FAR_ARGS);
#undef PB_FAR_ARGS
            ::pb::count_launch();
        }
        if (m->n_band) {
            Rule fine = mesh_ref_rule(m), coarse = mesh_rule(m);
            const double ppairs = 0.5 * m->n_band * (Qb * Qb + Q * Q);
            Timer tm(ctx, PB_KERNEL_NEAR_BAND, s, ppairs,
                     0.5 * m->n_band * (band_flops(m->Qr, true) + band_flops(m->Q, false)) / ppairs);
            // few entries: smaller shares, so that every SM has some
            int span = BAND_SPAN;
            while (span > 2 * BAND_THREADS && m->n_band < (int64_t)4 * ctx->num_sms * span) span /= 2;
            const unsigned gb = (unsigned)((m->n_band + span - 1) / span);
#define PB_BAND_ARGS m->verts, m->tris, m->tgeo, m->band_ptr, m->band_s, m->band_t, m->n_band, span, m->n_adj, fine, \
                     coarse, kappa, ss, m->status
            if (m->Qr == 6 && m->Q == 3) k_band_pairs<6, 3><<<gb, BAND_THREADS, 0, s>>>(PB_BAND_ARGS);
            else if (m->Qr == 6 && m->Q == 1) k_band_pairs<6, 1><<<gb, BAND_THREADS, 0, s>>>(PB_BAND_ARGS);
            else if (m->Qr == 3 && m->Q == 1) k_band_pairs<3, 1><<<gb, BAND_THREADS, 0, s>>>(PB_BAND_ARGS);
            else rc = set_error(PB_EINVAL, "band rule %d with far rule %d", m->Qr, m->Q);
#undef PB_BAND_ARGS
            tm.stop();
            ::pb::count_launch();
        }
        cudaMemsetAsync(nf->diag, 0, sizeof(double) * N_VALS * m->nv, s);
        {
            const int batch = sizeof(double) * row_warp_doubles(128, m->max_row) <= (227u << 10) ? 128 : 32;
            const size_t per_warp = sizeof(double) * row_warp_doubles(batch, m->max_row);
            const int warps = (int)std::max<size_t>(1, std::min<size_t>(8, (200u << 10) / per_warp));
            const size_t sm = per_warp * warps;
            if (sm > (227u << 10)) {
                rc = set_error(PB_EINVAL, "near pattern rows too long (%d entries) for one warp's shared memory",
                               m->max_row);
            } else {
                const auto rows = batch == 128 ? k_near_rows<128> : k_near_rows<32>;
                // the largest allowed (227 KB), not this launch's sm: builds on other host threads
                // set the same value, so none lowers it under another's launch
                cudaFuncSetAttribute((const void*)rows, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 << 10);
                rows<<<(unsigned)((m->nv + warps - 1) / warps), 32 * warps, sm, s>>>(
                    m->nv, m->nnz, m->max_row, warps, m->row_ptr, m->col, m->v2t_ptr, m->v2t, m->tris, m->adj_ptr,
                    m->pairs, m->n_band ? m->band_ptr : nullptr, m->band_s, m->n_adj, m->tgeo, ss, far, nf->val,
                    nf->diag);
                ::pb::count_launch();
            }
        }
        // the mass matrix on its own pattern
        if (rc == PB_OK) {
            const int64_t nv = m->nv, cap = m->nnz;
            int32_t* cnt = nf->mrow_ptr + (nv + 1);
            nf->mcol = cnt + (nv + 1);
            int64_t* total = (int64_t*)(((uintptr_t)(nf->mcol + cap) + 15) & ~(uintptr_t)15);
            nf->mval = (double*)(total + 1);
            const unsigned nb = (unsigned)((nv + 127) / 128);
            k_mass_rows<<<nb, 128, 0, s>>>(nv, m->nnz, 0, m->row_ptr, m->col, nf->val, cnt, nullptr, nullptr,
                                           nullptr);
            ::pb::count_launch();
            rc = device_scan(nv, cnt, nf->mrow_ptr, total, s);
            k_mass_rows<<<nb, 128, 0, s>>>(nv, m->nnz, 1, m->row_ptr, m->col, nf->val, nullptr, nf->mrow_ptr,
                                           nf->mcol, nf->mval);
            ::pb::count_launch();
        }
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        int st = 0;
        if (e == cudaSuccess && m->n_band) e = cudaMemcpy(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) rc = set_error(PB_ECUDA, "near build: %s", cudaGetErrorString(e));
        else if (st == PB_EMESH) rc = set_error(PB_EMESH, "internal: band pair without reverse");
    }
    return rc;
}

int near_build(pb_ctx* ctx, const pb_mesh* mesh, double kappa, pb_near** out, cudaStream_t s, bool pooled) {
    if (!ctx || !mesh || !out) return set_error(PB_EINVAL, "pb_near_build: NULL argument");
    if (!(kappa >= 0.0) || !std::isfinite(kappa)) return set_error(PB_EINVAL, "kappa must be >= 0");
    *out = nullptr;
    PB_CUDA(cudaSetDevice(ctx->device));
    pb_near* nf = new pb_near();
    int rc = build(ctx, mesh, kappa, nf, s, pooled);
    if (rc != PB_OK) {
        free_near(nf);
        delete nf;
        return rc;
    }
    *out = nf;
    return PB_OK;
}

__global__ void k_exp_selftest(const double* __restrict__ x, double* __restrict__ y, int64_t n) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) y[i] = exp_nonpos(x[i]);
}

}  // namespace pb

using namespace pb;

extern "C" int pb_near_build(pb_ctx* ctx, const pb_mesh* mesh, double kappa, pb_near** out, void* stream) {
    return near_build(ctx, mesh, kappa, out, (cudaStream_t)stream, true);
}

extern "C" int pb_selftest_exp(pb_ctx* ctx, const double* x, double* y, int64_t n, void* stream) {
    if (!ctx || (n > 0 && (!x || !y)) || n < 0) return set_error(PB_EINVAL, "pb_selftest_exp: bad argument");
    if (n == 0) return PB_OK;
    PB_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    k_exp_selftest<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(x, y, n);
    ::pb::count_launch();
    PB_CUDA(cudaGetLastError());
    PB_CUDA(cudaStreamSynchronize(s));
    return PB_OK;
}

extern "C" int pb_free_near(pb_near* nf) {
    if (!nf) return PB_OK;
    free_near(nf);
    delete nf;
    return PB_OK;
}
