// Pseudofermion action S = phi^+ (M^+ M)^-1 phi and its force per link.
//
// With Y solving M^+ Y = phi and X solving M X = Y, S = |Y|^2 and, for a
// link variation U_mu(x) -> exp(eps L) U_mu(x) with L in su(3),
//   dS/deps = -2 Re <Y, (dM/deps) X> = Re tr(L G_mu(x)),
// and the force is the traceless anti-Hermitian projection
//   F = TA(G) = (G - G^+)/2 - tr(G - G^+)/6.
// TA is the orthogonal projection onto su(3) for <A, B> = Re tr(A^+ B), so G
// only matters through Re tr(L G) with L anti-Hermitian: G and G' give the
// same F whenever they differ by a Hermitian matrix or a multiple of 1.  In
// particular, for any complex c and matrix B, c B^+ and -conj(c) B give the
// same F.  The kernel uses this to move U_mu(x) to the far left of every
// term and forms F = TA(U H) from one 3x3 matrix H per link.
//
// Hopping part (the forward hop at x and the backward hop at x+mu use the
// link; p the time-boundary factor of the hop):
//   G_hop = 2 kappa p [ sum_s (U (1-g_mu) X(x+mu))_s Y_s(x)^+
//                       - sum_s ((1+g_mu) X(x))_s Y_s(x+mu)^+ U^+ ]
//   H_hop = 2 kappa p sum_s [ ((1-g_mu) X(x+mu))_s Y_s(x)^+
//                             + Y_s(x+mu) ((1+g_mu) X(x))_s^+ ].
//
// Clover part: T = i csw kappa sum_{a<b} sigma_ab (x) Fhat_ab, so
//   <Y, dT X> = sum_y sum_{a<b} (i csw kappa / 8)(tr(dQ Xi) - tr(dQ^+ Xi))
// with Xi_ab(y) the traceless part of sum_{s,t} sigma_ab[s][t] X_t(y) Y_s(y)^+.
// For the link (x, mu) and each plaquette containing it -- corners c0 = x,
// c1 = x+mu, c2 = x+mu+d nu, c3 = x+d nu (d = +-1), loop links U = L0, L1,
// L2, L3 in that order -- every clover leaf based at corner c_k contributes
// through W_k(Z) = L0 ... L_{k-1} Z L_k ... L3 (k = 1..4, corner c_{k mod 4}):
//   G += c sum_k [W_k(Xi(c_k)) + W_k(Xi(c_k)^+)^+],  c = -(i csw kappa / 4) sigma
// where sigma = +1 when the loop c0 c1 c2 c3 runs counter-clockwise in the
// (a, b) = (min(mu,nu), max(mu,nu)) plane (the leaves' orientation) and -1
// when the leaves run through the link backwards.  As c is imaginary, the
// second term gives the same F as c W_k(Xi^+), so only the Hermitian
// Xh = Xi + Xi^+ enters (k_xi stores it, 9 reals per plane and site), and
//   sum_k W_k(Xh_k) = U [ Xh(c1) T + L1 (S2 Xh(x) + (Xh(c2) L2 + L2 Xh(c3)) L3) ]
// with S2 = L2 L3 and T = L1 S2.
//
// The four links of a plaquette see the same insertions, so k_force_plaq
// forms what they share once per plaquette.  Let L0 = U_a(x), L1 = U_b(x+a), V =
// U_a(x+b), W = U_b(x) be the links of the plaquette of (a, b), a < b, at x, Z0,
// Z1, Z2, Z3 = Xh_ab at x, x+a, x+a+b, x+b, and Hm(M) = (M + M^+)/2.  As c is
// imaginary, F = TA(c M) = c Hm(M) - trace, and Hm(M) = Hm(M^+).  With
//   D = L1 V^+, r = L1 Z2 V^+, Q = D W^+, C = L0 D, m = L0 (r + Z1 D)
//   P = L0 Q, P1 = Q L0, P3 = W^+ C          the loop from x, x+a and x+b
// the links get, in units of c with sigma = +1,
//   U_a(x)      Hm(G),  G = (m + C Z3) W^+ + P Z0
//   U_b(x)     -Hm(G + [Z0, P]) = -(Hm(G) + Hm(Z0 X)),  X = P - P^+
//   U_b(x+a)    Hm(((r + D Z3) W^+ + Q Z0) L0 + P1 Z1)
//   U_a(x+b)   -Hm(W^+ (m + Z0 C) + Z3 P3)
// (the two links at a corner begin the same loop in its two directions, which
// moves one insertion from its end to its front): about 2070 FP64 operations
// per plaquette, 12 400 a site, where the four insertions of each leaf pair
// taken link by link are 19 000.  (Carrying Hm(G) and X from corner to corner with
// U^+ (.) U takes 1680, but U^+ U = 1 only as far as the links are unitary: for
// links rounded to FP32 the force was off by 1.8e-8, and for exact ones its
// rounding errors were 1.7 times as large.)  k_force_link adds the six
// contributions of a link and its hopping part; two planes at a time, the
// pairs (xy, zt), (xz, yt), (yz, xt) that contain every direction once.
//
// Everything here but the first two link passes is bound by the FP64 pipe (97 %
// busy in the plaquettes, 91 % in the last link pass).  At 16^3x32 (k_xi + the
// force): 244 + 4650 us link by link; now the plaquettes 3 x 947, the link
// passes 50 + 50 + 316.

#include <math.h>

#include "wc_internal.cuh"
#include "wc_solver.cuh"
#include "wc_solver_kernels.cuh"
#include "wc_stencil.cuh"

namespace wc {


namespace {

struct M3 {
    cx<double> m[3][3];
};

__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b)
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cx<double> s = a.m[i][0] * b.m[0][j];
            s = cfma(a.m[i][1], b.m[1][j], s);
            s = cfma(a.m[i][2], b.m[2][j], s);
            r.m[i][j] = s;
        }
    return r;
}

__device__ __forceinline__ M3 dag(const M3 &a)
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) r.m[i][j] = conj(a.m[j][i]);
    return r;
}

__device__ __forceinline__ M3 link(const GaugeStore &g, int V, int mu, int x)
{
    cx<double> u[6], r2[3];
    P64::load_link(g, V, mu, x, u, r2);
    M3 r;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        r.m[0][j] = u[j];
        r.m[1][j] = u[3 + j];
        r.m[2][j] = r2[j];
    }
    return r;
}

// plane index of (a, b), a < b: xy xz xt yz yt zt
__device__ __forceinline__ int plane_of(int a, int b)
{
    return a == 0 ? b - 1 : a == 1 ? b + 1 : 5;
}

// Hermitian 3x3 matrix: real diagonal d, upper entries o = (h01, h02, h12)
struct H3 {
    double d[3];
    cx<double> o[3];
};

// off-diagonal entry (i, k), i != k (constants once the callers are unrolled)
__device__ __forceinline__ cx<double> hoff(const H3 &h, int i, int k)
{
    const cx<double> v = h.o[i + k - 1];
    return i < k ? v : conj(v);
}

// acc + H B
__device__ __forceinline__ void fma_hm(const H3 &h, const M3 &b, M3 &acc)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cx<double> s = acc.m[i][j];
            s.re = fma(h.d[i], b.m[i][j].re, s.re);
            s.im = fma(h.d[i], b.m[i][j].im, s.im);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k != i) s = cfma(hoff(h, i, k), b.m[k][j], s);
            acc.m[i][j] = s;
        }
}

// acc + A H
__device__ __forceinline__ void fma_mh(const M3 &a, const H3 &h, M3 &acc)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cx<double> s = acc.m[i][j];
            s.re = fma(a.m[i][j].re, h.d[j], s.re);
            s.im = fma(a.m[i][j].im, h.d[j], s.im);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k != j) s = cfma(a.m[i][k], hoff(h, k, j), s);
            acc.m[i][j] = s;
        }
}

__device__ __forceinline__ M3 zero3()
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) r.m[i][j] = mkc(0.0, 0.0);
    return r;
}

__device__ __forceinline__ M3 mul_dag(const M3 &a, const M3 &b) { return mul(a, dag(b)); }

// off-diagonal entry q of an H3 / X3: rows and columns
__device__ __forceinline__ int off_row(int q) { return q == 2 ? 1 : 0; }
__device__ __forceinline__ int off_col(int q) { return q == 0 ? 1 : 2; }

// anti-Hermitian 3x3 matrix: i d on the diagonal, upper entries o
struct X3 {
    double d[3];
    cx<double> o[3];
};

__device__ __forceinline__ H3 operator+(const H3 &a, const H3 &b)
{
    H3 r;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r.d[k] = a.d[k] + b.d[k];
        r.o[k] = a.o[k] + b.o[k];
    }
    return r;
}

__device__ __forceinline__ H3 operator-(const H3 &a, const H3 &b)
{
    H3 r;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r.d[k] = a.d[k] - b.d[k];
        r.o[k] = a.o[k] - b.o[k];
    }
    return r;
}

// entry (i, j) of X, i != j
__device__ __forceinline__ cx<double> xoff(const X3 &x, int i, int j)
{
    const cx<double> v = x.o[i + j - 1];
    return i < j ? v : -conj(v);
}

// 2 Hm(E W^+ + P Z)
__device__ __forceinline__ H3 herm2(const M3 &e, const M3 &w, const M3 &p, const H3 &z)
{
    // entry (i, j) of E W^+ + P Z
    const auto at = [&](int i, int j) {
        cx<double> s = mkc(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < 3; ++k) s = cfma_conj(w.m[j][k], e.m[i][k], s);
        s.re = fma(p.m[i][j].re, z.d[j], s.re);
        s.im = fma(p.m[i][j].im, z.d[j], s.im);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k != j) s = cfma(p.m[i][k], hoff(z, k, j), s);
        return s;
    };
    H3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) s = fma(e.m[i][k].re, w.m[i][k].re, fma(e.m[i][k].im, w.m[i][k].im, s));
        s = fma(p.m[i][i].re, z.d[i], s);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k != i) {
                const cx<double> h = hoff(z, k, i);
                s = fma(p.m[i][k].re, h.re, fma(-p.m[i][k].im, h.im, s));
            }
        r.d[i] = 2.0 * s;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = off_row(q), j = off_col(q);
        r.o[q] = at(i, j) + conj(at(j, i));
    }
    return r;
}

// 2 Hm(Z X)
__device__ __forceinline__ H3 herm2_zx(const H3 &z, const X3 &x)
{
    H3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double s = 0.0;   // Re (Z X)_ii: Z_ii times the imaginary X_ii drops out
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k != i) {
                const cx<double> h = hoff(z, i, k), a = xoff(x, k, i);
                s = fma(h.re, a.re, fma(-h.im, a.im, s));
            }
        r.d[i] = 2.0 * s;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = off_row(q), j = off_col(q), k = 3 - i - j;
        const auto at = [&](int a, int b) {
            const cx<double> xab = xoff(x, a, b), zab = hoff(z, a, b);
            cx<double> s = mkc(z.d[a] * xab.re, z.d[a] * xab.im);
            s.re = fma(-zab.im, x.d[b], s.re);   // Z_ab i X_bb
            s.im = fma(zab.re, x.d[b], s.im);
            return cfma(hoff(z, a, k), xoff(x, k, b), s);
        };
        r.o[q] = at(i, j) + conj(at(j, i));
    }
    return r;
}

__device__ __forceinline__ void store_h3(double *p, int V, int x, const H3 &h)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) p[(size_t)k * V + x] = h.d[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[(size_t)(3 + 2 * k) * V + x] = h.o[k].re;
        p[(size_t)(4 + 2 * k) * V + x] = h.o[k].im;
    }
}

__device__ __forceinline__ H3 load_h3(const double *p, int V, int x)
{
    H3 h;
#pragma unroll
    for (int k = 0; k < 3; ++k) h.d[k] = __ldg(p + (size_t)k * V + x);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        h.o[k] = mkc(__ldg(p + (size_t)(3 + 2 * k) * V + x), __ldg(p + (size_t)(4 + 2 * k) * V + x));
    return h;
}

// Xh_ab(y) = Xi + Xi^+ for the six planes, Xi the traceless part of
// sum_{s,t} sigma_ab[s][t] X_t(y) Y_s(y)^+.  Layout [6][9][V] doubles:
// h00 h11 h22, re/im of h01, h02, h12.  On spin pair 0 / 1 sigma is (s1, s2, s3
// the Pauli matrices) xy -s3, xz s2, xt -/+s1, yz -s1, yt -/+s2, zt -/+s3: the
// Hermitian parts of the three Pauli sums of each pair, added and subtracted.
__global__ void __launch_bounds__(64) k_xi(Geom g, const double2 *X, const double2 *Y, double *xh)
{
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= g.V) return;
    const int V = g.V;
    H3 s[2][3];   // [pair][Pauli]: S + S^+
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        cx<double> x[6], w[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 u = __ldg(X + (size_t)(6 * b + k) * V + y), v = __ldg(Y + (size_t)(6 * b + k) * V + y);
            x[k] = mkc(u.x, u.y);
            w[k] = mkc(v.x, v.y);
        }
        // O_st = X_t Y_s^+
        const auto o = [&](int sp, int t, int i, int j) { return cmul_conj(w[3 * sp + j], x[3 * t + i]); };
        const auto osub = [&](int sp, int t, int i, int j, cx<double> a) { return cfma_conj(w[3 * sp + j], -x[3 * t + i], a); };
#pragma unroll
        for (int q = 0; q < 6; ++q) {   // the diagonal, then the three pairs (i, j)
            const int i = q < 3 ? q : off_row(q - 3), j = q < 3 ? q : off_col(q - 3);
            const cx<double> a01 = o(0, 1, i, j), a10 = o(1, 0, i, j), a3 = osub(1, 1, i, j, o(0, 0, i, j));
            const cx<double> p1 = a01 + a10, p2 = times_i(a10 - a01);
            if (q < 3) {
                s[b][0].d[q] = 2.0 * p1.re;
                s[b][1].d[q] = 2.0 * p2.re;
                s[b][2].d[q] = 2.0 * a3.re;
            } else {
                const cx<double> c01 = o(0, 1, j, i), c10 = o(1, 0, j, i), c3 = osub(1, 1, j, i, o(0, 0, j, i));
                s[b][0].o[q - 3] = p1 + conj(c01 + c10);
                s[b][1].o[q - 3] = p2 + conj(times_i(c10 - c01));
                s[b][2].o[q - 3] = a3 + conj(c3);
            }
        }
    }
    // planes xy xz xt yz yt zt: Pauli matrix and the signs of the two pairs
    constexpr int pauli[6] = {2, 1, 0, 0, 1, 2};
    constexpr double s0[6] = {-1.0, 1.0, -1.0, -1.0, -1.0, -1.0}, s1[6] = {-1.0, 1.0, 1.0, -1.0, 1.0, 1.0};
#pragma unroll
    for (int pl = 0; pl < 6; ++pl) {
        const H3 &a = s[0][pauli[pl]], &c = s[1][pauli[pl]];
        H3 h;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            h.d[k] = s0[pl] * a.d[k] + s1[pl] * c.d[k];
            h.o[k] = mkc(s0[pl] * a.o[k].re + s1[pl] * c.o[k].re, s0[pl] * a.o[k].im + s1[pl] * c.o[k].im);
        }
        const double t = (1.0 / 3.0) * (h.d[0] + h.d[1] + h.d[2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) h.d[k] -= t;
        store_h3(xh + (size_t)pl * 9 * V, V, y, h);
    }
}

// Where the contributions of the plaquettes of two planes go: [9][V] for each
// plane and each of its four slots.
struct ForceSlots {
    double *at[2][4];
};

// The contributions of one plaquette to its four links (see above), twice
// each, in units of c: slot 0 U_a(x), 1 U_b(x), 2 U_b(x+a), 3 U_a(x+b), the signs of
// 1 and 3 left to k_force_link, at the index of x.  Plane (planes.x, planes.y) for blockIdx.y = 0, (planes.z,
// planes.w) for 1.
__global__ void __launch_bounds__(64) k_force_plaq(Geom g, GaugeStore G, const double *xh, int4 planes, ForceSlots ws)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V) return;
    const int V = g.V;
    const int a = blockIdx.y ? planes.z : planes.x, b = blockIdx.y ? planes.w : planes.y;
    const double *xp = xh + (size_t)plane_of(a, b) * 9 * V;
    int c[4];
    site_coords(g, x, c);
    const int xa = wc_idx(c[a] == g.L[a] - 1 ? x - (g.L[a] - 1) * g.stride[a] : x + g.stride[a], V);
    const int xb = wc_idx(c[b] == g.L[b] - 1 ? x - (g.L[b] - 1) * g.stride[b] : x + g.stride[b], V);
    const int xab = wc_idx(c[b] == g.L[b] - 1 ? xa - (g.L[b] - 1) * g.stride[b] : xa + g.stride[b], V);
    const auto put = [&](int slot, const H3 &h) { store_h3(ws.at[blockIdx.y][slot], V, x, h); };
    M3 D, r;
    {
        const M3 L1 = link(G, V, b, xa), Vd = dag(link(G, V, a, xb));
        M3 s = zero3();
        fma_mh(L1, load_h3(xp, V, xab), s);
        r = mul(s, Vd);
        D = mul(L1, Vd);
    }
    const M3 L0 = link(G, V, a, x), W = link(G, V, b, x);
    const M3 Q = mul_dag(D, W);
    {
        M3 n = r;
        fma_mh(D, load_h3(xp, V, xb), n);
        n = mul_dag(n, W);
        fma_mh(Q, load_h3(xp, V, x), n);
        put(2, herm2(n, dag(L0), mul(Q, L0), load_h3(xp, V, xa)));
    }
    fma_hm(load_h3(xp, V, xa), D, r);
    const M3 m = mul(L0, r), C = mul(L0, D);
    {
        M3 e = m;
        fma_mh(C, load_h3(xp, V, xb), e);
        const M3 P = mul(L0, Q);
        X3 X;
#pragma unroll
        for (int i = 0; i < 3; ++i) X.d[i] = 2.0 * P.m[i][i].im;
#pragma unroll
        for (int q = 0; q < 3; ++q) X.o[q] = P.m[off_row(q)][off_col(q)] - conj(P.m[off_col(q)][off_row(q)]);
        const H3 Z0 = load_h3(xp, V, x), H = herm2(e, W, P, Z0);
        put(0, H);
        put(1, H + herm2_zx(Z0, X));
    }
    {
        M3 y = m;
        fma_hm(load_h3(xp, V, x), C, y);
        put(3, herm2(dag(y), dag(W), dag(mul(dag(W), C)), load_h3(xp, V, xb)));
    }
}

// two-spinor of (1 + S g_mu) psi at site x of an FP64 field
template <int MU, int S>
__device__ __forceinline__ void half_spinor(const double2 *f, int V, int x, cx<double> h[6])
{
    cx<double> p[12];
    P64::load_spinor(f, nullptr, V, x, p);
    project<MU, S>(p, h);
}

// Z += sum over two spins of a_s b_s^+
__device__ __forceinline__ void fma_outer2(const cx<double> a[6], const cx<double> b[6], M3 &z)
{
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = 0; q < 3; ++q) z.m[p][q] = cfma_conj(b[3 * s + q], a[3 * s + p], z.m[p][q]);
}

// sum_s [((1-g) X(x+mu))_s Y_s(x)^+ + Y_s(x+mu) ((1+g) X(x))_s^+]: 1 -+ g is
// Hermitian and twice a projector, so the sums over four spins are those over
// the two spins of both projected spinors
template <int MU>
__device__ __forceinline__ M3 hop_outer(const double2 *X, const double2 *Y, int V, int x, int xf)
{
    M3 z = zero3();
    cx<double> a[6], b[6];
    half_spinor<MU, -1>(X, V, xf, a);
    half_spinor<MU, -1>(Y, V, x, b);
    fma_outer2(a, b, z);
    half_spinor<MU, +1>(Y, V, xf, a);
    half_spinor<MU, +1>(X, V, x, b);
    fma_outer2(a, b, z);
    return z;
}

// Link (x, mu), mu = blockIdx.y: the contributions of the planes of this step
// added to those parked in F (9 doubles of a link's 18); with LAST, the hopping
// part too and F = TA(G) in the canonical layout [V][4][3][3].
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(64) k_force_link(Geom g, GaugeStore G, const double2 *X, const double2 *Y, int4 planes,
                                                   ForceSlots ws, double kappa, double csw, double2 *F)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, mu = blockIdx.y;
    if (x >= g.V) return;
    const int V = g.V;
    int c[4];
    site_coords(g, x, c);
    H3 h = {};
    double2 *out = F + ((size_t)x * 4 + mu) * 9;
    if (csw != 0.0) {
        // the plane of this step that contains mu: (a, b) with a = mu or b = mu
        const int second = mu == planes.z || mu == planes.w;
        const int a = second ? planes.z : planes.x, b = second ? planes.w : planes.y;
        const int nu = mu == a ? b : a;
        const int xd = wc_idx(c[nu] == 0 ? x + (g.L[nu] - 1) * g.stride[nu] : x - g.stride[nu], V);
        h = load_h3(ws.at[second][mu == a ? 0 : 2], V, mu == a ? x : xd) -
            load_h3(ws.at[second][mu == a ? 3 : 1], V, mu == a ? xd : x);
        if (!FIRST) {
            H3 p;
            const double2 d0 = out[0], d1 = out[1];
            p.d[0] = d0.x, p.d[1] = d0.y, p.d[2] = d1.x;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double2 v = out[2 + k];
                p.o[k] = mkc(v.x, v.y);
            }
            h = h + p;
        }
    }
    if (!LAST) {
        out[0] = make_double2(h.d[0], h.d[1]);
        out[1] = make_double2(h.d[2], 0.0);
#pragma unroll
        for (int k = 0; k < 3; ++k) out[2 + k] = make_double2(h.o[k].re, h.o[k].im);
        return;
    }
    const bool wrap = c[mu] == g.L[mu] - 1;
    const int xf = wc_idx(wrap ? x - (g.L[mu] - 1) * g.stride[mu] : x + g.stride[mu], V);
    const double k2 = kappa * ((mu == 3 && wrap) ? (double)g.tbc : 1.0);
    M3 z;
    if (mu == 0) z = hop_outer<0>(X, Y, V, x, xf);
    else if (mu == 1) z = hop_outer<1>(X, Y, V, x, xf);
    else if (mu == 2) z = hop_outer<2>(X, Y, V, x, xf);
    else z = hop_outer<3>(X, Y, V, x, xf);
    const M3 u = mul(link(G, V, mu, x), z);
    // G - G^+ = 2 kappa p (U z - (U z)^+) + 2 c H, H = h / 2, c = -i csw kappa / 4
    const double cb = -csw * kappa / 8.0;
    const double f0 = fma(cb, h.d[0], 2.0 * k2 * u.m[0][0].im), f1 = fma(cb, h.d[1], 2.0 * k2 * u.m[1][1].im),
                 f2 = fma(cb, h.d[2], 2.0 * k2 * u.m[2][2].im);
    const double t = (1.0 / 3.0) * (f0 + f1 + f2);
    out[0] = make_double2(0.0, f0 - t);
    out[4] = make_double2(0.0, f1 - t);
    out[8] = make_double2(0.0, f2 - t);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = off_row(q), j = off_col(q);
        const cx<double> d = u.m[i][j] - conj(u.m[j][i]);
        const cx<double> v = mkc(fma(k2, d.re, -cb * h.o[q].im), fma(k2, d.im, cb * h.o[q].re));
        out[3 * i + j] = make_double2(v.re, v.im);
        out[3 * j + i] = make_double2(-v.re, v.im);
    }
}

bool is_device_ptr(const void *p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

// Slots in the work vectors of a solver state, which are free between solves:
// from slot number `have` on, up to eight in all; returns the new number.  The
// even-odd and FP64 solvers leave all eight, so that a force takes no more
// memory than Xh (432 B a site; with slots of its own it took 1008).
static int borrow_slots(const SolverState &S, size_t bytes, double **slot, int have)
{
    for (const wc_field_s *f : S.work) {
        if (!f) continue;
        char *p = static_cast<char *>(f->data);
        for (size_t left = spinor_bytes(f->prec, f->lat->g.V); left >= bytes && have < 8; left -= bytes, p += bytes)
            slot[have++] = reinterpret_cast<double *>(p);
    }
    return have;
}

// F from X, Y (FP64 fields) into the canonical force layout at dst (device).
wc_status force_from_solutions(wc_lattice lat, wc_field X, wc_field Y, double2 *dst)
{
    const int V = lat->g.V;
    cudaStream_t s = lat->stream;
    const double2 *x = static_cast<const double2 *>(X->data), *y = static_cast<const double2 *>(Y->data);
    // Xh of the six planes, and the slots that idle solver vectors do not give
    ForceSlots ws{};
    const size_t slot_bytes = sizeof(double) * 9 * (size_t)V;
    int have = borrow_slots(lat->st, slot_bytes, &ws.at[0][0], 0);
    if (lat->half) have = borrow_slots(lat->half->st, slot_bytes, &ws.at[0][0], have);
    double *xh = nullptr;
    wc_status st = check_cuda(lat, cudaMalloc(&xh, sizeof(double) * 54 * (size_t)V + slot_bytes * (8 - have)),
                              "cudaMalloc(force)");
    if (st != WC_OK) return st;
    for (int k = have; k < 8; ++k) (&ws.at[0][0])[k] = xh + (size_t)(54 + 9 * (k - have)) * V;
    const int4 pair[3] = {make_int4(0, 1, 2, 3), make_int4(0, 2, 1, 3), make_int4(1, 2, 0, 3)};
    const unsigned blocks = (V + 63) / 64;
    const bool clover = lat->csw != 0.0;
    if (clover) k_xi<<<blocks, 64, 0, s>>>(lat->g, x, y, xh);
    for (int p = clover ? 0 : 2; p < 3; ++p) {
        if (clover) k_force_plaq<<<dim3(blocks, 2), 64, 0, s>>>(lat->g, lat->gauge, xh, pair[p], ws);
        const auto kern = p == 2 ? (clover ? k_force_link<false, true> : k_force_link<true, true>)
                                 : p == 0 ? k_force_link<true, false> : k_force_link<false, false>;
        kern<<<dim3(blocks, 4), 64, 0, s>>>(lat->g, lat->gauge, x, y, pair[p], ws, lat->kappa, lat->csw, dst);
    }
    st = check_launch(lat, "force");
    cudaStreamSynchronize(s);
    cudaFree(xh);
    return st;
}

}  // namespace wc

using namespace wc;

namespace wc {
namespace {

// out = scale * F U per link (3x3 complex, canonical [4V][3][3] order)
__global__ void k_force_times_links(long long nlinks, const double2 *F, const double2 *U, double scale, double2 *out)
{
    const long long l = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (l >= nlinks) return;
    const double2 *f = F + 9 * l, *u = U + 9 * l;
    cx<double> a[9], b[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        a[k] = mkc(f[k].x, f[k].y);
        b[k] = mkc(u[k].x, u[k].y);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            cx<double> acc = a[3 * i] * b[j];
            acc = cfma(a[3 * i + 1], b[3 + j], acc);
            acc = cfma(a[3 * i + 2], b[6 + j], acc);
            out[9 * l + 3 * i + j] = make_double2(scale * acc.re, scale * acc.im);
        }
}

}  // namespace
}  // namespace wc

extern "C" {

wc_status wc_force_times_links(wc_lattice lat, const double *force, const double *U, double scale, double *out)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (!force || !U || !out) return set_error(lat, WC_ERR_ARG, "NULL argument");
    if (!is_device_ptr(force) || !is_device_ptr(U) || !is_device_ptr(out))
        return set_error(lat, WC_ERR_ARG, "force, U and out must be device pointers");
    const long long n = 4LL * lat->g.V;
    k_force_times_links<<<(unsigned)((n + 255) / 256), 256, 0, lat->stream>>>(
        n, reinterpret_cast<const double2 *>(force), reinterpret_cast<const double2 *>(U), scale,
        reinterpret_cast<double2 *>(out));
    return check_cuda(lat, cudaGetLastError(), "force_times_links");
}

wc_status wc_action_force(wc_lattice lat, wc_field phi, double *S_out, double *force, const wc_solve_params *p)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (!phi || !p || !S_out || !force) return set_error(lat, WC_ERR_ARG, "NULL argument");
    if (phi->lat != lat || phi->prec != WC_F64) return set_error(lat, WC_ERR_ARG, "phi must be an FP64 field of lat");
    wc_field X = nullptr, Y = nullptr;
    wc_status st = wc_field_create(lat, WC_F64, &Y);
    if (st == WC_OK) st = wc_field_create(lat, WC_F64, &X);
    if (st == WC_OK) st = check_solve_args(lat, Y, phi, p);
    wc_solve_info info{};
    if (st == WC_OK) st = bicgstab(lat, 1, Y, phi, *p, &info);   // M^+ Y = phi
    if (st == WC_OK) st = bicgstab(lat, 0, X, Y, *p, &info);     // M X = Y
    double S = 0.0;
    if (st == WC_OK) st = reduce_norm2(lat, Y, &S);
    if (st == WC_OK) {
        const int V = lat->g.V;
        const size_t bytes = sizeof(double2) * 36 * (size_t)V;
        if (is_device_ptr(force)) {
            st = force_from_solutions(lat, X, Y, reinterpret_cast<double2 *>(force));
        } else {
            double2 *tmp = nullptr;
            st = check_cuda(lat, cudaMalloc(&tmp, bytes), "cudaMalloc(force)");
            if (st == WC_OK) st = force_from_solutions(lat, X, Y, tmp);
            if (st == WC_OK) st = check_cuda(lat, cudaMemcpy(force, tmp, bytes, cudaMemcpyDeviceToHost), "copy force");
            cudaFree(tmp);
        }
    }
    if (st == WC_OK) *S_out = S;
    wc_field_destroy(X);
    wc_field_destroy(Y);
    return st;
}

}  // extern "C"
