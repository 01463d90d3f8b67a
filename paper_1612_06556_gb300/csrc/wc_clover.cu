// Clover term A = 1 + T of the loaded links (FP64 arithmetic).
//
// Fhat_munu(x) = (1/8)[(Q - Q^+) - tr(Q - Q^+)/3], Q the sum of the four
// plaquette leaves at x.  The four leaves that pass through one plaquette
// are the same loop begun at its four corners.  With its two-link paths
//   A = U_mu(x) U_nu(x+mu)         B = U_nu(x) U_mu(x+nu)
//   C = U_nu(x+mu) U_mu(x+nu)^+    D = U_mu(x)^+ U_nu(x)
// they are
//   at x  A B^+     at x + mu + nu  B^+ A     at x + mu  C D^+     at x + nu  D^+ C
// of which only the anti-Hermitian part X = P - P^+ (9 reals) is wanted: four
// products of 108 FP64 operations and four X of 96 per plaquette, 816 a site and
// plane, against 12 products of 108 for the four leaves taken site by site.
// (Forming X once and carrying it to the other corners, U^+ X U, takes 738, but
// U^+ U = 1 only as far as the links are unitary: for links rounded to FP32 the
// term was off by 4e-9, and its rounding errors were a fifth larger.)  The
// build is bound by the FP64 pipe (one warp instruction per 64 cycles on
// each of its four units per SM; 95 % busy): at 16^3x32 3 x 369 us in k_leaves,
// 1929 us for the whole build site by site.
//
// k_leaves writes the four X per plaquette at the index of x, plane
// by plane; k_gather adds the leaves that arrive at a site (fixed order)
// and forms the clover entries; two planes per pass, since the entries need
// the pairs (xy, zt), (yz, xt), (xz, yt).  The leaves of two planes are 576 B
// a site, the size of the double-FP32 copy of the clover term, which is
// written last and holds them until then.  One thread per
// (site, plane, pair of leaves) in k_leaves: twelve times as many warps as
// sites / 32, which is what small lattices need to reach all FP64 units.
#include "wc_internal.cuh"

namespace wc {

namespace {

struct M3 {
    cx<double> m[3][3];
};

// anti-Hermitian 3x3 matrix: i d on the diagonal, upper entries (0,1) (0,2)
// (1,2) in o
struct X3 {
    double d[3];
    cx<double> o[3];
};

__device__ __forceinline__ M3 load_u(const GaugeStore &g, int V, int mu, int x)
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

__device__ __forceinline__ M3 m3_mul(const M3 &a, const M3 &b)
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

__device__ __forceinline__ M3 m3_dag(const M3 &a)
{
    M3 r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) r.m[i][j] = conj(a.m[j][i]);
    return r;
}

// a * conj(b), accumulated
__device__ __forceinline__ cx<double> mul_conj(cx<double> a, cx<double> b, cx<double> acc)
{
    acc.re = fma(a.re, b.re, acc.re);
    acc.re = fma(a.im, b.im, acc.re);
    acc.im = fma(a.im, b.re, acc.im);
    acc.im = fma(-a.re, b.im, acc.im);
    return acc;
}

// P - P^+ of P = A B^+
__device__ __forceinline__ X3 anti_of_abdag(const M3 &a, const M3 &b)
{
    X3 x;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double s = 0.0;   // Im P_ii
#pragma unroll
        for (int k = 0; k < 3; ++k) s = fma(a.m[i][k].im, b.m[i][k].re, fma(-a.m[i][k].re, b.m[i][k].im, s));
        x.d[i] = 2.0 * s;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int i = q == 2 ? 1 : 0, j = q == 0 ? 1 : 2;
        cx<double> u = mkc(0.0, 0.0), l = u;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            u = mul_conj(a.m[i][k], b.m[j][k], u);
            l = mul_conj(a.m[j][k], b.m[i][k], l);
        }
        x.o[q] = u - conj(l);
    }
    return x;
}

// scratch of one plane: double [4 corners][9][V]
__device__ __forceinline__ void store_x(double *w, int V, int x, const X3 &a)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) w[(size_t)k * V + x] = a.d[k];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        w[(size_t)(3 + 2 * k) * V + x] = a.o[k].re;
        w[(size_t)(4 + 2 * k) * V + x] = a.o[k].im;
    }
}

__device__ __forceinline__ void add_x(const double *w, int V, int x, X3 &a)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) a.d[k] += __ldg(w + (size_t)k * V + x);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a.o[k].re += __ldg(w + (size_t)(3 + 2 * k) * V + x);
        a.o[k].im += __ldg(w + (size_t)(4 + 2 * k) * V + x);
    }
}

__device__ __forceinline__ int up(const Geom &g, int x, const int c[4], int mu)
{
    return wc_idx(c[mu] == g.L[mu] - 1 ? x - (g.L[mu] - 1) * g.stride[mu] : x + g.stride[mu], g.V);
}

__device__ __forceinline__ int down(const Geom &g, int x, const int c[4], int mu)
{
    return wc_idx(c[mu] == 0 ? x + (g.L[mu] - 1) * g.stride[mu] : x - g.stride[mu], g.V);
}

// Leaves of the plaquettes of plane (planes.x, planes.y) (blockIdx.y = 0) or
// (planes.z, planes.w) (blockIdx.y = 1): A B^+ and B^+ A (blockIdx.z = 0), or C D^+
// and D^+ C (blockIdx.z = 1).  The two pairs in one thread take 254 registers,
// or 1.8 KB of spills at 168.
__global__ void __launch_bounds__(64) k_leaves(Geom g, GaugeStore G, int4 planes, double *ws)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V) return;
    const int V = g.V;
    const int mu = blockIdx.y ? planes.z : planes.x, nu = blockIdx.y ? planes.w : planes.y;
    double *w = ws + (size_t)blockIdx.y * 36 * V;
    int c[4];
    site_coords(g, x, c);
    const int xm = up(g, x, c, mu), xn = up(g, x, c, nu);
    M3 a, b;
    if (blockIdx.z == 0) {
        a = m3_mul(load_u(G, V, mu, x), load_u(G, V, nu, xm));
        b = m3_mul(load_u(G, V, nu, x), load_u(G, V, mu, xn));
    } else {
        a = m3_mul(load_u(G, V, nu, xm), m3_dag(load_u(G, V, mu, xn)));
        b = m3_mul(m3_dag(load_u(G, V, mu, x)), load_u(G, V, nu, x));
    }
    store_x(w + (size_t)(blockIdx.z == 0 ? 0 : 9) * V, V, x, anti_of_abdag(a, b));
    store_x(w + (size_t)(blockIdx.z == 0 ? 27 : 18) * V, V, x, anti_of_abdag(m3_dag(b), m3_dag(a)));
}

// 8 Fhat of plane (mu, nu) at x from its leaves
__device__ __forceinline__ X3 gather(const Geom &g, const double *w, int x, const int c[4], int mu, int nu)
{
    const int V = g.V;
    X3 f = {};
    const int xm = down(g, x, c, mu), xn = down(g, x, c, nu);
    add_x(w, V, x, f);
    add_x(w + (size_t)9 * V, V, xm, f);
    add_x(w + (size_t)18 * V, V, xn, f);
    add_x(w + (size_t)27 * V, V, down(g, xm, c, nu), f);
    const double t = (1.0 / 3.0) * (f.d[0] + f.d[1] + f.d[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) f.d[k] -= t;
    return f;
}

// entry (i, j) of X
__device__ __forceinline__ cx<double> entry(const X3 &x, int i, int j)
{
    if (i == j) return mkc(0.0, x.d[i]);
    const cx<double> v = x.o[i + j - 1];
    return i < j ? v : -conj(v);
}

// s a + t b
__device__ __forceinline__ X3 combine(double s, const X3 &a, double t, const X3 &b)
{
    X3 r;
#pragma unroll
    for (int k = 0; k < 3; ++k) r.d[k] = fma(s, a.d[k], t * b.d[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        r.o[k] = mkc(fma(s, a.o[k].re, t * b.o[k].re), fma(s, a.o[k].im, t * b.o[k].im));
    return r;
}

// In the chiral basis sigma_munu restricted to spin pair b is (eta = -1 for
// b = 0, +1 for b = 1):
//   sigma_xy = -s3, sigma_xz = s2, sigma_yz = -s1,
//   sigma_xt = eta s1, sigma_yt = eta s2, sigma_zt = eta s3,
// so the block of A is 1 + i csw kappa [[E3, E1 - i E2], [E1 + i E2, -E3]] with
// E1 = -F_yz + eta F_xt, E2 = F_xz + eta F_yt, E3 = -F_xy + eta F_zt.
// STEP 0 (planes xy, zt): E3, the diagonal 3x3 blocks.  STEP 1 (yz, xt): E1,
// parked in planes 6..10 of the block's entries.  STEP 2 (xz, yt): E2 and the
// lower 3x3 block i csw kappa (E1 + i E2).  Written to the FP64 store; f =
// csw kappa / 8.
template <int STEP>
__global__ void __launch_bounds__(128) k_gather(Geom g, CloverStore C, int4 planes, const double *ws, double f)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= g.V) return;
    const int V = g.V;
    int c[4];
    site_coords(g, x, c);
    const X3 fa = gather(g, ws, x, c, planes.x, planes.y);
    const X3 fb = gather(g, ws + (size_t)36 * V, x, c, planes.z, planes.w);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const double eta = b == 0 ? -f : f;
        double2 *o = C.c64 + (size_t)b * 18 * V + x;
        const X3 e = combine(STEP == 2 ? f : -f, fa, eta, fb);
        if (STEP == 0) {
            o[0] = make_double2(1.0 - e.d[0], 1.0 - e.d[1]);
            o[(size_t)V] = make_double2(1.0 - e.d[2], 1.0 + e.d[0]);
            o[(size_t)2 * V] = make_double2(1.0 + e.d[1], 1.0 + e.d[2]);
#pragma unroll
            for (int q = 0; q < 3; ++q) {   // entries (1,0) (2,0) (2,1), and (4,3) (5,3) (5,4)
                const int i = q == 0 ? 1 : 2, j = q == 2 ? 1 : 0;
                const cx<double> v = times_i(entry(e, i, j));
                o[(size_t)(3 + q) * V] = make_double2(v.re, v.im);
                o[(size_t)(q == 0 ? 12 : 15 + q) * V] = make_double2(-v.re, -v.im);
            }
        } else if (STEP == 1) {
            o[(size_t)6 * V] = make_double2(e.d[0], e.d[1]);
            o[(size_t)7 * V] = make_double2(e.d[2], 0.0);
#pragma unroll
            for (int k = 0; k < 3; ++k) o[(size_t)(8 + k) * V] = make_double2(e.o[k].re, e.o[k].im);
        } else {
            X3 e1;
            const double2 d0 = o[(size_t)6 * V], d1 = o[(size_t)7 * V];
            e1.d[0] = d0.x;
            e1.d[1] = d0.y;
            e1.d[2] = d1.x;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double2 v = o[(size_t)(8 + k) * V];
                e1.o[k] = mkc(v.x, v.y);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    // row 3 + i holds its entries from plane 6, 9, 13 on
                    const cx<double> v = times_i(entry(e1, i, j) + times_i(entry(e, i, j)));
                    o[(size_t)((i == 0 ? 6 : i == 1 ? 9 : 13) + j) * V] = make_double2(v.re, v.im);
                }
        }
    }
}

// the other precisions of the FP64 entries, one block of one site per thread
__global__ void __launch_bounds__(128) k_store_clover(int V, CloverStore C)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (x >= V) return;
    double r[36];
    P64::load_clover(C, V, x, b, r);
    store_clover_a<false>(C, V, x, b, r);
}

}  // namespace

cudaError_t launch_build_clover(wc_lattice lat, double csw, double kappa, cudaStream_t stream)
{
    const Geom &g = lat->g;
    static_assert(sizeof(float4) * 36 == sizeof(double) * 2 * 36, "leaves of two planes fit the double-FP32 store");
    double *ws = reinterpret_cast<double *>(lat->clover.cdf);
    const double f = csw * kappa / 8.0;
    const int4 pair[3] = {make_int4(0, 1, 2, 3), make_int4(1, 2, 0, 3), make_int4(0, 2, 1, 3)};
    const dim3 gl((g.V + 63) / 64, 2, 2), gg((g.V + 127) / 128), gs((g.V + 127) / 128, 2);
    for (int s = 0; s < 3; ++s) {
        k_leaves<<<gl, 64, 0, stream>>>(g, lat->gauge, pair[s], ws);
        if (s == 0) k_gather<0><<<gg, 128, 0, stream>>>(g, lat->clover, pair[s], ws, f);
        if (s == 1) k_gather<1><<<gg, 128, 0, stream>>>(g, lat->clover, pair[s], ws, f);
        if (s == 2) k_gather<2><<<gg, 128, 0, stream>>>(g, lat->clover, pair[s], ws, f);
    }
    k_store_clover<<<gs, 128, 0, stream>>>(g.V, lat->clover);
    return cudaGetLastError();
}

}  // namespace wc
