// Even-odd (Schur complement) preconditioning of M.  Sec. 2: both the FP64
// outer solver and the FP32 inner solver of CCS-QCD act on the even-odd
// site preconditioned matrix; the elimination below is the standard one.
//
// Ordering the sites by parity, M = [[A_ee, -k H_eo], [-k H_oe, A_oo]], so
//   b^_e = b_e + k H_eo A_oo^-1 b_o
//   M^ x_e = b^_e,   M^ = A_ee - k^2 H_eo A_oo^-1 H_oe   (even sites only)
//   x_o = A_oo^-1 (b_o + k H_oe x_e)
// and M^+ = gamma5 M^ gamma5 (gamma5 commutes with A and anticommutes with
// each hop).  The solvers run unchanged on half-volume fields of a
// "half lattice" (same gauge field and clover term, V/2 sites); its operator
// is M^.
//
// Half-volume layout: a field of parity p stores site (x,y,z,t) at index
// i = (x + Lx (y + Ly (z + Lz t))) >> 1; all extents are even (so that
// every hop, also across the boundary, flips the parity), hence every x-row
// holds Lx/2 sites of each parity and i is unique within a parity.
#include <math.h>

#include <algorithm>
#include <new>

#include "wc_internal.cuh"
#include "wc_reduce.cuh"
#include "wc_solver_kernels.cuh"
#include "wc_stencil.cuh"
#include "wc_dfsplit.cuh"

namespace wc {

namespace {

// ------------------------------------------------------------------------
// clover inverse: A^-1 as two packed Hermitian 6x6 blocks (FP64 arithmetic)
// ------------------------------------------------------------------------

__device__ __forceinline__ void unpack_block(const double r[36], cx<double> m[6][6])
{
    for (int i = 0; i < 6; ++i) m[i][i] = mkc(r[i], 0.0);
    int k = 6;
    for (int i = 1; i < 6; ++i)
        for (int j = 0; j < i; ++j) {
            m[i][j] = mkc(r[k], r[k + 1]);
            m[j][i] = conj(m[i][j]);
            k += 2;
        }
}

__device__ void pack_block(cx<double> m[6][6], double r[36])
{
    // Hermitian by construction; symmetrise the rounding
    for (int i = 0; i < 6; ++i) r[i] = m[i][i].re;
    int k = 6;
    for (int i = 1; i < 6; ++i)
        for (int j = 0; j < i; ++j) {
            const cx<double> a = m[i][j], b = conj(m[j][i]);
            r[k++] = 0.5 * (a.re + b.re);
            r[k++] = 0.5 * (a.im + b.im);
        }
}

// Gauss-Jordan inverse with partial pivoting (6x6 complex, in place).
// Returns false if a pivot is below 1e-12 of the block's largest entry
// (numerically singular: the inverse would carry no significant digit).
__device__ bool invert6(cx<double> a[6][6])
{
    double amax = 0.0;
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) amax = fmax(amax, fabs(a[i][j].re) + fabs(a[i][j].im));
    const double tiny2 = (1e-12 * amax) * (1e-12 * amax);
    cx<double> inv[6][6];
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) inv[i][j] = mkc(i == j ? 1.0 : 0.0, 0.0);
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        double best = a[c][c].re * a[c][c].re + a[c][c].im * a[c][c].im;
        for (int r = c + 1; r < 6; ++r) {
            const double v = a[r][c].re * a[r][c].re + a[r][c].im * a[r][c].im;
            if (v > best) {
                best = v;
                piv = r;
            }
        }
        if (!(best > tiny2) || !(best > 0.0)) return false;
        if (piv != c)
            for (int j = 0; j < 6; ++j) {
                cx<double> t = a[c][j];
                a[c][j] = a[piv][j];
                a[piv][j] = t;
                t = inv[c][j];
                inv[c][j] = inv[piv][j];
                inv[piv][j] = t;
            }
        const cx<double> p = a[c][c];
        const double d = p.re * p.re + p.im * p.im;
        const cx<double> pinv = mkc(p.re / d, -p.im / d);
        for (int j = 0; j < 6; ++j) {
            a[c][j] = pinv * a[c][j];
            inv[c][j] = pinv * inv[c][j];
        }
        for (int r = 0; r < 6; ++r) {
            if (r == c) continue;
            const cx<double> f = a[r][c];
            for (int j = 0; j < 6; ++j) {
                a[r][j] = a[r][j] - f * a[c][j];
                inv[r][j] = inv[r][j] - f * inv[c][j];
            }
        }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) a[i][j] = inv[i][j];
    return true;
}

// Inverse of a packed Hermitian 6x6 block B as K^+ D^-1 K from B = L D L^+, K =
// L^-1 (unit lower triangular), without pivoting: about 500 FP64 operations in
// registers, against 1700 for the pivoted Gauss-Jordan elimination, which keeps
// its 6x6 arrays in local memory (indexed at run time).  False unless every
// pivot stays above 5/8 of the block's largest entry: the caller then takes
// the elimination, which also decides what is singular.  Nothing near singular
// passes (the determinant is the product of the pivots), and what passes is
// inverted as accurately as by the elimination: mean error of the inverse
// over 8192 blocks of Haar links, by this form / by elimination, csw 1 1.23 /
// 1.28e-16, csw 2 1.26 / 1.31, csw 3 1.34 / 1.37 (88 % of the blocks pass), csw 5
// 4.6 / 4.6 (13 %); a bound of 1/4 would pass 84 % at csw 5, at 4.8e-16.
// (By 3x3 blocks and cofactors: 1.65 1.67 1.79 5.4e-16.)  At 16^3x32 297 us for
// both blocks of all sites and their copies, FP64 pipe 88 % busy; 1637 with every
// block eliminated.
__device__ __forceinline__ bool invert_block(const double r[36], double inv[36])
{
    double big = 0.0, d[6], e[6];
    cx<double> l[6][6];   // below the diagonal: what is left of B, then L, then K
#pragma unroll
    for (int k = 0; k < 36; ++k) big = fmax(big, fabs(r[k]));
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        d[i] = r[i];
#pragma unroll
        for (int j = 0; j < i; ++j) l[i][j] = mkc(r[6 + i * (i - 1) + 2 * j], r[7 + i * (i - 1) + 2 * j]);
    }
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        ok = ok && fabs(d[c]) > 0.625 * big;   // false for a NaN
        e[c] = 1.0 / d[c];
        cx<double> w[6];
#pragma unroll
        for (int i = c + 1; i < 6; ++i) {
            // w / d, the product with 1 / d corrected once
            w[i] = l[i][c];
            const cx<double> q = e[c] * w[i];
            l[i][c] = mkc(fma(fma(-q.re, d[c], w[i].re), e[c], q.re), fma(fma(-q.im, d[c], w[i].im), e[c], q.im));
        }
#pragma unroll
        for (int i = c + 1; i < 6; ++i) {
            d[i] = fma(-l[i][c].re, w[i].re, fma(-l[i][c].im, w[i].im, d[i]));
#pragma unroll
            for (int j = c + 1; j < i; ++j) l[i][j] = cfma_conj(w[j], -l[i][c], l[i][j]);
        }
    }
    if (!ok) return false;
    // row by row: K_ij = -(L_ij + sum_k L_ik K_kj), j < k < i
#pragma unroll
    for (int i = 1; i < 6; ++i) {
        cx<double> row[6];
#pragma unroll
        for (int j = 0; j < i; ++j) {
            row[j] = -l[i][j];
#pragma unroll
            for (int k = j + 1; k < i; ++k) row[j] = cfma(-l[i][k], l[k][j], row[j]);
        }
#pragma unroll
        for (int j = 0; j < i; ++j) l[i][j] = row[j];
    }
    // (B^-1)_ij = sum_k conj(K_ki) K_kj / d_k over k >= i
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double s = 0.0;
#pragma unroll
        for (int k = 5; k > i; --k) s = fma(e[k], fma(l[k][i].re, l[k][i].re, l[k][i].im * l[k][i].im), s);
        inv[i] = e[i] + s;
#pragma unroll
        for (int j = 0; j < i; ++j) {
            cx<double> t = mkc(0.0, 0.0);
#pragma unroll
            for (int k = 5; k > i; --k) t = cfma_conj(l[k][i], e[k] * l[k][j], t);
            inv[6 + i * (i - 1) + 2 * j] = fma(e[i], l[i][j].re, t.re);
            inv[7 + i * (i - 1) + 2 * j] = fma(e[i], l[i][j].im, t.im);
        }
    }
    return true;
}

// the pivoted elimination on a packed block, out of line: few blocks need it
__device__ __noinline__ bool invert_block_pivoted(const double *r, double *inv)
{
    cx<double> m[6][6];
    unpack_block(r, m);
    const bool ok = invert6(m);
    pack_block(m, inv);
    return ok;
}

// Parity-ordered copies for the even-odd kernels: within every component
// plane, position parity(x) * V/2 + (x >> 1), so that the threads of one
// parity read contiguous memory (full-volume order would fetch every other
// site's entries with them).  Ce: A = 1 + T; Ci: A^-1.  One block of one
// site per thread.
__global__ void __launch_bounds__(64) k_clover_invert(Geom g, CloverStore C, CloverStore Ce, CloverStore Ci, int *bad)
{
    const int V = g.V;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (x >= V) return;
    int c[4];
    site_coords(g, x, c);
    const int pos = ((c[0] + c[1] + c[2] + c[3]) & 1) * (V >> 1) + (x >> 1);
    double r[36], inv[36];
    P64::load_clover(C, V, x, b, r);
    store_clover_a<true>(Ce, V, pos, b, r);
    if (!invert_block(r, inv) && !invert_block_pivoted(r, inv)) atomicExch(bad, 1);
    store_clover_block(Ci, V, pos, b, inv);
}

// ------------------------------------------------------------------------
// parity stencil
// ------------------------------------------------------------------------

// full site of half index i of parity p: 2 i is the full index of the site
// with x rounded down to even (all extents are even)
__device__ __forceinline__ int full_site(const Geom &g, int i, int p, int c[4])
{
    site_coords_fast(g, 2 * i, c);
    const int bit = (p + c[1] + c[2] + c[3]) & 1;
    c[0] += bit;
    return wc_idx(2 * i + bit, g.V);
}

// hops of the opposite-parity half field `in` into site x (full index x,
// coordinates c), accumulated into acc with coefficient k (boundary phase
// included); links from the full-volume store
template <class P, int MU, int SF, int SB>
__device__ __forceinline__ void eo_hop_dir(const Geom &g, const GaugeStore &U, const void *in, const float *in_nrm,
                                           int Vh, int x, const int c[4], typename P::real k,
                                           cx<typename P::real> acc[12])
{
    using R = typename P::real;
    const int L = g.L[MU], st = g.stride[MU];
    {
        const bool wrap = c[MU] == L - 1;
        const int xf = wc_idx(wrap ? x - (L - 1) * st : x + st, g.V);
        cx<R> p[12], h[6], u[6], r2[3], w[6];
        const R scale = P::load_spinor_raw(in, in_nrm, Vh, xf >> 1, p);
        const R coef = ((MU == 3 && wrap) ? k * R(g.tbc) : k) * scale;
        project<MU, SF>(p, h);
        P::load_link(U, g.V, MU, x, u, r2);
        su3_mul(u, r2, h, coef, w);
        reconstruct_add<MU, SF>(acc, w);
    }
    {
        const bool wrap = c[MU] == 0;
        const int xb = wc_idx(wrap ? x + (L - 1) * st : x - st, g.V);
        cx<R> p[12], h[6], u[6], r2[3], w[6];
        const R scale = P::load_spinor_raw(in, in_nrm, Vh, xb >> 1, p);
        const R coef = ((MU == 3 && wrap) ? k * R(g.tbc) : k) * scale;
        project<MU, SB>(p, h);
        P::load_link(U, g.V, MU, xb, u, r2);
        su3_adj_mul(u, r2, h, coef, w);
        reconstruct_add<MU, SB>(acc, w);
    }
}

// y = A v (INV: A^-1 v) at position pos of the parity-ordered store
template <class P, bool INV>
__device__ __forceinline__ void clover_eo(const CloverStore &S, int V, int pos, const cx<typename P::real> v[12],
                                          cx<typename P::real> y[12])
{
    if constexpr (!INV) {
        clover_a<P>(S, V, pos, 0, v, y);
        clover_a<P>(S, V, pos, 1, v + 6, y + 6);
    } else {
        using R = typename P::real;
        R r0[36], r1[36];
        P::load_clover(S, V, pos, 0, r0);
        P::load_clover(S, V, pos, 1, r1);
        clover_block_mul(r0, v, y);
        clover_block_mul(r1, v + 6, y + 6);
    }
}

// o = C v + beta h
template <class P>
__device__ __forceinline__ void add_clover_eo(const Geom &g, int p, const CloverStore &C, double beta, int Vh, int i,
                                              const cx<typename P::real> v[12], const cx<typename P::real> h[12],
                                              cx<typename P::real> o[12])
{
    using R = typename P::real;
    const R bt = R(beta);
    clover_eo<P, false>(C, g.V, wc_idx(p * Vh + i, g.V), v, o);
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k] = o[k] + bt * h[k];
}

// h = the hops of hin (opposite parity) to full-lattice site x
template <class P, int DAG>
__device__ __forceinline__ void eo_hops(const Geom &g, const GaugeStore &U, const void *hin, const float *hin_nrm, int Vh,
                                        int x, const int c[4], cx<typename P::real> h[12])
{
    using R = typename P::real;
#pragma unroll
    for (int k = 0; k < 12; ++k) h[k] = mkc(R(0), R(0));
    constexpr int SF = DAG ? +1 : -1;
    constexpr int SB = -SF;
    if constexpr (std::is_same<P, P16>::value) {
        const auto half = [](int y) { return y >> 1; };
        hop_dir_h16<0, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, 1.f, h, half);
        hop_dir_h16<1, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, 1.f, h, half);
        hop_dir_h16<2, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, 1.f, h, half);
        hop_dir_h16<3, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, 1.f, h, half);
    } else {
        const R one = R(1);
        eo_hop_dir<P, 0, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, one, h);
        eo_hop_dir<P, 1, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, one, h);
        eo_hop_dir<P, 2, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, one, h);
        eo_hop_dir<P, 3, SF, SB>(g, U, hin, hin_nrm, Vh, x, c, one, h);
    }
}

// One pass of the even-odd operators, for the sites of parity p (half index
// i); h = sum of the hops of `hin` (opposite parity), C, Ci: clover term and
// inverse in parity order (k_clover_invert):
//   MODE 0: out = Ci h
//        1: out = C vin + beta h
//   and on FP64 fields
//        2: out = vin + beta h
//        4: out = Ci vin
//        5: out = Ci w and out2 = w - C out, w = vin + beta h (with
//           vin = b_o, h = H_oe x_e, beta = k: the reconstructed x_o and
//           the odd-site residual b_o - (A_oo x_o - k H_oe x_e) of the
//           x_o as stored, in one pass)
// (FP32 and FP16 fields.  One CTA per SM is all that is asked of the register
// allocation: without that it keeps fewer loads in flight, a solver step at
// 16^3x32 in binary16 136 instead of 122 us; four CTAs measured the same, five
// and six 4 and 8 % slower.  Site coordinates by multiplication and the
// binary16 hops formed from the stored halves took 2 to 3 % off a step:
// 16^3x32 FP32 112 -> 109 us, 24^3x32 binary16 188 -> 183.)
template <class P, int DAG, int MODE>
__global__ void __launch_bounds__(128, 1) k_eo(Geom g, int p, GaugeStore U, CloverStore C, CloverStore Ci,
                                            const void *hin, const float *hin_nrm, const void *vin,
                                            const float *vin_nrm, void *out, float *out_nrm, double beta,
                                            const int *skip)
{
    griddep_wait();
    griddep_launch_dependents();
    if (skip && *skip) return;
    static_assert(MODE == 0 || MODE == 1, "the other modes are for FP64 fields");
    using R = typename P::real;
    const int Vh = g.V >> 1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Vh) return;
    int c[4];
    const int x = full_site(g, i, p, c);
    cx<R> h[12], o[12];
    eo_hops<P, DAG>(g, U, hin, hin_nrm, Vh, x, c, h);
    if (MODE == 0) {
        clover_eo<P, true>(Ci, g.V, wc_idx(p * Vh + i, g.V), h, o);
    } else {
        cx<R> v[12];
        P::load_spinor(vin, vin_nrm, Vh, i, v);
        add_clover_eo<P>(g, p, C, beta, Vh, i, v, h, o);
    }
    P::store_spinor(out, out_nrm, Vh, i, o);
}

// k_eo in FP64 on four warps per 32 sites (hop_split64): warp w finishes
// components 3 w .. 3 w + 2; a product with A or A^-1 takes its vector from
// shared memory.
template <int DAG, int MODE>
__global__ void __launch_bounds__(kSplit64 * kSplit64Sites, 3)
    k_eo_split64(Geom g, int p, GaugeStore U, CloverStore C, CloverStore Ci, const void *hin, const double2 *vin,
                 double2 *out, double2 *out2, double beta, const int *skip)
{
    griddep_wait();
    griddep_launch_dependents();
    if (skip && *skip) return;
    __shared__ Split64Mem sm;
    const int Vh = g.V >> 1;
    const int s = threadIdx.x & (kSplit64Sites - 1), w = threadIdx.x / kSplit64Sites;
    const int i = blockIdx.x * kSplit64Sites + s;
    const bool valid = i < Vh;
    if (MODE != 4 && valid) {
        int c[4];
        const int x = full_site(g, i, p, c);
        hop_split64<DAG ? +1 : -1>(g, U, hin, Vh, x, c, sm, w, s, [](int y) { return y >> 1; });
    }
    __syncthreads();
    cx<double> v[3], o[3], vb[6];
    if (valid) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int k = 3 * w + r;
            const cx<double> h = MODE == 4 ? mkc(0.0, 0.0) : sum_split64(sm, k, s);
            if (MODE == 0) {
                v[r] = h;
            } else if (MODE == 1) {
                v[r] = beta * h;
            } else {
                const double2 a = vin[(size_t)k * Vh + i];
                v[r] = MODE == 4 ? mkc(a.x, a.y) : mkc(fma(beta, h.re, a.x), fma(beta, h.im, a.y));
            }
        }
    }
    // every thread reads and writes column s, component k only in its own
    // warp until the barrier
    const auto share = [&](const cx<double> a[3]) {
        if (valid)
#pragma unroll
            for (int r = 0; r < 3; ++r) sm[0][3 * w + r][s] = make_double2(a[r].re, a[r].im);
        __syncthreads();
        if (valid)
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const double2 b = sm[0][(w >> 1) * 6 + k][s];
                vb[k] = mkc(b.x, b.y);
            }
    };
    const auto store = [&](double2 *f, const cx<double> a[3]) {
#pragma unroll
        for (int r = 0; r < 3; ++r) f[(size_t)(3 * w + r) * Vh + i] = make_double2(a[r].re, a[r].im);
    };
    if (MODE == 2) {
        if (valid) store(out, v);
        return;
    }
    const int pos = wc_idx(p * Vh + (valid ? i : 0), g.V);
    if (MODE == 1) {
        if (!valid) return;
        const double2 *q = vin + (size_t)(w >> 1) * 6 * Vh + i;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 a = q[(size_t)k * Vh];
            vb[k] = mkc(a.x, a.y);
        }
        clover_rows64(C, g.V, pos, w, vb, v);
        store(out, v);
        return;
    }
    share(v);
    if (valid) {
#pragma unroll
        for (int r = 0; r < 3; ++r) o[r] = mkc(0.0, 0.0);
        clover_rows64(Ci, g.V, pos, w, vb, o);
        store(out, o);
    }
    if (MODE == 5) {
        __syncthreads();   // vb is read
        share(o);
        if (valid) {
            cx<double> y[3] = {times_iq<2>(v[0]), times_iq<2>(v[1]), times_iq<2>(v[2])};   // A x_o - v
            clover_rows64(C, g.V, pos, w, vb, y);
#pragma unroll
            for (int r = 0; r < 3; ++r) y[r] = times_iq<2>(y[r]);
            store(out2, y);
        }
    }
}

// k_eo in mode 1 as the second half of a solver step's operator: the pass
// also forms the sums of alpha (or OMEGA: of omega) with `ss.with`, in CTAs
// of W warps.  The sums are those of out as stored.
template <class P, int DAG, int W, bool OMEGA>
__global__ void __launch_bounds__(32 * W, 1) k_eo_sum(Geom g, int p, GaugeStore U, CloverStore C, const void *hin,
                                                      const float *hin_nrm, const void *vin, const float *vin_nrm,
                                                      void *out, float *out_nrm, double beta, StepSum ss)
{
    griddep_wait();
    griddep_launch_dependents();
    if (ss.sc->skip) return;
    using R = typename P::real;
    const int Vh = g.V >> 1;
    const int i = blockIdx.x * 32 * W + threadIdx.x;
    R acc[step_sums<OMEGA, R>] = {};
    if (i < Vh) {
        int c[4];
        const int x = full_site(g, i, p, c);
        cx<R> h[12], v[12], o[12];
        eo_hops<P, DAG>(g, U, hin, hin_nrm, Vh, x, c, h);
        P::load_spinor(vin, vin_nrm, Vh, i, v);
        add_clover_eo<P>(g, p, C, beta, Vh, i, v, h, o);
        P::store_spinor(out, out_nrm, Vh, i, o);
        P::as_stored(o);
        P::load_spinor(ss.with, ss.with_nrm, Vh, i, v);
        add_step_sums<OMEGA, 12>(o, v, acc);
    }
    reduce_step_sums<OMEGA, W, R>(acc, ss);
}

// The same in FP64 on four warps per 32 sites (k_eo_split64).
template <int DAG, bool OMEGA>
__global__ void __launch_bounds__(kSplit64 * kSplit64Sites, 3)
    k_eo_split64_sum(Geom g, int p, GaugeStore U, CloverStore C, const void *hin, const double2 *vin, double2 *out,
                     double beta, StepSum ss)
{
    griddep_wait();
    griddep_launch_dependents();
    if (ss.sc->skip) return;
    __shared__ Split64Mem sm;
    const int Vh = g.V >> 1;
    const int s = threadIdx.x & (kSplit64Sites - 1), w = threadIdx.x / kSplit64Sites;
    const int i = blockIdx.x * kSplit64Sites + s;
    const bool valid = i < Vh;
    if (valid) {
        int c[4];
        const int x = full_site(g, i, p, c);
        hop_split64<DAG ? +1 : -1>(g, U, hin, Vh, x, c, sm, w, s, [](int y) { return y >> 1; });
    }
    __syncthreads();
    double acc[step_sums<OMEGA, double>] = {};
    if (valid) {
        cx<double> vb[6], o[3], a[3];
        const double2 *q = vin + (size_t)(w >> 1) * 6 * Vh + i;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 b = q[(size_t)k * Vh];
            vb[k] = mkc(b.x, b.y);
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) o[r] = beta * sum_split64(sm, 3 * w + r, s);
        clover_rows64(C, g.V, wc_idx(p * Vh + i, g.V), w, vb, o);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const size_t k = (size_t)(3 * w + r) * Vh + i;
            out[k] = make_double2(o[r].re, o[r].im);
            const double2 b = static_cast<const double2 *>(ss.with)[k];
            a[r] = mkc(b.x, b.y);
        }
        add_step_sums<OMEGA, 3>(o, a, acc);
    }
    reduce_step_sums<OMEGA, kSplit64, double>(acc, ss);
}

// An FP64 half field as z2 values (wc_dfsplit.cuh), for the hops of the next
// pass: each of its spinors is read eight times.
__global__ void __launch_bounds__(256) k_to_df(long long n, const double2 *in, float4 *out, const int *skip)
{
    griddep_wait();
    griddep_launch_dependents();
    if (skip && *skip) return;
    const long long step = (long long)gridDim.x * blockDim.x;
    // four reads in flight
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += 4 * step) {
        double2 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = i + k * step < n ? in[i + k * step] : make_double2(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * step < n) out[i + k * step] = dfs::to4(dfs::of_double(v[k]));
    }
}

// k_eo of FP64 fields in double-FP32 arithmetic, on four warps per 32 sites as
// k_eo_split64.  hin, and the output of modes 0 and 4, which the next pass takes
// its hops from, are kept as z2 values.
template <int DAG, int MODE>
__global__ void __launch_bounds__(kSplit64 * kSplit64Sites, dfs::kCtas)
    k_eo_splitdf(Geom g, int p, GaugeStore U, CloverStore C, CloverStore Ci, const void *hin, const double2 *vin,
                 void *out, double2 *out2, double beta, const int *skip)
{
    using dfs::z2;
    griddep_wait();
    griddep_launch_dependents();
    if (skip && *skip) return;
    __shared__ dfs::Mem sm;
    const int Vh = g.V >> 1;
    const int s = threadIdx.x & (kSplit64Sites - 1), w = threadIdx.x / kSplit64Sites;
    const int i = blockIdx.x * kSplit64Sites + s;
    const bool valid = i < Vh;
    if (MODE != 4 && valid) {
        int c[4];
        const int x = full_site(g, i, p, c);
        dfs::hops<DAG ? +1 : -1, true>(g, U, hin, Vh, x, c, sm, w, s, [](int y) { return y >> 1; });
    }
    __syncthreads();
    const df bt(beta);
    z2 v[3], vb[6];
    if (valid) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int k = 3 * w + r;
            const z2 h = MODE == 4 ? dfs::zero() : dfs::sum(sm, k, s);
            if (MODE == 0) {
                v[r] = h;
            } else if (MODE == 1) {
                dfs::Sum t = dfs::first_term(bt, h);
                v[r] = dfs::finish(t);
            } else {
                const z2 a = dfs::of_double(vin[(size_t)k * Vh + i]);
                dfs::Sum t = dfs::start(a);
                if (MODE != 4) dfs::add_term(t, bt, h);
                v[r] = dfs::finish(t);
            }
        }
    }
    // component k is read and written only by its own warp until the barrier
    const auto share = [&](const z2 a[3]) {
        if (valid)
#pragma unroll
            for (int r = 0; r < 3; ++r) sm[0][3 * w + r][s] = dfs::to4(a[r]);
        __syncthreads();
        if (valid)
#pragma unroll
            for (int k = 0; k < 6; ++k) vb[k] = dfs::of4(sm[0][(w >> 1) * 6 + k][s]);
    };
    const auto store = [&](const z2 a[3]) {
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const size_t at = (size_t)(3 * w + r) * Vh + i;
            if (MODE == 0 || MODE == 4) static_cast<float4 *>(out)[at] = dfs::to4(a[r]);
            else static_cast<double2 *>(out)[at] = dfs::to_double(a[r]);
        }
    };
    if (MODE == 2) {
        if (valid) store(v);
        return;
    }
    const int pos = wc_idx(p * Vh + (valid ? i : 0), g.V);
    if (MODE == 1) {
        if (!valid) return;
        const double2 *q = vin + (size_t)(w >> 1) * 6 * Vh + i;
#pragma unroll
        for (int k = 0; k < 6; ++k) vb[k] = dfs::of_double(q[(size_t)k * Vh]);
        dfs::Sum y[3] = {dfs::start(v[0]), dfs::start(v[1]), dfs::start(v[2])};
        dfs::clover_rows(C, g.V, pos, w, vb, y);
        const z2 o[3] = {dfs::finish(y[0]), dfs::finish(y[1]), dfs::finish(y[2])};
        store(o);
        return;
    }
    share(v);
    z2 o[3];
    if (valid) {
        dfs::Sum y[3] = {dfs::start(dfs::zero()), dfs::start(dfs::zero()), dfs::start(dfs::zero())};
        dfs::clover_rows(Ci, g.V, pos, w, vb, y);
#pragma unroll
        for (int r = 0; r < 3; ++r) o[r] = dfs::finish(y[r]);
        store(o);
    }
    if (MODE == 5) {
        // the residual of x_o as the caller receives it (the stored value)
        if (valid)
#pragma unroll
            for (int r = 0; r < 3; ++r) o[r] = dfs::of_double(dfs::to_double(o[r]));
        __syncthreads();   // vb is read
        share(o);
        if (valid) {
            dfs::Sum y[3] = {dfs::start(dfs::neg(v[0])), dfs::start(dfs::neg(v[1])), dfs::start(dfs::neg(v[2]))};
            dfs::clover_rows(C, g.V, pos, w, vb, y);
#pragma unroll
            for (int r = 0; r < 3; ++r) out2[(size_t)(3 * w + r) * Vh + i] = dfs::to_double(dfs::neg(dfs::finish(y[r])));
        }
    }
}

// full field <-> the two half fields (parity 0 = even, 1 = odd)
template <class P>
__global__ void k_split(Geom g, const void *full, const float *full_nrm, void *ev, float *ev_nrm, void *od,
                        float *od_nrm)
{
    const int Vh = g.V >> 1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Vh) return;
    int c[4];
    cx<typename P::real> s[12];
    P::load_spinor(full, full_nrm, g.V, full_site(g, i, 0, c), s);
    P::store_spinor(ev, ev_nrm, Vh, i, s);
    if (!od) return;   // odd half not wanted
    P::load_spinor(full, full_nrm, g.V, full_site(g, i, 1, c), s);
    P::store_spinor(od, od_nrm, Vh, i, s);
}

template <class P>
__global__ void k_merge(Geom g, const void *ev, const float *ev_nrm, const void *od, const float *od_nrm,
                        void *full, float *full_nrm)
{
    const int Vh = g.V >> 1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Vh) return;
    int c[4];
    cx<typename P::real> s[12];
    P::load_spinor(ev, ev_nrm, Vh, i, s);
    P::store_spinor(full, full_nrm, g.V, full_site(g, i, 0, c), s);
    if (od) {
        P::load_spinor(od, od_nrm, Vh, i, s);
    } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) s[k] = mkc(typename P::real(0), typename P::real(0));
    }
    P::store_spinor(full, full_nrm, g.V, full_site(g, i, 1, c), s);
}

template <int DAG>
cudaError_t launch_eo_split64(const wc_lattice_s *full, int parity, int mode, const wc_field_s *hin,
                              const wc_field_s *vin, wc_field_s *out, double beta, cudaStream_t stream,
                              wc_field_s *out2, const int *skip, bool pdl)
{
    if (mode == 5 && (!out2 || out2->prec != WC_F64)) return cudaErrorInvalidValue;
    const int Vh = full->g.V >> 1;
    const dim3 grid((Vh + kSplit64Sites - 1) / kSplit64Sites);
    const void *hd = hin ? hin->data : nullptr;
    const double2 *vd = vin ? static_cast<const double2 *>(vin->data) : nullptr;
    double2 *od = static_cast<double2 *>(out->data), *o2 = out2 ? static_cast<double2 *>(out2->data) : nullptr;
#define WC_EO(M)                                                                                                 \
    return launch_step(pdl && pdl_grid(grid.x), k_eo_split64<DAG, M>, grid, kSplit64 *kSplit64Sites, stream, full->g, parity, full->gauge, \
                       full->ceo, full->cinv, hd, vd, od, o2, beta, skip)
    switch (mode) {
    case 0: WC_EO(0); break;
    case 1: WC_EO(1); break;
    case 2: WC_EO(2); break;
    case 4: WC_EO(4); break;
    case 5: WC_EO(5); break;
    default: return cudaErrorInvalidValue;
    }
#undef WC_EO
}

template <int DAG>
cudaError_t launch_eo_splitdf(const wc_lattice_s *full, int parity, int mode, const wc_field_s *hin,
                              const wc_field_s *vin, wc_field_s *out, double beta, cudaStream_t stream,
                              wc_field_s *out2, const int *skip, bool pdl)
{
    if (mode == 5 && (!out2 || out2->prec != WC_F64)) return cudaErrorInvalidValue;
    const int Vh = full->g.V >> 1;
    const dim3 grid((Vh + kSplit64Sites - 1) / kSplit64Sites);
    const void *hd = hin ? hin->data : nullptr;
    const double2 *vd = vin ? static_cast<const double2 *>(vin->data) : nullptr;
    double2 *o2 = out2 ? static_cast<double2 *>(out2->data) : nullptr;
#define WC_EO(M)                                                                                                    \
    return launch_step(pdl && pdl_grid(grid.x), k_eo_splitdf<DAG, M>, grid, kSplit64 *kSplit64Sites, stream, full->g, \
                       parity, full->gauge, full->ceo, full->cinv, hd, vd, out->data, o2, beta, skip)
    switch (mode) {
    case 0: WC_EO(0); break;
    case 1: WC_EO(1); break;
    case 2: WC_EO(2); break;
    case 4: WC_EO(4); break;
    case 5: WC_EO(5); break;
    default: return cudaErrorInvalidValue;
    }
#undef WC_EO
}

// CTAs of 128 sites; on small lattices (fewer than two such CTAs per SM)
// CTAs of 32, so that the sites spread over more SMs
int eo_threads(int Vh) { return Vh < 2 * 128 * sm_count() ? 32 : 128; }

template <class P, int DAG>
cudaError_t launch_eo_p(const wc_lattice_s *full, int parity, int mode, const wc_field_s *hin, const wc_field_s *vin,
                        wc_field_s *out, double beta, cudaStream_t stream, const int *skip, bool pdl)
{
    const int Vh = full->g.V >> 1;
    const int threads = eo_threads(Vh);
    const dim3 grid((Vh + threads - 1) / threads);
    const void *hd = hin ? hin->data : nullptr;
    const float *hn = hin ? hin->nrm : nullptr;
    const void *vd = vin ? vin->data : nullptr;
    const float *vn = vin ? vin->nrm : nullptr;
#define WC_EO(M)                                                                                                \
    return launch_step(pdl && pdl_grid(grid.x), k_eo<P, DAG, M>, grid, threads, stream, full->g, parity, full->gauge, full->ceo,    \
                       full->cinv, hd, hn, vd, vn, out->data, out->nrm, beta, skip)
    switch (mode) {
    case 0: WC_EO(0); break;
    case 1: WC_EO(1); break;
    default: return cudaErrorInvalidValue;   // the others: FP64 fields only
    }
#undef WC_EO
}

template <class P, int DAG>
cudaError_t launch_eo_sum(const wc_lattice_s *full, const wc_field_s *hin, const wc_field_s *vin, wc_field_s *out,
                          double beta, cudaStream_t stream, const StepSum &ss, bool omega, bool pdl)
{
    const int Vh = full->g.V >> 1, threads = eo_threads(Vh);
    const dim3 grid((Vh + threads - 1) / threads);
    const auto kern = threads == 32 ? (omega ? k_eo_sum<P, DAG, 1, true> : k_eo_sum<P, DAG, 1, false>)
                                    : (omega ? k_eo_sum<P, DAG, 4, true> : k_eo_sum<P, DAG, 4, false>);
    return launch_step(pdl && pdl_grid(grid.x), kern, grid, threads, stream, full->g, 0, full->gauge, full->ceo,
                       hin->data, hin->nrm, vin->data, vin->nrm, out->data, out->nrm, beta, ss);
}

template <int DAG>
cudaError_t launch_eo_sum64(const wc_lattice_s *full, const wc_field_s *hin, const wc_field_s *vin, wc_field_s *out,
                            double beta, cudaStream_t stream, const StepSum &ss, bool omega, bool pdl)
{
    const dim3 grid(((full->g.V >> 1) + kSplit64Sites - 1) / kSplit64Sites);
    const auto kern = omega ? k_eo_split64_sum<DAG, true> : k_eo_split64_sum<DAG, false>;
    return launch_step(pdl && pdl_grid(grid.x), kern, grid, kSplit64 * kSplit64Sites, stream, full->g, 0, full->gauge,
                       full->ceo, hin->data, static_cast<const double2 *>(vin->data), static_cast<double2 *>(out->data),
                       beta, ss);
}

}  // namespace

// one parity-stencil step on half fields of the full lattice `full`
cudaError_t launch_eo(const wc_lattice_s *full, int parity, int mode, int dagger, const wc_field_s *hin,
                      const wc_field_s *vin, wc_field_s *out, double beta, cudaStream_t stream, wc_field_s *out2,
                      const int *skip, bool pdl)
{
    const wc_prec pr = out->prec;
    if (pr == WC_F64 && full->fp64_arith == WC_ARITH_DF32)
        return dagger ? launch_eo_splitdf<1>(full, parity, mode, hin, vin, out, beta, stream, out2, skip, pdl)
                      : launch_eo_splitdf<0>(full, parity, mode, hin, vin, out, beta, stream, out2, skip, pdl);
    if (pr == WC_F64)
        return dagger ? launch_eo_split64<1>(full, parity, mode, hin, vin, out, beta, stream, out2, skip, pdl)
                      : launch_eo_split64<0>(full, parity, mode, hin, vin, out, beta, stream, out2, skip, pdl);
    if (pr == WC_F32)
        return dagger ? launch_eo_p<P32, 1>(full, parity, mode, hin, vin, out, beta, stream, skip, pdl)
                      : launch_eo_p<P32, 0>(full, parity, mode, hin, vin, out, beta, stream, skip, pdl);
    return dagger ? launch_eo_p<P16, 1>(full, parity, mode, hin, vin, out, beta, stream, skip, pdl)
                  : launch_eo_p<P16, 0>(full, parity, mode, hin, vin, out, beta, stream, skip, pdl);
}

cudaError_t launch_to_df(long long n, const wc_field_s *in, wc_field_s *out, cudaStream_t stream, const int *skip,
                         bool pdl)
{
    const int blocks = (int)std::min<long long>((n + 255) / 256, 8 * sm_count());
    return launch_step(pdl && pdl_grid(blocks), k_to_df, dim3(blocks), 256, stream, n,
                       static_cast<const double2 *>(in->data), static_cast<float4 *>(out->data), skip);
}

bool eo_split(const wc_lattice_s *full, const wc_field_s *f)
{
    return f->prec == WC_F64 && full->fp64_arith == WC_ARITH_DF32;
}

// od may be NULL: only the even half is written
cudaError_t launch_split(const wc_lattice_s *full, const wc_field_s *f, wc_field_s *ev, wc_field_s *od,
                         cudaStream_t stream)
{
    const int Vh = full->g.V >> 1;
    dim3 grid((Vh + 255) / 256), block(256);
    void *od_d = od ? od->data : nullptr;
    float *od_n = od ? od->nrm : nullptr;
    if (f->prec == WC_F64)
        k_split<P64><<<grid, block, 0, stream>>>(full->g, f->data, f->nrm, ev->data, ev->nrm, od_d, od_n);
    else if (f->prec == WC_F32)
        k_split<P32><<<grid, block, 0, stream>>>(full->g, f->data, f->nrm, ev->data, ev->nrm, od_d, od_n);
    else
        k_split<P16><<<grid, block, 0, stream>>>(full->g, f->data, f->nrm, ev->data, ev->nrm, od_d, od_n);
    return cudaGetLastError();
}

// od may be NULL: the odd sites of f are set to zero
cudaError_t launch_merge(const wc_lattice_s *full, const wc_field_s *ev, const wc_field_s *od, wc_field_s *f,
                         cudaStream_t stream)
{
    const int Vh = full->g.V >> 1;
    dim3 grid((Vh + 255) / 256), block(256);
    const void *od_d = od ? od->data : nullptr;
    const float *od_n = od ? od->nrm : nullptr;
    if (f->prec == WC_F64)
        k_merge<P64><<<grid, block, 0, stream>>>(full->g, ev->data, ev->nrm, od_d, od_n, f->data, f->nrm);
    else if (f->prec == WC_F32)
        k_merge<P32><<<grid, block, 0, stream>>>(full->g, ev->data, ev->nrm, od_d, od_n, f->data, f->nrm);
    else
        k_merge<P16><<<grid, block, 0, stream>>>(full->g, ev->data, ev->nrm, od_d, od_n, f->data, f->nrm);
    return cudaGetLastError();
}

// out = M^ in (or M^+ in) on half fields of the half lattice `half`: t = A_oo^-1 H_oe in,
// out = A_ee in - k^2 H_eo t.  t: the half lattice's scratch of out's precision.
cudaError_t launch_schur(wc_lattice half, wc_field out, wc_field in, int dagger, cudaStream_t stream, wc_field tmp,
                         const int *skip, bool pdl)
{
    const wc_lattice_s *full = half->schur_parent;
    wc_field_s *t = tmp ? tmp : half->schur_tmp[out->prec];
    // in double-FP32 the passes exchange split values: out holds those of in
    // until the second pass writes it
    const bool df = eo_split(full, out);
    cudaError_t e = df ? launch_to_df(6LL * full->g.V, in, out, stream, skip, pdl) : cudaSuccess;
    if (e == cudaSuccess)
        e = launch_eo(full, 1, 0, dagger, df ? out : in, nullptr, t, 0.0, stream, nullptr, skip, pdl);
    if (e == cudaSuccess)
        e = launch_eo(full, 0, 1, dagger, t, in, out, -full->kappa * full->kappa, stream, nullptr, skip, pdl);
    return e;
}

cudaError_t launch_apply(wc_lattice lat, wc_field out, wc_field in, int kind, SolverState &S, bool step)
{
    const int *skip = step ? &S.scal->skip : nullptr;
    if (!lat->schur_parent) {
        wc_field split = S.work[kDfSlot];
        if (split && eo_split(lat, in)) return launch_apply_df(lat, out, in, split, kind, S.stream, skip, S.pdl);
        return launch_apply(lat, out, in, kind, S.stream, skip, S.pdl);
    }
    return launch_schur(lat, out, in, kind == 1, S.stream, S.work[kSchurSlot + out->prec], skip, S.pdl);
}

cudaError_t launch_apply_sum(wc_lattice lat, wc_field out, wc_field in, int kind, SolverState &S, bool omega,
                             wc_field with)
{
    const StepSum ss{with->data, with->nrm, S.red, S.scal};
    const wc_prec pr = out->prec;
    const wc_lattice_s *full = lat->schur_parent;
    // sites and warps of a CTA of the pass that would form the sums
    const int sites = pr == WC_F64 ? kSplit64Sites : eo_threads(lat->g.V), warps = pr == WC_F64 ? kSplit64 : sites / 32;
    const bool fused = (full ? !eo_split(full, out) : pr == WC_F64 && !eo_split(lat, out)) && kind != 2 &&
                       sum_in_pass(S.red, (lat->g.V + sites - 1) / sites, warps);
    if (fused && !full) {
        const cudaError_t e = launch_apply64_sum(lat, out, in, kind, S.stream, ss, omega, S.pdl);
        if (e != cudaErrorNotSupported) return e;
    } else if (fused) {
        const bool dag = kind == 1;
        const int *skip = &S.scal->skip;
        wc_field_s *t = S.work[kSchurSlot + pr] ? S.work[kSchurSlot + pr] : lat->schur_tmp[pr];
        const double beta = -full->kappa * full->kappa;
        cudaError_t e = launch_eo(full, 1, 0, dag, in, nullptr, t, 0.0, S.stream, nullptr, skip, S.pdl);
        if (e != cudaSuccess) return e;
#define WC_SUM(F, ...) F<__VA_ARGS__>(full, t, in, out, beta, S.stream, ss, omega, S.pdl)
        if (pr == WC_F64) return dag ? WC_SUM(launch_eo_sum64, 1) : WC_SUM(launch_eo_sum64, 0);
        if (pr == WC_F32) return dag ? WC_SUM(launch_eo_sum, P32, 1) : WC_SUM(launch_eo_sum, P32, 0);
        return dag ? WC_SUM(launch_eo_sum, P16, 1) : WC_SUM(launch_eo_sum, P16, 0);
#undef WC_SUM
    }
    const cudaError_t e = launch_apply(lat, out, in, kind, S, true);
    if (e != cudaSuccess) return e;
    if (pr == WC_F64) {
        const double2 *o = static_cast<const double2 *>(out->data), *a = static_cast<const double2 *>(with->data);
        return omega ? bicg_omega(lat, S, o, a) : bicg_alpha(lat, S, a, o);
    }
    return omega ? lo_omega(lat, S, out, with) : lo_alpha(lat, S, with, out);
}

wc_status build_clover_inverse(wc_lattice lat)
{
    if (lat->cinv_loaded) return WC_OK;
    const int V = lat->g.V;
    wc_status st = WC_OK;
    for (CloverStore *c : {&lat->cinv, &lat->ceo}) {
        if (c->c64) continue;
        st = check_cuda(lat, cudaMalloc(&c->c64, sizeof(double2) * 36 * (size_t)V), "cudaMalloc(clover inverse)");
        if (st == WC_OK)
            st = check_cuda(lat, cudaMalloc(&c->cdf, sizeof(float4) * 36 * (size_t)V), "cudaMalloc(clover inverse)");
        if (c == &lat->cinv) {
            if (st == WC_OK)
                st = check_cuda(lat, cudaMalloc(&c->c32, sizeof(float4) * 18 * (size_t)V), "cudaMalloc(clover inverse)");
            if (st == WC_OK)
                st = check_cuda(lat, cudaMalloc(&c->c16, sizeof(uint4) * 9 * (size_t)V), "cudaMalloc(clover inverse)");
        } else if (st == WC_OK) {
            st = alloc_clover_a(lat, *c);
        }
        if (st != WC_OK) {
            free_clover(*c);   // c64 says that a store is complete
            return st;
        }
    }
    int *bad = nullptr;
    st = check_cuda(lat, cudaMalloc(&bad, sizeof(int)), "cudaMalloc");
    if (st != WC_OK) return st;
    st = check_cuda(lat, cudaMemsetAsync(bad, 0, sizeof(int), lat->stream), "memset");
    if (st == WC_OK) {
        k_clover_invert<<<dim3((V + 63) / 64, 2), 64, 0, lat->stream>>>(lat->g, lat->clover, lat->ceo, lat->cinv, bad);
        st = check_launch(lat, "clover_invert");
    }
    int h = 0;
    if (st == WC_OK) st = check_cuda(lat, cudaMemcpyAsync(&h, bad, sizeof(int), cudaMemcpyDeviceToHost, lat->stream),
                                     "copy");
    if (st == WC_OK) st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync");
    cudaFree(bad);
    if (st != WC_OK) return st;
    if (h) return set_error(lat, WC_ERR_BREAKDOWN, "clover term is singular at some site");
    lat->cinv_loaded = true;
    return WC_OK;
}

// The half lattice of lat (created on first use): V/2 sites, operator M^.
wc_status half_lattice(wc_lattice lat, wc_lattice *out)
{
    // every hop must change the parity, also across the (anti)periodic
    // boundary: all four extents even
    for (int mu = 0; mu < 4; ++mu)
        if (lat->g.L[mu] % 2 != 0) return set_error(lat, WC_ERR_ARG, "even-odd needs even lattice extents");
    wc_status st = build_clover_inverse(lat);
    if (st != WC_OK) return st;
    if (!lat->half) {
        wc_lattice h = new (std::nothrow) wc_lattice_s();
        if (!h) return set_error(lat, WC_ERR_ARG, "out of host memory");
        h->g = lat->g;
        h->g.V = lat->g.V / 2;
        h->schur_parent = lat;
        h->gauge_loaded = h->clover_loaded = true;
        h->kappa = lat->kappa;
        h->csw = lat->csw;
        h->stream = lat->stream;
        st = state_init(lat, h->st);
        for (int pr = 0; pr < 3 && st == WC_OK; ++pr) st = wc_field_create(h, (wc_prec)pr, &h->schur_tmp[pr]);
        if (st != WC_OK) {
            for (auto &f : h->schur_tmp) wc_field_destroy(f);
            state_free(h->st);
            delete h;
            return st;
        }
        lat->half = h;
    }
    lat->half->stream = lat->stream;
    lat->half->kappa = lat->kappa;
    *out = lat->half;
    return WC_OK;
}

void free_batch_pool(wc_lattice lat)
{
    for (auto &s : lat->batch_states) state_free(s);
    lat->batch_states.clear();
    for (auto f : lat->batch_fields) wc_field_destroy(f);
    lat->batch_fields.clear();
}

void free_half(wc_lattice lat)
{
    if (!lat->half) return;
    free_batch_pool(lat->half);
    for (auto f : lat->batch_fields) wc_field_destroy(f);   // half-lattice fields
    lat->batch_fields.clear();
    for (auto *half_fields : {&lat->ras_half, &lat->schur_io})
        for (auto &pr : *half_fields)
            for (auto &f : pr) {
                wc_field_destroy(f);
                f = nullptr;
            }
    for (auto &f : lat->half->schur_tmp) wc_field_destroy(f);
    state_free(lat->half->st);
    delete lat->half;
    lat->half = nullptr;
}

}  // namespace wc
