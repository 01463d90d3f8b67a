// The FP64 operator in double-FP32 arithmetic, a site's four directions on
// four warps (hop_split64's layout: a CTA of 32 sites, warp w takes the two
// hops of direction w and finishes components 3 w .. 3 w + 2).
//
// A complex value is two 64-bit registers, H = (re.hi, im.hi) and L = (re.lo,
// im.lo), operated on by paired instructions (wc_df2.cuh).  Sums of products
// are formed as compensated dot products (Ogita, Rump and Oishi 2005, "Dot2"):
// every product's rounding error, its cross terms and the error of adding it
// to the running sum go into one FP32 error sum.  That sum is rounded at its
// own size, so it is kept small: hi + lo is normalised every second term (13.5
// paired instructions a term and a chain of seven through the running sum,
// where a multiply-add of double-word numbers that normalises each time takes
// 16 and a chain of twelve), and the diagonal of a clover block, its largest
// term, comes last.  Relative errors against 64 bits, M / H / M^: 2.0e-15 /
// 4.6e-15 / 5.5e-15 at kappa 0.12 (a site per thread with double-word
// multiply-adds and a split of FP64 values cut off at 47 bits: 6.1e-15 / 9.0e-15
// / 1.5e-14, though its hops in x were in FP64).
//
// One site per thread at 128 registers spilled 1 KB and ran 22 500 warp
// instructions per 32 sites of an even-odd pass in 38 % of the issue slots;
// a third of them split FP64 spinors into floats, eight times per spinor.
// Here nothing spills, and the field the hops read is split once before (or
// kept split, where a pass writes it for the next).
#pragma once

#include "wc_internal.cuh"
#include "wc_stencil.cuh"

namespace wc {
namespace dfs {

using f2::u64;
using f2::z2;

constexpr int kSites = kSplit64Sites;
// CTAs per SM: 128 registers, no spills; even-odd passes at 24^3x32 178 + 144
// us, 324 + 295 with a site per thread.  (Before the normalisation of every
// second term: 172 + 137 us, 198 + 146 with three CTAs (168 registers), 179 +
// 141 with five (96 registers, 100 B of spills).)
constexpr int kCtas = 4;
using Mem = float4[kSplit64][12][kSites];   // z2 as float4 (H, L)

__device__ __forceinline__ z2 of4(float4 v) { return z2{f2::pk(v.x, v.y), f2::pk(v.z, v.w)}; }
__device__ __forceinline__ float4 to4(z2 a)
{
    float4 v;
    f2::upk(a.h, v.x, v.y);
    f2::upk(a.l, v.z, v.w);
    return v;
}
__device__ __forceinline__ z2 of_double(double2 v)
{
    const df a = df_from_double(v.x), b = df_from_double(v.y);
    return z2{f2::pk(a.hi, b.hi), f2::pk(a.lo, b.lo)};
}
__device__ __forceinline__ double2 to_double(z2 a)
{
    const float4 v = to4(a);
    return make_double2(df_to_double(df(v.x, v.z)), df_to_double(df(v.y, v.w)));
}
__device__ __forceinline__ z2 neg(z2 a) { return z2{f2::neg(a.h), f2::neg(a.l)}; }
__device__ __forceinline__ z2 zero() { return z2{0ull, 0ull}; }
// i a = (-im, re)
__device__ __forceinline__ u64 rot(u64 a)
{
    float x, y;
    f2::upk(a, x, y);
    return f2::pk(-y, x);
}
__device__ __forceinline__ z2 times_i(z2 a) { return z2{rot(a.h), rot(a.l)}; }
// i^Q a
template <int Q>
__device__ __forceinline__ z2 times_iq(z2 a)
{
    if (Q == 1) return times_i(a);
    if (Q == 2) return neg(a);
    if (Q == 3) return neg(times_i(a));
    return a;
}

// A sum of products under way: s + e
struct Sum {
    u64 s, e;
};

__device__ __forceinline__ Sum start(z2 a) { return Sum{a.h, a.l}; }

// + b x for a real b, the same in both lanes
__device__ __forceinline__ void add_term(Sum &t, df b, z2 x)
{
    const u64 nb = f2::pk(-b.hi, -b.hi), bh = f2::pk(b.hi, b.hi), bl = f2::pk(b.lo, b.lo);
    const u64 np = f2::mul(nb, x.h);              // -fl(b x)
    const u64 q = f2::fma(bl, x.h, f2::fma(bh, x.l, f2::fma(bh, x.h, np)));   // its rounding error, the cross terms
    const u64 s = f2::sub(t.s, np);               // TwoSum(t.s, -np)
    const u64 bb = f2::sub(s, t.s);
    const u64 e1 = f2::sub(t.s, f2::sub(s, bb)), e2 = f2::add(np, bb);
    t.e = f2::add(t.e, f2::add(q, f2::sub(e1, e2)));
    t.s = s;
}
// the error sum back below half a unit of s
__device__ __forceinline__ void normalise(Sum &t)
{
    const u64 hi = f2::add(t.s, t.e);
    t.e = f2::sub(t.e, f2::sub(hi, t.s));
    t.s = hi;
}
// + (re + i im) x, with ix = i x
__device__ __forceinline__ void add_pair(Sum &t, df re, z2 x, df im, z2 ix)
{
    add_term(t, re, x);
    add_term(t, im, ix);
    normalise(t);
}
// the first term
__device__ __forceinline__ Sum first_term(df b, z2 x)
{
    const u64 nb = f2::pk(-b.hi, -b.hi), bh = f2::pk(b.hi, b.hi), bl = f2::pk(b.lo, b.lo);
    const u64 np = f2::mul(nb, x.h);
    Sum t;
    t.s = f2::neg(np);
    t.e = f2::fma(bl, x.h, f2::fma(bh, x.l, f2::fma(bh, x.h, np)));
    return t;
}
__device__ __forceinline__ z2 finish(Sum t)
{
    const u64 hi = f2::add(t.s, t.e);
    return z2{hi, f2::sub(t.e, f2::sub(hi, t.s))};
}

// the spinor of site y of an FP64 field, or (SPLIT) of a field kept as z2
template <bool SPLIT>
__device__ __forceinline__ z2 load(const void *f, int V, int k, int y)
{
    if (SPLIT) return of4(static_cast<const float4 *>(f)[(size_t)k * V + y]);
    return of_double(static_cast<const double2 *>(f)[(size_t)k * V + y]);
}

// h = two-spinor of (1 + S g_mu) psi; a, b: the spins that give h0 and h1 by
// h = u + i^Q (lower spin)
template <bool SPLIT, int QA, int QB, int SA, int SB>
__device__ __forceinline__ void project_as(const void *f, int V, int y, z2 h[6])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        h[c] = f2::dadd(load<SPLIT>(f, V, c, y), times_iq<QA>(load<SPLIT>(f, V, 3 * SA + c, y)));
        h[3 + c] = f2::dadd(load<SPLIT>(f, V, 3 + c, y), times_iq<QB>(load<SPLIT>(f, V, 3 * SB + c, y)));
    }
}

template <bool SPLIT, int S>
__device__ __forceinline__ void project(int mu, const void *f, int V, int y, z2 h[6])
{
    constexpr int P = S > 0 ? 0 : 2, N = 2 - P;   // i^P = S, i^N = -S
    if (mu == 0) project_as<SPLIT, (P + 1) & 3, (P + 1) & 3, 3, 2>(f, V, y, h);
    else if (mu == 1) project_as<SPLIT, P, N, 3, 2>(f, V, y, h);
    else if (mu == 2) project_as<SPLIT, (P + 1) & 3, (N + 1) & 3, 2, 3>(f, V, y, h);
    else project_as<SPLIT, P, P, 2, 3>(f, V, y, h);
}

// w = U h, or U^+ h (ADJ), per spin of the two-spinor
template <bool ADJ>
__device__ __forceinline__ void link_mul(const GaugeStore &U, int V, int mu, int x, const z2 h[6], z2 w[6])
{
    const float4 *p = U.udf + (size_t)mu * 9 * V + x;
    float4 u[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = __ldg(p + (size_t)k * V);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        z2 ih[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) ih[j] = times_i(h[3 * s + j]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Sum t;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float4 m = ADJ ? u[3 * j + i] : u[3 * i + j];
                const df re(m.x, m.y), im = ADJ ? df(-m.z, -m.w) : df(m.z, m.w);
                if (j == 0) t = first_term(re, h[3 * s]);
                else normalise(t), add_term(t, re, h[3 * s + j]);
                add_term(t, im, ih[j]);
            }
            w[3 * s + i] = finish(t);
        }
    }
}

// Warp mu: the two hops of direction mu of site x into sm[mu]
template <int SF, bool SPLIT, class SiteIdx>
__device__ __forceinline__ void hops(const Geom &g, const GaugeStore &U, const void *in, int Vin, int x, const int c[4],
                                     Mem &sm, int mu, int s, SiteIdx sidx)
{
    const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
    const int L = g.L[mu], st = g.stride[mu];
    const bool wf = cm == L - 1, wb = cm == 0;
    const int xf = wc_idx(wf ? x - (L - 1) * st : x + st, g.V), xb = wc_idx(wb ? x + (L - 1) * st : x - st, g.V);
    z2 h[6], a[6], b[6];
    project<SPLIT, SF>(mu, in, Vin, sidx(xf), h);
    link_mul<false>(U, g.V, mu, x, h, a);
    project<SPLIT, -SF>(mu, in, Vin, sidx(xb), h);
    link_mul<true>(U, g.V, mu, xb, h, b);
    if (mu == 3 && g.tbc < 0) {
        const u64 mf = wf ? 0x8000000080000000ull : 0ull, mb = wb ? 0x8000000080000000ull : 0ull;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            a[k] = z2{a[k].h ^ mf, a[k].l ^ mf};
            b[k] = z2{b[k].h ^ mb, b[k].l ^ mb};
        }
    }
    // upper spins from the sum, lower ones from the difference (hop_pair64)
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        sm[mu][k][s] = to4(f2::dadd(a[k], b[k]));
        a[k] = f2::dadd(a[k], neg(b[k]));
    }
    constexpr int P = SF > 0 ? 0 : 2, N = 2 - P;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        z2 l0, l1;
        if (mu == 0) l0 = times_iq<(N + 1) & 3>(a[3 + k]), l1 = times_iq<(N + 1) & 3>(a[k]);
        else if (mu == 1) l0 = times_iq<N>(a[3 + k]), l1 = times_iq<P>(a[k]);
        else if (mu == 2) l0 = times_iq<(N + 1) & 3>(a[k]), l1 = times_iq<(P + 1) & 3>(a[3 + k]);
        else l0 = times_iq<P>(a[k]), l1 = times_iq<P>(a[3 + k]);
        sm[mu][6 + k][s] = to4(l0);
        sm[mu][9 + k][s] = to4(l1);
    }
}

// component k of the sum over the directions
__device__ __forceinline__ z2 sum(const Mem &sm, int k, int s)
{
    return f2::dadd(f2::dadd(of4(sm[0][k][s]), of4(sm[1][k][s])), f2::dadd(of4(sm[2][k][s]), of4(sm[3][k][s])));
}

// rows I0 .. I0 + 2 of y + B v, block b of a packed double-FP32 store
template <int I0>
__device__ __forceinline__ void clover_rows_at(const CloverStore &C, int V, int x, int b, const z2 v[6], Sum y[3])
{
    const float4 *p = C.cdf + (size_t)b * 18 * V + x;
    df d[3];
    if (I0 == 0) {
        const float4 a = __ldg(p), e = __ldg(p + (size_t)V);
        d[0] = df(a.x, a.y), d[1] = df(a.z, a.w), d[2] = df(e.x, e.y);
    } else {
        const float4 a = __ldg(p + (size_t)V), e = __ldg(p + (size_t)2 * V);
        d[0] = df(a.z, a.w), d[1] = df(e.x, e.y), d[2] = df(e.z, e.w);
    }
    z2 iv[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) iv[k] = times_i(v[k]);
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            const bool row = i >= I0 && i < I0 + 3, col = j >= I0 && j < I0 + 3;
            if (!row && !col) continue;
            const float4 e = __ldg(p + (size_t)(3 + i * (i - 1) / 2 + j) * V);
            const df re(e.x, e.y), im(e.z, e.w);
            if (row) {
                add_pair(y[i - I0], re, v[j], im, iv[j]);
            }
            if (col) {   // the mirror entry: conjugate
                add_pair(y[j - I0], re, v[i], -im, iv[i]);
            }
        }
    // the diagonal, the largest term, at the end: the error sums of the others
    // stay small
#pragma unroll
    for (int r = 0; r < 3; ++r) add_term(y[r], d[r], v[I0 + r]);
}

__device__ __forceinline__ void clover_rows(const CloverStore &C, int V, int x, int w, const z2 v[6], Sum y[3])
{
    if (w & 1) clover_rows_at<3>(C, V, x, w >> 1, v, y);
    else clover_rows_at<0>(C, V, x, w >> 1, v, y);
}

}  // namespace dfs
}  // namespace wc
