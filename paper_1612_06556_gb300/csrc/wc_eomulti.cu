// Multi-right-hand-side even-odd (Schur complement) operator:
//   out_r = M^ in_r = A_ee in_r - kappa^2 H_eo A_oo^-1 H_oe in_r   (or M^+)
// for up to kMrhsMax half-lattice fields of one lattice, in two launches
// (odd-site pass, even-site pass) that serve every right-hand side.
//
// The right-hand sides of a propagator share the gauge field, A and A^-1.
// In one pass a site reads its 8 links (4 forward U_mu(x), 4 backward
// U_mu(x - mu)) and one clover-type block (A^-1 on the odd pass, A on the
// even pass): 672 / 592 B per site in FP32, 336 / 296 B in FP16 storage,
// against 96 / 52 B per spinor read or written.  A CTA covers S consecutive
// sites of one parity for all n right-hand sides: it stages those shared
// words once in shared memory (coalesced along the sites), then thread
// (s, r) computes site s of right-hand side r from the staged links and
// block and the 8 neighbour spinors of field r (through L1/L2).  A CTA takes
// 32 sites for up to 6 fields and 16 above: more and smaller CTAs on an SM,
// one of them staging while the others compute.  M^ with 16 / 32 sites, FP32 at
// 16^3x32 4 fields 105 / 103 us, 5 123 / 119, 6 125 / 126, 7 140 / 139, 8 145 /
// 148, at 24^3x32 5 313 / 312, 6 318 / 327, 8 389 / 403, 12 559 / 585, 16 748 /
// 978; binary16 at 24^3x32 5 256 / 236, 6 251 / 252, 7 315 / 304, 8 309 / 322, 12
// 440 / 472, 16 583 / 771 (at 64 registers 16 sites spill, 696 for 12 FP32 fields
// at 24^3x32).  The third
// row of each link is rebuilt once per site after staging (into shared
// memory), not once per right-hand side.  The arithmetic per (site,
// right-hand side) is otherwise that of the single-field pass (spin
// projection, the block product, beta = -kappa^2 on the even pass).  Per-field device flags (the
// skip word of a lockstep batch's solver scalars) may skip fields.
#include <mutex>
#include <string>
#include <type_traits>

#include "wc_internal.cuh"
#include "wc_stencil.cuh"

namespace wc {

namespace {

struct EoMultiArgs {
    int n;
    const void *hin[kMrhsMax];     // hop input (opposite parity)
    const float *hin_nrm[kMrhsMax];
    const void *vin[kMrhsMax];     // site input (even pass)
    const float *vin_nrm[kMrhsMax];
    void *out[kMrhsMax];
    float *out_nrm[kMrhsMax];
    const int *skip[kMrhsMax];     // nullable: *skip[r] != 0 skips right-hand side r
    // even pass only: partial sums of field r for the solver step that
    // follows, per CTA, written to part[(r * gridDim.x + blockIdx.x) * 4 + c]:
    // red 1: <dot[r], out> (c = 0, 1: real, imaginary part); red 2: <out, vin>,
    // |out|^2, |vin|^2.  FP32 fields only.
    int red;
    const void *dot[kMrhsMax];
    double *part;
};

// the staged words of one site: 4 forward and 4 backward links, then the
// block of the pass: A^-1 (MODE 0) or A (MODE 1, see CloverStore)
template <class P>
struct EoMStage;

template <>
struct EoMStage<P32> {
    using W = float4;
    template <int MODE>
    static constexpr int words = 24 + (MODE == 0 ? 18 : 13);   // links [fwd/bwd][mu][3], block
    static __device__ __forceinline__ W link_word(const GaugeStore &U, int V, int mu, int x, int j)
    {
        return __ldg(U.u32 + ((size_t)mu * 3 + j) * V + x);
    }
    template <int MODE>
    static __device__ __forceinline__ void stage(const GaugeStore &U, const CloverStore &C, int V, int item, int x,
                                                 int xb_mu[4], int pos, W &out)
    {
        if (item < 12)
            out = link_word(U, V, item / 3, x, item % 3);
        else if (item < 24)
            out = link_word(U, V, (item - 12) / 3, xb_mu[(item - 12) / 3], (item - 12) % 3);
        else
            out = __ldg((MODE == 0 ? C.c32 : C.a32) + (size_t)(item - 24) * V + pos);
    }
    // the two stored rows of link lam = 4 bwd + mu
    template <int S>
    static __device__ __forceinline__ void rows(const W (*st)[S], int s, int lam, cx<float> a[6])
    {
        const int base = (lam >= 4 ? 12 : 0) + 3 * (lam & 3);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float4 v = st[base + j][s];
            a[2 * j] = mkc(v.x, v.y);
            a[2 * j + 1] = mkc(v.z, v.w);
        }
    }
    // y = A^-1 v or A v, block b
    template <int MODE, int S>
    static __device__ __forceinline__ void block_mul(const W (*st)[S], int s, int b, const cx<float> v[6],
                                                     cx<float> y[6])
    {
        if (MODE == 0) {
            float r[36];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const float4 w = st[24 + 9 * b + q][s];
                r[4 * q] = w.x;
                r[4 * q + 1] = w.y;
                r[4 * q + 2] = w.z;
                r[4 * q + 3] = w.w;
            }
            clover_block_mul(r, v, y);
        } else {
            const auto word = [&](int k) {
                const float4 w = st[24 + (k < 12 ? 6 * b + (k >> 1) : 12)][s];
                return (k < 12 ? k & 1 : b) ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
            };
            clover_a_mul<false>(word, v, y, 0.f);
        }
    }
};

template <>
struct EoMStage<P16> {
    using W = uint4;
    // links: [fwd/bwd][mu] as (uint4 row 0 + entry (1,0)) then the uint2
    // (entries (1,1), (1,2)) of two directions per word; block [9] or [6 + 1]
    template <int MODE>
    static constexpr int words = 8 + 4 + (MODE == 0 ? 9 : 7);
    template <int MODE>
    static __device__ __forceinline__ void stage(const GaugeStore &U, const CloverStore &C, int V, int item, int x,
                                                 int xb_mu[4], int pos, W &out)
    {
        if (item < 8) {
            const int mu = item & 3, y = item < 4 ? x : xb_mu[mu];
            out = __ldg(U.u16a + (size_t)mu * V + y);
        } else if (item < 12) {
            const int k = item - 8;   // words of (fwd mu 0,1), (fwd 2,3), (bwd 0,1), (bwd 2,3)
            const bool bwd = k >= 2;
            const int mu0 = 2 * (k & 1);
            const uint2 a = __ldg(U.u16b + (size_t)mu0 * V + (bwd ? xb_mu[mu0] : x));
            const uint2 b = __ldg(U.u16b + (size_t)(mu0 + 1) * V + (bwd ? xb_mu[mu0 + 1] : x));
            out = make_uint4(a.x, a.y, b.x, b.y);
        } else if (MODE == 0) {
            out = __ldg(C.c16 + (size_t)(item - 12) * V + pos);
        } else if (item < 18) {
            out = __ldg(C.a16 + (size_t)(item - 12) * V + pos);
        } else {
            const uint2 a = __ldg(C.a16b + pos);
            out = make_uint4(a.x, a.y, 0u, 0u);
        }
    }
    template <int S>
    static __device__ __forceinline__ void rows(const W (*st)[S], int s, int lam, cx<float> a[6])
    {
        const int mu = lam & 3;
        const bool bwd = lam >= 4;
        const uint4 v = st[(bwd ? 4 : 0) + mu][s];
        const uint4 w = st[8 + (bwd ? 2 : 0) + (mu >> 1)][s];
        a[0] = h2c(v.x);
        a[1] = h2c(v.y);
        a[2] = h2c(v.z);
        a[3] = h2c(v.w);
        a[4] = h2c((mu & 1) ? w.z : w.x);
        a[5] = h2c((mu & 1) ? w.w : w.y);
    }
    static __device__ __forceinline__ unsigned part(const uint4 &v, int k)
    {
        return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w;
    }
    template <int MODE, int S>
    static __device__ __forceinline__ void block_mul(const W (*st)[S], int s, int b, const cx<float> v[6],
                                                     cx<float> y[6])
    {
        if (MODE == 0) {
            float r[36];
#pragma unroll
            for (int k = 0; k < 18; ++k) {
                const int q = 18 * b + k;   // half2 index among the 36 of a site
                const cx<float> f = h2c(part(st[12 + (q >> 2)][s], q & 3));
                r[2 * k] = f.re;
                r[2 * k + 1] = f.im;
            }
            clover_block_mul(r, v, y);
        } else {
            const auto word = [&](int k) {
                const cx<float> f = h2c(k < 12 ? part(st[12 + 3 * b + (k >> 2)][s], k & 3) : part(st[18][s], b));
                return make_float2(f.re, f.im);
            };
            clover_a_mul<false>(word, v, y, 0.f);
        }
    }
};

// the two hops of direction MU of site x (full index, coordinates c) of the
// half field `in` (opposite parity), or (FIN) of a full-lattice field read at
// the full index; links from the stage, their third rows rebuilt there
template <class P, int MU, int SF, bool FIN, int S>
__device__ __forceinline__ void eom_hops(const Geom &g, const typename EoMStage<P>::W (*st)[S],
                                        const float2 (*r3)[3][S], int s, const void *in, const float *in_nrm, int Vh,
                                        int x, const int c[4], cx<float> acc[12])
{
    const int Vin = FIN ? g.V : Vh;
    const int L = g.L[MU], stride = g.stride[MU];
    const bool wf = c[MU] == L - 1, wb = c[MU] == 0;
    const int xf = wc_idx(wf ? x - (L - 1) * stride : x + stride, g.V);
    const int xb = wc_idx(wb ? x + (L - 1) * stride : x - stride, g.V);
    const auto load = [&](int y, bool wrap, cx<float> p[12]) {   // the factor of the hop
        const float scale = P::load_spinor_raw(in, in_nrm, Vin, FIN ? y : y >> 1, p);
        return (MU == 3 && wrap) ? (float)g.tbc * scale : scale;
    };
    const auto link = [&](int lam, cx<float> u[6], cx<float> r2[3]) {
        EoMStage<P>::rows(st, s, lam, u);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float2 v = r3[lam][j][s];
            r2[j] = mkc(v.x, v.y);
        }
    };
    const auto scaled = [&](float f, cx<float> h[6]) {
        if (std::is_same<P, P32>::value && (MU != 3 || f == 1.f)) return;
#pragma unroll
        for (int k = 0; k < 6; ++k) h[k] = f * h[k];
    };
    {
        cx<float> p[12], h[6], u[6], r2[3];
        const float f = load(xf, wf, p);
        project<MU, SF>(p, h);
        scaled(f, h);
        link(MU, u, r2);
        mul_reconstruct_add<MU, SF, true>(u, r2, h, acc);
    }
    {
        cx<float> p[12], h[6], u[6], r2[3];
        const float f = load(xb, wb, p);
        project<MU, -SF>(p, h);
        scaled(f, h);
        link(4 + MU, u, r2);
        mul_reconstruct_add<MU, -SF, false>(u, r2, h, acc);
    }
}

// full index and coordinates of half index i of parity p (all extents
// even): 2i is the full index of the site with x rounded down to even
__device__ __forceinline__ int eom_full_site(const Geom &g, int i, int p, int c[4])
{
    site_coords_fast(g, 2 * i, c);
    const int bit = (p + c[1] + c[2] + c[3]) & 1;
    c[0] += bit;
    return wc_idx(2 * i + bit, g.V);
}

// MODE 0 (odd pass): out_r = Blk H hin_r      (Blk = A^-1)
// MODE 1 (even pass): out_r = Blk vin_r + beta H hin_r   (Blk = A)
// FULL: the operator's input (hin of the odd pass, vin of the even pass) and
// output are full-lattice fields, the odd-site intermediate stays a half
// field: the even pass writes its site and the zero of the odd site beside
// it, so wc_apply_schur_multi needs no split and merge passes (at
// 16^3x32 with 12 FP32 fields two launches instead of 26: 48 of them, 264
// us, in an M^+ M^ pair before).
template <class P, int DAG, int MODE, bool FULL, int S>
__global__ void __maxnreg__(80) k_eo_multi(Geom g, int p, GaugeStore U, CloverStore Blk,
                                                                   const __grid_constant__ EoMultiArgs a,
                                                                   double beta)
{
    using W = typename EoMStage<P>::W;
    constexpr int NW = EoMStage<P>::template words<MODE>;
    __shared__ W st[NW][S];
    __shared__ float2 r3[8][3][S];   // third rows of the 8 links
    const int Vh = g.V >> 1;
    const int i0 = blockIdx.x * S;
    // blockDim is a multiple of S: a thread stages and computes the
    // same site s
    const int s = threadIdx.x % S, r = threadIdx.x / S, i = i0 + s;
    int c[4] = {0, 0, 0, 0}, x = 0;
    if (i < Vh) {
        x = eom_full_site(g, i, p, c);
        int xb[4];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu)
            xb[mu] = wc_idx(c[mu] == 0 ? x + (g.L[mu] - 1) * g.stride[mu] : x - g.stride[mu], g.V);
        const int pos = wc_idx(p * Vh + i, g.V);
        for (int item = r; item < NW; item += blockDim.x / S)
            EoMStage<P>::template stage<MODE>(U, Blk, g.V, item, x, xb, pos, st[item][s]);
    }
    __syncthreads();
    // the third row of every staged link, once per site
    for (int q = threadIdx.x; q < 8 * S; q += blockDim.x) {
        const int ss = q % S, lam = q / S;
        if (i0 + ss >= Vh) continue;
        cx<float> u[6], c3[3];
        EoMStage<P>::rows(st, ss, lam, u);
        reconstruct_row2(u, c3);
#pragma unroll
        for (int j = 0; j < 3; ++j) r3[lam][j][ss] = make_float2(c3[j].re, c3[j].im);
    }
    __syncthreads();
    if (r >= a.n) return;
    if (a.skip[r] && *a.skip[r]) return;   // all S threads of the field
    float red[4] = {0.f, 0.f, 0.f, 0.f};
    if (i < Vh) {
    constexpr int SF = DAG ? +1 : -1;
    constexpr bool FIN = FULL && MODE == 0;
    cx<float> h[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) h[k] = mkc(0.f, 0.f);
    eom_hops<P, 0, SF, FIN>(g, st, r3, s, a.hin[r], a.hin_nrm[r], Vh, x, c, h);
    eom_hops<P, 1, SF, FIN>(g, st, r3, s, a.hin[r], a.hin_nrm[r], Vh, x, c, h);
    eom_hops<P, 2, SF, FIN>(g, st, r3, s, a.hin[r], a.hin_nrm[r], Vh, x, c, h);
    eom_hops<P, 3, SF, FIN>(g, st, r3, s, a.hin[r], a.hin_nrm[r], Vh, x, c, h);
    cx<float> v[12], o[12];
    const float bt = (float)beta;
    if (MODE == 0) {
#pragma unroll
        for (int k = 0; k < 12; ++k) v[k] = h[k];
    } else {
        P::load_spinor(a.vin[r], a.vin_nrm[r], FULL ? g.V : Vh, FULL ? x : i, v);
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) EoMStage<P>::template block_mul<MODE>(st, s, b, v + 6 * b, o + 6 * b);
    if (MODE == 1)
#pragma unroll
        for (int k = 0; k < 12; ++k) o[k] = o[k] + bt * h[k];
    if constexpr (FULL && MODE == 1) {
        P::store_spinor(a.out[r], a.out_nrm[r], g.V, x, o);
        cx<float> z[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) z[k] = mkc(0.f, 0.f);
        P::store_spinor(a.out[r], a.out_nrm[r], g.V, wc_idx(x ^ 1, g.V), z);   // the row's odd site beside x
    } else {
        P::store_spinor(a.out[r], a.out_nrm[r], Vh, i, o);
    }
    if (MODE == 1 && a.red == 1) {
        cx<float> d[12];
        P32::load_spinor(a.dot[r], nullptr, Vh, i, d);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            red[0] = fmaf(d[k].re, o[k].re, fmaf(d[k].im, o[k].im, red[0]));
            red[1] = fmaf(d[k].re, o[k].im, fmaf(-d[k].im, o[k].re, red[1]));
        }
    } else if (MODE == 1 && a.red == 2) {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            red[0] = fmaf(o[k].re, v[k].re, fmaf(o[k].im, v[k].im, red[0]));
            red[1] = fmaf(o[k].re, v[k].im, fmaf(-o[k].im, v[k].re, red[1]));
            red[2] = fmaf(o[k].re, o[k].re, fmaf(o[k].im, o[k].im, red[2]));
            red[3] = fmaf(v[k].re, v[k].re, fmaf(v[k].im, v[k].im, red[3]));
        }
    }
    }   // i < Vh
    if (MODE == 1 && a.red != 0) {
        // S adjacent lanes hold the sites of this CTA for field r; the other
        // field of the warp may have left it
        const unsigned lanes = S == 32 ? 0xffffffffu : 0xffffu << (threadIdx.x & 16);
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int o2 = S / 2; o2 > 0; o2 >>= 1) red[c] += __shfl_xor_sync(lanes, red[c], o2);
        if (s == 0)
#pragma unroll
            for (int c = 0; c < 4; ++c) a.part[((size_t)r * gridDim.x + blockIdx.x) * 4 + c] = (double)red[c];
    }
}

template <class P, int DAG, bool FULL, int S>
cudaError_t launch_eom_s(const wc_lattice_s *full, int n, wc_field_s *const *outs, wc_field_s *const *ins,
                       wc_field_s *const *tmps, const int *const *skip, int red, wc_field const *dots, double *part,
                       cudaStream_t stream)
{
    const int Vh = full->g.V >> 1;
    const dim3 grid((Vh + S - 1) / S), block(S * n);
    EoMultiArgs a{};
    a.n = n;
    for (int r = 0; r < n; ++r) {
        a.skip[r] = skip ? skip[r] : nullptr;
        a.hin[r] = ins[r]->data;
        a.hin_nrm[r] = ins[r]->nrm;
        a.out[r] = tmps[r]->data;
        a.out_nrm[r] = tmps[r]->nrm;
    }
    // odd sites: tmp = A_oo^-1 H_oe in
    k_eo_multi<P, DAG, 0, FULL, S><<<grid, block, 0, stream>>>(full->g, 1, full->gauge, full->cinv, a, 0.0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // even sites: out = A_ee in - kappa^2 H_eo tmp
    for (int r = 0; r < n; ++r) {
        a.hin[r] = tmps[r]->data;
        a.hin_nrm[r] = tmps[r]->nrm;
        a.vin[r] = ins[r]->data;
        a.vin_nrm[r] = ins[r]->nrm;
        a.out[r] = outs[r]->data;
        a.out_nrm[r] = outs[r]->nrm;
    }
    a.red = red;
    a.part = part;
    for (int r = 0; r < n && red == 1; ++r) a.dot[r] = dots[r]->data;
    k_eo_multi<P, DAG, 1, FULL, S><<<grid, block, 0, stream>>>(full->g, 0, full->gauge, full->ceo, a,
                                                      -full->kappa * full->kappa);
    return cudaGetLastError();
}

constexpr int kEomSmall = 6;   // fields up to which a CTA takes 32 sites

template <class P, int DAG, bool FULL>
cudaError_t launch_eom(const wc_lattice_s *full, int n, wc_field_s *const *outs, wc_field_s *const *ins,
                       wc_field_s *const *tmps, const int *const *skip, int red, wc_field const *dots, double *part,
                       cudaStream_t stream)
{
    return n > kEomSmall ? launch_eom_s<P, DAG, FULL, 16>(full, n, outs, ins, tmps, skip, red, dots, part, stream)
                         : launch_eom_s<P, DAG, FULL, 32>(full, n, outs, ins, tmps, skip, red, dots, part, stream);
}

}  // namespace

cudaError_t launch_schur_multi(wc_lattice half, int n, wc_field const *outs, wc_field const *ins,
                               wc_field const *tmps, const int *const *skip, cudaStream_t stream, int red,
                               wc_field const *dots, double *part)
{
    if (n < 1 || n > kMrhsMax || !half->schur_parent) return cudaErrorInvalidValue;
    const wc_lattice_s *full = half->schur_parent;
    const wc_prec pr = ins[0]->prec;
    if (red != 0 && (pr != WC_F32 || !part || (red == 1 && !dots))) return cudaErrorInvalidValue;
    if (pr == WC_F32) return launch_eom<P32, 0, false>(full, n, outs, ins, tmps, skip, red, dots, part, stream);
    if (pr == WC_F16) return launch_eom<P16, 0, false>(full, n, outs, ins, tmps, skip, 0, nullptr, nullptr, stream);
    return cudaErrorInvalidValue;
}

int schur_multi_blocks(wc_lattice half, int n)
{
    const int S = n > kEomSmall ? 16 : 32;
    return (half->g.V + S - 1) / S;
}

}  // namespace wc

using namespace wc;

// outs[r] = M^ ins[r] (even sites; odd sites of outs set to zero) for FP32
// or FP16 full-lattice fields of one lattice
extern "C" wc_status wc_apply_schur_multi(wc_lattice lat, int n, wc_field *outs, wc_field *ins, int dagger)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (n < 1 || n > kMrhsMax || !outs || !ins)
        return set_error(lat, WC_ERR_ARG, "n must be in 1.." + std::to_string(kMrhsMax) + ", outs/ins non-NULL");
    for (int r = 0; r < n; ++r) {
        if (!outs[r] || !ins[r] || outs[r]->lat != lat || ins[r]->lat != lat)
            return set_error(lat, WC_ERR_ARG, "fields must belong to the lattice");
        if (ins[r]->prec != ins[0]->prec || outs[r]->prec != ins[0]->prec || ins[0]->prec == WC_F64)
            return set_error(lat, WC_ERR_ARG, "the multi-RHS Schur operator takes FP32 or FP16 fields of one precision");
        for (int q = 0; q < n; ++q)
            if (outs[r] == ins[q] || (q < r && outs[r] == outs[q]))
                return set_error(lat, WC_ERR_ARG, "out fields must be distinct from each other and from the inputs");
    }
    wc_status st = require_operator(lat);
    if (st != WC_OK) return st;
    wc_lattice h = nullptr;
    st = half_lattice(lat, &h);
    if (st != WC_OK) return st;
    const wc_prec pr = ins[0]->prec;
    const int Vh = h->g.V;
    // n odd-site intermediates in the lattice's workspace, kept between
    // calls up to kKeptWorkspace (allocating three half fields per right-hand
    // side on every call cost 2.7 ms of a 2.9 ms call at 12 right-hand sides and
    // 16^3x32; a larger workspace goes with a call of milliseconds); one
    // call at a time uses it: the lock is held until the stream has finished
    const size_t data_bytes = (spinor_bytes(pr, Vh) + 255) / 256 * 256;
    const size_t nrm_bytes = pr == WC_F16 ? ((size_t)Vh * sizeof(float) + 255) / 256 * 256 : 0;
    std::lock_guard<std::mutex> lk(lat->eom_mutex);
    if (lat->eom_ws_bytes < (data_bytes + nrm_bytes) * n) {
        cudaFree(lat->eom_ws);
        lat->eom_ws = nullptr;
        lat->eom_ws_bytes = 0;
        st = check_cuda(lat, cudaMalloc(&lat->eom_ws, (data_bytes + nrm_bytes) * n), "cudaMalloc(schur_multi)");
        if (st != WC_OK) return st;
        lat->eom_ws_bytes = (data_bytes + nrm_bytes) * n;
    }
    wc_field_s tmp[kMrhsMax];
    wc_field_s *tmps[kMrhsMax];
    char *ws = static_cast<char *>(lat->eom_ws);
    for (int k = 0; k < n; ++k, ws += data_bytes + nrm_bytes) {
        tmp[k].lat = h;
        tmp[k].prec = pr;
        tmp[k].data = ws;
        tmp[k].nrm = nrm_bytes ? reinterpret_cast<float *>(ws + data_bytes) : nullptr;
        tmps[k] = &tmp[k];
    }
    cudaError_t e;
    if (pr == WC_F32)
        e = dagger ? launch_eom<P32, 1, true>(lat, n, outs, ins, tmps, nullptr, 0, nullptr, nullptr, lat->stream)
                   : launch_eom<P32, 0, true>(lat, n, outs, ins, tmps, nullptr, 0, nullptr, nullptr, lat->stream);
    else
        e = dagger ? launch_eom<P16, 1, true>(lat, n, outs, ins, tmps, nullptr, 0, nullptr, nullptr, lat->stream)
                   : launch_eom<P16, 0, true>(lat, n, outs, ins, tmps, nullptr, 0, nullptr, nullptr, lat->stream);
    st = check_cuda(lat, e, "schur_multi");
    if (st == WC_OK) st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync");
    if (lat->eom_ws_bytes > kKeptWorkspace) {
        cudaFree(lat->eom_ws);
        lat->eom_ws = nullptr;
        lat->eom_ws_bytes = 0;
    }
    return st;
}
