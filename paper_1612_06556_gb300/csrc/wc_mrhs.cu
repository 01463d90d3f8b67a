// Multi-right-hand-side Wilson-Clover operator: out_r = M in_r (or M^+ in_r)
// for up to kMrhsMax fields of one lattice in one launch.
//
// The right-hand sides of a propagator share the gauge field and the clover
// term, which are 400 of the 592 bytes per site of a single FP32 apply.  A
// CTA covers S consecutive sites for all n right-hand sides: it
// first stages, once, the 4 forward links of its sites, the 4 backward links
// U_mu(x - mu) of their neighbours and their clover blocks in shared memory
// (37 float4 per site, coalesced along the sites), then thread (s, r)
// computes site s of right-hand side r, reading links and clover from
// shared memory and the 9 spinors of field r from global memory (neighbours
// through L1/L2); the third row of each link is rebuilt once per site
// after staging.  Compulsory bytes per site and right-hand side:
// 2 x 96 (spinor in, out) + 400 / n, i.e. 225 B at n = 12 against 592 B for
// separate applies.
//
// What bounds it is the latency of the neighbour spinors in L2 (the CTA's own
// sites serve two of the nine reads from L1) and the L1 data path, so warps
// per SM count, and CTAs small enough that one stages while others compute:
// 16 sites and 64 registers (32 warps) above four right-hand sides, 32 sites
// and 80 registers up to four, where a CTA has few warps anyway.  24^3x32,
// 16 x 64 / 32 x 80: 298 / 313 us for one field (16^3x32 87 / 83), 210 / 206 for
// 2, 204 / 189 for 3, 219 / 204 for 4, 236 / 258 for 5, 232 / 265 for 6, 277 /
// 324 for 8, 410 / 468 for 12, 527 / 791 for 16; 96 registers 491 / 686 for 12, 8
// sites 544.
#include "wc_internal.cuh"
#include "wc_stencil.cuh"

namespace wc {

namespace {

constexpr int kStageF4 = 37;   // float4 per site: 12 forward link, 12 backward link, 13 clover

struct MrhsArgs {
    int n;
    const float4 *in[kMrhsMax];
    float4 *out[kMrhsMax];
};

template <int S>
struct Stage {
    float4 w[kStageF4][S];
    float2 r3[8][3][S];   // third rows of the 8 links
};

// the two stored rows of staged link lam (mu, or 4 + mu for U_mu(x - mu))
template <int S>
__device__ __forceinline__ void rows_from_stage(const Stage<S> &st, int lam, int s, cx<float> a[6])
{
#pragma unroll
    for (int j = 0; j < 3; ++j) {   // words 0-11 forward, 12-23 backward links
        const float4 v = st.w[3 * lam + j][s];
        a[2 * j] = mkc(v.x, v.y);
        a[2 * j + 1] = mkc(v.z, v.w);
    }
}

// the hop from site y: acc += ph W (1 + SG g_MU) in(y), W the staged link lam
// (FWD) or its adjoint
template <int MU, int SG, bool FWD, int S>
__device__ __forceinline__ void hop_mrhs(const Stage<S> &st, int s, const float4 *in, int V, int y, float ph,
                                         cx<float> acc[12])
{
    constexpr int lam = FWD ? MU : 4 + MU;
    cx<float> h[6], u[6], r2[3];
    {
        // never a programmatic dependent, so that the read-only path is open:
        // 410 us for 12 fields at 24^3x32, 417 by ordinary loads
        cx<float> p[12];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const float4 v = __ldg(in + (size_t)j * V + y);
            p[2 * j] = mkc(v.x, v.y);
            p[2 * j + 1] = mkc(v.z, v.w);
        }
        project<MU, SG>(p, h);
    }
    if (MU == 3 && ph != 1.f) {
#pragma unroll
        for (int k = 0; k < 6; ++k) h[k] = ph * h[k];
    }
    rows_from_stage(st, lam, s, u);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float2 v = st.r3[lam][j][s];
        r2[j] = mkc(v.x, v.y);
    }
    mul_reconstruct_add<MU, SG, FWD>(u, r2, h, acc);
}

template <int MU, int SF, int S>
__device__ __forceinline__ void hops_mrhs(const Geom &g, const Stage<S> &st, int s, const float4 *in, int x,
                                          const int c[4], cx<float> acc[12])
{
    const int L = g.L[MU], stl = g.stride[MU];
    const bool wf = c[MU] == L - 1, wb = c[MU] == 0;
    const int xf = wc_idx(wf ? x - (L - 1) * stl : x + stl, g.V), xb = wc_idx(wb ? x + (L - 1) * stl : x - stl, g.V);
    hop_mrhs<MU, SF, true>(st, s, in, g.V, xf, MU == 3 && wf ? (float)g.tbc : 1.f, acc);
    hop_mrhs<MU, -SF, false>(st, s, in, g.V, xb, MU == 3 && wb ? (float)g.tbc : 1.f, acc);
}

// KIND 0: M, 1: M^+.  blockDim = S * n.
template <int KIND, int S>
__global__ void __maxnreg__(S == 16 ? 64 : 80)
    k_apply_mrhs(Geom g, GaugeStore U, CloverStore C, const __grid_constant__ MrhsArgs a, double kappa)
{
    __shared__ Stage<S> st;
    const int x0 = blockIdx.x * S;
    // blockDim is a multiple of S: a thread stages and computes the same site s
    const int s = threadIdx.x % S, r = threadIdx.x / S, x = x0 + s;
    int c[4] = {0, 0, 0, 0};
    if (x < g.V) {
        site_coords_fast(g, x, c);
        for (int item = r; item < kStageF4; item += blockDim.x / S) {
            float4 v;
            if (item < 12) {                               // U_mu(x), plane item of [4][3][V]
                v = __ldg(U.u32 + (size_t)item * g.V + x);
            } else if (item < 24) {                        // U_mu(x - mu)
                const int mu = (item - 12) / 3, j = (item - 12) % 3;
                const int xb = wc_idx(c[mu] == 0 ? x + (g.L[mu] - 1) * g.stride[mu] : x - g.stride[mu], g.V);
                v = __ldg(U.u32 + ((size_t)mu * 3 + j) * g.V + xb);
            } else {                                       // clover plane item - 24 of [13][V]
                v = __ldg(C.a32 + (size_t)(item - 24) * g.V + x);
            }
            st.w[item][s] = v;
        }
    }
    __syncthreads();
    // the third row of every staged link, once per site
    for (int q = threadIdx.x; q < 8 * S; q += blockDim.x) {
        const int ss = q % S, lam = q / S;
        if (x0 + ss >= g.V) continue;
        cx<float> u[6], c3[3];
        rows_from_stage(st, lam, ss, u);
        reconstruct_row2(u, c3);
#pragma unroll
        for (int j = 0; j < 3; ++j) st.r3[lam][j][ss] = make_float2(c3[j].re, c3[j].im);
    }
    __syncthreads();
    if (r >= a.n || x >= g.V) return;
    const float4 *in = a.in[r];
    cx<float> acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = mkc(0.f, 0.f);
    constexpr int SF = KIND == 1 ? +1 : -1;
    hops_mrhs<0, SF>(g, st, s, in, x, c, acc);
    hops_mrhs<1, SF>(g, st, s, in, x, c, acc);
    hops_mrhs<2, SF>(g, st, s, in, x, c, acc);
    hops_mrhs<3, SF>(g, st, s, in, x, c, acc);
    // A in - kappa (hops), a clover block at a time
    const float mk = (float)(-kappa);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        cx<float> v[6];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float4 w = __ldg(in + (size_t)(3 * b + j) * g.V + x);
            v[2 * j] = mkc(w.x, w.y);
            v[2 * j + 1] = mkc(w.z, w.w);
        }
        const auto word = [&](int k) {
            const float4 w = st.w[24 + (k < 12 ? 6 * b + (k >> 1) : 12)][s];
            return (k < 12 ? k & 1 : b) ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
        };
        clover_a_mul<true>(word, v, acc + 6 * b, mk);
    }
    P32::store_spinor(a.out[r], nullptr, g.V, x, acc);
}

}  // namespace

cudaError_t launch_apply_multi(wc_lattice lat, int n, const wc_field *outs, const wc_field *ins, int kind,
                               cudaStream_t stream)
{
    if (n < 1 || n > kMrhsMax) return cudaErrorInvalidValue;
    MrhsArgs a{};
    a.n = n;
    for (int r = 0; r < n; ++r) {
        a.in[r] = static_cast<const float4 *>(ins[r]->data);
        a.out[r] = static_cast<float4 *>(outs[r]->data);
    }
    const Geom &g = lat->g;
    const int S = n > 4 ? 16 : 32;
    const auto kern = S == 16 ? (kind == 1 ? k_apply_mrhs<1, 16> : k_apply_mrhs<0, 16>)
                              : (kind == 1 ? k_apply_mrhs<1, 32> : k_apply_mrhs<0, 32>);
    kern<<<(g.V + S - 1) / S, S * n, 0, stream>>>(g, lat->gauge, lat->clover, a, lat->kappa);
    return cudaGetLastError();
}

}  // namespace wc
