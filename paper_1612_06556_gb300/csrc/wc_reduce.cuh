// Grid sums in one launch, the scalar updates of BiCGStab that follow them, and
// the sums that an operator pass forms from the field it has just computed.
#pragma once

#include <math.h>

#include "wc_internal.cuh"

namespace wc {

// Sums of v[0..N) over the lanes, N = 1, 2 or 4: lane l returns the sum of
// v[l / (32 / N)].
template <int N, class T>
__device__ __forceinline__ T warp_sums(T (&v)[N])
{
    static_assert(N == 1 || N == 2 || N == 4, "one, two or four sums");
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int half = N / 2, o = 16; half > 0; half /= 2, o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const T give = up ? v[i] : v[half + i], keep = up ? v[half + i] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (int o = 16 / N; o > 0; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

constexpr int kRedBlock = 256;
constexpr int kRedWarps = kRedBlock / 32;

// Sum i over w[.][k] where warp k of the block has put its sums (lane i * W +
// k of the calling warp reads it): every lane of i * W .. i * W + W - 1.
template <int N, int W, class T>
__device__ __forceinline__ T block_sums(const T (&w)[N][W])
{
    static_assert(N * W <= 32 && (W & (W - 1)) == 0, "a lane for each value");
    const int lane = threadIdx.x & 31;
    T u = lane < N * W ? w[lane / W][lane % W] : T(0);
#pragma unroll
    for (int o = W / 2; o > 0; o /= 2) u += __shfl_xor_sync(0xffffffffu, u, o);
    return u;
}

struct NoUpdate {
    __device__ void operator()(double, const double *) const {}
};
struct NoAhead {
    __device__ double operator()() const { return 0.0; }
};


// Reduce acc[0..M) over the grid (blocks of 32 W threads, one dimension x; at
// least 4 gridDim.x doubles of partials).  The last block to arrive leaves the
// grid sums in out[0..M), summed in a fixed order, and its warp 0 calls
// post(t, extra) with sum i in lane i (zero above).  ahead() runs meanwhile in
// the last warp of that block; extra[l] is what lane l of it returned.
template <int M, int W = kRedWarps, class T, class Post = NoUpdate, class Ahead = NoAhead>
__device__ __forceinline__ void grid_reduce(T (&acc)[M], const ReduceScratch &rs, double *out, Post post = Post(),
                                            Ahead ahead = Ahead())
{
    constexpr int N = M == 3 ? 4 : M;
    __shared__ T sm[N][W];
    __shared__ double fin[W < N ? N : W], extra[32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = i < M ? acc[i] : T(0);
    const T t = warp_sums(v);
    if (lane % (32 / N) == 0) sm[lane / (32 / N)][wid] = t;
    __syncthreads();
    if (wid == 0) {
        const T u = block_sums(sm);
        if (lane < M * W && lane % W == 0) rs.partials[(size_t)blockIdx.x * 4 + lane / W] = (double)u;
        __syncwarp();
        // the fences stand between the other lanes' partials and this
        // lane's ticket, and between the ticket and the block's reads
        if (lane == 0) {
            __threadfence();
            last = atomicAdd(rs.ticket, 1u) == gridDim.x - 1;
            __threadfence();
        }
    }
    __syncthreads();
    if (!last) return;
    if constexpr (W < N) {
        // a single warp: all sums in one loop, so that their loads overlap
        static_assert(W == 1, "one warp, or one for each sum");
        double p[N] = {};
#pragma unroll 4
        for (int b = lane; b < (int)gridDim.x; b += 32)
#pragma unroll
            for (int i = 0; i < M; ++i) p[i] += __ldcg(rs.partials + (size_t)b * 4 + i);
        const double s = warp_sums(p);
        if (lane % (32 / N) == 0) fin[lane / (32 / N)] = s;
    } else {
        // warp w adds the partials of sum w % N
        double s = 0.0;
        const int i = wid % N;
        if (i < M) {
#pragma unroll 4
            for (int b = (wid / N) * 32 + lane; b < (int)gridDim.x; b += 32 * W / N)
                s += __ldcg(rs.partials + (size_t)b * 4 + i);
            double one[1] = {s};
            s = warp_sums(one);
        }
        if (lane == 0) fin[wid] = s;
    }
    if (wid == W - 1) extra[lane] = ahead();
    __syncthreads();
    if (wid != 0) return;
    double u = lane < (W < N ? N : W) ? fin[lane] : 0.0;
#pragma unroll
    for (int o = N; o < W; o *= 2) u += __shfl_xor_sync(0xffffffffu, u, o);
    if (lane >= M) u = 0.0;
    if (lane < M) out[lane] = u;
    if (lane == 0) *rs.ticket = 0u;
    post(u, extra);
}

__device__ __forceinline__ cx<double> c_of(double2 a) { return {a.x, a.y}; }

// ---- scalar updates, run by one warp -------------------------------------
// t: sum i of the reduction in lane i.

__device__ __forceinline__ double sum_of(double t, int i) { return __shfl_sync(0xffffffffu, t, i); }

// a / b, the real part in even lanes, the imaginary part in odd ones
__device__ __forceinline__ double cdiv_part(cx<double> a, cx<double> b)
{
    const bool im = threadIdx.x & 1;
    const double d = b.re * b.re + b.im * b.im;
    const double p = im ? a.im : a.re, q = im ? -a.re : a.im;
    return (p * b.re + q * b.im) / d;
}

// alpha = rho / <rhat, v>
__device__ __forceinline__ void alpha_update(double t, SolverScalars *sc)
{
    const int lane = threadIdx.x & 31;
    const cx<double> rv = mkc(sum_of(t, 0), sum_of(t, 1));
    const double a = cdiv_part(c_of(sc->rho), rv);
    const bool zero = rv.re == 0.0 && rv.im == 0.0;
    if (lane < 2) (&sc->alpha.x)[lane] = zero ? 0.0 : a;
    if (lane == 0) {
        if (!isfinite(rv.re) || !isfinite(rv.im)) sc->flags |= FLAG_NAN;
        if (zero) sc->flags |= FLAG_BREAKDOWN;
    }
}

// omega = <t, s> / <t, t>
__device__ __forceinline__ void omega_update(double t, SolverScalars *sc)
{
    const int lane = threadIdx.x & 31;
    const double tt = sum_of(t, 2);
    const bool bad = !isfinite(tt) || !isfinite(sum_of(t, 0)) || !isfinite(sum_of(t, 1));
    const double om = t / tt;
    if (lane < 2) (&sc->omega.x)[lane] = tt > 0.0 ? om : 0.0;
    if (lane == 0) {
        sc->tt = tt;
        if (bad) sc->flags |= FLAG_NAN;
    }
}

// omega from <t, s>, <t, t>, <s, s>
__device__ __forceinline__ void lo_omega_update(double t, SolverScalars *sc)
{
    const int lane = threadIdx.x & 31;
    const double tr = sum_of(t, 0), ti = sum_of(t, 1), tt = sum_of(t, 2), ss = sum_of(t, 3);
    double om = tt > 0.0 ? t / tt : 0.0;
    // omega stabilisation (Sleijpen & van der Vorst): when t and s are
    // nearly orthogonal, |<t,s>| / (|t||s|) < 0.7, the minimising omega is
    // tiny and BiCGStab loses accuracy in finite precision; enlarge it
    // (the squares first: the roots are wanted only then)
    const double c2 = tr * tr + ti * ti;
    if (tt > 0.0 && ss > 0.0 && c2 > 0.0 && c2 < 0.5 * (tt * ss)) {
        const double rho_t = sqrt(c2) / sqrt(tt * ss);
        if (rho_t < 0.7) om *= 0.7 / rho_t;
    }
    if (lane < 2) (&sc->omega.x)[lane] = om;
    if (lane == 0) {
        sc->tt = tt;
        if (!isfinite(tt) || !isfinite(tr) || !isfinite(ti) || !isfinite(ss)) sc->flags |= FLAG_NAN;
    }
}

// ---- sums formed by the operator pass of a solver step -------------------
// The pass that produces v = op phat (or t = op shat) has every component in
// registers: with one more read, of rhat (or s), it forms the sums of alpha
// (or omega) too, and its last CTA the scalar.  That saves the pass over both
// vectors, its launch and its share of the tail, twice a step: FP64 at 8^4
// 63.2 -> 55.0 us a step, even-odd FP64 at 12^4 180.6 -> 167.3, binary16 at
// 16^3x32 121.7 -> 116.3.

// The pass forms the sums itself if its last CTA has no more than two partials
// per SM to add up for each of its warps.  Its few warps read them one after
// the other, where a reduction of 256 threads has eight warps and four blocks
// per SM: at 16^4 (1024 CTAs of one warp) 95.3 us a step with separate passes
// and 96.0 in the operator's, binary16 at 24^3x32 (1728 CTAs of four) 217 and
// 222; at 16^3x32 (512 CTAs of four) 121.7 and 116.3.
inline bool sum_in_pass(const ReduceScratch &rs, int ctas, int warps)
{
    return ctas <= rs.max_blocks / 2 * warps && ctas <= 2 * rs.max_blocks;   // the partials hold four sums of each
}

struct StepSum {
    const void *with;        // rhat, or s
    const float *with_nrm;
    ReduceScratch rs;
    SolverScalars *sc;
};

// The contribution of N components: y of v or t, a of rhat or s
template <bool OMEGA, int N, class R, int M>
__device__ __forceinline__ void add_step_sums(const cx<R> *y, const cx<R> *a, R (&acc)[M])
{
#pragma unroll
    for (int k = 0; k < N; ++k) {
        // <rhat, v> or <t, s>
        const cx<R> l = OMEGA ? y[k] : a[k], r = OMEGA ? a[k] : y[k];
        acc[0] = fma(l.re, r.re, fma(l.im, r.im, acc[0]));
        acc[1] = fma(l.re, r.im, fma(-l.im, r.re, acc[1]));
        if (M > 2) acc[2] = fma(y[k].re, y[k].re, fma(y[k].im, y[k].im, acc[2]));
        if (M > 3) acc[3] = fma(a[k].re, a[k].re, fma(a[k].im, a[k].im, acc[3]));
    }
}

// number of sums: alpha two, omega three in FP64, four in the low precisions
template <bool OMEGA, class R>
constexpr int step_sums = !OMEGA ? 2 : sizeof(R) == sizeof(double) ? 3 : 4;

template <bool OMEGA, int W, class R, int M>
__device__ __forceinline__ void reduce_step_sums(R (&acc)[M], const StepSum &ss)
{
    SolverScalars *sc = ss.sc;
    grid_reduce<M, W>(acc, ss.rs, ss.rs.result, [=](double t, const double *) {
        if (!OMEGA) alpha_update(t, sc);
        else if (M == 3) omega_update(t, sc);
        else lo_omega_update(t, sc);
    });
}

}  // namespace wc
