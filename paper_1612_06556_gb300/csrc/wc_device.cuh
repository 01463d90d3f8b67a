// Device-side types of libwc: complex arithmetic, lattice geometry, the
// device layouts of links and clover, and the per-precision load/store
// traits shared by all kernels.
//
// Device layouts (V = lattice volume, every array plane-major so that one
// warp's 16-byte loads of one component plane are contiguous):
//   spinor  F64: double2 [12][V]       component k = 3*spin + colour
//           F32: float4  [6][V]        chunk j = components 2j, 2j+1
//           F16: uint4   [3][V]        chunk j = components 4j..4j+3 (half2
//                each), times float scale[V] (max |real| of the site)
//   links   FP32/FP16: rows 0 and 1 of U_mu(x) (6 complex, row-major); row 2
//           is rebuilt in registers as conj(row0 x row1) (paper Sec. 2,
//           SU(3) reconstruction) -- these kernels are bandwidth-bound.
//           FP64: all three rows, the third computed once at load time by
//           the same formula: on GB300 the FP64 operator is bound by the
//           FP64 pipe, not by bandwidth, so the rebuild is not repeated.
//           F64: double2 [4][9][V]     F32: float4 [4][3][V]
//           F16: uint4 [4][V] (complex 0..3) + uint2 [4][V] (complex 4, 5)
//   clover  A = 1 + T as two Hermitian 6x6 blocks (spins {0,1} and {2,3},
//           index 3*s_local + colour): per block 6 real diagonal entries then
//           the 15 complex entries below the diagonal in row order
//           (1,0) (2,0) (2,1) (3,0) ... (5,4); 72 reals per site
//           F64: double2 [36][V]; the inverse A^-1 of the even-odd kernels
//           F32: float4 [18][V]    F16: uint4 [9][V]
//           A itself in FP32 and FP16: a block is 1 + [[P, Q^+], [Q, -P]]
//           with P traceless Hermitian and Q any 3x3 matrix (field strengths
//           times csw kappa), 26 reals: the words (P00, P11), P10, P20, P21,
//           Q00, Q01, ... Q22 of two reals each, 13 per block
//           F32: float4 [13][V], block b in planes 6 b .. 6 b + 5 and half b
//           of plane 12;   F16: uint4 [6][V], block b in planes 3 b .. 3 b +
//           2, and uint2 [V], word b: the block's last
//           208 / 104 bytes a site instead of 288 / 144, and the stored
//           values are the small ones: rounding 1 + P to the storage had
//           cost up to 2^-24 / 2^-11 of 1
//   FP64 links and clover are also kept split into double-FP32 pairs (same
//   planes, float4 = hi, lo of the real part, hi, lo of the imaginary part)
//   for the double-FP32 operator (wc_df.cuh).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "wc_check.cuh"
#include "wc_df.cuh"

namespace wc {

// ------------------------------------------------------------------------
// complex arithmetic
// ------------------------------------------------------------------------

template <class R>
struct cx {
    R re, im;
};

template <class R>
__host__ __device__ __forceinline__ cx<R> mkc(R a, R b) { return cx<R>{a, b}; }
template <class R>
__host__ __device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <class R>
__host__ __device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <class R>
__host__ __device__ __forceinline__ cx<R> operator-(cx<R> a) { return {-a.re, -a.im}; }
template <class R>
__host__ __device__ __forceinline__ cx<R> operator*(cx<R> a, cx<R> b)
{
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <class R>
__host__ __device__ __forceinline__ cx<R> operator*(R s, cx<R> a) { return {s * a.re, s * a.im}; }
template <class R>
__host__ __device__ __forceinline__ cx<R> conj(cx<R> a) { return {a.re, -a.im}; }
// i * a
template <class R>
__host__ __device__ __forceinline__ cx<R> times_i(cx<R> a) { return {-a.im, a.re}; }
// conj(a) * b
template <class R>
__host__ __device__ __forceinline__ cx<R> cmul_conj(cx<R> a, cx<R> b)
{
    return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re};
}
// acc + a * b
template <class R>
__host__ __device__ __forceinline__ cx<R> cfma(cx<R> a, cx<R> b, cx<R> acc)
{
    acc.re = fma(a.re, b.re, acc.re);
    acc.re = fma(-a.im, b.im, acc.re);
    acc.im = fma(a.re, b.im, acc.im);
    acc.im = fma(a.im, b.re, acc.im);
    return acc;
}
// acc + conj(a) * b
template <class R>
__host__ __device__ __forceinline__ cx<R> cfma_conj(cx<R> a, cx<R> b, cx<R> acc)
{
    acc.re = fma(a.re, b.re, acc.re);
    acc.re = fma(a.im, b.im, acc.re);
    acc.im = fma(a.re, b.im, acc.im);
    acc.im = fma(-a.im, b.re, acc.im);
    return acc;
}

}  // namespace wc

// the same operators for complex double-FP32 values, on packed float pairs
#include "wc_df2.cuh"

namespace wc {

// ------------------------------------------------------------------------
// geometry
// ------------------------------------------------------------------------

// Division of a non-negative index n < 2^31 by a fixed divisor d without
// the integer-divide instruction sequence: q = floor(n m / 2^k) with
// k = 31 + ceil(log2 d) and m = ceil(2^k / d) < 2^32 is floor(n / d) for
// every such n (Granlund and Montgomery, "Division by invariant integers
// using multiplication", 1994: m d - 2^k < d <= 2^(k - 31)).
struct FastDiv {
    unsigned m;
    int k;
};

inline FastDiv make_fastdiv(int d)
{
    int l = 0;
    while ((1LL << l) < d) ++l;
    const int k = 31 + l;
    const unsigned long long p = 1ULL << k;
    return FastDiv{(unsigned)((p + (unsigned long long)d - 1) / (unsigned long long)d), k};
}

__host__ __device__ __forceinline__ int fast_div(int n, FastDiv f)
{
    return (int)(((unsigned long long)(unsigned)n * f.m) >> f.k);
}

struct Geom {
    int L[4];
    int stride[4];  // 1, Lx, Lx*Ly, Lx*Ly*Lz
    int V;
    int tbc;        // +1 or -1
    FastDiv div[3]; // by L[0], L[1], L[2]
};

// the fast divisors of g.L (host, after L is set)
inline void geom_set_div(Geom &g)
{
    for (int m = 0; m < 3; ++m) g.div[m] = make_fastdiv(g.L[m]);
}

__device__ __forceinline__ void site_coords(const Geom &g, int s, int c[4])
{
    c[0] = s % g.L[0];
    s /= g.L[0];
    c[1] = s % g.L[1];
    s /= g.L[1];
    c[2] = s % g.L[2];
    c[3] = s / g.L[2];
}

// site_coords with the divisions by multiplication.  Measured per operator:
// the whole-lattice FP16 kernel (bound by instruction issue) gains 3 %, the FP32
// one (at 80 registers, bandwidth-bound) loses 2 % and keeps the divisions; the
// four-warp FP64 and double-FP32 kernels, the even-odd passes and the
// multi-field kernels use it.
__device__ __forceinline__ void site_coords_fast(const Geom &g, int s, int c[4])
{
    int q = fast_div(s, g.div[0]);
    c[0] = s - q * g.L[0];
    s = q;
    q = fast_div(s, g.div[1]);
    c[1] = s - q * g.L[1];
    s = q;
    q = fast_div(s, g.div[2]);
    c[2] = s - q * g.L[2];
    c[3] = q;
}

// ------------------------------------------------------------------------
// raw device stores of a lattice
// ------------------------------------------------------------------------

struct GaugeStore {
    double2 *u64 = nullptr;   // [4][9][V]
    float4 *udf = nullptr;    // [4][9][V] u64 as double-FP32 pairs
    float4 *u32 = nullptr;    // [4][3][V]
    uint4 *u16a = nullptr;    // [4][V]  row 0, row 1 entry 0
    uint2 *u16b = nullptr;    // [4][V]  row 1 entries 1, 2
};

struct CloverStore {
    double2 *c64 = nullptr;   // [36][V]
    float4 *cdf = nullptr;    // [36][V] c64 as double-FP32 pairs
    float4 *c32 = nullptr;    // [18][V]  the inverse only
    uint4 *c16 = nullptr;     // [9][V]   the inverse only
    float4 *a32 = nullptr;    // [13][V]  A only
    uint4 *a16 = nullptr;     // [6][V]   A only
    uint2 *a16b = nullptr;    // [V]      A only
};

// Programmatic dependent launch: a kernel launched with the programmatic
// stream serialization attribute may start while the previous kernel of the
// stream drains; griddepcontrol.wait then blocks until that kernel has
// completed and its writes are visible.  launch_dependents lets the next
// such kernel start once every CTA of this grid is running.  Both are no-ops
// for kernels launched without the attribute.
//
// Vectors are read by ordinary loads: a dependent is on the SMs while the
// kernel before it writes its input, and the non-coherent path (__ldg) is for
// data that nothing writes in a kernel's whole lifetime.  Links and clover
// term, which no kernel of a solve writes, keep it.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }

// What the host reads after each step of a solve: written by the step's last
// kernel into page-locked host memory, seq last.
struct StepReport {
    double rr;
    int flags, action;
    volatile unsigned long long seq;
};

// Scalars of one BiCGStab solve, resident on the device.
struct SolverScalars {
    double2 rho, rho0, alpha, omega, beta;
    double rr;       // |r|^2
    double pp, ss;   // |p|^2, |s|^2 (scales of the defect correction)
    double tt;
    int flags;       // bit 0: breakdown, bit 1: non-finite value
    int skip;        // 1: the kernels of a solver step return at once -- this
                     // right-hand side of a lockstep batch has stopped, or a
                     // host-driven solve has to act before its next step
    // host-driven solves: what ends or interrupts the run of steps, decided
    // with the last sum of a step (track_step)
    int track;       // TRACK_*
    int action;      // ACT_*
    double tol2, d2, defer2;        // |r|^2 to reach; delta^2; see reliable_bicgstab
    double rmax2, prev, rr_refresh; // largest |r|^2 since the last refresh, of the last step, of the refresh
};

enum { FLAG_BREAKDOWN = 1, FLAG_NAN = 2 };
enum { TRACK_NONE = 0, TRACK_FP64 = 1, TRACK_RELIABLE = 2, TRACK_INNER = 3 };
enum { ACT_NONE = 0, ACT_STOP = 1, ACT_DIVERGED = 2, ACT_BREAKDOWN = 3, ACT_DEFER = 4, ACT_REFRESH = 5 };

// Reduction scratch: per-block partial sums and a completion ticket.
struct ReduceScratch {
    double *partials = nullptr;   // [2 max_blocks][4]
    unsigned *ticket = nullptr;
    double *result = nullptr;     // [8] final sums (device)
    double *host_result = nullptr;  // [8] pinned host mirror
    int max_blocks = 0;
};

// ------------------------------------------------------------------------
// precision traits: loads and stores of the device layouts
// ------------------------------------------------------------------------

__device__ __forceinline__ cx<float> h2c(unsigned v)
{
    __half2 h = *reinterpret_cast<__half2 *>(&v);
    float2 f = __half22float2(h);
    return {f.x, f.y};
}

__device__ __forceinline__ unsigned c2h(float re, float im)
{
    __half2 h = __floats2half2_rn(re, im);
    return *reinterpret_cast<unsigned *>(&h);
}

// max(a, b, c) in one instruction (three-input max.f32)
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// third row of an SU(3) matrix from its first two: c = conj(a x b)
template <class R>
__device__ __forceinline__ void reconstruct_row2(const cx<R> u[6], cx<R> c[3])
{
    c[0] = conj(u[1] * u[5] - u[2] * u[4]);
    c[1] = conj(u[2] * u[3] - u[0] * u[5]);
    c[2] = conj(u[0] * u[4] - u[1] * u[3]);
}

struct P64 {
    using real = double;
    // register caps of the operator's launch shapes (bit 0: cap 1, bit 1:
    // cap 2) and the minimum resident 256-thread CTAs that cap 1 stands for
    static constexpr int kCaps = 0;   // ALU-bound on the FP64 pipe: no cap
    static constexpr int kCap1MinBlocks = 1;
    static __device__ __forceinline__ void load_spinor(const void *d, const float *, int V, int x,
                                                       cx<double> s[12])
    {
        const double2 *p = static_cast<const double2 *>(d);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            double2 v = p[(size_t)k * V + x];
            s[k] = {v.x, v.y};
        }
    }
    // the stored values and the factor they must be multiplied by (1 here)
    static __device__ __forceinline__ double load_spinor_raw(const void *d, const float *n, int V, int x,
                                                             cx<double> s[12])
    {
        load_spinor(d, n, V, x, s);
        return 1.0;
    }
    static __device__ __forceinline__ void store_spinor(void *d, float *, int V, int x,
                                                        const cx<double> s[12])
    {
        double2 *p = static_cast<double2 *>(d);
#pragma unroll
        for (int k = 0; k < 12; ++k) p[(size_t)k * V + x] = make_double2(s[k].re, s[k].im);
    }
    // U_mu(x): a[0..2] = row 0, a[3..5] = row 1, c[0..2] = row 2
    static __device__ __forceinline__ void load_link(const GaugeStore &g, int V, int mu, int x,
                                                     cx<double> a[6], cx<double> c[3])
    {
        const double2 *p = g.u64 + (size_t)mu * 9 * V + x;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            double2 v = __ldg(p + (size_t)k * V);
            a[k] = {v.x, v.y};
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            double2 v = __ldg(p + (size_t)(6 + k) * V);
            c[k] = {v.x, v.y};
        }
    }
    // the 36 reals of clover block b
    static __device__ __forceinline__ void load_clover(const CloverStore &c, int V, int x, int b,
                                                       double r[36])
    {
        const double2 *p = c.c64 + (size_t)b * 18 * V + x;
#pragma unroll
        for (int k = 0; k < 18; ++k) {
            double2 v = __ldg(p + (size_t)k * V);
            r[2 * k] = v.x;
            r[2 * k + 1] = v.y;
        }
    }
};

struct P32 {
    using real = float;
    static constexpr int kCaps = 3;   // cap 1: 64 registers, cap 2: 85
    static constexpr int kCap1MinBlocks = 4;
    static __device__ __forceinline__ void load_spinor(const void *d, const float *, int V, int x,
                                                       cx<float> s[12])
    {
        const float4 *p = static_cast<const float4 *>(d);
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            float4 v = p[(size_t)j * V + x];
            s[2 * j] = {v.x, v.y};
            s[2 * j + 1] = {v.z, v.w};
        }
    }
    static __device__ __forceinline__ float load_spinor_raw(const void *d, const float *n, int V, int x,
                                                            cx<float> s[12])
    {
        load_spinor(d, n, V, x, s);
        return 1.f;
    }
    static __device__ __forceinline__ void store_spinor(void *d, float *, int V, int x,
                                                        const cx<float> s[12])
    {
        float4 *p = static_cast<float4 *>(d);
#pragma unroll
        for (int j = 0; j < 6; ++j)
            p[(size_t)j * V + x] = make_float4(s[2 * j].re, s[2 * j].im, s[2 * j + 1].re, s[2 * j + 1].im);
    }
    // s as a store_spinor followed by a load_spinor returns it (without the way
    // through memory)
    static __device__ __forceinline__ void as_stored(cx<float> s[12]) {}
    static __device__ __forceinline__ void load_link(const GaugeStore &g, int V, int mu, int x,
                                                     cx<float> a[6], cx<float> c[3])
    {
        const float4 *p = g.u32 + (size_t)mu * 3 * V + x;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float4 v = __ldg(p + (size_t)j * V);
            a[2 * j] = {v.x, v.y};
            a[2 * j + 1] = {v.z, v.w};
        }
        reconstruct_row2(a, c);
    }
    static __device__ __forceinline__ void load_clover(const CloverStore &c, int V, int x, int b,
                                                       float r[36])
    {
        const float4 *p = c.c32 + (size_t)b * 9 * V + x;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            float4 v = __ldg(p + (size_t)k * V);
            r[4 * k] = v.x;
            r[4 * k + 1] = v.y;
            r[4 * k + 2] = v.z;
            r[4 * k + 3] = v.w;
        }
    }
};

// FP64 storage, double-FP32 arithmetic (the operator's FP64 path when the
// lattice selects it): spinors are converted on load and store, links and
// clover come from their pre-split copies.
struct PDF {
    using real = df;
    static constexpr int kCaps = 1;   // cap 1: 128 registers (2 CTAs of 256)
    static constexpr int kCap1MinBlocks = 2;
    static __device__ __forceinline__ void load_spinor(const void *d, const float *, int V, int x, cx<df> s[12])
    {
        const double2 *p = static_cast<const double2 *>(d);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const double2 v = p[(size_t)k * V + x];
            s[k] = {df_from_double(v.x), df_from_double(v.y)};
        }
    }
    static __device__ __forceinline__ df load_spinor_raw(const void *d, const float *n, int V, int x, cx<df> s[12])
    {
        load_spinor(d, n, V, x, s);
        return df(1.0f, 0.0f);
    }
    static __device__ __forceinline__ void store_spinor(void *d, float *, int V, int x, const cx<df> s[12])
    {
        double2 *p = static_cast<double2 *>(d);
#pragma unroll
        for (int k = 0; k < 12; ++k) p[(size_t)k * V + x] = make_double2(df_to_double(s[k].re), df_to_double(s[k].im));
    }
    static __device__ __forceinline__ void load_link(const GaugeStore &g, int V, int mu, int x, cx<df> a[6],
                                                     cx<df> c[3])
    {
        const float4 *p = g.udf + (size_t)mu * 9 * V + x;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const float4 v = __ldg(p + (size_t)k * V);
            a[k] = {df(v.x, v.y), df(v.z, v.w)};
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float4 v = __ldg(p + (size_t)(6 + k) * V);
            c[k] = {df(v.x, v.y), df(v.z, v.w)};
        }
    }
    static __device__ __forceinline__ void load_clover(const CloverStore &c, int V, int x, int b, df r[36])
    {
        const float4 *p = c.cdf + (size_t)b * 18 * V + x;
#pragma unroll
        for (int k = 0; k < 18; ++k) {
            const float4 v = __ldg(p + (size_t)k * V);
            r[2 * k] = df(v.x, v.y);
            r[2 * k + 1] = df(v.z, v.w);
        }
    }
};

struct P16 {
    using real = float;
    static constexpr int kCaps = 3;   // cap 1: 64 registers, cap 2: 85
    static constexpr int kCap1MinBlocks = 4;
    // stored (unit-scaled) values; returns the site's scale, to be folded
    // into a later coefficient instead of multiplying all 24 components
    static __device__ __forceinline__ float load_spinor_raw(const void *d, const float *nrm, int V, int x,
                                                            cx<float> s[12])
    {
        const uint4 *p = static_cast<const uint4 *>(d);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            uint4 v = p[(size_t)j * V + x];
            s[4 * j] = h2c(v.x);
            s[4 * j + 1] = h2c(v.y);
            s[4 * j + 2] = h2c(v.z);
            s[4 * j + 3] = h2c(v.w);
        }
        return nrm[x];
    }
    static __device__ __forceinline__ void load_spinor(const void *d, const float *nrm, int V, int x,
                                                       cx<float> s[12])
    {
        const uint4 *p = static_cast<const uint4 *>(d);
        const float sc = nrm[x];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            uint4 v = p[(size_t)j * V + x];
            s[4 * j] = sc * h2c(v.x);
            s[4 * j + 1] = sc * h2c(v.y);
            s[4 * j + 2] = sc * h2c(v.z);
            s[4 * j + 3] = sc * h2c(v.w);
        }
    }
    static __device__ __forceinline__ void store_spinor(void *d, float *nrm, int V, int x,
                                                        const cx<float> s[12])
    {
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 12; ++k) m = fmax3(m, fabsf(s[k].re), fabsf(s[k].im));
        const float inv = m > 0.f ? 1.f / m : 0.f;
        uint4 *p = static_cast<uint4 *>(d);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            uint4 v;
            v.x = c2h(s[4 * j].re * inv, s[4 * j].im * inv);
            v.y = c2h(s[4 * j + 1].re * inv, s[4 * j + 1].im * inv);
            v.z = c2h(s[4 * j + 2].re * inv, s[4 * j + 2].im * inv);
            v.w = c2h(s[4 * j + 3].re * inv, s[4 * j + 3].im * inv);
            p[(size_t)j * V + x] = v;
        }
        nrm[x] = m;
    }
    // s as a store_spinor followed by a load_spinor returns it
    static __device__ __forceinline__ void as_stored(cx<float> s[12])
    {
        float m = 0.f;
#pragma unroll
        for (int k = 0; k < 12; ++k) m = fmax3(m, fabsf(s[k].re), fabsf(s[k].im));
        const float inv = m > 0.f ? 1.f / m : 0.f;
#pragma unroll
        for (int k = 0; k < 12; ++k) s[k] = m * h2c(c2h(s[k].re * inv, s[k].im * inv));
    }
    static __device__ __forceinline__ void load_link(const GaugeStore &g, int V, int mu, int x,
                                                     cx<float> a[6], cx<float> c[3])
    {
        uint4 v = __ldg(g.u16a + (size_t)mu * V + x);
        uint2 w = __ldg(g.u16b + (size_t)mu * V + x);
        a[0] = h2c(v.x);
        a[1] = h2c(v.y);
        a[2] = h2c(v.z);
        a[3] = h2c(v.w);
        a[4] = h2c(w.x);
        a[5] = h2c(w.y);
        reconstruct_row2(a, c);
    }
    static __device__ __forceinline__ void load_clover(const CloverStore &c, int V, int x, int b,
                                                       float r[36])
    {
        // block b occupies reals 36b .. 36b+35 = chunks 4.5b ... : load all 9
        // chunks' halves that belong to it
        const uint4 *p = c.c16 + x;
#pragma unroll
        for (int k = 0; k < 18; ++k) {
            const int q = 18 * b + k;           // half2 index among 36 per site
            uint4 v = __ldg(p + (size_t)(q >> 2) * V);
            const unsigned w = (q & 3) == 0 ? v.x : (q & 3) == 1 ? v.y : (q & 3) == 2 ? v.z : v.w;
            cx<float> f = h2c(w);
            r[2 * k] = f.re;
            r[2 * k + 1] = f.im;
        }
    }
};

// one packed block of A (36 reals) at position pos of its store in the other
// precisions, and in FP64 too when F64
template <bool F64>
__device__ __forceinline__ void store_clover_a(const CloverStore &S, int V, int pos, int b, const double r[36])
{
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        const double2 v = make_double2(r[2 * q], r[2 * q + 1]);
        if (F64) S.c64[((size_t)b * 18 + q) * V + pos] = v;
        S.cdf[((size_t)b * 18 + q) * V + pos] = df_pack(v);
    }
    // words of two reals: (P00, P11), the lower entries of P, the rows of Q
    constexpr int at[13] = {0, 3, 4, 5, 6, 7, 8, 9, 10, 11, 13, 14, 15};
    float2 w[13];
    w[0] = make_float2((float)(r[0] - 1.0), (float)(r[1] - 1.0));
#pragma unroll
    for (int q = 1; q < 13; ++q) w[q] = make_float2((float)r[2 * at[q]], (float)r[2 * at[q] + 1]);
#pragma unroll
    for (int q = 0; q < 6; ++q)
        S.a32[((size_t)b * 6 + q) * V + pos] = make_float4(w[2 * q].x, w[2 * q].y, w[2 * q + 1].x, w[2 * q + 1].y);
    reinterpret_cast<float2 *>(S.a32 + (size_t)12 * V + pos)[b] = w[12];
    unsigned h[13];
#pragma unroll
    for (int q = 0; q < 13; ++q) h[q] = c2h(w[q].x, w[q].y);
#pragma unroll
    for (int q = 0; q < 3; ++q)
        S.a16[((size_t)b * 3 + q) * V + pos] = make_uint4(h[4 * q], h[4 * q + 1], h[4 * q + 2], h[4 * q + 3]);
    reinterpret_cast<unsigned *>(S.a16b + pos)[b] = h[12];
}

// one packed block (36 reals) of the inverse at position pos of its store, in
// all precisions; 16-byte stores, but for the 8 bytes of each block in the
// binary16 word the two blocks share
__device__ __forceinline__ void store_clover_block(const CloverStore &S, int V, int pos, int b, const double r[36])
{
#pragma unroll
    for (int q = 0; q < 18; ++q) {
        const double2 v = make_double2(r[2 * q], r[2 * q + 1]);
        S.c64[((size_t)b * 18 + q) * V + pos] = v;
        S.cdf[((size_t)b * 18 + q) * V + pos] = df_pack(v);
    }
#pragma unroll
    for (int q = 0; q < 9; ++q)
        S.c32[((size_t)b * 9 + q) * V + pos] =
            make_float4((float)r[4 * q], (float)r[4 * q + 1], (float)r[4 * q + 2], (float)r[4 * q + 3]);
    unsigned h[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) h[q] = c2h((float)r[2 * q], (float)r[2 * q + 1]);
#pragma unroll
    for (int q = 0; q < 4; ++q)
        S.c16[(size_t)((b == 0 ? 0 : 5) + q) * V + pos] =
            make_uint4(b == 0 ? h[4 * q] : h[4 * q + 2], b == 0 ? h[4 * q + 1] : h[4 * q + 3],
                       b == 0 ? h[4 * q + 2] : h[4 * q + 4], b == 0 ? h[4 * q + 3] : h[4 * q + 5]);
    reinterpret_cast<uint2 *>(S.c16 + (size_t)4 * V + pos)[b] =
        b == 0 ? make_uint2(h[16], h[17]) : make_uint2(h[0], h[1]);
}

// Hermitian 6x6 block (packed) times a 6-vector: y = B v
template <class R>
__device__ __forceinline__ void clover_block_mul(const R r[36], const cx<R> v[6], cx<R> y[6])
{
#pragma unroll
    for (int i = 0; i < 6; ++i) y[i] = r[i] * v[i];
    int k = 6;
#pragma unroll
    for (int i = 1; i < 6; ++i) {
#pragma unroll
        for (int j = 0; j < i; ++j) {
            const cx<R> l = mkc(r[k], r[k + 1]);
            k += 2;
            y[i] = cfma(l, v[j], y[i]);        // lower entry (i, j)
            y[j] = cfma_conj(l, v[i], y[j]);   // its mirror (j, i) = conj(l)
        }
    }
}

// y = s y + A v for block b of A in FP32 or FP16 storage: word(k) returns the
// reals of word k as float2.  HAVE: y holds a value (s ignored otherwise).
// The words are used as they arrive, so that few of them are live together.
template <bool HAVE, class Word>
__device__ __forceinline__ void clover_a_mul(Word word, const cx<float> v[6], cx<float> y[6], float s)
{
    const float2 d01 = word(0);
    const float d[3] = {d01.x, d01.y, -(d01.x + d01.y)};
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const float di = i < 3 ? d[i] : -d[i - 3];
        const cx<float> u = HAVE ? mkc(fmaf(s, y[i].re, v[i].re), fmaf(s, y[i].im, v[i].im)) : v[i];
        y[i] = mkc(fmaf(di, v[i].re, u.re), fmaf(di, v[i].im, u.im));
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {   // P10, P20, P21
        const int i = q == 0 ? 1 : 2, j = q == 2 ? 1 : 0;
        const float2 e = word(1 + q);
        const cx<float> l = mkc(e.x, e.y);
        y[i] = cfma(l, v[j], y[i]);
        y[j] = cfma_conj(l, v[i], y[j]);
        y[3 + i] = cfma(l, -v[3 + j], y[3 + i]);
        y[3 + j] = cfma_conj(l, -v[3 + i], y[3 + j]);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float2 e = word(4 + 3 * i + j);
            const cx<float> l = mkc(e.x, e.y);
            y[3 + i] = cfma(l, v[j], y[3 + i]);
            y[j] = cfma_conj(l, v[3 + i], y[j]);
        }
}

// word k of block b at position pos
__device__ __forceinline__ float2 clover_a_word(P32, const CloverStore &C, int V, int pos, int b, int k)
{
    const float4 w = __ldg(C.a32 + (size_t)(k < 12 ? 6 * b + (k >> 1) : 12) * V + pos);
    return (k < 12 ? k & 1 : b) ? make_float2(w.z, w.w) : make_float2(w.x, w.y);
}

// binary16 word k (two halves) of block b at position pos
__device__ __forceinline__ unsigned clover_a_half(const CloverStore &C, int V, int pos, int b, int k)
{
    if (k == 12) {
        const uint2 w = __ldg(C.a16b + pos);
        return b ? w.y : w.x;
    }
    const uint4 w = __ldg(C.a16 + (size_t)(3 * b + (k >> 2)) * V + pos);
    return (k & 3) == 0 ? w.x : (k & 3) == 1 ? w.y : (k & 3) == 2 ? w.z : w.w;
}
__device__ __forceinline__ float2 clover_a_word(P16, const CloverStore &C, int V, int pos, int b, int k)
{
    const cx<float> f = h2c(clover_a_half(C, V, pos, b, k));
    return make_float2(f.re, f.im);
}

// y = A v for block b at position pos of the store of A
template <class P>
__device__ __forceinline__ void clover_a(const CloverStore &C, int V, int pos, int b, const cx<typename P::real> v[6],
                                         cx<typename P::real> y[6])
{
    if constexpr (sizeof(typename P::real) == sizeof(float)) {
        clover_a_mul<false>([&](int k) { return clover_a_word(P(), C, V, pos, b, k); }, v, y, 0.f);
    } else {
        typename P::real r[36];
        P::load_clover(C, V, pos, b, r);
        clover_block_mul(r, v, y);
    }
}

}  // namespace wc
