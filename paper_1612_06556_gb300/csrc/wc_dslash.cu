// Wilson-Clover operator kernels: out = M in, M^+ in, H in; field casts.
//
// One thread per site.  Sites map to threads either in lexicographic order
// or by 4-D tiles (a CTA covers a tx*ty*tz*tt brick, x fastest, so a warp's
// loads stay 128-byte contiguous and the x/y/z neighbours of most sites lie
// in the same CTA); the 8-fold reuse of each input spinor is served by
// L1/L2.  The mapping, CTA size and register cap are picked per lattice
// extent, precision and operator by a small autotuner (first use, timed with
// CUDA events; not while the stream is being captured).  Per direction the neighbour spinor is spin
// projected to a two-spinor before the SU(3) multiply, halving the matvec
// work (paper Sec. 2/3, the hopping multiplication "MULT"); links are read as
// two rows and the third rebuilt in registers (SU(3) reconstruction).  The
// clover term (two packed Hermitian 6x6 blocks) is applied to the centre
// spinor first and the hops are accumulated into that result with the
// coefficient -kappa, so out = (1 + T) in - kappa H in is written once.
//
#include <array>
#include <map>
#include <mutex>
#include <type_traits>

#include "wc_internal.cuh"
#include "wc_reduce.cuh"
#include "wc_stencil.cuh"
#include "wc_dfsplit.cuh"

namespace wc {

namespace {

constexpr int kApplyMaxThreads = 256;

// Site of (block, thread) under a launch shape: tile[] = {0,0,0,0} means
// lexicographic order, else tile extents (x fastest) tiling the lattice.
struct TileMap {
    int tile[4];
    int ntile[3];   // tiles along x, y, z
};

__device__ __forceinline__ int site_of_thread(const Geom &g, const TileMap &m, int blk, bool &valid)
{
    if (m.tile[0] == 0) {
        const int x = blk * blockDim.x + threadIdx.x;
        valid = x < g.V;
        return x;
    }
    int t = threadIdx.x, b = blk;
    const int cx = (b % m.ntile[0]) * m.tile[0] + t % m.tile[0];
    t /= m.tile[0];
    b /= m.ntile[0];
    const int cy = (b % m.ntile[1]) * m.tile[1] + t % m.tile[1];
    t /= m.tile[1];
    b /= m.ntile[1];
    const int cz = (b % m.ntile[2]) * m.tile[2] + t % m.tile[2];
    t /= m.tile[2];
    b /= m.ntile[2];
    const int ct = b * m.tile[3] + t;
    valid = true;
    return cx + g.stride[1] * cy + g.stride[2] * cz + g.stride[3] * ct;
}

template <class P, int KIND>
__device__ __forceinline__ void apply_site(const Geom &g, const TileMap &tm, int blk, const GaugeStore &U,
                                           const CloverStore &C, const void *in, const float *in_nrm, void *out,
                                           float *out_nrm, double kappa)
{
    bool valid;
    const int x = site_of_thread(g, tm, blk, valid);
    if (valid) apply_site_at<P, KIND>(g, x, U, C, in, in_nrm, out, out_nrm, kappa);
}

// Bulk L2 prefetch of n bytes at p (both 16-byte multiples); only a cache
// hint: L2 is the point of coherence, so data still being written by the
// previous kernel is read correctly by the loads after griddep_wait().
__device__ __forceinline__ void prefetch_l2(const void *p, unsigned n)
{
    if (n >= 16 && (reinterpret_cast<uintptr_t>(p) & 15) == 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(n & ~15u) : "memory");
}

// The links and clover term of sites [x0, x0 + n) (lexicographic block),
// one contiguous range per component plane; plane i is issued by thread i.
template <class P>
__device__ __forceinline__ void prefetch_block(const Geom &g, const GaugeStore &U, const CloverStore &C, int x0,
                                               int n, int i)
{
    const size_t V = g.V;
    if (std::is_same<P, P32>::value) {
        if (i < 12) prefetch_l2(U.u32 + i * V + x0, 16u * n);                   // [4][3][V] float4
        else if (i < 25) prefetch_l2(C.a32 + (i - 12) * V + x0, 16u * n);      // [13][V] float4
    } else if (std::is_same<P, P16>::value) {
        if (i < 4) prefetch_l2(U.u16a + i * V + x0, 16u * n);                   // [4][V] uint4
        else if (i < 8) prefetch_l2(U.u16b + (i - 4) * V + x0, 8u * n);        // [4][V] uint2
        else if (i < 14) prefetch_l2(C.a16 + (i - 8) * V + x0, 16u * n);       // [6][V] uint4
        else if (i < 15) prefetch_l2(C.a16b + x0, 8u * n);                     // [V] uint2
    }
}

// KIND 0: out = M in, 1: out = M^+ in, 2: out = H in.  MINB: minimum
// resident CTAs of kApplyMaxThreads threads per SM (caps registers).  The
// grid may be smaller than the nlogical logical blocks (persistent launch:
// each CTA walks the logical blocks with stride gridDim.x).  kFlagPdl: the launch is a programmatic
// dependent of the previous kernel (lexicographic site maps only): the CTA
// warms L2 with the links and clover of its first sites, which no kernel of
// a solve writes, before it waits for the previous kernel's output.
constexpr int kFlagPdl = 1;

template <class P, int KIND, int MINB>
__global__ void __launch_bounds__(kApplyMaxThreads, MINB)
    k_apply(Geom g, TileMap tm, int nlogical, GaugeStore U, CloverStore C, const void *in, const float *in_nrm,
            void *out, float *out_nrm, double kappa, int flags, const int *skip)
{
    if (flags & kFlagPdl) {
        const int x0 = blockIdx.x * blockDim.x;
        const int n = g.V - x0 < (int)blockDim.x ? g.V - x0 : (int)blockDim.x;
        if (n > 0) prefetch_block<P>(g, U, C, x0, n, threadIdx.x);
        griddep_wait();
    }
    griddep_launch_dependents();
    if (skip && *skip) return;
    for (int blk = blockIdx.x; blk < nlogical; blk += gridDim.x)
        apply_site<P, KIND>(g, tm, blk, U, C, in, in_nrm, out, out_nrm, kappa);
}

// The FP64 operator on four warps per 32 sites (hop_split64).  168 registers,
// three CTAs per SM: three warps for each FP64 unit (four CTAs of 128
// registers measured the same).
template <int KIND>
__global__ void __launch_bounds__(kSplit64 * kSplit64Sites, 3)
    k_apply_split64(Geom g, GaugeStore U, CloverStore C, const void *in, void *out, double kappa, const int *skip)
{
    griddep_wait();
    griddep_launch_dependents();
    if (skip && *skip) return;
    __shared__ Split64Mem sm;
    const int s = threadIdx.x & (kSplit64Sites - 1), w = threadIdx.x / kSplit64Sites;
    const int x = blockIdx.x * kSplit64Sites + s;
    const bool valid = x < g.V;
    if (valid) {
        int c[4];
        site_coords_fast(g, x, c);
        hop_split64<KIND == 1 ? +1 : -1, KIND == 2>(g, U, in, g.V, x, c, sm, w, s, [](int y) { return y; });
    }
    __syncthreads();
    if (!valid) return;
    cx<double> y[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        y[r] = sum_split64(sm, 3 * w + r, s);
        if (KIND != 2) y[r] = -kappa * y[r];
    }
    if (KIND != 2) {
        cx<double> v[6];
        const double2 *p = static_cast<const double2 *>(in) + (size_t)(w >> 1) * 6 * g.V + x;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 a = p[(size_t)k * g.V];
            v[k] = mkc(a.x, a.y);
        }
        clover_rows64(C, g.V, x, w, v, y);
    }
    double2 *o = static_cast<double2 *>(out) + (size_t)3 * w * g.V + x;
#pragma unroll
    for (int r = 0; r < 3; ++r) o[(size_t)r * g.V] = make_double2(y[r].re, y[r].im);
}

// k_apply_split64 as the operator of a solver step: the pass also forms the
// sums of alpha (or OMEGA: of omega) with `ss.with`.
template <int KIND, bool OMEGA>
__global__ void __launch_bounds__(kSplit64 * kSplit64Sites, 3)
    k_apply_split64_sum(Geom g, GaugeStore U, CloverStore C, const void *in, void *out, double kappa, StepSum ss)
{
    griddep_wait();
    griddep_launch_dependents();
    if (ss.sc->skip) return;
    __shared__ Split64Mem sm;
    const int s = threadIdx.x & (kSplit64Sites - 1), w = threadIdx.x / kSplit64Sites;
    const int x = blockIdx.x * kSplit64Sites + s;
    const bool valid = x < g.V;
    if (valid) {
        int c[4];
        site_coords_fast(g, x, c);
        hop_split64<KIND == 1 ? +1 : -1>(g, U, in, g.V, x, c, sm, w, s, [](int y) { return y; });
    }
    __syncthreads();
    double acc[step_sums<OMEGA, double>] = {};
    if (valid) {
        cx<double> v[6], y[3], a[3];
        const double2 *p = static_cast<const double2 *>(in) + (size_t)(w >> 1) * 6 * g.V + x;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 b = p[(size_t)k * g.V];
            v[k] = mkc(b.x, b.y);
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) y[r] = -kappa * sum_split64(sm, 3 * w + r, s);
        clover_rows64(C, g.V, x, w, v, y);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const size_t k = (size_t)(3 * w + r) * g.V + x;
            static_cast<double2 *>(out)[k] = make_double2(y[r].re, y[r].im);
            const double2 b = static_cast<const double2 *>(ss.with)[k];
            a[r] = mkc(b.x, b.y);
        }
        add_step_sums<OMEGA, 3>(y, a, acc);
    }
    reduce_step_sums<OMEGA, kSplit64, double>(acc, ss);
}

// The same with the hops in double-FP32 arithmetic (wc_dfsplit.cuh); HDF: hin
// holds split values of in.  The clover term stays in FP64: its 66
// instructions per warp run on the FP64 units while the other warps' hops
// fill the FP32 pipes, and the largest term of out keeps all its bits.
template <int KIND, bool HDF>
__global__ void __launch_bounds__(kSplit64 * kSplit64Sites, dfs::kCtas)
    k_apply_splitdf(Geom g, GaugeStore U, CloverStore C, const void *hin, const void *in, void *out, double kappa,
                    const int *skip)
{
    griddep_wait();
    griddep_launch_dependents();
    if (skip && *skip) return;
    __shared__ dfs::Mem sm;
    const int s = threadIdx.x & (kSplit64Sites - 1), w = threadIdx.x / kSplit64Sites;
    const int x = blockIdx.x * kSplit64Sites + s;
    const bool valid = x < g.V;
    if (valid) {
        int c[4];
        site_coords_fast(g, x, c);
        dfs::hops<KIND == 1 ? +1 : -1, HDF>(g, U, hin, g.V, x, c, sm, w, s, [](int y) { return y; });
    }
    __syncthreads();
    if (!valid) return;
    cx<double> y[3];
    if (KIND != 2) {
        cx<double> v[6];
        const double2 *p = static_cast<const double2 *>(in) + (size_t)(w >> 1) * 6 * g.V + x;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const double2 a = p[(size_t)k * g.V];
            v[k] = mkc(a.x, a.y);
        }
        clover_rows64<true>(C, g.V, x, w, v, y);
    }
    double2 *o = static_cast<double2 *>(out) + (size_t)3 * w * g.V + x;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const double2 h = dfs::to_double(dfs::sum(sm, 3 * w + r, s));
        o[(size_t)r * g.V] = KIND == 2 ? h : make_double2(fma(-kappa, h.x, y[r].re), fma(-kappa, h.y, y[r].im));
    }
}

// ---- launch shapes and their autotuner ---------------------------------

struct ApplyShape {
    int threads;
    int tile[4];     // {0,0,0,0}: lexicographic
    int capped;      // register cap: 0 none, 1: 64 per thread (4 CTAs of 256), 2: 85 (3 CTAs of 256)
    int persistent;  // 1: grid = resident CTAs, each walks logical blocks
    int pdl;         // 1: programmatic dependent launch (lexicographic only; not inside a capture)
};

constexpr ApplyShape kShapes[] = {
    {128, {0, 0, 0, 0}, 0, 0}, {128, {0, 0, 0, 0}, 1, 0}, {256, {0, 0, 0, 0}, 0, 0}, {256, {0, 0, 0, 0}, 1, 0},
    {128, {8, 4, 4, 1}, 0, 0}, {128, {8, 4, 4, 1}, 1, 0}, {128, {8, 4, 2, 2}, 0, 0}, {128, {4, 4, 4, 2}, 0, 0},
    {256, {8, 4, 4, 2}, 0, 0}, {256, {8, 4, 4, 2}, 1, 0}, {256, {8, 8, 4, 1}, 0, 0}, {128, {0, 0, 0, 0}, 2, 0},
    {256, {0, 0, 0, 0}, 2, 0}, {128, {8, 4, 4, 1}, 2, 0}, {256, {8, 4, 4, 2}, 2, 0}, {128, {8, 4, 2, 2}, 2, 0},
    {128, {0, 0, 0, 0}, 2, 1}, {256, {0, 0, 0, 0}, 2, 1}, {128, {0, 0, 0, 0}, 0, 1}, {256, {0, 0, 0, 0}, 0, 1},
    {128, {0, 0, 0, 0}, 2, 1, 1}, {256, {0, 0, 0, 0}, 2, 1, 1},
    // small lattices: CTAs of 32 or 64 sites spread a few thousand sites
    // over more SMs (the FP64 operator is bound by the FP64 pipe of the SMs
    // it runs on)
    {32, {0, 0, 0, 0}, 0, 0}, {64, {0, 0, 0, 0}, 0, 0},
};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);
// What the FP64 operator takes unless a caller pins one of the shapes above:
// it measured faster than the best of them on every lattice (4^4 13
// against 39 us, 8^4 14 / 39, 12^4 49 / 60, 16^3x32 245 / 266, 24^3x32
// 809 / 863, 17x19x21x23 299 / 331, 32^3x64 3811 / 4014), so nothing is timed
// for it.
constexpr int kShapeSplit64 = kNumShapes;
// In double-FP32 arithmetic up to this many sites; above, one of the shapes
// is timed and taken.  Each hop splits its spinor anew, which costs more than it
// gains on large lattices: 8^4 17 against 47 us, 16^3x32 190 / 209, 17x19x21x23
// 227 / 250, 20^3x32 367 / 376, 24^3x24 477 / 466, 24^3x32 632 / 596, 28^3x32 1007 /
// 905.  The line is one of size, not of times measured in a process: the two
// forms round differently, and a result must not depend on a timing (the
// shapes all give the same bits).  A solve splits its vector once
// (launch_apply_df).
constexpr int kSplitDfSites = 1 << 18;

// caps: bit c-1 set if register cap c is compiled for the operator (P::kCaps)
bool shape_fits(const Geom &g, const ApplyShape &s, int caps)
{
    if (s.capped && !((caps >> (s.capped - 1)) & 1)) return false;
    if (s.tile[0] == 0) return true;
    for (int m = 0; m < 4; ++m)
        if (g.L[m] % s.tile[m] != 0) return false;
    return s.tile[0] * s.tile[1] * s.tile[2] * s.tile[3] == s.threads;
}

// Resident CTAs per SM of one kernel instantiation, asked of the runtime at
// every launch of a persistent shape.
template <class K>
int resident_ctas(K kernel, int threads)
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 1;
    }
    return n;
}

template <class P>
cudaError_t launch_split64(wc_lattice lat, wc_field out, wc_field in, int kind, cudaStream_t stream,
                           const int *skip, bool pdl)
{
    const Geom &g = lat->g;
    const dim3 grid((g.V + kSplit64Sites - 1) / kSplit64Sites);
    if constexpr (std::is_same<P, PDF>::value) {
        const auto kern = kind == 0 ? k_apply_splitdf<0, false>
                                    : kind == 1 ? k_apply_splitdf<1, false> : k_apply_splitdf<2, false>;
        return launch_step(pdl && pdl_grid(grid.x), kern, grid, kSplit64 * kSplit64Sites, stream, g, lat->gauge,
                           lat->clover, in->data, in->data, out->data, lat->kappa, skip);
    } else {
        const auto kern = kind == 0 ? k_apply_split64<0> : kind == 1 ? k_apply_split64<1> : k_apply_split64<2>;
        return launch_step(pdl && pdl_grid(grid.x), kern, grid, kSplit64 * kSplit64Sites, stream, g, lat->gauge,
                           lat->clover, in->data, out->data, lat->kappa, skip);
    }
}

template <class P>
cudaError_t launch_shape(wc_lattice lat, wc_field out, wc_field in, int kind, int index, cudaStream_t stream,
                         const int *skip = nullptr, bool step_pdl = false)
{
    if (index == kShapeSplit64) return launch_split64<P>(lat, out, in, kind, stream, skip, step_pdl);
    const ApplyShape &sh = kShapes[index];
    const Geom &g = lat->g;
    TileMap tm{};
    int nlogical;
    if (sh.tile[0] == 0) {
        nlogical = (g.V + sh.threads - 1) / sh.threads;
    } else {
        for (int m = 0; m < 4; ++m) tm.tile[m] = sh.tile[m];
        for (int m = 0; m < 3; ++m) tm.ntile[m] = g.L[m] / sh.tile[m];
        nlogical = g.V / sh.threads;
    }
    int pdl = 0;
    if (sh.pdl && sh.tile[0] == 0) {
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        cudaStreamIsCapturing(stream, &cs);
        pdl = cs == cudaStreamCaptureStatusNone;
    }
#define WC_LAUNCH(K, MB)                                                                                      \
    do {                                                                                                      \
        auto kern = k_apply<P, K, MB>;                                                                        \
        int grid = nlogical;                                                                                  \
        if (sh.persistent) {                                                                                  \
            const int cap = resident_ctas(kern, sh.threads) * sm_count();                                   \
            grid = nlogical < cap ? nlogical : cap;                                                           \
        }                                                                                                     \
        if (pdl) {                                                                                            \
            cudaLaunchConfig_t cfg = {};                                                                      \
            cudaLaunchAttribute attr[1];                                                                      \
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;                                  \
            attr[0].val.programmaticStreamSerializationAllowed = 1;                                           \
            cfg.gridDim = dim3(grid);                                                                         \
            cfg.blockDim = dim3(sh.threads);                                                                  \
            cfg.stream = stream;                                                                              \
            cfg.attrs = attr;                                                                                 \
            cfg.numAttrs = 1;                                                                                 \
            return cudaLaunchKernelEx(&cfg, kern, g, tm, nlogical, lat->gauge, lat->clover, in->data,         \
                                      (const float *)in->nrm, out->data, out->nrm, lat->kappa, kFlagPdl, skip); \
        }                                                                                                     \
        kern<<<grid, sh.threads, 0, stream>>>(g, tm, nlogical, lat->gauge, lat->clover, in->data, in->nrm,    \
                                              out->data, out->nrm, lat->kappa, 0, skip);                      \
    } while (0)
    // minimum resident CTAs of 256 threads for caps 1 and 2 (1: not compiled)
    constexpr bool c1 = P::kCaps & 1, c2 = P::kCaps & 2;
    constexpr int MB1 = c1 ? P::kCap1MinBlocks : 1, MB2 = c2 ? 3 : 1;
    if (kind == 0) {
        if (c1 && sh.capped == 1) WC_LAUNCH(0, MB1);
        else if (c2 && sh.capped == 2) WC_LAUNCH(0, MB2);
        else WC_LAUNCH(0, 1);
    } else if (kind == 1) {
        if (c1 && sh.capped == 1) WC_LAUNCH(1, MB1);
        else if (c2 && sh.capped == 2) WC_LAUNCH(1, MB2);
        else WC_LAUNCH(1, 1);
    } else {
        if (c1 && sh.capped == 1) WC_LAUNCH(2, MB1);
        else if (c2 && sh.capped == 2) WC_LAUNCH(2, MB2);
        else WC_LAUNCH(2, 1);
    }
#undef WC_LAUNCH
    return cudaGetLastError();
}

std::mutex g_shape_mutex;
struct ShapeChoice {
    int index;
    bool pinned;   // by a caller (wc_apply_shape)
};
std::map<std::array<int, 6>, ShapeChoice> g_shape_choice;   // by (L, prec, kind)

std::array<int, 6> shape_key(const Geom &g, int pcode, int kind)
{
    return {g.L[0], g.L[1], g.L[2], g.L[3], pcode, kind};
}

// the double-FP32 operator has its own entries
constexpr int kPrecDf = 3;

// whether a caller has pinned a shape (g_shape_mutex held by nobody)
bool shape_pinned(const Geom &g, int pcode, int kind)
{
    std::lock_guard<std::mutex> lk(g_shape_mutex);
    const auto it = g_shape_choice.find(shape_key(g, pcode, kind));
    return it != g_shape_choice.end() && it->second.pinned;
}

// Time every fitting shape (three rounds of 16 launches after one warm-up,
// best round kept, candidates interleaved so that clock drift affects all
// alike) and keep the fastest.  Needs an uncaptured stream; out is
// overwritten by the real launch that follows.
template <class P>
int tune_shape(wc_lattice lat, wc_field out, wc_field in, int kind, cudaStream_t stream)
{
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return 0;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return 0;
    }
    // the candidates are timed on four input / output pairs in turn (the
    // caller's and three copies of its input), so that on lattices whose
    // fields outgrow L2 every launch streams its spinors from HBM as the
    // solvers' applies do; without memory for the copies, on the caller's
    // pair alone
    const size_t bytes = spinor_bytes(in->prec, lat->g.V);
    wc_field ins[4] = {in, nullptr, nullptr, nullptr}, outs[4] = {out, nullptr, nullptr, nullptr};
    int npair = 1;
    for (int k = 1; k < 4; ++k) {
        if (wc_field_create(lat, in->prec, &ins[k]) != WC_OK) break;
        if (wc_field_create(lat, in->prec, &outs[k]) != WC_OK) {
            wc_field_destroy(ins[k]);
            ins[k] = nullptr;
            break;
        }
        cudaMemcpyAsync(ins[k]->data, in->data, bytes, cudaMemcpyDeviceToDevice, stream);
        if (in->nrm) cudaMemcpyAsync(ins[k]->nrm, in->nrm, sizeof(float) * lat->g.V, cudaMemcpyDeviceToDevice, stream);
        npair = k + 1;
    }
    cudaGetLastError();
    float best_ms[kNumShapes];
    for (int i = 0; i < kNumShapes; ++i) best_ms[i] = 1e30f;
    for (int round = 0; round < 3; ++round) {
        for (int i = 0; i < kNumShapes; ++i) {
            if (!shape_fits(lat->g, kShapes[i], P::kCaps)) continue;
            if (launch_shape<P>(lat, out, in, kind, i, stream) != cudaSuccess) continue;
            cudaEventRecord(e0, stream);
            for (int r = 0; r < 16; ++r)
                launch_shape<P>(lat, outs[r % npair], ins[r % npair], kind, i, stream);
            cudaEventRecord(e1, stream);
            if (cudaEventSynchronize(e1) != cudaSuccess) continue;
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ms < best_ms[i]) best_ms[i] = ms;
        }
    }
    int best = 0;
    for (int i = 1; i < kNumShapes; ++i)
        if (best_ms[i] < best_ms[best]) best = i;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    for (int k = 1; k < npair; ++k) {
        wc_field_destroy(ins[k]);
        wc_field_destroy(outs[k]);
    }
    cudaGetLastError();
    return best;
}

template <class P>
cudaError_t launch_apply_p(wc_lattice lat, wc_field out, wc_field in, int kind, cudaStream_t stream,
                           const int *skip, bool pdl)
{
    constexpr bool df = std::is_same<P, PDF>::value;
    const std::array<int, 6> key = shape_key(lat->g, df ? kPrecDf : (int)in->prec, kind);
    int choice = -1;
    {
        std::lock_guard<std::mutex> lk(g_shape_mutex);
        auto it = g_shape_choice.find(key);
        if (it != g_shape_choice.end()) choice = it->second.index;
    }
    if (choice < 0) {
        bool keep = true;
        if (std::is_same<P, P64>::value || (df && lat->g.V <= kSplitDfSites)) {
            choice = kShapeSplit64;
        } else {
            cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
            cudaStreamIsCapturing(stream, &cs);
            keep = cs == cudaStreamCaptureStatusNone;
            choice = keep ? tune_shape<P>(lat, out, in, kind, stream) : 0;   // no timing inside a capture
        }
        if (keep) {
            std::lock_guard<std::mutex> lk(g_shape_mutex);
            choice = g_shape_choice.emplace(key, ShapeChoice{choice, false}).first->second.index;
        }
    }
    return launch_shape<P>(lat, out, in, kind, choice, stream, skip, pdl);
}

// ------------------------------------------------------------------------
// precision conversion / scaling: dst = scale * src
// ------------------------------------------------------------------------

template <class PS, class PD>
__global__ void k_copy(int V, const void *src, const float *src_nrm, void *dst, float *dst_nrm, double scale,
                       const double *dev_norm2, int invert)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= V) return;
    double sc = scale;
    if (dev_norm2) {
        const double n2 = *dev_norm2;
        const double n = sqrt(n2);
        sc *= invert ? (n > 0.0 ? 1.0 / n : 0.0) : n;
    }
    cx<typename PS::real> a[12];
    PS::load_spinor(src, src_nrm, V, x, a);
    cx<typename PD::real> b[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        // scale in the wider of the two precisions, then round once
        const double re = sc * (double)a[k].re, im = sc * (double)a[k].im;
        b[k] = mkc((typename PD::real)re, (typename PD::real)im);
    }
    PD::store_spinor(dst, dst_nrm, V, x, b);
}

template <class PS>
cudaError_t launch_copy_s(wc_lattice lat, wc_field dst, wc_field src, double scale, const double *dn, int inv,
                          cudaStream_t stream)
{
    const int V = lat->g.V;
    dim3 grid((V + 255) / 256), block(256);
    switch (dst->prec) {
    case WC_F64:
        k_copy<PS, P64><<<grid, block, 0, stream>>>(V, src->data, src->nrm, dst->data, dst->nrm, scale, dn, inv);
        break;
    case WC_F32:
        k_copy<PS, P32><<<grid, block, 0, stream>>>(V, src->data, src->nrm, dst->data, dst->nrm, scale, dn, inv);
        break;
    default:
        k_copy<PS, P16><<<grid, block, 0, stream>>>(V, src->data, src->nrm, dst->data, dst->nrm, scale, dn, inv);
    }
    return cudaGetLastError();
}

}  // namespace

// Query or pin the launch shape of (lat extent, prec, kind): force >= 0 pins
// shape #force (false if it does not fit), -2 forgets what was pinned or
// timed; out = {threads, tile[4], flags}, all -1 when no shape was chosen yet.
bool apply_shape(wc_lattice lat, wc_prec prec, int kind, int force, int out[6])
{
    // FP64 fields on a lattice in double-FP32 mode use that operator's entry
    const int pcode = (prec == WC_F64 && lat->fp64_arith == WC_ARITH_DF32) ? kPrecDf : (int)prec;
    const std::array<int, 6> key = shape_key(lat->g, pcode, kind);
    for (int i = 0; i < 6; ++i) out[i] = -1;
    std::lock_guard<std::mutex> lk(g_shape_mutex);
    if (force >= 0) {
        const int caps = prec != WC_F64 ? P32::kCaps : pcode == kPrecDf ? PDF::kCaps : P64::kCaps;
        if (force >= kNumShapes || !shape_fits(lat->g, kShapes[force], caps)) return false;
        g_shape_choice[key] = ShapeChoice{force, true};
    } else if (force == -2) {
        g_shape_choice.erase(key);
    }
    auto it = g_shape_choice.find(key);
    if (it == g_shape_choice.end()) return true;
    if (it->second.index == kShapeSplit64) {
        out[0] = kSplit64 * kSplit64Sites;
        for (int m = 0; m < 4; ++m) out[1 + m] = 0;
        out[5] = 64;
        return true;
    }
    const ApplyShape &s = kShapes[it->second.index];
    out[0] = s.threads;
    for (int m = 0; m < 4; ++m) out[1 + m] = s.tile[m];
    out[5] = s.capped + 4 * s.persistent + 16 * s.pdl;
    return true;
}

int apply_shape_count() { return kNumShapes; }

cudaError_t launch_apply(wc_lattice lat, wc_field out, wc_field in, int kind, cudaStream_t stream, const int *skip,
                         bool pdl)
{
    if (lat->schur_parent) return launch_schur(lat, out, in, kind == 1, stream, nullptr, skip, pdl);   // half lattice: M^
    switch (in->prec) {
    case WC_F64:
        return lat->fp64_arith == WC_ARITH_DF32 ? launch_apply_p<PDF>(lat, out, in, kind, stream, skip, pdl)
                                                : launch_apply_p<P64>(lat, out, in, kind, stream, skip, pdl);
    case WC_F32: return launch_apply_p<P32>(lat, out, in, kind, stream, skip, pdl);
    default: return launch_apply_p<P16>(lat, out, in, kind, stream, skip, pdl);
    }
}

cudaError_t launch_apply64_sum(wc_lattice lat, wc_field out, wc_field in, int kind, cudaStream_t stream,
                               const StepSum &ss, bool omega, bool pdl)
{
    const Geom &g = lat->g;
    if (shape_pinned(g, (int)WC_F64, kind)) return cudaErrorNotSupported;   // a pinned launch shape stays in use
    const dim3 grid((g.V + kSplit64Sites - 1) / kSplit64Sites);
    const auto kern = kind == 0 ? (omega ? k_apply_split64_sum<0, true> : k_apply_split64_sum<0, false>)
                                : (omega ? k_apply_split64_sum<1, true> : k_apply_split64_sum<1, false>);
    return launch_step(pdl && pdl_grid(grid.x), kern, grid, kSplit64 * kSplit64Sites, stream, g, lat->gauge, lat->clover,
                       in->data, out->data, lat->kappa, ss);
}

cudaError_t launch_apply_df(wc_lattice lat, wc_field out, wc_field in, wc_field split, int kind, cudaStream_t stream,
                            const int *skip, bool pdl)
{
    const Geom &g = lat->g;
    if (shape_pinned(g, kPrecDf, kind)) return launch_apply(lat, out, in, kind, stream, skip, pdl);   // stays in use
    cudaError_t e = launch_to_df(12LL * g.V, in, split, stream, skip, pdl);
    if (e != cudaSuccess) return e;
    const dim3 grid((g.V + kSplit64Sites - 1) / kSplit64Sites);
    const auto kern = kind == 0 ? k_apply_splitdf<0, true> : kind == 1 ? k_apply_splitdf<1, true> : k_apply_splitdf<2, true>;
    return launch_step(pdl && pdl_grid(grid.x), kern, grid, kSplit64 * kSplit64Sites, stream, g, lat->gauge, lat->clover,
                       split->data, in->data, out->data, lat->kappa, skip);
}

cudaError_t launch_copy(wc_lattice lat, wc_field dst, wc_field src, double scale, const double *dev_scale,
                        int invert_scale, cudaStream_t stream)
{
    switch (src->prec) {
    case WC_F64: return launch_copy_s<P64>(lat, dst, src, scale, dev_scale, invert_scale, stream);
    case WC_F32: return launch_copy_s<P32>(lat, dst, src, scale, dev_scale, invert_scale, stream);
    default: return launch_copy_s<P16>(lat, dst, src, scale, dev_scale, invert_scale, stream);
    }
}

}  // namespace wc
