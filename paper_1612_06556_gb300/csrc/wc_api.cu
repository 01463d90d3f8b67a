// C ABI entry points: lattices, fields, gauge/clover loading, applies.
//
// Field transfers convert between the caller's canonical layout (complex128
// or complex64, site-major) and the plane-major device layouts in one kernel
// per call.  The synchronous calls stage host data in a lattice-owned
// buffer and return when the caller's memory may be reused; the
// asynchronous calls take device or page-locked host memory, copy host data
// in on a second stream of the lattice (so that the next input crosses the
// host link while the current step computes and copies its result out) and
// leave the caller to wc_sync.
#include <math.h>
#include <stdio.h>

#include <mutex>
#include <new>
#include <type_traits>

#include <vector>

#include "wc_internal.cuh"

namespace wc {

namespace {
thread_local std::string g_global_error;
}

wc_status set_error(wc_lattice lat, wc_status st, const std::string &msg)
{
    if (st == WC_OK) return st;
    if (lat)
        lat->err = msg;
    else
        g_global_error = msg;
    return st;
}

wc_status check_cuda(wc_lattice lat, cudaError_t e, const char *what)
{
    if (e == cudaSuccess) return WC_OK;
    cudaGetLastError();   // reported here: not again by the next launch check
    return set_error(lat, WC_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

wc_status check_launch(wc_lattice lat, const char *what) { return check_cuda(lat, cudaGetLastError(), what); }

int sm_count()
{
    static int n = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    });
    return n;
}

namespace {

bool is_device_pointer(const void *p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// ------------------------------------------------------------------------
// canonical <-> internal
// ------------------------------------------------------------------------

// A site's 12 components lie together in the canonical layout (96 or 192
// bytes) and in 12 planes in the device layouts.  On export a CTA turns
// kXferSites sites round in shared memory, so that both sides move 16
// contiguous bytes per thread and a warp whole 128-byte lines; one thread per
// site writing its row left the memory system with 12 partly used sectors per
// request (24^3x32 FP32 -> complex64 27 us = 3.1 TB/s, 12.4 us now;
// binary16 -> complex64 at 32^3x64 110 us, 42 now).  A row in shared memory
// is one 16-byte unit longer than in the canonical layout: the eight lanes
// of a 16-byte access phase then fall on different banks.
//
// On import the rows are read, and the sectors that one load of a warp leaves
// partly used are in L1 for the next: a thread per site is the faster form but
// where the rows are short beside what is written of them (complex64 ->
// binary16), and on lattices of less than a CTA of kXferSites per SM, where its
// loads wait for one another.  Thread per site / turned round, us: complex128 ->
// FP32 at 8^4 3.2 / 2.8, 16^4 4.9 / 5.7, 24^3x32 23 / 27, 32^3x64 91 / 109; ->
// FP64 3.1 / 2.3, 4.9 / 4.5, 28 / 31, 120 / 136; complex64 -> FP32 2.1 / 2.0,
// 3.0 / 3.2, 15.0 / 16.2, 61 / 68; -> binary16 2.1 / 2.2, 2.8 / 2.8, 12.5 / 12.0,
// 48.9 / 46.6.
// T: double2 (canonical complex128) or float2 (canonical complex64)
constexpr int kXferSites = 128;

template <class T>
struct XferRow {
    static constexpr int kUnits = 12 * sizeof(T) / 16;   // 16-byte units of a canonical row
    static constexpr int kPitch = kUnits + 1;
    float4 sm[kXferSites * kPitch];
    __device__ __forceinline__ T *row(int i) { return reinterpret_cast<T *>(sm + i * kPitch); }
};

// the canonical rows of sites [x0, x0 + n) to or from shared memory, in
// 16-byte units, or in units of T where the caller's complex64 data is not
// aligned to 16 bytes
template <class T, bool OUT, class C>
__device__ __forceinline__ void xfer_rows(XferRow<T> &b, C *data, int x0, int n)
{
    using X = XferRow<T>;
    if ((reinterpret_cast<uintptr_t>(data) & 15) == 0) {
        using V4 = std::conditional_t<OUT, float4, const float4>;
        V4 *g = reinterpret_cast<V4 *>(data) + (size_t)x0 * X::kUnits;
        for (int q = threadIdx.x; q < n * X::kUnits; q += kXferSites) {
            const int at = q / X::kUnits * X::kPitch + q % X::kUnits;
            if constexpr (OUT) g[q] = b.sm[at];
            else b.sm[at] = g[q];
        }
    } else {
        C *g = data + (size_t)x0 * 12;
        for (int q = threadIdx.x; q < n * 12; q += kXferSites) {
            if constexpr (OUT) g[q] = b.row(q / 12)[q % 12];
            else b.row(q / 12)[q % 12] = g[q];
        }
    }
}

template <class P, class T>
__global__ void __launch_bounds__(kXferSites) k_import(int V, const T *src, void *dst, float *nrm)
{
    __shared__ XferRow<T> b;
    const int x0 = blockIdx.x * kXferSites, n = min(kXferSites, V - x0);
    xfer_rows<T, false>(b, src, x0, n);
    __syncthreads();
    if ((int)threadIdx.x >= n) return;
    using R = typename P::real;
    cx<R> s[12];
    const T *row = b.row(threadIdx.x);
#pragma unroll
    for (int k = 0; k < 12; ++k) s[k] = mkc((R)row[k].x, (R)row[k].y);
    P::store_spinor(dst, nrm, V, x0 + threadIdx.x, s);
}

// the same, a thread per site
template <class P, class T>
__global__ void __launch_bounds__(256) k_import_rows(int V, const T *src, void *dst, float *nrm)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= V) return;
    using R = typename P::real;
    cx<R> s[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const T v = src[(size_t)x * 12 + k];
        s[k] = mkc((R)v.x, (R)v.y);
    }
    P::store_spinor(dst, nrm, V, x, s);
}

template <class P, class T>
__global__ void __launch_bounds__(kXferSites) k_export(int V, const void *src, const float *nrm, T *dst)
{
    __shared__ XferRow<T> b;
    const int x0 = blockIdx.x * kXferSites, n = min(kXferSites, V - x0);
    if ((int)threadIdx.x < n) {
        using E = decltype(T::x);
        cx<typename P::real> s[12];
        P::load_spinor(src, nrm, V, x0 + threadIdx.x, s);
        T *row = b.row(threadIdx.x);
#pragma unroll
        for (int k = 0; k < 12; ++k) row[k] = T{(E)s[k].re, (E)s[k].im};
    }
    __syncthreads();
    xfer_rows<T, true>(b, dst, x0, n);
}

// queue the conversion of canonical data (device) into f, or of f into it
template <class P, class T>
void launch_import_p(wc_field f, const T *src, cudaStream_t stream)
{
    const int V = f->lat->g.V;
    const bool turn = (std::is_same<P, P16>::value && std::is_same<T, float2>::value) || V < kXferSites * sm_count();
    if (turn) k_import<P, T><<<(V + kXferSites - 1) / kXferSites, kXferSites, 0, stream>>>(V, src, f->data, f->nrm);
    else k_import_rows<P, T><<<(V + 255) / 256, 256, 0, stream>>>(V, src, f->data, f->nrm);
}

template <class T>
void launch_import(wc_field f, const T *src, cudaStream_t stream)
{
    if (f->prec == WC_F64) launch_import_p<P64>(f, src, stream);
    else if (f->prec == WC_F32) launch_import_p<P32>(f, src, stream);
    else launch_import_p<P16>(f, src, stream);
}

template <class T>
void launch_export(wc_field f, T *dst, cudaStream_t stream)
{
    const int V = f->lat->g.V, grid = (V + kXferSites - 1) / kXferSites;
    if (f->prec == WC_F64) k_export<P64, T><<<grid, kXferSites, 0, stream>>>(V, f->data, f->nrm, dst);
    else if (f->prec == WC_F32) k_export<P32, T><<<grid, kXferSites, 0, stream>>>(V, f->data, f->nrm, dst);
    else k_export<P16, T><<<grid, kXferSites, 0, stream>>>(V, f->data, f->nrm, dst);
}

// canonical U[V][4][3][3] -> two-row stores in three precisions
__global__ void k_pack_gauge(int V, const double2 *U, GaugeStore g)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 4 * V) return;
    const int x = i % V, mu = i / V;
    const double2 *u = U + ((size_t)x * 4 + mu) * 9;  // rows 0 and 1 = entries 0..5
    double2 a[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k] = u[k];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        g.u64[((size_t)mu * 9 + k) * V + x] = a[k];
        g.udf[((size_t)mu * 9 + k) * V + x] = df_pack(a[k]);
    }
    cx<double> r01[6], r2[3];
#pragma unroll
    for (int k = 0; k < 6; ++k) r01[k] = mkc(a[k].x, a[k].y);
    reconstruct_row2(r01, r2);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double2 v = make_double2(r2[k].re, r2[k].im);
        g.u64[((size_t)mu * 9 + 6 + k) * V + x] = v;
        g.udf[((size_t)mu * 9 + 6 + k) * V + x] = df_pack(v);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
        g.u32[((size_t)mu * 3 + j) * V + x] =
            make_float4((float)a[2 * j].x, (float)a[2 * j].y, (float)a[2 * j + 1].x, (float)a[2 * j + 1].y);
    uint4 h;
    h.x = c2h((float)a[0].x, (float)a[0].y);
    h.y = c2h((float)a[1].x, (float)a[1].y);
    h.z = c2h((float)a[2].x, (float)a[2].y);
    h.w = c2h((float)a[3].x, (float)a[3].y);
    uint2 h2;
    h2.x = c2h((float)a[4].x, (float)a[4].y);
    h2.y = c2h((float)a[5].x, (float)a[5].y);
    g.u16a[(size_t)mu * V + x] = h;
    g.u16b[(size_t)mu * V + x] = h2;
}

template <class T>
cudaError_t dalloc(T **p, size_t bytes)
{
    return cudaMalloc(reinterpret_cast<void **>(p), bytes);
}

void free_gauge(GaugeStore &g)
{
    cudaFree(g.u64);
    cudaFree(g.udf);
    cudaFree(g.u32);
    cudaFree(g.u16a);
    cudaFree(g.u16b);
    g = GaugeStore{};
}

wc_status need_staging(wc_lattice lat, size_t bytes)
{
    if (lat->staging_bytes >= bytes) return WC_OK;
    cudaFree(lat->staging);
    lat->staging = nullptr;
    lat->staging_bytes = 0;
    wc_status st = check_cuda(lat, dalloc(&lat->staging, bytes), "cudaMalloc(staging)");
    if (st == WC_OK) lat->staging_bytes = bytes;
    return st;
}

wc_status check_field(wc_lattice lat, wc_field f, const char *name)
{
    if (!f) return set_error(lat, WC_ERR_ARG, std::string(name) + " is NULL");
    if (f->lat != lat) return set_error(lat, WC_ERR_ARG, std::string(name) + " belongs to another lattice");
    return WC_OK;
}

}  // namespace

void free_clover(CloverStore &c)
{
    cudaFree(c.c64);
    cudaFree(c.cdf);
    cudaFree(c.c32);
    cudaFree(c.c16);
    cudaFree(c.a32);
    cudaFree(c.a16);
    cudaFree(c.a16b);
    c = CloverStore{};
}

// the FP32 and FP16 parts of a store of A
wc_status alloc_clover_a(wc_lattice lat, CloverStore &c)
{
    const size_t V = lat->g.V;
    wc_status st = check_cuda(lat, dalloc(&c.a32, sizeof(float4) * 13 * V), "cudaMalloc(clover)");
    if (st == WC_OK) st = check_cuda(lat, dalloc(&c.a16, sizeof(uint4) * 6 * V), "cudaMalloc(clover)");
    if (st == WC_OK) st = check_cuda(lat, dalloc(&c.a16b, sizeof(uint2) * V), "cudaMalloc(clover)");
    return st;
}

// readers of the per-translation-unit violation counters (checked build)
std::vector<cudaError_t (*)(unsigned *)> &check_readers()
{
    static std::vector<cudaError_t (*)(unsigned *)> r;
    return r;
}

void register_check_counter(cudaError_t (*read)(unsigned *)) { check_readers().push_back(read); }

wc_status require_operator(wc_lattice lat, bool need_clover)
{
    if (lat->split_mask)
        return set_error(lat, WC_ERR_ARG,
                         "sub-domain lattice: its operator needs the neighbours' face data (wc_halo_pack, "
                         "wc_apply_interior, wc_apply_surface)");
    if (!lat->gauge_loaded) return set_error(lat, WC_ERR_STATE, "gauge field not loaded");
    if (need_clover && !lat->clover_loaded) return set_error(lat, WC_ERR_STATE, "clover term not loaded");
    return WC_OK;
}

wc_status state_init(wc_lattice lat, SolverState &s)
{
    // four blocks of 256 per SM: the last block adds one partial per block
    // and sum, so more blocks lengthen its tail and fewer leave the loads of
    // the vectors uncovered (lo_alpha at 16^3x32 10.0 / 7.7 / 8.1 / 8.2 us,
    // lo_xr 12.1 / 11.5 / 12.9 / 13.2 us with 8 / 4 / 3 / 2 per SM)
    const int max_blocks = 4 * sm_count();
    s.red.max_blocks = max_blocks;
    wc_status st = check_cuda(lat, dalloc(&s.red.partials, sizeof(double) * 8 * max_blocks), "cudaMalloc");
    if (st == WC_OK) st = check_cuda(lat, dalloc(&s.red.ticket, sizeof(unsigned)), "cudaMalloc");
    if (st == WC_OK) st = check_cuda(lat, dalloc(&s.red.result, sizeof(double) * 8), "cudaMalloc");
    if (st == WC_OK)
        st = check_cuda(lat, cudaMallocHost(reinterpret_cast<void **>(&s.red.host_result), sizeof(double) * 8),
                        "cudaMallocHost");
    if (st == WC_OK) st = check_cuda(lat, dalloc(&s.scal, sizeof(SolverScalars)), "cudaMalloc");
    if (st == WC_OK)
        st = check_cuda(lat, cudaMallocHost(reinterpret_cast<void **>(&s.scal_host), sizeof(SolverScalars)),
                        "cudaMallocHost");
    if (st == WC_OK)
        st = check_cuda(lat, cudaMallocHost(reinterpret_cast<void **>(&s.report), sizeof(StepReport) * kReportSlots),
                        "cudaMallocHost");
    for (int i = 0; i < kReportSlots && st == WC_OK; ++i) s.report[i].seq = 0;
    if (st == WC_OK) st = check_cuda(lat, cudaMemset(s.red.ticket, 0, sizeof(unsigned)), "cudaMemset");
    if (st == WC_OK) st = check_cuda(lat, cudaMemset(s.scal, 0, sizeof(SolverScalars)), "cudaMemset");
    if (st != WC_OK) state_free(s);
    return st;
}

void state_free(SolverState &s)
{
    if (s.inner) {
        state_free(*s.inner);
        delete s.inner;
        s.inner = nullptr;
    }
    for (auto &w : s.work) {
        wc_field_destroy(w);
        w = nullptr;
    }
    cudaFree(s.red.partials);
    cudaFree(s.red.ticket);
    cudaFree(s.red.result);
    cudaFreeHost(s.red.host_result);
    cudaFree(s.scal);
    cudaFreeHost(s.scal_host);
    cudaFreeHost(s.report);
    s = SolverState{};
}

wc_field state_work(wc_lattice lat, SolverState &s, int slot, wc_prec prec, wc_status *st)
{
    if (!s.work[slot]) {
        *st = wc_field_create(lat, prec, &s.work[slot]);
        if (*st != WC_OK) return nullptr;
    }
    *st = WC_OK;
    return s.work[slot];
}

namespace {
}  // namespace
}  // namespace wc

using namespace wc;

namespace {

template <class T>
wc_status field_import(wc_field f, const T *data)
{
    if (!f) return set_error(nullptr, WC_ERR_ARG, "field is NULL");
    wc_lattice lat = f->lat;
    if (!data) return set_error(lat, WC_ERR_ARG, "data is NULL");
    const int V = lat->g.V;
    const size_t bytes = sizeof(T) * 12 * (size_t)V;
    const T *src = data;
    wc_status st = WC_OK;
    const bool host = !is_device_pointer(data);
    if (host) {
        st = need_staging(lat, bytes);
        if (st != WC_OK) return st;
        st = check_cuda(lat, cudaMemcpyAsync(lat->staging, data, bytes, cudaMemcpyHostToDevice, lat->stream),
                        "cudaMemcpyAsync(import)");
        if (st != WC_OK) return st;
        src = reinterpret_cast<const T *>(lat->staging);
    }
    launch_import(f, src, lat->stream);
    st = check_launch(lat, "import");
    if (st == WC_OK && host) st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync(import)");
    return st;
}

template <class T>
wc_status field_export(wc_field f, T *data)
{
    if (!f) return set_error(nullptr, WC_ERR_ARG, "field is NULL");
    wc_lattice lat = f->lat;
    if (!data) return set_error(lat, WC_ERR_ARG, "data is NULL");
    const int V = lat->g.V;
    const size_t bytes = sizeof(T) * 12 * (size_t)V;
    const bool host = !is_device_pointer(data);
    T *dst = data;
    wc_status st = WC_OK;
    if (host) {
        st = need_staging(lat, bytes);
        if (st != WC_OK) return st;
        dst = reinterpret_cast<T *>(lat->staging);
    }
    launch_export(f, dst, lat->stream);
    st = check_launch(lat, "export");
    if (st == WC_OK && host) {
        st = check_cuda(lat, cudaMemcpyAsync(data, lat->staging, bytes, cudaMemcpyDeviceToHost, lat->stream),
                        "cudaMemcpyAsync(export)");
        if (st == WC_OK) st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync(export)");
    }
    return st;
}

bool is_pinned_host(const void *p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeHost;
}

// copy stream, events and the two staging buffers of the asynchronous path.
// Everything is created into locals and handed to the lattice only when
// every step succeeded (the copy stream is set last: it marks the set-up as
// done); after a failure the partial resources are released and the next
// asynchronous call tries again.
wc_status async_setup(wc_lattice lat)
{
    if (lat->copy_stream) return WC_OK;
    const size_t bytes = sizeof(double2) * 12 * (size_t)lat->g.V;
    cudaStream_t cs = nullptr, co = nullptr;
    cudaEvent_t ev[6] = {};   // in ready, in free, out ready 0/1, out free 0/1
    double2 *in = nullptr, *out[2] = {nullptr, nullptr};
    wc_status st = check_cuda(lat, cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking), "cudaStreamCreate(copy)");
    if (st == WC_OK)
        st = check_cuda(lat, cudaStreamCreateWithFlags(&co, cudaStreamNonBlocking), "cudaStreamCreate(copy out)");
    for (int k = 0; k < 6 && st == WC_OK; ++k)
        st = check_cuda(lat, cudaEventCreateWithFlags(&ev[k], cudaEventDisableTiming), "cudaEventCreate");
    if (st == WC_OK) st = check_cuda(lat, dalloc(&in, bytes), "cudaMalloc(staging)");
    for (int b = 0; b < 2 && st == WC_OK; ++b) st = check_cuda(lat, dalloc(&out[b], bytes), "cudaMalloc(staging)");
    // nothing to wait for before the first copies
    if (st == WC_OK) st = check_cuda(lat, cudaEventRecord(ev[1], lat->stream), "cudaEventRecord");
    for (int b = 0; b < 2 && st == WC_OK; ++b)
        st = check_cuda(lat, cudaEventRecord(ev[4 + b], co), "cudaEventRecord");
    if (st != WC_OK) {
        if (cs) cudaStreamDestroy(cs);
        if (co) cudaStreamDestroy(co);
        for (auto e : ev)
            if (e) cudaEventDestroy(e);
        cudaFree(in);
        cudaFree(out[0]);
        cudaFree(out[1]);
        return st;
    }
    lat->ev_in_ready = ev[0];
    lat->ev_in_free = ev[1];
    for (int b = 0; b < 2; ++b) {
        lat->ev_out_ready[b] = ev[2 + b];
        lat->ev_out_free[b] = ev[4 + b];
        lat->astage_out[b] = out[b];
    }
    lat->astage_in = in;
    lat->out_buf = 0;
    lat->copy_out_stream = co;
    lat->copy_stream = cs;
    return WC_OK;
}

template <class T>
wc_status field_import_async(wc_field f, const T *data)
{
    if (!f) return set_error(nullptr, WC_ERR_ARG, "field is NULL");
    wc_lattice lat = f->lat;
    if (!data) return set_error(lat, WC_ERR_ARG, "data is NULL");
    const bool dev = is_device_pointer(data);
    if (!dev && !is_pinned_host(data))
        return set_error(lat, WC_ERR_ARG, "asynchronous import needs device or page-locked host memory");
    const int V = lat->g.V;
    const T *src = data;
    wc_status st = WC_OK;
    if (!dev) {
        st = async_setup(lat);
        if (st != WC_OK) return st;
        // the previous import kernel must have read the staging buffer
        st = check_cuda(lat, cudaStreamWaitEvent(lat->copy_stream, lat->ev_in_free, 0), "wait");
        if (st == WC_OK)
            st = check_cuda(lat, cudaMemcpyAsync(lat->astage_in, data, sizeof(T) * 12 * (size_t)V,
                                                 cudaMemcpyHostToDevice, lat->copy_stream), "cudaMemcpyAsync(import)");
        if (st == WC_OK) st = check_cuda(lat, cudaEventRecord(lat->ev_in_ready, lat->copy_stream), "record");
        if (st == WC_OK) st = check_cuda(lat, cudaStreamWaitEvent(lat->stream, lat->ev_in_ready, 0), "wait");
        if (st != WC_OK) return st;
        src = reinterpret_cast<const T *>(lat->astage_in);
    }
    launch_import(f, src, lat->stream);
    st = check_launch(lat, "import");
    if (st == WC_OK && !dev) st = check_cuda(lat, cudaEventRecord(lat->ev_in_free, lat->stream), "record");
    return st;
}

template <class T>
wc_status field_export_async(wc_field f, T *data)
{
    if (!f) return set_error(nullptr, WC_ERR_ARG, "field is NULL");
    wc_lattice lat = f->lat;
    if (!data) return set_error(lat, WC_ERR_ARG, "data is NULL");
    const bool dev = is_device_pointer(data);
    if (!dev && !is_pinned_host(data))
        return set_error(lat, WC_ERR_ARG, "asynchronous export needs device or page-locked host memory");
    const int V = lat->g.V;
    T *dst = data;
    wc_status st = WC_OK;
    const int b = lat->out_buf;
    if (!dev) {
        st = async_setup(lat);
        if (st != WC_OK) return st;
        // the copy out that last used buffer b must be done
        st = check_cuda(lat, cudaStreamWaitEvent(lat->stream, lat->ev_out_free[b], 0), "wait");
        if (st != WC_OK) return st;
        dst = reinterpret_cast<T *>(lat->astage_out[b]);
    }
    launch_export(f, dst, lat->stream);
    st = check_launch(lat, "export");
    if (st == WC_OK && !dev) {
        st = check_cuda(lat, cudaEventRecord(lat->ev_out_ready[b], lat->stream), "record");
        if (st == WC_OK)
            st = check_cuda(lat, cudaStreamWaitEvent(lat->copy_out_stream, lat->ev_out_ready[b], 0), "wait");
        if (st == WC_OK)
            st = check_cuda(lat, cudaMemcpyAsync(data, lat->astage_out[b], sizeof(T) * 12 * (size_t)V,
                                                 cudaMemcpyDeviceToHost, lat->copy_out_stream),
                            "cudaMemcpyAsync(export)");
        if (st == WC_OK) st = check_cuda(lat, cudaEventRecord(lat->ev_out_free[b], lat->copy_out_stream), "record");
        if (st == WC_OK) lat->out_buf = b ^ 1;
    }
    return st;
}

}  // namespace

extern "C" {

wc_status wc_create_lattice(const int dims[4], int t_bc, void *cuda_stream, wc_lattice *out)
{
    if (!dims || !out) return set_error(nullptr, WC_ERR_ARG, "dims and out must not be NULL");
    *out = nullptr;
    long long V = 1;
    for (int m = 0; m < 4; ++m) {
        if (dims[m] < 2) return set_error(nullptr, WC_ERR_ARG, "every lattice extent must be >= 2");
        V *= dims[m];
    }
    if (V > (1LL << 30)) return set_error(nullptr, WC_ERR_ARG, "lattice volume above 2^30 sites");
    if (t_bc != 1 && t_bc != -1) return set_error(nullptr, WC_ERR_ARG, "t_bc must be +1 or -1");
    wc_lattice lat = new (std::nothrow) wc_lattice_s();
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "out of host memory");
    for (int m = 0; m < 4; ++m) lat->g.L[m] = dims[m];
    lat->g.stride[0] = 1;
    lat->g.stride[1] = dims[0];
    lat->g.stride[2] = dims[0] * dims[1];
    lat->g.stride[3] = dims[0] * dims[1] * dims[2];
    lat->g.V = (int)V;
    lat->g.tbc = t_bc;
    geom_set_div(lat->g);
    lat->stream = static_cast<cudaStream_t>(cuda_stream);
    wc_status st = state_init(lat, lat->st);
    if (st != WC_OK) {
        set_error(nullptr, st, lat->err);
        wc_destroy_lattice(lat);
        return st;
    }
    *out = lat;
    return WC_OK;
}

wc_status wc_destroy_lattice(wc_lattice lat)
{
    if (!lat) return WC_OK;
    cudaStreamSynchronize(lat->stream);
    free_batch_pool(lat);
    free_half(lat);
    state_free(lat->st);
    free_gauge(lat->gauge);
    free_clover(lat->clover);
    free_clover(lat->cinv);
    free_clover(lat->ceo);
    cudaFree(lat->staging);
    cudaFree(lat->eom_ws);
    for (cudaStream_t cs : {lat->copy_stream, lat->copy_out_stream})
        if (cs) {
            cudaStreamSynchronize(cs);
            cudaStreamDestroy(cs);
        }
    for (cudaEvent_t e : {lat->ev_in_ready, lat->ev_in_free, lat->ev_out_ready[0], lat->ev_out_ready[1],
                          lat->ev_out_free[0], lat->ev_out_free[1]})
        if (e) cudaEventDestroy(e);
    cudaFree(lat->astage_in);
    cudaFree(lat->astage_out[0]);
    cudaFree(lat->astage_out[1]);
    wc_destroy_lattice(lat->ext);
    delete lat;
    return WC_OK;
}

wc_status wc_set_stream(wc_lattice lat, void *cuda_stream)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    lat->stream = static_cast<cudaStream_t>(cuda_stream);
    if (lat->ext) lat->ext->stream = lat->stream;
    return WC_OK;
}

wc_status wc_set_fp64_arith(wc_lattice lat, int arith)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (arith != WC_ARITH_F64 && arith != WC_ARITH_DF32) return set_error(lat, WC_ERR_ARG, "unknown FP64 arithmetic");
    lat->fp64_arith = arith;
    return WC_OK;
}

wc_status wc_load_gauge(wc_lattice lat, const double *data)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (!data) return set_error(lat, WC_ERR_ARG, "gauge data is NULL");
    const int V = lat->g.V;
    GaugeStore &g = lat->gauge;
    wc_status st = WC_OK;
    if (!g.u64) {
        st = check_cuda(lat, dalloc(&g.u64, sizeof(double2) * 36 * (size_t)V), "cudaMalloc(gauge)");
        if (st == WC_OK) st = check_cuda(lat, dalloc(&g.udf, sizeof(float4) * 36 * (size_t)V), "cudaMalloc(gauge)");
        if (st == WC_OK) st = check_cuda(lat, dalloc(&g.u32, sizeof(float4) * 12 * (size_t)V), "cudaMalloc(gauge)");
        if (st == WC_OK) st = check_cuda(lat, dalloc(&g.u16a, sizeof(uint4) * 4 * (size_t)V), "cudaMalloc(gauge)");
        if (st == WC_OK) st = check_cuda(lat, dalloc(&g.u16b, sizeof(uint2) * 4 * (size_t)V), "cudaMalloc(gauge)");
        if (st != WC_OK) {
            free_gauge(g);
            return st;
        }
    }
    if (lat->split_mask) {
        // a sub-domain: data is the gauge field extended by one site across
        // every cut face; it is loaded on the extended lattice (where the
        // clover term will be built) and its interior copied here
        lat->ext->stream = lat->stream;
        st = wc_load_gauge(lat->ext, data);
        if (st != WC_OK) return set_error(lat, st, "extended gauge field: " + lat->ext->err);
        st = check_cuda(lat, extract_gauge(lat, lat->stream), "extract gauge");
        lat->gauge_loaded = (st == WC_OK);
        lat->clover_loaded = false;
        lat->cinv_loaded = false;
        return st;
    }
    const size_t bytes = sizeof(double2) * 36 * (size_t)V;
    const double2 *src = reinterpret_cast<const double2 *>(data);
    if (!is_device_pointer(data)) {
        st = need_staging(lat, bytes);
        if (st != WC_OK) return st;
        st = check_cuda(lat, cudaMemcpyAsync(lat->staging, data, bytes, cudaMemcpyHostToDevice, lat->stream),
                        "cudaMemcpyAsync(gauge)");
        if (st != WC_OK) return st;
        src = lat->staging;
    }
    k_pack_gauge<<<(4 * V + 255) / 256, 256, 0, lat->stream>>>(V, src, g);
    st = check_launch(lat, "pack_gauge");
    if (st != WC_OK) return st;
    // the host buffer must stay valid until the copy ran
    if (src == lat->staging) st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync(gauge)");
    lat->gauge_loaded = (st == WC_OK);
    lat->clover_loaded = false;
    lat->cinv_loaded = false;
    return st;
}

wc_status wc_load_clover(wc_lattice lat, double csw, double kappa)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (!lat->gauge_loaded) return set_error(lat, WC_ERR_STATE, "wc_load_clover before wc_load_gauge");
    if (!isfinite(csw) || !isfinite(kappa)) return set_error(lat, WC_ERR_ARG, "csw and kappa must be finite");
    const int V = lat->g.V;
    CloverStore &c = lat->clover;
    wc_status st = WC_OK;
    if (!c.c64) {
        st = check_cuda(lat, dalloc(&c.c64, sizeof(double2) * 36 * (size_t)V), "cudaMalloc(clover)");
        if (st == WC_OK) st = check_cuda(lat, dalloc(&c.cdf, sizeof(float4) * 36 * (size_t)V), "cudaMalloc(clover)");
        if (st == WC_OK) st = alloc_clover_a(lat, c);
        if (st != WC_OK) {
            free_clover(c);
            return st;
        }
    }
    if (lat->split_mask) {
        // a sub-domain: built on the extended lattice, whose halo sites hold
        // the neighbours' links the face sites' clover leaves reach
        lat->ext->stream = lat->stream;
        st = wc_load_clover(lat->ext, csw, kappa);
        if (st != WC_OK) return set_error(lat, st, "extended lattice clover: " + lat->ext->err);
        st = check_cuda(lat, extract_clover(lat, lat->stream), "extract clover");
    } else {
        st = check_cuda(lat, launch_build_clover(lat, csw, kappa, lat->stream), "build_clover");
    }
    if (st != WC_OK) return st;
    lat->csw = csw;
    lat->kappa = kappa;
    lat->clover_loaded = true;
    lat->cinv_loaded = false;
    return WC_OK;
}

wc_status wc_field_create(wc_lattice lat, wc_prec prec, wc_field *out)
{
    if (!lat || !out) return set_error(lat, WC_ERR_ARG, "lattice and out must not be NULL");
    *out = nullptr;
    if (prec != WC_F64 && prec != WC_F32 && prec != WC_F16) return set_error(lat, WC_ERR_ARG, "bad precision");
    wc_field f = new (std::nothrow) wc_field_s();
    if (!f) return set_error(lat, WC_ERR_ARG, "out of host memory");
    f->lat = lat;
    f->prec = prec;
    wc_status st = check_cuda(lat, cudaMalloc(&f->data, spinor_bytes(prec, lat->g.V)), "cudaMalloc(field)");
    if (st == WC_OK && prec == WC_F16)
        st = check_cuda(lat, dalloc(&f->nrm, sizeof(float) * (size_t)lat->g.V), "cudaMalloc(field)");
    if (st == WC_OK) st = check_cuda(lat, cudaMemsetAsync(f->data, 0, spinor_bytes(prec, lat->g.V), lat->stream),
                                     "cudaMemset(field)");
    if (st == WC_OK && f->nrm)
        st = check_cuda(lat, cudaMemsetAsync(f->nrm, 0, sizeof(float) * (size_t)lat->g.V, lat->stream),
                        "cudaMemset(field)");
    if (st != WC_OK) {
        wc_field_destroy(f);
        return st;
    }
    *out = f;
    return WC_OK;
}

wc_status wc_field_destroy(wc_field f)
{
    if (!f) return WC_OK;
    // cudaFree waits for outstanding device work that may use the buffers
    cudaFree(f->data);
    cudaFree(f->nrm);
    delete f;
    return WC_OK;
}

wc_status wc_field_import(wc_field f, const double *data)
{
    return field_import(f, reinterpret_cast<const double2 *>(data));
}

wc_status wc_field_export(wc_field f, double *data)
{
    return field_export(f, reinterpret_cast<double2 *>(data));
}

wc_status wc_field_import_f32(wc_field f, const float *data)
{
    return field_import(f, reinterpret_cast<const float2 *>(data));
}

wc_status wc_field_import_async(wc_field f, const void *data, int complex64)
{
    return complex64 ? field_import_async(f, static_cast<const float2 *>(data))
                     : field_import_async(f, static_cast<const double2 *>(data));
}

wc_status wc_field_export_async(wc_field f, void *data, int complex64)
{
    return complex64 ? field_export_async(f, static_cast<float2 *>(data))
                     : field_export_async(f, static_cast<double2 *>(data));
}

wc_status wc_sync(wc_lattice lat)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    wc_status st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync");
    if (st == WC_OK && lat->copy_stream) st = check_cuda(lat, cudaStreamSynchronize(lat->copy_stream), "sync");
    if (st == WC_OK && lat->copy_out_stream)
        st = check_cuda(lat, cudaStreamSynchronize(lat->copy_out_stream), "sync");
    return st;
}

wc_status wc_field_export_f32(wc_field f, float *data)
{
    return field_export(f, reinterpret_cast<float2 *>(data));
}

wc_status wc_field_copy(wc_field dst, wc_field src, double scale)
{
    if (!dst || !src) return set_error(nullptr, WC_ERR_ARG, "field is NULL");
    wc_lattice lat = dst->lat;
    if (src->lat != lat) return set_error(lat, WC_ERR_ARG, "fields belong to different lattices");
    if (!isfinite(scale)) return set_error(lat, WC_ERR_ARG, "scale must be finite");
    return check_cuda(lat, launch_copy(lat, dst, src, scale, nullptr, 0, lat->stream), "field_copy");
}

static wc_status apply_common(wc_lattice lat, wc_field out, wc_field in, int kind)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    wc_status st = check_field(lat, out, "out");
    if (st == WC_OK) st = check_field(lat, in, "in");
    if (st != WC_OK) return st;
    if (out == in || out->data == in->data) return set_error(lat, WC_ERR_ARG, "out and in must be distinct fields");
    if (out->prec != in->prec) return set_error(lat, WC_ERR_ARG, "out and in must have the same precision");
    st = require_operator(lat, kind != 2);
    if (st != WC_OK) return st;
    return check_cuda(lat, launch_apply(lat, out, in, kind, lat->stream), "apply");
}

wc_status wc_apply_M(wc_lattice lat, wc_field out, wc_field in) { return apply_common(lat, out, in, 0); }

wc_status wc_apply_multi(wc_lattice lat, int n, wc_field *outs, wc_field *ins, int dagger)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    if (n < 1 || n > kMrhsMax || !outs || !ins)
        return set_error(lat, WC_ERR_ARG, "n must be in 1.." + std::to_string(kMrhsMax) + ", outs/ins non-NULL");
    for (int r = 0; r < n; ++r) {
        wc_status st = check_field(lat, outs[r], "out");
        if (st == WC_OK) st = check_field(lat, ins[r], "in");
        if (st != WC_OK) return st;
        if (outs[r]->prec != WC_F32 || ins[r]->prec != WC_F32)
            return set_error(lat, WC_ERR_ARG, "the multi-RHS operator takes FP32 fields");
        for (int q = 0; q < n; ++q)
            if (outs[r] == ins[q] || (q < r && outs[r] == outs[q]))
                return set_error(lat, WC_ERR_ARG, "out fields must be distinct from each other and from the inputs");
    }
    wc_status st = require_operator(lat);
    if (st != WC_OK) return st;
    return check_cuda(lat, launch_apply_multi(lat, n, outs, ins, dagger ? 1 : 0, lat->stream),
                      "apply_multi");
}

wc_status wc_apply_schur(wc_lattice lat, wc_field out, wc_field in, int dagger)
{
    if (!lat) return set_error(nullptr, WC_ERR_ARG, "lattice is NULL");
    wc_status st = check_field(lat, out, "out");
    if (st == WC_OK) st = check_field(lat, in, "in");
    if (st != WC_OK) return st;
    if (out == in || out->prec != in->prec)
        return set_error(lat, WC_ERR_ARG, "out and in must be distinct fields of one precision");
    st = require_operator(lat);
    if (st != WC_OK) return st;
    wc_lattice h = nullptr;
    st = half_lattice(lat, &h);
    if (st != WC_OK) return st;
    // the half fields are kept between calls up to kKeptWorkspace (creating and
    // freeing three per call had cost 0.4 ms, the FP64 operator itself takes
    // 0.3 ms at 16^3x32); the lock is held until the stream has finished
    std::lock_guard<std::mutex> lk(lat->eom_mutex);
    wc_field *io = lat->schur_io[in->prec];
    for (int k = 0; k < 2 && st == WC_OK; ++k)
        if (!io[k]) st = wc_field_create(h, in->prec, &io[k]);
    if (st == WC_OK) st = check_cuda(lat, launch_split(lat, in, io[0], nullptr, lat->stream), "split");
    if (st == WC_OK) st = check_cuda(lat, launch_schur(h, io[1], io[0], dagger ? 1 : 0, lat->stream), "schur");
    if (st == WC_OK) st = check_cuda(lat, launch_merge(lat, io[1], nullptr, out, lat->stream), "merge");
    if (st == WC_OK) st = check_cuda(lat, cudaStreamSynchronize(lat->stream), "sync");
    if (2 * spinor_bytes(in->prec, h->g.V) > kKeptWorkspace)
        for (int k = 0; k < 2; ++k) {
            wc_field_destroy(io[k]);
            io[k] = nullptr;
        }
    return st;
}
wc_status wc_apply_Mdag(wc_lattice lat, wc_field out, wc_field in) { return apply_common(lat, out, in, 1); }
wc_status wc_apply_hop(wc_lattice lat, wc_field out, wc_field in) { return apply_common(lat, out, in, 2); }

wc_status wc_apply_shape(wc_lattice lat, wc_prec prec, int kind, int force_index, int shape_out[6])
{
    if (!lat || !shape_out) return set_error(lat, WC_ERR_ARG, "lattice and shape_out must not be NULL");
    if (prec != WC_F64 && prec != WC_F32 && prec != WC_F16) return set_error(lat, WC_ERR_ARG, "bad precision");
    if (kind < 0 || kind > 2) return set_error(lat, WC_ERR_ARG, "kind must be 0 (M), 1 (M^+) or 2 (H)");
    if (force_index < -2 || force_index >= apply_shape_count())
        return set_error(lat, WC_ERR_ARG, "force_index out of range");
    if (!apply_shape(lat, prec, kind, force_index, shape_out))
        return set_error(lat, WC_ERR_ARG, "launch shape does not fit this lattice / precision");
    return WC_OK;
}

wc_status wc_checked_violations(unsigned long long *count)
{
    if (!count) return set_error(nullptr, WC_ERR_ARG, "count is NULL");
    *count = 0;
    if (!kChecked) return set_error(nullptr, WC_ERR_STATE, "not a checked build (compile with -DWC_CHECKED)");
    wc_status st = check_cuda(nullptr, cudaDeviceSynchronize(), "sync");
    for (auto read : check_readers()) {
        if (st != WC_OK) break;
        unsigned v = 0;
        st = check_cuda(nullptr, read(&v), "read violation counter");
        *count += v;
    }
    return st;
}

const char *wc_last_error(wc_lattice lat)
{
    if (lat) return lat->err.c_str();
    return g_global_error.c_str();
}

}  // extern "C"
