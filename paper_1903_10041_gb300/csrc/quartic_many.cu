// Algorithm 1 + clamp on many independent quartics (the quartic benchmark
// of Sec. III-C): admm_quartic_min (FP64, quartic_min64_seeded) and
// admm_quartic_min_f32 (FP32 on packed pairs, quartic_min32x2_wells, branch
// decisions as FP64 would take them).  Each thread takes consecutive
// elements (pairs in FP32) in a grid-stride loop: 7 streams of one value
// each, coalesced.  Invalid elements (A < 0, A = C = 0, lo > hi, non-finite)
// get x = NaN and are counted, per thread first, then once per block in a
// word of pinned host memory that the call owns while it runs, so a call
// allocates and copies nothing for it.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <mutex>

#include <cuda_runtime.h>

#include "internal.h"
#include "trace.h"
#include "quartic32.cuh"

using namespace admm_impl;

namespace {

// Comparisons on the integer pipes: see quartic64.cuh.
__device__ __forceinline__ bool quartic_ok(double A, double B, double C, double D, double lo, double hi)
{
    const long long a = __double_as_longlong(A), l = __double_as_longlong(lo), h = __double_as_longlong(hi);
    const bool zero_a = (a << 1) == 0;
    auto top = [](double v) { return __double2hiint(v) & 0x7fffffff; }; // >= 0x7ff00000: not finite
    auto is_nan = [](long long v) { return (unsigned long long)(v << 1) > 0xffe0000000000000ull; };
    return max(max(top(A), top(B)), max(top(C), top(D))) < 0x7ff00000 && !is_nan(l) && !is_nan(h) &&
           (a > 0 || (zero_a && __double_as_longlong(C) > 0)) && (ord64(lo) <= ord64(hi) || ((l | h) << 1) == 0);
}
__device__ __forceinline__ bool quartic_ok(float A, float B, float C, float D, float lo, float hi)
{
    return isfinite(A) && isfinite(B) && isfinite(C) && isfinite(D) && A >= 0.0f && (A > 0.0f || C > 0.0f) && lo <= hi;
}

// Adds a block's invalid elements to the call's word.
__device__ __forceinline__ void report_bad(int n, int *bad)
{
    const int t = __syncthreads_count(n > 0); // most calls have none
    if (t == 0) return;
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n > 0) atomicAdd(bad, n);
}

__global__ void __launch_bounds__(256) quartic_many_f64(const double *A, const double *B, const double *C,
                                                        const double *D, const double *lo, const double *hi,
                                                        int64_t count, int mode, double *x, int *bad)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool in = t < count;
    const int64_t u = in ? t : count - 1;
    double a = A[u], b = B[u], c = C[u], d = D[u], l = lo[u], h = hi[u];
    const bool ok = quartic_ok(a, b, c, d, l, h);
    if (!ok) a = b = d = l = h = 0.0, c = 1.0;
    const double r = quartic_min64_seeded(a, b, c, d, l, h, mode);
    if (in) x[t] = ok ? r : NAN;
    const int nbad = in && !ok;
    report_bad(nbad, bad);
}

// The lanes that the packed code left (a NaN in r): solved alone, or counted as invalid.  Out of line.
__device__ __noinline__ float2 quartic_pair_rest(float2 a, float2 b, float2 c, float2 d, float2 l, float2 h, float2 r,
                                                 int mode, int *nbad)
{
    unsigned esc = 0;
    if (isnan(r.x)) {
        if (quartic_ok(a.x, b.x, c.x, d.x, l.x, h.x)) r.x = quartic_min32(a.x, b.x, c.x, d.x, l.x, h.x, mode, esc);
        else ++*nbad;
    }
    if (isnan(r.y)) {
        if (quartic_ok(a.y, b.y, c.y, d.y, l.y, h.y)) r.y = quartic_min32(a.y, b.y, c.y, d.y, l.y, h.y, mode, esc);
        else ++*nbad;
    }
    return r;
}

// One pair; an element's bits depend on its own data alone.
__device__ __forceinline__ float2 quartic_pair(float2 a, float2 b, float2 c, float2 d, float2 l, float2 h, int mode,
                                               int *nbad)
{
    // finite coefficients (their magnitudes' sum is) and lo <= hi; anything else is looked at lane by lane
    const float2 m = add2(add2(abs2(a), abs2(b)), add2(abs2(c), abs2(d)));
    bool okx, oky;
    const float2 r = quartic_min32x2_wells(a, b, c, d, l, h, mode, okx, oky);
    okx = okx && m.x < INFINITY && l.x <= h.x;
    oky = oky && m.y < INFINITY && l.y <= h.y;
    if (okx && oky) return r;
    return quartic_pair_rest(a, b, c, d, l, h, make_float2(okx ? r.x : NAN, oky ? r.y : NAN), mode, nbad);
}

// The last element of an odd count, paired with x^4 + x^2.  Out of line.
__device__ __noinline__ float quartic_odd(float a, float b, float c, float d, float l, float h, int mode, int *nbad)
{
    return quartic_pair(make_float2(a, 1.0f), make_float2(b, 0.0f), make_float2(c, 1.0f), make_float2(d, 0.0f),
                        make_float2(l, -1.0f), make_float2(h, 1.0f), mode, nbad)
        .x;
}

constexpr int kThreads32 = 128, kPerSm = 64;
__global__ void __launch_bounds__(kThreads32, 8) quartic_many_f32(const float *A, const float *B, const float *C,
                                                        const float *D, const float *lo, const float *hi,
                                                        int64_t count, int mode, float *x, int *bad)
{
    const int64_t pairs = count / 2;
    int nbad = 0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    float2 na, nb, nc, nd, nl, nh; // the thread's next pair, loaded while this one is solved
    auto load = [&](int64_t u) {
        na = ((const float2 *)A)[u];
        nb = ((const float2 *)B)[u];
        nc = ((const float2 *)C)[u];
        nd = ((const float2 *)D)[u];
        nl = ((const float2 *)lo)[u];
        nh = ((const float2 *)hi)[u];
    };
    if (t < pairs) load(t);
    for (; t < pairs; t += step) {
        const float2 a = na, b = nb, c = nc, d = nd, l = nl, h = nh;
        if (t + step < pairs) load(t + step);
        ((float2 *)x)[t] = quartic_pair(a, b, c, d, l, h, mode, &nbad);
    }
    if (count % 2 == 1 && blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t u = count - 1; // the odd element
        x[u] = quartic_odd(A[u], B[u], C[u], D[u], lo[u], hi[u], mode, &nbad);
    }
    report_bad(nbad, bad);
}

// The calls' counters: words of one pinned, device-mapped host page, taken
// by a call and given back when it returns (any thread, stream or device).
// With every word taken, a call waits for none and allocates a page of its own.
class BadWords {
    static constexpr int kWords = 64, kStride = 32; // ints: one word per 128 bytes
    std::mutex mu_;
    int *page_ = nullptr;
    uint64_t taken_ = 0;

public:
    struct Word {
        int *p = nullptr;
        int slot = -1; // -1: a page of its own
    };
    cudaError_t take(Word &w)
    {
        std::lock_guard<std::mutex> lk(mu_);
        if (page_) { // gone if the device was reset since
            cudaPointerAttributes at{};
            if (cudaPointerGetAttributes(&at, page_) != cudaSuccess || at.type != cudaMemoryTypeHost) {
                cudaGetLastError();
                page_ = nullptr;
                taken_ = 0;
            }
        }
        if (!page_) {
            const cudaError_t e = cudaHostAlloc((void **)&page_, sizeof(int) * kWords * kStride,
                                                cudaHostAllocMapped | cudaHostAllocPortable);
            if (e != cudaSuccess) return page_ = nullptr, e;
        }
        for (int t = 0; t < kWords; ++t)
            if (!(taken_ >> t & 1)) {
                taken_ |= 1ull << t;
                w = {page_ + t * kStride, t};
                *w.p = 0;
                return cudaSuccess;
            }
        const cudaError_t e = cudaHostAlloc((void **)&w.p, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable);
        if (e == cudaSuccess) *w.p = 0;
        return e;
    }
    void give(Word &w)
    {
        if (!w.p) return;
        if (w.slot < 0) {
            cudaFreeHost(w.p);
        } else {
            std::lock_guard<std::mutex> lk(mu_);
            taken_ &= ~(1ull << w.slot);
        }
        w.p = nullptr;
    }
};
BadWords g_bad_words;

// CTAs of the FP32 kernel: a pair per thread up to kPerSm CTAs per SM (eight
// resident, the rest handed out as others finish), then more pairs per thread,
// whose next loads run beside the solve.  2^26 quartics: 389 us with a pair per
// thread and no prefetch, 350 (80 % of HBM) so.
int quartic_grid(int64_t pairs)
{
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int64_t want = (pairs + kThreads32 - 1) / kThreads32;
    return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)std::max(nsm, 1) * kPerSm));
}

template <class T>
admm_status quartic_min_impl(const T *A, const T *B, const T *C, const T *D, const T *lo, const T *hi, int64_t count,
                             T *x, int32_t xmin_mode, int32_t on_device, void *stream)
{
    TraceRange trace_("admm_quartic_min");
    clear_last_error();
    if (count < 0 || (count > 0 && (!A || !B || !C || !D || !lo || !hi || !x)))
        return set_last_error("NULL array or negative count"), ADMM_EINVAL;
    if (xmin_mode != ADMM_XMIN_EXACT && xmin_mode != ADMM_XMIN_PAPER)
        return set_last_error("bad xmin_mode"), ADMM_EINVAL;
    if (count == 0) return ADMM_OK;
    if (on_device) { // the kernel dereferences these: they must be device-accessible
        const void *ptrs[7] = {A, B, C, D, lo, hi, x};
        for (const void *ptr : ptrs) {
            cudaPointerAttributes at{};
            if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess ||
                (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)) {
                cudaGetLastError(); // clear a sticky query error
                return set_last_error("on_device = 1 but an array is not device memory"), ADMM_EINVAL;
            }
        }
    }
    if (sizeof(T) == 4 && on_device &&
        ((uintptr_t)A | (uintptr_t)B | (uintptr_t)C | (uintptr_t)D | (uintptr_t)lo | (uintptr_t)hi | (uintptr_t)x) % 8)
        return set_last_error("FP32 device arrays must be 8-byte aligned"), ADMM_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = sizeof(T) * (size_t)count;
    T *d[7] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    BadWords::Word bad;
    int *dbad = nullptr;
    cudaError_t e = g_bad_words.take(bad);
    if (e == cudaSuccess) e = cudaHostGetDevicePointer((void **)&dbad, bad.p, 0);
    const T *src[6] = {A, B, C, D, lo, hi};
    if (!on_device)
        for (int t = 0; t < 7 && e == cudaSuccess; ++t) {
            e = cudaMallocAsync(&d[t], bytes, st);
            if (e == cudaSuccess && t < 6) e = cudaMemcpyAsync(d[t], src[t], bytes, cudaMemcpyHostToDevice, st);
        }
    if (e == cudaSuccess) {
        const T *a[6];
        for (int t = 0; t < 6; ++t) a[t] = on_device ? src[t] : d[t];
        T *xo = on_device ? x : d[6];
        if constexpr (sizeof(T) == 8)
            quartic_many_f64<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(a[0], a[1], a[2], a[3], a[4], a[5], count,
                                                                  xmin_mode, xo, dbad);
        else
            quartic_many_f32<<<quartic_grid((count + 1) / 2), kThreads32, 0, st>>>(a[0], a[1], a[2], a[3], a[4], a[5],
                                                                          count, xmin_mode, xo, dbad);
        e = cudaGetLastError();
        if (e == cudaSuccess && !on_device) e = cudaMemcpyAsync(x, d[6], bytes, cudaMemcpyDeviceToHost, st);
    }
    for (T *p : d)
        if (p) cudaFreeAsync(p, st);
    const cudaError_t es = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = es;
    const int hbad = e == cudaSuccess ? *(volatile int *)bad.p : 0;
    g_bad_words.give(bad);
    if (e != cudaSuccess) {
        set_last_error(cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? ADMM_ENOMEM : ADMM_ECUDA;
    }
    if (hbad > 0) {
        char m[96];
        snprintf(m, sizeof m, "%d invalid quartics (x = NaN there)", hbad);
        set_last_error(m);
        return ADMM_EINVAL;
    }
    return ADMM_OK;
}

} // namespace

extern "C" {

admm_status admm_quartic_min(const double *A, const double *B, const double *C, const double *D, const double *lo,
                             const double *hi, int64_t count, double *x, int32_t xmin_mode, int32_t on_device,
                             void *stream)
{
    return quartic_min_impl<double>(A, B, C, D, lo, hi, count, x, xmin_mode, on_device, stream);
}

admm_status admm_quartic_min_f32(const float *A, const float *B, const float *C, const float *D, const float *lo,
                                 const float *hi, int64_t count, float *x, int32_t xmin_mode, int32_t on_device,
                                 void *stream)
{
    return quartic_min_impl<float>(A, B, C, D, lo, hi, count, x, xmin_mode, on_device, stream);
}

} // extern "C"
