// Device helpers shared by the solver kernels: bounded grid barrier,
// deterministic warp/block reductions, L2-coherent loads.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace admm_impl {

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ int ld_volatile_i32(const int *p)
{
    return *(const volatile int *)p;
}

// Bounds-checked builds (compiled with -DADMM_DEBUG_BOUNDS, libadmm_debug.so):
// an element-array index is checked against the instance's range of that
// array before the access; an index outside it is recorded in *rec (array
// id in the top byte, the index below; the first violation wins) and
// replaced by 0, so the access stays inside the allocation and the kernel
// carries on.  The host turns a record into ADMM_EBOUNDS.  Release builds
// use the index as it is.
#ifdef ADMM_DEBUG_BOUNDS
__device__ __forceinline__ size_t dbg_index(size_t idx, size_t need, size_t len, unsigned long long *rec, int id)
{
    if (idx + need <= len) return idx;
    if (rec) atomicCAS(rec, 0ull, ((unsigned long long)(id + 1) << 56) | (idx & 0x00FFFFFFFFFFFFFFull));
    return 0;
}
#define ADMM_IDX(idx, need, len, rec, id) ::admm_impl::dbg_index((idx), (need), (len), (rec), (id))
#else
#define ADMM_IDX(idx, need, len, rec, id) (idx)
#endif
// array ids of the bounds records
enum { DBG_COL = 0, DBG_X = 1, DBG_COEF = 2, DBG_BOUND = 3, DBG_SELFTEST = 15 };

// Loads that bypass L1: data written by other SMs since this SM last cached it.
__device__ __forceinline__ double ldcg(const double *p) { return __ldcg(p); }

// Grid-wide barrier for a cooperative launch.  `bar` counts arrivals and is
// zeroed before the launch; barrier number b (1, 2, ...) waits for b * grid
// arrivals.  The arrival is a release and the poll an acquire at GPU scope
// (cumulative over the CTA's writes ordered by the first __syncthreads), so
// no fences are needed around them: 2690 -> 2380 cycles for 150 CTAs.  The
// wait is bounded: after spin_ns nanoseconds it records timeout_code in
// *status and returns false; it also returns false as soon as another CTA
// has recorded an error.  Never traps.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned target, int *status,
                                             long long spin_ns, int timeout_code)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(1u) : "memory");
        unsigned long long t0 = 0;
        int ok = 1;
        for (unsigned spins = 1;; ++spins) {
            unsigned v = ld_acquire_u32(bar);
            if ((int)(v - target) >= 0)
                break;
            if ((spins & 15) == 0) { // error flag and time limit every 16 polls
                if (ld_volatile_i32(status) != 0) { ok = 0; break; }
                if (t0 == 0) t0 = globaltimer_ns();
                if ((long long)(globaltimer_ns() - t0) > spin_ns) {
                    atomicCAS(status, 0, timeout_code);
                    ok = 0;
                    break;
                }
            }
            __nanosleep(32); // leave issue slots to co-resident CTAs still computing
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <class T> __device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <class T> __device__ __forceinline__ T warp_max(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// Maxima of non-negative doubles (residual terms, absolute values): for
// x, y >= 0 the order of their IEEE-754 bit patterns read as signed 64-bit
// integers is the order of the values, so these run on the integer pipes
// instead of the FP64 pipe (1/64 of the FP32 rate on this GPU).  A NaN without
// its sign ranks above infinity, so it is kept and fails the stop test; the FP32
// forms are there for that alone.
__device__ __forceinline__ double max_nonneg(double a, double b)
{
    return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
__device__ __forceinline__ float max_nonneg(float a, float b)
{
    return __uint_as_float(max(__float_as_uint(a), __float_as_uint(b)));
}
__device__ __forceinline__ float warp_max_nonneg(float v)
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_max_nonneg(double v)
{
    long long b = __double_as_longlong(v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
    return __longlong_as_double(b);
}
template <class T> __device__ __forceinline__ T warp_min(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Warp sums (or maxima, minima) of M values per lane at once: while more than
// one value is left, a step halves the values by keeping one half in the
// lanes with the step's bit clear and the other in those with it set, so M
// values take M - 1 + log2(32 / M) combinations instead of 5 M.  The total of
// value slot_of<M>(lane) ends up in every lane of its group of 32 / M.
template <int M> __device__ __forceinline__ int slot_of(int lane)
{
    return M == 2 ? lane >> 4 : (M == 4 ? lane >> 3 : lane >> 2);
}
template <int M, class T, class F> __device__ __forceinline__ T warp_many(T *v, F comb)
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int c = M; c > 1; c >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int t = 0; t < M / 2; ++t)
            if (t < c / 2) {
                const T keep = up ? v[t + c / 2] : v[t], send = up ? v[t] : v[t + c / 2];
                v[t] = comb(keep, send, o);
            }
        o >>= 1;
    }
    T r = v[0];
#pragma unroll
    for (int u = 16 / M; u > 0; u >>= 1) r = comb(r, r, u);
    return r;
}

__device__ __forceinline__ double clampd(double v, double lo, double hi)
{
    return v < lo ? lo : (v > hi ? hi : v);
}
__device__ __forceinline__ float clampf(float v, float lo, float hi)
{
    return v < lo ? lo : (v > hi ? hi : v);
}

} // namespace admm_impl
