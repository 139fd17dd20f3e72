// Host side of the single-instance solve kernel (single_kernel.cuh): variants,
// launch shape, launch, and the row conversions of the C ABI's state import
// and export.  The cluster variants are instantiated in single_cluster.cu.
#include <algorithm>

#include "single_kernel.cuh"

namespace admm_impl {

namespace {

template <int M> void *single_fn(int precision, int wide)
{
    switch (precision) {
    case ADMM_MIXED:
        return wide == 1 ? (void *)single_kernel<M, ADMM_MIXED, kBlock, false>
                         : (void *)single_kernel<M, ADMM_MIXED, kBlockWide, false>;
    case ADMM_MIXED_FP64CUBIC:
        return wide == 1 ? (void *)single_kernel<M, ADMM_MIXED_FP64CUBIC, kBlock, false>
                         : (void *)single_kernel<M, ADMM_MIXED_FP64CUBIC, kBlockWide, false>;
    default: return (void *)single_kernel<M, ADMM_FP64, kBlockF64, false>;
    }
}

void *pick(int precision, int m, int wide)
{
    if (wide == 0) return single_cluster_fn(precision, m);
    switch (single_mbound(m)) {
    case 2: return single_fn<2>(precision, wide);
    case 4: return single_fn<4>(precision, wide);
    default: return single_fn<8>(precision, wide);
    }
}

} // namespace

int single_mbound(int m) { return m <= 2 ? 2 : (m <= 4 ? 4 : 8); }

// FP64: 12 warps (one CTA per SM, up to 168 registers a thread); the FP64
// units are shared by the SM, so more warps hide more of their latency.
// The cluster variant (wide = 0) takes a column per thread on one warp per
// scheduler: fewer warps make its barriers cheaper.
int single_threads(int precision, int wide)
{
    if (precision != ADMM_FP64) return wide == 2 ? kBlockWide : kBlock;
    return wide == 0 ? kBlockF64Cluster : kBlockF64;
}

// Launch configuration of the cluster variant: one cluster of `ctas` CTAs.
static void cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr, int precision, int ctas, size_t smem,
                           cudaStream_t st)
{
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(single_threads(precision, 0));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

size_t single_smem_bytes(int m, int q, int precision)
{
    const int mb = single_mbound(m);
    size_t stage = 0; // the rolling stage of the mixed kernels, one per warp
    if (precision != ADMM_FP64 && mb <= 4)
        stage = (size_t)(kBlockWide / 32) * (mb == 2 ? roll_slots<2>() : roll_slots<4>()) * 32 * sizeof(float2);
    return single_carve_bytes(m, q) + stage;
}

int single_blocks_per_sm(int precision, int m, int wide, size_t smem)
{
    void *fn = pick(precision, m, wide);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, single_threads(precision, wide), smem) != cudaSuccess)
        return 0;
    return nb;
}

static bool cluster_resident(int precision, int m, int ctas, size_t smem)
{
    void *fn = pick(precision, m, 0);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return cudaGetLastError(), false;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cluster_config(cfg, attr, precision, ctas, smem, 0);
    int nc = 0;
    if (cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) != cudaSuccess) return cudaGetLastError(), false;
    return nc >= 1;
}

SingleShape single_shape(int precision, int m, int q, int64_t rs, int nsm, size_t smem)
{
    SingleShape sh{};
    const bool mixed = precision != ADMM_FP64;
    const int64_t unit = mixed ? kMixedVW : 1;   // mixed: vectors of kMixedVW columns
    const int64_t ncols = (int64_t)q * rs;
    // Small problems: one cluster, each CTA one piece of one row with at most a
    // column (mixed: a column pair) per thread, so the element phase takes as
    // long as on more SMs (a warp's FP64 instruction takes the scheduler's 64
    // cycles anyway) and the cluster barrier and distributed shared memory save
    // the grid barrier and the records' way through L2.  Up to 8 CTAs, the
    // portable cluster size; beyond that a CTA would need several rounds.
    // us per iteration on the grid -> as a cluster, at one CTA and at eight: FP64,
    // m = 2: n = 100 9.5 -> 7.2, n = 1000 9.5 -> 7.4; m = 4, n = 1000 12.9 -> 11.4;
    // mixed: n = 100, m = 2 6.0 -> 4.5, n = 4000, m = 4 7.6 -> 6.5 (short solves,
    // the call's own time included).
    {
        const int64_t cap = mixed ? (int64_t)kBlock * unit : kBlockF64Cluster;
        const int64_t p = (rs + cap - 1) / cap;
        if (q * p <= kClusterCtas && cluster_resident(precision, m, (int)(q * p), smem)) {
            sh.wide = 0;
            sh.pieces = (int)p;
            sh.grid = (int)(q * p);
            sh.nbmax = (int)p;
            sh.chunk = cap;
            return sh;
        }
    }
    // Contiguous equal column chunks over as many SMs as there are warps of
    // work (FP64 throughput per SM is the scarce resource), one CTA per SM;
    // mixed: the wide variant where 256 threads per SM would take more than one
    // pass (see NT at single_kernel).
    sh.wide = (mixed && ncols > (int64_t)nsm * single_threads(precision, 1) * unit) ? 2 : 1;
    const int per_sm = single_blocks_per_sm(precision, m, sh.wide, smem);
    if (per_sm < 1) return sh;
    const int64_t g = std::min<int64_t>((int64_t)nsm * per_sm, std::max<int64_t>(1, ncols / (32 * unit)));
    sh.chunk = ((ncols + g - 1) / g + unit - 1) / unit * unit;
    // Row-aligned split when every row gets whole pieces and the largest
    // piece is within 5 % of the flat chunk: no CTA then straddles two rows
    // (a straddling CTA reduces two segments and finishes last).
    const int p = (int)(g / q);
    if (p >= 1) {
        int64_t big = 0;
        for (int t = 0; t < p; ++t)
            big = std::max(big, piece_bound(t + 1, rs, p, (int)unit) - piece_bound(t, rs, p, (int)unit));
        if (piece_bound(1, rs, p, (int)unit) > 0 && 20 * big <= 21 * sh.chunk) {
            sh.pieces = p;
            sh.grid = q * p;
            sh.nbmax = p;
            return sh;
        }
    }
    sh.pieces = 0;
    sh.grid = (int)((ncols + sh.chunk - 1) / sh.chunk);
    sh.nbmax = 1;
    for (int j = 0; j < q; ++j) {
        const int64_t r0 = (int64_t)j * rs, r1 = r0 + rs - 1;
        sh.nbmax = std::max(sh.nbmax, (int)(r1 / sh.chunk - r0 / sh.chunk + 1));
    }
    return sh;
}

cudaError_t launch_single(int precision, int wide, const SingleArgs &a, size_t smem, cudaStream_t st)
{
    void *fn = pick(precision, a.m, wide);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    SingleArgs copy = a;
    void *args[] = {(void *)&copy};
    if (wide == 0) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cluster_config(cfg, attr, precision, a.grid, smem, st);
        return cudaLaunchKernelExC(&cfg, fn, args);
    }
    return cudaLaunchCooperativeKernel(fn, dim3(a.grid), dim3(single_threads(precision, wide)), args, smem, st);
}

} // namespace admm_impl

namespace admm_impl {
namespace {
template <class S, class D>
__global__ void convert_rows_kernel(D *dst, int64_t dld, const S *src, int64_t sld, int n, int64_t rows)
{
    const int64_t total = rows * n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / n;
        const int k = (int)(t - r * n);
        dst[r * dld + k] = (D)src[r * sld + k];
    }
}
int conv_grid(int64_t total) { return (int)std::max<int64_t>(1, std::min<int64_t>(4096, (total + 255) / 256)); }
} // namespace

void convert_rows_f32_to_f64(double *dst, int64_t dld, const float *src, int64_t sld, int n, int64_t rows,
                             cudaStream_t st)
{
    convert_rows_kernel<float, double><<<conv_grid(rows * n), 256, 0, st>>>(dst, dld, src, sld, n, rows);
}
namespace {
__global__ void ff_to_f64_kernel(double *dst, int64_t dld, const float *hi, const float *lo, int64_t sld, int n,
                                 int64_t rows)
{
    const int64_t total = rows * n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / n;
        const int k = (int)(t - r * n);
        dst[r * dld + k] = (double)hi[r * sld + k] + (double)lo[r * sld + k];
    }
}
__global__ void f64_to_ff_kernel(float *hi, float *lo, int64_t dld, const double *src, int64_t sld, int n,
                                 int64_t rows)
{
    const int64_t total = rows * n;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / n;
        const int k = (int)(t - r * n);
        const double v = src[r * sld + k];
        const float h = (float)v;
        hi[r * dld + k] = h;
        lo[r * dld + k] = (float)(v - (double)h);
    }
}
} // namespace

void convert_rows_ff_to_f64(double *dst, int64_t dld, const float *hi, const float *lo, int64_t sld, int n,
                            int64_t rows, cudaStream_t st)
{
    ff_to_f64_kernel<<<conv_grid(rows * n), 256, 0, st>>>(dst, dld, hi, lo, sld, n, rows);
}
void split_rows_f64_to_ff(float *hi, float *lo, int64_t dld, const double *src, int64_t sld, int n, int64_t rows,
                          cudaStream_t st)
{
    f64_to_ff_kernel<<<conv_grid(rows * n), 256, 0, st>>>(hi, lo, dld, src, sld, n, rows);
}

void convert_rows_f64_to_f32(float *dst, int64_t dld, const double *src, int64_t sld, int n, int64_t rows,
                             cudaStream_t st)
{
    convert_rows_kernel<double, float><<<conv_grid(rows * n), 256, 0, st>>>(dst, dld, src, sld, n, rows);
}
} // namespace admm_impl
