// Cluster variants of the single-instance solve kernel (small problems), in a
// translation unit of their own so that the two compile in parallel.
#include "single_kernel.cuh"

namespace admm_impl {

namespace {
template <int M> void *cluster_fn(int precision)
{
    switch (precision) {
    case ADMM_MIXED: return (void *)single_kernel<M, ADMM_MIXED, kBlock, true>;
    case ADMM_MIXED_FP64CUBIC: return (void *)single_kernel<M, ADMM_MIXED_FP64CUBIC, kBlock, true>;
    default: return (void *)single_kernel<M, ADMM_FP64, kBlockF64Cluster, true>;
    }
}
} // namespace

void *single_cluster_fn(int precision, int m)
{
    switch (single_mbound(m)) {
    case 2: return cluster_fn<2>(precision);
    case 4: return cluster_fn<4>(precision);
    default: return cluster_fn<8>(precision);
    }
}

} // namespace admm_impl
