// Check of the batched kernel's shared memory per CTA (batch.cu): for every
// source count, row count, CTA size, cluster size and team kind no more than
// `accepted`, the size that decides which shapes the batch and server calls
// have always taken, and within it at the shapes where an SM's shared memory
// just suffices.
#include <cstddef>
#include <cstdio>

#include "batch.h"

using namespace admm_impl;

static size_t team(int m, int q, int items, int warps)
{
    const int mq = m * q;
    return (size_t)scal_size(m, q) + 2 * (size_t)items * m * 4 + 4 * (size_t)warps + 24 + mq + 8 + kWarpsMax * 8 +
           2 * ((mq + 1) / 2) + 8;
}

static size_t accepted(int m, int q, int warps, int cluster, bool warp_teams)
{
    const size_t slice = (team(m, q, q, 1) + 3) / 4 * 4;
    size_t bytes = (8 * team(m, q, q + warps * cluster, warps) + 15) / 16 * 16;
    if (m <= 4) bytes += (size_t)warps * 34 * 32 * 8 + (size_t)warps * 32 * 11 * 4;
    if (warp_teams && 8 * slice * warps > bytes) bytes = 8 * slice * warps;
    return bytes;
}

int main()
{
    const size_t sm = 232448; // shared memory a CTA may have
    int edge = 0;
    for (int m = 1; m <= ADMM_MAX_M; ++m)
        for (int q = 1; q <= ADMM_BATCH_MAX_PAIRS; ++q)
            for (int warps = 4; warps <= 16; warps *= 2)
                for (int cluster = 1; cluster <= 8; cluster *= 2)
                    for (int wt = 0; wt < 2; ++wt) {
                        const size_t was = accepted(m, q, warps, cluster, wt != 0);
                        const size_t is = batch_cta_smem(m, q, warps, cluster, wt != 0, batch_slice_doubles(m, q)).bytes;
                        if (is > was) {
                            std::fprintf(stderr, "m %d q %d warps %d cluster %d warp teams %d: %zu > %zu bytes\n", m, q,
                                         warps, cluster, wt, is, was);
                            return 1;
                        }
                        if (was <= sm && was + 2048 > sm) ++edge;
                    }
    if (edge < 20) return std::fprintf(stderr, "few shapes at the edge: %d\n", edge), 1;
    std::puts("shared memory ok");
    return 0;
}
