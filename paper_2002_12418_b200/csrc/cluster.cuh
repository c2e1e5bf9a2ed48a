// Thread-block cluster helpers: ranks, cluster addresses, barriers, and the sum of partial accumulators over the CTAs of a
// cluster that share one work item's K loop.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mnnb {
namespace ptx {

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Cluster address of the shared-memory location `addr` (an address of this CTA) in the CTA of rank `rank`.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float ld_cluster_f32(uint32_t cluster_addr)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr) : "memory");
    return v;
}

// Split accumulators lie in every CTA's shared memory as [column][128 rows] fp32 from `smem_base` on.  Calls
// emit(column, sum) for this rank's share of the bn columns (a multiple of 16) and the given row; the partial sums are
// added in rank order, so the result does not depend on timing.
template <typename Emit>
__device__ __forceinline__ void cluster_reduce_columns(uint32_t smem_base, int bn, uint32_t rank, int split, int row, int first, int step,
                                                       Emit&& emit)
{
    const int c0 = bn * (int)rank / split, c1 = bn * ((int)rank + 1) / split;
    for (int c = c0 + first; c < c1; c += 2 * step) {
        float v[2][8];
#pragma unroll
        for (int s = 0; s < 8; ++s)
            if (s < split) {
                const uint32_t a = map_to_rank(smem_base, (uint32_t)s) + (uint32_t)(c * 128 + row) * 4u;
                v[0][s] = ld_cluster_f32(a);
                if (c + step < c1) v[1][s] = ld_cluster_f32(a + (uint32_t)step * 512u);
            }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (c + h * step < c1) {
                float sum = v[h][0];
#pragma unroll
                for (int s = 1; s < 8; ++s)
                    if (s < split) sum += v[h][s];
                emit(c + h * step, sum);
            }
    }
}

}  // namespace ptx
}  // namespace mnnb
