// Pieces shared by the Gram-matrix kernels (calib_cov.cu, quantize.cu): the sum of partial tiles over a cluster.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rosaq {

// Lets the next kernel of the stream start.  To be called when little is left to do: the bounded waits of that kernel run from its
// start, and the time of a Gram matrix grows with its tokens without a bound.
__device__ __forceinline__ void cov_grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void cov_grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void cov_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void cov_epi_bar() { asm volatile("bar.sync 1, 128;" ::: "memory"); }   // the four epilogue warps

// Rows [r_begin, r_end) of the tile staged at `stage` (shared address `addr`, `pitch` floats per row) become the sum over the
// cluster's Z tiles, added in order of the splits.  The tile of split k lies at the same address of cluster rank
// ranks_per_split * k + rank_in_split.  Only these rows of this CTA's tile change, and nobody else reads them.
// `cols` is a power of two and (r_end - r_begin) * cols a multiple of 8 * threads.
__device__ __forceinline__ void cov_sum_rows(uint32_t addr, float *stage, int pitch, int cols, int r_begin, int r_end, int Z,
                                             int ranks_per_split, uint32_t rank_in_split, int tid, int threads) {
  const int n = (r_end - r_begin) * cols, shift = 31 - __clz(cols);
  for (int i0 = tid; i0 < n; i0 += 8 * threads) {
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    for (int k0 = 0; k0 < Z; k0 += 4) {                      // 32 loads in flight: a round trip costs 200 ns
      float v[4][8];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k0 + k < Z) {
          uint32_t remote;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"((uint32_t)(ranks_per_split * (k0 + k)) + rank_in_split));
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int i = i0 + e * threads;
            asm volatile("ld.shared::cluster.f32 %0, [%1];"
                         : "=f"(v[k][e])
                         : "r"(remote + (uint32_t)((r_begin + (i >> shift)) * pitch + (i & (cols - 1))) * 4u));
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k0 + k < Z)
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] = __fadd_rn(acc[e], v[k][e]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = i0 + e * threads;
      stage[(r_begin + (i >> shift)) * pitch + (i & (cols - 1))] = acc[e];
    }
  }
}

// How many CTAs of a cluster share the tokens of a tile: the largest power of two that the cluster size, the
// tokens (`most_by_work` splits leave each enough of them) and the CTAs resident at once allow.
inline int cov_splits(long long ctas, int slots, long long most_by_work, int most) {
  int z = 1;
  while (2 * z <= most && 2 * z <= most_by_work && 2 * z * ctas <= slots) z *= 2;
  return z;
}

// cluster of x_dim CTAs along x times `splits` along z
template <typename K, typename... Args>
int cov_launch(K kern, dim3 grid, int threads, size_t smem, int x_dim, int splits, cudaStream_t s, const Args &...args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[na].val.programmaticStreamSerializationAllowed = 1;
  ++na;
  if (x_dim * splits > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = x_dim;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = splits;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  if (cudaLaunchKernelEx(&cfg, kern, args...) != cudaSuccess) {
    (void)cudaGetLastError();
    return ROSAQ_ERR_CUDA;
  }
  return ROSAQ_OK;
}

}  // namespace rosaq
