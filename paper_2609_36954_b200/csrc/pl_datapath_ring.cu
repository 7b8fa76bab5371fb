// Datapath for gathering rings, and for reducing rings whose hops are asked for (PL_OPT_RING_HOPS; else they are
// folded, see pl_datapath_flat.cu), with the grid left to the library: a thread-block cluster per tile, one CTA per
// rank, the hops through distributed shared memory.
//
// A ring moves the partial sums of a partition from rank to rank, in a wider type than the data, so
// most of its bytes are partial sums: written by one rank, read once by the next.  On the op
// queues each of them goes through global memory, with a flag per hop.  Here rank r of a tile is
// CTA r of a cluster: it adds its own data to the partial sum in its shared memory and stores the
// result into the shared memory of CTA r + 1, and the cluster barrier (release / acquire) is the
// flag.  Only inputs and outputs touch global memory.  Clusters are independent of one another, so
// none has to be resident with another; a barrier is reached by every thread of a cluster
// whatever the data, so nothing waits for what may not come.
//
// A large message is bound by the stores into the neighbours and the barriers between them, a small
// one by R - 1 (or 2 R - 2) times a hop of about 0.6 us.  Own data is loaded a step ahead.  On the op
// queues -> here: reduce-scatter 8 x 64 MiB bf16 349 -> 238 us, all-reduce 8 x 64 MiB 469 -> 394,
// 4 x 1 MiB fp32 13.5 -> 7.6, 8 x 64 KiB bf16 28.8 -> 9.4, 16 x 16 MiB 335 -> 248; all-gather
// 8 x 64 KiB 15.2 -> 7.8.  Tiles handed out by a counter in global memory, and op queues in
// wavefront order, took the same as the queues: their partial sums went through global memory still.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "pl_device.cuh"
#include "pl_internal.h"
#include "pl_kernels.h"
#include "pl_ptx.cuh"

namespace pl {
namespace {

using namespace dev;

__device__ __forceinline__ uint4 lds16(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
// store into the shared memory of another CTA of the cluster (address from map_to_rank)
__device__ __forceinline__ void st_cluster16(uint32_t a, const uint4& v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t a, uint32_t cta) {
  uint32_t o;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(cta));
  return o;
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Two buffers for what arrives, alternated by step; a partial sum lies in two planes of 16 bytes per
// unit (sums / corrections, or the halves of eight fp32 sums).
template <int DT, int U>
__global__ void __launch_bounds__(kRingThreads) pl_ring_kernel(const __grid_constant__ RingHopParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr bool kWide = DT == PL_BF16 || DT == PL_F32;  // partial sums take 32 bytes per unit
  const uint32_t R = (uint32_t)P.n_ranks, nthr = blockDim.x, tid = threadIdx.x;
  const uint32_t c = blockIdx.x / R, r = blockIdx.x - c * R, q = r ? r - 1 : R - 1;
  const uint32_t plane = P.tile * 16u, base = ptx::smem_u32(smem);
  const uint32_t next = map_to_rank(base, r + 1 == R ? 0u : r + 1);
  const uint64_t u0 = (uint64_t)c * P.tile;
  const uint32_t units = (uint32_t)min((uint64_t)P.tile, P.part_units - u0);
  auto buffer = [&](uint32_t step) { return (step & 1u) * (kWide ? 2u : 1u) * plane; };
  auto part_off = [&](uint32_t k, uint32_t i) { return (k * P.part_units + u0 + tid + i * nthr) * 16ull; };
  auto live = [&](uint32_t i) { return tid + i * nthr < units; };
  pdl_launch_dependents();
  cluster_arrive();  // every CTA of the cluster runs before one stores into another
  cluster_wait();
  pdl_wait();

  uint32_t step = 0;
  if constexpr (DT != PL_U8) {
    if (P.reduce) {
      uint4 b[U], a[U];
      uint32_t k = r >= 2 ? r - 2 : r + R - 2;  // partition that reaches rank r at step 0; one lower at each later step
#pragma unroll
      for (uint32_t i = 0; i < U; ++i)
        if (live(i)) {
          a[i] = ld16(static_cast<const char*>(P.in[q]) + part_off(k, i));
          b[i] = ld16(static_cast<const char*>(P.in[r]) + part_off(k, i));
        }
      for (; step + 1 < R; ++step) {
        const bool last = step + 2 == R;
        const uint32_t k_next = k ? k - 1 : R - 1;
        uint4 b_next[U];
        if (!last) {  // own data of the next step: travels while this step's partial sums do
#pragma unroll
          for (uint32_t i = 0; i < U; ++i)
            if (live(i)) b_next[i] = ld16(static_cast<const char*>(P.in[r]) + part_off(k_next, i));
        }
#pragma unroll
        for (uint32_t i = 0; i < U; ++i) {
          if (!live(i)) continue;
          const uint32_t at = (tid + i * nthr) * 16u;
          Acc<DT> acc;
          acc.zero();
          if constexpr (DT == PL_BF16) {
            if (step == 0) acc.add_bf16(a[i]);
            else acc.add_f32(lds16(base + buffer(step) + at), lds16(base + buffer(step) + plane + at));
            acc.add_bf16(b[i]);
          } else if constexpr (DT == PL_F32) {
            if (step == 0) acc.add(a[i]);
            else acc.add_pair(lds16(base + buffer(step) + at), lds16(base + buffer(step) + plane + at));
            acc.add(b[i]);
          } else {
            acc.add(step == 0 ? a[i] : lds16(base + buffer(step) + at));
            acc.add(b[i]);
          }
          const uint32_t to = next + buffer(step + 1) + at;
          if (!last) {
            if constexpr (DT == PL_BF16) {
              st_cluster16(to, make_uint4(__float_as_uint(acc.v[0]), __float_as_uint(acc.v[1]), __float_as_uint(acc.v[2]), __float_as_uint(acc.v[3])));
              st_cluster16(to + plane, make_uint4(__float_as_uint(acc.v[4]), __float_as_uint(acc.v[5]), __float_as_uint(acc.v[6]), __float_as_uint(acc.v[7])));
            } else if constexpr (DT == PL_F32) {
              st_cluster16(to, acc.sums());
              st_cluster16(to + plane, acc.corrections());
            } else {
              st_cluster16(to, acc.result());
            }
          } else {
            uint4 v;
            if constexpr (DT == PL_BF16) v = acc.to_bf16(P.out_scale);
            else v = acc.result(P.out_scale);
            st16(static_cast<char*>(P.out[r]) + part_off(P.gather ? r : 0u, i), v);
            if (P.gather) st_cluster16(to, v);
          }
        }
        if (last && !P.gather) break;
        cluster_arrive();
        k = k_next;
#pragma unroll
        for (uint32_t i = 0; i < U; ++i) b[i] = b_next[i];
        cluster_wait();
      }
    }
  }
  if (P.gather) {
    if (!P.reduce) {  // all-gather: a rank's own contribution starts on its way
#pragma unroll
      for (uint32_t i = 0; i < U; ++i) {
        if (!live(i)) continue;
        const uint4 v = ld16(static_cast<const char*>(P.in[r]) + part_off(0u, i));
        st16(static_cast<char*>(P.out[r]) + part_off(r, i), v);
        st_cluster16(next + buffer(step) + (tid + i * nthr) * 16u, v);
      }
      cluster_arrive();
      cluster_wait();
    }
    uint32_t k = q;  // partition that reaches rank r at the first gather step
    for (uint32_t j = 0; j + 1 < R; ++j, ++step) {
      const bool last = j + 2 == R;
#pragma unroll
      for (uint32_t i = 0; i < U; ++i) {
        if (!live(i)) continue;
        const uint32_t at = (tid + i * nthr) * 16u;
        const uint4 v = lds16(base + buffer(step) + at);
        if (!last) st_cluster16(next + buffer(step + 1) + at, v);
        st16(static_cast<char*>(P.out[r]) + part_off(k, i), v);
      }
      if (last) break;
      k = k ? k - 1 : R - 1;
      cluster_arrive();
      cluster_wait();
    }
  }
}

void configure(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int R, const RingLaunch& L) {
  cfg.gridDim = dim3((unsigned)L.grid);
  cfg.blockDim = dim3((unsigned)L.threads);
  cfg.dynamicSmemBytes = L.smem_bytes;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)R;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

template <int DT, int U>
cudaError_t launch_t(const RingHopParams& P, const RingLaunch& L, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  configure(cfg, attr, P.n_ranks, L);
  cfg.stream = stream;
  return cudaLaunchKernelEx(&cfg, pl_ring_kernel<DT, U>, P);
}

// Raises the limits the launch needs on the current device; clusters that can be resident at once.
template <int DT, int U>
int prepare_t(int R, const RingLaunch& L) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  configure(cfg, attr, R, L);
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(pl_ring_kernel<DT, U>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * kRingThreads * 64) != cudaSuccess ||
      (R > 8 && cudaFuncSetAttribute(pl_ring_kernel<DT, U>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
      cudaOccupancyMaxActiveClusters(&n, pl_ring_kernel<DT, U>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

template <typename F>
auto pick(int dtype, int units, F f) {
  auto by_units = [&](auto dt) {
    if (units == 1) return f(dt, std::integral_constant<int, 1>{});
    return f(dt, std::integral_constant<int, 4>{});
  };
  switch (dtype) {
    case PL_BF16: return by_units(std::integral_constant<int, PL_BF16>{});
    case PL_F32: return by_units(std::integral_constant<int, PL_F32>{});
    case PL_I32: return by_units(std::integral_constant<int, PL_I32>{});
    // bytes are only gathered, in tiles of one unit per thread (ring_shape() gives four to two ranks and 256 threads,
    // which an all-gather of two ranks is too small for)
    default: return f(std::integral_constant<int, PL_U8>{}, std::integral_constant<int, 1>{});
  }
}

}  // namespace

int ring_prepare(int dtype, int R, const RingLaunch& L) {
  return pick(dtype, L.units, [&](auto dt, auto u) { return prepare_t<dt(), u()>(R, L); });
}

cudaError_t launch_ring(int dtype, const RingHopParams& P, const RingLaunch& L, cudaStream_t stream) {
  return pick(dtype, L.units, [&](auto dt, auto u) { return launch_t<dt(), u()>(P, L, stream); });
}

}  // namespace pl
