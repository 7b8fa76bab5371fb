// Datapath for layered direct-fused all-reduces (the decode shape: L small all-reduces in one
// launch) whose grid is left to the library.
//
// Such a schedule is regular: every queue holds exactly one op per layer, the ops of layer l
// read and write the same slice of every rank's buffers l messages further on, and every op of
// layer l + 1 waits for every op of layer l.  The register executor runs it too, but pays on
// every layer for being able to run anything: descriptors through shared memory, 512 threads at
// two CTA barriers whatever the slice needs, input lines that come from DRAM only after the flag.
// A layer is a serial chain (flag seen -> inputs -> sum -> outputs acknowledged -> flag), so what
// counts is what sits on that chain:
//   - a CTA has as many threads as its slice has 16-byte units (32 at the small end), one unit per
//     thread, addresses from the kernel parameters;
//   - the lines of a later layer's inputs are asked into L2 while the flag of this layer travels
//     (a prefetch is not a read: the values are loaded after the flag, from the point of
//     coherence);
//   - CLUSTER: when the whole schedule fits 16 CTAs, they form one thread-block cluster and the
//     flag is the cluster barrier (release / acquire): one hop instead of an increment in L2 and a
//     poll that has to see it.
// What bounds it: at the small end the chain (outputs acknowledged by L2 about 0.6 us, barrier 0.1 or
// flag 0.6 us, inputs from L2 0.3 us), at 1 MiB the chain plus 16 MiB of L2 traffic per layer
// (2.6 us at DRAM rate, which the prefetch and the write-back overlap with the chain).
// Measured on B200, R = 8, bf16, 80 layers in one launch, three sets of buffers in turn, us per
// layer, register executor -> this kernel: 4 KiB 2.0 -> 1.01, 16 KiB 2.16 -> 1.12, 32 KiB 1.41 (cluster); 64 KiB 3.20 -> 1.74,
// 128 KiB 3.28 -> 1.78, 512 KiB 3.86 -> 2.49, 1 MiB 5.00 -> 3.46 (flags).  Clock stamps of a 16 KiB layer, cycles: loads
// issued 66, arrived 445, summed and stored 290, acknowledged (release) 1160, barrier 200.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "pl_device.cuh"
#include "pl_internal.h"
#include "pl_kernels.h"

namespace pl {
namespace {

using namespace dev;

constexpr int kMaxThreads = kLayerThreads, kMaxClusterThreads = kLayerClusterThreads;  // threads that move data; CLUSTER adds one warp that asks for lines ahead

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// One unit (16 bytes of every source) of a layer: NR bounds the ranks, all loads before the adds.
// EXACT: there are NR ranks, so the loads and stores follow one another without a test of the rank between them, which
// costs a load 37 cycles (8 ranks, 16 KiB: the loads are issued in 66 cycles instead of 299).  The compiler may
// then spread them over the additions, which waits for memory several times over (8 x 64 KiB 146 -> 212 us for 80
// layers): one word of each goes through a shuffle to its own lane, and every lane of the warp waits there for all.
// So all 32 lanes come here, and one with nothing to do (`live` false) loads what another loads and stores nothing.
template <int DT, int NR, bool HOOK, bool EXACT>
__device__ __forceinline__ void layer_unit(const ExecParams& P, uint64_t in_off, uint64_t out_off, bool live) {
  const int R = EXACT ? NR : P.n_ranks;
  uint4 q[NR];
#pragma unroll
  for (int s = 0; s < NR; ++s)
    if (s < R) q[s] = ld16(static_cast<const char*>(P.base[kSlotIn + s]) + in_off);
  if constexpr (EXACT) {
#pragma unroll
    for (int s = 0; s < NR; ++s) q[s].w = __shfl_sync(0xFFFFFFFFu, q[s].w, (int)(threadIdx.x & 31u));
    if (!live) return;
  }
  uint4 second[HOOK ? NR : 1];
  if constexpr (HOOK) {
    if (P.hook & PL_HOOK_RESIDUAL) {
#pragma unroll
      for (int s = 0; s < NR; ++s)
        if (s < R) second[s] = ld16(static_cast<const char*>(P.base[kSlotAux + s]) + in_off);
    }
  }
  Acc<DT> acc;
  acc.zero();
#pragma unroll
  for (int s = 0; s < NR; ++s)
    if (s < R) {
      if constexpr (DT == PL_BF16) acc.add_bf16(q[s]);
      else acc.add(q[s]);
    }
  if constexpr (HOOK) {
#pragma unroll
    for (int k = 0; k < NR; ++k)
      if (k < R) store_final_q<DT>(acc, P.out_scale, P.hook, static_cast<char*>(P.base[kSlotOut + k]) + out_off, second[k]);
  } else {
    uint4 r;
    if constexpr (DT == PL_BF16) r = acc.to_bf16(P.out_scale);
    else r = acc.result(P.out_scale);
#pragma unroll
    for (int k = 0; k < NR; ++k)
      if (k < R) st16(static_cast<char*>(P.base[kSlotOut + k]) + out_off, r);
  }
}

// The units of one layer that fall to this thread, `n` apart: one as a rule.
template <int DT, int NR, bool HOOK, bool EXACT>
__device__ __forceinline__ void layer_slice(const ExecParams& P, uint64_t in_off, uint64_t out_off, uint32_t out_unit, uint32_t units, uint32_t t, uint32_t n) {
#pragma unroll 1
  for (uint32_t u = t; EXACT ? (u & ~31u) < units : u < units; u += n) {  // EXACT: the same number of turns for a whole warp
    const uint32_t at = EXACT ? min(u, units - 1u) : u;
    layer_unit<DT, NR, HOOK, EXACT>(P, in_off + at * 16ull, out_off + (uint64_t)at * out_unit, u < units);
  }
}

// Lines of one layer's operands for this CTA's slice into L2: line j of rank s by the thread with
// number j * NR + s modulo n.  The slice starts on a 16-byte boundary, so it can touch one line
// more than its bytes fill; that one is left to the load.
// ROLLED: one turn after another.  The shorter code is ahead (8 x 4 KiB 42.2 -> 40.7 us for 40 layers, 2 x 128 KiB 62.9 -> 55.5), but not with a
// residual of up to four ranks, which asks for twice the lines (2 x 64 KiB 48.5, rolled 56.1 us, 4 x 512 KiB 93.6 / 99.2; 8 x 32 KiB 82.1 / 77.8).
template <int NR, bool ROLLED>
__device__ __forceinline__ void ask_for_layer(const ExecParams& P, uint64_t in_off, uint32_t units, uint32_t t, uint32_t n) {
  const uint32_t lines = (units + 7u) >> 3;
  const bool residual = P.hook & PL_HOOK_RESIDUAL;
  auto ask = [&](uint32_t j) {
    const uint32_t line = j / NR, s = j % NR;
    if (s >= (uint32_t)P.n_ranks) return;
    const uint64_t off = in_off + (uint64_t)line * 128u;
    prefetch_l2(static_cast<const char*>(P.base[kSlotIn + s]) + off);
    if (residual) prefetch_l2(static_cast<const char*>(P.base[kSlotAux + s]) + off);
  };
  if constexpr (ROLLED) {
#pragma unroll 1
    for (uint32_t j = t; j < lines * NR; j += n) ask(j);
  } else {
    for (uint32_t j = t; j < lines * NR; j += n) ask(j);
  }
}

// FULL: with the stamps of a trace and the hook that breaks a wait.  They are a kernel of their own because the code in
// the loop costs a layer time even if it is not run (80 layers of 4 KiB 86 -> 81 us without it).
template <int DT, int NR, bool HOOK, bool CLUSTER, bool EXACT, bool FULL>
__global__ void __launch_bounds__(CLUSTER ? kMaxClusterThreads + 32 : kMaxThreads) pl_layers_kernel(const __grid_constant__ ExecParams P,
                                                                                  const __grid_constant__ LayerParams Y) {
  __shared__ int s_abort;
  const uint32_t tid = threadIdx.x, q = blockIdx.x, nq = P.n_queues;
  pdl_launch_dependents();
  // descriptors are immutable: read before the wait for the launch in front
  const DevOp* const op0 = P.ops + q;
  const uint64_t in_off0 = P.srcs[(uint64_t)q * P.src_stride] & 0xFFFFFFFFFFFFull;  // the same in every rank's input
  const uint64_t out_off0 = op0->dst & 0xFFFFFFFFFFFFull;
  const uint32_t units = (uint32_t)(op0->count / Acc<DT>::kElems);
  const uint32_t out_unit = (HOOK && DT == PL_BF16 && (P.hook & PL_HOOK_F32_OUT)) ? 32u : 16u;
  if (tid == 0) s_abort = 0;
  uint32_t topo = op0->topo;
  pdl_wait();

  if constexpr (CLUSTER) {
    const uint32_t movers = blockDim.x - 32u;
    for (uint32_t l = 0; l < Y.n_layers; ++l) {
      if (FULL && (int)l == Y.break_layer) {
        // test hook: a wait that nothing satisfies.  Every CTA leaves here; the one whose op was
        // broken gives up after the time limit and says so.
        if ((int)q == Y.break_queue && tid == 0) {
          const unsigned long long t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 <= P.timeout_ns) {}
          record_timeout(P, (int)q, topo, op0->signal + l - 1u, nq, 0);
        }
        break;
      }
      const uint64_t in_off = in_off0 + l * Y.in_stride, out_off = out_off0 + l * Y.out_stride;
      if (FULL && P.trace && tid == 0) P.trace[2ull * topo] = globaltimer_ns();
      if (tid < movers) {
        layer_slice<DT, NR, HOOK, EXACT>(P, in_off, out_off, out_unit, units, tid, movers);
      } else if (l + 1 < Y.n_layers) {
        ask_for_layer<NR, !HOOK || (NR > 4)>(P, in_off + Y.in_stride, units, tid - movers, 32u);
      }
      if (l + 1 < Y.n_layers) {
        if (FULL && P.trace) {
          __syncthreads();
          if (tid == 0) P.trace[2ull * topo + 1] = globaltimer_ns();
        }
        __syncwarp();
        cluster_arrive_release();
        cluster_wait_acquire();
      } else if (FULL && P.trace) {
        __syncthreads();
        if (tid == 0) P.trace[2ull * topo + 1] = globaltimer_ns();
      }
      topo += nq;
    }
  } else {
    const unsigned long long epoch = *reinterpret_cast<volatile unsigned long long*>(P.epoch) + 1ull;
    bool aborted = false;
    unsigned long long* flag = P.flags + op0->signal;  // this layer's; the next layer's is the next word
    for (uint32_t l = 0; l < Y.n_layers; ++l) {
      if (l > 0) {
        if (tid == 0) {
          // every CTA signals once per layer; acquire, bounded by the time limit
          const unsigned long long need = epoch * (gridDim.x + ((FULL && (int)l == Y.break_layer && (int)q == Y.break_queue) ? 1ull : 0ull));
          unsigned long long seen = ld_acquire_u64(flag);
          if (seen < need) {
            const unsigned long long t0 = globaltimer_ns();
            uint32_t spins = 0;
            while ((seen = ld_acquire_u64(flag)) < need) {
              if ((++spins & 63u) == 0) {
                if (ld_volatile_s32(P.status + 8)) { s_abort = 1; break; }
                if (globaltimer_ns() - t0 > P.timeout_ns) {
                  record_timeout(P, (int)q, topo, (uint32_t)(flag - P.flags), need, seen);
                  s_abort = 1;
                  break;
                }
              }
            }
          }
        }
        ++flag;
        __syncthreads();
        if (s_abort) { aborted = true; break; }
      }
      const uint64_t in_off = in_off0 + l * Y.in_stride, out_off = out_off0 + l * Y.out_stride;
      if (FULL && P.trace && tid == 0) P.trace[2ull * topo] = globaltimer_ns();
      layer_slice<DT, NR, HOOK, EXACT>(P, in_off, out_off, out_unit, units, tid, blockDim.x);
      if (l + 1 < Y.n_layers || (FULL && P.trace)) {
        __syncthreads();  // every thread's writes are done
        if (tid == 0) {
          if (FULL && P.trace) P.trace[2ull * topo + 1] = globaltimer_ns();
          // cumulative: covers the other threads' stores, observed through the barrier
          if (l + 1 < Y.n_layers) red_release_add_u64(flag, 1ull);
        }
      }
      if (l + 1 < Y.n_layers) {
        topo += nq;
        // while the flag travels (asking two layers ahead measured the same)
        if (Y.ask_ahead) ask_for_layer<NR, !HOOK || (NR > 4)>(P, in_off + Y.in_stride, units, tid, blockDim.x);
      }
    }
    __syncthreads();
    if (tid == 0 && !aborted) {
      // last CTA to finish advances the epoch for the next execute
      const unsigned long long prev = atomicAdd(P.epoch + 1, 1ull);
      if (prev == (unsigned long long)gridDim.x - 1ull) {
        P.epoch[1] = 0ull;
        __threadfence();
        *reinterpret_cast<volatile unsigned long long*>(P.epoch) = epoch;
      }
    }
  }
}

void configure(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int grid, int threads, bool cluster, bool overlap) {
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)(threads + (cluster ? 32 : 0)));
  int na = 0;
  if (cluster) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)grid;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  if (overlap) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
}

using LayerKernel = void (*)(ExecParams, LayerParams);

// The kernel of a launch: a processing phase has one form, with everything in it, and so have traces and broken waits.
template <int DT, int NR, bool HOOK, bool CLUSTER>
LayerKernel kernel_t(int R, bool full) {
  if constexpr (HOOK) return pl_layers_kernel<DT, NR, true, CLUSTER, false, true>;
  else if (full) return pl_layers_kernel<DT, NR, false, CLUSTER, false, true>;
  else {
    auto exact = [](auto n) -> LayerKernel { return pl_layers_kernel<DT, n(), false, CLUSTER, true, false>; };
    switch (R) {
      case 2: return exact(std::integral_constant<int, 2>{});
      case 3: return exact(std::integral_constant<int, 3>{});
      case 4: return exact(std::integral_constant<int, 4>{});
      case 5: return exact(std::integral_constant<int, 5>{});
      case 6: return exact(std::integral_constant<int, 6>{});
      case 7: return exact(std::integral_constant<int, 7>{});
      case 8: return exact(std::integral_constant<int, 8>{});
      case 12: return exact(std::integral_constant<int, 12>{});
      case 16: return exact(std::integral_constant<int, 16>{});
      default: return pl_layers_kernel<DT, PL_MAX_RANKS, false, CLUSTER, false, false>;  // 9 to 15 but for 12
    }
  }
}

// Up to 16 CTAs: more than the portable 8 needs the opt-in (a per-device attribute of the function, raised here, when
// the schedule is built, and kept).
bool cluster_fits(LayerKernel kernel, int grid, int threads) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  int n = 0;
  configure(cfg, attr, grid, threads, true, false);
  const void* f = reinterpret_cast<const void*>(kernel);
  if ((grid > 8 && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) ||
      cudaOccupancyMaxActiveClusters(&n, f, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= 1;
}

// f(dtype, rank bound, hook) over the instantiations; int32 has no hooks.
template <typename F>
auto pick(int dtype, int R, bool hook, F f) {
  auto ranks = [&](auto dt, auto hk) {
    if (R <= 4) return f(dt, std::integral_constant<int, 4>{}, hk);
    if (R <= 8) return f(dt, std::integral_constant<int, 8>{}, hk);
    return f(dt, std::integral_constant<int, PL_MAX_RANKS>{}, hk);
  };
  if (dtype == PL_BF16) return hook ? ranks(std::integral_constant<int, PL_BF16>{}, std::true_type{}) : ranks(std::integral_constant<int, PL_BF16>{}, std::false_type{});
  if (dtype == PL_F32) return hook ? ranks(std::integral_constant<int, PL_F32>{}, std::true_type{}) : ranks(std::integral_constant<int, PL_F32>{}, std::false_type{});
  return ranks(std::integral_constant<int, PL_I32>{}, std::false_type{});
}

}  // namespace

cudaError_t launch_layers(int dtype, const ExecParams& P, const LayerParams& Y, int grid, int threads, bool cluster, cudaStream_t stream) {
  if (dtype == PL_U8 || (dtype == PL_I32 && P.hook)) return cudaErrorInvalidValue;
  const bool full = P.trace || Y.break_layer >= 0;
  const LayerKernel kernel = pick(dtype, P.n_ranks, P.hook != 0, [&](auto dt, auto nr, auto hk) {
    return cluster ? kernel_t<dt(), nr(), hk(), true>(P.n_ranks, full) : kernel_t<dt(), nr(), hk(), false>(P.n_ranks, full);
  });
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  configure(cfg, attr, grid, threads, cluster, P.overlap_launch);
  cfg.stream = stream;
  return cudaLaunchKernelEx(&cfg, kernel, P, Y);
}

// Both kernels that a schedule may launch: the hook that breaks a wait can be set after the build.
bool layers_cluster_fits(int dtype, int R, bool hook, int grid, int threads) {
  return pick(dtype, R, hook, [&](auto dt, auto nr, auto hk) {
    return cluster_fits(kernel_t<dt(), nr(), hk(), true>(R, false), grid, threads) && cluster_fits(kernel_t<dt(), nr(), hk(), true>(R, true), grid, threads);
  });
}

}  // namespace pl
