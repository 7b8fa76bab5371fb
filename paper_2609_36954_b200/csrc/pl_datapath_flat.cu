// Datapath for schedules without flags whose grid is left to the library: no op waits for another,
// so nothing has to be resident together and no CTA needs a queue.  The ops are laid end to end
// as spans (runs of consecutive bytes with the same sources and destinations, see flat_plan()), the
// spans are cut into tiles of a few KiB per operand, and every tile is a CTA of its own.
//
// What bounds it is HBM, and what this form gains over a persistent CTA per queue is the order in
// which HBM is touched: the hardware hands out the next tile whenever a CTA retires, so all SMs
// work inside one narrow window that sweeps through every operand, and no SM has a queue left
// over at the end.  Queues of a persistent grid drift apart (equal work, unequal service) and touch
// 144 windows at once.  B200, R = 8, bf16, back to back over three sets of buffers, queue executor
// -> this: reduce-scatter + all-gather 64 MiB per rank 189 -> 175 us, fused all-reduce 256 MiB
// 657 -> 631 us, 16 MiB 50.9 -> 42.1 us, 4 MiB 15.6 -> 11.9 us, 16 MiB with residual 82.6 -> 60.6 us,
// 4 MiB with residual 34.8 -> 18.0 us, all-to-all-v of 24 MiB 67.5 -> 61.0 us.
//
// A reducing ring comes here too, folded: the hops of a unit are a chain of additions in ring order, which one
// thread makes with the same rounding (its span names the rank to start with).  A ring's bytes are mostly partial
// sums in a wider type than the data; folded it reads inputs and writes outputs, like a direct reduction.  Through
// neighbours' shared memory -> folded: reduce-scatter 8 x 64 MiB bf16 237 -> 87 us, fp32 277 -> 90, all-reduce
// 8 x 64 MiB bf16 392 -> 160, 4 x 1 MiB fp32 7.55 -> 2.6, 8 x 64 KiB bf16 9.3 -> 2.7, 16 x 48 MiB fp32 814 -> 242.
//
// Two forms, by the schedule's datapath:
//   register   the working set sits in L2 or nearly: one unit (16 bytes per operand) or a few per
//              thread, all loads of a thread before its first add or store;
//   bulk copy  streaming from HBM: one bulk asynchronous load per operand and tile into shared
//              memory; reduce ops add from there and store from registers, copies leave by bulk
//              stores.  Several CTAs per SM take the place of a ring of slots.
// Bulk copies store evict-first, which keeps in L2 what the next launch reads of a stream's inputs.  The
// register form stores plainly: its results fit L2, and whoever reads them next finds them there (8 x 8 MiB
// all-gather and a reader of the results 44.9 us evict-first, 39.7 plain; 8 x 4 MiB 28.7 / 25.4; back to back without a
// reader evict-first is ahead, 12.5 / 13.0 and 6.6 / 7.3).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include "pl_device.cuh"
#include "pl_internal.h"
#include "pl_kernels.h"
#include "pl_ptx.cuh"

namespace pl {
namespace {

using namespace dev;

struct Tile {
  FlatSpan span;
  uint64_t first;  // first unit of the tile inside the span
  uint32_t units;
};

// The tile of this CTA.  A run is worked out from the parameters: nothing is uploaded, and no load stands in front of a
// tile's own.  The span is the second dimension of the grid (dealt in the same order; found by a division it cost more than the
// load: one-shot 6 x 2 MiB bf16 7.73 us, 8.06 by division, 8.53 from memory; reduce-scatter 8 x 1 MiB 1.74, 1.88, 2.01).
// Else every warp finds the span whose blocks contain it (lane i looks at spans i, i + 32, ...); spans are written
// when the schedule is built, so this may run ahead of the wait for the launch in front.
__device__ __forceinline__ Tile my_tile(const FlatParams& P) {
  const uint32_t b = blockIdx.x, lane = threadIdx.x & 31u;
  if (!P.spans) {
    const uint32_t k = blockIdx.y;
    Tile t;
    t.span.src_off = k * P.run.src_step;
    t.span.dst_off = k * P.run.dst_step;
    t.span.units = P.run.units;
    t.span.first_block = 0;
    t.span.ranks = P.run.ranks + k * P.run.rank_step;
    t.first = (uint64_t)b * P.tile;
    t.units = (uint32_t)min((uint64_t)P.tile, t.span.units - t.first);
    return t;
  }
  uint32_t k = 0;
  if (P.n_spans > 1) {
    uint32_t below = 0;  // spans that start at or before this block
    for (uint32_t i = 0; i < P.n_spans; i += 32)
      below += __popc(__ballot_sync(0xFFFFFFFFu, i + lane < P.n_spans && __ldg(&P.spans[i + lane].first_block) <= b));
    k = below - 1u;
  }
  Tile t;
  const uint4* s = reinterpret_cast<const uint4*>(P.spans + k);
  const uint4 lo = __ldg(s), hi = __ldg(s + 1);
  t.span.src_off = ((uint64_t)lo.y << 32) | lo.x;
  t.span.dst_off = ((uint64_t)lo.w << 32) | lo.z;
  t.span.units = ((uint64_t)hi.y << 32) | hi.x;
  t.span.first_block = hi.z;
  t.span.ranks = hi.w;
  t.first = (uint64_t)(b - t.span.first_block) * P.tile;
  t.units = (uint32_t)min((uint64_t)P.tile, t.span.units - t.first);
  return t;
}
__device__ __forceinline__ uint32_t src_rank(const FlatSpan& s) { return s.ranks & 0xFFu; }
__device__ __forceinline__ uint32_t dst_rank(const FlatSpan& s) { return (s.ranks >> 8) & 0xFFu; }
__device__ __forceinline__ uint32_t first_rank(const FlatSpan& s) { return s.ranks >> 16; }

__device__ __forceinline__ uint4 ld16_hint(const void* p, uint64_t policy) {
  uint4 v;
  asm volatile("ld.global.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
  return v;
}
template <int DT>
__device__ __forceinline__ void add_unit(Acc<DT>& acc, const uint4& q) {
  if constexpr (DT == PL_BF16) acc.add_bf16(q);
  else acc.add(q);
}

// Sum of one unit to one destination, as every executor finishes a reduce op.  `second`: the unit
// of the destination's second operand (HOOK).
template <int DT, bool HOOK>
__device__ __forceinline__ void store_sum(const FlatParams& P, const Acc<DT>& acc, void* dst, const uint4& second) {
  if constexpr (HOOK) {
    store_final_q<DT>(acc, P.out_scale, P.hook, static_cast<char*>(dst), second);
  } else {
    uint4 r;
    if constexpr (DT == PL_BF16) r = acc.to_bf16(P.out_scale);
    else r = acc.result(P.out_scale);
    st16(dst, r);
  }
}

// ---- register form ---------------------------------------------------------------------------
// Which launches release the one behind them at their start is flat_release()'s.
// Units per thread of a reduce: about 8 operand vectors in flight (16 with a second operand per rank).
template <int NR, bool HOOK>
struct FlatUnits {
  static constexpr int value = HOOK ? (NR <= 2 ? 2 : 1) : (NR <= 2 ? 4 : NR <= 4 ? 2 : 1);
};

// NR bounds the ranks, so that the register of every operand is a compile-time constant.  EXACT: there are NR ranks, and
// the loads follow one another without a test between them; a word of each source goes through a shuffle to its own
// lane, where the warp waits for all of them (see layer_unit() in pl_datapath_layers.cu).  A unit past the end of the
// tile is then loaded from its last one and not stored.  With a processing phase that is faster at every size (residual,
// bf16, us: 4 x 4 MiB 9.5 -> 8.9, 8 x 1.6 MiB 9.3 -> 9.0, 8 x 4 MiB 18.1 -> 17.2, 16 x 4 MiB 33.6 -> 31.9; fp32 8 x 2 MiB 11.1 -> 10.2);
// without one the bursts are slower where inputs and outputs take 20 to 40 MB of L2 (8 x 2 MiB 6.4 / 8.2, 16 x 1 MiB
// 6.9 / 8.3, while 16 x 2 MiB 13.0 / 12.2; measured with the launch behind released early), so it goes with HOOK.
// FOLDED: the sum starts with a rank that the span names, so the pointer of every load is looked up at run time.  Where it is not,
// the pointers are constants (looked up in every sum: one-shot 6 x 8 MiB bf16 33.8 -> 35.8 us, fp32 43.7 -> 46.5, reduce-scatter 2 x 8 MiB
// with residual 5.0 -> 5.9).
// HINT: the loads carry the evict-first hint.  Known when compiled, but for sums of more than 8 ranks to one rank, which test for it in
// front of every load: that keeps the loads of up to 16 sources in front of the first addition (us, so / as an argument /
// one test for all loads: one-shot 12 x 2 MiB int32 24.0 / 30.8 / 34.2, 16 x 2 MiB bf16 49.2 / 51.3 / 52.9, reduce-scatter 12 x 1 MiB bf16 2.01 / 2.36
// / 2.50, though 16 x 4 MiB 13.8 / 13.0 / 12.9; up to 8 ranks: one-shot 8 x 2 MiB bf16 12.1 / 11.6 / 12.0, reduce-scatter 8 x 4 MiB
// fp32 8.3 / 7.1 / 7.1, and to every rank 16 x 2 MiB 15.1 / 13.4 / 13.3, 12 x 4 KiB 2.35 / 2.51 / 2.60).
template <int DT, int NR, bool HOOK, bool ALL, bool EXACT, bool FOLDED, bool HINT>
__global__ void __launch_bounds__(kFlatThreads, 2) pl_flat_reduce_kernel(const __grid_constant__ FlatParams P) {
  constexpr int U = FlatUnits<NR, HOOK>::value;
  if (P.release) pdl_launch_dependents();
  const Tile t = my_tile(P);
  const uint32_t R = EXACT ? (uint32_t)NR : (uint32_t)P.n_ranks, to = dst_rank(t.span);
  const bool residual = HOOK && (P.hook & PL_HOOK_RESIDUAL);
  const uint32_t out_b = (HOOK && DT == PL_BF16 && (P.hook & PL_HOOK_F32_OUT)) ? 32u : 16u;
  constexpr bool kTested = NR > 8 && !ALL && !EXACT;
  const bool hint = kTested ? (P.hints & 1u) != 0 : HINT;
  const uint64_t policy = hint ? ptx::policy_evict_first() : 0ull;
  pdl_wait();
  uint64_t in_off[U], at[U];  // byte offset of the unit in every source, unit index in the destination
  bool live[U];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    uint32_t u = threadIdx.x + (uint32_t)(j * kFlatThreads);
    live[j] = u < t.units;
    if (EXACT) u = min(u, t.units - 1u);
    at[j] = t.span.dst_off + t.first + u;
    in_off[j] = (t.span.src_off + t.first + u) * 16ull;
  }
  uint4 q[U][NR];
  const uint32_t first = FOLDED ? first_rank(t.span) : 0u;
  auto load = [&](auto ld) {
#pragma unroll
    for (int j = 0; j < U; ++j)
#pragma unroll
      for (int s = 0; s < NR; ++s)
        if (EXACT || (live[j] && s < (int)R)) {
          const uint32_t rank = !FOLDED ? (uint32_t)s : first + s < R ? first + s : first + s - R;
          q[j][s] = ld(static_cast<const char*>(P.in[rank]) + in_off[j]);
        }
  };
  if constexpr (kTested) load([&](const char* src) { return hint ? ld16_hint(src, policy) : ld16(src); });
  else if (hint) load([&](const char* src) { return ld16_hint(src, policy); });
  else load([](const char* src) { return ld16(src); });
  // second operands: of 8 ranks at a time when the results go to every rank (16 of them and 16
  // sources would not fit the registers), else the one of the destination
  constexpr int NS = !HOOK ? 1 : !ALL ? 1 : NR < 8 ? NR : 8;
  uint4 second[U][NS];
  if (residual) {
#pragma unroll
    for (int j = 0; j < U; ++j)
#pragma unroll
      for (int k = 0; k < NS; ++k)
        if (EXACT || (live[j] && (!ALL || k < (int)R))) second[j][k] = ld16(static_cast<const char*>(P.aux[ALL ? k : (int)to]) + at[j] * 16ull);
  }
  if constexpr (EXACT) {
    const int lane = (int)(threadIdx.x & 31u);
#pragma unroll
    for (int j = 0; j < U; ++j) {
#pragma unroll
      for (int s = 0; s < NR; ++s) q[j][s].w = __shfl_sync(0xFFFFFFFFu, q[j][s].w, lane);
    }
  }
#pragma unroll
  for (int j = 0; j < U; ++j) {
    if (!live[j]) continue;
    Acc<DT> acc;
    acc.zero();
#pragma unroll
    for (int s = 0; s < NR; ++s)
      if (s < (int)R) add_unit<DT>(acc, q[j][s]);
    if constexpr (!ALL) {
      store_sum<DT, HOOK>(P, acc, static_cast<char*>(P.out[to]) + at[j] * out_b, second[j][0]);
    } else {
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        if (k >= (int)R) continue;
        if constexpr (HOOK && NR > 8) {
          if (residual && k == 8) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if (8 + i < (int)R) second[j][i] = ld16(static_cast<const char*>(P.aux[8 + i]) + at[j] * 16ull);
          }
        }
        store_sum<DT, HOOK>(P, acc, static_cast<char*>(P.out[k]) + at[j] * out_b, second[j][HOOK ? k % NS : 0]);
      }
    }
  }
}

template <int U, bool ALL>
__global__ void __launch_bounds__(kFlatThreads) pl_flat_copy_kernel(const __grid_constant__ FlatParams P) {
  if (P.release) pdl_launch_dependents();
  const Tile t = my_tile(P);
  const uint64_t policy = (P.hints & 1u) ? ptx::policy_evict_first() : 0ull;
  pdl_wait();
  const char* src = static_cast<const char*>(P.in[src_rank(t.span)]) + (t.span.src_off + t.first) * 16ull;
  const uint64_t at = (t.span.dst_off + t.first) * 16ull;
  uint4 q[U];
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const uint32_t u = threadIdx.x + (uint32_t)(j * kFlatThreads);
    if (u < t.units) q[j] = (P.hints & 1u) ? ld16_hint(src + u * 16ull, policy) : ld16(src + u * 16ull);
  }
  auto put = [&](uint32_t r) {
    char* dst = static_cast<char*>(P.out[r]) + at;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const uint32_t u = threadIdx.x + (uint32_t)(j * kFlatThreads);
      if (u < t.units) st16(dst + u * 16ull, q[j]);
    }
  };
  if constexpr (ALL) {
    for (int r = 0; r < P.n_ranks; ++r) put((uint32_t)r);
  } else {
    put(dst_rank(t.span));
  }
}

// ---- bulk-copy form --------------------------------------------------------------------------
constexpr int kBarBytes = 128;  // the mbarrier, ahead of the tiles

// Bounded wait for the tile's loads.  On expiry the status is recorded and the loads get a last
// bounded chance to land, so that none is in flight when the CTA leaves.
__device__ __forceinline__ bool wait_tile(const FlatParams& P, uint64_t* bar) {
  if (ptx::mbar_try_wait(bar, 0)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (uint32_t spins = 1;; ++spins) {
    if (ptx::mbar_try_wait(bar, 0)) return true;
    if ((spins & 255u) == 0 && globaltimer_ns() - t0 > 2ull * P.timeout_ns + 1000000ull) {
      record_timeout_at(P.status, (int)blockIdx.x, 0xFFFFFFFFu, 0xFFFFFFFFu, 0, 0);
      ptx::mbar_wait_bounded(bar, 0, 1u << 20);
      return false;
    }
  }
}

template <int DT, bool HOOK, bool ALL>
__global__ void __launch_bounds__(kFlatBulkThreads) pl_flat_bulk_reduce_kernel(const __grid_constant__ FlatParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
  unsigned char* tiles = smem + kBarBytes;
  pdl_launch_dependents();
  const Tile t = my_tile(P);
  const uint32_t tid = threadIdx.x, R = (uint32_t)P.n_ranks, to = dst_rank(t.span);
  const bool residual = HOOK && (P.hook & PL_HOOK_RESIDUAL);
  const uint32_t n_aux = residual ? (ALL ? R : 1u) : 0u, stride = P.tile * 16u, bytes = t.units * 16u;
  const uint64_t at = t.span.dst_off + t.first;
  if (tid == 0) {
    ptx::mbar_init(bar, 1);
    ptx::mbar_init_fence();
  }
  pdl_wait();
  if (tid < 32) {
    if (tid == 0) ptx::mbar_expect_tx(bar, bytes * (R + n_aux));
    __syncwarp();
    if (tid < R + n_aux) {  // lane s: source s in order of addition; lane R + k: second operand of rank k (or of the destination)
      const uint32_t s = first_rank(t.span) + tid, rank = s < R ? s : s - R;
      const char* from = tid < R ? static_cast<const char*>(P.in[rank]) + (t.span.src_off + t.first) * 16ull
                                 : static_cast<const char*>(P.aux[ALL ? tid - R : to]) + at * 16ull;
      if ((P.hints & 1u) && tid < R) ptx::bulk_g2s_hint(tiles + tid * stride, from, bytes, bar, ptx::policy_evict_first());
      else ptx::bulk_g2s(tiles + tid * stride, from, bytes, bar);
    }
  }
  __syncthreads();  // the barrier is initialised before the other warps look at it
  if (!wait_tile(P, bar)) return;
  const uint32_t out_b = (HOOK && DT == PL_BF16 && (P.hook & PL_HOOK_F32_OUT)) ? 32u : 16u;
  for (uint32_t u = tid; u < t.units; u += kFlatBulkThreads) {
    const unsigned char* p = tiles + u * 16u;
    Acc<DT> acc;
    acc.zero();
    uint32_t s = 0;
    for (; s + 4 <= R; s += 4, p += 4 * stride) {
      const uint4 a = *reinterpret_cast<const uint4*>(p), b = *reinterpret_cast<const uint4*>(p + stride);
      const uint4 c = *reinterpret_cast<const uint4*>(p + 2 * stride), d = *reinterpret_cast<const uint4*>(p + 3 * stride);
      add_unit<DT>(acc, a);
      add_unit<DT>(acc, b);
      add_unit<DT>(acc, c);
      add_unit<DT>(acc, d);
    }
    for (; s < R; ++s, p += stride) add_unit<DT>(acc, *reinterpret_cast<const uint4*>(p));
    uint4 second = make_uint4(0, 0, 0, 0);  // p stands at the first second operand
    if constexpr (!ALL) {
      if (residual) second = *reinterpret_cast<const uint4*>(p);
      store_sum<DT, HOOK>(P, acc, static_cast<char*>(P.out[to]) + (at + u) * out_b, second);
    } else {
#pragma unroll 4
      for (uint32_t k = 0; k < R; ++k) {
        if (residual) second = *reinterpret_cast<const uint4*>(p + k * stride);
        store_sum<DT, HOOK>(P, acc, static_cast<char*>(P.out[k]) + (at + u) * out_b, second);
      }
    }
  }
}

template <bool ALL>
__global__ void __launch_bounds__(32) pl_flat_bulk_copy_kernel(const __grid_constant__ FlatParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
  unsigned char* tile = smem + kBarBytes;
  pdl_launch_dependents();
  const Tile t = my_tile(P);
  const uint32_t lane = threadIdx.x, bytes = t.units * 16u;
  const uint64_t policy = ptx::policy_evict_first();
  if (lane == 0) {
    ptx::mbar_init(bar, 1);
    ptx::mbar_init_fence();
  }
  pdl_wait();
  if (lane == 0) {
    const char* from = static_cast<const char*>(P.in[src_rank(t.span)]) + (t.span.src_off + t.first) * 16ull;
    ptx::mbar_expect_tx(bar, bytes);
    if (P.hints & 1u) ptx::bulk_g2s_hint(tile, from, bytes, bar, policy);
    else ptx::bulk_g2s(tile, from, bytes, bar);
  }
  __syncwarp();
  if (!wait_tile(P, bar)) return;
  if (lane < (ALL ? (uint32_t)P.n_ranks : 1u)) {
    char* to = static_cast<char*>(P.out[ALL ? lane : dst_rank(t.span)]) + (t.span.dst_off + t.first) * 16ull;
    if (P.hints & 2u) ptx::bulk_s2g_hint(to, tile, bytes, policy);
    else ptx::bulk_s2g(to, tile, bytes);
    ptx::bulk_commit();
    ptx::bulk_wait<0>();
  }
}

template <void (*kernel)(const FlatParams)>
cudaError_t launch(const FlatParams& P, const FlatLaunch& F, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = P.spans ? dim3(F.blocks) : dim3(F.blocks / P.n_spans, P.n_spans);
  cfg.blockDim = dim3((unsigned)F.threads);
  cfg.dynamicSmemBytes = F.smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (F.smem_bytes > 48 * 1024) {
    // the opt-in is a per-device attribute of the function: one bit per device and instantiation
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured.load(std::memory_order_acquire) & bit)) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
      if (e != cudaSuccess) return e;
      configured.fetch_or(bit, std::memory_order_release);
    }
  }
  return cudaLaunchKernelEx(&cfg, kernel, P);
}

template <int DT, int NR, bool HOOK, bool EXACT, bool FOLDED = false>
cudaError_t launch_all(const FlatParams& P, const FlatLaunch& F, cudaStream_t stream) {
  auto by_hint = [&](auto all) {
    if constexpr (all() || NR <= 8 || EXACT) {
      if (P.hints & 1u) return launch<pl_flat_reduce_kernel<DT, NR, HOOK, all(), EXACT, FOLDED, true>>(P, F, stream);
    }
    return launch<pl_flat_reduce_kernel<DT, NR, HOOK, all(), EXACT, FOLDED, false>>(P, F, stream);
  };
  return F.all ? by_hint(std::true_type{}) : by_hint(std::false_type{});
}
template <int DT, int NR, bool HOOK>
cudaError_t launch_reduce(const FlatParams& P, const FlatLaunch& F, cudaStream_t stream) {
  if constexpr (HOOK) {  // EXACT for 2, 3, 4, 6, 8 and 16 ranks, the counts it was measured at; another takes the next bound's
    if constexpr (NR == 4) {
      if (P.n_ranks == 3) return launch_all<DT, 3, true, true>(P, F, stream);
    }
    if constexpr (NR == 8) {
      if (P.n_ranks == 6) return launch_all<DT, 6, true, true>(P, F, stream);
    }
    if (NR <= 4 || P.n_ranks == NR) return launch_all<DT, NR, true, true>(P, F, stream);
  } else if (F.folded) {
    return launch_all<DT, NR, false, false, true>(P, F, stream);
  }
  if constexpr (!HOOK || NR > 4) return launch_all<DT, NR, HOOK, false>(P, F, stream);
  else return cudaErrorInvalidValue;  // not reached
}
template <int DT, bool HOOK>
cudaError_t launch_dt(const FlatParams& P, const FlatLaunch& F, cudaStream_t stream) {
  if (F.bulk) return F.all ? launch<pl_flat_bulk_reduce_kernel<DT, HOOK, true>>(P, F, stream) : launch<pl_flat_bulk_reduce_kernel<DT, HOOK, false>>(P, F, stream);
  if (P.n_ranks <= 2) return launch_reduce<DT, 2, HOOK>(P, F, stream);
  if (P.n_ranks <= 4) return launch_reduce<DT, 4, HOOK>(P, F, stream);
  if (P.n_ranks <= 8) return launch_reduce<DT, 8, HOOK>(P, F, stream);
  return launch_reduce<DT, PL_MAX_RANKS, HOOK>(P, F, stream);
}

}  // namespace

FlatLaunch flat_launch(int R, bool reduce, bool all, bool bulk, uint32_t hook, uint64_t total_units, int sm_count) {
  FlatLaunch F;
  F.reduce = reduce;
  F.all = all;
  F.bulk = bulk;
  F.smem_bytes = 0;
  F.threads = bulk ? (reduce ? kFlatBulkThreads : 32) : kFlatThreads;
  if (bulk && reduce) {
    // about 16 KiB of sources: 128 units of 8 ranks (8 x 64 MiB reduce-scatter 86.6 us; 64 units 87.0,
    // 256 units 86.3, 512 units 87.4; fused with residual 232 us against 233 with 256 units)
    F.tile = R <= 2 ? 512u : R <= 4 ? 256u : 128u;
    const uint32_t n_aux = (hook & PL_HOOK_RESIDUAL) ? (all ? (uint32_t)R : 1u) : 0u;
    F.smem_bytes = kBarBytes + ((uint32_t)R + n_aux) * F.tile * 16u;
  } else if (bulk) {
    // all-gather 8 x 64 MiB 93.2 us with 128 units, 95.1 with 256, 99.4 with 1024.  With two or three stores for a load a CTA
    // of 128 is over too soon: reduce-scatter + all-gather 2 x 64 MiB 66.3 us, 256 units 52.9, 512 54.0; 2 x 128 MiB 129.0,
    // 114.8, 115.2; 3 x 64 MiB 77.7, 74.7; 4 x 64 MiB 93.4, 93.5; 5 x 64 MiB 117.5, 117.7
    F.tile = all && R > 3 ? 128u : 256u;
    F.smem_bytes = kBarBytes + F.tile * 16u;
  } else if (reduce) {
    const int U = hook ? (R <= 2 ? 2 : 1) : (R <= 2 ? 4 : R <= 4 ? 2 : 1);  // FlatUnits
    F.tile = (uint32_t)(U * kFlatThreads);
  } else {
    // one unit per thread where it goes to every rank (all-gather of 4 MiB: 6.4 us, 4 units 12.9 us)
    // or where 4 units would leave SMs without two CTAs
    F.units = (!all && total_units >= 4ull * kFlatThreads * 2 * (uint64_t)sm_count) ? 4 : 1;
    F.tile = (uint32_t)(F.units * kFlatThreads);
  }
  return F;
}

cudaError_t launch_flat(int dtype, const FlatParams& P, const FlatLaunch& F, cudaStream_t stream) {
  if (!F.reduce) {
    if (F.bulk) return F.all ? launch<pl_flat_bulk_copy_kernel<true>>(P, F, stream) : launch<pl_flat_bulk_copy_kernel<false>>(P, F, stream);
    if (F.all) return launch<pl_flat_copy_kernel<1, true>>(P, F, stream);
    return F.units == 4 ? launch<pl_flat_copy_kernel<4, false>>(P, F, stream) : launch<pl_flat_copy_kernel<1, false>>(P, F, stream);
  }
  switch (dtype) {
    case PL_BF16: return P.hook ? launch_dt<PL_BF16, true>(P, F, stream) : launch_dt<PL_BF16, false>(P, F, stream);
    case PL_F32: return P.hook ? launch_dt<PL_F32, true>(P, F, stream) : launch_dt<PL_F32, false>(P, F, stream);
    case PL_I32: return P.hook ? cudaErrorInvalidValue : launch_dt<PL_I32, false>(P, F, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pl
