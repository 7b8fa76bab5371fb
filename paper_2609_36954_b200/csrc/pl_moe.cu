// MoE expert-parallel dispatch / combine: an all-to-all-v of token rows whose counts are
// only known on the device (Table 2 of the paper names the pattern; Sec. 4 uses prefix sums
// for the variable-length offsets).
//
// dispatch = count (per 256-token block, per expert, via bit masks) -> scan (one CTA per
// source rank: exclusive prefix sums over its blocks, totals per expert and destination) ->
// place (segment bases in (source rank, expert, token) order, row index of every
// (token, slot), receive metadata) -> move (each token row is read once into
// shared memory by a bulk async copy and written to its K destinations by K bulk stores);
// with up to 1024 routing entries per source all of it in one launch (moe_small_kernel).
// combine = gate-weighted fp32 sum of the K expert rows of every token, ascending slot.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstring>
#include <new>
#include <vector>

#include "pl_api_internal.h"
#include "pl_internal.h"
#include "pl_ptx.cuh"

using namespace pl;

namespace {

constexpr int kTB = 256;             // tokens per count/place block
constexpr int kMaskWords = kTB / 32;
constexpr int kMaxTopk = 32;
constexpr int kCombineThreads = 256, kCombinePartThreads = 128;

// Kernels here are launched while the one in front drains, and that one may be what writes their
// routing (the caller's router, moe_derive_ranks_kernel).  So what a launch in front can write is
// read with coherent loads behind griddepcontrol.wait, never with __ldg: __ldcg where a word is read once (its
// loads go out in batches; plain ones cost a one-launch dispatch of 192 tokens 1.5 of 10 us), plain ones where the lines are
// used again from L1 (with __ldcg a deduplicated dispatch of 8 x 64 tokens takes 19.8 us instead of 15.5).  A
// non-coherent load wants data that nobody writes while the kernel lives.

struct DispatchPtrs {
  const void* x[PL_MAX_RANKS];
  const int32_t* idx[PL_MAX_RANKS];
  void* recv[PL_MAX_RANKS];
  int32_t* meta[PL_MAX_RANKS];
};
struct CombinePtrs {
  const void* y[PL_MAX_RANKS];
  const float* gates[PL_MAX_RANKS];
  void* out[PL_MAX_RANKS];
};
struct MoeGeo {
  int R, T, E, K, NB, epr;
  uint32_t row_bytes;
  uint32_t move_rows, move_parts;  // mover: token rows per tile, or tiles per row
  unsigned long long cap;
  int32_t* blockcnt;   // [R][NB][E]: per-block counts, turned into exclusive block offsets by scan
  long long* counts;   // [R][R]
  long long* ecounts;  // [R][E]
  int32_t* pos;        // [R][T][K] row in the destination's receive buffer, -1 if dropped
  int32_t* prank;      // [R][T][K] destination rank
  int* flags;          // [0] overflow, [1] invalid expert id, [2] copy engine wait gave up, [3] grid barrier gave up (sticky)
  unsigned int* sync;  // fused bookkeeping: [0] CTAs that reached the grid barrier, [1] CTAs that left the kernel
  const int32_t* slotmask;  // optional [R][T][K]: written into the metadata instead of the slot index
  int epr_shift;            // log2(epr), -1 if it is no power of two
  int gates_are_logits;     // combine: the gate input holds the K selected logits; softmax them first
  uint32_t parts, width;    // combine by parts: CTAs per row, threads per token
  uint64_t pad[4];
};
static_assert(cheap_params(sizeof(MoeGeo)) && sizeof(DispatchPtrs) % 64 == 0 && sizeof(CombinePtrs) % 64 == 0, "launch cost");

__device__ __forceinline__ void build_mask(const MoeGeo& g, const int32_t* idx, uint32_t* mask, int t, int tid) {
  for (int i = tid; i < g.E * kMaskWords; i += kTB) mask[i] = 0u;
  __syncthreads();
  if (t < g.T)
    for (int j = 0; j < g.K; ++j) {
      const int e = idx[(size_t)t * g.K + j];
      if (e < 0) continue;  // empty slot (deduplicated routing pads with -1)
      if (e < g.E) atomicOr(&mask[e * kMaskWords + (tid >> 5)], 1u << (tid & 31));
      else g.flags[1] = 1;
    }
  __syncthreads();
}

__global__ void __launch_bounds__(kTB) moe_count_kernel(const __grid_constant__ DispatchPtrs P, const __grid_constant__ MoeGeo g) {
  extern __shared__ uint32_t mask[];
  const int b = blockIdx.x, p = blockIdx.y, tid = threadIdx.x;
  build_mask(g, P.idx[p], mask, b * kTB + tid, tid);
  for (int e = tid; e < g.E; e += kTB) {
    int c = 0;
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) c += __popc(mask[e * kMaskWords + w]);
    g.blockcnt[((size_t)p * g.NB + b) * g.E + e] = c;
  }
}

// One CTA per source rank p: exclusive scan of the per-block counts of every expert, the totals
// per expert (ecounts) and per destination rank (counts).  Segment bases, which need the counts
// of all source ranks, are computed by the place kernel.
__global__ void __launch_bounds__(256) moe_scan_kernel(const __grid_constant__ MoeGeo g) {
  const int tid = threadIdx.x, n = blockDim.x, p = blockIdx.x;
  if (p == 0 && tid < 3) g.flags[tid] = 0;
  for (int e = tid; e < g.E; e += n) {
    int run = 0;
    // exclusive scan over the token blocks, eight independent loads at a time
    for (int b0 = 0; b0 < g.NB; b0 += 8) {
      int v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        v[i] = (b0 + i < g.NB) ? g.blockcnt[((size_t)p * g.NB + b0 + i) * g.E + e] : 0;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (b0 + i < g.NB) {
          g.blockcnt[((size_t)p * g.NB + b0 + i) * g.E + e] = run;
          run += v[i];
        }
    }
    g.ecounts[p * g.E + e] = run;
  }
  __syncthreads();  // this CTA's ecounts are visible to its own threads
  for (int r = tid; r < g.R; r += n) {
    long long s = 0;
    for (int e = r * g.epr; e < (r + 1) * g.epr; ++e) s += g.ecounts[p * g.E + e];
    g.counts[p * g.R + r] = s;
  }
}

__global__ void __launch_bounds__(kTB) moe_place_kernel(const __grid_constant__ DispatchPtrs P, const __grid_constant__ MoeGeo g) {
  extern __shared__ uint32_t mask[];
  int32_t* s_base = reinterpret_cast<int32_t*>(mask + (size_t)g.E * kMaskWords);  // [E] row of this source's segments
  const int b = blockIdx.x, p = blockIdx.y, tid = threadIdx.x, t = b * kTB + tid;
  const int32_t* idx = P.idx[p];
  // first row of expert e's run inside the receive buffer of its rank: everything sources
  // q < p send to that rank, then this source's rows for the rank's earlier experts
  for (int e = tid; e < g.E; e += kTB) {
    const int r = e / g.epr;
    long long off = 0;
    for (int q = 0; q < p; ++q) off += g.counts[q * g.R + r];
    for (int e2 = r * g.epr; e2 < e; ++e2) off += g.ecounts[p * g.E + e2];
    s_base[e] = (int32_t)off;
  }
  if (b == 0 && p == 0 && tid < g.R) {  // capacity check, once
    long long total = 0;
    for (int q = 0; q < g.R; ++q) total += g.counts[q * g.R + tid];
    if ((unsigned long long)total > g.cap) g.flags[0] = 1;
  }
  build_mask(g, idx, mask, t, tid);  // ends with a barrier: s_base is visible
  if (t >= g.T) return;
  const int w = tid >> 5;
  const uint32_t below = (1u << (tid & 31)) - 1u;
  for (int j = 0; j < g.K; ++j) {
    const int e = idx[(size_t)t * g.K + j];
    const size_t o = ((size_t)p * g.T + t) * g.K + j;
    if ((unsigned)e >= (unsigned)g.E) { g.pos[o] = -1; g.prank[o] = 0; continue; }
    int rank = __popc(mask[e * kMaskWords + w] & below);
    for (int w2 = 0; w2 < w; ++w2) rank += __popc(mask[e * kMaskWords + w2]);
    const long long row = (long long)s_base[e] + g.blockcnt[((size_t)p * g.NB + b) * g.E + e] + rank;
    const int r = e / g.epr;
    g.prank[o] = r;
    if ((unsigned long long)row < g.cap) {
      g.pos[o] = (int32_t)row;
      if (P.meta[r]) reinterpret_cast<int4*>(P.meta[r])[row] = make_int4(p, t, g.slotmask ? g.slotmask[o] : j, e);
    } else {
      g.pos[o] = -1;
    }
  }
}


// ---- fused bookkeeping: count -> (grid barrier) -> offsets -> place in ONE launch ------------
// Grid (NB, R), all CTAs co-resident (checked on the host).  Phase 1: the block's expert masks
// stay in shared memory and its per-expert counts go to global memory.  After a grid-wide
// barrier every CTA reads all R * NB * E counts (128 KiB at the C4 shape, from L2), derives the
// per-source totals, the segment bases of its own source rank and its own block offsets, and
// places its tokens.  The barrier is an arrival counter with a bounded wait; the last CTA to
// leave the kernel clears it, so nothing has to be reset between dispatches (or graph replays).
// Launched while the kernel in front drains, which takes 2 us off a dispatch (4 x 313 tokens of 1 KiB
// 16.5 -> 14.8 us, 4 x 360 deduplicated 24.8 -> 21.4, 8 x 1024 x 14 KiB 177 -> 175).
__global__ void __launch_bounds__(kTB) moe_plan_kernel(const __grid_constant__ DispatchPtrs P, const __grid_constant__ MoeGeo g) {
  extern __shared__ __align__(16) uint32_t mask[];
  int32_t* s_base = reinterpret_cast<int32_t*>(mask + (size_t)g.E * kMaskWords);  // [E]
  int32_t* s_ecnt = s_base + g.E;                                                 // [R][E] totals per (source, expert)
  int32_t* s_cnt = s_ecnt + (size_t)g.R * g.E;                                    // [R][R] rows source -> destination
  __shared__ int s_bad, s_giveup;
  const int b = blockIdx.x, p = blockIdx.y, tid = threadIdx.x, t = b * kTB + tid;
  const int32_t* idx = P.idx[p];
  if (tid == 0) { s_bad = 0; s_giveup = 0; }
  // ---- phase 1: masks and counts of this block
  for (int i = tid; i < g.E * kMaskWords; i += kTB) mask[i] = 0u;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Only now: the row mover's CTAs are to find the SMs empty, or they crowd on those that the launch in
  // front leaves first (4 x 313 tokens of 1 KiB, dispatch and combine: 25.4 us with the release before
  // the wait, 18.4 after it).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __syncthreads();
  if (t < g.T)
    for (int j0 = 0; j0 < g.K; j0 += 8) {
      int ev[8];  // eight slots at a time: the loads are independent of one another
#pragma unroll
      for (int k = 0; k < 8; ++k) ev[k] = (j0 + k < g.K) ? idx[(size_t)t * g.K + j0 + k] : -1;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int e = ev[k];
        if (e < 0) continue;  // empty slot (deduplicated routing pads with -1)
        if (e < g.E) atomicOr(&mask[e * kMaskWords + (tid >> 5)], 1u << (tid & 31));
        else s_bad = 1;
      }
    }
  __syncthreads();
  for (int e = tid; e < g.E; e += kTB) {
    int c = 0;
#pragma unroll
    for (int w = 0; w < kMaskWords; ++w) c += __popc(mask[e * kMaskWords + w]);
    g.blockcnt[((size_t)p * g.NB + b) * g.E + e] = c;
  }
  if (b == 0 && p == 0 && tid < 3) g.flags[tid] = 0;  // ordered before every later flag write by the barrier
  // ---- grid barrier
  __syncthreads();
  if (tid == 0) {
    const unsigned int n_ctas = gridDim.x * gridDim.y;
    __threadfence();
    atomicAdd(g.sync, 1u);
    unsigned int seen;
    unsigned long long t0 = 0;
    uint32_t spins = 0;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(g.sync) : "memory");
      if (seen >= n_ctas) break;
      if ((++spins & 63u) == 0) {
        unsigned long long now;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(now));
        if (t0 == 0) t0 = now;
        if (now - t0 > 2000000000ull) { s_giveup = 1; g.flags[3] = 1; break; }
      }
    }
  }
  __syncthreads();
  if (!s_giveup) {
    // ---- phase 2: totals per (source, expert); this block's offset inside its source's run.
    // Loads go out eight blocks at a time (independent, so one L2 latency per batch).
    if ((g.E & 3) == 0) {
      const int E4 = g.E >> 2;
      for (int i = tid; i < g.R * E4; i += kTB) {
        const int q = i / E4, e = (i - q * E4) << 2;
        int4 total = make_int4(0, 0, 0, 0), before = total;
        for (int b0 = 0; b0 < g.NB; b0 += 8) {
          int4 v[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            v[k] = (b0 + k < g.NB) ? __ldcg(reinterpret_cast<const int4*>(&g.blockcnt[((size_t)q * g.NB + b0 + k) * g.E + e]))
                                   : make_int4(0, 0, 0, 0);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (b0 + k == b) before = total;
            total.x += v[k].x; total.y += v[k].y; total.z += v[k].z; total.w += v[k].w;
          }
        }
        *reinterpret_cast<int4*>(&s_ecnt[q * g.E + e]) = total;
        if (q == p) *reinterpret_cast<int4*>(&s_base[e]) = before;
      }
    } else {
      for (int i = tid; i < g.R * g.E; i += kTB) {
        const int q = i / g.E, e = i - q * g.E;
        int total = 0, before = 0;
        for (int b0 = 0; b0 < g.NB; b0 += 8) {
          int v[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) v[k] = (b0 + k < g.NB) ? __ldcg(&g.blockcnt[((size_t)q * g.NB + b0 + k) * g.E + e]) : 0;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            if (b0 + k == b) before = total;
            total += v[k];
          }
        }
        s_ecnt[i] = total;
        if (q == p) s_base[e] = before;
      }
    }
    __syncthreads();
    for (int i = tid; i < g.R * g.R; i += kTB) {
      const int q = i / g.R, r = i - q * g.R;
      int c = 0;
      for (int e = r * g.epr; e < (r + 1) * g.epr; ++e) c += s_ecnt[q * g.E + e];
      s_cnt[i] = c;
    }
    __syncthreads();
    // first row of expert e's run in the receive buffer of its rank: what sources q < p send
    // there, then this source's rows for the rank's earlier experts, then the earlier blocks
    for (int e = tid; e < g.E; e += kTB) {
      const int r = e / g.epr;
      long long off = s_base[e];
      for (int q = 0; q < p; ++q) off += s_cnt[q * g.R + r];
      for (int e2 = r * g.epr; e2 < e; ++e2) off += s_ecnt[p * g.E + e2];
      s_base[e] = (int32_t)off;
      if (b == 0) g.ecounts[p * g.E + e] = s_ecnt[p * g.E + e];
    }
    if (b == 0 && tid < g.R) g.counts[p * g.R + tid] = s_cnt[p * g.R + tid];
    if (b == 0 && p == 0 && tid < g.R) {  // capacity check, once
      long long total = 0;
      for (int q = 0; q < g.R; ++q) total += s_cnt[q * g.R + tid];
      if ((unsigned long long)total > g.cap) g.flags[0] = 1;
    }
    if (tid == 0 && s_bad) g.flags[1] = 1;
    __syncthreads();
    // ---- phase 3: place this block's tokens
    if (t < g.T) {
      const int w = tid >> 5;
      const uint32_t below = (1u << (tid & 31)) - 1u;
      for (int j0 = 0; j0 < g.K; j0 += 8) {
        int ev[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) ev[k] = (j0 + k < g.K) ? idx[(size_t)t * g.K + j0 + k] : -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int j = j0 + k;
          if (j >= g.K) break;
          const int e = ev[k];
          const size_t o = ((size_t)p * g.T + t) * g.K + j;
          if ((unsigned)e >= (unsigned)g.E) { g.pos[o] = -1; g.prank[o] = 0; continue; }
          int rank = __popc(mask[e * kMaskWords + w] & below);
          for (int w2 = 0; w2 < w; ++w2) rank += __popc(mask[e * kMaskWords + w2]);
          const long long row = (long long)s_base[e] + rank;
          const int r = e / g.epr;
          g.prank[o] = r;
          if ((unsigned long long)row < g.cap) {
            g.pos[o] = (int32_t)row;
            if (P.meta[r]) reinterpret_cast<int4*>(P.meta[r])[row] = make_int4(p, t, g.slotmask ? g.slotmask[o] : j, e);
          } else {
            g.pos[o] = -1;
          }
        }
      }
    }
  }
  // ---- the last CTA to leave clears the barrier words for the next dispatch
  __syncthreads();
  if (tid == 0) {
    const unsigned int n_ctas = gridDim.x * gridDim.y;
    __threadfence();
    if (atomicAdd(g.sync + 1, 1u) == n_ctas - 1u) {
      g.sync[0] = 0u;
      g.sync[1] = 0u;
      __threadfence();
    }
  }
}

// Deduplicated routing: for every token the distinct destination ranks in ascending order
// (padded with -1) and, per destination, the mask of slots whose expert lives there.
struct DeriveParams {
  const int32_t* idx[PL_MAX_RANKS];
  int R, T, K, epr, KR;  // KR: destinations per token
  int32_t *ridx, *rmask;
  uint64_t pad[7];
};
static_assert(cheap_params(sizeof(DeriveParams)), "launch cost");
__global__ void __launch_bounds__(256) moe_derive_ranks_kernel(const __grid_constant__ DeriveParams P) {
  const int R = P.R, T = P.T, K = P.K, epr = P.epr, KR = P.KR;
  int32_t *const ridx = P.ridx, *const rmask = P.rmask;
  const long long tok = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tok >= (long long)R * T) return;
  const int p = (int)(tok / T);
  const long long t = tok % T;
  const int32_t* idx = P.idx[p] + t * K;
  unsigned masks[PL_MAX_RANKS];
#pragma unroll
  for (int r = 0; r < PL_MAX_RANKS; ++r) masks[r] = 0u;
  for (int j = 0; j < K; ++j) {
    const int e = idx[j];
    const int r = (e >= 0) ? e / epr : -1;
#pragma unroll
    for (int q = 0; q < PL_MAX_RANKS; ++q)
      if (q == r) masks[q] |= 1u << j;
  }
  int n = 0;
#pragma unroll
  for (int r = 0; r < PL_MAX_RANKS; ++r)
    if (r < R && masks[r]) {
      ridx[tok * KR + n] = r;
      rmask[tok * KR + n] = (int32_t)masks[r];
      ++n;
    }
  for (; n < KR; ++n) {
    ridx[tok * KR + n] = -1;
    rmask[tok * KR + n] = 0;
  }
}

// ---- small dispatches in one launch --------------------------------------------------------
// A CTA takes `rows` consecutive tokens of one source rank: it asks for their rows first, works out
// where its own rows go from the routing of everybody while they travel, and stores them.
// Each CTA reads all routing in front of its own (16 KiB of indices at 8 x 64 tokens x 8 slots),
// so nothing is counted, published and read back between launches or across a grid barrier.  A
// dispatch of this size is bound by its chain (indices from DRAM, counting, rows out) and by the
// launches; small_dispatch_rows() says where it is used.
// The row of (p, t, j) at rank r = entries of sources before p that go to r, plus entries of p that
// go to r with a lower expert, or with the same expert and an earlier token.
// DEDUP: an entry is (token, destination rank); the row is the number of earlier tokens, over
// sources and then tokens, with a slot on r.
struct SmallParams {
  uint32_t rows;            // tokens per CTA
  int K0, epr0;             // DEDUP: slots per token and experts per rank of the routing
  uint32_t release;         // release the launch behind at the start
  int32_t* ridx;            // DEDUP: distinct destination ranks per token, padded with -1, and the slots on each
  int32_t* rmask;
  uint64_t pad[4];
};
static_assert(sizeof(SmallParams) % 64 == 0, "launch cost");  // it goes with a MoeGeo

// Bounded wait for the first phase of `bar` (a CTA's rows have landed).
__device__ __forceinline__ bool wait_rows(uint64_t* bar) {
  if (ptx::mbar_try_wait(bar, 0)) return true;
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t0));
  for (uint32_t tries = 1;; ++tries) {
    if (ptx::mbar_try_wait(bar, 0)) return true;
    if ((tries & 1023u) == 0) {
      asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t1));
      if (t1 - t0 > 2000000000ull) return false;
    }
  }
}
// Adds one to rank r's 8-bit field (r < 16); a thread adds at most 255 entries.
__device__ __forceinline__ void count_rank(unsigned long long (&c)[2], int r) {
  const unsigned long long one = 1ull << ((r & 7) * 8);
  if (r < 8) c[0] += one;
  else c[1] += one;
}
// Sums the CTA's per-thread fields into s_cnt[16] (zeroed, a barrier before the call; none after).
__device__ __forceinline__ void sum_ranks(const unsigned long long (&c)[2], int R, int32_t* s_cnt) {
  const unsigned long long m = 0x00FF00FF00FF00FFull;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (h * 8 >= R) break;
    unsigned long long even = c[h] & m, odd = (c[h] >> 8) & m;  // 16-bit fields: a warp's 32 x 255 fit
#pragma unroll
    for (int d = 16; d; d >>= 1) {
      even += __shfl_xor_sync(0xFFFFFFFFu, even, d);
      odd += __shfl_xor_sync(0xFFFFFFFFu, odd, d);
    }
    const int lane = threadIdx.x & 31;
    if (lane < 8) {
      const int v = (int)(((lane & 1 ? odd : even) >> ((lane >> 1) * 16)) & 0xFFFFull);
      if (v) atomicAdd(&s_cnt[h * 8 + lane], v);
    }
  }
}
// Ranks that token `idx` (K slots) sends to, as a bit mask (dropping slots that name no expert).
__device__ __forceinline__ uint32_t rank_set(const int32_t* idx, int K, int epr, int R) {
  uint32_t set = 0;
  for (int j0 = 0; j0 < K; j0 += 8) {
    int ev[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) ev[k] = (j0 + k < K) ? idx[j0 + k] : -1;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (ev[k] >= 0 && ev[k] < epr * R) set |= 1u << (ev[k] / epr);
  }
  return set;
}

template <bool DEDUP>
__global__ void __launch_bounds__(kSmallThreads) moe_small_kernel(const __grid_constant__ DispatchPtrs P, const __grid_constant__ MoeGeo g,
                                                                  const __grid_constant__ SmallParams Q) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);
  unsigned char* tile = smem + 128;
  __shared__ int32_t s_cnt[16], s_total[16];
  __shared__ int32_t s_before[kSmallTargets];          // per target: this source's rows in front of it
  __shared__ int32_t s_set[kSmallTargets];             // DEDUP: rank sets of the CTA's tokens
  __shared__ int32_t s_own[DEDUP ? 1 : kSmallOwn];     // the source's routing
  __shared__ int32_t s_hist[DEDUP ? 1 : kSmallExperts];
  __shared__ int s_bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, R = g.R, T = g.T, K = DEDUP ? Q.K0 : g.K, TK = T * K;
  const uint32_t groups = ((uint32_t)T + Q.rows - 1) / Q.rows;
  // The first R CTAs count a source's entries, the one behind them all entries; the others move rows.
  // (Counted by the CTAs that move a source's first tokens it came on top of the longest chain: dispatch
  // and combine of 8 x 8 tokens of 14 KiB 13.8 us, now 10.5; 8 x 8 of 4 KiB deduplicated 11.3, now 9.3.)
  const uint32_t counters = (uint32_t)R + 1u;
  const bool counts = blockIdx.x < counters;
  const int p = counts ? (int)min(blockIdx.x, (uint32_t)R - 1u) : (int)((blockIdx.x - counters) / groups);
  const int t0 = counts ? 0 : (int)((blockIdx.x - counters - (uint32_t)p * groups) * Q.rows);
  const int nrows = min((int)Q.rows, T - t0), Kd = g.K, n_tgt = nrows * Kd;  // Kd: entries per token (DEDUP: ranks)
  if (!DEDUP && Q.release) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid < 16) s_cnt[tid] = s_total[tid] = 0;
  if (tid == 0) {
    s_bad = 0;
    ptx::mbar_init(full, 1);
    ptx::mbar_init_fence();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (tid == 0 && !counts) {
    const uint32_t bytes = (uint32_t)nrows * g.row_bytes;
    ptx::mbar_expect_tx(full, bytes);
    ptx::bulk_g2s_hint(tile, static_cast<const char*>(P.x[p]) + (size_t)t0 * g.row_bytes, bytes, full, ptx::policy_evict_first());
  }
  const int32_t* own = P.idx[p];
  auto rank_of = [&](int e) { return g.epr_shift >= 0 ? e >> g.epr_shift : e / g.epr; };
  // entries per rank of the sources [0, n), in this thread's 8-bit fields
  auto count_sources = [&](int n, unsigned long long (&into)[2], bool check) {
    bool vec = (TK & 3) == 0;
    for (int q = 0; q < n; ++q) vec = vec && ((uintptr_t)P.idx[q] & 15) == 0;
    if (vec) {  // 16 bytes at a time, over all sources
      const int nv = TK >> 2, all = n * nv;
      for (int i0 = tid; i0 < all; i0 += 4 * kSmallThreads) {
        int4 ev[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = i0 + k * kSmallThreads, q = i / nv;
          ev[k] = i < all ? __ldcg(reinterpret_cast<const int4*>(P.idx[q]) + (i - q * nv)) : make_int4(-1, -1, -1, -1);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int e = m == 0 ? ev[k].x : m == 1 ? ev[k].y : m == 2 ? ev[k].z : ev[k].w;
            if ((unsigned)e < (unsigned)g.E) count_rank(into, rank_of(e));
            else if (check && e >= 0) s_bad = 1;
          }
      }
      return;
    }
    for (int i = tid; i < TK; i += kSmallThreads)
      for (int q0 = 0; q0 < n; q0 += 8) {
        int ev[8];  // independent loads: one L2 latency per batch
#pragma unroll
        for (int k = 0; k < 8; ++k) ev[k] = (q0 + k < n) ? __ldcg(&P.idx[q0 + k][i]) : -1;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if ((unsigned)ev[k] < (unsigned)g.E) count_rank(into, rank_of(ev[k]));
          else if (check && ev[k] >= 0) s_bad = 1;
        }
      }
  };
  auto count_tokens = [&](int from, int to, unsigned long long (&into)[2]) {  // DEDUP: tokens numbered over the sources
    for (int i = from + tid; i < to; i += kSmallThreads) {
      const int q = i / T;
      for (uint32_t set = rank_set(P.idx[q] + (size_t)(i - q * T) * K, K, Q.epr0, R); set; set &= set - 1) count_rank(into, __ffs(set) - 1);
    }
  };
  unsigned long long c[2] = {0ull, 0ull};
  if (counts) {
    __syncthreads();
    if (blockIdx.x < (uint32_t)R) {
      if constexpr (DEDUP) {
        count_tokens(p * T, (p + 1) * T, c);
        sum_ranks(c, R, s_total);
        __syncthreads();
        if (tid < R) g.counts[p * R + tid] = g.ecounts[p * R + tid] = s_total[tid];
      } else {
        for (int e = tid; e < g.E; e += kSmallThreads) s_hist[e] = 0;
        __syncthreads();
        for (int i = tid; i < TK; i += kSmallThreads) {
          const int e = __ldcg(&own[i]);
          if ((unsigned)e < (unsigned)g.E) atomicAdd(&s_hist[e], 1);
        }
        __syncthreads();
        for (int e = tid; e < g.E; e += kSmallThreads) g.ecounts[(size_t)p * g.E + e] = s_hist[e];
        if (tid < R) {
          long long n = 0;
          for (int e = tid * g.epr; e < (tid + 1) * g.epr; ++e) n += s_hist[e];
          g.counts[p * R + tid] = n;
        }
      }
    } else {  // the whole routing: does every rank's share fit, does every slot name an expert
      if constexpr (DEDUP) count_tokens(0, R * T, c);
      else count_sources(R, c, true);
      sum_ranks(c, R, s_total);
      __syncthreads();
      if (tid == 0) {
        int over = 0;
        for (int q = 0; q < R; ++q) over |= (unsigned long long)s_total[q] > g.cap;
        g.flags[0] = over;
        g.flags[1] = s_bad;
        g.flags[2] = 0;
      }
    }
    return;
  }
  // ---- what goes to each rank in front of this CTA's tokens
  if constexpr (DEDUP) {
    if (tid < nrows) s_set[tid] = (int32_t)rank_set(own + (size_t)(t0 + tid) * K, K, Q.epr0, R);
    count_tokens(0, p * T + t0, c);
  } else {
    for (int i = tid; i < TK; i += kSmallThreads) s_own[i] = __ldcg(&own[i]);
    count_sources(p, c, false);
  }
  __syncthreads();
  sum_ranks(c, R, s_cnt);
  if constexpr (!DEDUP) {
    // this source's entries in front of each target: lower expert of the rank, or same expert and
    // an earlier token.  Warp w takes targets w, w + 8, ...; its lanes share the entries.
    for (int k = warp; k < n_tgt; k += kSmallThreads / 32) {
      const int t = t0 + k / K, e = s_own[t0 * K + k];
      if ((unsigned)e >= (unsigned)g.E) continue;
      const int lo = rank_of(e) * g.epr;  // first expert of the rank
      int n = 0;
#pragma unroll 4
      for (int i = lane; i < TK; i += 32) {
        const int o = s_own[i];
        n += (o >= lo && (o < e || (o == e && i < t * K))) ? 1 : 0;
      }
      n = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)n);
      if (lane == 0) s_before[k] = n;
    }
  }
  __syncthreads();
  // ---- place: thread k owns target k
  int row = -1, r = 0, src = 0, meta_j = 0, meta_e = 0;
  if (tid < n_tgt) {
    src = tid / Kd;
    const int j = tid - src * Kd, t = t0 + src;
    bool live;
    if constexpr (DEDUP) {
      uint32_t set = (uint32_t)s_set[src], mask = 0;
      for (int k = 0; k < j; ++k) set &= set - 1;
      live = set != 0;
      if (live) {
        r = __ffs(set) - 1;
        row = s_cnt[r];
        for (int k = 0; k < src; ++k) row += (int)(((uint32_t)s_set[k] >> r) & 1u);
        for (int k = 0; k < K; ++k) {
          const int e = own[(size_t)t * K + k];
          if (e >= 0 && e / Q.epr0 == r) mask |= 1u << k;
        }
      }
      const size_t o = ((size_t)p * T + t) * Kd + j;
      Q.ridx[o] = live ? r : -1;
      Q.rmask[o] = (int32_t)mask;
      meta_j = (int)mask;
      meta_e = r;
    } else {
      meta_j = j;
      meta_e = s_own[t * K + j];
      live = (unsigned)meta_e < (unsigned)g.E;
      if (live) {
        r = rank_of(meta_e);
        row = s_cnt[r] + s_before[tid];
      }
    }
    if (live && (unsigned long long)row >= g.cap) row = -1;
  }
  // ---- the rows have landed (bounded wait): one bulk store per target
  bool ok = true;
  if (tid < n_tgt) {
    ok = wait_rows(full);
    if (ok && row >= 0) {
      ptx::bulk_s2g_hint(static_cast<char*>(P.recv[r]) + (size_t)row * g.row_bytes, tile + (size_t)src * g.row_bytes, g.row_bytes, ptx::policy_evict_first());
      ptx::bulk_commit();
    }
    // bookkeeping while the rows leave
    const size_t o = ((size_t)p * T + t0 + src) * Kd + (tid - src * Kd);
    g.pos[o] = row;
    g.prank[o] = r;
    if (row >= 0 && P.meta[r]) reinterpret_cast<int4*>(P.meta[r])[row] = make_int4(p, t0 + src, meta_j, meta_e);
  }
  if (tid < n_tgt) {
    ptx::bulk_wait<0>();
    if (!ok) {
      g.flags[3] = 1;  // reported and cleared by the next read of the plan
      ptx::mbar_wait_bounded(full, 0, 1u << 20);
    }
  }
}

// ---- rows to their destinations ---------------------------------------------------------------
// A CTA of one warp moves one tile: a part of a token's row, or `rows` consecutive short rows of one
// source (contiguous in its input).  One bulk load, then a bulk store per destination.  Bound by HBM
// (1 read : K writes); the order in which the tiles are dealt keeps all SMs inside one window of
// the input, and tiles of 2 KiB were served best (8 x 4096 tokens of 14,336 bytes, top-8, whole
// dispatch: 660 us; 3584 bytes 684, 7168 bytes 667, whole rows 666; a persistent ring of 56 KiB
// loads on 132 SMs 742).
constexpr uint32_t kMoveTile = 2048;
__global__ void __launch_bounds__(32) moe_move_kernel(const __grid_constant__ DispatchPtrs P, const __grid_constant__ MoeGeo g) {
  __shared__ __align__(128) unsigned char tile[kMoveTile];
  __shared__ uint64_t full;
  const uint32_t lane = threadIdx.x, T = (uint32_t)g.T, K = (uint32_t)g.K;
  uint32_t p, t, nrows = 1, off = 0, bytes;  // tokens [t, t + nrows) of source p, bytes [off, off + bytes) of each
  if (g.move_rows > 1) {
    const uint32_t groups = (T + g.move_rows - 1) / g.move_rows;
    p = blockIdx.x / groups;
    t = (blockIdx.x - p * groups) * g.move_rows;
    nrows = min(g.move_rows, T - t);
    bytes = g.row_bytes;
  } else {
    const uint32_t tok = blockIdx.x / g.move_parts;
    p = tok / T;
    t = tok - p * T;
    off = (blockIdx.x - tok * g.move_parts) * kMoveTile;
    bytes = min(kMoveTile, g.row_bytes - off);
  }
  if (lane == 0) {
    ptx::mbar_init(&full, 1);
    ptx::mbar_init_fence();
    ptx::mbar_expect_tx(&full, nrows * bytes);
  }
  __syncwarp();
  // launched with programmatic stream serialization: wait for the bookkeeping kernel to complete
  // before anything it wrote (pos, prank) is read
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (lane == 0)
    ptx::bulk_g2s_hint(tile, static_cast<const char*>(P.x[p]) + (size_t)t * g.row_bytes + off, nrows * bytes, &full, ptx::policy_evict_first());
  const size_t at = ((size_t)p * T + t) * K;
  const uint32_t n_st = nrows * K;
  int row = -1, r = 0;  // this lane's first store, fetched before the wait
  if (lane < n_st) {
    row = g.pos[at + lane];
    r = g.prank[at + lane];
  }
  if (!wait_rows(&full)) {
    g.flags[2] = 1;
    ptx::mbar_wait_bounded(&full, 0, 1u << 20);
    return;
  }
  for (uint32_t i = lane; i < n_st; i += 32) {
    if (i >= 32) {
      row = g.pos[at + i];
      r = g.prank[at + i];
    }
    // every token row is read once and every received row written once: both stream through L2
    if (row >= 0)
      ptx::bulk_s2g_hint(static_cast<char*>(P.recv[r]) + (size_t)row * g.row_bytes + off, tile + (size_t)(i / K) * bytes, bytes, ptx::policy_evict_first());
  }
  ptx::bulk_commit();
  ptx::bulk_wait<0>();
}

// fp32 softmax over a token's K logits (max-subtracted); lane j < K of a warp holds logit j
__device__ __forceinline__ float softmax_gate(float logit, int K) {
  const unsigned lanes = (K >= 32) ? 0xFFFFFFFFu : ((1u << K) - 1u);
  float m = logit;
  for (int j = 0; j < K; ++j) m = fmaxf(m, __shfl_sync(lanes, logit, j));
  const float e = expf(logit - m);
  float sum = 0.f;
  for (int j = 0; j < K; ++j) sum += __shfl_sync(lanes, e, j);  // ascending slot order on every lane
  return e / sum;
}
__device__ __forceinline__ void add_gated(float (&acc)[8], float gate, const uint4& q) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    acc[2 * i] = fmaf(gate, __uint_as_float(w[i] << 16), acc[2 * i]);
    acc[2 * i + 1] = fmaf(gate, __uint_as_float(w[i] & 0xFFFF0000u), acc[2 * i + 1]);
  }
}
__device__ __forceinline__ uint4 round_row(const float (&acc)[8]) {
  uint4 o;
  __nv_bfloat162 a = __floats2bfloat162_rn(acc[0], acc[1]), b = __floats2bfloat162_rn(acc[2], acc[3]);
  __nv_bfloat162 c = __floats2bfloat162_rn(acc[4], acc[5]), d = __floats2bfloat162_rn(acc[6], acc[7]);
  o.x = *reinterpret_cast<uint32_t*>(&a);
  o.y = *reinterpret_cast<uint32_t*>(&b);
  o.z = *reinterpret_cast<uint32_t*>(&c);
  o.w = *reinterpret_cast<uint32_t*>(&d);
  return o;
}

// Neither combine kernel releases its dependents: the launch behind it is set up as its CTAs exit.  Released
// earlier, the few CTAs of the next dispatch's bookkeeping all crowd on the first SM that has room and share
// it (dispatch and combine, 256 experts, top-8, released at the start / at the end: 8 x 256 tokens of 14 KiB 120 / 103 us,
// of 1 KiB 38 / 20, 8 x 1024 of 4 KiB 132 / 115, 16 x 256 of 14 KiB 203 / 187; one-launch dispatch 8 x 8 of 14 KiB 13.3 / 7.9;
// nothing is slower).
//
// combine: CTA per token (grid-strided), 16-byte column units across threads, the K source
// rows and gates of the next token are fetched while the current one is summed.
__global__ void __launch_bounds__(kCombineThreads) moe_combine_kernel(const __grid_constant__ CombinePtrs P, const __grid_constant__ MoeGeo g) {
  __shared__ const char* s_row[2][kMaxTopk];
  __shared__ float s_gate[2][kMaxTopk];
  const int tid = threadIdx.x;
  const unsigned long long n_tok = (unsigned long long)g.R * g.T;
  auto load_meta = [&](unsigned long long tok, int buf) {
    if (tid < g.K) {
      const int p = (int)(tok / g.T);
      const unsigned long long t = tok % g.T;
      const int row = g.pos[tok * g.K + tid];
      const int r = g.prank[tok * g.K + tid];
      s_row[buf][tid] = row >= 0 ? static_cast<const char*>(P.y[r]) + (size_t)row * g.row_bytes : nullptr;
      float gate = P.gates[p][t * g.K + tid];
      if (g.gates_are_logits) gate = softmax_gate(gate, g.K);
      s_gate[buf][tid] = gate;
    }
  };
  asm volatile("griddepcontrol.wait;" ::: "memory");
  unsigned long long tok = blockIdx.x;
  if (tok < n_tok) load_meta(tok, 0);
  __syncthreads();
  const uint32_t units = g.row_bytes >> 4;
  for (int it = 0; tok < n_tok; tok += gridDim.x, ++it) {
    const int buf = it & 1;
    if (tok + gridDim.x < n_tok) load_meta(tok + gridDim.x, buf ^ 1);
    const int p = (int)(tok / g.T);
    char* out = static_cast<char*>(P.out[p]) + (tok % g.T) * g.row_bytes;
    for (uint32_t u = tid; u < units; u += kCombineThreads) {
      float acc[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] = 0.f;
      for (int j0 = 0; j0 < g.K; j0 += 8) {
        uint4 q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const char* rowp = (j0 + j < g.K) ? s_row[buf][j0 + j] : nullptr;
          q[j] = rowp ? __ldcg(reinterpret_cast<const uint4*>(rowp) + u) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (j0 + j < g.K) add_gated(acc, s_gate[buf][j0 + j], q[j]);
        }
      }
      __stcg(reinterpret_cast<uint4*>(out) + u, round_row(acc));
    }
    __syncthreads();
  }
}

// The same for few tokens or short rows: CTA per (token, part of the row) or per several tokens of a
// short row, one 16-byte unit per thread, so that the work divides over the SMs whatever the token
// count is.  `width` threads (whole warps) work on one token.  KB source rows are loaded at a time:
// with few slots per token the registers of eight would cost half of the resident CTAs.
template <int KB>
__global__ void __launch_bounds__(kCombinePartThreads) moe_combine_parts_kernel(const __grid_constant__ CombinePtrs P, const __grid_constant__ MoeGeo g) {
  const uint32_t parts = g.parts, width = g.width;
  constexpr int kTokens = kCombinePartThreads / 32;
  __shared__ const char* s_row[kTokens][kMaxTopk];
  __shared__ float s_gate[kTokens][kMaxTopk];
  const uint32_t sub = threadIdx.x / width, tid = threadIdx.x - sub * width;  // token of this CTA, thread of that token
  uint32_t tok, part = 0;
  if (parts > 1) {
    tok = blockIdx.x / parts;
    part = blockIdx.x - tok * parts;
  } else {
    tok = blockIdx.x * (blockDim.x / width) + sub;
  }
  const bool live = tok < (uint32_t)g.R * (uint32_t)g.T;
  const uint32_t p = live ? tok / (uint32_t)g.T : 0u, t = tok - p * (uint32_t)g.T;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (live && tid < (uint32_t)g.K) {
    const int row = g.pos[(size_t)tok * g.K + tid];
    const int r = g.prank[(size_t)tok * g.K + tid];
    float gate = P.gates[p][(size_t)t * g.K + tid];
    s_row[sub][tid] = row >= 0 ? static_cast<const char*>(P.y[r]) + (size_t)row * g.row_bytes : nullptr;
    if (g.gates_are_logits) gate = softmax_gate(gate, g.K);
    s_gate[sub][tid] = gate;
  }
  __syncthreads();
  const uint32_t units = g.row_bytes >> 4, u = part * width + tid;
  if (!live || u >= units) return;
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  for (int j0 = 0; j0 < g.K; j0 += KB) {
    uint4 q[KB];
#pragma unroll
    for (int j = 0; j < KB; ++j) {
      const char* rowp = (j0 + j < g.K) ? s_row[sub][j0 + j] : nullptr;
      q[j] = rowp ? __ldcg(reinterpret_cast<const uint4*>(rowp) + u) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < KB; ++j)
      if (j0 + j < g.K) add_gated(acc, s_gate[sub][j0 + j], q[j]);
  }
  __stcg(reinterpret_cast<uint4*>(static_cast<char*>(P.out[p]) + (size_t)t * g.row_bytes) + u, round_row(acc));
}

// A launch set up while the one in front drains (programmatic stream serialization, unless
// `overlap` is false): the kernel waits for everything in front before it reads or writes.
template <typename... Params, typename... Args>
bool launch_after(bool overlap, void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t cs, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = cs;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  if (cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The dynamic shared-memory limit is an attribute of the FUNCTION (per device), not of a plan:
// it is raised once per device to the most any plan can ask for, so that creating a second,
// smaller plan cannot lower it under the feet of the first.
constexpr int kMaxExperts = 4096;
constexpr size_t kPlanSmemMax = 200 * 1024;  // the fused bookkeeping kernel is used while its tables fit this

size_t plan_smem_bytes(const MoeGeo& g) {
  return ((size_t)g.E * kMaskWords + (size_t)g.E + (size_t)g.R * g.E + (size_t)g.R * g.R) * 4;
}
bool configure_kernels(int device) {
  static std::atomic<unsigned long long> configured{0};
  const unsigned long long bit = 1ull << (device & 63);
  if (configured.load(std::memory_order_acquire) & bit) return true;
  if (cudaFuncSetAttribute(moe_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxExperts * kMaskWords * 4) != cudaSuccess ||
      cudaFuncSetAttribute(moe_place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxExperts * kMaskWords * 4 + kMaxExperts * 4) != cudaSuccess ||
      cudaFuncSetAttribute(moe_small_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemMax) != cudaSuccess ||
      cudaFuncSetAttribute(moe_small_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemMax) != cudaSuccess ||
      cudaFuncSetAttribute(moe_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPlanSmemMax) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  configured.fetch_or(bit, std::memory_order_release);
  return true;
}

}  // namespace

struct pl_moe_plan_s {
  pl_comm_t comm = nullptr;
  MoeGeo g{};
  char* d_blob = nullptr;
  size_t blob_bytes = 0;
  int sm_count = 148;
  int combine_per_sm = 4;  // resident CTAs of the combine kernel per SM (occupancy query at plan creation)
  bool fused = false, fused_dedup = false;  // bookkeeping in one launch (grid co-resident, tables fit shared memory)
  uint32_t small_rows = 0, small_rows_dedup = 0;  // > 0: dispatched in one launch with this many tokens per CTA
  bool dispatched = false;
  // deduplicated variant: the same machinery run over "one expert per rank" routing
  MoeGeo gd{};
  int32_t* d_ridx = nullptr;   // [R][T][KR] distinct destination ranks, -1 padded
  int32_t* d_rmask = nullptr;  // [R][T][KR] slot masks
  float* d_ones = nullptr;     // [T][KR] unit gates
  char* d_blob2 = nullptr;
  bool dispatched_dedup = false;
};

extern "C" {

pl_status_t pl_moe_plan_create(pl_comm_t comm, int tokens_per_rank, int hidden, int n_experts, int topk,
                               size_t recv_capacity_rows, pl_moe_plan_t* out) {
  if (!comm || !out) return PL_ERR_INVALID_ARG;
  *out = nullptr;
  if (comm->planner) return PL_ERR_UNSUPPORTED;
  if (!on_comm_device(comm)) return PL_ERR_INVALID_ARG;
  const int R = comm->R;
  if (tokens_per_rank < 1 || hidden < 1 || n_experts < R || topk < 1 || topk > kMaxTopk) return PL_ERR_INVALID_ARG;
  if (n_experts % R || n_experts > kMaxExperts || topk > n_experts) return PL_ERR_INVALID_ARG;
  if (recv_capacity_rows == 0 || recv_capacity_rows > 0x7FFFFFFFull) return PL_ERR_INVALID_ARG;
  const size_t row_bytes = (size_t)hidden * elem_size(comm->dtype);
  if (row_bytes % 16) return PL_ERR_ALIGNMENT;
  if (row_bytes > (1u << 30)) return PL_ERR_INVALID_ARG;
  pl_moe_plan_s* pl = new (std::nothrow) pl_moe_plan_s();
  if (!pl) return PL_ERR_OOM;
  pl->comm = comm;
  pl->sm_count = comm->sm_count;
  {
    // The combine kernel deals tokens to CTAs by a fixed stride, so its grid must be exactly one
    // resident wave: with 1.5 waves (6 CTAs per SM against 4 resident) the second half wave ran
    // alone and the launch took 703 us instead of 612 us (C4 shape).
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, moe_combine_kernel, kCombineThreads, 0) != cudaSuccess || occ < 1) {
      cudaGetLastError();
      occ = 1;
    }
    pl->combine_per_sm = occ;
  }
  MoeGeo& g = pl->g;
  g.R = R;
  g.T = tokens_per_rank;
  g.E = n_experts;
  g.K = topk;
  g.NB = (tokens_per_rank + kTB - 1) / kTB;
  g.epr = n_experts / R;
  g.epr_shift = -1;
  for (int b = 0; b < 13; ++b)
    if (g.epr == 1 << b) g.epr_shift = b;
  g.row_bytes = (uint32_t)row_bytes;
  g.move_rows = (uint32_t)std::max<size_t>(1, std::min<size_t>(32, kMoveTile / row_bytes));
  g.move_parts = (uint32_t)((row_bytes + kMoveTile - 1) / kMoveTile);
  g.cap = recv_capacity_rows;
  size_t off = 0;
  auto place = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
  const size_t o_bc = place((size_t)R * g.NB * g.E * 4);
  const size_t o_cnt = place((size_t)R * R * 8), o_ecnt = place((size_t)R * g.E * 8);
  const size_t o_pos = place((size_t)R * g.T * g.K * 4), o_prank = place((size_t)R * g.T * g.K * 4);
  const size_t o_flags = place(32);  // 4 flag words + 2 barrier words
  pl->blob_bytes = off;
  if (cudaMalloc(&pl->d_blob, off) != cudaSuccess) { cudaGetLastError(); delete pl; return PL_ERR_OOM; }
  if (cudaMemset(pl->d_blob, 0, off) != cudaSuccess) { cudaGetLastError(); cudaFree(pl->d_blob); delete pl; return PL_ERR_CUDA; }
  g.blockcnt = reinterpret_cast<int32_t*>(pl->d_blob + o_bc);
  g.counts = reinterpret_cast<long long*>(pl->d_blob + o_cnt);
  g.ecounts = reinterpret_cast<long long*>(pl->d_blob + o_ecnt);
  g.pos = reinterpret_cast<int32_t*>(pl->d_blob + o_pos);
  g.prank = reinterpret_cast<int32_t*>(pl->d_blob + o_prank);
  g.flags = reinterpret_cast<int*>(pl->d_blob + o_flags);
  g.sync = reinterpret_cast<unsigned int*>(pl->d_blob + o_flags + 16);
  if (!configure_kernels(comm->device)) {
    cudaFree(pl->d_blob);
    delete pl;
    return PL_ERR_CUDA;
  }
  // second set of bookkeeping for the deduplicated variant: R "experts" (one per rank),
  // at most min(topk, R) destinations per token
  {
    MoeGeo& d = pl->gd;
    d = g;
    d.E = R;
    d.epr = 1;
    d.epr_shift = 0;
    d.K = std::min(topk, R);
    size_t off2 = 0;
    auto place2 = [&](size_t bytes) { size_t o = off2; off2 = align_up(off2 + bytes, 256); return o; };
    const size_t tk = (size_t)R * g.T * d.K;
    const size_t q_bc = place2((size_t)R * g.NB * R * 4);
    const size_t q_cnt = place2((size_t)R * R * 8), q_ecnt = place2((size_t)R * R * 8);
    const size_t q_pos = place2(tk * 4), q_prank = place2(tk * 4), q_ridx = place2(tk * 4), q_rmask = place2(tk * 4);
    const size_t q_ones = place2((size_t)g.T * d.K * 4), q_flags = place2(32);
    if (cudaMalloc(&pl->d_blob2, off2) != cudaSuccess) { cudaGetLastError(); cudaFree(pl->d_blob); delete pl; return PL_ERR_OOM; }
    std::vector<float> ones((size_t)g.T * d.K, 1.0f);
    if (cudaMemset(pl->d_blob2, 0, off2) != cudaSuccess ||
        cudaMemcpy(pl->d_blob2 + q_ones, ones.data(), ones.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess) {
      cudaGetLastError();
      cudaFree(pl->d_blob);
      cudaFree(pl->d_blob2);
      delete pl;
      return PL_ERR_CUDA;
    }
    d.blockcnt = reinterpret_cast<int32_t*>(pl->d_blob2 + q_bc);
    d.counts = reinterpret_cast<long long*>(pl->d_blob2 + q_cnt);
    d.ecounts = reinterpret_cast<long long*>(pl->d_blob2 + q_ecnt);
    d.pos = reinterpret_cast<int32_t*>(pl->d_blob2 + q_pos);
    d.prank = reinterpret_cast<int32_t*>(pl->d_blob2 + q_prank);
    d.flags = reinterpret_cast<int*>(pl->d_blob2 + q_flags);
    d.sync = reinterpret_cast<unsigned int*>(pl->d_blob2 + q_flags + 16);
    pl->d_ridx = reinterpret_cast<int32_t*>(pl->d_blob2 + q_ridx);
    pl->d_rmask = reinterpret_cast<int32_t*>(pl->d_blob2 + q_rmask);
    pl->d_ones = reinterpret_cast<float*>(pl->d_blob2 + q_ones);
    d.slotmask = pl->d_rmask;
  }
  {
    // one-launch bookkeeping needs every CTA of its grid resident at once (they meet at a barrier)
    auto feasible = [&](const MoeGeo& q) {
      const size_t smem = plan_smem_bytes(q);
      if (smem > kPlanSmemMax) return false;
      int per_sm = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, moe_plan_kernel, kTB, smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
      }
      return (long long)q.NB * q.R <= (long long)per_sm * comm->sm_count;
    };
    pl->fused = feasible(pl->g);
    pl->fused_dedup = feasible(pl->gd);
    pl->small_rows = small_dispatch_rows(false, R, tokens_per_rank, topk, n_experts, row_bytes, comm->sm_count);
    pl->small_rows_dedup = small_dispatch_rows(true, R, tokens_per_rank, topk, n_experts, row_bytes, comm->sm_count);
  }
  comm->n_plans += 1;
  *out = pl;
  return PL_OK;
}

pl_status_t pl_moe_plan_destroy(pl_moe_plan_t plan) {
  if (!plan) return PL_ERR_INVALID_ARG;
  if (plan->d_blob) cudaFree(plan->d_blob);
  if (plan->d_blob2) cudaFree(plan->d_blob2);
  plan->comm->n_plans -= 1;
  delete plan;
  return PL_OK;
}

// count / scan / place (or the fused kernel), then the row mover launched so that its set-up
// overlaps the tail of the bookkeeping.  Returns the number of kernels launched, 0 on error.
static int launch_dispatch(pl_moe_plan_t plan, const DispatchPtrs& P, const MoeGeo& g, bool fused, cudaStream_t cs) {
  int launched = 0;
  const size_t mask_smem = (size_t)g.E * kMaskWords * 4;
  dim3 grid(g.NB, g.R);
  if (fused) {
    if (!launch_after(true, moe_plan_kernel, grid, kTB, plan_smem_bytes(g), cs, P, g)) return 0;
    launched = 1;
  } else {
    moe_count_kernel<<<grid, kTB, mask_smem, cs>>>(P, g);
    moe_scan_kernel<<<g.R, 256, 0, cs>>>(g);
    moe_place_kernel<<<grid, kTB, mask_smem + (size_t)g.E * 4, cs>>>(P, g);
    launched = 3;
  }
  if (cudaGetLastError() != cudaSuccess) return 0;
  const unsigned long long tiles = g.move_rows > 1 ? (unsigned long long)g.R * ((g.T + g.move_rows - 1) / g.move_rows)
                                                   : (unsigned long long)g.R * g.T * g.move_parts;
  if (tiles > 0x7FFFFFFFull) return 0;
  // only the fused kernel releases its dependents early
  if (!launch_after(fused, moe_move_kernel, dim3((unsigned)tiles), 32, 0, cs, P, g)) return 0;
  return launched + 1;
}

// The launch behind is released early where few bytes are written; else, and deduplicated, it is set up as the CTAs exit.  Dispatch and
// combine in turn, us, released / not, one by one and in a graph: top-2 8 x 8 tokens of 1 KiB 6.7 / 6.9 and 5.2 / 5.4, top-8 8 x 8 of 1 KiB 6.7 / 6.8 and 5.5
// / 6.0, top-2 4 x 256 of 4 KiB 11.3 / 11.5 and 11.0 / 11.3; from 12 MiB of rows on 4 x 64 top-8 of 14 KiB 14.15 / 13.88 and 13.5 / 13.6, 8 x 64 26.0 / 25.8 and 25.65 /
// 25.84, top-2 8 x 64 10.8 / 10.5 and 10.2 / 10.3; deduplicated top-2 8 x 64 of 1 KiB 8.3 / 7.5 and 7.9 / 7.2, top-8 8 x 8 of 4 KiB 8.9 / 8.4 and 7.8 / 8.2.
static bool launch_small(const DispatchPtrs& P, const MoeGeo& g, SmallParams Q, bool dedup, cudaStream_t cs) {
  Q.release = (uint64_t)g.R * g.T * g.K * g.row_bytes < (12ull << 20);
  const dim3 grid((unsigned)g.R * (((unsigned)g.T + Q.rows - 1) / Q.rows) + (unsigned)g.R + 1u);
  return launch_after(true, dedup ? moe_small_kernel<true> : moe_small_kernel<false>, grid, kSmallThreads, 128 + (size_t)Q.rows * g.row_bytes, cs, P, g, Q);
}

pl_status_t pl_moe_dispatch(pl_moe_plan_t plan, const void* const* x, const int32_t* const* topk_idx,
                            void* const* recv, int32_t* const* recv_meta, void* stream) {
  if (!plan || !x || !topk_idx || !recv) return PL_ERR_INVALID_ARG;
  if (!on_comm_device(plan->comm)) return PL_ERR_INVALID_ARG;
  const MoeGeo& g = plan->g;
  DispatchPtrs P;
  std::memset(&P, 0, sizeof(P));
  for (int r = 0; r < g.R; ++r) {
    if (!x[r] || !topk_idx[r] || !recv[r]) return PL_ERR_INVALID_ARG;
    if (((uintptr_t)x[r] & 15) || ((uintptr_t)recv[r] & 15) || ((uintptr_t)topk_idx[r] & 3)) return PL_ERR_ALIGNMENT;
    if (recv_meta && recv_meta[r] && ((uintptr_t)recv_meta[r] & 15)) return PL_ERR_ALIGNMENT;
    P.x[r] = x[r];
    P.idx[r] = topk_idx[r];
    P.recv[r] = recv[r];
    P.meta[r] = recv_meta ? recv_meta[r] : nullptr;
  }
  if (plan->small_rows) {
    if (!launch_small(P, g, SmallParams{plan->small_rows, g.K, g.epr, 0, nullptr, nullptr}, false, static_cast<cudaStream_t>(stream))) return PL_ERR_CUDA;
    g_launches.fetch_add(1);
    plan->dispatched = true;
    return PL_OK;
  }
  const int launched = launch_dispatch(plan, P, g, plan->fused, static_cast<cudaStream_t>(stream));
  if (!launched) return PL_ERR_CUDA;
  g_launches.fetch_add(launched);
  plan->dispatched = true;
  return PL_OK;
}

// Launched overlapped like the register executor: both kernels wait for everything in front before they read.
static bool launch_combine(pl_moe_plan_t plan, const CombinePtrs& P, MoeGeo g, cudaStream_t cs) {
  const uint32_t units = g.row_bytes >> 4, parts = (units + kCombinePartThreads - 1) / kCombinePartThreads;
  const unsigned long long n_tok = (unsigned long long)g.R * g.T, turns = (unsigned long long)plan->sm_count * plan->combine_per_sm;
  const bool by_parts = combine_by_parts(n_tok, units, g.K, turns) && n_tok * parts <= 0x7FFFFFFFull;
  const uint32_t width = ((units + parts - 1) / parts + 31) / 32 * 32, tokens = parts > 1 ? 1u : kCombinePartThreads / width;
  if (!by_parts) return launch_after(true, moe_combine_kernel, dim3((unsigned)std::min(n_tok, turns)), kCombineThreads, 0, cs, P, g);
  g.parts = parts;
  g.width = width;
  return launch_after(true, g.K <= 2 ? moe_combine_parts_kernel<2> : g.K <= 4 ? moe_combine_parts_kernel<4> : moe_combine_parts_kernel<8>,
                      dim3((unsigned)((n_tok * parts + tokens - 1) / tokens)), tokens * width, 0, cs, P, g);
}

static pl_status_t combine_impl(pl_moe_plan_t plan, const void* const* y, const float* const* gates, void* const* out,
                                void* stream, bool gates_are_logits) {
  if (!plan || !y || !gates || !out) return PL_ERR_INVALID_ARG;
  if (plan->comm->dtype != PL_BF16) return PL_ERR_UNSUPPORTED;
  if (!plan->dispatched) return PL_ERR_INVALID_ARG;
  if (!on_comm_device(plan->comm)) return PL_ERR_INVALID_ARG;
  MoeGeo g = plan->g;  // by value: the mode below belongs to this call, not to the plan
  g.gates_are_logits = gates_are_logits ? 1 : 0;
  CombinePtrs P;
  std::memset(&P, 0, sizeof(P));
  for (int r = 0; r < g.R; ++r) {
    if (!y[r] || !gates[r] || !out[r]) return PL_ERR_INVALID_ARG;
    if (((uintptr_t)y[r] & 15) || ((uintptr_t)out[r] & 15) || ((uintptr_t)gates[r] & 3)) return PL_ERR_ALIGNMENT;
    P.y[r] = y[r];
    P.gates[r] = gates[r];
    P.out[r] = out[r];
  }
  if (!launch_combine(plan, P, g, static_cast<cudaStream_t>(stream))) return PL_ERR_CUDA;
  g_launches.fetch_add(1);
  return PL_OK;
}

pl_status_t pl_moe_combine(pl_moe_plan_t plan, const void* const* y, const float* const* gates, void* const* out,
                           void* stream) {
  return combine_impl(plan, y, gates, out, stream, false);
}

pl_status_t pl_moe_combine_logits(pl_moe_plan_t plan, const void* const* y, const float* const* logits,
                                  void* const* out, void* stream) {
  return combine_impl(plan, y, logits, out, stream, true);
}

pl_status_t pl_moe_plan_read(pl_moe_plan_t plan, int32_t* pos, int64_t* counts, int64_t* expert_counts, void* stream) {
  if (!plan) return PL_ERR_INVALID_ARG;
  const MoeGeo& g = plan->g;
  if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) { cudaGetLastError(); return PL_ERR_CUDA; }
  int flags[4] = {0, 0, 0, 0};
  bool ok = cudaMemcpy(flags, g.flags, 16, cudaMemcpyDeviceToHost) == cudaSuccess;
  if (ok && flags[3]) {  // the grid barrier of the bookkeeping kernel gave up: report once, clear barrier state
    flags[2] = 1;
    ok = cudaMemset(g.flags + 3, 0, 4 + 8) == cudaSuccess;  // flags[3] and the two barrier words behind it
  }
  if (ok && pos) ok = cudaMemcpy(pos, g.pos, (size_t)g.R * g.T * g.K * 4, cudaMemcpyDeviceToHost) == cudaSuccess;
  if (ok && counts) ok = cudaMemcpy(counts, g.counts, (size_t)g.R * g.R * 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  if (ok && expert_counts) ok = cudaMemcpy(expert_counts, g.ecounts, (size_t)g.R * g.E * 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  if (!ok) { cudaGetLastError(); return PL_ERR_CUDA; }
  if (flags[2]) return PL_ERR_TIMEOUT;
  if (flags[1]) return PL_ERR_INVALID_ARG;
  if (flags[0]) return PL_ERR_OVERFLOW;
  return PL_OK;
}

pl_status_t pl_moe_dispatch_dedup(pl_moe_plan_t plan, const void* const* x, const int32_t* const* topk_idx,
                                  void* const* recv, int32_t* const* recv_meta, void* stream) {
  if (!plan || !x || !topk_idx || !recv) return PL_ERR_INVALID_ARG;
  if (!on_comm_device(plan->comm)) return PL_ERR_INVALID_ARG;
  const MoeGeo& g = plan->g;
  const MoeGeo& d = plan->gd;
  DispatchPtrs P;
  DeriveParams D{};
  std::memset(&P, 0, sizeof(P));
  for (int r = 0; r < g.R; ++r) {
    if (!x[r] || !topk_idx[r] || !recv[r]) return PL_ERR_INVALID_ARG;
    if (((uintptr_t)x[r] & 15) || ((uintptr_t)recv[r] & 15) || ((uintptr_t)topk_idx[r] & 3)) return PL_ERR_ALIGNMENT;
    if (recv_meta && recv_meta[r] && ((uintptr_t)recv_meta[r] & 15)) return PL_ERR_ALIGNMENT;
    D.idx[r] = topk_idx[r];
    P.x[r] = x[r];
    P.idx[r] = plan->d_ridx + (size_t)r * g.T * d.K;  // the derived per-rank routing
    P.recv[r] = recv[r];
    P.meta[r] = recv_meta ? recv_meta[r] : nullptr;
  }
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  if (plan->small_rows_dedup) {
    for (int r = 0; r < g.R; ++r) P.idx[r] = topk_idx[r];
    if (!launch_small(P, d, SmallParams{plan->small_rows_dedup, g.K, g.epr, 0, plan->d_ridx, plan->d_rmask}, true, cs)) return PL_ERR_CUDA;
    g_launches.fetch_add(1);
    plan->dispatched_dedup = true;
    return PL_OK;
  }
  const long long n_tok = (long long)g.R * g.T;
  D.R = g.R;
  D.T = g.T;
  D.K = g.K;
  D.epr = g.epr;
  D.KR = d.K;
  D.ridx = plan->d_ridx;
  D.rmask = plan->d_rmask;
  if (!launch_after(true, moe_derive_ranks_kernel, dim3((unsigned)((n_tok + 255) / 256)), 256, 0, cs, D))
    return PL_ERR_CUDA;
  const int launched = launch_dispatch(plan, P, d, plan->fused_dedup, cs);
  if (!launched) return PL_ERR_CUDA;
  g_launches.fetch_add(1 + launched);
  plan->dispatched_dedup = true;
  return PL_OK;
}

pl_status_t pl_moe_combine_dedup(pl_moe_plan_t plan, const void* const* z, void* const* out, void* stream) {
  if (!plan || !z || !out) return PL_ERR_INVALID_ARG;
  if (plan->comm->dtype != PL_BF16) return PL_ERR_UNSUPPORTED;
  if (!plan->dispatched_dedup) return PL_ERR_INVALID_ARG;
  if (!on_comm_device(plan->comm)) return PL_ERR_INVALID_ARG;
  const MoeGeo& d = plan->gd;
  CombinePtrs P;
  std::memset(&P, 0, sizeof(P));
  for (int r = 0; r < d.R; ++r) {
    if (!z[r] || !out[r]) return PL_ERR_INVALID_ARG;
    if (((uintptr_t)z[r] & 15) || ((uintptr_t)out[r] & 15)) return PL_ERR_ALIGNMENT;
    P.y[r] = z[r];
    P.gates[r] = plan->d_ones;  // the expert layer has already applied the gates
    P.out[r] = out[r];
  }
  if (!launch_combine(plan, P, d, static_cast<cudaStream_t>(stream))) return PL_ERR_CUDA;
  g_launches.fetch_add(1);
  return PL_OK;
}

pl_status_t pl_moe_plan_read_dedup(pl_moe_plan_t plan, int32_t* pos, int64_t* counts, void* stream) {
  if (!plan) return PL_ERR_INVALID_ARG;
  const MoeGeo& d = plan->gd;
  if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) { cudaGetLastError(); return PL_ERR_CUDA; }
  int flags[4] = {0, 0, 0, 0};
  bool ok = cudaMemcpy(flags, d.flags, 16, cudaMemcpyDeviceToHost) == cudaSuccess;
  if (ok && flags[3]) {
    flags[2] = 1;
    ok = cudaMemset(d.flags + 3, 0, 4 + 8) == cudaSuccess;
  }
  if (ok && counts) ok = cudaMemcpy(counts, d.counts, (size_t)d.R * d.R * 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  if (ok && pos) {
    const size_t tk = (size_t)d.R * d.T * d.K;
    std::vector<int32_t> ridx(tk), rpos(tk);
    ok = cudaMemcpy(ridx.data(), plan->d_ridx, tk * 4, cudaMemcpyDeviceToHost) == cudaSuccess &&
         cudaMemcpy(rpos.data(), d.pos, tk * 4, cudaMemcpyDeviceToHost) == cudaSuccess;
    if (ok) {
      const size_t n_tok = (size_t)d.R * d.T;
      for (size_t i = 0; i < n_tok * d.R; ++i) pos[i] = -1;
      for (size_t t = 0; t < n_tok; ++t)
        for (int j = 0; j < d.K; ++j)
          if (ridx[t * d.K + j] >= 0) pos[t * d.R + ridx[t * d.K + j]] = rpos[t * d.K + j];
    }
  }
  if (!ok) { cudaGetLastError(); return PL_ERR_CUDA; }
  if (flags[2]) return PL_ERR_TIMEOUT;
  if (flags[1]) return PL_ERR_INVALID_ARG;
  if (flags[0]) return PL_ERR_OVERFLOW;
  return PL_OK;
}

}  // extern "C"
