// Launch wrappers implemented in the .cu files (kept free of kernel code so that host-only
// translation units can include it).
#pragma once
#include <cuda_runtime.h>

#include "pl_internal.h"

namespace pl {

// register (ld/st) executor
cudaError_t launch_exec(int dtype, const ExecParams& P, int grid, int threads, cudaStream_t stream);
int exec_max_ctas_per_sm(int dtype, int threads);
int exec_max_threads();

// TMA (bulk-copy, shared-memory ring) executor
cudaError_t launch_exec_tma(int dtype, const ExecParams& P, int grid, cudaStream_t stream);
int exec_tma_max_ctas_per_sm(int dtype, int stages, uint32_t stage_bytes);
// threads per CTA of the two variants: general (16 consumer warps) and pipelined reduce (12)
int exec_tma_threads(bool pipelined);
size_t exec_tma_smem_bytes(int stages, uint32_t stage_bytes);

// layered direct-fused all-reduces with one op per queue and layer (`cluster`: the grid is one
// thread-block cluster and the cluster barrier takes the place of the flags)
cudaError_t launch_layers(int dtype, const ExecParams& P, const LayerParams& Y, int grid, int threads, bool cluster, cudaStream_t stream);
// whether such a cluster can be resident; raises the limit its launches need, so it goes before the first of them
bool layers_cluster_fits(int dtype, int R, bool hook, int grid, int threads);

// schedules without flags, one CTA per tile
FlatLaunch flat_launch(int R, bool reduce, bool all, bool bulk, uint32_t hook, uint64_t total_units, int sm_count);
cudaError_t launch_flat(int dtype, const FlatParams& P, const FlatLaunch& F, cudaStream_t stream);

// ring schedules, a cluster per tile.  ring_prepare: clusters that can be resident at once (0: none)
int ring_prepare(int dtype, int R, const RingLaunch& L);
cudaError_t launch_ring(int dtype, const RingHopParams& P, const RingLaunch& L, cudaStream_t stream);

// packet executor (latency path): rank = cluster of ctas_per_rank CTAs
cudaError_t launch_exec_packet(int dtype, const PacketParams& P, int threads, bool overlap, cudaStream_t stream);
int exec_packet_max_groups(int dtype, int ctas_per_rank, int threads);
int exec_packet_max_units_per_thread();
int exec_packet_max_threads();

}  // namespace pl
