// The host-only rules that pick an executor and its launch, callable from a test without a GPU.
#include <cstdio>
#include <vector>

#include "pl_internal.h"

using namespace pl;

extern "C" {

// Lowers a collective, lays its ops out for the flat executor and returns the number of spans (at most `cap`
// written as src_off, dst_off, units, source rank, destination rank; 255 = every rank), -1 if the ops are not of that
// form, -2 if the request is refused.
int t_flat_plan(int R, int dtype, int coll, int algo, uint64_t count, uint64_t chunk, const uint64_t* counts_v, int root, uint32_t hook,
                uint64_t* spans, int cap, int* reduce, int* all) {
  BuildRequest rq{};
  rq.R = R;
  rq.dtype = dtype;
  rq.coll = coll;
  rq.algo = algo;
  rq.count_per_rank = count;
  rq.chunk_bytes = chunk;
  rq.counts_v = counts_v;
  rq.root = root;
  rq.hook = hook;
  rq.sm_count = 148;
  rq.pol = default_policy(rq, 148);
  Lowered L;
  std::string err;
  if (lower(rq, &L, &err) != PL_OK) return -2;
  bool r = false, a = false;
  std::vector<FlatSpan> f;
  if (!flat_plan(L, R, dtype, &f, &r, &a)) return -1;
  *reduce = r;
  *all = a;
  for (int i = 0; i < (int)f.size() && i < cap; ++i) {
    spans[5 * i] = f[i].src_off;
    spans[5 * i + 1] = f[i].dst_off;
    spans[5 * i + 2] = f[i].units;
    spans[5 * i + 3] = f[i].ranks & 0xFFu;
    spans[5 * i + 4] = (f[i].ranks >> 8) & 0xFFu;
  }
  return (int)f.size();
}

int t_queues_faster(int R, int dtype, uint32_t hook, int algo, int reduce, int all, int tma, uint64_t message_bytes) {
  return queues_faster(R, dtype, hook, algo, reduce, all, tma, message_bytes);
}

int t_ring_folds(int R, int gather, uint64_t part_units) { return ring_folds(R, gather, part_units, 148); }

int t_flat_release(int R, int reduce, int all, int bulk, int run, uint64_t blocks) { return flat_release(R, reduce, all, bulk, run, blocks); }

int t_combine_by_parts(uint64_t n_tok, uint32_t units, int topk, uint64_t turns) { return combine_by_parts(n_tok, units, topk, turns); }

int t_small_dispatch_rows(int dedup, int R, int tokens, int topk, int experts, uint64_t row_bytes) {
  return (int)small_dispatch_rows(dedup, R, tokens, topk, experts, row_bytes, 148);
}

// bit 0: the layer executor runs it, bit 1: and asks for the next layer's lines
int t_layers(int R, uint64_t message_bytes, int hook) {
  return (layer_executor_faster(R, message_bytes, hook) ? 1 : 0) | (layer_asks_ahead(R, message_bytes) ? 2 : 0);
}

// 0 if the queues run the ring, else its threads, units per thread, tile and grid
int t_ring_shape(int R, int dtype, int reduce, int gather, uint64_t part_units, uint64_t chunk_bytes, int* shape) {
  RingLaunch L{};
  if (!ring_shape(R, dtype, reduce, gather, part_units, chunk_bytes, 148, &L)) return 0;
  shape[0] = L.threads;
  shape[1] = L.units;
  shape[2] = (int)L.tile;
  shape[3] = L.grid;
  return (int)L.smem_bytes;
}

// Spans of a folded ring: src_off, dst_off, units, first rank of the sum, destination rank (255 = every rank).
int t_ring_plan(int R, int gather, uint64_t part_units, uint64_t* spans) {
  std::vector<FlatSpan> f;
  ring_plan(R, gather, part_units, &f);
  for (size_t i = 0; i < f.size(); ++i) {
    const uint64_t row[5] = {f[i].src_off, f[i].dst_off, f[i].units, f[i].ranks >> 16, (f[i].ranks >> 8) & 0xFFu};
    for (int k = 0; k < 5; ++k) spans[5 * i + k] = row[k];
  }
  return (int)f.size();
}

// Whether spans (rows as t_flat_plan writes them) are a run, and the run's spans written over them.
int t_flat_run(uint64_t* spans, int n) {
  std::vector<FlatSpan> f;
  for (int i = 0; i < n; ++i) {
    const uint64_t* s = spans + 5 * i;
    f.push_back(FlatSpan{s[0], s[1], s[2], 0, (uint32_t)(s[3] | s[4] << 8)});
  }
  FlatRun run;
  if (!flat_run(f, &run)) return 0;
  for (uint64_t k = 0; k < (uint64_t)n; ++k) {
    const uint32_t ranks = run.ranks + (uint32_t)k * run.rank_step;
    const uint64_t row[5] = {k * run.src_step, k * run.dst_step, run.units, ranks & 0xFFu, ranks >> 8 & 0xFFu};
    for (int i = 0; i < 5; ++i) spans[5 * k + i] = row[i];
  }
  return 1;
}

// Validates a lowered schedule after a change to op `which`: 0 none, 1 another op with the same destination, 2 the op's
// output shortened by 16 bytes, 3 the op's destination moved up by 16 bytes.
int t_validate_changed(int R, int dtype, int coll, int algo, uint64_t count, uint64_t chunk, int n_layers, int which, int change, char* msg, int cap) {
  BuildRequest rq{};
  rq.R = R;
  rq.dtype = dtype;
  rq.coll = coll;
  rq.algo = algo;
  rq.count_per_rank = count;
  rq.chunk_bytes = chunk;
  rq.n_layers = n_layers;
  rq.sm_count = 148;
  rq.pol = default_policy(rq, 148);
  Lowered L;
  std::string err;
  if (lower(rq, &L, &err) != PL_OK) return -2;
  HostOp& op = L.ops[which];
  const HostOp copy = op;
  const int es = copy.kind == PL_OP_COPY ? 1 : elem_size(dtype);
  if (change == 2) op.count -= 16 / es;
  if (change == 3) op.dst.offset += 16, op.count -= 16 / es;
  if (change == 1) L.ops.insert(L.ops.begin() + which + 1, copy);
  assign_queues(&L, R, rq.pol.n_ctas);
  const pl_status_t st = validate(L, R, &err, false);
  std::snprintf(msg, (size_t)cap, "%s", err.c_str());
  return st;
}
}
