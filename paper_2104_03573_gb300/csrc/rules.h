// Rules the launches and kernels follow that are plain arithmetic on sizes:
// C++ without CUDA headers, so that the host compiler builds them too.
#pragma once

#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define MCBTE_RULE __host__ __device__ __forceinline__
#else
#define MCBTE_RULE inline
#endif

namespace mcbte {

// Last event of a tail round that begins after event e and covers `span`
// events: never past the run's last one, so that it lies beyond e (the round
// makes progress) until e + 1 = max_events ends the particle.  e + span alone
// wraps within `span` of 2^32.
MCBTE_RULE uint32_t round_end(uint32_t e, uint32_t span, uint32_t max_events) {
  const uint32_t left = max_events - 1u - e;
  return e + (span < left ? span : left);
}

// Bins up to which an FP32 relaxation takes one Philox block; the tail computes
// draws ahead only there.
constexpr int kOneBlockBins = 65536;

// Shared-memory plan of the persistent FP32 tracers.
struct SmemPlan {
  int relax_in_smem;   // alias records ~ C/tau in shared memory
  int binf_in_smem;    // per-bin {v, 1/v, Lambda} in shared memory
  int qbin_in_smem;    // frequency-resolved flux privatised per block
  int cells_in_smem;   // cell tallies privatised per block
  int tail_slots;      // the tail's draw slots per warp, 0 without (first in the layout)
  int grad_in_smem;    // the gradient accumulator privatised per block
  int snap_in_smem;    // a pore-hit snapshot per thread (measure-valued d/dp; after the warps' records)
  int batch_slots;     // the main kernel's emitted batch: slots per warp, 0 without (first in the layout)
  size_t bytes;
};

// Tables and per-block tallies by use per event: the relaxation alias records
// and the per-bin constants (every relaxation), the cell tallies (every
// flight), the per-bin flux (every relaxation period), the gradient
// accumulator (every period of a gradient pass), the pore-hit snapshots of the
// measure-valued d/dp (64 bytes per thread).  Each is placed while room
// remains in `budget`.
inline SmemPlan plan_tables(int n_bins, int n_geoms, int n_cells, int per_bin, size_t budget, int grad_acc = 0,
                            int snap_threads = 0) {
  SmemPlan S{0, 0, 0, 0, 0, 0, 0, 0, 0};
  auto place = [&](bool wanted, size_t bytes) {
    const bool in = wanted && S.bytes + bytes <= budget;
    if (in) S.bytes += bytes;
    return in ? 1 : 0;
  };
  const size_t n = (size_t)n_bins;
  S.relax_in_smem = place(true, n * 16);
  S.binf_in_smem = place(true, n * 16);
  S.cells_in_smem = place(n_cells > 0 && n_geoms == 1, ((size_t)n_cells * 8 + 4) * 8);
  S.qbin_in_smem = place(per_bin != 0 && n_geoms == 1, n * 8);
  S.grad_in_smem = place(grad_acc != 0, n * 8);
  S.snap_in_smem = place(snap_threads > 0, (size_t)snap_threads * 64);
  return S;
}

// Bytes the steady tracers' tables and tallies may take, and all that a block
// lays out (of 227 KB, the rest for the static shared memory).  What lies
// between them is kept for the records every warp has of its own (the tail's
// draw slots), at half their count at least, so that no table size leaves a
// warp without them.
constexpr size_t kTableBytes = 200 * 1024;
constexpr size_t kPlanBytes = 226 * 1024;

// The tail kernel's draw slots.  64 per warp where they fit beside the tables,
// else 32; without any a lone particle draws inline and its events take two to
// three times as long (2e5 particles, per-bin flux: pore film of 4650 bins
// 17.8 ms without, 6.7 with 64; of 5100 bins 6.6 with 32.  1e5 particles,
// measure-valued gradient of 5400 bins: 51.2 ms without, 14.8 with).
constexpr int kTailThreads = 256;
constexpr int kTailSlots = 64;
constexpr size_t kTailSlotBytes = 80;

inline SmemPlan plan_tail(int n_bins, int n_geoms, int n_cells, int per_bin, int grad_acc, int snap_threads) {
  SmemPlan S = plan_tables(n_bins, n_geoms, n_cells, per_bin, kTableBytes, grad_acc, snap_threads);
  const size_t slot = (size_t)(kTailThreads / 32) * kTailSlotBytes;   // one in every warp
  if (n_bins > kOneBlockBins) return S;
  S.tail_slots = S.bytes + kTailSlots * slot <= kPlanBytes ? kTailSlots : kTailSlots / 2;
  S.bytes += (size_t)S.tail_slots * slot;
  return S;
}

// The main kernel's emitted batches (Refill, EmitBatch): 32 slots per warp
// where they fit beside the tables, else 16.  A table or tally in global memory
// costs far more (silicon-like slab, 2e6 particles, 50 cells: 5700 bins
// 139 ms with 32 slots and the cells outside, 5.5 with 16; 4650 bins 13.4 ms
// with the per-bin flux outside, 5.8).  Blocks of 1024 threads take none: their
// 64 registers spill with them, into the L1 whose room they take (the same
// slab, 1e7 particles, 3000 / 4200 / 7800 bins: 18.7 / 24.9 / 27.3 ms with,
// 16.9 / 17.3 / 17.9 without).
constexpr int kUnbatchedThreads = 1024;   // and more
constexpr int kBatchSlots = 32;
constexpr size_t kRefillBytes = 48, kBatchBytes = 1296, kBatchBytesExt = 1424;   // a record holds 32 slots

inline SmemPlan plan_main(int threads, bool ext, int n_bins, int n_geoms, int n_cells, int per_bin, int grad_acc,
                          int snap_threads) {
  SmemPlan S = plan_tables(n_bins, n_geoms, n_cells, per_bin, kTableBytes, grad_acc, snap_threads);
  if (threads >= kUnbatchedThreads) return S;
  const size_t warps = (size_t)(threads / 32), rec = ext ? kBatchBytesExt : kBatchBytes;
  auto bytes = [&](int slots) { return warps * kRefillBytes + (warps * (size_t)slots / kBatchSlots) * rec; };
  S.batch_slots = S.bytes + bytes(kBatchSlots) <= kPlanBytes ? kBatchSlots : kBatchSlots / 2;
  S.bytes += bytes(S.batch_slots);
  return S;
}

}  // namespace mcbte
