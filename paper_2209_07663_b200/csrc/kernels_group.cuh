// One launch over several tables (Section 3.1 of the Monolith paper: a production model
// holds many embedding tables of very uneven size, most of them far too small to fill a
// GPU on their own).  Every kernel of the hot path exists a second time as a grouped
// kernel: its grid is the concatenation of the grids the tables would have launched one by
// one, a block first finds the table it belongs to, and then runs the same body on that
// table's view, scratch and batch.  The bodies are the single-table kernels' own.
#pragma once

#include "kernels_adagrad.cuh"
#include "kernels_dedup.cuh"
#include "kernels_forward.cuh"
#include "kernels_table.cuh"

namespace mono {

// One table's share of a grouped call.
struct GroupItem {
  TableView tv;
  Work wk;
  const unsigned long long* ids;
  const long long* off;
  long long n_ids, n_bags;
  float* out;                    // lookup
  uint32_t* occ_row;             // lookup: where a tile's rows go that do not fit its block's shared memory
  const float* grad;             // push
  unsigned long long dedup_seed;
  uint32_t now;
  uint32_t prepared;             // lookup: 1 = rows from the per-call set (the batch was announced), 0 = from the key store
  uint32_t lane_class;           // 0..3: lane groups of 4 / 8 / 16 / 32 with one column vector per lane;
                                 // 4..6: 32 lanes with 2 / 4 / 8 vectors per lane
  uint32_t pool_wide;            // lookup: 32-byte accesses (classes 4..6 only)
  uint32_t tile_bags;            // lookup: bags per block
  RowGrid row_grid;              // push: the row updates' blocks
  uint32_t active;               // 0: the table takes no part in this call (empty batch)
};

// Which table a block of a grouped launch belongs to: start[i] .. start[i+1] are table i's
// blocks.  Returns the table and the block's number within it.  Every warp searches, 32 places at a time: one at a time was
// six reads one after the other for 64 tables, in every block of seven kernels (180 -> 176 us per step).
__device__ inline uint32_t find_table(const uint32_t* __restrict__ start, uint32_t n_tables, uint32_t block,
                                      uint32_t* vblock, uint32_t* vgrid) {
  uint32_t lo = 0, n = n_tables;                         // it is in [lo, lo + n), where start[lo] <= block
  while (n > 1) {
    const uint32_t step = (n + 31) / 32, at = (threadIdx.x & 31) * step;
    const bool before = at < n && __ldg(start + lo + at) <= block;
    const uint32_t c = __popc(__ballot_sync(0xFFFFFFFFu, before)) - 1;
    lo += c * step;
    n = min(step, n - c * step);
  }
  const uint32_t s0 = __ldg(start + lo), s1 = __ldg(start + lo + 1);
  *vblock = block - s0;
  *vgrid = s1 - s0;
  return lo;
}

// A grouped call's descriptors and block maps, from the host's pinned copy: n words, of which the smaller of the two
// buffers holds `room`.  (A copy by the DMA engine, and the way to it and from there to the next kernel, left the GPU
// idle for ten microseconds: 64 tables 199.5 -> 180 us per step, three calls.)
__global__ void __launch_bounds__(256)
group_upload_kernel(uint4* __restrict__ dst, const uint4* src, uint32_t n, uint32_t room, unsigned int* error_bits) { after_previous_kernel();
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && MONO_INDEX_OK(error_bits, i, room)) dst[i] = __ldcv(src + i);
}

// A block's table: its descriptor, `it`, is copied to shared memory (read where it lies, in global memory, its fields
// filled the registers and the kernels spilled: 64 tables 180.4 -> 178.9 us per step).
#define MONO_GROUP_PROLOGUE                                                              \
  after_previous_kernel();                                                               \
  uint32_t vblock, vgrid;                                                                \
  __shared__ GroupItem it;                                                               \
  {                                                                                      \
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(items + find_table(start, n_tables, blockIdx.x, &vblock, &vgrid)); \
    for (uint32_t i = threadIdx.x; i < sizeof(GroupItem) / 8; i += blockDim.x) reinterpret_cast<unsigned long long*>(&it)[i] = __ldg(src + i); \
  }                                                                                      \
  __syncthreads()

__global__ void __launch_bounds__(256)
group_fill_occ_bag_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  fill_occ_bag_body(it.off, it.n_bags, it.n_ids, it.wk.occ_bag, it.wk.call, vblock, vgrid);
}

__global__ void __launch_bounds__(kTileThreads, 6)
group_dedup_tile_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  dedup_tile_body(it.wk, it.ids, it.n_ids, it.off, it.n_bags, it.dedup_seed, vblock);
}

template <int MODE>
__global__ void __launch_bounds__(256, 6)
group_table_update_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  table_update_body<MODE>(it.tv, it.wk, it.now, vblock, vgrid);
}

__global__ void __launch_bounds__(256)
group_sketch_add_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  if (it.tv.sketch_depth) sketch_add_body(it.tv, it.wk, vblock, vgrid);
}

__global__ void __launch_bounds__(256)
group_table_insert_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  table_insert_body(it.tv, it.wk, it.now, vblock, vgrid);
}

// (of a push whose batch was not pulled since it was announced, or not announced)
__global__ void __launch_bounds__(256)
group_file_segments_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  file_segments_body(it.wk, it.n_ids, it.n_bags, vblock, vgrid);
}

// The kernels whose bodies are compiled per lane-group width.  A block's table decides the
// width, so the tables of a launch can have different dims.  WIDE = 0 covers dims up to 128
// (one 16-byte column vector per lane, classes 0..3) in one launch; the wider rows (classes
// 4..6), whose bodies need twice to four times the registers, get a launch of their own.
template <int WIDE, typename F>
__device__ inline void by_lane_class(uint32_t lane_class, F&& f) {
  if (WIDE == 0) {
    switch (lane_class) {
      case 0: f(std::integral_constant<int, 4>{}, std::integral_constant<int, 1>{}); break;
      case 1: f(std::integral_constant<int, 8>{}, std::integral_constant<int, 1>{}); break;
      case 2: f(std::integral_constant<int, 16>{}, std::integral_constant<int, 1>{}); break;
      case 3: f(std::integral_constant<int, 32>{}, std::integral_constant<int, 1>{}); break;
      default: break;
    }
  } else {
    switch (lane_class) {
      case 4: f(std::integral_constant<int, 32>{}, std::integral_constant<int, 2>{}); break;
      case 5: f(std::integral_constant<int, 32>{}, std::integral_constant<int, 4>{}); break;
      case 6: f(std::integral_constant<int, 32>{}, std::integral_constant<int, 8>{}); break;
      default: break;
    }
  }
}

// The rows of a table of the group, whose batch may have been announced or not.
struct AnyRows {
  const GroupItem& it;
  __device__ __forceinline__ void resolve(long long first, uint32_t n, uint32_t* dst) const {
    if (it.prepared) FiledRows<1>{it.wk, it.n_bags, (uint32_t)it.tv.capacity}.resolve(first, n, dst);
    else ProbedRows<1, false>{it.tv, it.ids, it.tv.st->stash_hw}.resolve(first, n, dst);
  }
};

// (Three blocks per SM for the wide rows, whose bodies share the widest one's registers: eight tables of 260 to 512 columns
// 72 -> 65 us with 8192 short bags each, 35 -> 33 with long bags, of 516 to 1024 columns 118 -> 107 and 59 -> 53,
// of 132 to 256 49 -> 47 and 22.5, against four.)
template <int WIDE>
__global__ void __launch_bounds__(kPoolThreads, WIDE ? 3 : 6)
group_pool_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  __shared__ PoolTile sh;                                // (one for all widths: a block has one)
  const auto pool = [&](auto g, auto nv, auto vw) {
    pool_tile_body<pool_batch<decltype(vw)::value, false>(), decltype(g)::value, decltype(nv)::value, decltype(vw)::value>(it.tv, AnyRows{it}, it.occ_row, it.n_ids, it.off, it.n_bags, it.out,
                                                                                 it.tile_bags, vblock, sh);
  };
  if (WIDE && it.pool_wide) {
    using W = std::integral_constant<int, 32>;
    using V8 = std::integral_constant<int, 8>;
    switch (it.lane_class) {
      case 4: pool(W{}, std::integral_constant<int, 1>{}, V8{}); break;
      case 5: pool(W{}, std::integral_constant<int, 2>{}, V8{}); break;
      case 6: pool(W{}, std::integral_constant<int, 4>{}, V8{}); break;
      default: break;
    }
    return;
  }
  by_lane_class<WIDE>(it.lane_class, [&](auto g, auto nv) { pool(g, nv, std::integral_constant<int, 4>{}); });
}

template <int WIDE>
__global__ void __launch_bounds__(kRowThreads, WIDE ? 4 : 8)
group_update_rows_kernel(const GroupItem* __restrict__ items, const uint32_t* __restrict__ start, uint32_t n_tables) {
  MONO_GROUP_PROLOGUE;
  by_lane_class<WIDE>(it.lane_class, [&](auto g, auto nv) {
    update_rows_body<decltype(g)::value, decltype(nv)::value, false>(it.tv, it.wk, it.grad, it.n_bags, false, it.row_grid, vblock);
  });
}

#undef MONO_GROUP_PROLOGUE

}  // namespace mono
