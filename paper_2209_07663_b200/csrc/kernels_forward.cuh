// Forward: cuckoo look-up of every ID of a batch, gather of the rows that
// exist, sum per bag in ID order (the HashTable look-up operation of Section 2.1 serving the
// parameter pull of Section 2.2; sum pooling per bag).
#pragma once

#include "kernels_dedup.cuh"
#include "table_layout.cuh"

namespace mono {

// The rest of a read-only look-up that missed the preferred cell, for pulls that are bound by latency: the
// seven other keys of both buckets are asked for together.
__device__ inline bool thread_lookup_rest(const TableView& tv, unsigned long long id, unsigned stash_hw, unsigned long long* meta) {
  const unsigned long long h0 = tv.hash0(id);
  const uint32_t first = (uint32_t)(h0 >> 62);
  const Cell* b0 = tv.cells + (h0 & tv.bucket_mask) * kCellsPerBucket;
  const Cell* b1 = tv.cells + tv.bucket1(id) * kCellsPerBucket;
  unsigned long long k0[3], k1[4];
#pragma unroll
  for (uint32_t k = 0; k < 3; ++k) k0[k] = __ldg(&b0[(first + 1u + k) & 3u].key);
#pragma unroll
  for (uint32_t k = 0; k < 4; ++k) k1[k] = __ldg(&b1[k].key);
  const Cell* at = nullptr;
#pragma unroll
  for (uint32_t k = 0; k < 4; ++k) if (k1[k] == id) at = b1 + k;
#pragma unroll
  for (uint32_t k = 0; k < 3; ++k) if (k0[k] == id) at = b0 + ((first + 1u + k) & 3u);
  for (unsigned i = 0; at == nullptr && i < stash_hw; ++i)
    if (__ldg(&tv.stash[i].key) == id) at = tv.stash + i;
  if (at) *meta = __ldg(&at->meta);
  return at != nullptr;
}

// Read-only look-up by one thread.  An insertion tries the cell named by the
// top bits of the hash first, so that cell is read first and alone; the other
// three cells of the bucket, the second bucket and the stash follow only on a
// miss.  Returns true and the metadata when the ID is tracked.
__device__ inline bool thread_lookup(const TableView& tv, unsigned long long id, unsigned stash_hw,
                                     unsigned long long* meta) {
  const unsigned long long h0 = tv.hash0(id);
  const Cell* b = tv.cells + (h0 & tv.bucket_mask) * kCellsPerBucket;
  const uint32_t first = (uint32_t)(h0 >> 62);
  const Cell c0 = load_cell_ro(b + first);
  if (c0.key == id) { *meta = c0.meta; return true; }
  // the other three cells of the bucket, requested together (named values, not an array: an
  // indexed array here ends up in local memory)
  const Cell c1 = load_cell_ro(b + ((first + 1u) & 3u));
  const Cell c2 = load_cell_ro(b + ((first + 2u) & 3u));
  const Cell c3 = load_cell_ro(b + ((first + 3u) & 3u));
  if (c1.key == id) { *meta = c1.meta; return true; }
  if (c2.key == id) { *meta = c2.meta; return true; }
  if (c3.key == id) { *meta = c3.meta; return true; }
  b = tv.cells + tv.bucket1(id) * kCellsPerBucket;
  const Cell d0 = load_cell_ro(b), d1 = load_cell_ro(b + 1), d2 = load_cell_ro(b + 2), d3 = load_cell_ro(b + 3);
  if (d0.key == id) { *meta = d0.meta; return true; }
  if (d1.key == id) { *meta = d1.meta; return true; }
  if (d2.key == id) { *meta = d2.meta; return true; }
  if (d3.key == id) { *meta = d3.meta; return true; }
  for (unsigned i = 0; i < stash_hw; ++i) {
    const Cell s = load_cell_ro(tv.stash + i);
    if (s.key == id) { *meta = s.meta; return true; }
  }
  return false;
}

// The same look-up for a caller that goes on to modify the entry: it also returns where
// the entry is (index into cells[], or n_cells + i for stash cell i; kNoCell if nowhere).
// Its kernel stores metadata into the cells it reads, so the loads are ordinary (coherent)
// 16-byte loads, not the read-only path.
constexpr unsigned long long kNoCell = 0xFFFFFFFFFFFFFFFFull;

__device__ inline unsigned long long thread_locate(const TableView& tv, unsigned long long id, unsigned stash_hw,
                                                   unsigned long long* meta) {
  const unsigned long long h0 = tv.hash0(id);
  const unsigned long long base0 = (h0 & tv.bucket_mask) * kCellsPerBucket;
  const uint32_t first = (uint32_t)(h0 >> 62);
  const Cell c0 = load_cell_whole(tv.cells + base0 + first);
  if (c0.key == id) { *meta = c0.meta; return base0 + first; }
  // On a miss the keys of the other three cells are asked for together, then those of the second
  // bucket: most of these IDs are new to the table and in neither bucket, and a warp waits for its
  // slowest lane, so eight reads one after the other were what the look-up took (a key store at load 0.89:
  // 50 -> 42 us for 300 000 distinct IDs; all seven keys at once read a line more than most need: 48).
  unsigned long long at = kNoCell, k0[3], k1[4];
#pragma unroll
  for (uint32_t k = 0; k < 3; ++k) k0[k] = tv.cells[base0 + ((first + 1u + k) & 3u)].key;
#pragma unroll
  for (uint32_t k = 0; k < 3; ++k) if (k0[k] == id) at = base0 + ((first + 1u + k) & 3u);
  if (at == kNoCell) {
    const unsigned long long base1 = tv.bucket1(id) * kCellsPerBucket;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) k1[k] = tv.cells[base1 + k].key;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) if (k1[k] == id) at = base1 + k;
  }
  if (at != kNoCell) { *meta = tv.cells[at].meta; return at; }
  for (unsigned i = 0; i < stash_hw; ++i) {
    const Cell s = load_cell_whole(tv.stash + i);
    if (s.key == id) { *meta = s.meta; return (tv.bucket_mask + 1) * kCellsPerBucket + i; }
  }
  return kNoCell;
}

// ---- pooling ---------------------------------------------------------------

constexpr int kPoolThreads = 256;

// A lane's share of a row: VW consecutive floats, moved as one access of 16 bytes (VW = 4) or 32 (VW = 8).
template <int VW>
struct Vec { float x[VW]; };

template <int VW>
__device__ __forceinline__ Vec<VW> load_ro(const float* p) {
  Vec<VW> v;
  if constexpr (VW == 8) {
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(v.x[0]), "=f"(v.x[1]), "=f"(v.x[2]), "=f"(v.x[3]), "=f"(v.x[4]), "=f"(v.x[5]), "=f"(v.x[6]), "=f"(v.x[7]) : "l"(p));
  } else {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    v.x[0] = q.x; v.x[1] = q.y; v.x[2] = q.z; v.x[3] = q.w;
  }
  return v;
}
template <int VW>
__device__ __forceinline__ void store_vec(float* p, const Vec<VW>& v) {
  if constexpr (VW == 8) {
    asm volatile("st.global.v8.f32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"
                 :: "f"(v.x[0]), "f"(v.x[1]), "f"(v.x[2]), "f"(v.x[3]), "f"(v.x[4]), "f"(v.x[5]), "f"(v.x[6]), "f"(v.x[7]), "l"(p) : "memory");
  } else {
    *reinterpret_cast<float4*>(p) = make_float4(v.x[0], v.x[1], v.x[2], v.x[3]);
  }
}

// sum += rows idx[0..K), in that order; all K loads are issued before the first add.
template <int K, int G, int NV, int VW>
__device__ __forceinline__ void add_rows(const float* __restrict__ rows, uint32_t dim, const uint32_t* idx, int gl, Vec<VW> (&sum)[NV]) {
  uint32_t row[K];
#pragma unroll
  for (int k = 0; k < K; ++k) row[k] = idx[k];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const uint32_t c = (gl + v * G) * VW;
    if (c < dim) {
      Vec<VW> x[K];
#pragma unroll
      for (int k = 0; k < K; ++k) x[k] = load_ro<VW>(rows + (size_t)row[k] * 2u * dim + c);
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int e = 0; e < VW; ++e) sum[v].x[e] += x[k].x[e];
    }
  }
}

// dst[0..dim) = sum of the rows idx[0..n), in that order, by a group of G lanes.  The rows go in
// batches of K, what is left in one batch of its exact size: no
// per-row tests (an ID without a row points at the table's all-zero row), no loads for padding.
template <int K, int G, int NV, int VW>
__device__ __forceinline__ void pool_bag(const float* __restrict__ rows, uint32_t dim, const uint32_t* idx, uint32_t n, int gl, float* __restrict__ dst) {
  Vec<VW> sum[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int e = 0; e < VW; ++e) sum[v].x[e] = 0.f;
  uint32_t i = 0;
  for (; i + K <= n; i += K) add_rows<K, G, NV, VW>(rows, dim, idx + i, gl, sum);
  switch (n - i) {
    case 11: if constexpr (K > 11) add_rows<11, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 10: if constexpr (K > 10) add_rows<10, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 9: if constexpr (K > 9) add_rows<9, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 8: if constexpr (K > 8) add_rows<8, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 7: if constexpr (K > 7) add_rows<7, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 6: if constexpr (K > 6) add_rows<6, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 5: if constexpr (K > 5) add_rows<5, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 4: if constexpr (K > 4) add_rows<4, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 3: add_rows<3, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 2: add_rows<2, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    case 1: add_rows<1, G, NV, VW>(rows, dim, idx + i, gl, sum); break;
    default: break;
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const uint32_t c = (gl + v * G) * VW;
    if (c < dim) store_vec<VW>(dst + c, sum[v]);
  }
}

// Where a tile's rows come from.  resolve(first, n, dst) leaves the row of occurrence first + i in
// dst[i], with all threads of the block; an ID without a row gets the table's all-zero row, one
// past the capacity.
//
// A batch that was not announced: every occurrence is looked up in the key store.  The preferred
// cells of P occurrences are asked for together; the rest of a look-up follows only on a miss.
template <int P, bool TOGETHER>
struct ProbedRows {
  const TableView& tv;
  const unsigned long long* __restrict__ ids;
  unsigned stash_hw;
  __device__ __forceinline__ void resolve(long long first, uint32_t n, uint32_t* dst) const {
    for (uint32_t i = threadIdx.x; i < n; i += kPoolThreads * P) {
      unsigned long long id[P];
      Cell c[P];
#pragma unroll
      for (int k = 0; k < P; ++k) id[k] = i + k * kPoolThreads < n ? ids[first + i + k * kPoolThreads] : kEmptyKey;
#pragma unroll
      for (int k = 0; k < P; ++k) {
        c[k] = empty_cell();
        if (id[k] != kEmptyKey) {
          const unsigned long long h0 = tv.hash0(id[k]);
          c[k] = load_cell_ro(tv.cells + (h0 & tv.bucket_mask) * kCellsPerBucket + (h0 >> 62));
        }
      }
#pragma unroll
      for (int k = 0; k < P; ++k) {
        if (i + k * kPoolThreads >= n) continue;
        bool found = id[k] != kEmptyKey;
        if (found && c[k].key != id[k]) found = TOGETHER ? thread_lookup_rest(tv, id[k], stash_hw, &c[k].meta) : thread_lookup(tv, id[k], stash_hw, &c[k].meta);
        dst[i + k * kPoolThreads] = found && meta_resident(c[k].meta) ? meta_row(c[k].meta) : (uint32_t)tv.capacity;
      }
    }
  }
};

// A batch that was announced: every distinct ID was looked up then, and its slot of the per-call
// set holds its row.  While it is there, every occurrence of a repeated ID is filed for the push:
// its bag goes into the ID's segment of bag_of_sorted[], at the occurrence's rank.
template <int P>
struct FiledRows {
  const Work& wk;
  long long n_bags;
  uint32_t zero_row;
  // An occurrence's slot of the per-call set: key (x, y), start of the ID's segment, row.
  __device__ __forceinline__ uint4 slot_of(const uint2 o) const {
    if (o.x == kNoSlot || !MONO_INDEX_OK(wk.error_bits, o.x, wk.n_slots())) return make_uint4(0u, 0u, kNoSegment, kNoRow);
    return __ldg(reinterpret_cast<const uint4*>(wk.bset + o.x));
  }
  __device__ __forceinline__ void file(const uint2 o, const uint4 bs, uint32_t bag) const {
    if (bs.z != kNoSegment && bag < n_bags && MONO_INDEX_OK(wk.error_bits, (unsigned long long)bs.z + o.y, wk.max_ids))
      wk.bag_of_sorted[bs.z + o.y] = bag;                                         // (an ID that occurs once has no segment)
  }
  // The filing alone, of one occurrence.
  __device__ __forceinline__ void file(long long j) const {
    const uint2 o = wk.occ[j];
    const uint4 bs = slot_of(o);
    if (bs.z != kNoSegment) file(o, bs, wk.occ_bag[j]);
  }
  __device__ __forceinline__ void resolve(long long first, uint32_t n, uint32_t* dst) const {
    for (uint32_t i = threadIdx.x; i < n; i += kPoolThreads * P) {
      uint2 o[P];
      uint4 bs[P];
      uint32_t bag[P];
#pragma unroll
      for (int k = 0; k < P; ++k) {
        const uint32_t at = i + k * kPoolThreads;
        o[k] = at < n ? wk.occ[first + at] : make_uint2(kNoSlot, 0u);
        bag[k] = at < n ? wk.occ_bag[first + at] : 0xFFFFFFFFu;
      }
#pragma unroll
      for (int k = 0; k < P; ++k) bs[k] = slot_of(o[k]);
#pragma unroll
      for (int k = 0; k < P; ++k) {
        const uint32_t at = i + k * kPoolThreads;
        if (at >= n) continue;
        file(o[k], bs[k], bag[k]);
        dst[at] = bs[k].w != kNoRow ? bs[k].w : zero_row;
      }
    }
  }
};

// Forward: one block per tile of consecutive bags (the HashTable look-up of Section 2.1 serving the
// parameter pull of Section 2.2).
//   1. all threads resolve the tile's IDs to rows, into shared memory: independent random reads, as
//      many in flight as the block has threads;
//   2. lane groups of G (chosen from dim, so that a lane owns NV vectors of VW floats) each add up
//      a bag at a time, in ID order, so that the fp32 sum has one fixed order.
// Bound by the latency of scattered reads (more than half of the warp-cycles per issue wait for memory, with DRAM at
// about half and L1 at two thirds of their peaks on the largest announced batch: profiles/), so everything here
// is about reads in flight:
//  - blocks of one kernel are in both steps at any time, which two kernels one after the other never
//    are, and the rows' indices do not travel through memory;
//  - the tile's bags are put in order of length (a counting sort of at most 256 entries in shared
//    memory), because the groups of a warp wait for the longest of their bags; warps take the next
//    bags from a counter;
//  - bags of one ID, which come last, are copies: kCopies of them in flight per group;
//  - rows of more than 128 columns go as 32-byte accesses, one per lane instead of two.
// Measured against a kernel for step 1 and another for step 2: 1.6 M bags of 64 columns 403 -> 340 us,
// 213 000 of 32 columns 43.8 -> 31.5, 41 000 long bags of 200 columns 116 -> 87, one request of 208
// bags (latency) 6.1 -> 4.7; one warp per tile instead of a block 357 / 36 / 98 us.
// Tile sizes: pool_tile() on the host.
constexpr int kPoolBags = 256;          // most bags of a tile: one per thread
constexpr int kPoolIds = 1024;          // most IDs of a tile whose rows fit the shared memory; a tile with more goes through `spill`
constexpr int kPoolBins = 32;           // bag lengths told apart when the tile's bags are put in order

struct PoolTile {
  uint32_t row[kPoolIds];
  uint32_t begin[kPoolBags];            // first ID of the bag
  uint32_t len[kPoolBags];
  uint32_t count[kPoolBins];            // bags per length, then the place of the first of them
  uint8_t order[kPoolBags];             // the tile's bags, longest first
  unsigned int next;
};

template <int K, int G, int NV, int VW, typename Rows>
__device__ __forceinline__ void pool_tile_body(const TableView& tv, const Rows& rows, uint32_t* __restrict__ spill, long long n_ids,
                                               const long long* __restrict__ offsets, long long n_bags, float* __restrict__ out,
                                               uint32_t tile_bags, uint32_t vblock, PoolTile& sh) {
  constexpr int kGroups = 32 / G;
  const int lane = threadIdx.x & 31, gl = lane % G, grp = lane / G;
  const uint32_t dim = tv.dim;
  const long long b0 = (long long)vblock * tile_bags;
  const uint32_t nb = (uint32_t)(n_bags - b0 < tile_bags ? n_bags - b0 : tile_bags);
  if (threadIdx.x < kPoolBins) sh.count[threadIdx.x] = 0;
  if (threadIdx.x == 0) sh.next = 0;
  long long lo = 0, hi = 0;
  bool ok = true;
  if (threadIdx.x < nb) {
    lo = offsets[b0 + threadIdx.x];
    hi = offsets[b0 + threadIdx.x + 1];
    ok = bag_ok(lo, hi, n_ids);
    if (!ok) { atomicOr(&tv.st->error_bits, 4u /* MONO_DEV_BAD_OFFSETS */); lo = hi = 0; }      // flagged, and treated as empty
  }
  const bool well_formed = __syncthreads_and(ok) != 0;
  const uint32_t n = (uint32_t)(hi - lo);                                        // (a call has fewer than 2^31 IDs)
  const uint32_t bin = n < kPoolBins ? kPoolBins - 1 - n : 0;                    // longest first
  uint32_t place = 0;
  const uint32_t* idx;
  {
    const long long first = offsets[b0], last = offsets[b0 + nb];
    const bool fits = well_formed && last - first <= kPoolIds;
    uint32_t* dst = fits ? sh.row : spill;
    idx = dst;
    if (threadIdx.x < nb) {
      place = atomicAdd(&sh.count[bin], 1u);
      sh.begin[threadIdx.x] = (uint32_t)(fits ? lo - first : lo);
      sh.len[threadIdx.x] = n;
    }
    // the tile's IDs are one run, unless its offsets are malformed: then bag by bag
    const uint32_t runs = well_formed ? 1u : nb;
    for (uint32_t r = 0; r < runs; ++r) {
      long long from = first, to = last;
      if (!well_formed) {
        from = offsets[b0 + r];
        to = offsets[b0 + r + 1];
        if (!bag_ok(from, to, n_ids)) continue;
      }
      rows.resolve(from, (uint32_t)(to - from), dst + (fits ? 0 : from));
    }
  }
  __syncthreads();
  if (threadIdx.x < kPoolBins) {
    const uint32_t c = sh.count[threadIdx.x];
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += v;
    }
    sh.count[threadIdx.x] = incl - c;
  }
  __syncthreads();
  if (threadIdx.x < nb) sh.order[sh.count[bin] + place] = (uint8_t)threadIdx.x;
  __syncthreads();
  const uint32_t n_sums = sh.count[kPoolBins - 2];                               // bags of two IDs and more
  for (;;) {
    uint32_t i = 0;
    if (lane == 0) i = atomicAdd(&sh.next, (unsigned)kGroups);
    i = __shfl_sync(0xFFFFFFFFu, i, 0);
    if (i >= n_sums) break;
    i += grp;
    if (i < n_sums) {
      const uint32_t b = sh.order[i];
      pool_bag<K, G, NV, VW>(tv.rows, dim, idx + sh.begin[b], sh.len[b], gl, out + (b0 + b) * (long long)dim);
    }
    __syncwarp();
  }
  constexpr int kCopies = VW == 8 ? 2 : 4;
  for (uint32_t i = n_sums + ((threadIdx.x >> 5) * kGroups + grp) * kCopies; i < nb; i += (kPoolThreads / 32) * kGroups * kCopies) {
    uint32_t b[kCopies], r[kCopies];
#pragma unroll
    for (int k = 0; k < kCopies; ++k) {
      b[k] = i + k < nb ? sh.order[i + k] : 0xFFFFFFFFu;
      r[k] = b[k] != 0xFFFFFFFFu && sh.len[b[k]] ? idx[sh.begin[b[k]]] : (uint32_t)tv.capacity;
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint32_t c = (gl + v * G) * VW;
      if (c < dim) {
        Vec<VW> x[kCopies];
#pragma unroll
        for (int k = 0; k < kCopies; ++k) x[k] = load_ro<VW>(tv.rows + (size_t)r[k] * 2u * dim + c);
#pragma unroll
        for (int k = 0; k < kCopies; ++k) if (b[k] != 0xFFFFFFFFu) store_vec<VW>(out + (b0 + b[k]) * (long long)dim + c, x[k]);
      }
    }
  }
}

// Blocks per SM and look-ups in flight per thread: narrow rows, whose groups are small, do best with
// all the warps an SM holds (213 000 bags of 32 columns 31.5 us against 36.9 with six blocks), wider
// ones with the registers for more rows in flight (long bags of 64 columns 22.7 against 25 us).  Rows of more than
// 512 columns in 32-byte accesses need 80 registers, three blocks: at the 64 of four they spill, and the pull of 2048 bags of
// up to 64 IDs of 1024 columns took 54 us against 40, of 65 536 bags of up to 8 IDs 106 against 98.  (In 16-byte
// accesses four stay: three are 50 -> 40 us for the long bags of 516 columns, but 72.7 -> 76.8 for the many short ones.)
// DEEP, for long bags in batches that are bound by the latency of their rows rather than of their look-ups (pools_deep() on the
// host has the rule and the figures): half as many rows again in flight per lane group, at four blocks.
template <int G, int NV, int VW, bool DEEP> constexpr int pool_blocks_per_sm() { return DEEP ? 4 : NV * VW == 32 && VW == 8 ? 3 : NV > 1 ? 4 : G <= 8 ? 8 : 6; }
template <int VW, bool DEEP> __host__ __device__ constexpr int pool_batch() { return VW == 8 ? (DEEP ? 6 : 4) : (DEEP ? 12 : 8); }
// (Filing is a chain of two reads, a batch's own record and its ID's slot of the per-call set: four at a time, 8 M IDs of
// 64 columns 1365 -> 1346 us per step, timed in turn; at the 32 registers of the narrow rows they spill, 4 M IDs 343 -> 359.)
template <int G> constexpr int kProbesInFlight = G <= 8 ? 1 : 2;
template <int G> constexpr int kFiledInFlight = G <= 8 ? 1 : 4;

// TOGETHER (launch_pool): of a look-up that misses the preferred cell, the rest at once.  It needs
// the registers of six blocks per SM, which narrow rows only have to spare in a batch of one wave of blocks
// (one request of 208 bags 5.7 -> 4.8 us; 213 000 bags 31.8 -> 32.8, so larger ones look on bucket by bucket).
template <int G, int NV, int VW, bool TOGETHER, bool DEEP>
__global__ void __launch_bounds__(kPoolThreads, (TOGETHER && G <= 8 ? 6 : pool_blocks_per_sm<G, NV, VW, DEEP>()))
probe_pool_kernel(TableView tv, const unsigned long long* __restrict__ ids, uint32_t* __restrict__ spill, long long n_ids,
                  const long long* __restrict__ offsets, long long n_bags, float* __restrict__ out, uint32_t tile_bags) { after_previous_kernel();
  __shared__ PoolTile sh;
  pool_tile_body<pool_batch<VW, DEEP>(), G, NV, VW>(tv, ProbedRows<kProbesInFlight<G>, TOGETHER>{tv, ids, tv.st->stash_hw}, spill, n_ids, offsets, n_bags, out, tile_bags, blockIdx.x, sh);
}

template <int G, int NV, int VW, bool DEEP>
__global__ void __launch_bounds__(kPoolThreads, (pool_blocks_per_sm<G, NV, VW, DEEP>()))
gather_pool_kernel(TableView tv, Work wk, uint32_t* __restrict__ spill, long long n_ids, const long long* __restrict__ offsets,
                 long long n_bags, float* __restrict__ out, uint32_t tile_bags) { after_previous_kernel();
  __shared__ PoolTile sh;
  pool_tile_body<pool_batch<VW, DEEP>(), G, NV, VW>(tv, FiledRows<kFiledInFlight<G>>{wk, n_bags, (uint32_t)tv.capacity}, spill, n_ids, offsets, n_bags, out, tile_bags, blockIdx.x, sh);
}

}  // namespace mono
