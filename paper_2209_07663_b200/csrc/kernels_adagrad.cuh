// Backward, last phase: per distinct ID that owns a row, sum the pooled
// gradients of its occurrences' bags (fp64 accumulation, one rounding to fp32)
// and apply one Adagrad step to the row, in place.  This is the parameter push
// of Section 2.2 for the sparse rows; the optimizer itself is not named in the
// paper.
//
// Three cases, by how often the ID occurs in the batch:
// Every repeated ID has a segment of bag_of_sorted[] that lists the bags of its
// occurrences (filed by the pull, gather_pool_kernel, when the batch was announced, else by
// file_segments_kernel inside the push).
//  - once (most distinct IDs of a long-tailed batch): its gradient is the
//    pooled gradient of its one bag, so the row is updated straight from that
//    bag's gradient row;
//  - 2 .. kSegChunk times: one lane group gathers the gradient rows of the
//    segment's bags;
//  - more (the head of the Zipf distribution: one ID can own several percent of
//    a batch): the segment is cut into parts of kSegChunk that separate groups
//    reduce into fp64 partial sums, which are added up in a fixed tree.
#pragma once

#include "kernels_dedup.cuh"
#include "kernels_forward.cuh"
#include "kernels_table.cuh"

namespace mono {

struct D4 { double x, y, z, w; };

__device__ inline void add4(D4& a, const float4 v) { a.x += (double)v.x; a.y += (double)v.y; a.z += (double)v.z; a.w += (double)v.w; }

// acc += G*G;  w -= lr*G/(sqrt(acc)+eps), each operation rounded to fp32 on its
// own (no fused multiply-add), so the result does not depend on contraction.
__device__ inline void adagrad4(float4& w, float4& a, const float4 g, float lr, float eps) {
  const float gx = g.x, gy = g.y, gz = g.z, gw = g.w;
  a.x = __fadd_rn(a.x, __fmul_rn(gx, gx));
  a.y = __fadd_rn(a.y, __fmul_rn(gy, gy));
  a.z = __fadd_rn(a.z, __fmul_rn(gz, gz));
  a.w = __fadd_rn(a.w, __fmul_rn(gw, gw));
  w.x = __fsub_rn(w.x, __fdiv_rn(__fmul_rn(lr, gx), __fadd_rn(__fsqrt_rn(a.x), eps)));
  w.y = __fsub_rn(w.y, __fdiv_rn(__fmul_rn(lr, gy), __fadd_rn(__fsqrt_rn(a.y), eps)));
  w.z = __fsub_rn(w.z, __fdiv_rn(__fmul_rn(lr, gz), __fadd_rn(__fsqrt_rn(a.z), eps)));
  w.w = __fsub_rn(w.w, __fdiv_rn(__fmul_rn(lr, gw), __fadd_rn(__fsqrt_rn(a.w), eps)));
}

// Load (or, for a row admitted in this call, create) the row, update, store.
__device__ inline void update_row(const TableView& tv, uint32_t row_word, unsigned long long id,
                                  uint32_t c4, const D4& g) {
  const uint32_t row = row_word & ~kFreshBit;
  float4* pw = reinterpret_cast<float4*>(tv.w_row(row)) + c4;
  float4* pa = reinterpret_cast<float4*>(tv.acc_row(row)) + c4;
  float4 w, a;
  if (row_word & kFreshBit) {
    w = init_vec(tv, id, c4);
    a = make_float4(tv.init_acc, tv.init_acc, tv.init_acc, tv.init_acc);
  } else {
    w = *pw;
    a = *pa;
  }
  adagrad4(w, a, make_float4((float)g.x, (float)g.y, (float)g.z, (float)g.w), tv.lr, tv.eps);
  *pw = w;
  *pa = a;
}

// The per-call set must be empty again when the push ends.  Its primary tier is wiped as a whole
// (clear_primary: a streaming write costs less than one scattered store per ID); an ID
// that overflowed into the secondary tier, which is far larger and almost empty, has its slot
// emptied by the kernel that updates its row.
__device__ inline void clear_overflow_slot(const Work& wk, uint32_t slot) {
  if (slot > wk.primary_mask) {
    BatchSlot e; e.key = kEmptyKey; e.a = 0; e.b = 0;
    wk.bset[slot] = e;
  }
}

__device__ inline void clear_primary(const Work& wk, uint32_t vblock, uint32_t vgrid) {
  const uint32_t n = wk.primary_mask + 1u;
  ulonglong2 e; e.x = kEmptyKey; e.y = 0ull;
  for (uint32_t i = vblock * blockDim.x + threadIdx.x; i < n; i += vgrid * blockDim.x)
    *reinterpret_cast<ulonglong2*>(wk.bset + i) = e;
}
// Sum of the grad rows of bags bag_of_sorted[begin], [begin + STEP], ... below end for the NV column
// vectors this lane owns.  Eight independent row loads in flight per trip.
template <int G, int NV, int STEP = 1>
__device__ inline void reduce_segment(const Work& wk, const float* __restrict__ grad, long long n_bags,
                                      uint32_t dim, int gl, uint32_t begin, uint32_t end, D4 (&s)[NV]) {
  constexpr int kDepth = NV == 1 ? 8 : 4;
  uint32_t i = begin;
  for (; i + (kDepth - 1) * STEP < end; i += kDepth * STEP) {
    uint32_t b[kDepth];
#pragma unroll
    for (int k = 0; k < kDepth; ++k) b[k] = wk.bag_of_sorted[i + k * STEP];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint32_t c4 = gl + v * G;
      if (c4 * 4u < dim) {
        float4 x[kDepth];
#pragma unroll
        for (int k = 0; k < kDepth; ++k)
          x[k] = b[k] < n_bags ? __ldg(reinterpret_cast<const float4*>(grad + (size_t)b[k] * dim) + c4)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kDepth; ++k) add4(s[v], x[k]);
      }
    }
  }
  if (i < end) {
    // the ragged tail, again with all its loads issued before the adds
    uint32_t b[kDepth];
#pragma unroll
    for (int k = 0; k < kDepth; ++k) b[k] = i + k * STEP < end ? wk.bag_of_sorted[i + k * STEP] : 0xFFFFFFFFu;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint32_t c4 = gl + v * G;
      if (c4 * 4u < dim) {
        float4 x[kDepth];
#pragma unroll
        for (int k = 0; k < kDepth; ++k)
          x[k] = b[k] < n_bags ? __ldg(reinterpret_cast<const float4*>(grad + (size_t)b[k] * dim) + c4)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kDepth; ++k) add4(s[v], x[k]);
      }
    }
  }
}

// The same for one lane group of a grouped call's block, whose pointers are not constants of the launch: the lanes read the
// bags' numbers together and hand them round, a load and its address less per row (64 tables: the row updates 60.5 ->
// 56 us; a table's own launch, whose pointers are, gains nothing: 8 M IDs 642 -> 655, 1 M the same).
template <int G, int NV>
__device__ __forceinline__ void reduce_segment_together(const Work& wk, const float* __restrict__ grad, long long n_bags, uint32_t dim,
                                                        int gl, uint32_t begin, uint32_t end, D4 (&s)[NV]) {
  constexpr int kDepth = NV == 1 ? 8 : 4;
  constexpr int kEach = kDepth > G ? kDepth / G : 1;                      // numbers a lane reads per chunk
  const unsigned mask = G == 32 ? 0xFFFFFFFFu : ((1u << (G & 31)) - 1u) << ((threadIdx.x & 31) / G * G);
  for (uint32_t i = begin; i < end; i += G * kEach) {                     // the same for the group
    uint32_t mine[kEach];
#pragma unroll
    for (int r = 0; r < kEach; ++r) mine[r] = i + r * G + gl < end ? wk.bag_of_sorted[i + r * G + gl] : 0xFFFFFFFFu;
#pragma unroll 1
    for (int k0 = 0; k0 < G * kEach && i + k0 < end; k0 += kDepth) {
      uint32_t b[kDepth];
#pragma unroll
      for (int k = 0; k < kDepth; ++k) b[k] = __shfl_sync(mask, mine[kEach > 1 ? k / G : 0], kEach > 1 ? k % G : k0 + k, G);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint32_t c4 = gl + v * G;
        if (c4 * 4u < dim) {
          float4 x[kDepth];
#pragma unroll
          for (int k = 0; k < kDepth; ++k)
            x[k] = b[k] < n_bags ? __ldg(reinterpret_cast<const float4*>(grad + (size_t)b[k] * dim) + c4)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int k = 0; k < kDepth; ++k) add4(s[v], x[k]);
        }
      }
    }
  }
}

// The filing pass of a push whose batch was not announced, or not pulled since (otherwise the pull
// has filed the bags, FiledRows): one pass over the occurrences.
__device__ inline void file_segments_body(const Work& wk, long long n_ids, long long n_bags, uint32_t vblock, uint32_t vgrid) {
  const long long stride = (long long)vgrid * blockDim.x;
  const FiledRows<1> rows{wk, n_bags, 0u};
  for (long long j = (long long)vblock * blockDim.x + threadIdx.x; j < n_ids; j += stride) rows.file(j);
}
__global__ void __launch_bounds__(256)
file_segments_kernel(Work wk, long long n_ids, long long n_bags) { after_previous_kernel();
  file_segments_body(wk, n_ids, n_bags, blockIdx.x, gridDim.x);
}

// ---- the row updates of a push: one kernel -----------------------------------
// Blocks of one grid take different kinds of work, the heaviest first: parts of long segments, short
// segments, what occurs once.  None waits for another, so the blocks of the next kind fill the SMs
// as those of the one before run out, and a small batch has all of them resident at once.  Measured
// against eight kernels on two streams (clear, expand, reduce twice, singles, fold, combine, finish),
// whole step: 20 000 IDs 54 -> 36 us, 1 M IDs 180 -> 153, 4 M drifting 360 -> 348, 8 M 1404 -> 1395; against the
// three kinds one after the other in every block, 47 / 163 / 411 / 1437.
// What bounds it: gradient rows gathered at random for the first two kinds (latency; ten blocks of 128
// threads per SM at 48 registers: eight at 64 measured 3 % of a step slower, twelve spill; rows of 132 to 256 columns
// seven at 72, 198 -> 167 us per step against four), HBM for the third.

// The lanes that work on one part of a long segment: PG of them, PG / G lane groups that take turns at the
// rows to add up.
template <int PG, int G>
struct Team {
  static constexpr int kGroups = PG / G;
  int lane = threadIdx.x % PG, gl = threadIdx.x % G, grp = threadIdx.x % PG / G;
  unsigned mask = PG == 32 ? 0xFFFFFFFFu : ((1u << (PG & 31)) - 1u) << ((threadIdx.x & 31) / PG * PG);

  // the groups have each summed a share: afterwards every one of them has the whole
  template <int NV>
  __device__ __forceinline__ void add_groups(D4 (&s)[NV]) const {
#pragma unroll
    for (int o = G; o < PG; o <<= 1)
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        s[v].x += __shfl_xor_sync(mask, s[v].x, o);
        s[v].y += __shfl_xor_sync(mask, s[v].y, o);
        s[v].z += __shfl_xor_sync(mask, s[v].z, o);
        s[v].w += __shfl_xor_sync(mask, s[v].w, o);
      }
  }

  // s = src[0] + src[stride] + ... (n of them).  They were written by other blocks: read past L1.
  template <int NV>
  __device__ __forceinline__ void sum_partials(const double* src, uint32_t n, size_t stride, uint32_t dim, D4 (&s)[NV]) const {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint32_t c4 = gl + v * G;
      s[v] = D4{0.0, 0.0, 0.0, 0.0};
      if (c4 * 4u < dim) {
#pragma unroll 4
        for (uint32_t i = grp; i < n; i += kGroups) {
          const double2* p = reinterpret_cast<const double2*>(src + i * stride) + c4 * 2;
          const double2 x = __ldcg(p), y = __ldcg(p + 1);
          s[v].x += x.x; s[v].y += x.y; s[v].z += y.x; s[v].w += y.y;
        }
      }
    }
    add_groups<NV>(s);
  }

  // The long ID that part p belongs to: the last one whose first part is not after p, PG places at a time.
  __device__ __forceinline__ uint32_t owner_of_part(const Work& wk, uint32_t n_long, uint32_t p) const {
    uint32_t lo = 0, n = n_long;                                         // it is in [lo, lo + n)
    while (n > 1) {
      const uint32_t step = (n + PG - 1) / PG, at = lane * step;
      const bool before = at < n && wk.long_part0[lo + at] <= p;
      const uint32_t c = __popc(__ballot_sync(mask, before)) - 1;
      lo += c * step;
      n = min(step, n - c * step);
    }
    return lo;
  }
};

// The parts of the long segments.  A team of PG lanes sums one part into fp64 partial sums in scratch.
// Partial sums are added up in a tree: the team that finishes the last of kFanIn neighbours adds
// them up and goes on to the next level, and the one that reaches the top updates the row.  The
// order of every addition is fixed by the parts' numbers, whoever does it.  (A tree, because one ID
// can own a tenth of a batch: with 64 neighbours at a time and then all the rest, adding up the
// 11 000 parts of such an ID was a serial chain of 50 us.)
template <int PG, int G, int NV, bool TOGETHER>
__device__ inline void reduce_parts(const TableView& tv, const Work& wk, const float* __restrict__ grad, long long n_bags,
                                    bool ordered, unsigned long long longs, uint32_t vblock, uint32_t vgrid) {
  const uint32_t n_parts = (uint32_t)longs, n_long = (uint32_t)(longs >> 32);
  const Team<PG, G> team;
  const uint32_t teams = (vgrid * blockDim.x) / PG;
  for (uint32_t item = (vblock * blockDim.x + threadIdx.x) / PG; item < n_parts; item += teams) {
    const uint32_t p = ordered ? wk.part_order[item] : item;
    if (!MONO_INDEX_OK(wk.error_bits, p, wk.max_parts)) continue;
    const uint32_t li = ordered ? wk.part_u[p] : team.owner_of_part(wk, n_long, p);
    if (!MONO_INDEX_OK(wk.error_bits, li, wk.max_long)) continue;
    const uint32_t u = wk.long_u[li], p0 = wk.long_part0[li];
    const uint32_t row_word = wk.urow[u], m = wk.ulen[u], seg = wk.useg[u];
    if (row_word == kNoRow) continue;                                    // no row: gradient dropped, by every part
    uint32_t k = p - p0;
    const uint32_t begin = seg + k * kSegChunk, end = (k + 1) * kSegChunk < m ? begin + kSegChunk : seg + m;
    if (!MONO_INDEX_OK(wk.error_bits, (unsigned long long)end - 1, wk.max_ids)) continue;
    D4 s[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = D4{0.0, 0.0, 0.0, 0.0};
    if constexpr (TOGETHER) reduce_segment_together<G, NV>(wk, grad, n_bags, tv.dim, team.gl, begin, end, s);
    else reduce_segment<G, NV, PG / G>(wk, grad, n_bags, tv.dim, team.gl, begin + team.grp, end, s);
    team.template add_groups<NV>(s);
    const uint32_t parts = (m + kSegChunk - 1) / kSegChunk;
    bool top = true;
    for (uint32_t level = 0, step = 1; step < parts; ++level, step *= kFanIn) {
      // s is the sum of the parts [k, k + step) of the ID, cut off at the last: leave it where the level above finds it
      double* dst = wk.partials + (size_t)(p0 + k) * tv.dim;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const uint32_t c4 = team.gl + v * G;
        if (team.grp == 0 && c4 * 4u < tv.dim) {
          reinterpret_cast<double2*>(dst)[c4 * 2] = make_double2(s[v].x, s[v].y);
          reinterpret_cast<double2*>(dst)[c4 * 2 + 1] = make_double2(s[v].z, s[v].w);
        }
      }
      k = k / (step * kFanIn) * (step * kFanIn);
      const uint32_t want = min(kFanIn, (parts - k + step - 1) / step);
      uint32_t* counter = wk.part_done + p0 + k;                         // five bits per level: kFanIn at most
      __threadfence();
      __syncwarp(team.mask);
      uint32_t before = 0;
      if (team.lane == 0) before = atomicAdd(counter, 1u << (5 * level));
      before = __shfl_sync(team.mask, before, 0, PG) >> (5 * level) & 31u;
      if (before != want - 1u) { top = false; break; }
      __threadfence();
      if (team.lane == 0) atomicSub(counter, want << (5 * level));       // zero again for the next call
      team.template sum_partials<NV>(wk.partials + (size_t)(p0 + k) * tv.dim, want, (size_t)step * tv.dim, tv.dim, s);
    }
    if (!top) continue;
    const unsigned long long id = wk.uid[u];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint32_t c4 = team.gl + v * G;
      if (team.grp == 0 && c4 * 4u < tv.dim) update_row(tv, row_word, id, c4, s[v]);
    }
    __syncwarp(team.mask);
  }
}

// The repeated IDs: a team of PG lanes each, which reduces the segment, if it is short, and updates the row.
// (Measured against one packed record per repeated ID, read a trip ahead: the separate arrays were 2 %
// of a step faster on the largest configuration.)
template <int PG, int G, int NV, bool TOGETHER>
__device__ inline void reduce_short(const TableView& tv, const Work& wk, const float* __restrict__ grad, long long n_bags,
                                    uint32_t n, uint32_t vblock, uint32_t vgrid) {
  const Team<PG, G> team;
  const uint32_t teams = (vgrid * blockDim.x) / PG;
  for (uint32_t item = (vblock * blockDim.x + threadIdx.x) / PG; item < n; item += teams) {
    const uint32_t u = wk.multi_list[item];
    if (team.lane == 0) clear_overflow_slot(wk, wk.uslot[u]);
    const uint32_t m = wk.ulen[u];
    const uint32_t row_word = wk.urow[u];
    if (row_word == kNoRow || m > kSegChunk) continue;                   // no row: gradient dropped; long: in parts
    const uint32_t begin = wk.useg[u];
    D4 s[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = D4{0.0, 0.0, 0.0, 0.0};
    if constexpr (TOGETHER) reduce_segment_together<G, NV>(wk, grad, n_bags, tv.dim, team.gl, begin, begin + m, s);
    else reduce_segment<G, NV, PG / G>(wk, grad, n_bags, tv.dim, team.gl, begin + team.grp, begin + m, s);
    team.template add_groups<NV>(s);
    const unsigned long long id = wk.uid[u];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const uint32_t c4 = team.gl + v * G;
      if (team.grp == 0 && c4 * 4u < tv.dim) update_row(tv, row_word, id, c4, s[v]);
    }
  }
}

// The IDs that occur once in the batch (most distinct IDs of a long-tailed batch): the
// gradient of such an ID is the pooled gradient of its one bag, so its row is updated
// straight from there.  One warp per 32 consecutive distinct IDs, which are numbered in
// the order the batch first shows them, so the gradient rows are read roughly in order;
// the lanes whose ID occurs once and has a row are served in turn by lane groups of G,
// which read the bag's gradient row, the table row and its accumulator, and write both
// back updated.
template <int G, int NV>
__device__ inline void update_singletons(const TableView& tv, const Work& wk, const float* __restrict__ grad,
                                              long long n_bags, uint32_t n, uint32_t vblock, uint32_t vgrid) {
  constexpr int kGroups = 32 / G;
  // Two rows of a lane group in flight (1.3 M single rows of 64 columns 5 % faster, whole step 1395 -> 1380 us; 99 000 of
  // 100 columns 137 -> 130); rows of several vectors per lane have their own loads to overlap.
  constexpr int kRows = NV == 1 ? 2 : 1;
  const int lane = threadIdx.x & 31;
  const int gl = lane % G, grp = lane / G;
  const uint32_t n_warps = (vgrid * blockDim.x) >> 5;
  const uint32_t n_rounds = (n + 31) / 32;
  unsigned int n_single = 0;
  for (uint32_t r = (vblock * blockDim.x + threadIdx.x) >> 5; r < n_rounds; r += n_warps) {
    const uint32_t u = r * 32 + lane;
    uint32_t row_word = kNoRow, bag = 0;
    unsigned long long id = 0;
    bool single = false;
    if (u < n && wk.ulen[u] == 1u) {
      const uint32_t slot = wk.uslot[u];
      row_word = wk.urow[u];
      if (row_word != kNoRow && MONO_INDEX_OK(wk.error_bits, wk.uocc[u], wk.max_ids)) {
        bag = wk.occ_bag[wk.uocc[u]];
        single = bag < n_bags;
        if (row_word & kFreshBit) id = wk.uid[u];
      }
      clear_overflow_slot(wk, slot);                     // (after the loads: a store in between would hold them back)
    }
    unsigned todo = __ballot_sync(0xFFFFFFFFu, single);
    n_single += __popc(todo);
    while (todo) {
      // the next kGroups * kRows flagged lanes, kRows for each lane group; all their loads before the first store
      uint32_t rw[kRows], bg[kRows];
      unsigned long long key[kRows];
      bool mine[kRows];
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        int src = -1;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
          const int l = todo ? __ffs(todo) - 1 : -1;
          if (l >= 0) todo &= todo - 1;
          if (g == grp) src = l;
        }
        mine[k] = src >= 0;
        const int from = src < 0 ? 0 : src;
        rw[k] = __shfl_sync(0xFFFFFFFFu, row_word, from);
        bg[k] = __shfl_sync(0xFFFFFFFFu, bag, from);
        key[k] = __shfl_sync(0xFFFFFFFFu, id, from);
      }
      float4 x[kRows][NV], w[kRows][NV], a[kRows][NV];
#pragma unroll
      for (int k = 0; k < kRows; ++k)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const uint32_t c4 = gl + v * G;
          if (!mine[k] || c4 * 4u >= tv.dim) continue;
          const uint32_t row = rw[k] & ~kFreshBit;
          x[k][v] = __ldg(reinterpret_cast<const float4*>(grad + (size_t)bg[k] * tv.dim) + c4);
          if (!(rw[k] & kFreshBit)) {
            w[k][v] = reinterpret_cast<const float4*>(tv.w_row(row))[c4];
            a[k][v] = reinterpret_cast<const float4*>(tv.acc_row(row))[c4];
          }
        }
#pragma unroll
      for (int k = 0; k < kRows; ++k)
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const uint32_t c4 = gl + v * G;
          if (!mine[k] || c4 * 4u >= tv.dim) continue;
          const uint32_t row = rw[k] & ~kFreshBit;
          if (rw[k] & kFreshBit) {
            w[k][v] = init_vec(tv, key[k], c4);
            a[k][v] = make_float4(tv.init_acc, tv.init_acc, tv.init_acc, tv.init_acc);
          }
          adagrad4(w[k][v], a[k][v], x[k][v], tv.lr, tv.eps);
          reinterpret_cast<float4*>(tv.w_row(row))[c4] = w[k][v];
          reinterpret_cast<float4*>(tv.acc_row(row))[c4] = a[k][v];
        }
    }
  }
  if (lane == 0 && n_single) atomicAdd(&tv.st->sum_single_resident, (unsigned long long)n_single);
}
constexpr int kRowThreads = 128;
constexpr uint32_t kFewParts = 4096;     // a warp for each is resident
constexpr uint32_t kHardlyAny = 256;
// How the grid is shared out: blocks [0, parts) take the parts, the next `shorts` the short segments,
// the rest what occurs once.
struct RowGrid { uint32_t parts, shorts, singles; };

template <int G, int NV, bool FEW>
__device__ __forceinline__ void update_rows_body(const TableView& tv, const Work& wk, const float* __restrict__ grad, long long n_bags,
                                                 bool ordered, const RowGrid& grid, uint32_t vblock) {
  if (vblock < grid.parts) {
    const unsigned long long longs = wk.call->longs;
    // Few parts (they are resident all at once): a warp each, because the longest chain of loads is what
    // counts (step of 20 000 IDs 35.8 -> 28.4 us, of 135 000 56 -> 47).  Many: a lane group each, which
    // spends nothing on adding groups up (a warp each: 1 M IDs 154 -> 160 us, 4 M drifting 351 -> 370).
    // (A grouped call, whose tables share the SMs, has no use for it: FEW is false.)
    if (G < 32 && (!FEW || (uint32_t)longs > kFewParts)) reduce_parts<G, G, NV, !FEW>(tv, wk, grad, n_bags, ordered, longs, vblock, grid.parts);
    else reduce_parts<32, G, NV, !FEW && G == 32>(tv, wk, grad, n_bags, ordered, longs, vblock, grid.parts);
  } else if (vblock - grid.parts < grid.shorts) {
    // Likewise: up to 64 bags, eight or four at a time by a small lane group, are the longest chain of a small batch (20 000 IDs of 16
    // columns 10.1 -> 8.6 us, of 32 13.6 -> 13.2; with up to 8192 of them a warp each, 1 M IDs 55.3 -> 58.7).  Where
    // hardly any ID is repeated, adding the groups up is all it adds (160 IDs 6.1 -> 6.7).
    const uint32_t n_multi = wk.call->n_multi;
    if (G < 32 && (!FEW || n_multi > kFewParts || n_multi < kHardlyAny)) reduce_short<G, G, NV, !FEW>(tv, wk, grad, n_bags, n_multi, vblock - grid.parts, grid.shorts);
    else reduce_short<32, G, NV, !FEW && G == 32>(tv, wk, grad, n_bags, n_multi, vblock - grid.parts, grid.shorts);
  } else {
    update_singletons<G, NV>(tv, wk, grad, n_bags, wk.call->n_unique, vblock - grid.parts - grid.shorts, grid.singles);
    clear_primary(wk, vblock - grid.parts - grid.shorts, grid.singles);
  }
}
template <int G, int NV>
__global__ void __launch_bounds__(kRowThreads, NV == 1 ? 10 : NV == 2 ? 7 : 4)
update_rows_kernel(TableView tv, Work wk, const float* __restrict__ grad, long long n_bags, int ordered, RowGrid grid) {
  after_previous_kernel();
  update_rows_body<G, NV, true>(tv, wk, grad, n_bags, ordered != 0, grid, blockIdx.x);
}

}  // namespace mono
