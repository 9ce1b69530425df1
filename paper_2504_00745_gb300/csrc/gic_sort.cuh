// gic_sort.cuh -- device side of a1 (the stable Morton sort): the passes of
// the LSD radix sort as CTA-wide functions over tiles, shared by gic_sort's
// kernels (one launch per pass) and by gic_step's rebuild kernel (all passes in
// one cooperative launch, a grid barrier between them).
//
// A CTA has NT = 256 or 128 threads (NT / 32 warps of kTile / NT chunks of 32 keys,
// kRadix / NT digits per thread).  The keys of a tile are loaded before the
// first of them is ranked: the ranking's warp votes would otherwise put one
// chunk's load latency after another's.
//
// Stability: inside a tile each warp ranks its consecutive chunks of 32 keys in
// order, warps own consecutive sub-ranges and tiles are offset by the counts
// of earlier tiles, so equal keys keep their input order in every pass.
//
// What one pass writes and a later one reads (keys, values, counts, totals,
// the permutation) has no __restrict__ and no read-only load: in the one-launch
// form another SM wrote it during the same kernel, before a grid barrier.
#pragma once

#include "gic_internal.cuh"

namespace gic {

constexpr int kTile = 1024;  // keys per tile (one CTA at a time)
constexpr int kRadix = 256;

struct SortLayout {
  int64_t n;
  int tiles;
  int passes;
  size_t off_keys_a, off_vals_a, off_keys_b, off_vals_b, off_counts, off_totals, total;
};

// The workspace of a sort of n granules on grid G.
SortLayout sort_layout(const DGrid& G, int64_t n);

__device__ __forceinline__ uint32_t digit_of(uint32_t key, int shift) { return (key >> shift) & (kRadix - 1); }

struct ScatterState {
  const int32_t* in_cell;
  const void* in_pos;
  const void* in_vel;
  const int32_t* in_id;
  int32_t* out_cell;
  void* out_pos;
  void* out_vel;
  int32_t* out_id;
  int32_t* perm;
  float4* out_posf;  // FP32 path: float copy of the sorted positions, or NULL
};

template <int NT>
struct SortShared {
  uint32_t warp_hist[NT / 32][kRadix];
  uint32_t base[kRadix];
  uint32_t scan[NT / 32];
  uint32_t carry;
};

// The CTA's exclusive scan of one value per thread; sh_scan holds a word per
// warp.  Two barriers.
template <int NT>
__device__ __forceinline__ uint32_t cta_exclusive(uint32_t v, uint32_t* sh_scan) {
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  uint32_t incl = v;
  for (int off = 1; off < 32; off <<= 1) {
    uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  __syncthreads();
  if (lane == 31) sh_scan[warp] = incl;
  __syncthreads();
  uint32_t wsum = 0;
  for (int w = 0; w < warp; ++w) wsum += sh_scan[w];
  return wsum + incl - v;
}

// Per-tile digit histogram of the tiles blockIdx.x, + gridDim.x, ...;
// counts[d * tiles + tile].  first: the keys come from the cells.
template <int NT>
__device__ __forceinline__ void sort_upsweep(SortShared<NT>& sh, int64_t n, int shift, bool first,
                                             const int32_t* __restrict__ cell, const uint32_t* keys, uint32_t* counts,
                                             int tiles) {
  constexpr int kChunks = kTile / NT;
  uint32_t* s_hist = sh.base;
  const int warp = threadIdx.x >> 5, lane = lane_id();
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    __syncthreads();  // the previous tile's counts are out
    for (int d = threadIdx.x; d < kRadix; d += NT) s_hist[d] = 0;
    __syncthreads();
    const int64_t base = (int64_t)tile * kTile + warp * (32 * kChunks) + lane;
    uint32_t key[kChunks];
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const int64_t idx = base + c * 32;
      key[c] = idx < n ? (first ? (uint32_t)cell[idx] : keys[idx]) : 0u;
    }
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const bool valid = base + c * 32 < n;
      const uint32_t k = first ? morton_of_cell((int32_t)key[c]) : key[c];
      uint32_t d = valid ? digit_of(k, shift) : 0xffffffffu;
      unsigned peers = __match_any_sync(0xffffffffu, d);
      if (valid && (peers & lanemask_lt()) == 0) atomicAdd(&s_hist[d], (uint32_t)__popc(peers));
    }
    __syncthreads();
    for (int d = threadIdx.x; d < kRadix; d += NT) counts[(int64_t)d * tiles + tile] = s_hist[d];
  }
}

// Digits of a scan that a CTA of NT threads takes at a time: a whole CTA per
// digit, or, when a digit has at most kWarpScanTiles tiles, a warp per digit.
constexpr int kWarpScanTiles = 256;

// Exclusive scan over the tiles of every digit; totals[d] = count of digit d.
// With table_head, CTA 0 also advances the cell-table epoch.
template <int NT>
__device__ __forceinline__ void sort_scan(SortShared<NT>& sh, uint32_t* counts, int tiles, uint32_t* totals,
                                          uint4* table_head) {
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  if (table_head && blockIdx.x == 0 && threadIdx.x == 0) {
    uint32_t e = table_head->x + 1u;
    table_head->x = e == 0u ? 1u : e;
  }
  if (tiles <= kWarpScanTiles) {
    for (int d = blockIdx.x * (NT / 32) + warp; d < kRadix; d += gridDim.x * (NT / 32)) {
      uint32_t* row = counts + (int64_t)d * tiles;
      uint32_t carry = 0;
      for (int base = 0; base < tiles; base += 32) {
        const int t = base + lane;
        const uint32_t v = t < tiles ? row[t] : 0u;
        uint32_t incl = v;
        for (int off = 1; off < 32; off <<= 1) {
          uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += o;
        }
        if (t < tiles) row[t] = carry + incl - v;
        carry += __shfl_sync(0xffffffffu, incl, 31);
      }
      if (lane == 0) totals[d] = carry;
    }
    return;
  }
  constexpr int kPer = 4;  // tiles per thread and step, loaded together
  for (int d = blockIdx.x; d < kRadix; d += gridDim.x) {
    uint32_t* row = counts + (int64_t)d * tiles;
    uint32_t carry = 0;
    for (int base = 0; base < tiles; base += kPer * NT) {
      const int t0 = base + kPer * threadIdx.x;
      uint32_t v[kPer], sum = 0;
#pragma unroll
      for (int q = 0; q < kPer; ++q) v[q] = t0 + q < tiles ? row[t0 + q] : 0u;
#pragma unroll
      for (int q = 0; q < kPer; ++q) sum += v[q];
      uint32_t run = carry + cta_exclusive<NT>(sum, sh.scan);
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (t0 + q < tiles) row[t0 + q] = run;
        run += v[q];
      }
      __syncthreads();
      if (threadIdx.x == NT - 1) sh.carry = run;
      __syncthreads();
      carry = sh.carry;
    }
    if (threadIdx.x == 0) totals[d] = carry;
  }
}

// Rank every key of the tiles blockIdx.x, + gridDim.x, ... stably and
// scatter.  Not-last passes write (key, value); the last pass writes the
// sorted key and the permutation.
template <int NT>
__device__ __forceinline__ void sort_downsweep(SortShared<NT>& sh, int64_t n, int shift, bool first, bool last,
                                               const int32_t* __restrict__ cell, const uint32_t* keys_in,
                                               const uint32_t* vals_in, uint32_t* keys_out, uint32_t* vals_out,
                                               const uint32_t* counts, const uint32_t* totals, int tiles,
                                               int32_t* perm) {
  constexpr int kChunks = kTile / NT, kWarps = NT / 32, kDigits = kRadix / NT;
  const int warp = threadIdx.x >> 5, lane = lane_id();
  // first key position of each digit: the exclusive scan of the totals (digits
  // threadIdx.x * kDigits ...), the same for every tile
  uint32_t tot[kDigits], sum = 0;
#pragma unroll
  for (int q = 0; q < kDigits; ++q) sum += tot[q] = totals[threadIdx.x * kDigits + q];
  uint32_t first_of[kDigits];
  first_of[0] = cta_exclusive<NT>(sum, sh.scan);
#pragma unroll
  for (int q = 1; q < kDigits; ++q) first_of[q] = first_of[q - 1] + tot[q - 1];
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t base = (int64_t)tile * kTile + warp * (32 * kChunks) + lane;
    uint32_t r_key[kChunks], r_val[kChunks], r_rank[kChunks];
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const int64_t idx = base + c * 32;
      const bool valid = idx < n;
      r_key[c] = valid ? (first ? (uint32_t)cell[idx] : keys_in[idx]) : 0u;
      r_val[c] = first ? (uint32_t)idx : (valid ? vals_in[idx] : 0u);
    }
    __syncthreads();  // the previous tile's reads of the shared arrays are done
    for (int w = 0; w < kWarps; ++w)
      for (int d = threadIdx.x; d < kRadix; d += NT) sh.warp_hist[w][d] = 0;
#pragma unroll
    for (int q = 0; q < kDigits; ++q) {
      const int d = threadIdx.x * kDigits + q;
      sh.base[d] = first_of[q] + counts[(int64_t)d * tiles + tile];
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      const bool valid = base + c * 32 < n;
      if (first) r_key[c] = morton_of_cell((int32_t)r_key[c]);
      uint32_t d = valid ? digit_of(r_key[c], shift) : 0xffffffffu;
      unsigned peers = __match_any_sync(0xffffffffu, d);
      unsigned before = peers & lanemask_lt();
      uint32_t prior = valid ? sh.warp_hist[warp][d] : 0u;
      __syncwarp();
      if (valid && before == 0) sh.warp_hist[warp][d] = prior + (uint32_t)__popc(peers);
      __syncwarp();
      r_rank[c] = valid ? prior + (uint32_t)__popc(before) : 0xffffffffu;
    }
    __syncthreads();
    // exclusive scan over warps, per digit
    for (int d = threadIdx.x; d < kRadix; d += NT) {
      uint32_t run = 0;
      for (int w = 0; w < kWarps; ++w) {
        uint32_t t = sh.warp_hist[w][d];
        sh.warp_hist[w][d] = run;
        run += t;
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
      if (r_rank[c] == 0xffffffffu) continue;
      uint32_t d = digit_of(r_key[c], shift);
      uint32_t pos = sh.base[d] + sh.warp_hist[warp][d] + r_rank[c];
      keys_out[pos] = r_key[c];
      if (!last)
        vals_out[pos] = r_val[c];
      else
        perm[pos] = (int32_t)r_val[c];
    }
  }
}

// Gather of granule k into sorted order (out[k] = in[perm[k]]: perm is close to
// the identity because the input is the previous substep's sorted order, so
// the reads are nearly coalesced), and the cell table entry
// {start, count, epoch, 0} of every occupied cell at 1 + its linear index.
template <typename T>
__device__ __forceinline__ void sort_gather(const DGrid& G, int64_t n, int64_t k, const uint32_t* keys,
                                            const ScatterState& S, uint4* table, uint32_t* status) {
  int32_t src = S.perm[k];
  int32_t c = S.in_cell[src];
  pos_t<T> p = ((const pos_t<T>*)S.in_pos)[src];
  S.out_cell[k] = c;
  ((pos_t<T>*)S.out_pos)[k] = p;
  ((vec_t<T>*)S.out_vel)[k] = ((const vec_t<T>*)S.in_vel)[src];
  if (S.out_id) S.out_id[k] = S.in_id ? S.in_id[src] : src;
  if constexpr (sizeof(T) == 4) {
    if (S.out_posf)
      S.out_posf[k] = posf_of(c, p);
  }
  uint32_t key = keys[k];
  if (k > 0 && keys[k - 1] == key) return;
  int64_t e = k + 1;
  while (e < n && keys[e] == key) ++e;
  int x = cell_x(c), y = cell_y(c), z = cell_z(c);
  if (x >= G.nc[0] || y >= G.nc[1] || z >= G.nc[2]) {
    raise_status(status, GIC_STATUS_BAD_CELL);
    return;
  }
  uint32_t epoch = table[0].x;
  table[table_index(G, x, y, z)] = make_uint4((uint32_t)k, (uint32_t)(e - k), epoch, 0u);
}

}  // namespace gic
