// gic_tile.cuh -- a CTA's neighbourhood of contact cells staged in shared
// memory (the cell-table entries of its box and the float positions of every
// granule in it), and the Verlet-list build on it.  Shared by gic_contact's
// staged kernel, gic_neighbors_build and gic_step's rebuild kernel.
#pragma once

#include "gic_contact.cuh"

namespace gic {

// The float positions (contact-cell units, absolute) and radii of a state's
// granules: the FP32 state's copies, or formed from its fixed-point records
// (the same values), or from an FP64 state (off by at most one float rounding,
// which kPosfTol covers as it does for the copies).
template <typename T>
struct FloatPos {
  const int32_t* cell;
  const pos_t<T>* pos;
  const float4* posf;
  __device__ __forceinline__ float4 operator()(int64_t j) const {
    if constexpr (sizeof(T) == 4) {
      return posf ? __ldg(&posf[j]) : posf_of(__ldg(&cell[j]), __ldg(&pos[j]));
    } else {
      const int32_t c = __ldg(&cell[j]);
      const d4 p = ldg(&pos[j]);
      return make_float4((float)cell_x(c) + (float)(p.x * inv_hc), (float)cell_y(c) + (float)(p.y * inv_hc),
                         (float)cell_z(c) + (float)(p.z * inv_hc), (float)p.w);
    }
  }
  double inv_hc;
};

// ----------------------------------------------------------------- staged neighbourhood
//
// One CTA = NT consecutive granules of the Morton-sorted state: a compact
// blob of contact cells.  The CTA marks the cells within one of any of its
// granules' cells, stages the cell-table entries of the marked cells of the
// blob's bounding box and the float positions of every granule in them in
// shared memory, and each thread then walks its 27 neighbour cells there.  A
// Morton range of 256 granules is a few boxes side by side, whose common
// bounding box holds two to three times the cells that any of its granules
// looks at; with the unmarked ones left out, and one buffer shared by the box's
// entries (6 bytes a cell) and the granules (16), 97 to 99.8% of the CTAs fit
// (dam break, sweep, polydisperse bed, dense packing; 41 to 57% with every cell of
// the box in two fixed arrays of the same size).  The others (a Morton range
// that jumps across the domain) take the global-memory path; the results are
// identical.  A gic_step call that rebuilds: 16M sweep 5907 -> 4643 us, 8M bed
// 5794 -> 4361, FP64 dam break of 1M 1752 -> 1040.
//
// The buffers: 22 KB for 128 granules (gic_contact, gic_neighbors_build: 90 to 98%
// of the CTAs fit, and several are resident), or the 48 KB
// that a CTA of the fused substep has anyway.

constexpr int kTileThreads = 128;

// The CTA's staged neighbourhood in shared memory.
template <int NT>
struct TileShared {
  static constexpr int kBytes = NT == 256 ? 48 * 1024 - 256 : (NT == 128 ? 22 * 1024 : 24 * 1024);
  static constexpr int kCells = kBytes / 12;  // at most half the buffer
  __align__(16) unsigned char buf[kBytes];
  int wlo[3][NT / 32], whi[3][NT / 32];
  uint32_t wsum[NT / 32];
  unsigned rmax_bits;  // the largest staged radius (float bits)
};

struct TileBox {
  bool staged;             // the neighbourhood is in shared memory (uniform over the CTA)
  int bx0, by0, bz0, bx, by, bz;
  uint32_t* start;         // by box cell: sorted index of its first granule
  uint16_t* off;           // by box cell: slot of its first granule; off[b + 1] ends it
  float4* pf;              // by slot
};

// CTA-wide (every thread calls it once): the bounding box of the CTA's contact
// cells with a one-cell halo, clipped to the grid; the table entries (start,
// count of this epoch) of its marked cells, their exclusive scan and the float
// positions of their granules, relative to the box corner.  valid / ci: this
// thread's granule and cell.
template <int NT, typename T>
__device__ __forceinline__ TileBox tile_stage(TileShared<NT>& sh, const DGrid& G, const uint4* table, uint32_t epoch,
                                              const FloatPos<T>& fpos, bool valid, int32_t ci) {
  constexpr int kCells = TileShared<NT>::kCells, kW = NT / 32;
  static_assert((kW & (kW - 1)) == 0 && kW <= 32, "lanes read the warps' extents in turn");
  const int warp = threadIdx.x >> 5, cx = cell_x(ci), cy = cell_y(ci), cz = cell_z(ci);
  const int c3[3] = {cx, cy, cz};
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int l = __reduce_min_sync(0xffffffffu, valid ? c3[a] : kMaxCellsPerAxis - 1);
    const int h = __reduce_max_sync(0xffffffffu, valid ? c3[a] : -1);
    if (lane_id() == 0) {
      sh.wlo[a][warp] = l;
      sh.whi[a][warp] = h;
    }
  }
  if (threadIdx.x == 0) sh.rmax_bits = 0u;
  __syncthreads();
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lo[a] = __reduce_min_sync(0xffffffffu, sh.wlo[a][lane_id() & (kW - 1)]);
    hi[a] = __reduce_max_sync(0xffffffffu, sh.whi[a][lane_id() & (kW - 1)]);
  }
  TileBox B;
  B.bx0 = max(lo[0] - 1, 0);
  B.by0 = max(lo[1] - 1, 0);
  B.bz0 = max(lo[2] - 1, 0);
  B.bx = min(hi[0] + 1, G.nc[0] - 1) - B.bx0 + 1;
  B.by = min(hi[1] + 1, G.nc[1] - 1) - B.by0 + 1;
  B.bz = min(hi[2] + 1, G.nc[2] - 1) - B.bz0 + 1;
  const int ncell = B.bx * B.by * B.bz;
  // a CTA without granules stages nothing, nor does one with a granule in a cell beyond
  // the grid (GIC_STATUS_BAD_CELL), whose own cell and slot the box does not hold
  B.staged = hi[0] >= 0 && hi[0] < G.nc[0] && hi[1] < G.nc[1] && hi[2] < G.nc[2] && ncell <= kCells;
  B.start = reinterpret_cast<uint32_t*>(sh.buf);
  B.off = nullptr;
  B.pf = nullptr;
  if (!B.staged) return B;
  const int nr = (ncell + 8) & ~7;  // ncell + 1 entries, to a multiple of 8
  B.off = reinterpret_cast<uint16_t*>(sh.buf + 4 * nr);
  B.pf = reinterpret_cast<float4*>(sh.buf + 6 * nr);
  // mark the cells around the granules' (the first lane of a run in one cell marks for it)
  for (int w = threadIdx.x; w < nr / 2; w += NT) reinterpret_cast<uint32_t*>(B.off)[w] = 0u;
  __syncthreads();
  const int32_t prev = __shfl_up_sync(0xffffffffu, ci, 1);
  if (valid && (lane_id() == 0 || prev != ci)) {
    const int xa = max(cx - 1, 0) - B.bx0, xb = min(cx + 1, G.nc[0] - 1) - B.bx0;
    for (int z = max(cz - 1, 0); z <= min(cz + 1, G.nc[2] - 1); ++z)
      for (int y = max(cy - 1, 0); y <= min(cy + 1, G.nc[1] - 1); ++y) {
        uint16_t* row = B.off + B.bx * ((y - B.by0) + B.by * (z - B.bz0));
        for (int x = xa; x <= xb; ++x) row[x] = 1;
      }
  }
  __syncthreads();
  // the table entries of the marked cells; box index -> coordinates with float
  // reciprocals: (b + 1/2) / d stays >= 1 / (2 d) from an integer
  const float ibx = __fdividef(1.0f, (float)B.bx), ibxy = __fdividef(1.0f, (float)(B.bx * B.by));
  constexpr int kU = 4;  // loads in flight per thread
  for (int b0 = threadIdx.x; b0 < ncell; b0 += kU * NT) {
    uint4 e[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int b = b0 + u * NT;
      e[u] = make_uint4(0u, 0u, 0u, 0u);
      if (b < ncell && B.off[b]) {
        const int z = (int)(((float)b + 0.5f) * ibxy);
        const int rem = b - z * B.bx * B.by;
        const int y = (int)(((float)rem + 0.5f) * ibx);
        e[u] = __ldg(&table[table_index(G, B.bx0 + rem - y * B.bx, B.by0 + y, B.bz0 + z)]);
        if (e[u].z != epoch) e[u].y = 0u;
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int b = b0 + u * NT;
      if (b >= ncell) break;
      B.start[b] = e[u].x;
      B.off[b] = (uint16_t)min(e[u].y, 0xffffu);  // a count cut off here is beyond the buffer
    }
  }
  __syncthreads();
  // exclusive scan of the counts: consecutive cells per thread, then the threads
  const int per = (ncell + NT - 1) / NT, first = min((int)threadIdx.x * per, ncell), last = min(first + per, ncell);
  uint32_t sum = 0;
  for (int b = first; b < last; ++b) sum += B.off[b];
  uint32_t incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane_id() >= d) incl += o;
  }
  if (lane_id() == 31) sh.wsum[warp] = incl;
  __syncthreads();
  const uint32_t ws = lane_id() < kW ? sh.wsum[lane_id()] : 0u;
  const uint32_t total = __reduce_add_sync(0xffffffffu, ws);
  B.staged = 6u * (uint32_t)nr + 16ull * total <= (uint32_t)TileShared<NT>::kBytes;  // then total < 2^16
  if (!B.staged) return B;
  uint32_t run = __reduce_add_sync(0xffffffffu, lane_id() < warp ? ws : 0u) + incl - sum;
  for (int b = first; b < last; ++b) {
    const uint32_t c = B.off[b];
    B.off[b] = (uint16_t)run;
    run += c;
  }
  if (threadIdx.x == 0) B.off[ncell] = (uint16_t)total;
  __syncthreads();
  // stage the float positions: cell b's granules go to slots off[b] ...
  // off[b + 1] - 1.  A cell takes one lane, or eight where cells hold many
  // granules; the first granules of kU cells are in flight together.  Positions
  // are in units of contact cells relative to the box corner (exact
  // differences of the absolute copies): the three cells of an x-row are
  // consecutive slots, and no cell offset is needed
  float rmax = 0.f;
  const int sh8 = total > 2u * (uint32_t)ncell ? 3 : 0;
  auto put = [&](uint32_t t, const float4& p) {
    B.pf[t] = make_float4(p.x - (float)B.bx0, p.y - (float)B.by0, p.z - (float)B.bz0, p.w);
    rmax = fmaxf(rmax, p.w);
  };
  for (int w0 = threadIdx.x; w0 < ncell << sh8; w0 += kU * NT) {
    float4 pv[kU];
    uint32_t at[kU], end[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int w = w0 + u * NT;
      at[u] = end[u] = 0u;
      pv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (w < ncell << sh8) {
        const int b = w >> sh8;
        const uint32_t o = B.off[b];
        at[u] = o + (uint32_t)(w - (b << sh8));
        end[u] = B.off[b + 1];
        if (at[u] < end[u]) pv[u] = fpos(B.start[b] + (at[u] - o));
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (at[u] >= end[u]) continue;
      put(at[u], pv[u]);
      const int b = (w0 + u * NT) >> sh8;
      const uint32_t base = B.start[b] - B.off[b];
      for (uint32_t t = at[u] + (1u << sh8); t < end[u]; t += 1u << sh8) put(t, fpos(base + t));
    }
  }
  const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(rmax));  // radii >= 0
  if (lane_id() == 0) atomicMax(&sh.rmax_bits, m);
  __syncthreads();
  return B;
}

// Walk of granule i's 27 cells in a staged neighbourhood, in the order of
// for_each_partner, with candidates beyond reach(r_j) (contact cells) left out: hit(t,
// b, code, d2, r_j) for slot t of box cell b at offset code = (ox + 1) + 3 (oy + 1) +
// 9 (oz + 1).  fi: the granule's float position.
//
// Cells farther than the largest reach of any staged partner (plus a margin
// past the float rounding of d2) hold no partner: whole rows (oy, oz) and the
// end cells of a row are skipped.  A staged copy lies in its closed cell, so its
// distance is at least the cell's.  (One loop over the slots of all rows instead of
// one per row is slower, 2250 -> 2610 us for gic_contact on the 16M sweep: the lanes of
// a warp share cells, so their rows are alike and their loads broadcast.)
template <int NT, typename Reach, typename F>
__device__ __forceinline__ void tile_walk(const TileShared<NT>& sh, const TileBox& B, int64_t i, int32_t ci,
                                          const float4& fi, Reach reach, F hit) {
  const int lx = cell_x(ci) - B.bx0, ly = cell_y(ci) - B.by0, lz = cell_z(ci) - B.bz0;
  const float xi = fi.x - (float)B.bx0, yi = fi.y - (float)B.by0, zi = fi.z - (float)B.bz0;
  const float Rmax = reach(__uint_as_float(sh.rmax_bits)) + 1e-3f;
  const float R2 = Rmax * Rmax;
  const int bown = lx + B.bx * (ly + B.by * lz);
  const uint32_t tself = B.off[bown] + (uint32_t)(i - (int64_t)B.start[bown]);
  const float dxl = xi - (float)lx, dxh = (float)(lx + 1) - xi;  // to the own cell's x faces
  for (int oz = -1; oz <= 1; ++oz) {
    const int z = lz + oz;
    if (z < 0 || z >= B.bz) continue;
    const float dz = oz < 0 ? zi - (float)lz : (oz > 0 ? (float)(lz + 1) - zi : 0.f);
    for (int oy = -1; oy <= 1; ++oy) {
      const int y = ly + oy;
      if (y < 0 || y >= B.by) continue;
      const float dy = oy < 0 ? yi - (float)ly : (oy > 0 ? (float)(ly + 1) - yi : 0.f);
      const float dyz = fmaf(dy, dy, dz * dz);
      if (dyz >= R2) continue;
      const int xa = (lx > 0 && fmaf(dxl, dxl, dyz) < R2) ? lx - 1 : lx;
      const int xb = (lx + 1 < B.bx && fmaf(dxh, dxh, dyz) < R2) ? lx + 1 : lx;
      const int rb = B.bx * (y + B.by * z);
      const uint32_t t0 = B.off[rb + xa], t1 = B.off[rb + xb + 1];
      for (uint32_t t = t0; t < t1; ++t) {
        const float4 fj = B.pf[t];
        const float rx = fj.x - xi, ry = fj.y - yi, rz = fj.z - zi;
        const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
        const float Rs = reach(fj.w);
        if (d2 < Rs * Rs) {
          if (t == tself) continue;
          int bj = rb + xa;
          while (B.off[bj + 1] <= t) ++bj;  // the cell of slot t (cells of the row in x order)
          hit(t, bj, (bj - rb - lx + 1) + 3 * (oy + 1) + 9 * (oz + 1), d2, fj.w);
        }
      }
    }
  }
}

// ----------------------------------------------------------------- staged list build
//
// The row of granule i (contact cell ci) of the sorted state on the
// neighbourhood staged by its CTA: the partners within r_i + r_j + skin by the float
// pre-test of verlet_pair (kCap: within grow (r_i + r_j) + skin, the bridges'
// reach), in the order of the 27-cell walk, slot = sorted index, and the
// granule's reference entries; no forces (the substep then walks the fresh
// rows).  A row beyond cap entries sets the overflow word (kStep: and has the
// count kNbWalked); returns whether it did.
template <int NT, typename T, bool kCap, bool kStep>
__device__ __forceinline__ bool build_row(const TileShared<NT>& sh, const TileBox& B, const DGrid& G, int64_t n,
                                          int64_t i, int32_t ci, const FloatPos<T>& fpos, const int32_t* id,
                                          const uint4* table, uint32_t epoch, const NbDev& nb, float skin, float grow) {
  if (i >= n) return false;
  const int cx = cell_x(ci), cy = cell_y(ci), cz = cell_z(ci);
  const float4 fi = fpos(i);
  const float ri = fi.w;
  auto reach = [&](float rj) {
    return kCap ? fmaf(fmaf(ri + rj, grow, skin), G.inv_hc_f, kPosfTol) : fmaf(ri + rj + skin, G.inv_hc_f, kPosfTol);
  };
  int32_t* row = nb.list + i * nb.cap;
  int cnt = 0;
  bool over = false;
  auto keep = [&](int64_t j) {
    if (cnt < nb.cap)
      row[cnt++] = (int32_t)j;
    else
      over = true;
  };
  if (B.staged) {
    // the walk's test in one multiply-add, wider than reach() by more than their
    // roundings differ; reach() then decides, as on the other paths
    const float g = kCap ? grow : 1.f, per_r = g * G.inv_hc_f;
    const float own = fmaf(fmaf(ri, g, skin), G.inv_hc_f, kPosfTol) + 4e-6f;
    tile_walk<NT>(sh, B, i, ci, fi, [&](float rj) { return fmaf(rj, per_r, own); },
                  [&](uint32_t t, int bj, int, float d2, float rj) {
                    const float Rs = reach(rj);
                    if (d2 < Rs * Rs) keep((int64_t)B.start[bj] + (t - B.off[bj]));
                  });
  } else {  // the box exceeds the tile: the 27 cells from global memory
    auto walk = [&](auto at) {
      for_each_partner(G, table, epoch, i, cx, cy, cz, [&](int64_t j, int, int, int) {
        const float4 fj = at(j);
        const float rx = fj.x - fi.x, ry = fj.y - fi.y, rz = fj.z - fi.z;
        const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
        const float Rs = reach(fj.w);
        if (d2 < Rs * Rs) keep(j);
      });
    };
    // gic_neighbors_build has float copies: without the question for every candidate
    // 10,976 granules in cells of 190 take 358 us instead of 465.  (gic_step may have
    // none; both walks in its kernel made the 16M sweep's rebuild 1.3% slower.)
    if constexpr (sizeof(T) == 4 && !kStep)
      walk([&](int64_t j) { return __ldg(&fpos.posf[j]); });
    else
      walk(fpos);
  }
  nb.count[i] = kStep && over ? kNbWalked : cnt;
  nb.at[i] = (int32_t)i;
  nb.cur[i] = (int32_t)i;
  nb.ref_cell[i] = ci;
  reinterpret_cast<pos_t<T>*>(nb.ref_pos)[i] = ldg(&fpos.pos[i]);
  const int32_t idi = __ldg(&id[i]);
  if (idi >= 0 && (int64_t)idi < n) nb.slot[idi] = (int32_t)i;
  if (over) atomicOr(&nb.flags[kNbOverflow], 1u);
  return over;
}

}  // namespace gic
