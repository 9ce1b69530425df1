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
// blob of contact cells.  The CTA stages the cell-table entries of the
// blob's bounding box (+1 cell halo) and the float positions of every
// granule in those cells in shared memory, then each thread walks its 27
// neighbour cells there.  A CTA whose box or granule count exceeds the
// shared-memory budget (a Morton range that jumps across the domain) takes
// the global-memory path instead; the results are identical.
//
// The budgets: 128 granules, 22 KB (gic_contact, gic_neighbors_build; more
// CTAs per SM suit the monodisperse packings), or 256 granules in the 46 KB
// that a CTA of the fused substep has anyway.

constexpr int kTileThreads = 128;

// The CTA's staged neighbourhood in shared memory.
template <int NT>
struct TileShared {
  static constexpr int kCells = NT <= 128 ? 512 : 768;
  static constexpr int kGranules = NT <= 128 ? 1152 : 2304;
  int lo[3], hi[3];
  uint32_t start[kCells];
  uint32_t off[kCells + 1];  // first slot of each cell; at first its granule count
  float4 pf[kGranules];
  uint32_t wsum[NT / 32];
  int mode;             // 0: staged, 1: global fallback
  unsigned rmax_bits;   // the largest staged radius (float bits)
};

struct TileBox {
  int bx0, by0, bz0, bx, by, bz;
};

// CTA-wide (every thread calls it): the bounding box of the CTA's contact
// cells with a one-cell halo, clipped to the grid; its table entries (start,
// count of this epoch), their exclusive scan and the float positions of every
// granule in the box, relative to the box corner.  sh.mode = 1 when the box or
// its granules exceed the tile.  valid / ci: this thread's granule and cell.
template <int NT, typename T>
__device__ __forceinline__ TileBox tile_stage(TileShared<NT>& sh, const DGrid& G, const uint4* table, uint32_t epoch,
                                              const FloatPos<T>& fpos, bool valid, int32_t ci) {
  constexpr int kCells = TileShared<NT>::kCells, kGranules = TileShared<NT>::kGranules;
  __syncthreads();  // the last use of sh is over
  if (threadIdx.x < 3) {
    sh.lo[threadIdx.x] = 1 << 30;
    sh.hi[threadIdx.x] = -1;
  }
  if (threadIdx.x == 0) sh.rmax_bits = 0u;
  __syncthreads();
  if (valid) {
    atomicMin(&sh.lo[0], cell_x(ci));
    atomicMin(&sh.lo[1], cell_y(ci));
    atomicMin(&sh.lo[2], cell_z(ci));
    atomicMax(&sh.hi[0], cell_x(ci));
    atomicMax(&sh.hi[1], cell_y(ci));
    atomicMax(&sh.hi[2], cell_z(ci));
  }
  __syncthreads();
  TileBox B;
  B.bx0 = max(sh.lo[0] - 1, 0);
  B.by0 = max(sh.lo[1] - 1, 0);
  B.bz0 = max(sh.lo[2] - 1, 0);
  B.bx = min(sh.hi[0] + 1, G.nc[0] - 1) - B.bx0 + 1;
  B.by = min(sh.hi[1] + 1, G.nc[1] - 1) - B.by0 + 1;
  B.bz = min(sh.hi[2] + 1, G.nc[2] - 1) - B.bz0 + 1;
  const int ncell = B.bx * B.by * B.bz;
  if (threadIdx.x == 0) sh.mode = (ncell > kCells || sh.hi[0] < 0) ? 1 : 0;
  __syncthreads();
  if (sh.mode == 0) {
    // stage the table entries of the box
    // box index -> coordinates with float reciprocals (exact for these small integers)
    const float ibx = 1.0f / (float)B.bx, ibxy = 1.0f / (float)(B.bx * B.by);
    constexpr int kU = 4;  // loads in flight per thread
    for (int b0 = threadIdx.x; b0 < ncell; b0 += kU * NT) {
      uint4 e[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int b = b0 + u * NT;
        if (b >= ncell) break;
        int z = (int)(((float)b + 0.5f) * ibxy);
        int rem = b - z * B.bx * B.by;
        int y = (int)(((float)rem + 0.5f) * ibx);
        int x = B.bx0 + rem - y * B.bx;
        y += B.by0;
        z += B.bz0;
        e[u] = __ldg(&table[table_index(G, x, y, z)]);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int b = b0 + u * NT;
        if (b >= ncell) break;
        const bool ok = e[u].z == epoch;
        sh.start[b] = ok ? e[u].x : 0u;
        sh.off[b] = ok ? e[u].y : 0u;
      }
    }
    __syncthreads();
    // exclusive scan of the counts (kCells / NT per thread)
    {
      const int per = (kCells + NT - 1) / NT;
      uint32_t loc[per];
      uint32_t sum = 0;
#pragma unroll
      for (int k = 0; k < per; ++k) {
        int b = threadIdx.x * per + k;
        loc[k] = b < ncell ? sh.off[b] : 0u;
        sum += loc[k];
      }
      uint32_t incl = sum;
      for (int off = 1; off < 32; off <<= 1) {
        uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane_id() >= off) incl += o;
      }
      if (lane_id() == 31) sh.wsum[threadIdx.x >> 5] = incl;
      __syncthreads();
      uint32_t base = 0;
      for (int w = 0; w < (threadIdx.x >> 5); ++w) base += sh.wsum[w];
      uint32_t run = base + incl - sum;
#pragma unroll
      for (int k = 0; k < per; ++k) {
        int b = threadIdx.x * per + k;
        if (b < kCells) sh.off[b] = run;
        run += loc[k];
      }
      if (threadIdx.x == NT - 1) sh.off[kCells] = run;
    }
    __syncthreads();
    const uint32_t total = sh.off[kCells];
    if (total > (uint32_t)kGranules) {
      if (threadIdx.x == 0) sh.mode = 1;
    } else {
      // stage the float positions: cell b's granules go to slots off[b] ...
      // off[b + 1] - 1.  A cell takes one lane, or eight where cells hold
      // many granules; the first granules of kU cells are in flight together
      float rmax = 0.f;
      const int sh8 = total > 4u * (uint32_t)ncell ? 3 : 0;
      // positions in units of contact cells relative to the box corner (exact
      // differences of the absolute copies): the three cells of an x-row are
      // consecutive slots, and no cell offset is needed
      auto put = [&](uint32_t t, const float4& p) {
        sh.pf[t] = make_float4(p.x - (float)B.bx0, p.y - (float)B.by0, p.z - (float)B.bz0, p.w);
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
            at[u] = sh.off[b] + (uint32_t)(w - (b << sh8));
            end[u] = sh.off[b + 1];
            if (at[u] < end[u]) pv[u] = fpos(sh.start[b] + (at[u] - sh.off[b]));
          }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          if (at[u] >= end[u]) continue;
          put(at[u], pv[u]);
          const int b = (w0 + u * NT) >> sh8;
          const uint32_t first = sh.start[b] - sh.off[b];
          for (uint32_t t = at[u] + (1u << sh8); t < end[u]; t += 1u << sh8) put(t, fpos(first + t));
        }
      }
      const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(rmax));  // radii >= 0
      if (lane_id() == 0) atomicMax(&sh.rmax_bits, m);
    }
    __syncthreads();
  }
  return B;
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
  if (sh.mode == 0) {
    const int lx = cx - B.bx0, ly = cy - B.by0, lz = cz - B.bz0;
    const float xi = fi.x - (float)B.bx0, yi = fi.y - (float)B.by0, zi = fi.z - (float)B.bz0;
    const int bown = lx + B.bx * (ly + B.by * lz);
    const uint32_t tself = sh.off[bown] + (uint32_t)(i - (int64_t)sh.start[bown]);
    // Cells farther than the largest pre-test radius of any staged partner
    // (plus a margin past the float rounding of d2) hold no partner: whole
    // rows (oy, oz) and the end cells of a row are skipped.  A staged copy
    // lies in its closed cell, so its distance is at least the cell's.
    const float Rmax = reach(__uint_as_float(sh.rmax_bits)) + 1e-3f;
    const float R2 = Rmax * Rmax;
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
        const uint32_t t0 = sh.off[rb + xa], t1 = sh.off[rb + xb + 1];
        for (uint32_t t = t0; t < t1; ++t) {
          if (t == tself) continue;
          const float4 fj = sh.pf[t];
          const float rx = fj.x - xi, ry = fj.y - yi, rz = fj.z - zi;
          const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
          const float Rs = reach(fj.w);
          if (d2 < Rs * Rs) {
            int bj = rb + xa;
            while (sh.off[bj + 1] <= t) ++bj;  // the cell of slot t (cells of the row in x order)
            keep((int64_t)sh.start[bj] + (t - sh.off[bj]));
          }
        }
      }
    }
  } else {  // the box exceeds the tile: the 27 cells from global memory
    for_each_partner(G, table, epoch, i, cx, cy, cz, [&](int64_t j, int, int, int) {
      const float4 fj = fpos(j);
      const float rx = fj.x - fi.x, ry = fj.y - fi.y, rz = fj.z - fi.z;
      const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
      const float Rs = reach(fj.w);
      if (d2 < Rs * Rs) keep(j);
    });
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
