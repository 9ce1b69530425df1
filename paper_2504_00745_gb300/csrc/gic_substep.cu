// gic_substep.cu -- one SandSubstep (Alg. 2) after the sort, fused into one
// pass over the sorted state: contact forces from the Verlet lists (or, on a
// substep that rebuilds them, from the 27-cell walk that builds them), the G2P coupling
// (Sec. 3.3), the virtual-mass integration (Sec. 5.2) into the next state,
// and the P2G scatter of F_s at the old positions and, when asked, of
// alpha_s at the new ones.  The per-granule force arrays of the separate
// entry points (F_c, F_fl, a_f, f_ex) never leave registers.
#include <type_traits>

#include "gic_capillary.cuh"
#include "gic_contact.cuh"
#include "gic_grid.cuh"
#include "gic_integrate.cuh"
#include "gic_sort.cuh"
#include "gic_tile.cuh"

namespace gic {

// CTAs of 256 threads; a small FP64 state takes CTAs of 64, at most three per SM, so
// that it is spread over the chip: 8,000 granules in 32 CTAs kept 32 SMs busy and
// 120 idle, and FP64 instructions issue at 1.8 lanes per clock and SM.  Windows of 20
// substeps in CTAs of 256 and of 64 (152 SMs: the line at 29,184), dense packing: 2590
// and 1746 us at 9,000 granules, 2925 and 2549 at 27,000, 2974 and 2941 at 32,000, 3029
// and 3079 at 37,000; loose packing, where the staging of the tiles weighs more: 727
// and 687 at 8,000, 831 and 837 at 29,000, 792 and 855 at 32,000, 1221 and 1422 at 50,000.
// (FP32 stays at 256: 467 against 446 us at 7,000 granules, and two partners'
// opposite deposits cancel exactly inside one CTA's integer tile only.)
constexpr int kSubstepThreads = kSubThreads;
constexpr int kSmallThreads = 64;
constexpr int kSmallPerSm = 3;

// The granule arrays a substep reads.
template <typename T>
struct StateIn {
  const int32_t* cell;
  const pos_t<T>* pos;
  const float4* posf;
  const vec_t<T>* vel;
  const int32_t* id;
};

template <typename T>
static StateIn<T> state_in(const GicGranules* s) {
  return StateIn<T>{s->cell, (const pos_t<T>*)s->pos, sizeof(T) == 4 ? (const float4*)s->posf : nullptr,
                    (const vec_t<T>*)s->vel, s->id};
}

// The shared memory of a substep CTA: the tile (FP32), and before it, in a
// gic_step call that rebuilds, the staged neighbourhood of the list build.
// Dynamic, so that the out-of-line build addresses it as shared memory.
extern __shared__ __align__(16) unsigned char g_substep_smem[];
template <typename T, int NT>
using SubShared = std::conditional_t<sizeof(T) == 4, SubTile, SubTile64<NT>>;
template <typename T, int NT>
constexpr size_t kSubSmem = sizeof(SubShared<T, NT>) > sizeof(TileShared<NT>) ? sizeof(SubShared<T, NT>)
                                                                             : sizeof(TileShared<NT>);
static_assert(kSubSmem<float, kSubstepThreads> <= 48 * 1024, "more shared memory than a kernel has without asking");

// Contact (and bridge) force of sorted granule i from the 27 cells, walls
// excluded, into vel_out[i] (which the granule's own thread reads and then
// overwrites): for a granule whose row overflowed.
template <typename T, bool kCap>
__device__ __forceinline__ void contact_walk(const DGrid& G, const DParams<T>& P, const StateIn<T>& S, const T* af,
                                             const uint4* table, uint32_t epoch, int64_t i, vec_t<T>* vel_out,
                                             uint32_t* status) {
  const int32_t* cell = S.cell;
  const pos_t<T>* pos = S.pos;
  const vec_t<T>* vel = S.vel;
  const int32_t ci = cell[i];
  const int cx = cell_x(ci), cy = cell_y(ci), cz = cell_z(ci);
  const pos_t<T> pi = pos[i];
  const vec_t<T> vi = vel[i];
  const T ri = radius_of(pi);
  const T mi = granule_mass(P, ri);
  T F0 = T(0), F1 = T(0), F2 = T(0);
  bool coincident = false;
  auto contact = [&](int64_t j, const PairGeom<T>& g) {
    add_force(P, g, vi, ldg(&vel[j]), mi, radius_of(ldg(&pos[j])), F0, F1, F2, coincident);
  };
  if constexpr (kCap) {
    const T sri = moisture_ratio_at(G, P, af, ci, pi, (T*)nullptr);
    for_each_partner(G, table, epoch, i, cx, cy, cz, [&](int64_t j, int ox, int oy, int oz) {
      const pos_t<T> pj = ldg(&pos[j]);
      const T rj = radius_of(pj);
      PairGeom<T> g;
      if (!pair_within(G, pi, pj, ox, oy, oz, ri, rj, P.kappa * (ri + rj), g)) return;
      if (g.overlap > T(0))
        contact(j, g);
      else
        add_bridge(P, g, ri, rj, sri,
                   moisture_ratio_at(G, P, af, pack_cell(cx + ox, cy + oy, cz + oz), pj, (T*)nullptr), F0, F1, F2);
    });
  } else {
    for_each_contact<T>(G, table, epoch, i, cx, cy, cz, pi, ri, pos, S.posf, contact);
  }
  if (coincident) raise_status(status, GIC_STATUS_COINCIDENT);
  vel_out[i] = make_vec<T>(F0, F1, F2);
}

// The CTA's share of a rebuild: the rows of its granules of the sorted state
// (each is read only by its own granule's thread, so no CTA waits for
// another's).  Out of line, at the kernel's start: it costs the calls that keep
// their lists no registers, and no launch of its own (an idle launch of one CTA
// per 128 granules costs 2.3 ns per CTA: 20 us of every call on 1M granules).
// The references are to the kernel's parameters.
template <typename T, int NT, bool kCap>
static __device__ __noinline__ void step_build(const DGrid& G, const DParams<T>& P, const StateIn<T>& S,
                                               const NbDev& nb, int64_t n, const T* af, const uint4* table, T skin,
                                               vec_t<T>* vel_out, uint32_t* status) {
  TileShared<NT>& sh = *reinterpret_cast<TileShared<NT>*>(g_substep_smem);
  const uint32_t epoch = __ldg(&table[0].x);
  const int64_t i = blockIdx.x * (int64_t)NT + threadIdx.x;
  const bool valid = i < n;
  const int32_t ci = valid ? __ldg(&S.cell[i]) : 0;
  const FloatPos<T> fpos{S.cell, S.pos, S.posf, G.inv_hc};
  const TileBox B = tile_stage<NT, T>(sh, G, table, epoch, fpos, valid, ci);
  const bool over = build_row<NT, T, kCap, true>(sh, B, G, n, i, ci, fpos, S.id, table, epoch, nb,
                                                              (float)skin, (float)(T(1) + P.kappa));
  if (over) contact_walk<T, kCap>(G, P, S, af, table, epoch, i, vel_out, status);
  __syncthreads();  // the shared memory is the tile's from here on
}

// The moisture ratio of every granule of the state that a gic_step call steps, for
// the capillary walk: from each of its ~11 partners a granule otherwise
// interpolates the partner's fluid fraction again (8 gathers and ~130
// instructions each).  The same values; 300,000 wet granules: 92 -> 79 us per call
// that keeps its lists, this kernel's 5 included.  In the sort's second key and
// index lists, which nothing uses after the sort.
template <typename T>
__global__ void __launch_bounds__(256) k_moisture(const __grid_constant__ DGrid G,
                                                  const __grid_constant__ DParams<T> P, int64_t n,
                                                  const __grid_constant__ StateIn<T> state,
                                                  const __grid_constant__ StateIn<T> sorted, const uint32_t* flags,
                                                  const T* __restrict__ af, T* __restrict__ sr) {
  const int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x;
  if (i >= n || flags[kNbSorted] == kNbStalled) return;
  const bool resorted = flags[kNbSorted] != 0u;  // as k_substep
  sr[i] = moisture_ratio_at(G, P, af, resorted ? sorted.cell[i] : state.cell[i],
                            resorted ? sorted.pos[i] : state.pos[i], (T*)nullptr);
}

// The substep of a call whose sort stalled: `next` becomes a copy of `state`, so that
// what the caller does with it (ids are indices in gic_unpack) stays in bounds.  (In line:
// out of line, nvcc 13.0's FP64 kernel with bridges stored x alone of each record.)
template <typename T, int NT>
static __device__ __forceinline__ void step_stalled(int64_t n, const StateIn<T>& S, int32_t* cell_out, pos_t<T>* pos_out,
                                                 vec_t<T>* vel_out, int32_t* id_out, float4* posf_out) {
  const int64_t i = blockIdx.x * (int64_t)NT + threadIdx.x;
  if (i >= n) return;
  const int32_t c = S.cell[i];
  const pos_t<T> p = S.pos[i];
  cell_out[i] = c;
  pos_out[i] = p;
  vel_out[i] = S.vel[i];
  if (id_out && S.id) id_out[i] = S.id[i];
  if constexpr (sizeof(T) == 4)
    if (posf_out) posf_out[i] = posf_of(c, p);
}

// kMode: kGeneral is gic_substep's kernel, which reads from the list flags
// whether it rebuilds; kStep and kStepCap are gic_step's, without and with the
// capillary force: in a call that rebuilds they read `sorted` and build its rows
// first, out of line, so that the other calls' path carries no build code (a
// smaller instruction footprint: 2% on the 16M sweep).  kNoAlpha: a call without
// alpha_s (the kernel then carries none of its code).
enum SubMode { kGeneral, kStep, kStepCap };

template <typename T, int kMode, bool kNoAlpha = false, int NT = kSubstepThreads>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 || NT == kSmallThreads ? 4 : 2)
    k_substep(const __grid_constant__ DGrid G, const __grid_constant__ DParams<T> P, int64_t n,
              const __grid_constant__ StateIn<T> state, const __grid_constant__ StateIn<T> sorted,
              const __grid_constant__ NbDev nb, const uint4* __restrict__ table, T skin,
              const __grid_constant__ Fields<T> Fd, int32_t* __restrict__ cell_out, pos_t<T>* __restrict__ pos_out,
              vec_t<T>* __restrict__ vel_out, int32_t* __restrict__ id_out, float4* __restrict__ posf_out,
              vec_t<T>* __restrict__ fex_out, double* __restrict__ alpha, T* __restrict__ Fs_u,
              T* __restrict__ Fs_v, T* __restrict__ Fs_w, double* __restrict__ sums, uint32_t* status,
              const T* moisture) {
  // after gic_step's sort kernel, whose launch may overlap it (see substep_launch):
  // returns when that kernel is complete
  if constexpr (kMode != kGeneral) asm volatile("griddepcontrol.wait;" ::: "memory");
  // uniform over the launch
  const uint32_t sort_done = kMode != kGeneral ? nb.flags[kNbSorted] : 0u;
  if (kMode != kGeneral && sort_done == kNbStalled) {  // no sorted state, perhaps no rows
    step_stalled<T, NT>(n, state, cell_out, pos_out, vel_out, id_out, posf_out);
    return;
  }
  const bool resorted = sort_done != 0u;
  const bool rebuild = kMode == kGeneral && (nb.flags[kNbRebuild] | nb.flags[kNbSticky]) != 0u;
  const StateIn<T> S = resorted ? sorted : state;
  const int32_t* __restrict__ cell = S.cell;
  const pos_t<T>* __restrict__ pos = S.pos;
  const float4* __restrict__ posf = S.posf;
  const vec_t<T>* __restrict__ vel = S.vel;
  const int32_t* __restrict__ id = S.id;
  if constexpr (kMode != kGeneral)
    if (resorted)
      step_build<T, NT, kMode == kStepCap>(G, P, sorted, nb, n, Fd.af, table, skin, vel_out, status);
  SubShared<T, NT>& sh = *reinterpret_cast<SubShared<T, NT>*>(g_substep_smem);
  const bool do_a = !kNoAlpha && alpha != nullptr, do_f = Fs_u != nullptr;
  const int64_t i = blockIdx.x * (int64_t)NT + threadIdx.x;
  const bool valid = i < n;
  const int32_t ci = valid ? cell[i] : 0;
  // the granule's own records, prefetched into L2 before the CTA's tile
  // barriers (the loads themselves come after them; no register is held)
  pos_t<T> pi{}, po{};
  vec_t<T> vi{};
  int32_t idi = 0;
  if (valid) {
    prefetch_l2(&pos[i]);
    prefetch_l2(&vel[i]);
    if (id_out && id) prefetch_l2(&id[i]);
    if (!rebuild) {
      const int32_t sl = nb.ident ? (int32_t)i : nb.at[i];
      prefetch_l2(&nb.count[sl]);  // (not the row: a whole line for a few entries)
      prefetch_l2(&nb.ref_cell[sl]);
      prefetch_l2(reinterpret_cast<const pos_t<T>*>(nb.ref_pos) + sl);
    }
  }
  // the candidates' list of the contact walk: the words in which this thread parks
  // its stencils afterwards, or alpha_s is accumulated
  constexpr bool kHitList = sizeof(T) == 4 && kMode != kStepCap;
  // the CTA's tile: the fields staged for G2P, and (FP32) F_s / alpha_s accumulators
  SubBox B;
  if constexpr (sizeof(T) == 4)
    B = sub_tile_begin(sh, G, Fd, valid, ci, do_a && !kHitList, do_f);
  else
    B = sub_tile64_begin<NT>(sh, G, Fd, valid, ci);

  int32_t co = 0;
  T fe[3] = {T(0), T(0), T(0)};
  bool far = false;
  const bool spread = sizeof(T) == 4 && do_f && !do_a && B.tile;  // uniform over the CTA
  if constexpr (sizeof(T) == 4)
    if (spread && !valid) spread_put_stencil(sh, false, SubStencil{});
  if (valid) {
    pi = pos[i];
    vi = vel[i];
    if (id_out && id) idi = id[i];
    const T ri = radius_of(pi);
    const T mi = granule_mass(P, ri);
    uint32_t flags = 0;
    if (T(2) * ri > grid_hc<T>(G)) flags |= GIC_STATUS_RADIUS;
    // a2: contact
    T F0 = 0, F1 = 0, F2 = 0;
    bool coincident = false;
    {
      const int cx = cell_x(ci), cy = cell_y(ci), cz = cell_z(ci);
      const bool has_f = sizeof(T) == 4 && posf != nullptr;
      float4 fi = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (sizeof(T) == 4) fi = posf_of(ci, pi);  // its record in posf
      if (kMode != kGeneral && nb.count[i] < 0) {  // the row overflowed: step_build left the force here
        const vec_t<T> Fc = vel_out[i];
        F0 = Fc.x;
        F1 = Fc.y;
        F2 = Fc.z;
      } else if (kMode == kStepCap || (kMode == kGeneral && P.cap)) {  // with the capillary bridges (Sec. 5.4): contacts and bridge candidates
        auto ratio = [&](int64_t j, int32_t cj, const pos_t<T>& pj) {  // kStepCap: k_moisture's
          if constexpr (kMode == kStepCap)
            return __ldg(&moisture[j]);
          else
            return moisture_ratio_at(G, P, Fd.af, cj, pj, (T*)nullptr);
        };
        const T sri = ratio(i, ci, pi);
        auto near = [&](int64_t j, int32_t cj, const pos_t<T>& pj, const PairGeom<T>& g) {
          if (g.overlap > T(0))
            add_force(P, g, vi, ldg(&vel[j]), mi, radius_of(pj), F0, F1, F2, coincident);
          else
            add_bridge(P, g, ri, radius_of(pj), sri, ratio(j, cj, pj), F0, F1, F2);
        };
        if (rebuild)
          verlet_build_row_near<T>(G, P, nb, table, n, i, cx, cy, cz, ci, pi, ri, skin, id, pos, near);
        else
          for_each_list_near<T>(G, P, nb, i, cx, cy, cz, pi, ri, has_f, fi, cell, pos, posf, near);
      } else if (rebuild) {  // this substep rebuilds the lists: walk the 27 cells
        verlet_build_granule(G, P, nb, table, n, i, cx, cy, cz, ci, pi, ri, mi, vi, has_f, fi, skin, id, pos, posf,
                             vel, F0, F1, F2, coincident);
      } else {
        bool walked = false;
        if constexpr (kHitList)
          if (has_f) {
            for_each_list_hit(G, nb, i, cx, cy, cz, pi, ri, fi, cell, pos, posf, vel, spread_words(sh), kSpreadStride,
                              kSpreadWords, [&](uint32_t, const PairGeom<float>& g, const float4& vj, float rj) {
                                add_force(P, g, vi, vj, mi, rj, F0, F1, F2, coincident);
                              });
            walked = true;
          }
        if (!walked)
          verlet_list_force(G, P, nb, i, cx, cy, cz, ci, pi, ri, mi, vi, has_f, fi, cell, pos, posf, vel, F0, F1, F2,
                            coincident);
      }
      if (P.walls) {
        if constexpr (sizeof(T) == 4)
          add_walls_f32(G, P, pi, ri, mi, vi, cx, cy, cz, F0, F1, F2, status);
        else
          add_walls(G, P, pi, ri, mi, vi, cx, cy, cz, F0, F1, F2, status);
      }
      if (coincident) flags |= GIC_STATUS_COINCIDENT;
      if (!finite_bits(F0) || !finite_bits(F1) || !finite_bits(F2)) flags |= GIC_STATUS_NONFINITE;
    }
    // a3: G2P coupling
    T Ffl[3], af[3];
    T sp;
    if constexpr (sizeof(T) == 4) {
      if (B.tile) {
        const SubStencil St = sub_stencil(B, G, ci, pi);
        if (spread) spread_put_stencil(sh, true, St);
        sp = sub_g2p(sh, B, St, G, P, pi, vi, Ffl, af);
      } else {
        const G2POut o = g2p_global_f32(G, P, Fd, ci, pi, vi);
        sp = o.sp;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          Ffl[d] = o.F[d];
          af[d] = o.a[d];
        }
      }
    } else
      sp = sub_g2p64<NT>(sh, B, G, P, Fd, ci, pi, vi, Ffl, af);
    if (!finite_bits(sp)) flags |= GIC_STATUS_NONFINITE;
    // the record of the last build for the displacement test below, loaded before
    // the stores (which may not be moved past)
    int32_t rc = ci;
    pos_t<T> rp = pi;  // (after a build this call's positions are the reference)
    if (!rebuild) {
      const int32_t sl = nb.ident ? (int32_t)i : nb.at[i];
      rc = nb.ref_cell[sl];
      rp = reinterpret_cast<const pos_t<T>*>(nb.ref_pos)[sl];
    }
    // a4: integrate into the next state
    vec_t<T> vo;
    integrate_granule(G, P, ci, pi, vi, F0, F1, F2, Ffl[0], Ffl[1], Ffl[2], af[0], af[1], af[2], co, po, vo, fe[0],
                      fe[1], fe[2], flags);
    if (flags) raise_status(status, flags);
    cell_out[i] = co;
    pos_out[i] = po;
    vel_out[i] = vo;
    if (id_out && id) id_out[i] = idi;
    if constexpr (sizeof(T) == 4) {
      if (posf_out) posf_out[i] = posf_of(co, po);
    }
    if (fex_out) fex_out[i] = make_vec<T>(fe[0], fe[1], fe[2]);
    // the next call's displacement test, on the positions just written
    far = moved_far(G, co, po, rc, rp, nb_lim2(nb, T(0)));
  }
  const bool cta_far = __any_sync(0xffffffffu, far) && lane_id() == 0;
  if (kMode == kGeneral && cta_far) atomicOr(&nb.flags[kNbNext], 1u);

  // a5: P2G
  if constexpr (sizeof(T) == 4) {
    const float fc[3] = {P.exch * fe[0], P.exch * fe[1], P.exch * fe[2]};
    float unit = 0.f, inv_unit = 0.f;
    if (do_f) {  // the CTA's fixed-point unit
      float Mt = 0.f;
      if (valid) {
        const float m = fmaxf(fabsf(fc[0]), fmaxf(fabsf(fc[1]), fabsf(fc[2])));
        Mt = m <= 3.0e38f ? m : INFINITY;  // NaN or inf: no fixed point for this CTA
      }
      if (spread && valid) spread_put_force(sh, fc);  // before the barrier in sub_fs_scale
      inv_unit = sub_fs_scale(sh, B, Mt, unit);
    }
    float* Fs[3] = {Fs_u, Fs_v, Fs_w};
    unsigned long long S = 0;
    if (kHitList && do_a) sub_zero_alpha(sh, B);
    if (valid && do_a) {
      int ia[3];
      long long va[8];
      alpha_deposits(G, co, po, ia, va, S);
      sub_add_alpha(sh, B, G, (unsigned long long*)alpha, ia, va);
    }
    if (inv_unit == 0.f) {  // (uniform) no tile for F_s
      if (valid && do_f) fs_deposit_global(G, Fs[0], Fs[1], Fs[2], ci, pi, fc[0], fc[1], fc[2]);
    } else if (spread) {
      spread_deposit(sh, B, G, inv_unit);
    } else if (!kNoAlpha && valid) {
      const SubStencil St = sub_stencil(B, G, ci, pi);
#pragma unroll
      for (int comp = 0; comp < 3; ++comp)
        sub_add_face(sh.f[comp], B, G, St.e0[comp], comp == 0 ? St.wf[0] : St.wc[0], comp == 1 ? St.wf[1] : St.wc[1],
                     comp == 2 ? St.wf[2] : St.wc[2], fc[comp] * inv_unit);
    }
    sub_tile_flush(sh, B, G, (unsigned long long*)alpha, Fs, do_a, inv_unit != 0.f, unit);
    if (sums) p2g_sums(sums, (long long)S);
  } else {
    // FP64: straight double atomics (alpha_s from V / dx^3 and the tent
    // weights at the new position, F_s at the old one)
    __shared__ double s_red[32];
    double Vi = 0.0;
    if (valid && do_a) {
      double r = (double)radius_of(po);
      Vi = 4.0 / 3.0 * kPi * r * r * r;
      int m[3];
      double t[3];
      granule_mac_fp64(G, co, po, m, t);
      Stencil3<double> S = make_stencil<double>(G, m, t, 3);
      double s = Vi * G.inv_dx * G.inv_dx * G.inv_dx;
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          double wyz = (b ? S.w[1] : 1.0 - S.w[1]) * (c ? S.w[2] : 1.0 - S.w[2]) * s;
          int64_t row = sample_index(G.nx, G.ny, S.i0[0], S.i0[1] + b, S.i0[2] + c);
          atomicAdd(&alpha[row], (1.0 - S.w[0]) * wyz);
          atomicAdd(&alpha[row + 1], S.w[0] * wyz);
        }
    }
    if (valid && do_f) {
      int m[3];
      T t[3];
      granule_mac<T>(G, ci, pi, m, t);
      T* Fs[3] = {Fs_u, Fs_v, Fs_w};
#pragma unroll
      for (int comp = 0; comp < 3; ++comp)
        add_face64(G, Fs[comp], make_stencil<T>(G, m, t, comp), P.exch * fe[comp]);
    }
    if (sums) {
      double s = block_sum(Vi, s_red);
      if (threadIdx.x == 0) atomicAdd(&sums[1], s);
    }
  }
  if constexpr (kMode == kGeneral)
    verlet_call_done(nb, rebuild);
  else
    step_call_done(nb, resorted, cta_far);
}

constexpr int kSubstepAdjThreads = 128;
constexpr int kAdjHits = 12;

// Adjoint of k_substep's granule outputs (next position, velocity, f_ex) for
// one granule of the sorted state: the integration's adjoint gives the
// granule's own F_c, F_fl and a_f gradients, the G2P adjoint adds its
// position and velocity parts, and the contact adjoint walks the granule's
// Verlet row (or the 27 cells, writing the row, on a substep that rebuilds
// it), forming each partner's F_c gradient from the partner's upstream
// gradients.  Writes the result through perm (the sort's scatter).
template <typename T>
__global__ void __launch_bounds__(kSubstepAdjThreads, sizeof(T) == 4 ? 6 : 3) k_substep_adj(
    DGrid G, DParams<T> P, int64_t n, const int32_t* __restrict__ cell, const pos_t<T>* __restrict__ pos,
    const float4* __restrict__ posf, const vec_t<T>* __restrict__ vel, const int32_t* __restrict__ id, NbDev nb,
    const uint4* __restrict__ table, T skin, Fields<T> Fd, const vec_t<T>* __restrict__ gxo,
    const vec_t<T>* __restrict__ gvo, const vec_t<T>* __restrict__ gfe, const int32_t* __restrict__ perm,
    vec_t<T>* __restrict__ gxi, vec_t<T>* __restrict__ gvi, double* __restrict__ g_cdrag,
    double* __restrict__ g_mu) {
  __shared__ double s_red[64];
  __shared__ uint32_t s_list[sizeof(T) == 4 ? kAdjHits : 1][kSubstepAdjThreads];  // candidates of the contact walk
  const bool rebuild = (nb.flags[kNbRebuild] | nb.flags[kNbSticky]) != 0u;  // uniform over the launch
  const int64_t i = blockIdx.x * (int64_t)kSubstepAdjThreads + threadIdx.x;
  T my_gc = T(0), my_gmu = T(0);
  if (i < n) {
    const int32_t ci = cell[i];
    const pos_t<T> pi = pos[i];
    const vec_t<T> vi = vel[i];
    const T ri = radius_of(pi);
    const T mi = granule_mass(P, ri);
    const vec_t<T> zero = make_vec<T>(0, 0, 0);
    // a4: x' = x + dt v', v' = v + dt a
    const vec_t<T> gxi_ = gxo[i];
    const IntegrateAdj<T> o = integrate_adj_granule(P, ri, gxi_, gvo[i], gfe ? gfe[i] : zero);
    T gx[3] = {gxi_.x, gxi_.y, gxi_.z};
    T gv[3] = {o.gvt[0], o.gvt[1], o.gvt[2]};
    // a3: F_fl and a_f at the granule
    {
      int m[3];
      T t[3], gdv[3];
      my_gc = g2p_adj_granule<T>(G, P, Fd, ci, pi, vi, o.gFfl, o.gaf, gx, gdv, m, t);
#pragma unroll
      for (int a = 0; a < 3; ++a) gv[a] -= gdv[a];
    }
    // a2: contact pairs (F_ji = -F_ij) and walls
    const T l0 = o.gFc[0], l1 = o.gFc[1], l2 = o.gFc[2];
    T gm = T(0);
    auto pair_of = [&](int64_t j, const PairGeom<T>& g, const vec_t<T>& vj, T rj) {
      const IntegrateAdj<T> oj =
          integrate_adj_granule(P, rj, ldg(&gxo[j]), ldg(&gvo[j]), gfe ? ldg(&gfe[j]) : zero);
      gm += pair_force_adj(P, g.x0, g.x1, g.x2, g.d, g.overlap, vi.x - vj.x, vi.y - vj.y, vi.z - vj.z,
                           pair_mass(P, mi, rj), l0 - oj.gFc[0], l1 - oj.gFc[1], l2 - oj.gFc[2], l0, l1, l2, gx[0],
                           gx[1], gx[2], gv[0], gv[1], gv[2]);
    };
    auto pair = [&](int64_t j, const PairGeom<T>& g) { pair_of(j, g, ldg(&vel[j]), radius_of(ldg(&pos[j]))); };
    const int cx = cell_x(ci), cy = cell_y(ci), cz = cell_z(ci);
    const bool has_f = sizeof(T) == 4 && posf != nullptr;
    const float4 fi = has_f ? __ldg(&posf[i]) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (P.cap) {  // contacts and capillary bridges; a bridge also depends on x_i through sr_i
      T gsr[3];
      const T sri = moisture_ratio_at(G, P, Fd.af, ci, pi, gsr);
      T wsr = T(0);  // sum over bridges of (lambda_i - lambda_j) . dF/d sr_mean
      auto near = [&](int64_t j, int32_t cj, const pos_t<T>& pj, const PairGeom<T>& g) {
        if (g.overlap > T(0)) {
          pair(j, g);
          return;
        }
        const T rj = radius_of(pj);
        const IntegrateAdj<T> oj =
            integrate_adj_granule(P, rj, ldg(&gxo[j]), ldg(&gvo[j]), gfe ? ldg(&gfe[j]) : zero);
        wsr += add_bridge_adj(P, g, ri, rj, sri, moisture_ratio_at(G, P, Fd.af, cj, pj, (T*)nullptr),
                              l0 - oj.gFc[0], l1 - oj.gFc[1], l2 - oj.gFc[2], gx[0], gx[1], gx[2]);
      };
      if (rebuild)
        verlet_build_row_near<T>(G, P, nb, table, n, i, cx, cy, cz, ci, pi, ri, skin, id, pos, near);
      else
        for_each_list_near<T>(G, P, nb, i, cx, cy, cz, pi, ri, has_f, fi, cell, pos, posf, near);
#pragma unroll
      for (int a = 0; a < 3; ++a) gx[a] += T(0.5) * wsr * gsr[a];
    } else if (rebuild) {
      verlet_build_row<T>(G, nb, table, n, i, cx, cy, cz, ci, pi, ri, has_f, fi, skin, id, pos, posf, pair);
    } else {
      bool walked = false;
      if constexpr (sizeof(T) == 4)
        if (has_f) {
          for_each_list_hit(G, nb, i, cx, cy, cz, pi, ri, fi, cell, pos, posf, vel, &s_list[0][threadIdx.x],
                            kSubstepAdjThreads, kAdjHits, pair_of);
          walked = true;
        }
      if (!walked) for_each_list_contact<T>(G, nb, i, cx, cy, cz, ci, pi, ri, has_f, fi, cell, pos, posf, pair);
    }
    if (P.walls)
      gm += add_walls_adj(G, P, pi, ri, mi, vi, cx, cy, cz, l0, l1, l2, gx[0], gx[1], gx[2], gv[0], gv[1], gv[2]);
    my_gmu = gm;
    const int64_t out = perm ? (int64_t)perm[i] : i;
    gxi[out] = make_vec<T>(gx[0], gx[1], gx[2]);
    gvi[out] = make_vec<T>(gv[0], gv[1], gv[2]);
  }
  if (g_cdrag || g_mu) {
    if constexpr (sizeof(T) == 4) {
      // FP32 path: the warp sums in FP32 (the terms are FP32 values), then the
      // CTA's warps in FP64: the FP64 pipe of this GPU runs at 1/64 of the
      // FP32 rate, and a per-thread FP64 shuffle tree cost as much as the
      // rest of the kernel's arithmetic
      float a = my_gc, b = my_gmu;
      for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
      }
      const int w = threadIdx.x >> 5;
      if (lane_id() == 0) {
        s_red[w] = (double)a;
        s_red[32 + w] = (double)b;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        double ga = 0.0, gb = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
          ga += s_red[k];
          gb += s_red[32 + k];
        }
        if (g_cdrag) atomicAdd(g_cdrag, ga);
        if (g_mu) atomicAdd(g_mu, gb);
      }
    } else {
      block_sum2(my_gc, my_gmu, s_red);
      if (threadIdx.x == 0) {
        if (g_cdrag) atomicAdd(g_cdrag, my_gc);
        if (g_mu) atomicAdd(g_mu, my_gmu);
      }
    }
  }
  verlet_call_done(nb, rebuild);  // its barrier also frees s_red
}

}  // namespace gic

using namespace gic;

namespace gic {

// [zero alpha_s] -> k_substep -> [alpha_s out].  sorted: null for gic_substep
// (the substep of s); else gic_step's, which reads `sorted` in a call that
// rebuilt and s otherwise.
static int substep_launch(const DGrid& G, const GicParams* params, const GicGranules* s, const GicGranules* sorted,
                          const void* cell_table, const GicNeighbors* nb, const NbDev& d, const void* u, const void* v,
                          const void* w, const void* p, const void* alpha_f, GicGranules* next, void* f_ex,
                          double* alpha_s, void* Fs_u, void* Fs_v, void* Fs_w, double* sums2, cudaStream_t stream,
                          void* scratch = nullptr, void* moisture = nullptr) {
  int rc;
  const int64_t ncell = (int64_t)G.nx * G.ny * G.nz;
  if (alpha_s && (rc = alpha_begin(alpha_s, ncell, sums2, stream, scratch))) return rc;
  if (s->n > 0) {
    auto go = [&](auto t, auto nt, auto* kern, const DParams<decltype(t)>& P) -> int {
      using T = decltype(t);
      constexpr int NT = decltype(nt)::value;
      constexpr size_t smem = kSubSmem<T, NT>;
      if (smem > 48 * 1024 &&
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return set_error(GIC_ERR_CUDA, "substep: %zu bytes of shared memory refused", smem);
      if (sorted && P.cap) {
        k_moisture<T><<<grid_blocks(s->n, 256), 256, 0, stream>>>(G, P, s->n, state_in<T>(s), state_in<T>(sorted),
                                                                  d.flags, (const T*)alpha_f, (T*)moisture);
        count_launches(1);
      }
      // In a gic_step call the kernel directly follows the sort kernel, which returns
      // at once unless the call rebuilds: it may be launched while that one runs,
      // and waits for it itself: 2 us of every call (29.0 -> 27.5 us on 8,000 FP64
      // granules, 68.4 -> 66.4 on the 1M dam break).  Not under capture, whose
      // graphs keep their plain edges, nor behind alpha_s's clearing.
      cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
      if (sorted && cudaStreamIsCapturing(stream, &cap) != cudaSuccess)
        return set_error(GIC_ERR_CUDA, "substep: the stream's capture status is not available");
      cudaLaunchAttribute early;
      early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
      early.val.programmaticStreamSerializationAllowed = 1;
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(grid_blocks(s->n, NT));
      cfg.blockDim = dim3(NT);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = stream;
      cfg.attrs = &early;
      cfg.numAttrs = sorted && !alpha_s && cap == cudaStreamCaptureStatusNone ? 1 : 0;
      const cudaError_t e = cudaLaunchKernelEx(
          &cfg, kern, G, P, s->n, state_in<T>(s), state_in<T>(sorted ? sorted : s), d, (const uint4*)cell_table,
          (T)nb->skin, fields<T>(u, v, w, p, alpha_f), next->cell, (pos_t<T>*)next->pos, (vec_t<T>*)next->vel,
          next->id, sizeof(T) == 4 ? (float4*)next->posf : (float4*)nullptr, (vec_t<T>*)f_ex, alpha_s, (T*)Fs_u,
          (T*)Fs_v, (T*)Fs_w, sums2, status_word(), (const T*)moisture);
      if (e != cudaSuccess) return set_error(GIC_ERR_CUDA, "substep: launch: %s", cudaGetErrorString(e));
      return GIC_OK;
    };
    constexpr std::integral_constant<int, kSubstepThreads> kWhole{};
    constexpr std::integral_constant<int, kSmallThreads> kSmall{};
    if (s->precision == GIC_FP32) {
      DParams<float> P;
      if ((rc = make_params(params, &P))) return rc;
      rc = go(0.f, kWhole,
              !sorted   ? k_substep<float, kGeneral>
              : P.cap   ? k_substep<float, kStepCap>
              : alpha_s ? k_substep<float, kStep>
                        : k_substep<float, kStep, true>,
              P);
    } else {
      DParams<double> P;
      if ((rc = make_params(params, &P))) return rc;
      if (sorted && s->n <= (int64_t)kSmallPerSm * kSmallThreads * sm_count())
        rc = go(0.0, kSmall,
                P.cap ? k_substep<double, kStepCap, false, kSmallThreads>
                      : k_substep<double, kStep, false, kSmallThreads>,
                P);
      else
        rc = go(0.0, kWhole,
                !sorted ? k_substep<double, kGeneral> : P.cap ? k_substep<double, kStepCap> : k_substep<double, kStep>,
                P);
    }
    if (rc) return rc;
    count_launches(1);
  }
  if (alpha_s && (rc = alpha_end(G, s->precision, alpha_s, ncell, sums2, stream, scratch))) return rc;
  return GIC_OK;
}

}  // namespace gic

extern "C" int gic_substep(const GicGrid* grid, const GicParams* params, const GicGranules* sorted,
                           const void* cell_table, const GicNeighbors* nb, const void* u, const void* v,
                           const void* w, const void* p, const void* alpha_f, GicGranules* next, void* f_ex,
                           double* alpha_s, void* Fs_u, void* Fs_v, void* Fs_w, double* sums2,
                           gic_stream_t stream) {
  GIC_RANGE("gic_substep");
  {  // parameters first, before any device work
    DParams<double> chk;
    if (int rc0 = make_params(params, &chk)) return rc0;
  }
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  const GicGranules* s = sorted;
  if ((rc = check_granules(s, "gic_substep sorted", true))) return rc;
  if ((rc = check_granules(next, "gic_substep next"))) return rc;
  if (next->n != s->n || next->precision != s->precision)
    return set_error(GIC_ERR_INVALID, "gic_substep: sorted/next differ in size or precision");
  if (!u || !v || !w || !p || !alpha_f) return set_error(GIC_ERR_INVALID, "gic_substep: null fluid field");
  bool fs = Fs_u || Fs_v || Fs_w;
  if (fs && !(Fs_u && Fs_v && Fs_w)) return set_error(GIC_ERR_INVALID, "gic_substep: give all three F_s arrays or none");
  if (sums2 && !alpha_s) return set_error(GIC_ERR_INVALID, "gic_substep: sums2 needs alpha_s");
  if ((rc = check_vecs(s->precision, "gic_substep", {f_ex}))) return rc;
  NbDev d;
  if ((rc = verlet_prelude(G, params, s, cell_table, nb, nullptr, stream, "gic_substep", &d, false))) return rc;
  if ((rc = substep_launch(G, params, s, nullptr, cell_table, nb, d, u, v, w, p, alpha_f, next, f_ex, alpha_s, Fs_u,
                           Fs_v, Fs_w, sums2, (cudaStream_t)stream)))
    return rc;
  GIC_CHECK_LAUNCH("gic_substep");
  return GIC_OK;
}

static bool share_array(const GicGranules* a, const GicGranules* b) {
  return a->cell == b->cell || a->pos == b->pos || a->vel == b->vel || a->id == b->id ||
         (a->posf && a->posf == b->posf);
}

static int check_sort_workspace(const GicGrid* grid, const GicGranules* s, const void* ws, size_t ws_bytes,
                                const char* what) {
  size_t need = 0;
  if (int rc = gic_workspace_size(grid, s->n, s->precision, &need)) return rc;
  if (!ws || ws_bytes < need)
    return set_error(GIC_ERR_WORKSPACE, "%s: workspace of %zu bytes needed, %zu given", what, need, ws_bytes);
  if ((uintptr_t)ws % 256) return set_error(GIC_ERR_ALIGN, "%s: workspace must be 256-byte aligned", what);
  return GIC_OK;
}

extern "C" int gic_step(const GicGrid* grid, const GicParams* params, const GicGranules* state, GicGranules* next,
                        GicGranules* sorted, int32_t* perm, void* cell_table, void* ws, size_t ws_bytes,
                        const GicNeighbors* nb, const void* u, const void* v, const void* w, const void* p,
                        const void* alpha_f, double* alpha_s, void* Fs_u, void* Fs_v, void* Fs_w, double* sums2,
                        gic_stream_t stream) {
  GIC_RANGE("gic_step");
  {  // parameters first, before any device work
    DParams<double> chk;
    if (int rc0 = make_params(params, &chk)) return rc0;
  }
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  if (!params) return set_error(GIC_ERR_INVALID, "gic_step: params is NULL");
  if ((rc = check_granules(state, "gic_step state", true))) return rc;
  if ((rc = check_granules(next, "gic_step next", true))) return rc;
  if ((rc = check_granules(sorted, "gic_step sorted", true))) return rc;
  if (next->n != state->n || next->precision != state->precision || sorted->n != state->n ||
      sorted->precision != state->precision)
    return set_error(GIC_ERR_INVALID, "gic_step: state/next/sorted size or precision differ");
  if (share_array(state, next) || share_array(state, sorted) || share_array(next, sorted))
    return set_error(GIC_ERR_INVALID, "gic_step: state, next and sorted must not share arrays");
  if (state->n > 0 && !perm) return set_error(GIC_ERR_INVALID, "gic_step: perm is NULL");
  if (!u || !v || !w || !p || !alpha_f) return set_error(GIC_ERR_INVALID, "gic_step: null fluid field");
  bool fs = Fs_u || Fs_v || Fs_w;
  if (fs && !(Fs_u && Fs_v && Fs_w)) return set_error(GIC_ERR_INVALID, "gic_step: give all three F_s arrays or none");
  if (sums2 && !alpha_s) return set_error(GIC_ERR_INVALID, "gic_step: sums2 needs alpha_s");
  if (!nb) return set_error(GIC_ERR_INVALID, "gic_step: neighbours struct is NULL");
  NbDev d;
  if ((rc = verlet_view(G, state, cell_table, nb, "gic_step", true, &d))) return rc;
  if (state->n == 0) return GIC_OK;
  if ((rc = check_sort_workspace(grid, state, ws, ws_bytes, "gic_step"))) return rc;
  const cudaStream_t st = (cudaStream_t)stream;
  if ((rc = launch_step_sort(G, state, sorted, perm, cell_table, ws, d.flags, kBarrierPolls, st))) return rc;
  if ((rc = substep_launch(G, params, state, sorted, cell_table, nb, d, u, v, w, p, alpha_f, next, nullptr, alpha_s,
                           Fs_u, Fs_v, Fs_w, sums2, st, ws, (char*)ws + sort_layout(G, state->n).off_keys_b)))
    return rc;
  GIC_CHECK_LAUNCH("gic_step");
  return GIC_OK;
}

extern "C" int gic_step_sort(const GicGrid* grid, const GicGranules* state, GicGranules* sorted, int32_t* perm,
                             void* cell_table, void* ws, size_t ws_bytes, const GicNeighbors* nb, int32_t polls,
                             gic_stream_t stream) {
  GIC_RANGE("gic_step_sort");
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  if ((rc = check_granules(state, "gic_step_sort state", true))) return rc;
  if ((rc = check_granules(sorted, "gic_step_sort sorted", true))) return rc;
  if (sorted->n != state->n || sorted->precision != state->precision)
    return set_error(GIC_ERR_INVALID, "gic_step_sort: state/sorted size or precision differ");
  if (share_array(state, sorted))
    return set_error(GIC_ERR_INVALID, "gic_step_sort: state and sorted must not share arrays");
  if (state->n > 0 && !perm) return set_error(GIC_ERR_INVALID, "gic_step_sort: perm is NULL");
  if (!nb) return set_error(GIC_ERR_INVALID, "gic_step_sort: neighbours struct is NULL");
  NbDev d;
  if ((rc = verlet_view(G, state, cell_table, nb, "gic_step_sort", true, &d))) return rc;
  if (state->n == 0) return GIC_OK;
  if ((rc = check_sort_workspace(grid, state, ws, ws_bytes, "gic_step_sort"))) return rc;
  if ((rc = launch_step_sort(G, state, sorted, perm, cell_table, ws, d.flags, polls < 0 ? kBarrierPolls : polls,
                             (cudaStream_t)stream)))
    return rc;
  GIC_CHECK_LAUNCH("gic_step_sort");
  return GIC_OK;
}

extern "C" int gic_substep_adj(const GicGrid* grid, const GicParams* params, const GicGranules* sorted,
                               const int32_t* perm, const void* cell_table, const GicNeighbors* nb, const void* u,
                               const void* v, const void* w, const void* p, const void* alpha_f,
                               const void* g_pos_out, const void* g_vel_out, const void* g_f_ex, void* g_pos_in,
                               void* g_vel_in, double* g_cdrag, double* g_mu, gic_stream_t stream) {
  GIC_RANGE("gic_substep_adj");
  {  // parameters first, before any device work
    DParams<double> chk;
    if (int rc0 = make_params(params, &chk)) return rc0;
  }
  DGrid G;
  int rc = make_grid(grid, &G);
  if (rc) return rc;
  const GicGranules* s = sorted;
  if ((rc = check_granules(s, "gic_substep_adj sorted", true))) return rc;
  if (!u || !v || !w || !p || !alpha_f) return set_error(GIC_ERR_INVALID, "gic_substep_adj: null fluid field");
  if (!g_pos_out || !g_vel_out || !g_pos_in || !g_vel_in)
    return set_error(GIC_ERR_INVALID, "gic_substep_adj: null gradient array");
  if ((rc = check_vecs(s->precision, "gic_substep_adj", {g_pos_out, g_vel_out, g_f_ex, g_pos_in, g_vel_in})))
    return rc;
  // partners read the upstream gradients while others are written
  const void* ins[3] = {g_pos_out, g_vel_out, g_f_ex};
  for (const void* q : ins)
    if (q && (q == g_pos_in || q == g_vel_in))
      return set_error(GIC_ERR_INVALID, "gic_substep_adj: an output aliases an input gradient");
  if (g_pos_in == g_vel_in) return set_error(GIC_ERR_INVALID, "gic_substep_adj: g_pos_in aliases g_vel_in");
  NbDev d;
  if ((rc = verlet_prelude(G, params, s, cell_table, nb, nullptr, stream, "gic_substep_adj", &d, false))) return rc;
  if (s->n == 0) return GIC_OK;
  const unsigned blocks = grid_blocks(s->n, kSubstepAdjThreads);
  if (s->precision == GIC_FP32) {
    DParams<float> P;
    if ((rc = make_params(params, &P))) return rc;
    k_substep_adj<float><<<blocks, kSubstepAdjThreads, 0, stream>>>(
        G, P, s->n, s->cell, (const uint4*)s->pos, (const float4*)s->posf, (const float4*)s->vel, s->id, d,
        (const uint4*)cell_table, (float)nb->skin, fields<float>(u, v, w, p, alpha_f), (const float4*)g_pos_out,
        (const float4*)g_vel_out, (const float4*)g_f_ex, perm, (float4*)g_pos_in, (float4*)g_vel_in, g_cdrag, g_mu);
  } else {
    DParams<double> P;
    if ((rc = make_params(params, &P))) return rc;
    k_substep_adj<double><<<blocks, kSubstepAdjThreads, 0, stream>>>(
        G, P, s->n, s->cell, (const d4*)s->pos, nullptr, (const d4*)s->vel, s->id, d, (const uint4*)cell_table,
        nb->skin, fields<double>(u, v, w, p, alpha_f), (const d4*)g_pos_out, (const d4*)g_vel_out,
        (const d4*)g_f_ex, perm, (d4*)g_pos_in, (d4*)g_vel_in, g_cdrag, g_mu);
  }
  count_launches(1);
  GIC_CHECK_LAUNCH("gic_substep_adj");
  return GIC_OK;
}
