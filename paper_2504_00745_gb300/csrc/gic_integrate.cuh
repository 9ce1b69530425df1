// gic_integrate.cuh -- device side of a4 (virtual-mass symplectic Euler,
// Sec. 5.2 Eq. sand kine; Alg. 2 MoveParticle), shared by the integrate
// kernel and the fused substep.
#pragma once

#include "gic_internal.cuh"

namespace gic {

template <typename T>
struct Masses {
  T m, ma, sum;  // granule, added mass, their sum (rounded once)
};

template <typename T>
__device__ __forceinline__ Masses<T> masses(const DParams<T>& P, T r) {
  T V = T(4.0 / 3.0 * kPi) * r * r * r;
  Masses<T> M;
  M.m = P.rho_s * V;
  M.ma = P.vm ? T(0.5) * P.rho_f * V : T(0);
  M.sum = fma(P.rho_s, V, M.ma);
  return M;
}

__device__ __forceinline__ void advance_axis(const DGrid& G, float dt, float v, uint32_t q, int c, int nc,
                                             uint32_t& q_out, int& c_out, uint32_t& flags) {
  float inc_f = dt * v * G.inv_unit_f;
  // a move of less than a cell that stays in the domain: 32-bit integers
  if (fabsf(inc_f) < 0x1p30f && q <= kFracMask) {
    const int s = (int)q + __float2int_rn(inc_f);
    const int cn = c + (s >> kFracBits);  // floor division by 2^30
    if (cn >= 0 && cn < nc) {
      q_out = (uint32_t)s & kFracMask;
      c_out = cn;
      return;
    }
  }
  // clamp far beyond one cell so the integer conversion is defined
  inc_f = fminf(fmaxf(inc_f, -0x1p40f), 0x1p40f);
  long long s = (long long)q + __float2ll_rn(inc_f);
  long long shift = s >> kFracBits;  // floor division by 2^30
  q_out = (uint32_t)(s & (long long)kFracMask);
  long long cn = (long long)c + shift;
  if (shift > 1 || shift < -1) flags |= GIC_STATUS_FAST;
  if (cn < 0) {
    cn = 0;
    q_out = 0;
    flags |= GIC_STATUS_OUT_OF_DOMAIN;
  } else if (cn > nc - 1) {
    cn = nc - 1;
    q_out = kFracMask;
    flags |= GIC_STATUS_OUT_OF_DOMAIN;
  }
  c_out = (int)cn;
}

__device__ __forceinline__ void advance_axis(const DGrid& G, double dt, double v, double o, int c, int nc,
                                             double& o_out, int& c_out, uint32_t& flags) {
  double x = fma(dt, v, o);
  // still in the cell: 0 <= x < h_c, compared as integers (a negative or NaN x is
  // above every such value), without the floor and its conversions; a cell beyond the
  // grid is clamped below
  if (c < nc && (unsigned long long)__double_as_longlong(x) < (unsigned long long)__double_as_longlong(G.hc)) {
    o_out = x;
    c_out = c;
    return;
  }
  double sh = floor(x * G.inv_hc);
  if (!(fabs(sh) < 1e9)) sh = x > 0 ? 1e9 : -1e9;
  long long shift = (long long)sh;
  x = fma(-sh, G.hc, x);
  // guard against rounding just outside [0, h_c)
  if (x < 0.0) x = 0.0;
  if (x >= G.hc) x = nextafter(G.hc, 0.0);
  if (shift > 1 || shift < -1) flags |= GIC_STATUS_FAST;
  long long cn = (long long)c + shift;
  if (cn < 0) {
    cn = 0;
    x = 0.0;
    flags |= GIC_STATUS_OUT_OF_DOMAIN;
  } else if (cn > nc - 1) {
    cn = nc - 1;
    x = nextafter(G.hc, 0.0);
    flags |= GIC_STATUS_OUT_OF_DOMAIN;
  }
  o_out = x;
  c_out = (int)cn;
}

// One granule: new cell / position record / velocity and the exchange force
// f_ex = F_fl + m_a (a_f - a) from the forces on it; status bits in flags.
template <typename T>
__device__ __forceinline__ void integrate_granule(const DGrid& G, const DParams<T>& P, int32_t c, const pos_t<T>& p,
                                                  const vec_t<T>& v, T fc0, T fc1, T fc2, T ff0, T ff1, T ff2,
                                                  T fa0, T fa1, T fa2, int32_t& c_out, pos_t<T>& p_out,
                                                  vec_t<T>& v_out, T& fe0, T& fe1, T& fe2, uint32_t& flags) {
  Masses<T> M = masses(P, radius_of(p));
  T inv = T(1) / M.sum;
  T a0 = fma(M.ma, fa0, fma(M.m, P.g[0], fc0 + ff0)) * inv;
  T a1 = fma(M.ma, fa1, fma(M.m, P.g[1], fc1 + ff1)) * inv;
  T a2 = fma(M.ma, fa2, fma(M.m, P.g[2], fc2 + ff2)) * inv;
  T v0 = fma(P.dt, a0, v.x), v1 = fma(P.dt, a1, v.y), v2 = fma(P.dt, a2, v.z);
  if (!finite_bits(v0) || !finite_bits(v1) || !finite_bits(v2)) flags |= GIC_STATUS_NONFINITE;
  int c3[3] = {cell_x(c), cell_y(c), cell_z(c)};
  int cn[3];
  p_out = p;
  advance_axis(G, P.dt, v0, p.x, c3[0], G.nc[0], p_out.x, cn[0], flags);
  advance_axis(G, P.dt, v1, p.y, c3[1], G.nc[1], p_out.y, cn[1], flags);
  advance_axis(G, P.dt, v2, p.z, c3[2], G.nc[2], p_out.z, cn[2], flags);
  c_out = pack_cell(cn[0], cn[1], cn[2]);
  v_out = make_vec<T>(v0, v1, v2);
  fe0 = fma(M.ma, fa0 - a0, ff0);
  fe1 = fma(M.ma, fa1 - a1, ff1);
  fe2 = fma(M.ma, fa2 - a2, ff2);
}

// Adjoint of integrate_granule: from the gradients gx, gv, gf of (x', v',
// f_ex) of a granule of radius r to those of v (gvt; x's is gx itself), F_c,
// F_fl and a_f.  x' = x + dt v', v' = v + dt a, a = (F_c + F_fl + m g +
// m_a a_f) / (m + m_a), f_ex = F_fl + m_a (a_f - a).
template <typename T>
struct IntegrateAdj {
  T gvt[3], gFc[3], gFfl[3], gaf[3];
};

template <typename T>
__device__ __forceinline__ IntegrateAdj<T> integrate_adj_granule(const DParams<T>& P, T r, const vec_t<T>& gx,
                                                                 const vec_t<T>& gv, const vec_t<T>& gf) {
  const Masses<T> M = masses(P, r);
  const T inv = T(1) / M.sum;
  IntegrateAdj<T> o;
  const T x[3] = {gx.x, gx.y, gx.z}, v[3] = {gv.x, gv.y, gv.z}, f[3] = {gf.x, gf.y, gf.z};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    o.gvt[a] = v[a] + P.dt * x[a];
    const T ga = P.dt * o.gvt[a] - M.ma * f[a];  // a enters v' (dt) and f_ex (-m_a)
    o.gFc[a] = ga * inv;
    o.gFfl[a] = ga * inv + f[a];
    o.gaf[a] = M.ma * (ga * inv + f[a]);
  }
  return o;
}

}  // namespace gic
