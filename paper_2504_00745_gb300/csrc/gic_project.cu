// gic_project.cu -- the velocity and density projections that consume
// alpha_s (Sec. 5.1: Eqs. discret momentum, backward Euler, bring2, ppe1 a/b
// and position change; the limits stated after Eq. position change; the face
// weight beta_j of the appendix on the Push-Out boundary condition).
//
// Both systems are A p = b with (A p)_c = sum over the cell's faces of
// beta_f (p_c - p_nb): beta_f the mean alpha_f' of the two cells, the inner
// cell's alpha_f' on an open side (p_nb = 0 beyond), no term on a solid side.
// A is symmetric positive definite (an open side is required).
//
// GB300's FP64 rate is a small fraction of its FP32 rate, and an all-FP32 CG
// stalls at a relative residual of order eps_32 * cond(A) (~1e-3 on a 128^3
// box with one open side).  So the solve is mixed-precision iterative
// refinement: the solution p and each residual b - A p are FP64 (one FP64
// stencil pass per refinement step), and each correction A e = r comes from
// an FP32 conjugate-gradient run, preconditioned by a geometric multigrid
// V-cycle, to a modest reduction.  The CG iterations are queued a few at a time
// between host reads of the stop flag.
// Reductions are deterministic: every block writes a partial sum, and the
// block that finishes last (an atomic ticket, no waiting) adds the partials
// in index order and writes the scalar that the next kernels read.
#include <math.h>
#include <string.h>

#include "gic_internal.cuh"

namespace gic {

constexpr int kProjThreads = 256;

struct PGrid {
  int nx, ny, nz;
  int64_t n;        // cells (< 2^30: cell and face indices are 32-bit)
  int64_t nxy;      // nx * ny
  int open[6];      // -x, +x, -y, +y, -z, +z
};

// Device scalars of the solver (in the workspace).
struct ProjRed {
  double dy;       // d . A d
  double rz[2];    // r . M^-1 r of the current and the next CG iterate
  double rr;       // r . r of the FP32 iterate
  double rr64, bb; // ||b - A p||^2 (FP64) and ||b||^2
  double rr_stop;  // the CG run stops when r . r <= rr_stop
  unsigned ticket; // blocks done with the current kernel
  int done, iters; // stop flag and iteration count of the CG run
};

// Every block calls it once with its partials (valid in thread 0); the
// block that arrives last sums all partials in index order into out[]
// (NV values, component-major partials P[v * gridDim.x + block]) and resets
// the ticket.  Returns true in that block (all threads).
template <int NV>
__device__ __forceinline__ bool reduce_last(const double (&v)[NV], double* __restrict__ P, ProjRed* red,
                                            double* const (&out)[NV]) {
  __shared__ bool last;
  __shared__ double smem[32];
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) P[q * gridDim.x + blockIdx.x] = v[q];
    __threadfence();
    last = atomicAdd(&red->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    double s = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) s += __ldcg(&P[q * gridDim.x + b]);
    s = block_sum(s, smem);
    if (threadIdx.x == 0) *out[q] = s;
  }
  if (threadIdx.x == 0) red->ticket = 0u;
  return true;
}

// Compensated FP32 sum (Kahan): the CG's per-thread dot-product partials stay
// off the FP64 pipe, whose rate on GB300 is a small fraction of FP32's.
struct KahanF {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float y = __fsub_rn(x, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
  }
};

// Sum of the CTA's compensated partials, in double, valid in thread 0: the warps
// add (hi, lo) float pairs with TwoSum, and only one value per warp takes the
// FP64 pipe (a tree of double shuffles in every warp cost 3 us of a pass at
// 128^3).  smem: one double per warp.
__device__ __forceinline__ double block_sum(const KahanF& k, double* smem) {
  float h = k.s, l = -k.c;
  for (int off = 16; off > 0; off >>= 1) {
    const float h2 = __shfl_down_sync(0xffffffffu, h, off), l2 = __shfl_down_sync(0xffffffffu, l, off);
    const float t = __fadd_rn(h, h2), b = __fsub_rn(t, h);
    l = __fadd_rn(__fadd_rn(l, l2), __fadd_rn(__fsub_rn(h, __fsub_rn(t, b)), __fsub_rn(h2, b)));
    h = t;
  }
  if (lane_id() == 0) smem[threadIdx.x >> 5] = (double)h + (double)l;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += smem[w];
  return r;
}

// alpha_f' = 1 - min(alpha_s, alpha_s_max); a NaN alpha_s stays NaN (and is reported)
__device__ __forceinline__ double target_fraction(double alpha_s, double amax) {
  return 1.0 - (alpha_s > amax ? amax : alpha_s);
}

// alpha_f' as float (the FP32 operator of the corrections; the FP64 residual
// forms it from alpha_s itself).
__global__ void __launch_bounds__(kProjThreads) k_proj_prep(PGrid g, const double* __restrict__ alpha_s, double amax,
                                                            float* __restrict__ ap32) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < g.n; c += (int64_t)gridDim.x * blockDim.x)
    ap32[c] = (float)target_fraction(alpha_s[c], amax);
}

struct ProjScales {
  double vel;       // rho h / dt: b1 = vel * (sum of beta v over low faces - over high faces)
  double den;       // -rho h^2 / dt^2: b2 = den * alpha' (1 - clamp(ratio))
  double rmin, rmax, amax;
};

// FP64 face weights of the operator (computed once per call, so that each
// residual pass spends its FP64 work on the stencil itself): the mean
// alpha_f' of the two cells, the inner cell's on an open side, 0 on a solid
// side.  Face arrays as the velocity components, x fastest.
__global__ void __launch_bounds__(kProjThreads) k_proj_faces64(PGrid g, unsigned open, const double* __restrict__ alpha_s,
                                                               double amax, double* __restrict__ fx,
                                                               double* __restrict__ fy, double* __restrict__ fz) {
  const unsigned nx = g.nx, ny = g.ny, nz = g.nz;
  const unsigned nu = (nx + 1) * ny * nz, nv = nx * (ny + 1) * nz, nw = nx * ny * (nz + 1);
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < nu + nv + nw; q += gridDim.x * blockDim.x) {
    unsigned a, f;
    if (q < nu) {
      a = 0, f = q;
    } else if (q < nu + nv) {
      a = 1, f = q - nu;
    } else {
      a = 2, f = q - nu - nv;
    }
    const unsigned sx = nx + (a == 0), sy = ny + (a == 1);
    const unsigned k = f / (sx * sy), rem = f - k * sx * sy, j = rem / sx, i = rem - j * sx;
    const unsigned pos = a == 0 ? i : (a == 1 ? j : k);
    const unsigned m = a == 0 ? nx : (a == 1 ? ny : nz);
    const unsigned stride = a == 0 ? 1u : (a == 1 ? nx : nx * ny);
    // the cell above the face (valid when pos < m) and the one below (pos > 0)
    const unsigned c_hi = i + nx * (j + ny * k), c_lo = c_hi - stride;
    double wgt;
    if (pos > 0 && pos < m)
      wgt = 0.5 * (target_fraction(alpha_s[c_hi], amax) + target_fraction(alpha_s[c_lo], amax));
    else if (pos == 0)
      wgt = (open >> (2 * a)) & 1u ? target_fraction(alpha_s[c_hi], amax) : 0.0;
    else
      wgt = (open >> (2 * a + 1)) & 1u ? target_fraction(alpha_s[c_lo], amax) : 0.0;
    (a == 0 ? fx : (a == 1 ? fy : fz))[f] = wgt;
  }
}

// Right-hand side b of system `which` (1: velocity, 2: density) in FP64, kept for
// the solve's later residuals: with p = 0 it is the first residual.  Starts the
// FP32 correction run: r32 = b, e = 0, and arms its stop test.  Scalars: ||b||^2
// as ||r||^2 and ||b||^2.
__global__ void __launch_bounds__(kProjThreads) k_proj_rhs(
    PGrid g, int which, ProjScales S, const double* __restrict__ alpha_s, const float* __restrict__ alpha_star,
    const float* __restrict__ u, const float* __restrict__ v, const float* __restrict__ w,
    const double* __restrict__ fx, const double* __restrict__ fy, const double* __restrict__ fz,
    double* __restrict__ b64, float* __restrict__ r32, float* __restrict__ e32, double inner_tol2,
    double* __restrict__ P, ProjRed* red, uint32_t* status) {
  __shared__ double smem[64];
  double bb = 0.0;
  const unsigned n = (unsigned)g.n, nx = g.nx, ny = g.ny, nxy = nx * ny;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    double b;
    if (which == 1) {
      const unsigned k = c / nxy, rem = c - k * nxy, j = rem / nx, i = rem - j * nx;
      const unsigned fu = i + (nx + 1) * (j + ny * k), fv = i + nx * (j + (ny + 1) * k);
      // b1 = (rho h / dt) (sum over low faces - sum over high faces) of beta v*
      const double flux = (fx[fu] * (double)u[fu] - fx[fu + 1] * (double)u[fu + 1]) +
                          (fy[fv] * (double)v[fv] - fy[fv + nx] * (double)v[fv + nx]) +
                          (fz[c] * (double)w[c] - fz[c + nxy] * (double)w[c + nxy]);
      b = S.vel * flux;
    } else {
      const double ac = target_fraction(alpha_s[c], S.amax);
      const double q = (double)alpha_star[c] / ac;
      const double ratio = q < S.rmin ? S.rmin : (q > S.rmax ? S.rmax : q);  // NaN stays NaN
      b = S.den * ac * (1.0 - ratio);
    }
    if (!isfinite(b)) raise_status(status, GIC_STATUS_NONFINITE);
    b64[c] = b;
    r32[c] = (float)b;
    e32[c] = 0.f;
    bb += b * b;
  }
  bb = block_sum(bb, smem);
  const double vals[2] = {bb, bb};
  double* const outs[2] = {&red->rr64, &red->bb};
  if (reduce_last<2>(vals, P, red, outs) && threadIdx.x == 0) {  // arm the CG run on this residual
    red->rr_stop = inner_tol2 * red->rr64;
    red->done = 0;
    red->iters = 0;
  }
}

// FP64 residual r = b - A p; starts the next FP32 correction run as k_proj_rhs
// does.  Bound by the FP64 pipe (15 operations per cell; with b formed again in
// every pass 30): 72 us at 128^3, 140 before.
__global__ void __launch_bounds__(kProjThreads) k_proj_residual(
    PGrid g, const double* __restrict__ b64, const double* __restrict__ fx, const double* __restrict__ fy,
    const double* __restrict__ fz, const double* __restrict__ p, float* __restrict__ r32, float* __restrict__ e32,
    double inner_tol2, double* __restrict__ P, ProjRed* red, uint32_t* status) {
  __shared__ double smem[32];
  double rr = 0.0;
  const unsigned n = (unsigned)g.n, nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    const unsigned k = c / nxy, rem = c - k * nxy, j = rem / nx, i = rem - j * nx;
    const unsigned fu = i + (nx + 1) * (j + ny * k), fv = i + nx * (j + (ny + 1) * k);
    const double pc = p[c];
    // (A p)_c as differences (a neighbour beyond an open side is 0; solid sides have weight 0)
    double Ap = 0.0;
    Ap = fma(fx[fu], i > 0 ? pc - p[c - 1] : pc, Ap);
    Ap = fma(fx[fu + 1], i + 1 < nx ? pc - p[c + 1] : pc, Ap);
    Ap = fma(fy[fv], j > 0 ? pc - p[c - nx] : pc, Ap);
    Ap = fma(fy[fv + nx], j + 1 < ny ? pc - p[c + nx] : pc, Ap);
    Ap = fma(fz[c], k > 0 ? pc - p[c - nxy] : pc, Ap);
    Ap = fma(fz[c + nxy], k + 1 < nz ? pc - p[c + nxy] : pc, Ap);
    const double r = b64[c] - Ap;
    if (!isfinite(r)) raise_status(status, GIC_STATUS_NONFINITE);
    r32[c] = (float)r;
    e32[c] = 0.f;
    rr += r * r;
  }
  rr = block_sum(rr, smem);
  const double vals[1] = {rr};
  double* const outs[1] = {&red->rr64};
  if (reduce_last<1>(vals, P, red, outs) && threadIdx.x == 0) {  // arm the CG run on this residual
    red->rr_stop = inner_tol2 * red->rr64;
    red->done = 0;
    red->iters = 0;
  }
}

// ---- multigrid preconditioner (FP32) ----
//
// A level is the operator (A x)_c = sum over c's faces of beta_f (x_c -
// x_nb) on an nx ny nz cell grid, with x_nb = 0 beyond the boundary: open
// sides carry their weight, solid sides weight 0, so every level is the same
// kind of operator.  Level 0 has the face weights of the projection; level
// l + 1 halves each axis (ceil), a coarse cell covering up to 2 x 2 x 2 fine
// cells, and its face weights are the sums of the fine face weights across
// each coarse face: the Galerkin product R A P with P the piecewise-constant
// interpolation and R = P^T.  The V-cycle smooths with red-black Gauss-Seidel
// (red then black before the coarse correction, black then red after it, so
// the preconditioner is symmetric), restricts the residual by summing the
// children, adds kMgOmega times the interpolated coarse correction (the
// constant interpolation under-corrects; 1.6 keeps the preconditioner
// positive definite and halves the CG iterations against 1.0), and runs the
// small levels, down to the coarsest (every axis <= 4 cells, solved by a
// palindromic sequence of Gauss-Seidel sweeps), in one CTA.
//
// A level takes four passes instead of a pass per half sweep and transfer.
// Down: the red half sweep from x = 0 is invd b, which the black cells form for
// their neighbours themselves (mg_down); the black cells' residuals then vanish,
// so the restriction reads the red children alone (mg_restrict).  Up: the black
// half sweep adds the coarse correction to its red neighbours as it reads them,
// and its own old value and the red cells' do not outlive the two half sweeps,
// so the interpolation is never stored (mg_up_black, mg_up_red).  A thread takes
// the two cells of a pair along x, one of each colour, so that no lane idles on
// the other colour.  128^3, per CG iteration: level 0 12 + 10 + 10 + 17 us (the
// last with r . z), the levels below 27 us, the tail 16 us, the CG passes 38 us;
// bound by the traffic between L2 and L1 (each array about 2.4 times through the
// halos of 64 x 8 x 4 cells).  Before, with a pass per half sweep and transfer,
// 230 us in 26 launches (now 16).  Runs of four cells per thread with 16-byte
// loads measured the same.
constexpr float kMgOmega = 1.6f;
constexpr int kMgCoarsePairs = 8;  // (black, red) sweep pairs after the first red sweep on the coarsest level
constexpr int kMgMaxLevels = 16;

struct MgLevel {
  int nx, ny, nz;
  float *bx, *by, *bz;  // face weights: (nx+1) ny nz, nx (ny+1) nz, nx ny (nz+1)
  float* invd;          // 1 / (sum of the cell's six face weights)
  const float* ap;      // level 0: alpha_f', from which its passes form the face weights again
  unsigned open;        // level 0: the open sides
  float *x, *b;         // correction and right-hand side
};

__device__ __forceinline__ bool stopped(const ProjRed* red) { return *(volatile const int*)&red->done != 0; }

__device__ __forceinline__ void level_ijk(const MgLevel& L, unsigned c, unsigned& i, unsigned& j, unsigned& k) {
  const unsigned nx = (unsigned)L.nx, nxy = nx * (unsigned)L.ny;
  k = c / nxy;
  const unsigned r = c - k * nxy;
  j = r / nx;
  i = r - j * nx;
}

// sum of the cell's six face weights
__device__ __forceinline__ float level_diag(const MgLevel& L, unsigned c, unsigned i, unsigned j, unsigned k) {
  const unsigned nx = (unsigned)L.nx, ny = (unsigned)L.ny, nxy = nx * ny;
  const unsigned fx = i + (nx + 1) * (j + ny * k);
  const unsigned fy = i + nx * (j + (ny + 1) * k);
  return ((L.bx[fx] + L.bx[fx + 1]) + (L.by[fy] + L.by[fy + nx])) + (L.bz[c] + L.bz[c + nxy]);
}

// Level-0 face weights from alpha_f' (float): the mean of the two cells, the
// inner cell's value on an open side, 0 on a solid side.
__global__ void __launch_bounds__(kProjThreads) k_mg_faces0(MgLevel L, unsigned open, const float* __restrict__ ap) {
  const unsigned nx = L.nx, ny = L.ny, nz = L.nz;
  const unsigned nu = (nx + 1) * ny * nz, nv = nx * (ny + 1) * nz, nw = nx * ny * (nz + 1);
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < nu + nv + nw; q += gridDim.x * blockDim.x) {
    unsigned a, f;
    if (q < nu) {
      a = 0, f = q;
    } else if (q < nu + nv) {
      a = 1, f = q - nu;
    } else {
      a = 2, f = q - nu - nv;
    }
    const unsigned sx = nx + (a == 0), sy = ny + (a == 1);
    const unsigned k = f / (sx * sy), rem = f - k * sx * sy, j = rem / sx, i = rem - j * sx;
    const unsigned pos = a == 0 ? i : (a == 1 ? j : k);
    const unsigned m = a == 0 ? nx : (a == 1 ? ny : nz);
    const unsigned stride = a == 0 ? 1u : (a == 1 ? nx : nx * ny);
    // the cell above the face (valid when pos < m) and the one below (pos > 0)
    const unsigned c_hi = i + nx * (j + ny * k), c_lo = c_hi - stride;
    float wgt;
    if (pos > 0 && pos < m)
      wgt = 0.5f * (ap[c_hi] + ap[c_lo]);
    else if (pos == 0)
      wgt = (open >> (2 * a)) & 1u ? ap[c_hi] : 0.f;
    else
      wgt = (open >> (2 * a + 1)) & 1u ? ap[c_lo] : 0.f;
    (a == 0 ? L.bx : (a == 1 ? L.by : L.bz))[f] = wgt;
  }
}

// Coarse face weights: the sum of the fine face weights across each coarse face.
__global__ void __launch_bounds__(kProjThreads) k_mg_coarsen(MgLevel F, MgLevel C) {
  const unsigned cx = C.nx, cy = C.ny, cz = C.nz;
  const unsigned nu = (cx + 1) * cy * cz, nv = cx * (cy + 1) * cz, nw = cx * cy * (cz + 1);
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < nu + nv + nw; q += gridDim.x * blockDim.x) {
    unsigned a, f;
    if (q < nu) {
      a = 0, f = q;
    } else if (q < nu + nv) {
      a = 1, f = q - nu;
    } else {
      a = 2, f = q - nu - nv;
    }
    const unsigned sx = cx + (a == 0), sy = cy + (a == 1);
    const unsigned K = f / (sx * sy), rem = f - K * sx * sy, J = rem / sx, I = rem - J * sx;
    const unsigned fnx = F.nx, fny = F.ny, fnz = F.nz;
    // the fine face position along axis a, and the 2 x 2 footprint on the other two axes
    unsigned lo[3] = {2 * I, 2 * J, 2 * K}, hi[3], lim[3] = {fnx, fny, fnz};
    for (int b = 0; b < 3; ++b) hi[b] = min(lo[b] + 2, lim[b]);
    lo[a] = min(lo[a], lim[a]);
    hi[a] = lo[a] + 1;
    const float* src = a == 0 ? F.bx : (a == 1 ? F.by : F.bz);
    const unsigned fsx = fnx + (a == 0), fsy = fny + (a == 1);
    float s = 0.f;
    for (unsigned k = lo[2]; k < hi[2]; ++k)
      for (unsigned j = lo[1]; j < hi[1]; ++j)
        for (unsigned i = lo[0]; i < hi[0]; ++i) s += src[i + fsx * (j + fsy * k)];
    (a == 0 ? C.bx : (a == 1 ? C.by : C.bz))[f] = s;
  }
}

__global__ void __launch_bounds__(kProjThreads) k_mg_diag(MgLevel L) {
  const unsigned n = (unsigned)L.nx * L.ny * L.nz;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    unsigned i, j, k;
    level_ijk(L, c, i, j, k);
    const float diag = level_diag(L, c, i, j, k);
    L.invd[c] = diag > 0.f ? 1.f / diag : 0.f;
  }
}

// Pair p of cells along x on a level: cells i0 = 2 p and i0 + 1 of row (j, k),
// one red ((i + j + k) even) and one black.
struct MgPair {
  unsigned j, k, ir, ib;   // x of the red and of the black cell
  unsigned row;            // index of cell (0, j, k)
  bool red, black;         // the cell exists (the last pair of an odd row has one)
};
__device__ __forceinline__ MgPair mg_pair(const MgLevel& L, unsigned p, unsigned j, unsigned k) {
  MgPair q;
  const unsigned odd = (j + k) & 1u;
  q.j = j;
  q.k = k;
  q.ir = 2 * p + odd;
  q.ib = 2 * p + 1 - odd;
  q.row = (unsigned)L.nx * (j + (unsigned)L.ny * k);
  q.red = q.ir < (unsigned)L.nx;
  q.black = q.ib < (unsigned)L.nx;
  return q;
}

// The six face weights of cell (i, j, k): low and high x, y, z.  kAp (level 0):
// from alpha_f' of the cell and its neighbours, the values k_mg_faces0 stores:
// 8 MB at 128^3 instead of 25, so that a CG iteration's arrays (67 MB) fit L2.
// Outside the grid the cell itself stands in (its index q), so that no load
// waits on a branch.
struct MgFaces {
  float w[6];
};
struct MgNear {
  unsigned q[6];  // indices of the six neighbours, the cell's own beyond a side
  bool in[6];
};
__device__ __forceinline__ MgNear mg_near(const MgLevel& L, unsigned c, unsigned i, unsigned j, unsigned k) {
  const unsigned nx = (unsigned)L.nx, nxy = nx * (unsigned)L.ny;
  MgNear m;
  m.in[0] = i > 0, m.in[1] = i + 1 < nx, m.in[2] = j > 0, m.in[3] = j + 1 < (unsigned)L.ny, m.in[4] = k > 0,
  m.in[5] = k + 1 < (unsigned)L.nz;
  m.q[0] = m.in[0] ? c - 1 : c, m.q[1] = m.in[1] ? c + 1 : c;
  m.q[2] = m.in[2] ? c - nx : c, m.q[3] = m.in[3] ? c + nx : c;
  m.q[4] = m.in[4] ? c - nxy : c, m.q[5] = m.in[5] ? c + nxy : c;
  return m;
}
template <bool kAp>
__device__ __forceinline__ MgFaces mg_faces(const MgLevel& L, const MgNear& m, unsigned c, unsigned i, unsigned j,
                                            unsigned k) {
  MgFaces F;
  if constexpr (kAp) {
    const float own = L.ap[c];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      const float w = 0.5f * (a & 1 ? L.ap[m.q[a]] + own : own + L.ap[m.q[a]]);  // high side + low side
      F.w[a] = m.in[a] ? w : ((L.open >> a) & 1u ? own : 0.f);
    }
  } else {
    const unsigned nx = (unsigned)L.nx, ny = (unsigned)L.ny, nxy = nx * ny;
    const unsigned fx = i + (nx + 1) * (j + ny * k);
    const unsigned fy = i + nx * (j + (ny + 1) * k);
    F.w[0] = L.bx[fx], F.w[1] = L.bx[fx + 1], F.w[2] = L.by[fy], F.w[3] = L.by[fy + nx], F.w[4] = L.bz[c],
    F.w[5] = L.bz[c + nxy];
  }
  return F;
}

// sum over the interior faces of cell (i, j, k) of beta_f f(neighbour), f given
// the neighbour's index and coordinates.  All loads are in flight together
// (behind tests of the sides they took 27 cycles per instruction).
template <bool kAp, typename F>
__device__ __forceinline__ float mg_gather(const MgLevel& L, unsigned c, unsigned i, unsigned j, unsigned k, F&& f) {
  const MgNear m = mg_near(L, c, i, j, k);
  const MgFaces w = mg_faces<kAp>(L, m, c, i, j, k);
  float v[6];
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    const unsigned d = m.in[a];
    v[a] = f(m.q[a], a == 0 ? i - d : (a == 1 ? i + d : i), a == 2 ? j - d : (a == 3 ? j + d : j),
             a == 4 ? k - d : (a == 5 ? k + d : k));
  }
  float t = 0.f;
#pragma unroll
  for (int a = 0; a < 6; ++a) t = fmaf(m.in[a] ? w.w[a] : 0.f, v[a], t);
  return t;
}

// Down: x of both colours from x = 0 (red invd b, black with those).
template <bool kAp>
__device__ __forceinline__ void mg_down(const MgLevel& L, const MgPair& q) {
  if (q.red) L.x[q.row + q.ir] = L.invd[q.row + q.ir] * L.b[q.row + q.ir];
  if (!q.black) return;
  const unsigned c = q.row + q.ib;
  const float s = mg_gather<kAp>(L, c, q.ib, q.j, q.k,
                            [&](unsigned d, unsigned, unsigned, unsigned) { return L.invd[d] * L.b[d]; });
  L.x[c] = L.invd[c] * (L.b[c] + s);
}

// Residual b - A x of the red child in pair (I, j, k) of level F after mg_down:
// its own row was solved in the red half sweep (with the black cells 0), so
// what is left is the black neighbours' part.  (The black cells' residuals
// vanish after theirs.)
template <bool kAp>
__device__ __forceinline__ float mg_residual(const MgLevel& F, unsigned I, unsigned j, unsigned k) {
  if (j >= (unsigned)F.ny || k >= (unsigned)F.nz) return 0.f;
  const MgPair q = mg_pair(F, I, j, k);
  if (!q.red) return 0.f;
  return mg_gather<kAp>(F, q.row + q.ir, q.ir, j, k, [&](unsigned d, unsigned, unsigned, unsigned) { return F.x[d]; });
}

// Coarse right-hand side of cell (I, J, K), the sum of its children's residuals:
// four lanes per cell, lane m (of the aligned four) the child row 2 J + (m & 1)
// of layer 2 K + (m >> 1).
template <bool kAp>
__device__ __forceinline__ void mg_restrict(const MgLevel& F, const MgLevel& C, unsigned I, unsigned m, unsigned J,
                                            unsigned K) {
  float r = mg_residual<kAp>(F, I, 2 * J + (m & 1u), 2 * K + (m >> 1));
  const unsigned quad = 0xfu << (lane_id() & 28);
  r += __shfl_xor_sync(quad, r, 1);
  r += __shfl_xor_sync(quad, r, 2);
  if (m == 0) C.b[I + (unsigned)C.nx * (J + (unsigned)C.ny * K)] = r;
}

// Up, black cells: x_c = invd (b + sum beta_f (x_nb + omega x_coarse(nb's parent))).
template <bool kAp>
__device__ __forceinline__ void mg_up_black(const MgLevel& L, const MgLevel& C, const MgPair& q) {
  if (!q.black) return;
  const unsigned c = q.row + q.ib;
  const float s = mg_gather<kAp>(L, c, q.ib, q.j, q.k, [&](unsigned d, unsigned i, unsigned j, unsigned k) {
    return fmaf(kMgOmega, C.x[(i >> 1) + (unsigned)C.nx * ((j >> 1) + (unsigned)C.ny * (k >> 1))], L.x[d]);
  });
  L.x[c] = L.invd[c] * (L.b[c] + s);
}

// One colour's half sweep at cell (i, j, k).
template <bool kAp>
__device__ __forceinline__ float mg_sweep(const MgLevel& L, unsigned c, unsigned i, unsigned j, unsigned k) {
  const float s = mg_gather<kAp>(L, c, i, j, k, [&](unsigned d, unsigned, unsigned, unsigned) { return L.x[d]; });
  const float x = L.invd[c] * (L.b[c] + s);
  L.x[c] = x;
  return x;
}

// The passes grid-wide: a CTA takes tiles of 2^lx pairs x 2^ly rows x 2^lz runs of kc
// layers (lx + ly + lz = 8: a thread per run), tile blockIdx.x, + gridDim.x, ... (two
// divisions per tile, none per cell).  f(p, j, k) for every pair (or coarse cell) p < np.
// kDeep: lz > 0.  A kernel of its own, because the split in three cost the other grids
// 0.9% of a call at 128^3 (another schedule of the same loop).
struct MgTiles {
  unsigned np, ny, nz;       // extent
  unsigned lx, ly, lz, kc;   // tile shape
  unsigned tx, ty, tiles;    // tiles along x, y; in all
};
static_assert(kProjThreads == 256, "mg_tiles splits 8 bits");
template <bool kDeep, typename F>
__device__ __forceinline__ void mg_tiles(const MgTiles& T, F&& f) {
  const unsigned px = threadIdx.x & ((1u << T.lx) - 1u);
  if constexpr (!kDeep) {
    const unsigned py = threadIdx.x >> T.lx;
    for (unsigned t = blockIdx.x; t < T.tiles; t += gridDim.x) {
      const unsigned txy = T.tx * T.ty, tz = t / txy, r = t - tz * txy, y = r / T.tx, x = r - y * T.tx;
      const unsigned p = (x << T.lx) + px, j = y * ((unsigned)kProjThreads >> T.lx) + py;
      if (p >= T.np || j >= T.ny) continue;
      const unsigned k1 = min((tz + 1) * T.kc, T.nz);
#pragma unroll 2
      for (unsigned k = tz * T.kc; k < k1; ++k) f(p, j, k);
    }
    return;
  }
  const unsigned py = (threadIdx.x >> T.lx) & ((1u << T.ly) - 1u), pz = threadIdx.x >> (T.lx + T.ly);
  for (unsigned t = blockIdx.x; t < T.tiles; t += gridDim.x) {
    const unsigned txy = T.tx * T.ty, tz = t / txy, r = t - tz * txy, y = r / T.tx, x = r - y * T.tx;
    const unsigned p = (x << T.lx) + px, j = (y << T.ly) + py;
    if (p >= T.np || j >= T.ny) continue;
    const unsigned k0 = ((tz << T.lz) + pz) * T.kc, k1 = min(k0 + T.kc, T.nz);
#pragma unroll 2
    for (unsigned k = k0; k < k1; ++k) f(p, j, k);
  }
}

template <bool kAp, bool kDeep>
__global__ void __launch_bounds__(kProjThreads, 4) k_mg_down(MgLevel L, MgTiles T, const ProjRed* red) {
  if (stopped(red)) return;
  mg_tiles<kDeep>(T, [&](unsigned p, unsigned j, unsigned k) { mg_down<kAp>(L, mg_pair(L, p, j, k)); });
}

template <bool kAp, bool kDeep>
__global__ void __launch_bounds__(kProjThreads, 4) k_mg_restrict(MgLevel F, MgLevel C, MgTiles T, const ProjRed* red) {
  if (stopped(red)) return;
  mg_tiles<kDeep>(T, [&](unsigned p, unsigned J, unsigned K) { mg_restrict<kAp>(F, C, p >> 2, p & 3u, J, K); });
}

template <bool kAp, bool kDeep>
__global__ void __launch_bounds__(kProjThreads, 4) k_mg_up_black(MgLevel L, MgLevel C, MgTiles T, const ProjRed* red) {
  if (stopped(red)) return;
  mg_tiles<kDeep>(T, [&](unsigned p, unsigned j, unsigned k) { mg_up_black<kAp>(L, C, mg_pair(L, p, j, k)); });
}

template <bool kDeep>
__global__ void __launch_bounds__(kProjThreads, 4) k_mg_up_red(MgLevel L, MgTiles T, const ProjRed* red) {
  if (stopped(red)) return;
  mg_tiles<kDeep>(T, [&](unsigned p, unsigned j, unsigned k) {
    const MgPair q = mg_pair(L, p, j, k);
    if (q.red) mg_sweep<false>(L, q.row + q.ir, q.ir, j, k);
  });
}

// The same on level 0, where x = z = M^-1 r is complete after it, with rho =
// r . z into red->rz[cur] (b is r): a thread has both cells of its pair at hand.
template <bool kDeep>
__global__ void __launch_bounds__(kProjThreads, 4) k_mg_up_red_dot(MgLevel L, MgTiles T, int cur,
                                                                   double* __restrict__ P, ProjRed* red) {
  __shared__ double smem[32];
  if (stopped(red)) return;
  KahanF sum;
  mg_tiles<kDeep>(T, [&](unsigned p, unsigned j, unsigned k) {
    const MgPair q = mg_pair(L, p, j, k);
    if (q.red) sum.add(L.b[q.row + q.ir] * mg_sweep<true>(L, q.row + q.ir, q.ir, j, k));
    if (q.black) sum.add(L.b[q.row + q.ib] * L.x[q.row + q.ib]);
  });
  const double rz = block_sum(sum, smem);
  const double vals[1] = {rz};
  double* const outs[1] = {&red->rz[cur]};
  reduce_last<1>(vals, P, red, outs);
}

// The levels from `first` (at most kMgTailCells cells) down to the coarsest
// in one CTA: their weights, invd and the right-hand side of `first` are copied
// to shared memory (all copies in flight together), and every pass runs there with a barrier after it (16^3
// and below: 16 us; with the levels in global memory, a barrier and an L2 round
// trip per pass, 29 us).  Up to 8192 cells, as many as fit: a level of 4500 to 7600
// cells costs less here than in four launches (call on 24 x 44 x 34: 4290 -> 3770 us,
// on 35 x 65 x 24: 5240 -> 4960).  On the coarsest level (every axis <= 4 cells, so
// at most 32 pairs: one warp) red from x = 0, then kMgCoarsePairs (black, red)
// sweep pairs.  Same-colour cells do not touch, so a half sweep reads only
// values no thread of the pass writes.
constexpr int kMgTailThreads = 1024;
constexpr int kMgTailCells = 8192;
constexpr size_t kMgTailSmem = 224 * 1024;
struct MgLevels {
  MgLevel l[kMgMaxLevels];
};
// Floats of one level in the tail's shared memory; its arrays start at multiples
// of four floats.
__host__ __device__ inline unsigned mg_pad(unsigned n) { return (n + 3u) & ~3u; }
__host__ __device__ inline unsigned mg_level_floats(unsigned nx, unsigned ny, unsigned nz) {
  return mg_pad((nx + 1) * ny * nz) + mg_pad(nx * (ny + 1) * nz) + mg_pad(nx * ny * (nz + 1)) + 3 * mg_pad(nx * ny * nz);
}

extern __shared__ __align__(16) float g_mg_smem[];

// Level L's arrays at `base` floats in shared memory.
__device__ __forceinline__ MgLevel mg_shared(const MgLevel& L, unsigned base) {
  const unsigned nx = L.nx, ny = L.ny, nz = L.nz, n = mg_pad(nx * ny * nz);
  MgLevel S = L;
  float* q = g_mg_smem + base;
  S.bx = q;
  q += mg_pad((nx + 1) * ny * nz);
  S.by = q;
  q += mg_pad(nx * (ny + 1) * nz);
  S.bz = q;
  q += mg_pad(nx * ny * (nz + 1));
  S.invd = q;
  S.x = q + n;
  S.b = q + 2 * n;
  return S;
}

// n floats to shared memory, not waited for (both sides 16-byte aligned).
__device__ __forceinline__ void mg_copy(float* dst, const float* src, unsigned n) {
  const unsigned to = (unsigned)__cvta_generic_to_shared(dst);
  for (unsigned q = threadIdx.x; q < n / 4; q += kMgTailThreads)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 16 * q), "l"(src + 4 * q) : "memory");
  const unsigned q = (n & ~3u) + threadIdx.x;
  if (q < n) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + 4 * q), "l"(src + q) : "memory");
}

// f(p, j, k) for the np x ny x nz pairs (or cells) by the whole CTA
template <typename F>
__device__ __forceinline__ void mg_cta(unsigned np, unsigned ny, unsigned nz, F&& f) {
  for (unsigned t = threadIdx.x; t < np * ny * nz; t += kMgTailThreads) {
    const unsigned k = t / (np * ny), r = t - k * np * ny, j = r / np;
    f(r - j * np, j, k);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kMgTailThreads) k_mg_tail(MgLevels Ls, int first, int top, const ProjRed* red) {
  if (stopped(red)) return;
  unsigned base = 0;
  for (int l = first; l <= top; ++l) {
    const MgLevel G = Ls.l[l], S = mg_shared(G, base);
    const unsigned nx = G.nx, ny = G.ny, nz = G.nz, n = nx * ny * nz;
    mg_copy(S.bx, G.bx, (nx + 1) * ny * nz);
    mg_copy(S.by, G.by, nx * (ny + 1) * nz);
    mg_copy(S.bz, G.bz, nx * ny * (nz + 1));
    mg_copy(S.invd, G.invd, n);
    if (l == first) mg_copy(S.b, G.b, n);
    base += mg_level_floats(G.nx, G.ny, G.nz);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  base = 0;
  for (int l = first; l < top; ++l) {
    const MgLevel S = mg_shared(Ls.l[l], base);
    base += mg_level_floats(S.nx, S.ny, S.nz);
    const MgLevel C = mg_shared(Ls.l[l + 1], base);
    mg_cta((S.nx + 1) / 2, S.ny, S.nz, [&](unsigned p, unsigned j, unsigned k) { mg_down<false>(S, mg_pair(S, p, j, k)); });
    mg_cta(4 * C.nx, C.ny, C.nz, [&](unsigned p, unsigned J, unsigned K) { mg_restrict<false>(S, C, p >> 2, p & 3u, J, K); });
  }
  {
    const MgLevel S = mg_shared(Ls.l[top], base);
    const unsigned np = (S.nx + 1) / 2, t = threadIdx.x;
    if (t < 32) {
      const bool any = t < np * S.ny * S.nz;
      const unsigned k = t / (np * S.ny), r = t - k * np * S.ny, j = r / np;
      const MgPair q = mg_pair(S, r - j * np, j, k);
      if (any) mg_down<false>(S, q);  // red from x = 0, then black
      __syncwarp();
      if (any && q.red) mg_sweep<false>(S, q.row + q.ir, q.ir, j, k);
      __syncwarp();
      for (int m = 1; m < kMgCoarsePairs; ++m) {
        if (any && q.black) mg_sweep<false>(S, q.row + q.ib, q.ib, j, k);
        __syncwarp();
        if (any && q.red) mg_sweep<false>(S, q.row + q.ir, q.ir, j, k);
        __syncwarp();
      }
    }
    __syncthreads();
  }
  for (int l = top - 1; l >= first; --l) {
    const MgLevel C = mg_shared(Ls.l[l + 1], base);
    base -= mg_level_floats(Ls.l[l].nx, Ls.l[l].ny, Ls.l[l].nz);
    const MgLevel S = mg_shared(Ls.l[l], base);
    const unsigned np = (S.nx + 1) / 2;
    mg_cta(np, S.ny, S.nz, [&](unsigned p, unsigned j, unsigned k) { mg_up_black<false>(S, C, mg_pair(S, p, j, k)); });
    mg_cta(np, S.ny, S.nz, [&](unsigned p, unsigned j, unsigned k) {
      const MgPair q = mg_pair(S, p, j, k);
      if (q.red) mg_sweep<false>(S, q.row + q.ir, q.ir, j, k);
    });
  }
  const MgLevel S = mg_shared(Ls.l[first], 0);
  float* x = Ls.l[first].x;
  for (unsigned c = threadIdx.x; c < (unsigned)(S.nx * S.ny * S.nz); c += kMgTailThreads) x[c] = S.x[c];
}

// ---- conjugate gradients on A e = r with the multigrid preconditioner ----

// rho = r . z (z = M^-1 r from the V-cycle) into red->rz[cur].
__global__ void __launch_bounds__(kProjThreads) k_cg_dot(int64_t n64, int cur, const float* __restrict__ r,
                                                         const float* __restrict__ z, double* __restrict__ P,
                                                         ProjRed* red) {
  __shared__ double smem[32];
  if (stopped(red)) return;
  const unsigned n = (unsigned)n64;
  KahanF k;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) k.add(r[c] * z[c]);
  const double rz = block_sum(k, smem);
  const double vals[1] = {rz};
  double* const outs[1] = {&red->rz[cur]};
  reduce_last<1>(vals, P, red, outs);
}

// d_new = z + beta d_old (beta = rho / rho_prev; 0 on a run's first
// iteration), y = A d_new and d_new . y into red->dy.  d_old and d_new are
// different buffers: neighbours' d_new is formed from their z and d_old.
// The face weights are formed again from alpha_f' (mg_faces).
template <bool kDeep>
__global__ void __launch_bounds__(kProjThreads, 4) k_cg_dir_apply(MgLevel L, MgTiles T, int cur,
                                                                  const float* __restrict__ z,
                                                                  const float* __restrict__ d_old,
                                                                  float* __restrict__ d_new, float* __restrict__ y,
                                                                  double* __restrict__ P, ProjRed* red) {
  __shared__ double smem[32];
  if (stopped(red)) return;
  // beta in FP32 (a double divide per thread would occupy GB300's slow FP64 pipe)
  const float be = red->iters == 0 ? 0.f : (float)red->rz[cur] / (float)red->rz[cur ^ 1];
  KahanF dyk;
  // beta = 0 takes z alone (the old direction is not read into the sum)
  auto dn = [&](unsigned q) { return be != 0.f ? fmaf(be, d_old[q], z[q]) : z[q]; };
  mg_tiles<kDeep>(T, [&](unsigned i, unsigned j, unsigned k) {
    const unsigned c = i + (unsigned)L.nx * (j + (unsigned)L.ny * k);
    const MgNear m = mg_near(L, c, i, j, k);
    const MgFaces w = mg_faces<true>(L, m, c, i, j, k);
    float v[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) v[a] = dn(m.q[a]);
    const float dc = dn(c);
    float acc = (((w.w[0] + w.w[1]) + (w.w[2] + w.w[3])) + (w.w[4] + w.w[5])) * dc;
#pragma unroll
    for (int a = 0; a < 6; ++a) acc = fmaf(m.in[a] ? -w.w[a] : 0.f, v[a], acc);
    d_new[c] = dc;
    y[c] = acc;
    dyk.add(dc * acc);
  });
  const double dy = block_sum(dyk, smem);
  const double vals[1] = {dy};
  double* const outs[1] = {&red->dy};
  reduce_last<1>(vals, P, red, outs);
}

// alpha = rho / (d . y); e += alpha d; r -= alpha y (float4); r . r into
// red->rr.  The last block counts the iteration and sets the stop flag when
// r . r <= rr_stop (or on a breakdown).
__global__ void __launch_bounds__(kProjThreads) k_cg_update(int64_t n64, int cur, const float* __restrict__ d,
                                                            const float* __restrict__ y, float* __restrict__ e,
                                                            float* __restrict__ r, double* __restrict__ P,
                                                            ProjRed* red) {
  __shared__ double smem[32];
  if (stopped(red)) return;
  const double dy = red->dy, rz = red->rz[cur];  // the same values in every block
  if (!(dy > 0.0) || !isfinite(rz)) {  // d = 0 (r = 0: converged) or breakdown: stop this run
    if (blockIdx.x == 0 && threadIdx.x == 0) red->done = 1;
    return;
  }
  const float al = (float)rz / (float)dy;  // FP32, as beta
  KahanF rrk;
  const unsigned n = (unsigned)n64, n4 = n / 4u;
  const unsigned t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (unsigned q = t0; q < n4; q += stride) {  // arrays are 256-byte aligned
    const float4 dq = reinterpret_cast<const float4*>(d)[q];
    const float4 yq = reinterpret_cast<const float4*>(y)[q];
    float4 eq = reinterpret_cast<const float4*>(e)[q];
    float4 rq = reinterpret_cast<const float4*>(r)[q];
    eq.x = fmaf(al, dq.x, eq.x);
    eq.y = fmaf(al, dq.y, eq.y);
    eq.z = fmaf(al, dq.z, eq.z);
    eq.w = fmaf(al, dq.w, eq.w);
    rq.x = fmaf(-al, yq.x, rq.x);
    rq.y = fmaf(-al, yq.y, rq.y);
    rq.z = fmaf(-al, yq.z, rq.z);
    rq.w = fmaf(-al, yq.w, rq.w);
    reinterpret_cast<float4*>(e)[q] = eq;
    reinterpret_cast<float4*>(r)[q] = rq;
    rrk.add(rq.x * rq.x + rq.y * rq.y + rq.z * rq.z + rq.w * rq.w);
  }
  for (unsigned c = 4u * n4 + t0; c < n; c += stride) {
    e[c] = fmaf(al, d[c], e[c]);
    const float rc = fmaf(-al, y[c], r[c]);
    r[c] = rc;
    rrk.add(rc * rc);
  }
  const double rr = block_sum(rrk, smem);
  const double vals[1] = {rr};
  double* const outs[1] = {&red->rr};
  if (reduce_last<1>(vals, P, red, outs) && threadIdx.x == 0) {
    red->iters += 1;
    if (!(red->rr > red->rr_stop)) red->done = 1;  // also stops on NaN
  }
}

// p += e (the FP32 correction into the FP64 solution).
__global__ void __launch_bounds__(kProjThreads) k_proj_add(int64_t n, double* __restrict__ p,
                                                           const float* __restrict__ e) {
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x)
    p[c] += (double)e[c];
}

// Face outputs: v' = v* - (dt/rho) grad p1 and dx = clamp(-(dt^2/rho) grad p2, -h, h);
// zero on solid sides' faces.  Faces of the three grids in one index range.
__global__ void __launch_bounds__(kProjThreads) k_proj_faces(
    PGrid g, double h, double dt_rho, double dt2_rho, const double* __restrict__ p1, const double* __restrict__ p2,
    const float* __restrict__ u, const float* __restrict__ v, const float* __restrict__ w, float* __restrict__ uo,
    float* __restrict__ vo, float* __restrict__ wo, float* __restrict__ dxu, float* __restrict__ dxv,
    float* __restrict__ dxw) {
  const int64_t nu = (int64_t)(g.nx + 1) * g.ny * g.nz, nv = (int64_t)g.nx * (g.ny + 1) * g.nz,
                nw = (int64_t)g.nx * g.ny * (g.nz + 1);
  const double inv_h = 1.0 / h;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nu + nv + nw;
       q += (int64_t)gridDim.x * blockDim.x) {
    int a;
    int64_t f;
    if (q < nu) {
      a = 0;
      f = q;
    } else if (q < nu + nv) {
      a = 1;
      f = q - nu;
    } else {
      a = 2;
      f = q - nu - nv;
    }
    // face (i, j, k) on grid a: x fastest with n_a + 1 samples along a
    int ns[3] = {g.nx, g.ny, g.nz};
    ns[a] += 1;
    const int64_t sxy = (int64_t)ns[0] * ns[1];
    const int k = (int)(f / sxy);
    const int64_t rem = f - (int64_t)k * sxy;
    const int j = (int)(rem / ns[0]);
    const int i = (int)(rem - (int64_t)j * ns[0]);
    const int idx[3] = {i, j, k};
    const int m = a == 0 ? g.nx : (a == 1 ? g.ny : g.nz);
    const int64_t stride = a == 0 ? 1 : (a == 1 ? g.nx : g.nxy);
    // the cell on the high side has index idx (if idx[a] < m), the low side idx - e_a (if idx[a] > 0)
    const int64_t cR = i + (int64_t)g.nx * (j + (int64_t)g.ny * k);  // valid when idx[a] < m
    const bool lo_in = idx[a] > 0, hi_in = idx[a] < m;
    const bool solid = (!lo_in && !g.open[2 * a]) || (!hi_in && !g.open[2 * a + 1]);
    float vo_ = 0.f, dx_ = 0.f;
    if (!solid) {
      const int64_t cL = cR - stride;
      const double pR1 = hi_in ? p1[cR] : 0.0, pL1 = lo_in ? p1[cL] : 0.0;
      const double pR2 = hi_in ? p2[cR] : 0.0, pL2 = lo_in ? p2[cL] : 0.0;
      const float* vin = a == 0 ? u : (a == 1 ? v : w);
      vo_ = (float)((double)vin[f] - dt_rho * (pR1 - pL1) * inv_h);
      const double dxf = -dt2_rho * (pR2 - pL2) * inv_h;
      dx_ = (float)(dxf < -h ? -h : (dxf > h ? h : dxf));
    }
    if (uo) (a == 0 ? uo : (a == 1 ? vo : wo))[f] = vo_;
    if (dxu) (a == 0 ? dxu : (a == 1 ? dxv : dxw))[f] = dx_;
  }
}

// ---- host side ----

struct ProjWs {
  double *fx, *fy, *fz;                // FP64 face weights (the residual's operator)
  double* b64;                         // right-hand side of the solve
  float *ap32, *r, *z, *d[2], *y, *e;  // d: the CG direction, double-buffered
  double* P;                           // 2 * nblk partial sums
  ProjRed* red;
  MgLevel lev[kMgMaxLevels];
  int levels;
};

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

static int proj_blocks(int64_t n) {
  const int64_t want = (n + kProjThreads - 1) / kProjThreads;
  const int64_t cap = 8 * (int64_t)sm_count();
  return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// Workspace of the call (laid out by the same walk that measures it): the
// FP32 CG vectors, the partial sums, the scalars and the multigrid levels
// (halving each axis until every axis has at most 4 cells).
static size_t proj_layout(const PGrid& g, int nblk, char* base, ProjWs* W) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + off : nullptr;
    off += align256(bytes);
    return p;
  };
  const size_t n = (size_t)g.n;
  ProjWs w;
  w.fx = (double*)take(8 * (size_t)(g.nx + 1) * g.ny * g.nz);
  w.fy = (double*)take(8 * (size_t)g.nx * (g.ny + 1) * g.nz);
  w.fz = (double*)take(8 * (size_t)g.nx * g.ny * (g.nz + 1));
  w.b64 = (double*)take(8 * n);
  w.ap32 = (float*)take(4 * n);
  w.r = (float*)take(4 * n);
  w.z = (float*)take(4 * n);
  w.d[0] = (float*)take(4 * n);
  w.d[1] = (float*)take(4 * n);
  w.y = (float*)take(4 * n);
  w.e = (float*)take(4 * n);
  w.P = (double*)take(2 * 8 * (size_t)nblk);
  w.red = (ProjRed*)take(sizeof(ProjRed));
  int nx = g.nx, ny = g.ny, nz = g.nz;
  w.levels = 0;
  for (;;) {
    MgLevel& L = w.lev[w.levels];
    L.nx = nx, L.ny = ny, L.nz = nz;
    const size_t nl = (size_t)nx * ny * nz;
    L.bx = (float*)take(4 * (size_t)(nx + 1) * ny * nz);
    L.by = (float*)take(4 * (size_t)nx * (ny + 1) * nz);
    L.bz = (float*)take(4 * (size_t)nx * ny * (nz + 1));
    L.invd = (float*)take(4 * nl);
    if (w.levels == 0) {
      L.x = w.z;
      L.b = w.r;
    } else {
      L.x = (float*)take(4 * nl);
      L.b = (float*)take(4 * nl);
    }
    ++w.levels;
    if ((nx <= 4 && ny <= 4 && nz <= 4) || w.levels == kMgMaxLevels) break;
    nx = (nx + 1) / 2, ny = (ny + 1) / 2, nz = (nz + 1) / 2;
  }
  if (W) *W = w;
  return off;
}

static int proj_grid(const GicGrid* grid, PGrid* g) {
  if (!grid) return set_error(GIC_ERR_INVALID, "gic_project: grid is NULL");
  if (grid->nx < 1 || grid->ny < 1 || grid->nz < 1) return set_error(GIC_ERR_INVALID, "gic_project: empty grid");
  if (!(grid->dx > 0.0) || !isfinite(grid->dx)) return set_error(GIC_ERR_INVALID, "gic_project: dx must be positive");
  g->nx = grid->nx;
  g->ny = grid->ny;
  g->nz = grid->nz;
  g->nxy = (int64_t)grid->nx * grid->ny;
  g->n = g->nxy * grid->nz;
  if (g->n >= ((int64_t)1 << 30)) return set_error(GIC_ERR_INVALID, "gic_project: 2^30 cells or more");
  return GIC_OK;
}

// The solver's scalars, read to the host.
static int read_red(const ProjRed* dev, ProjRed* host, cudaStream_t st) {
  if (cudaMemcpyAsync(host, dev, sizeof(ProjRed), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return set_error(GIC_ERR_CUDA, "gic_project: reading the solver's scalars failed");
  return wait_stream(st, 60000, "gic_project", 20);
}

}  // namespace gic

using namespace gic;

extern "C" int gic_project_workspace_size(const GicGrid* grid, size_t* bytes) {
  GIC_RANGE("gic_project_workspace_size");
  PGrid g;
  int rc = proj_grid(grid, &g);
  if (rc) return rc;
  if (!bytes) return set_error(GIC_ERR_INVALID, "gic_project_workspace_size: bytes is NULL");
  *bytes = proj_layout(g, proj_blocks(g.n), nullptr, nullptr);
  return GIC_OK;
}

extern "C" int gic_project(const GicGrid* grid, const GicProjParams* P, const double* alpha_s, const float* alpha_star,
                           const float* u, const float* v, const float* w, double* p1, double* p2, float* u_out,
                           float* v_out, float* w_out, float* dx_u, float* dx_v, float* dx_w, void* ws,
                           size_t ws_bytes, GicProjInfo* info, gic_stream_t stream_) {
  GIC_RANGE("gic_project");
  PGrid g;
  int rc = proj_grid(grid, &g);
  if (rc) return rc;
  if (!P) return set_error(GIC_ERR_INVALID, "gic_project: params is NULL");
  if (!(P->dt > 0.0) || !(P->rho_f > 0.0)) return set_error(GIC_ERR_INVALID, "gic_project: dt and rho_f must be positive");
  if (!(P->alpha_s_max > 0.0 && P->alpha_s_max < 1.0))
    return set_error(GIC_ERR_INVALID, "gic_project: alpha_s_max must lie in (0, 1)");
  if (!(P->ratio_min > 0.0 && P->ratio_min <= 1.0 && P->ratio_max >= 1.0 && isfinite(P->ratio_max)))
    return set_error(GIC_ERR_INVALID, "gic_project: need 0 < ratio_min <= 1 <= ratio_max");
  if (!(P->tol > 0.0) || !(P->inner_tol > 0.0 && P->inner_tol < 1.0))
    return set_error(GIC_ERR_INVALID, "gic_project: tol must be positive and inner_tol in (0, 1)");
  if (P->max_outer < 1 || P->max_inner < 1)
    return set_error(GIC_ERR_INVALID, "gic_project: max_outer and max_inner must be >= 1");
  bool any_open = false;
  for (int s = 0; s < 6; ++s) {
    if (P->open[s] != 0 && P->open[s] != 1) return set_error(GIC_ERR_INVALID, "gic_project: open[%d] must be 0 or 1", s);
    any_open |= P->open[s] == 1;
  }
  if (!any_open) return set_error(GIC_ERR_INVALID, "gic_project: at least one side must be open (p = 0 beyond it)");
  if (!alpha_s || !alpha_star || !u || !v || !w || !p1 || !p2)
    return set_error(GIC_ERR_INVALID, "gic_project: null input or pressure array");
  const bool vel_out = u_out || v_out || w_out, disp_out = dx_u || dx_v || dx_w;
  if (vel_out && !(u_out && v_out && w_out))
    return set_error(GIC_ERR_INVALID, "gic_project: give all three projected velocity arrays or none");
  if (disp_out && !(dx_u && dx_v && dx_w))
    return set_error(GIC_ERR_INVALID, "gic_project: give all three displacement arrays or none");
  unsigned open_bits = 0u;
  for (int s = 0; s < 6; ++s) {
    g.open[s] = P->open[s];
    if (P->open[s]) open_bits |= 1u << s;
  }
  const int nblk = proj_blocks(g.n);
  const size_t need = proj_layout(g, nblk, nullptr, nullptr);
  if (!ws || ws_bytes < need)
    return set_error(GIC_ERR_WORKSPACE, "gic_project: workspace of %zu bytes needed, %zu given", need, ws_bytes);
  if ((uintptr_t)ws % 256) return set_error(GIC_ERR_ALIGN, "gic_project: workspace must be 256-byte aligned");
  cudaStream_t st = (cudaStream_t)stream_;
  ProjWs W;
  proj_layout(g, nblk, (char*)ws, &W);
  for (int l = 0; l < W.levels; ++l) W.lev[l].ap = nullptr, W.lev[l].open = 0u;
  W.lev[0].ap = W.ap32;
  W.lev[0].open = open_bits;
  if (W.levels == kMgMaxLevels && !(W.lev[kMgMaxLevels - 1].nx <= 4 && W.lev[kMgMaxLevels - 1].ny <= 4 &&
                                    W.lev[kMgMaxLevels - 1].nz <= 4))
    return set_error(GIC_ERR_INVALID, "gic_project: grid too large for the multigrid hierarchy");
  uint32_t* status = status_word();
  const double h = grid->dx;
  ProjScales S;
  S.vel = P->rho_f * h / P->dt;
  S.den = -P->rho_f * h * h / (P->dt * P->dt);
  S.rmin = P->ratio_min;
  S.rmax = P->ratio_max;
  S.amax = P->alpha_s_max;
  GicProjInfo inf;
  memset(&inf, 0, sizeof(inf));
  ProjRed hr;
  int64_t launches = 0;
  int rc2 = GIC_OK;
  auto lblocks = [&](const MgLevel& L) { return proj_blocks((int64_t)L.nx * L.ny * L.nz); };
  auto fblocks = [&](const MgLevel& L) {
    return proj_blocks((int64_t)(L.nx + 1) * L.ny * L.nz + (int64_t)L.nx * (L.ny + 1) * L.nz +
                       (int64_t)L.nx * L.ny * (L.nz + 1));
  };

  if (cudaMemsetAsync(W.red, 0, sizeof(ProjRed), st) != cudaSuccess ||
      cudaMemsetAsync(W.d[0], 0, sizeof(float) * g.n, st) != cudaSuccess ||
      cudaMemsetAsync(W.d[1], 0, sizeof(float) * g.n, st) != cudaSuccess)
    return set_error(GIC_ERR_CUDA, "gic_project: clearing the workspace failed");
  // the operator's face weights on every level
  k_proj_faces64<<<fblocks(W.lev[0]), kProjThreads, 0, st>>>(g, open_bits, alpha_s, P->alpha_s_max, W.fx, W.fy, W.fz);
  k_proj_prep<<<nblk, kProjThreads, 0, st>>>(g, alpha_s, P->alpha_s_max, W.ap32);
  k_mg_faces0<<<fblocks(W.lev[0]), kProjThreads, 0, st>>>(W.lev[0], open_bits, W.ap32);
  k_mg_diag<<<lblocks(W.lev[0]), kProjThreads, 0, st>>>(W.lev[0]);
  launches += 4;
  for (int l = 1; l < W.levels; ++l) {
    k_mg_coarsen<<<fblocks(W.lev[l]), kProjThreads, 0, st>>>(W.lev[l - 1], W.lev[l]);
    k_mg_diag<<<lblocks(W.lev[l]), kProjThreads, 0, st>>>(W.lev[l]);
    launches += 2;
  }
  // the levels from `first` on run in one CTA (k_mg_tail): the largest that has
  // few cells and fits its shared memory with those below it
  MgLevels levels;
  for (int l = 0; l < W.levels; ++l) levels.l[l] = W.lev[l];
  const int top = W.levels - 1;
  int first = top;
  size_t tail_bytes = 4 * (size_t)mg_level_floats(W.lev[top].nx, W.lev[top].ny, W.lev[top].nz);
  while (first > 0) {
    const MgLevel& L = W.lev[first - 1];
    if ((int64_t)L.nx * L.ny * L.nz > kMgTailCells) break;
    const size_t more = 4 * (size_t)mg_level_floats(L.nx, L.ny, L.nz);
    if (tail_bytes + more > kMgTailSmem) break;
    tail_bytes += more;
    --first;
  }
  if (tail_bytes > 48 * 1024 &&
      cudaFuncSetAttribute(k_mg_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMgTailSmem) != cudaSuccess)
    return set_error(GIC_ERR_CUDA, "gic_project: shared memory of the coarse levels refused");
  // tiles of a pass over np x ny x nz pairs (or cells): wide enough for the rows (up to
  // a warp), the other lanes over rows and layers so that the fewest fall outside the
  // grid.  (All of them on rows, a column of 1 x 1 x 20000 cells had one lane of 256 at
  // work: 10.5 ms a call, now 2.5; 2 x 2 x 65536 13.0 -> 4.5, 4 x 4 x 4096 15.6 -> 10.9,
  // 300 x 1 x 300 6.9 -> 5.7; 128^3 keeps its 32 x 8 lanes, 10.6.)  And up to four
  // layers per thread where that still leaves a tile for every CTA that is resident at
  // once (four per SM)
  const uint64_t resident = 4 * (uint64_t)sm_count();
  auto tiles = [&](unsigned np, unsigned ny, unsigned nz) {
    MgTiles T;
    T.np = np, T.ny = ny, T.nz = nz;
    T.lx = 0;
    while (T.lx < 5 && (1u << T.lx) < np) ++T.lx;
    auto over = [](unsigned n, unsigned l) { return ((uint64_t)n + (1u << l) - 1) >> l; };  // ceil(n / 2^l)
    uint64_t fewest = UINT64_MAX;
    for (int ly = 8 - (int)T.lx; ly >= 0; --ly) {
      const unsigned lz = 8 - T.lx - ly;
      const uint64_t lanes = over(ny, ly) * over(nz, lz);
      if (lanes < fewest) fewest = lanes, T.ly = ly, T.lz = lz;
    }
    T.tx = (unsigned)over(np, T.lx);
    T.ty = (unsigned)over(ny, T.ly);
    T.kc = 1;
    unsigned lk = 0;  // log2 kc
    while (lk < 2 && (uint64_t)T.tx * T.ty * over(nz, T.lz + lk + 1) >= resident) ++lk;
    T.kc = 1u << lk;
    T.tiles = T.tx * T.ty * (unsigned)over(nz, T.lz + lk);
    return T;
  };
  auto deep = [](const MgTiles& T, auto* flat, auto* layered) { return T.lz ? layered : flat; };
  auto pairs = [&](const MgLevel& L) { return tiles((unsigned)(L.nx + 1) / 2, L.ny, L.nz); };
  auto quads = [&](const MgLevel& L) { return tiles(4 * (unsigned)L.nx, L.ny, L.nz); };  // four lanes per cell
  auto ctas = [&](const MgTiles& T) { return (int)(T.tiles < (unsigned)nblk ? T.tiles : (unsigned)nblk); };
  // one preconditioned CG iteration: z = V-cycle(r), rho = r . z, the new
  // direction with y = A d, the updates; all arguments but the parity are
  // fixed for the call
  auto cg_iteration = [&](int cur) {
    for (int l = 0; l < first; ++l) {
      const MgLevel &L = W.lev[l], &C = W.lev[l + 1];
      const MgTiles T = pairs(L), Q = quads(C);
      (l == 0 ? deep(T, k_mg_down<true, false>, k_mg_down<true, true>)
              : deep(T, k_mg_down<false, false>, k_mg_down<false, true>))<<<ctas(T), kProjThreads, 0, st>>>(L, T, W.red);
      (l == 0 ? deep(Q, k_mg_restrict<true, false>, k_mg_restrict<true, true>)
              : deep(Q, k_mg_restrict<false, false>, k_mg_restrict<false, true>))<<<ctas(Q), kProjThreads, 0, st>>>(
          L, C, Q, W.red);
    }
    k_mg_tail<<<1, kMgTailThreads, tail_bytes, st>>>(levels, first, top, W.red);
    for (int l = first - 1; l >= 0; --l) {
      const MgLevel &L = W.lev[l], &C = W.lev[l + 1];
      const MgTiles T = pairs(L);
      (l == 0 ? deep(T, k_mg_up_black<true, false>, k_mg_up_black<true, true>)
              : deep(T, k_mg_up_black<false, false>, k_mg_up_black<false, true>))<<<ctas(T), kProjThreads, 0, st>>>(
          L, C, T, W.red);
      if (l > 0)
        deep(T, k_mg_up_red<false>, k_mg_up_red<true>)<<<ctas(T), kProjThreads, 0, st>>>(L, T, W.red);
      else
        deep(T, k_mg_up_red_dot<false>, k_mg_up_red_dot<true>)<<<ctas(T), kProjThreads, 0, st>>>(L, T, cur, W.P,
                                                                                                 W.red);
    }
    if (first == 0) k_cg_dot<<<nblk, kProjThreads, 0, st>>>(g.n, cur, W.r, W.z, W.P, W.red);
    const MgTiles T = tiles(g.nx, g.ny, g.nz);
    deep(T, k_cg_dir_apply<false>, k_cg_dir_apply<true>)<<<ctas(T), kProjThreads, 0, st>>>(
        W.lev[0], T, cur, W.z, W.d[cur ^ 1], W.d[cur], W.y, W.P, W.red);
    k_cg_update<<<nblk, kProjThreads, 0, st>>>(g.n, cur, W.d[cur], W.y, W.e, W.r, W.P, W.red);
    launches += 4 * first + (first == 0 ? 4 : 3);
  };

  for (int which = 1; which <= 2 && rc2 == GIC_OK; ++which) {
    double* p = which == 1 ? p1 : p2;
    const int sys = which - 1;
    if (cudaMemsetAsync(p, 0, sizeof(double) * g.n, st) != cudaSuccess) {
      rc2 = set_error(GIC_ERR_CUDA, "gic_project: clearing p failed");
      break;
    }
    int last_iters = 0;  // of the previous CG run
    for (int outer = 0;; ++outer) {
      const double tol2 = P->inner_tol * P->inner_tol;
      if (outer == 0)  // p = 0
        k_proj_rhs<<<nblk, kProjThreads, 0, st>>>(g, which, S, alpha_s, alpha_star, u, v, w, W.fx, W.fy, W.fz, W.b64,
                                                  W.r, W.e, tol2, W.P, W.red, status);
      else
        k_proj_residual<<<nblk, kProjThreads, 0, st>>>(g, W.b64, W.fx, W.fy, W.fz, p, W.r, W.e, tol2, W.P, W.red,
                                                       status);
      ++launches;
      if ((rc2 = read_red(W.red, &hr, st))) break;
      if (!isfinite(hr.rr64) || !isfinite(hr.bb)) {
        rc2 = set_error(GIC_ERR_INVALID, "gic_project: non-finite residual (check alpha_s, alpha_star and v*)");
        break;
      }
      inf.outer[sys] = outer;
      inf.rel_residual[sys] = hr.bb > 0.0 ? sqrt(hr.rr64 / hr.bb) : 0.0;
      if (hr.bb == 0.0 || hr.rr64 <= P->tol * P->tol * hr.bb) {
        inf.converged[sys] = 1;
        break;
      }
      if (outer >= P->max_outer) break;
      // the FP32 preconditioned CG on A e = r to a reduction of inner_tol (of
      // the FP32 copy's r . r): as many iterations as the previous run took,
      // less one in runs of more than four (a read costs about as much as an
      // iteration queued past the stop, whose kernels return at once), three in the
      // first run, are queued before the stop flag is read, then two at a time
      int it = 0, want = last_iters == 0 ? 3 : last_iters > 4 ? last_iters - 1 : last_iters > 2 ? last_iters : 2;
      for (;;) {
        for (int q = 0; q < want && it < P->max_inner; ++q, ++it) cg_iteration(it & 1);
        cudaError_t le = cudaGetLastError();
        if (le != cudaSuccess) {
          rc2 = set_error(GIC_ERR_CUDA, "gic_project: %s", cudaGetErrorString(le));
          break;
        }
        if ((rc2 = read_red(W.red, &hr, st))) break;
        if (hr.done || it >= P->max_inner) break;
        want = 2;
      }
      last_iters = hr.iters;
      if (rc2) break;
      inf.inner[sys] += hr.iters;
      k_proj_add<<<nblk, kProjThreads, 0, st>>>(g.n, p, W.e);
      ++launches;
    }
  }
  if (rc2 == GIC_OK && (vel_out || disp_out)) {
    const int64_t nf = (int64_t)(g.nx + 1) * g.ny * g.nz + (int64_t)g.nx * (g.ny + 1) * g.nz +
                       (int64_t)g.nx * g.ny * (g.nz + 1);
    const int fb = (int)((nf + kProjThreads - 1) / kProjThreads < 4096 ? (nf + kProjThreads - 1) / kProjThreads : 4096);
    k_proj_faces<<<fb, kProjThreads, 0, st>>>(g, h, P->dt / P->rho_f, P->dt * P->dt / P->rho_f, p1, p2, u, v, w,
                                              u_out, v_out, w_out, dx_u, dx_v, dx_w);
    ++launches;
  }
  count_launches(launches);
  if (rc2) return rc2;
  GIC_CHECK_LAUNCH("gic_project");
  if (info) *info = inf;
  return GIC_OK;
}
