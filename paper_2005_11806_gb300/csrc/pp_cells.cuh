// Per-cell bodies of the stencil kernels, shared by the single-grid kernels
// (pp_kernels_stencil.cu) and the grouped multi-grid kernels (pp_batch.cu).
#pragma once
#include "pp_fft.cuh"

namespace pp {

struct CellIdx {
  int i, j, k;
  unsigned cim, cip, cjm, cjp;  // grids keep nx ny (nz + 1) below 2^31
};

// 32-bit divisions: three 64-bit ones cost more than the FP64 work of some of
// the bodies below.
__device__ __forceinline__ CellIdx cell_index(const Geo& g, size_t c64) {
  const unsigned nx = (unsigned)g.nx, ny = (unsigned)g.ny, c = (unsigned)c64;
  CellIdx x;
  const unsigned row = c / nx, i = c - row * nx, k = row / ny, j = row - k * ny;
  x.i = (int)i;
  x.j = (int)j;
  x.k = (int)k;
  x.cim = i == 0 ? c + nx - 1 : c - 1;
  x.cip = i + 1 == nx ? c + 1 - nx : c + 1;
  x.cjm = j == 0 ? c + (ny - 1) * nx : c - nx;
  x.cjp = j + 1 == ny ? c - (ny - 1) * nx : c + nx;
  return x;
}

// Face coefficients of cell c (beta = 2/(rho_a + rho_b) on its x-, y- and
// z-face "below", x/y coefficients scaled by the layer width dzf_k).  Wall
// faces get 0: the z walls, and with walls in y the y-face below row 0,
// which the periodic indexing also reaches as the face above row ny - 1.
// FP64-pipe bound: five operations a face (512^3: prep_faces and prep_diag
// together 9.4 -> 5.2 ms, most of it the IEEE divisions and 64-bit index divisions).
__device__ __forceinline__ void cell_prep_faces(const Geo& g, const double* __restrict__ rho,
                                                const Faces& fc, size_t c) {
  const CellIdx x = cell_index(g, c);
  const size_t plane = (size_t)g.nx * g.ny;
  const double r = rho[c];
  // layer factors 2 dzf / dx^2, 2 dzf / dy^2, 2 / dzc (0 on the walls); a product
  // of uniform factors costs as much of the FP64 pipe as one of the cell's own
  double fx = g.cw_d[x.k], fy = g.cw_d[g.nz + 1 + x.k], fz = g.cw_d[2 * (g.nz + 1) + x.k];
  if (g.ym) {  // stretched y: the row of cell j is scaled by dzf_k s_j; the y face below it carries t_j = dy / dyc_j
    fx *= g.ym[x.j];
    fy *= g.ym[g.ny + x.j];
    fz *= g.ym[x.j];
  }
  fc.cx[c] = fx * rcp_f64(r + rho[x.cim]);
  fc.cy[c] = (g.ywall && x.j == 0) ? 0.0 : fy * rcp_f64(r + rho[x.cjm]);
  fc.cz[c] = (x.k == 0) ? 0.0 : fz * rcp_f64(r + rho[c - plane]);
  if (x.k == g.nz - 1) fc.cz[c + plane] = 0.0;
  if (fc.rhof != nullptr) fc.rhof[c] = (float)r;
}

// diag = sum of the six (row-scaled) coefficients of cell c.
__device__ __forceinline__ void cell_prep_diag(const Geo& g, const Faces& fc, size_t c) {
  const CellIdx x = cell_index(g, c);
  const size_t plane = (size_t)g.nx * g.ny;
  fc.diag[c] = ((fc.cx[c] + fc.cx[x.cip]) + (fc.cy[c] + fc.cy[x.cjp])) + (fc.cz[c] + fc.cz[c + plane]);
  if (fc.diagf != nullptr) fc.diagf[c] = (float)fc.diag[c];
}

// d = D u* - (S - meanS) at cell c (wall values of w*, and of v* with walls
// in y, taken as zero); stores the row-scaled b_s = dzf_k d / dt (dzf_k s_j
// d / dt on a stretched y, where the row width is dyf_j = s_j dy) and
// returns d.
__device__ __forceinline__ double cell_rhs_b(const Geo& g, const double* __restrict__ us,
                                             const double* __restrict__ vs,
                                             const double* __restrict__ ws,
                                             const double* __restrict__ S, double meanS,
                                             double* __restrict__ b, double inv_dt, size_t c) {
  const CellIdx x = cell_index(g, c);
  const size_t plane = (size_t)g.nx * g.ny;
  const double wlo = (x.k == 0) ? 0.0 : ws[c];
  const double whi = (x.k == g.nz - 1) ? 0.0 : ws[c + plane];
  const double vlo = (g.ywall && x.j == 0) ? 0.0 : vs[c];
  const double vhi = (g.ywall && x.j == g.ny - 1) ? 0.0 : vs[x.cjp];
  double dv = vhi - vlo, wd = g.dzf[x.k] * inv_dt;
  if (g.ym) {
    dv *= g.ym[2 * g.ny + x.j];
    wd *= g.ym[x.j];
  }
  double d = fma(us[x.cip] - us[c], g.inv_dx, fma(dv, g.inv_dy, (whi - wlo) * g.inv_dzf[x.k]));
  if (S != nullptr) d -= (S[c] - meanS);
  b[c] = d * wd;
  return d;
}

// 2 div(k grad T) at cell c: D(k_f G T) with k_f the arithmetic mean of the
// two cells of a face, no flux through the z walls, nor through the y walls
// when y is bounded (Eqs. 30 and 34).
__device__ __forceinline__ double cell_conduction2(const Geo& g, const double* __restrict__ kc,
                                                   const double* __restrict__ T, size_t c) {
  const CellIdx x = cell_index(g, c);
  const size_t plane = (size_t)g.nx * g.ny;
  const double k0 = kc[c], t0 = T[c];
  const double sx = fma(k0 + kc[x.cip], T[x.cip] - t0, (k0 + kc[x.cim]) * (T[x.cim] - t0));
  // with walls in y no heat crosses the faces below row 0 and above row ny - 1
  const bool yhi = !(g.ywall && x.j + 1 == g.ny), ylo = !(g.ywall && x.j == 0);
  // stretched y: the face below row j is dyc_j = dy / t_j from the centre
  // below, and the row is dyf_j = s_j dy wide
  double fhi = yhi ? T[x.cjp] - t0 : 0.0, flo = ylo ? T[x.cjm] - t0 : 0.0;
  if (g.ym) {
    const double isj = g.ym[2 * g.ny + x.j];
    fhi *= yhi ? g.ym[g.ny + x.j + 1] * isj : 0.0;
    flo *= g.ym[g.ny + x.j] * isj;
  }
  const double sy = fma(k0 + kc[x.cjp], fhi, (k0 + kc[x.cjm]) * flo);
  double sz = 0.0;
  if (x.k + 1 < g.nz) sz = (k0 + kc[c + plane]) * ((T[c + plane] - t0) * g.inv_dzc[x.k + 1]);
  if (x.k > 0) sz = fma(k0 + kc[c - plane], (T[c - plane] - t0) * g.inv_dzc[x.k], sz);
  return fma(sx, g.inv_dx2, fma(sy, g.inv_dy2, sz * g.inv_dzf[x.k]));
}

// u = u* - dt beta G p at the faces of cell c (Eq. corr); w walls = 0, and
// with walls in y the wall row 0 of v = 0.
__device__ __forceinline__ void cell_correct(const Geo& g, const Faces& fc,
                                             const double* __restrict__ us,
                                             const double* __restrict__ vs,
                                             const double* __restrict__ ws,
                                             const double* __restrict__ p, double dt,
                                             double* __restrict__ u, double* __restrict__ v,
                                             double* __restrict__ w, size_t c) {
  const CellIdx x = cell_index(g, c);
  const size_t plane = (size_t)g.nx * g.ny;
  const double pc = p[c];
  // dt beta_x / dx = dt dx cx / dzf_k (cx carries dzf_k); on a stretched y
  // cx and cz also carry s_j, and dt beta_y / dyc_j = dt dy cy / dzf_k
  // (cy carries dzf_k t_j = dzf_k dy / dyc_j)
  double dz = dt;
  double ax = (dt * g.dx) * g.inv_dzf[x.k];
  const double ay = (dt * g.dy) * g.inv_dzf[x.k];
  if (g.ym) {
    const double is = g.ym[2 * g.ny + x.j];
    ax *= is;
    dz *= is;
  }
  u[c] = fma(-ax, fc.cx[c] * (pc - p[x.cim]), us[c]);
  v[c] = (g.ywall && x.j == 0) ? 0.0 : fma(-ay, fc.cy[c] * (pc - p[x.cjm]), vs[c]);
  w[c] = (x.k == 0) ? 0.0 : fma(-dz, fc.cz[c] * (pc - p[c - plane]), ws[c]);
  if (x.k == g.nz - 1) w[c + plane] = 0.0;
}

// Loop control of Algorithm 1 for one grid, run by thread 0 with the
// reduced residual sums s2 (sum e^2) and s1 (sum |e|).  kexact: recompute
// the residual exactly every kexact passes (<= 1: every pass); convergence
// is only accepted on an exact residual.
__device__ __forceinline__ void status_update(DevStatus* st, double s2, double s1, double rtol,
                                              int maxit, int kexact) {
  st->e2 = s2;
  st->e1 = s1;
  const double e20 = st->e2_0;
  const double rel = (e20 > 0.0) ? sqrt(s2 / e20) : 0.0;
  st->rel = rel;
  const int exact = st->need_exact;
  st->last_exact = exact;
  if (!isfinite(s2) || !isfinite(e20)) { st->done = 1; st->code = PP_ERR_NUMERIC; }
  else if (e20 == 0.0 || (rel <= rtol && exact)) { st->done = 1; st->code = PP_OK; }
  else if (st->iters >= maxit) { st->done = 1; st->code = PP_ERR_NOT_CONVERGED; }
  else {
    st->iters += 1;
    if (kexact <= 1) {
      st->need_exact = 1;
    } else if (exact) {
      st->need_exact = 0;
      st->since_exact = 1;
    } else {
      st->since_exact += 1;
      // an updated residual below the tolerance is confirmed by an exact one
      st->need_exact = (rel <= rtol || st->since_exact >= kexact) ? 1 : 0;
    }
  }
}

__device__ __forceinline__ void status_init(DevStatus* st) {
  st->e2 = 0; st->e1 = 0; st->e2_0 = 0; st->rel = 0; st->mean_S = 0; st->pmean = 0;
  st->iters = 0; st->done = 0; st->code = PP_OK; st->pad = 0;
  st->need_exact = 1; st->since_exact = 0; st->last_exact = 1;
}

}  // namespace pp
