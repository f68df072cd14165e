// Stencil, reduction and set-up kernels of the projection: mixture density
// (Eq. 22), face coefficients, the loop-invariant right-hand side of
// Algorithm 1, its loop control, the correction step (Eq. corr), the gauge
// removal, the adjoint stencils and the Thomas pivots of the z solve.
#include "pp_cells.cuh"

namespace pp {

namespace {
// Partial sums written by the reduction kernels: six blocks for each of the 152
// SMs (1024 blocks left 40 of them a seventh one; a third of it is two each).
constexpr int kRedBlocks = 912;
constexpr int kThreads = 256;

inline int grid_for(size_t n) {
  size_t b = (n + kThreads - 1) / kThreads;
  if (b > (size_t)152 * 64) b = (size_t)152 * 64;
  return (int)(b == 0 ? 1 : b);
}
}  // namespace

int reduce_blocks() { return kRedBlocks; }

__global__ void k_mixture(const double* __restrict__ phi, double rho_g, double rho_l,
                          double* __restrict__ rho, size_t n) {
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const double f = phi[c];
    rho[c] = rho_g * f + rho_l * (1.0 - f);
  }
}

// beta on every face: arithmetic face density, beta = 2 / (rho_a + rho_b);
// x/y coefficients carry the width dzf_k of their layer (row scaling).
__global__ void k_prep_faces(Geo g, const double* __restrict__ rho, Faces fc) {
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
    cell_prep_faces(g, rho, fc, c);
}

// diag = sum of the six (row-scaled) coefficients of each cell.
__global__ void k_prep_diag(Geo g, Faces fc) {
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
    cell_prep_diag(g, fc, c);
}

// Fixed-order partial sums of dzf_k * f (dzf_k s_j * f on a stretched y:
// the cell volume over dx dy) (grid of kRedBlocks blocks).
__global__ void k_weighted_partial(Geo g, const double* __restrict__ f, double* __restrict__ red) {
  __shared__ double sh[32];
  const unsigned nx = (unsigned)g.nx, ny = (unsigned)g.ny, n = nx * ny * (unsigned)g.nz;
  double s = 0.0;
  for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
    const unsigned row = c / nx, k = row / ny;
    const double w = g.ym ? g.dzf[k] * g.ym[row - k * ny] : g.dzf[k];
    s = fma(w, f[c], s);
  }
  s = block_sum<double>(s, sh);
  if (threadIdx.x == 0) red[blockIdx.x] = s;
}

// out = scale * sum_b red[b * stride + off]
__global__ void k_finalize(const double* __restrict__ red, int nblk, int stride, int off, double scale,
                           double* __restrict__ out) {
  __shared__ double sh[32];
  double s = 0.0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += red[(size_t)b * stride + off];
  s = block_sum<double>(s, sh);
  if (threadIdx.x == 0) *out = scale * s;
}

// b_s = dzf_k (D u* - (S - <S>_V)) / dt (row-scaled); wall values of w* are
// taken as zero; block partial sums of (D u* - S_c)^2.
__global__ void k_rhs_b(Geo g, const double* __restrict__ us, const double* __restrict__ vs,
                        const double* __restrict__ ws, const double* __restrict__ S,
                        const DevStatus* __restrict__ st, double* __restrict__ b,
                        double* __restrict__ red, double inv_dt) {
  __shared__ double sh[32];
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  const double meanS = st->mean_S;
  double s2 = 0.0;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const double d = cell_rhs_b(g, us, vs, ws, S, meanS, b, inv_dt, c);
    s2 += d * d;
  }
  s2 = block_sum<double>(s2, sh);
  if (threadIdx.x == 0) red[blockIdx.x] = s2;
}

__global__ void k_init_status(DevStatus* st) { status_init(st); }

// u = u* - dt beta G p  (Eq. corr); w wall planes are written as zero.
__global__ void k_correct(Geo g, Faces fc, const double* __restrict__ us, const double* __restrict__ vs,
                          const double* __restrict__ ws, const double* __restrict__ p, double dt,
                          double* __restrict__ u, double* __restrict__ v, double* __restrict__ w) {
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
    cell_correct(g, fc, us, vs, ws, p, dt, u, v, w, c);
}

__global__ void k_sub_mean(double* __restrict__ p, size_t n, const DevStatus* __restrict__ st) {
  const double m = st->pmean;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
    p[c] -= m;
}

// Inverse Thomas pivots of (L_z + lambda_x(kx) + lambda_y(ky)) per column.
__global__ void k_setup_pivots(Geo g, const double* __restrict__ lamx, const double* __restrict__ lamy,
                               double* __restrict__ invd, double* __restrict__ mtab) {
  const size_t ncol = (size_t)g.ny * g.nxh;
  const size_t col = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= ncol) return;
  const int j = (int)(col / g.nxh), kx = (int)(col % g.nxh);
  const double lam = lamx[kx] + lamy[j];
  double d = -(g.za[0] + g.zc[0]) + lam;
  if (mtab != nullptr) mtab[col] = 0.0;
  if (col == 0 && g.nz == 1) { invd[0] = 0.0; return; }
  invd[col] = 1.0 / d;
  for (int k = 1; k < g.nz; ++k) {
    const double dinv_prev = invd[(size_t)(k - 1) * ncol + col];
    if (mtab != nullptr) mtab[(size_t)k * ncol + col] = g.za[k] * dinv_prev;
    d = (-(g.za[k] + g.zc[k]) + lam) - g.za[k] * g.zc[k - 1] / d;
    const bool pin = (col == 0 && k == g.nz - 1);  // singular (0, 0) column: pin the last unknown
    invd[(size_t)k * ncol + col] = pin ? 0.0 : 1.0 / d;
  }
}

// Tables of the FP64-recurrence z solve (TriZ), one thread per table column
// tc = ky' nxh + kx with lambda = lambda_x(kx) + lambda_y(ky'): the same
// pivot recurrence as k_setup_pivots, stored as m_k = a_k / d_{k-1},
// e_k = c_k / d_k (FP64) and 1 / d_k (the spectrum's precision).  Column 0 is
// the singular (0, 0) system: its last inverse pivot is 0.
template <typename T>
__global__ void k_setup_z(Geo g, const double* __restrict__ lamx, const double* __restrict__ lamy, int nyt,
                            double* __restrict__ m, double* __restrict__ e, T* __restrict__ dinv) {
  const size_t ntc = (size_t)nyt * g.nxh;
  const size_t tc = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tc >= ntc) return;
  const int j = (int)(tc / g.nxh), kx = (int)(tc % g.nxh);
  const double lam = lamx[kx] + lamy[j];
  double d = -(g.za[0] + g.zc[0]) + lam;
  double inv_prev = 0.0;
  for (int k = 0; k < g.nz; ++k) {
    if (k > 0) d = (-(g.za[k] + g.zc[k]) + lam) - g.za[k] * g.zc[k - 1] / d;
    const bool pin = (tc == 0 && k == g.nz - 1);  // singular (0, 0) column: pin the last unknown
    const double inv = pin ? 0.0 : 1.0 / d;
    const size_t o = (size_t)k * ntc + tc;
    m[o] = (k == 0) ? 0.0 : g.za[k] * inv_prev;
    e[o] = (k + 1 < g.nz) ? g.zc[k] * inv : 0.0;
    dinv[o] = (T)inv;
    inv_prev = inv;
  }
}

// ---- Methods I and II (Sec. 3.3.1) -------------------------------------------
constexpr int kExtBlocks = kRedBlocks / 2;  // (min, max) pairs fit the partial-sum buffer

// Block partial minimum and maximum of rho into red[2 b], red[2 b + 1].
__global__ void k_rho_extrema(size_t n, const double* __restrict__ rho, double* __restrict__ red) {
  __shared__ double smin[kThreads / 32], smax[kThreads / 32];
  double lo = INFINITY, hi = -INFINITY;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const double r = rho[c];
    lo = fmin(lo, r);
    hi = fmax(hi, r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { smin[wid] = lo; smax[wid] = hi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) { lo = fmin(lo, smin[k]); hi = fmax(hi, smax[k]); }
    red[2 * (size_t)blockIdx.x] = lo;
    red[2 * (size_t)blockIdx.x + 1] = hi;
  }
}

// rho0 = min rho (Method I, Eq. poisson_me1); the harmonic mean
// 2 rho_min rho_max / (rho_min + rho_max) of the two phase densities
// (Method II, Eq. poisson_laizet).  One thread.
__global__ void k_rho_tilde(const double* __restrict__ red, int nblk, int method, double* __restrict__ out) {
  double lo = INFINITY, hi = -INFINITY;
  for (int b = 0; b < nblk; ++b) {
    lo = fmin(lo, red[2 * (size_t)b]);
    hi = fmax(hi, red[2 * (size_t)b + 1]);
  }
  *out = (method == 1) ? lo : 2.0 * lo * hi / (lo + hi);
}

// Eq. poisson_me2 with p^q = p - delta:
//   u = u* - dt beta G p + dt (beta - 1/rho0) G delta  on every face.
// beta is recovered from the row-scaled coefficients: cx = dzf_k beta / dx^2,
// cy = dzf_k beta / dy^2, cz = beta / dzc.
template <typename T>
__global__ void k_correct_method1(Geo g, Faces fc, const double* __restrict__ us,
                                  const double* __restrict__ vs, const double* __restrict__ ws,
                                  const double* __restrict__ p, const T* __restrict__ delta, double dt,
                                  double* __restrict__ u, double* __restrict__ v, double* __restrict__ w) {
  const size_t plane = (size_t)g.nx * g.ny, n = plane * g.nz;
  const double ir0 = 1.0 / *fc.rho_tilde;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    cell_correct(g, fc, us, vs, ws, p, dt, u, v, w, c);
    const CellIdx x = cell_index(g, c);
    const double idzf = g.inv_dzf[x.k];
    const double dc = (double)delta[c];
    // stretched y: cx, cz carry s_j and cy carries t_j = dy / dyc_j (t_0 = 0
    // on the walls, where v is not corrected)
    const double is = g.ym ? g.ym[2 * g.ny + x.j] : 1.0;
    const double tj = g.ym ? g.ym[g.ny + x.j] : 1.0;
    const double bx = fc.cx[c] * idzf * is / g.inv_dx2;
    u[c] += dt * (bx - ir0) * (dc - (double)delta[x.cim]) / g.dx;
    if (!(g.ywall && x.j == 0)) {
      const double by = fc.cy[c] * idzf / (g.inv_dy2 * tj);
      v[c] += dt * (by - ir0) * (dc - (double)delta[x.cjm]) * tj / g.dy;
    }
    if (x.k > 0) w[c] += dt * (fc.cz[c] * is - ir0 * g.inv_dzc[x.k]) * (dc - (double)delta[c - plane]);
  }
}

// ---- divergence source from the thermodynamics (Eqs. 30, 34, v_gas) ----------

// Block partial sums of Phi div(k grad T) dV, Phi div(u) dV and Phi dV into
// red[3 b + {0, 1, 2}] (wall values of w taken as zero).
__global__ void k_thermo_partial(Geo g, const double* __restrict__ phi, const double* __restrict__ kc,
                                 const double* __restrict__ T, const double* __restrict__ u,
                                 const double* __restrict__ v, const double* __restrict__ w,
                                 double* __restrict__ red) {
  __shared__ double sh[32];
  const size_t plane = (size_t)g.nx * g.ny, n = plane * g.nz;
  const double dxdy = g.dx * g.dy;
  double a = 0.0, b = 0.0, vg = 0.0;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const CellIdx x = cell_index(g, c);
    const double f = phi[c];
    const double fdv = f * (g.ym ? g.dzf[x.k] * g.ym[x.j] : g.dzf[x.k]);  // over dx dy
    const double wlo = (x.k == 0) ? 0.0 : w[c];
    const double whi = (x.k == g.nz - 1) ? 0.0 : w[c + plane];
    // the wall row of v (walls in y) carries no flux, like the wall planes of w
    const double vlo = (g.ywall && x.j == 0) ? 0.0 : v[c];
    const double vhi = (g.ywall && x.j == g.ny - 1) ? 0.0 : v[x.cjp];
    double dvy = vhi - vlo;
    if (g.ym) dvy *= g.ym[2 * g.ny + x.j];  // stretched y: dyf_j = s_j dy
    const double div = fma(u[x.cip] - u[c], g.inv_dx, fma(dvy, g.inv_dy, (whi - wlo) * g.inv_dzf[x.k]));
    a = fma(fdv, cell_conduction2(g, kc, T, c), a);
    b = fma(fdv, div, b);
    vg += fdv;
  }
  a = block_sum<double>(a, sh);
  __syncthreads();
  b = block_sum<double>(b, sh);
  __syncthreads();
  vg = block_sum<double>(vg, sh);
  if (threadIdx.x == 0) {
    red[3 * (size_t)blockIdx.x] = 0.5 * dxdy * a;
    red[3 * (size_t)blockIdx.x + 1] = dxdy * b;
    red[3 * (size_t)blockIdx.x + 2] = dxdy * vg;
  }
}

// out = {sum a, sum b, V_g, RP} with RP of Eq. 30 (RP = NaN when V_g = 0).
__global__ void k_thermo_rate(const double* __restrict__ red, int nblk, double p0, double gamma,
                              double* __restrict__ out) {
  __shared__ double sh[32];
  double s[3];
  for (int q = 0; q < 3; ++q) {
    double t = 0.0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) t += red[3 * (size_t)b + q];
    s[q] = block_sum<double>(t, sh);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = s[0];
    out[1] = s[1];
    out[2] = s[2];
    out[3] = (s[2] > 0.0) ? gamma / s[2] * ((gamma - 1.0) / gamma * s[0] - p0 * s[1]) : NAN;
  }
}

// S = (1/p0) [ (gamma - 1)/gamma div(k grad T) - dp0dt / gamma ] Phi  (Eq. 34);
// a = (gamma - 1) / (2 gamma p0), b = dp0dt / (gamma p0) come from the host
// (three divisions a thread were a quarter of the kernel).  FP64-pipe bound:
// 256^3 1.14 -> 0.79 ms.
__global__ void k_divergence_source(Geo g, const double* __restrict__ phi, const double* __restrict__ kc,
                                    const double* __restrict__ T, double a, double b, double* __restrict__ S) {
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x)
    S[c] = fma(a, cell_conduction2(g, kc, T, c), -b) * phi[c];
}

// ---- momentum predictor (Eqs. 29, 32) ---------------------------------------
struct PredArgs {
  const double *u, *v, *w, *rho, *mu;
  const double *fx, *fy, *fz;  // body force, entries may be null
  const double *pu, *pv, *pw;  // RU of the step before, null: forward Euler
  double gx, gy, gz, dta, dtb;      // dt a, dt b
  double idx, idy, hdx, hdy, tdx, tdy; // 1 / h, 1 / (2 h), 8 / h: uniform products cost FP64 issue like any other
  double *us, *vs, *ws;
  double *ru, *rv, *rw;        // RU, entries may be null
};
constexpr int kPredLanes = 30;  // useful lanes of a warp; lanes 0 and 31 hold the x neighbours

// Predicted velocity at the three low faces of cell (i, j, k): the u-face
// i-1/2, the v-face j-1/2 and (k >= 1) the w-face k-1/2.  RU = -C(u) +
// (1/rho_f)[div tau + f] + g with C(u) = div(u u) - u div(u) (central
// divergence form: normal products at cell centres, cross products at edges,
// a velocity carried to an edge by the mean of its two values) and the
// Newton-Stokes stress (normal parts at cell centres with the cell's mu,
// shear parts at edges with the mean mu of the cells around the edge;
// no-slip z walls: wall velocity zero, half-cell distance to the wall).
// With walls in y the y walls are no-slip too: the wall row of v is zero
// (read as zero, written as zero), the edges on y = 0 and y = ly carry the
// wall shear of u and w over half a cell and no convective flux, and the
// edges where a y wall meets a z wall carry nothing.  u* = u + dt (a RU - b
// RU_prev).
//
// Bound by the FP64 pipe.  A cell's edge and centre terms are shared with its
// neighbours: a warp holds 30 consecutive cells of one row (and one neighbour
// on each side, exchanged by shuffles) and marches in z, so x and z
// neighbours' terms come from registers and only those of the rows j - 1 and
// j + 1 are formed twice; about 160 FP64 operations a cell against about 365
// with every term formed at both of its cells and three IEEE divisions.
// 256^3: 9.7 ms -> 6.2 ms (FP64 pipe 86 % busy; 12 % of the lanes are the tiles'
// neighbours at 256).
//
// WHOLE (nx <= 32): a warp holds 32 / nx whole rows, neighbours by shuffles
// around each row, so no lane is a tile's neighbour and a short row does not
// leave most of the warp idle (8 x 64 x 500: 0.371 -> 0.117 ms, 32 x 96 x 96
// 0.228 -> 0.117, both with chunks as before).
template <bool WHOLE>
__global__ void __launch_bounds__(128) k_predictor(Geo g, PredArgs A, int ntile, int ngroup, int nchunk, int chunk) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int lane = threadIdx.x & 31;
  const unsigned wid = blockIdx.x * 4 + (threadIdx.x >> 5);
  const unsigned rest = WHOLE ? wid : wid / (unsigned)ntile;
  const int ch = (int)(rest / (unsigned)ngroup);
  if (ch >= nchunk) return;
  int i, j = (int)(rest - (unsigned)ch * ngroup);
  bool emit_lane;
  int from_left = 0, from_right = 0;  // WHOLE: the lanes of i - 1 and i + 1
  if constexpr (WHOLE) {
    const int rows = 32 / nx, q = lane / nx;
    i = lane - q * nx;
    j = j * rows + q;
    emit_lane = q < rows && j < ny;
    if (j >= ny) j = ny - 1;  // lanes without a row of their own only read
    from_left = i == 0 ? lane + nx - 1 : lane - 1;
    from_right = i + 1 == nx ? lane + 1 - nx : lane + 1;
  } else {
    const int at = (int)(wid - rest * ntile) * kPredLanes + lane - 1;  // -1 .. ; wraps
    i = at < 0 ? at + nx : at;
    while (i >= nx) i -= nx;
    emit_lane = lane >= 1 && lane <= kPredLanes && at < nx;
  }
  const int k0 = ch * chunk, k1 = min(k0 + chunk, nz);
  const bool ywall = g.ywall != 0;
  const bool wlo = ywall && j == 0, whi = ywall && j + 1 == ny;  // the row's low / high y edges are walls
  const int jm = j == 0 ? ny - 1 : j - 1, jp = j + 1 == ny ? 0 : j + 1;
  const bool vz_m = ywall && jm == 0, vz_p = ywall && jp == 0;   // rows whose v reads as zero
  const size_t plane = (size_t)nx * ny;
  const size_t oc = (size_t)j * nx + i, om = (size_t)jm * nx + i, op = (size_t)jp * nx + i;
  const double idx = A.idx, idy = A.idy;
  constexpr unsigned full = 0xffffffffu;
  auto left = [&](double a) {  // value at i - 1
    return WHOLE ? __shfl_sync(full, a, from_left) : __shfl_up_sync(full, a, 1);
  };
  auto right = [&](double a) {  // value at i + 1
    return WHOLE ? __shfl_sync(full, a, from_right) : __shfl_down_sync(full, a, 1);
  };

  const int ks = k0 > 0 ? k0 - 1 : 0;  // the layer below the chunk only leaves its upper edges and centre
  size_t o = (size_t)ks * plane;
  // layer k of rows j, j - 1, j + 1
  double uc = A.u[o + oc], um = A.u[o + om], up = A.u[o + op];
  double vc = wlo ? 0.0 : A.v[o + oc], vm = vz_m ? 0.0 : A.v[o + om], vp = vz_p ? 0.0 : A.v[o + op];
  // half the viscosity: the sum over an edge's four cells is then twice their
  // mean, and every stress is formed doubled
  double mc = 0.5 * A.mu[o + oc], mm = 0.5 * A.mu[o + om], mp = 0.5 * A.mu[o + op];
  double wc = A.w[o + oc], wm = A.w[o + om], wp = A.w[o + op];  // face k
  // sums of mu over cell pairs: x pairs of the three rows, y pairs
  double sx = mc + left(mc), sy = mc + mm, syp = mc + mp;
  // lower edges: x-z, y-z below row j, y-z above row j (4 x the convective
  // product, 2 x the stress); the z wall of layer 0, else set by the layer below
  double Fxz = 0.0, Txz, Fyz = 0.0, Tyz, Fyp = 0.0, Typ = 0.0;
  {
    const double h = 2.0 * g.inv_dzf[0];  // sx: the mean of the two cells
    Txz = sx * uc * h;
    Tyz = wlo ? 0.0 : sy * vc * h;
    Txz *= 2.0;
    Tyz *= 2.0;
  }
  double Dk = 0.0, Czk = 0.0, Tzk = 0.0, rk = 0.0;  // layer k - 1: divergence, centre terms, density
  for (int k = ks; k < k1; ++k, o += plane) {
    const bool top = k + 1 == nz;
    const size_t ou = o + plane;
    // ---- layer k + 1
    const double wuc = A.w[ou + oc], wum = A.w[ou + om], wup = A.w[ou + op];  // face k + 1
    double uu = 0.0, uum = 0.0, uup = 0.0, vu = 0.0, vum = 0.0, vup = 0.0, mu_ = 0.0, mum = 0.0, mup = 0.0;
    if (!top) {
      uu = A.u[ou + oc]; uum = A.u[ou + om]; uup = A.u[ou + op];
      vu = wlo ? 0.0 : A.v[ou + oc]; vum = vz_m ? 0.0 : A.v[ou + om]; vup = vz_p ? 0.0 : A.v[ou + op];
      mu_ = 0.5 * A.mu[ou + oc]; mum = 0.5 * A.mu[ou + om]; mup = 0.5 * A.mu[ou + op];
    }
    const double rc = A.rho[o + oc], rm = A.rho[o + om];
    const double idzf = g.inv_dzf[k], idzc = g.inv_dzc[k + 1];
    // ---- centres of layer k
    const double ur = right(uc), urm = right(um), vl = left(vc), vlp = left(vp), wl = left(wuc);
    const double dux = ur - uc, dvy = vp - vc, dvm = vc - vm, dwz = wuc - wc;
    const double D = fma(dux, idx, fma(dvy, idy, dwz * idzf));
    const double Dm = fma(urm - um, idx, fma(dvm, idy, (wum - wm) * idzf));  // row j - 1
    // 2 tau = (mu / 2) (8 d - 8/3 D)
    const double t83 = (-8.0 / 3.0) * D, t83m = (-8.0 / 3.0) * Dm;
    const double Tx = mc * fma(dux, A.tdx, t83), Ty = mc * fma(dvy, A.tdy, t83);
    const double Tym = mm * fma(dvm, A.tdy, t83m), Tz = mc * fma(dwz, 8.0 * idzf, t83);
    const double ax = uc + ur, ay = vc + vp, aym = vm + vc, az = wc + wuc;
    const double Cx = ax * ax, Cy = ay * ay, Cym = aym * aym, Cz = az * az;  // 4 x the products
    // ---- x-y edges below and above row j (4 x the convective product)
    const double sxm = mm + left(mm), sxp = mp + left(mp);
    double Fxy = 0.0, Txy, Fxyp = 0.0, Txyp;
    if (wlo) Txy = sx * uc * (0.5 * A.tdy);  // 2 x 2 mu u / dy
    else {
      Fxy = (uc + um) * (vc + vl);
      Txy = (sx + sxm) * fma(uc - um, idy, (vc - vl) * idx);
    }
    if (whi) Txyp = -sx * uc * (0.5 * A.tdy);
    else {
      Fxyp = (up + uc) * (vp + vlp);
      Txyp = (sx + sxp) * fma(up - uc, idy, (vp - vlp) * idx);
    }
    // ---- edges on face k + 1
    const double sxu = mu_ + left(mu_), syu = mu_ + mum, sypu = mu_ + mup;
    double FxzU = 0.0, TxzU, FyzU = 0.0, TyzU, FypU = 0.0, TypU = 0.0;
    if (top) {
      const double h = -4.0 * idzf;  // 2 x (-2 / dzf) times the mean of two cells
      TxzU = sx * uc * h;
      TyzU = wlo ? 0.0 : sy * vc * h;
    } else {
      FxzU = (uc + uu) * (wuc + wl);
      TxzU = (sx + sxu) * fma(uu - uc, idzc, (wuc - wl) * idx);
      const double mz = mc + mu_;
      if (wlo) TyzU = mz * wuc * (0.5 * A.tdy);  // 2 x 2 mu w / dy
      else {
        FyzU = (vc + vu) * (wuc + wum);
        TyzU = (sy + syu) * fma(vu - vc, idzc, (wuc - wum) * idy);
      }
      if (whi) TypU = -mz * wuc * (0.5 * A.tdy);
      else {
        FypU = (vp + vup) * (wup + wuc);
        TypU = (syp + sypu) * fma(vup - vp, idzc, (wup - wuc) * idy);
      }
    }
    // the neighbours' terms (every lane takes part)
    const double Cxl = left(Cx), Txl = left(Tx), Dl = left(D), rl = left(rc);
    const double Fxyr = right(Fxy), Txyr = right(Txy), Fxzr = right(Fxz), Txzr = right(Txz);
    if (k >= k0 && emit_lane) {
      const size_t c = o + oc;
      const double qz = 0.5 * idzf;  // cv: 2 x the convection
      // ---- x momentum at the u-face (i-1/2, j, k)
      {
        double cv = fma(Cx - Cxl, A.hdx, fma(Fxyp - Fxy, A.hdy, (FxzU - Fxz) * qz));
        cv = fma(-uc, D + Dl, cv);
        double vs = fma(Tx - Txl, idx, fma(Txyp - Txy, idy, (TxzU - Txz) * idzf));
        if (A.fx != nullptr) vs = fma(2.0, A.fx[c], vs);
        const double r = fma(-0.5, cv, fma(vs, rcp_f64(rc + rl), A.gx));
        double q = fma(A.dta, r, uc);
        if (A.pu != nullptr) q = fma(-A.dtb, A.pu[c], q);
        A.us[c] = q;
        if (A.ru != nullptr) A.ru[c] = r;
      }
      // ---- y momentum at the v-face (i, j-1/2, k); the wall row stays zero
      if (wlo) {
        A.vs[c] = 0.0;
        if (A.rv != nullptr) A.rv[c] = 0.0;
      } else {
        double cv = fma(Fxyr - Fxy, A.hdx, fma(Cy - Cym, A.hdy, (FyzU - Fyz) * qz));
        cv = fma(-vc, D + Dm, cv);
        double vs = fma(Txyr - Txy, idx, fma(Ty - Tym, idy, (TyzU - Tyz) * idzf));
        if (A.fy != nullptr) vs = fma(2.0, A.fy[c], vs);
        const double r = fma(-0.5, cv, fma(vs, rcp_f64(rc + rm), A.gy));
        double q = fma(A.dta, r, vc);
        if (A.pv != nullptr) q = fma(-A.dtb, A.pv[c], q);
        A.vs[c] = q;
        if (A.rv != nullptr) A.rv[c] = r;
      }
      // ---- z momentum at the w-face (i, j, k-1/2), interior faces only
      if (k == 0) {
        A.ws[c] = 0.0;
        if (A.rw != nullptr) A.rw[c] = 0.0;
      } else {
        const double ic = g.inv_dzc[k];
        double cv = fma(Fxzr - Fxz, A.hdx, fma(Fyp - Fyz, A.hdy, (Cz - Czk) * (0.5 * ic)));
        cv = fma(-wc, D + Dk, cv);
        double vs = fma(Txzr - Txz, idx, fma(Typ - Tyz, idy, (Tz - Tzk) * ic));
        if (A.fz != nullptr) vs = fma(2.0, A.fz[c], vs);
        const double r = fma(-0.5, cv, fma(vs, rcp_f64(rc + rk), A.gz));
        double q = fma(A.dta, r, wc);
        if (A.pw != nullptr) q = fma(-A.dtb, A.pw[c], q);
        A.ws[c] = q;
        if (A.rw != nullptr) A.rw[c] = r;
      }
      if (top) {
        A.ws[c + plane] = 0.0;
        if (A.rw != nullptr) A.rw[c + plane] = 0.0;
      }
    }
    // ---- on to layer k + 1
    uc = uu; um = uum; up = uup;
    vc = vu; vm = vum; vp = vup;
    mc = mu_; mm = mum; mp = mup;
    wc = wuc; wm = wum; wp = wup;
    sx = sxu; sy = syu; syp = sypu;
    Fxz = FxzU; Txz = TxzU; Fyz = FyzU; Tyz = TyzU; Fyp = FypU; Typ = TypU;
    Dk = D; Czk = Cz; Tzk = Tz; rk = rc;
  }
}

// ---- adjoint ---------------------------------------------------------------
// y = -dt * beta * W_f^{-1} g  (W_f = dzf of the layer on x/y faces, dzc on
// interior z faces; wall z-faces zero).
__global__ void k_adj_rhs(Geo g, const double* __restrict__ rho, const double* __restrict__ gu,
                          const double* __restrict__ gv, const double* __restrict__ gw, double dt,
                          double* __restrict__ yu, double* __restrict__ yv, double* __restrict__ yw) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const size_t plane = (size_t)nx * ny, n = plane * nz;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(c % nx);
    const int j = (int)((c / nx) % ny);
    const int k = (int)(c / plane);
    const size_t cim = c - i + (i == 0 ? nx - 1 : i - 1);
    const size_t cjm = c - (size_t)j * nx + (size_t)(j == 0 ? ny - 1 : j - 1) * nx;
    const double r = rho[c];
    const double idzf = g.inv_dzf[k];
    // stretched y (face weights dzf s_j on x faces, dzf / t_j on y faces,
    // dzc s_j on z faces; s_j = dyf_j / dy, t_j = dy / dyc_j)
    const double is = g.ym ? g.ym[2 * ny + j] : 1.0, tj = g.ym ? g.ym[ny + j] : 1.0;
    yu[c] = -dt * (2.0 / (r + rho[cim])) * gu[c] * idzf * is;
    // with walls in y the wall row of v is not an unknown: no gradient enters there
    yv[c] = (g.ywall && j == 0) ? 0.0 : -dt * (2.0 / (r + rho[cjm])) * gv[c] * idzf * tj;
    yw[c] = (k == 0) ? 0.0 : -dt * (2.0 / (r + rho[c - plane])) * gw[c] * g.inv_dzc[k] * is;
    if (k == nz - 1) yw[c + plane] = 0.0;
  }
}

// gus = g + W_f G mu; t = d beta/d rho * g_beta with g_beta = -dt (G p) gus.
__global__ void k_adj_finish(Geo g, const double* __restrict__ rho, const double* __restrict__ p,
                             const double* __restrict__ mu, double dt, const double* __restrict__ gu,
                             const double* __restrict__ gv, const double* __restrict__ gw,
                             double* __restrict__ gus, double* __restrict__ gvs, double* __restrict__ gws,
                             double* __restrict__ tx, double* __restrict__ ty, double* __restrict__ tz) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const size_t plane = (size_t)nx * ny, n = plane * nz;
  const double idx = 1.0 / g.dx, idy = 1.0 / g.dy;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(c % nx);
    const int j = (int)((c / nx) % ny);
    const int k = (int)(c / plane);
    const size_t cim = c - i + (i == 0 ? nx - 1 : i - 1);
    const size_t cjm = c - (size_t)j * nx + (size_t)(j == 0 ? ny - 1 : j - 1) * nx;
    const double dzf = g.dzf[k];
    const double r = rho[c];
    // stretched y: x-face weight dzf s_j, y-face weight dzf / t_j against
    // G_y = t_j / dy (the two cancel), z-face weight dzc s_j
    const double sj = g.ym ? g.ym[j] : 1.0, tj = g.ym ? g.ym[ny + j] : 1.0;
    const double a = gu[c] + dzf * sj * (mu[c] - mu[cim]) * idx;
    const bool vwall = g.ywall && j == 0;  // wall row of v: zero gradient, no density dependence
    const double bb = vwall ? 0.0 : gv[c] + dzf * (mu[c] - mu[cjm]) * idy;
    gus[c] = a;
    gvs[c] = bb;
    const double bx = 2.0 / (r + rho[cim]), by = 2.0 / (r + rho[cjm]);
    tx[c] = -0.5 * bx * bx * (-dt * (p[c] - p[cim]) * idx * a);
    ty[c] = vwall ? 0.0 : -0.5 * by * by * (-dt * (p[c] - p[cjm]) * idy * tj * bb);
    if (k == 0) {
      gws[c] = 0.0;
      tz[c] = 0.0;
    } else {
      const double cc = gw[c] + sj * (mu[c] - mu[c - plane]);
      gws[c] = cc;
      const double bz = 2.0 / (r + rho[c - plane]);
      tz[c] = -0.5 * bz * bz * (-dt * (p[c] - p[c - plane]) * g.inv_dzc[k] * cc);
    }
    if (k == nz - 1) { gws[c + plane] = 0.0; tz[c + plane] = 0.0; }
  }
}

__global__ void k_adj_grho(Geo g, const double* __restrict__ tx, const double* __restrict__ ty,
                           const double* __restrict__ tz, double* __restrict__ grho) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const size_t plane = (size_t)nx * ny, n = plane * nz;
  for (size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(c % nx);
    const int j = (int)((c / nx) % ny);
    const size_t cip = c - i + (i + 1 == nx ? 0 : i + 1);
    const size_t cjp = c - (size_t)j * nx + (size_t)(j + 1 == ny ? 0 : j + 1) * nx;
    grho[c] = tx[c] + tx[cip] + ty[c] + ty[cjp] + tz[c] + tz[c + plane];
  }
  (void)nz;
}

// ---------------------------------------------------------------------------
cudaError_t launch_mixture(const double* phi, double rho_g, double rho_l, double* rho, size_t n,
                           cudaStream_t s) {
  k_mixture<<<grid_for(n), kThreads, 0, s>>>(phi, rho_g, rho_l, rho, n);
  return cudaGetLastError();
}

cudaError_t launch_prep_faces(const Geo& g, const double* rho, Faces fc, cudaStream_t s) {
  k_prep_faces<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, rho, fc);
  k_prep_diag<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, fc);
  return cudaGetLastError();
}

cudaError_t launch_weighted_mean(const Geo& g, const double* f, double* red, double* out_mean,
                                 cudaStream_t s) {
  k_weighted_partial<<<kRedBlocks, kThreads, 0, s>>>(g, f, red);
  k_finalize<<<1, 1024, 0, s>>>(red, kRedBlocks, 1, 0, 1.0 / (g.lz * (double)g.nx * g.ny), out_mean);
  return cudaGetLastError();
}

cudaError_t launch_rhs_b(const Geo& g, const double* us, const double* vs, const double* ws,
                         const double* S, double* b, double* red, DevStatus* st, double inv_dt,
                         cudaStream_t s) {
  k_rhs_b<<<kRedBlocks, kThreads, 0, s>>>(g, us, vs, ws, S, st, b, red, inv_dt);
  k_finalize<<<1, 1024, 0, s>>>(red, kRedBlocks, 1, 0, inv_dt * inv_dt, &st->e2_0);
  return cudaGetLastError();
}

cudaError_t launch_init_status(DevStatus* st, cudaStream_t s) {
  k_init_status<<<1, 1, 0, s>>>(st);
  return cudaGetLastError();
}

cudaError_t launch_correct(const Geo& g, const Faces& fc, const double* us, const double* vs,
                           const double* ws, const double* p, double dt, double* u, double* v,
                           double* w, cudaStream_t s) {
  k_correct<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, fc, us, vs, ws, p, dt, u, v, w);
  return cudaGetLastError();
}

cudaError_t launch_rho_tilde(const Geo& g, const double* rho, int method, double* red, double* out,
                             cudaStream_t s) {
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  k_rho_extrema<<<kExtBlocks, kThreads, 0, s>>>(n, rho, red);
  k_rho_tilde<<<1, 1, 0, s>>>(red, kExtBlocks, method, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_correct_method1(const Geo& g, const Faces& fc, const double* us, const double* vs,
                                   const double* ws, const double* p, const T* delta, double dt,
                                   double* u, double* v, double* w, cudaStream_t s) {
  k_correct_method1<T><<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, fc, us, vs, ws, p, delta,
                                                                               dt, u, v, w);
  return cudaGetLastError();
}
template cudaError_t launch_correct_method1<double>(const Geo&, const Faces&, const double*, const double*,
                                                    const double*, const double*, const double*, double,
                                                    double*, double*, double*, cudaStream_t);
template cudaError_t launch_correct_method1<float>(const Geo&, const Faces&, const double*, const double*,
                                                   const double*, const double*, const float*, double,
                                                   double*, double*, double*, cudaStream_t);

cudaError_t launch_thermo_rate(const Geo& g, const double* phi, const double* kc, const double* T,
                               const double* u, const double* v, const double* w, double p0, double gamma,
                               double* red, double* out, cudaStream_t s) {
  constexpr int kThermoBlocks = kRedBlocks / 3;  // three partial sums per block fit the buffer
  k_thermo_partial<<<kThermoBlocks, kThreads, 0, s>>>(g, phi, kc, T, u, v, w, red);
  k_thermo_rate<<<1, 1024, 0, s>>>(red, kThermoBlocks, p0, gamma, out);
  return cudaGetLastError();
}

cudaError_t launch_divergence_source(const Geo& g, const double* phi, const double* kc, const double* T,
                                     double p0, double gamma, double dp0dt, double* S, cudaStream_t s) {
  k_divergence_source<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(
      g, phi, kc, T, 0.5 * (gamma - 1.0) / gamma / p0, dp0dt / gamma / p0, S);
  return cudaGetLastError();
}

cudaError_t launch_predictor(const Geo& g, const double* u, const double* v, const double* w, const double* rho,
                             const double* mu, const double* const f[3], const double* const prev[3],
                             const double grav[3], double dt, double a, double b, double* const out[3],
                             double* const ru[3], cudaStream_t s) {
  // A warp per 30 cells of a row (or per 32 / nx rows) and chunk of layers: long
  // chunks (a chunk repeats about 0.7 of a layer), but at least about 16 warps
  // an SM.  Where chunks of eight leave fewer, the warps are counted: a warp
  // takes about 6 us a layer, the FP64 unit's time, so an SM partition with a
  // second warp takes twice as long (40^3, four layers a chunk: 0.059 ms, 800
  // warps on 608 partitions; six layers, 560 warps: 0.047).
  const bool whole = g.nx <= 32;
  const int ntile = whole ? 1 : (g.nx + kPredLanes - 1) / kPredLanes;
  const int ngroup = whole ? (g.ny + 32 / g.nx - 1) / (32 / g.nx) : g.ny;
  const long long rows = (long long)ntile * ngroup;
  auto warps = [&](int c) { return rows * ((g.nz + c - 1) / c); };
  int chunk = 64;
  while (chunk > 8 && warps(chunk) < 152 * 16) chunk >>= 1;
  if (warps(chunk) < 152 * 16) {
    long long best = -1;
    for (int c = 1; c <= 32; ++c) {
      const long long cost = (warps(c) + 152 * 4 - 1) / (152 * 4) * (10 * c + 7);
      if (best < 0 || cost < best) {
        best = cost;
        chunk = c;
      }
    }
  }
  const int nchunk = (g.nz + chunk - 1) / chunk;
  const PredArgs A{u, v, w, rho, mu, f[0], f[1], f[2], prev[0], prev[1], prev[2], grav[0], grav[1], grav[2],
                   dt * a, dt * b, g.inv_dx, g.inv_dy, 0.5 * g.inv_dx, 0.5 * g.inv_dy, 8.0 * g.inv_dx,
                   8.0 * g.inv_dy, out[0], out[1], out[2], ru[0], ru[1], ru[2]};
  auto kern = whole ? k_predictor<true> : k_predictor<false>;
  kern<<<(unsigned)((rows * nchunk + 3) / 4), 128, 0, s>>>(g, A, ntile, ngroup, nchunk, chunk);
  return cudaGetLastError();
}

cudaError_t launch_remove_mean(const Geo& g, double* p, double* red, DevStatus* st, cudaStream_t s) {
  cudaError_t e = launch_weighted_mean(g, p, red, &st->pmean, s);
  if (e != cudaSuccess) return e;
  const size_t n = (size_t)g.nx * g.ny * g.nz;
  k_sub_mean<<<grid_for(n), kThreads, 0, s>>>(p, n, st);
  return cudaGetLastError();
}

cudaError_t launch_setup_pivots(const Geo& g, const double* lamx, const double* lamy, double* invd,
                                cudaStream_t s, double* mtab) {
  const size_t ncol = (size_t)g.ny * g.nxh;
  k_setup_pivots<<<(int)((ncol + 127) / 128), 128, 0, s>>>(g, lamx, lamy, invd, mtab);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_setup_z(const Geo& g, const double* lamx, const double* lamy, int nyt, double* m, double* e,
                           T* d, cudaStream_t s) {
  const size_t ntc = (size_t)nyt * g.nxh;
  k_setup_z<T><<<(int)((ntc + 127) / 128), 128, 0, s>>>(g, lamx, lamy, nyt, m, e, d);
  return cudaGetLastError();
}
template cudaError_t launch_setup_z<float>(const Geo&, const double*, const double*, int, double*, double*, float*,
                                           cudaStream_t);
template cudaError_t launch_setup_z<double>(const Geo&, const double*, const double*, int, double*, double*, double*,
                                            cudaStream_t);

cudaError_t launch_adj_rhs(const Geo& g, const double* rho, const double* gu, const double* gv,
                           const double* gw, double dt, double* yu, double* yv, double* yw,
                           cudaStream_t s) {
  k_adj_rhs<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, rho, gu, gv, gw, dt, yu, yv, yw);
  return cudaGetLastError();
}

cudaError_t launch_adj_finish(const Geo& g, const double* rho, const double* p, const double* mu,
                              double dt, const double* gu, const double* gv, const double* gw,
                              double* gus, double* gvs, double* gws, double* tx, double* ty,
                              double* tz, cudaStream_t s) {
  k_adj_finish<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, rho, p, mu, dt, gu, gv, gw,
                                                                         gus, gvs, gws, tx, ty, tz);
  return cudaGetLastError();
}

cudaError_t launch_adj_grho(const Geo& g, const double* tx, const double* ty, const double* tz,
                            double* grho, cudaStream_t s) {
  k_adj_grho<<<grid_for((size_t)g.nx * g.ny * g.nz), kThreads, 0, s>>>(g, tx, ty, tz, grho);
  return cudaGetLastError();
}

}  // namespace pp
