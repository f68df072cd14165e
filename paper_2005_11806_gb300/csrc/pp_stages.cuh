// Device-side stages of one constant-coefficient eigenexpansion solve
// (Sec. 3.3.1: the pressure equation with homogeneous boundary conditions
// solved exactly by the eigenexpansion method) and of Algorithm 1's pass:
// residual + forward x transform, y transforms, the per-(kx, ky) tridiagonal
// solve along z, and the inverse x transform fused with the pressure update.
// The single-grid kernels (pp_kernels_fft.cu) and the grouped multi-grid
// kernels (pp_batch.cu) both call these.
#pragma once
#include <type_traits>

#include "pp_cells.cuh"
#include "pp_fft.cuh"
#include "pp_zsweep.cuh"

namespace pp {

constexpr int kThreads = 256;
// FFT elements per block = kEpt * kThreads (two shared buffers of that many
// complex values).  8 was the fastest of {2, 4, 8, 16} for every kernel in a
// 512^3 sweep on GB300.
constexpr int kEpt = 8;
constexpr int kPrefetchInv = 8;  // p values prefetched per thread in the inverse x kernel

// Rows per block of the x kernels: (rows/2) complex sequences of length nx
// with at most ept * kThreads elements in the shared buffer.
inline int rows_per_block(int nx, int ept) {
  int nseq = (ept * kThreads) / nx;
  if (nseq > 32) nseq = 32;
  if (nseq < 1) nseq = 1;
  return 2 * nseq;
}

// kx columns per y tile: a power of two with tx * ny <= ept * kThreads.
inline int ffty_tile(int ny, size_t csize, int ept) {
  int tx = (int)(128 / csize);  // 128-byte row segments
  while (tx > 1 && ny * tx > ept * kThreads) tx >>= 1;
  return tx;
}

__device__ __forceinline__ bool stopped(const DevStatus* st) { return st != nullptr && st->done; }

// Transform dispatch: compile-time passes for FP64 lines of 512 (x, y and z) and
// of 256, 128 and 64 along z (cosine plans), the generic mixed-radix passes
// otherwise (same passes in the same order, so the same results).  FP32 lines
// of 512 take fft_dispatch_smem; x and y lines of the other powers of two the
// register transforms of pp_wfft.cuh.
#define PP_TRY_FIXED(NN, NBB)                                                                       \
  if (n == NN && nbatch == NBB) {                                                                   \
    if (BATCH_FAST) return fft_block_fixed<T, DIR, true, NN, NBB, NBB, 1>(a, b, tw, tid, nth);      \
    return fft_block_fixed<T, DIR, false, NN, NBB, 1, NN>(a, b, tw, tid, nth);                      \
  }

template <typename T, int DIR, bool BATCH_FAST>
__device__ __forceinline__ C2<T>* fft_dispatch(C2<T>* a, C2<T>* b, const FftDesc& d, int nbatch, int es, int bs,
                                               const C2<T>* __restrict__ tw, int tid, int nth) {
  const int n = d.n;
  const bool shape_ok = BATCH_FAST ? (es == nbatch && bs == 1) : (es == 1 && bs == n);
  if constexpr (std::is_same<T, double>::value) {
    if (shape_ok) {
      PP_TRY_FIXED(512, 4)
      if constexpr (BATCH_FAST) {
        PP_TRY_FIXED(256, 8)
        PP_TRY_FIXED(128, 8)
        PP_TRY_FIXED(64, 8)
      }
    }
  }
  return fft_block<T, DIR, BATCH_FAST>(a, b, d, nbatch, es, bs, tw, tid, nth);
}
#undef PP_TRY_FIXED

// Whether the FP32 fast path (fft_dispatch_smem) takes this shape.
__host__ __device__ inline bool fft_smem_shape(int n, int nbatch) { return n == 512 && nbatch == 4; }

// FP32 fast path (fft_block_smem) of that shape; returns the element offset of
// the result buffer.  twb: offset of the N-entry twiddle table.
template <int DIR, bool BATCH_FAST>
__device__ __forceinline__ int fft_dispatch_smem(int a, int b, int twb, int tid, int nth) {
  return fft_block_smem<DIR, BATCH_FAST, 512, 4, BATCH_FAST ? 4 : 1, BATCH_FAST ? 1 : 512>(a, b, twb, tid, nth);
}

// Copies the N-entry twiddle table into shared memory at element offset twb.
__device__ __forceinline__ void load_twiddles_smem(const float2* __restrict__ tw, int n, int twb) {
  float2* S = smem_f2();
  for (int i = threadIdx.x; i < n; i += blockDim.x) S[twb + i] = tw[i];
}

// ---------------------------------------------------------------------------
// Update pass of the mixed residual for nx % 4 == 0, vectorised: each thread
// takes the two rows of one complex sequence and four consecutive cells of
// each (16-byte loads of E, delta and the FP32 density), subtracts A delta
// from E, and writes the scaled residual of both rows as two interleaved
// complex pairs.
//
// A delta is formed from half fluxes G = (delta_b - delta_a) / (rho_a +
// rho_b), one per face: an add, an add, a reciprocal and a multiply, shared
// by the face's two cells where both are in the thread (5 x faces for 4
// cells; with two rows taken together 3 y faces for 2 cells), then
//   A delta = 2 [w_x (G_x+ - G_x-) + w_y+ G_y+ - w_y- G_y- + w_z+ G_z+ - w_z- G_z-]
// with the layer (and row) factors w.  Coefficients formed per cell and face,
// with the range checks of a division each, take 111 instructions a cell with
// the transform and 0.098 ms at 256^3, 0.678 ms at 512^3; this form takes 87,
// 0.091 ms and 0.644 ms.
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float half_flux(float da, float db, float ha, float hb) {
  return (db - da) * rcp_f32(ha + hb);
}
__device__ __forceinline__ float4 half_flux4(float4 da, float4 db, float4 ha, float4 hb) {
  return make_float4(half_flux(da.x, db.x, ha.x, hb.x), half_flux(da.y, db.y, ha.y, hb.y),
                     half_flux(da.z, db.z, ha.z, hb.z), half_flux(da.w, db.w, ha.w, hb.w));
}

// Factors of one row (all carry the 2 of the fluxes): x faces, y faces below
// and above, z faces below and above, 1 / dzf (1 / (dzf s_j) on a stretched
// y), the scaling of the residual where it is constant.
struct RowW {
  float x, yl, yh, zd, zu, iv;
};

// What the four cells of a row at offset c need beside their own delta and
// density: the x neighbours (il, ir), the layers above and below, E.
struct RowIn {
  float4 du, hu, dd, hd, e;
  float dl, dr, hl, hr;
};
__device__ __forceinline__ RowIn load_row(const float* __restrict__ E, const float* __restrict__ delta,
                                          const float* __restrict__ rhof, unsigned c, unsigned il, unsigned ir,
                                          unsigned plane, bool up, bool dn) {
  RowIn x;
  const unsigned cu = up ? c + plane : c, cd = dn ? c - plane : c;  // at a wall: the cell itself, no flux
  x.e = ld4(E + c);
  x.du = ld4(delta + cu);
  x.dd = ld4(delta + cd);
  x.hu = ld4(rhof + cu);
  x.hd = ld4(rhof + cd);
  x.dl = delta[il];
  x.dr = delta[ir];
  x.hl = rhof[il];
  x.hr = rhof[ir];
  return x;
}
// Keeps every load before it in flight together: left to itself the compiler
// sinks them to their uses, and a thread waits for memory several times in a
// step (residual 256^3 0.104 -> 0.094 ms, 512^3 0.672 -> 0.644 ms).
__device__ __forceinline__ void loads_issued() { asm volatile("" ::: "memory"); }

// The four cells of a row: their E updated in place, their scaled residuals
// returned, e^2 and |e| added to s2 and s1.  Gl, Gh: the half fluxes of the y
// faces below and above.
__device__ __forceinline__ float4 resid_row4(const RowW& w, const RowIn& x, float* __restrict__ E, unsigned c, float4 d,
                                             float4 h, float4 Gl, float4 Gh, bool scale, bool own, float rt_f,
                                             float& s2, float& s1) {
  float4 e = x.e;
  const float x0 = half_flux(x.dl, d.x, x.hl, h.x), x1 = half_flux(d.x, d.y, h.x, h.y),
              x2 = half_flux(d.y, d.z, h.y, h.z), x3 = half_flux(d.z, d.w, h.z, h.w),
              x4 = half_flux(d.w, x.dr, h.w, x.hr);
  const float4 Gu = half_flux4(d, x.du, h, x.hu), Gd = half_flux4(x.dd, d, x.hd, h);
  auto cell = [&](float xm, float xp, float gl, float gh, float gd, float gu, float& ev, float hv) -> float {
    float t = w.x * (xp - xm);
    t = fmaf(w.yh, gh, t);
    t = fmaf(-w.yl, gl, t);
    t = fmaf(w.zu, gu, t);
    t = fmaf(-w.zd, gd, t);
    ev = ev - t;
    const float ee = ev * w.iv;
    s2 = fmaf(ee, ee, s2);
    s1 += fabsf(ee);
    return scale ? (own ? hv : rt_f) * ee : ee;
  };
  float4 r;
  r.x = cell(x0, x1, Gl.x, Gh.x, Gd.x, Gu.x, e.x, h.x);
  r.y = cell(x1, x2, Gl.y, Gh.y, Gd.y, Gu.y, e.y, h.y);
  r.z = cell(x2, x3, Gl.z, Gh.z, Gd.z, Gu.z, e.z, h.z);
  r.w = cell(x3, x4, Gl.w, Gh.w, Gd.w, Gu.w, e.w, h.w);
  *reinterpret_cast<float4*>(E + c) = e;
  return r;
}

// Factors of row j of layer k.  The y faces of the walls are 0; a stretched y
// (YS) scales the x and z faces by s_j, the y faces below and above by t_j
// and t_{j+1}, the cell's value by 1 / s_j.
template <bool YS>
__device__ __forceinline__ RowW row_factors(const Geo& g, int k, int j) {
  const int nz1 = g.nz + 1, ny = g.ny;
  RowW w;
  w.x = 2.f * g.cw_f[k];
  w.yl = (g.ywall && j == 0) ? 0.f : 2.f * g.cw_f[nz1 + k];
  w.yh = (g.ywall && j + 1 == ny) ? 0.f : 2.f * g.cw_f[nz1 + k];
  w.zd = 2.f * g.cw_f[2 * nz1 + k];
  w.zu = 2.f * g.cw_f[2 * nz1 + k + 1];
  w.iv = g.inv_dzf_f[k];
  if constexpr (YS) {
    const float sj = g.ym_f[j];
    w.x *= sj;
    w.zd *= sj;
    w.zu *= sj;
    w.yl *= g.ym_f[ny + j];
    w.yh = (j + 1 < ny) ? w.yh * g.ym_f[ny + j + 1] : 0.f;
    w.iv *= g.ym_f[2 * ny + j];
  }
  return w;
}

// Odd ny: the two rows of a sequence one after the other.
template <bool YS>
__device__ __forceinline__ void resid_update_vec4(const Geo& g, const Faces& fc, float* __restrict__ E,
                                                  const float* __restrict__ delta, bool scale, bool own, float rt_f,
                                                  long row0, int rpb, float2* bufA, int seq_stride, float& s2,
                                                  float& s1, int tid, int nth) {
  // 32-bit cell offsets (grids keep nx ny (nz + 1) below 2^31); the first row
  // is split into (layer, row in layer) once, the others step from it (no
  // 64-bit division per cell group)
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int nrows = nz * ny;
  const unsigned plane = (unsigned)nx * ny;
  const int t4 = nx >> 2;
  const int npairs = rpb >> 1;
  const int lg4 = ((t4 & (t4 - 1)) == 0) ? 31 - __clz(t4) : -1;
  const int r0 = (int)row0;
  const int k0 = r0 / ny, j0 = r0 - k0 * ny;
  for (int w = tid; w < npairs * t4; w += nth) {
    const int qp = lg4 >= 0 ? (w >> lg4) : w / t4;
    const int i = (w - qp * t4) << 2;
    float4 rr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = r0 + 2 * qp + h;
      rr[h] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (row < nrows) {
        int k = k0, j = j0 + 2 * qp + h;
        while (j >= ny) { j -= ny; ++k; }
        const int jp = (j + 1 == ny) ? 0 : j + 1, jm = (j == 0) ? ny - 1 : j - 1;
        const unsigned rowoff = (unsigned)row * nx, kp = (unsigned)k * plane, c = rowoff + i;
        const unsigned cyp = kp + (unsigned)jp * nx + i, cym = kp + (unsigned)jm * nx + i;
        const float4 d = ld4(delta + c), hc = ld4(fc.rhof + c);
        const float4 dm = ld4(delta + cym), hm = ld4(fc.rhof + cym), dp = ld4(delta + cyp), hp = ld4(fc.rhof + cyp);
        const RowIn in = load_row(E, delta, fc.rhof, c, rowoff + (i == 0 ? nx - 1 : i - 1),
                                  rowoff + (i + 4 == nx ? 0 : i + 4), plane, k + 1 < nz, k > 0);
        loads_issued();
        rr[h] = resid_row4(row_factors<YS>(g, k, j), in, E, c, d, hc, half_flux4(dm, d, hm, hc),
                           half_flux4(d, dp, hc, hp), scale, own, rt_f, s2, s1);
      }
    }
    float4* dst = reinterpret_cast<float4*>(bufA + qp * seq_stride + i);
    dst[0] = make_float4(rr[0].x, rr[1].x, rr[0].y, rr[1].y);
    dst[1] = make_float4(rr[0].z, rr[1].z, rr[0].w, rr[1].w);
  }
}

// The same update with the two rows of a sequence taken together.  With ny
// even, rows 2q and 2q + 1 (the first row is even) lie in one layer and are y
// neighbours of each other: the rows j - 1 .. j + 2 of delta and of the
// density are loaded once each and the face between the two rows is formed
// once.
template <bool YS>
__device__ __forceinline__ void resid_update_pair4(const Geo& g, const Faces& fc, float* __restrict__ E,
                                                   const float* __restrict__ delta, bool scale, bool own, float rt_f,
                                                   long row0, int rpb, float2* bufA, int seq_stride, float& s2,
                                                   float& s1, int tid, int nth) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int nrows = nz * ny;
  const unsigned plane = (unsigned)nx * ny;
  const int t4 = nx >> 2;
  const int npairs = rpb >> 1;
  const int lg4 = ((t4 & (t4 - 1)) == 0) ? 31 - __clz(t4) : -1;
  const int r0 = (int)row0;
  const int k0 = r0 / ny, j0 = r0 - k0 * ny;
  for (int w = tid; w < npairs * t4; w += nth) {
    const int qp = lg4 >= 0 ? (w >> lg4) : w / t4;
    const int i = (w - qp * t4) << 2;
    const int row = r0 + 2 * qp;  // row A; row B = row + 1, same layer
    float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra;
    if (row < nrows) {
      int k = k0, j = j0 + 2 * qp;
      while (j >= ny) { j -= ny; ++k; }
      const int jm = (j == 0) ? ny - 1 : j - 1;
      const int jpp = (j + 2 == ny) ? 0 : j + 2;
      const unsigned oa = (unsigned)row * nx, ob = oa + nx;
      const unsigned kp = (unsigned)k * plane;
      const unsigned ca = oa + i, cb = ob + i;
      const unsigned cm = kp + (unsigned)jm * nx + i, cp = kp + (unsigned)jpp * nx + i;
      const int il = (i == 0) ? nx - 1 : i - 1, ir = (i + 4 == nx) ? 0 : i + 4;
      const bool up = k + 1 < nz, dn = k > 0;
      const float4 dA = ld4(delta + ca), dB = ld4(delta + cb);
      const float4 hA = ld4(fc.rhof + ca), hB = ld4(fc.rhof + cb);
      const float4 dM = ld4(delta + cm), hM = ld4(fc.rhof + cm), dP = ld4(delta + cp), hP = ld4(fc.rhof + cp);
      const RowIn inA = load_row(E, delta, fc.rhof, ca, oa + il, oa + ir, plane, up, dn);
      const RowIn inB = load_row(E, delta, fc.rhof, cb, ob + il, ob + ir, plane, up, dn);
      RowW wa = row_factors<YS>(g, k, j), wb = wa;
      if constexpr (YS) wb = row_factors<YS>(g, k, j + 1);
      else { wb.yl = wa.yh; wb.yh = (g.ywall && j + 2 == ny) ? 0.f : wa.yh; }
      loads_issued();
      const float4 Gm = half_flux4(dA, dB, hA, hB);
      ra = resid_row4(wa, inA, E, ca, dA, hA, half_flux4(dM, dA, hM, hA), Gm, scale, own, rt_f, s2, s1);
      rb = resid_row4(wb, inB, E, cb, dB, hB, Gm, half_flux4(dB, dP, hB, hP), scale, own, rt_f, s2, s1);
    }
    float4* dst = reinterpret_cast<float4*>(bufA + qp * seq_stride + i);
    dst[0] = make_float4(ra.x, rb.x, ra.y, rb.y);
    dst[1] = make_float4(ra.z, rb.z, ra.w, rb.w);
  }
}

// FP64 residual with the two rows of a sequence taken together (ny even: rows
// 2q and 2q + 1 are y neighbours in one layer): the y neighbours and the y
// coefficients between them are loaded once, and a thread has 23 loads in
// flight for two cells.  Per cell: seven FMAs, then the scaling and the norms.
template <bool YS>
__device__ __forceinline__ void resid_exact_pair(const Geo& g, const Faces& fc, const double* __restrict__ b,
                                                 const double* __restrict__ rho, const double* __restrict__ p,
                                                 bool scale, bool const_scale, double rt, long row0, int rpb,
                                                 double2* bufA, int seq_stride, double& s2, double& s1, int tid,
                                                 int nth) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int nrows = nz * ny;
  const unsigned plane = (unsigned)nx * ny;
  const int npairs = rpb >> 1;
  const int r0 = (int)row0;
  const int k0 = r0 / ny, j0 = r0 - k0 * ny;
  const int tpr = nx < nth ? nx : nth, par = nth / tpr;
  const int q0 = tid / tpr, i0 = tid - q0 * tpr;
  for (int q = q0; q < npairs && q0 < par; q += par) {
    const int row = r0 + 2 * q;
    if (row >= nrows) {
      for (int i = i0; i < nx; i += tpr) bufA[(size_t)q * seq_stride + i] = make_double2(0.0, 0.0);
      continue;
    }
    int k = k0, j = j0 + 2 * q;
    while (j >= ny) { j -= ny; ++k; }
    const unsigned kp = (unsigned)k * plane;
    const unsigned oa = (unsigned)row * nx, ob = oa + nx;
    const unsigned om = kp + (unsigned)(j == 0 ? ny - 1 : j - 1) * nx, op = kp + (unsigned)(j + 2 == ny ? 0 : j + 2) * nx;
    const bool up = k + 1 < nz, dn = k > 0;
    const double iva = g.inv_dzf[k] * (YS ? g.ym[2 * ny + j] : 1.0), ivb = YS ? g.inv_dzf[k] * g.ym[2 * ny + j + 1] : iva;
    for (int i = i0; i < nx; i += tpr) {
      const int ip = (i + 1 == nx) ? 0 : i + 1, im = (i == 0) ? nx - 1 : i - 1;
      const unsigned ca = oa + i, cb = ob + i;
      const double pa = p[ca], pb = p[cb], pm = p[om + i], pp = p[op + i];
      const double pal = p[oa + im], par_ = p[oa + ip], pbl = p[ob + im], pbr = p[ob + ip];
      const double xa = fc.cx[ca], xar = fc.cx[oa + ip], xb = fc.cx[cb], xbr = fc.cx[ob + ip];
      const double ya = fc.cy[ca], yb = fc.cy[cb], yp = fc.cy[op + i];
      const double za = fc.cz[ca], zau = fc.cz[ca + plane], zb = fc.cz[cb], zbu = fc.cz[cb + plane];
      double pau = 0.0, pbu = 0.0, pad = 0.0, pbd = 0.0;  // the wall faces' coefficients are 0
      if (up) { pau = p[ca + plane]; pbu = p[cb + plane]; }
      if (dn) { pad = p[ca - plane]; pbd = p[cb - plane]; }
      double ea = fma(fc.diag[ca], pa, b[ca]), eb = fma(fc.diag[cb], pb, b[cb]);
      const double ha = scale ? (const_scale ? rt : rho[ca]) : 1.0, hb = scale ? (const_scale ? rt : rho[cb]) : 1.0;
      ea = fma(-xar, par_, ea);
      eb = fma(-xbr, pbr, eb);
      ea = fma(-xa, pal, ea);
      eb = fma(-xb, pbl, eb);
      ea = fma(-yb, pb, ea);
      eb = fma(-yp, pp, eb);
      ea = fma(-ya, pm, ea);
      eb = fma(-yb, pa, eb);
      if (up) { ea = fma(-zau, pau, ea); eb = fma(-zbu, pbu, eb); }
      if (dn) { ea = fma(-za, pad, ea); eb = fma(-zb, pbd, eb); }
      ea *= iva;
      eb *= ivb;
      s2 = fma(ea, ea, s2);
      s1 += fabs(ea);
      s2 = fma(eb, eb, s2);
      s1 += fabs(eb);
      bufA[(size_t)q * seq_stride + i] = make_double2(scale ? ha * ea : ea, scale ? hb * eb : eb);
    }
  }
}

// ---------------------------------------------------------------------------
// Residual of the variable-coefficient equation and forward real x transform.
//   mode 0: r = f (constant-coefficient solve)
//   mode 1: e = (D u^s - S_c)/dt, evaluated in FP64 in the row-scaled form
//           dzf_k e = b_s - (sum_nb c_nb p_nb - diag p_c), b_s = dzf_k b / dt;
//           r = rho e (or e).  The mixed path narrows dzf_k e to FP32 and
//           finishes (scaling, norms, rho) in FP32.
//   Mixed path with E: E = dzf_k e is kept in FP32.  An exact pass stores
//   the FP64 value narrowed; an update pass subtracts A delta, evaluated in
//   FP32 as sum_nb c_nb (delta_nb - delta_c) (no diagonal needed).
// Two real rows are packed into one complex sequence (re = even row,
// im = odd row), transformed together and separated afterwards.
// The rows [row0, row0 + rpb) of the residual (the first step of the stage
// below) into bufA: complex sequence q = (row - row0) / 2 at element offset
// q * seq_stride (re = even row, im = odd row); s2, s1 accumulate e^2 and
// |e| of the thread's cells.  Called by nth threads (a block, or a warp), tid
// their index.
template <typename T, bool YS>
__device__ __forceinline__ void resid_rows(const Geo& g, const Faces& fc, const double* __restrict__ b,
                                           const double* __restrict__ rho, const double* __restrict__ p, int mode,
                                           int p_zero, int scale_rho, long row0, int rpb, bool need_exact,
                                           float* __restrict__ E, const float* __restrict__ delta, C2<T>* bufA,
                                           int seq_stride, T& s2, T& s1, int tid, int nth) {
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const bool update = (E != nullptr) && !p_zero && !need_exact;
  const int nrows = nz * ny;
  const size_t plane = (size_t)ny * nx;
  // constant scaling of Methods I and II (one device scalar for all cells)
  const bool const_scale = fc.rho_tilde != nullptr;
  const double rt = (const_scale && mode != 0) ? *fc.rho_tilde : 0.0;
  const float rt_f = (float)rt;
  // thread -> (row offset, first column); index math is done once per row
  const int tpr = nx < nth ? nx : nth;
  const int rows_par = nth / tpr;
  const int qoff = tid / tpr, i0 = tid - qoff * tpr;
  bool vec = update && sizeof(T) == sizeof(float) && (nx & 3) == 0;
  if (vec) {
    float a2 = 0.f, a1 = 0.f;
    if ((ny & 1) == 0)  // the two rows of a sequence share a layer
      resid_update_pair4<YS>(g, fc, E, delta, scale_rho != 0, !const_scale, rt_f, row0, rpb,
                             reinterpret_cast<float2*>(bufA), seq_stride, a2, a1, tid, nth);
    else
      resid_update_vec4<YS>(g, fc, E, delta, scale_rho != 0, !const_scale, rt_f, row0, rpb,
                            reinterpret_cast<float2*>(bufA), seq_stride, a2, a1, tid, nth);
    s2 += (T)a2;
    s1 += (T)a1;
  }
  if constexpr (sizeof(T) == sizeof(double)) {
    if (mode != 0 && !p_zero && (ny & 1) == 0) {
      resid_exact_pair<YS>(g, fc, b, rho, p, scale_rho != 0, const_scale, rt, row0, rpb,
                           reinterpret_cast<double2*>(bufA), seq_stride, s2, s1, tid, nth);
      vec = true;
    }
  }
  for (int q = qoff; !vec && q < rpb && qoff < rows_par; q += rows_par) {
    const int row = (int)row0 + q;
    const bool valid = row < nrows;
    const int k = valid ? row / ny : 0, j = valid ? row - k * ny : 0;
    const int jp = (j + 1 == ny) ? 0 : j + 1, jm = (j == 0) ? ny - 1 : j - 1;
    const size_t rowoff = (size_t)row * nx;
    const size_t kp = (size_t)k * plane;
    const size_t rowp = kp + (size_t)jp * nx, rowm = kp + (size_t)jm * nx;
    // stretched y: the row is scaled by dzf_k s_j (Geo::ym)
    const bool ys = YS && valid;
    const float idzf_f =
        (mode != 0 && sizeof(T) == sizeof(float)) ? g.inv_dzf_f[k] * (ys ? g.ym_f[2 * ny + j] : 1.f) : 0.f;
    const double idzf =
        (mode != 0 && sizeof(T) == sizeof(double)) ? g.inv_dzf[k] * (ys ? g.ym[2 * ny + j] : 1.0) : 0.0;
    const float ysj = ys ? g.ym_f[j] : 1.f, ytlo = ys ? g.ym_f[ny + j] : 1.f;
    const float ythi = ys ? ((j + 1 < ny) ? g.ym_f[ny + j + 1] : 0.f) : 1.f;
    for (int i = i0; i < nx; i += tpr) {
      T r = (T)0;
      if (valid) {
        const size_t c = rowoff + i;
        if (mode == 0) {
          r = (T)b[c];
        } else {
          const int ip = (i + 1 == nx) ? 0 : i + 1, im = (i == 0) ? nx - 1 : i - 1;
          double ep = 0.0;
          float ev = 0.f;  // FP32 dzf_k e of the mixed path
          if (update) {
            // E^s = E^{s-1} - A delta, A delta in FP32 with the FP32
            // coefficients formed from rhof (as in resid_update_vec4)
            const float dc = delta[c];
            const float rcc = fc.rhof[c];
            const int nz1 = nz + 1;
            const float wx = g.cw_f[k] * ysj, wy = g.cw_f[nz1 + k];
            const float wyl = (g.ywall && j == 0) ? 0.f : wy * ytlo;
            const float wyh = (g.ywall && j + 1 == ny) ? 0.f : wy * ythi;
            float t = wx * face_beta_f(rcc, fc.rhof[rowoff + ip]) * (delta[rowoff + ip] - dc);
            t = fmaf(wx * face_beta_f(fc.rhof[rowoff + im], rcc), delta[rowoff + im] - dc, t);
            t = fmaf(wyh * face_beta_f(rcc, fc.rhof[rowp + i]), delta[rowp + i] - dc, t);
            t = fmaf(wyl * face_beta_f(rcc, fc.rhof[rowm + i]), delta[rowm + i] - dc, t);
            if (k + 1 < nz)
              t = fmaf(g.cw_f[2 * nz1 + k + 1] * ysj * face_beta_f(rcc, fc.rhof[c + plane]), delta[c + plane] - dc, t);
            if (k > 0)
              t = fmaf(g.cw_f[2 * nz1 + k] * ysj * face_beta_f(rcc, fc.rhof[c - plane]), delta[c - plane] - dc, t);
            ev = E[c] - t;
            E[c] = ev;
          } else {
            ep = b[c];
            if (!p_zero) {  // b - (sum_nb c_nb p_nb - diag p_c), seven FMAs
              ep = fma(fc.diag[c], p[c], ep);
              ep = fma(-fc.cx[rowoff + ip], p[rowoff + ip], ep);
              ep = fma(-fc.cx[c], p[rowoff + im], ep);
              ep = fma(-fc.cy[rowp + i], p[rowp + i], ep);
              ep = fma(-fc.cy[c], p[rowm + i], ep);
              if (k + 1 < nz) ep = fma(-fc.cz[c + plane], p[c + plane], ep);
              if (k > 0) ep = fma(-fc.cz[c], p[c - plane], ep);
            }
            if (sizeof(T) == sizeof(float)) {
              ev = narrow_f64(ep);
              if (E != nullptr) E[c] = ev;
            }
          }
          if (sizeof(T) == sizeof(float)) {
            const float e = ev * idzf_f;
            s2 = fmaf(e, e, (float)s2);
            s1 += fabsf(e);
            r = (T)(scale_rho ? (const_scale ? rt_f : fc.rhof[c]) * e : e);
          } else {
            const double e = ep * idzf;
            s2 = (T)fma(e, e, (double)s2);
            s1 += (T)fabs(e);
            r = (T)(scale_rho ? (const_scale ? rt : rho[c]) * e : e);
          }
        }
      }
      C2<T>& z = bufA[(size_t)(q >> 1) * seq_stride + i];
      if (q & 1) z.y = r; else z.x = r;
    }
  }
}

// The last steps of a residual kernel, by one warp of each block after its
// block's partial sums are in red[2 blk + {0, 1}] (written by lane 0): the last
// block of each group adds the group's pairs, the last group adds the groups'
// and runs the loop control.  Every sum runs in a fixed order.  No block waits
// for another.  (A kernel of one block reduced the sums before: 0.004 to
// 0.028 ms and a launch a pass.)
__device__ __forceinline__ void resid_ticket(const LoopCheck& ck, const double* red, unsigned blk, unsigned nblk) {
  constexpr unsigned full = 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  const unsigned ngrp = (nblk + kCheckGroup - 1) / kCheckGroup, grp = blk / kCheckGroup;
  const unsigned first = grp * kCheckGroup, n = min((unsigned)kCheckGroup, nblk - first);
  auto last_of = [&](unsigned* t, unsigned count) {  // lane 0's earlier writes are visible to the last one
    unsigned last = 0u;
    if (lane == 0u) {
      unsigned before;
      asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(before) : "l"(t) : "memory");
      last = before == count - 1u ? 1u : 0u;
      if (last) *t = 0u;  // nobody else arrives in this launch
    }
    last = __shfl_sync(full, last, 0);
    __syncwarp();
    return last != 0u;
  };
  auto sum2 = [&](const double* src, unsigned count, double& a, double& b) {
    a = b = 0.0;
    for (unsigned i = lane; i < count; i += 32u) {
      a += __ldcg(src + 2 * (size_t)i);
      b += __ldcg(src + 2 * (size_t)i + 1);
    }
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(full, a, o);
      b += __shfl_xor_sync(full, b, o);
    }
  };
  if (!last_of(ck.tick + 1 + grp, n)) return;
  double a, b;
  sum2(red + 2 * (size_t)first, n, a, b);
  if (ngrp == 1u) {
    if (lane == 0u) status_update(ck.st, a, b, ck.rtol, ck.maxit, ck.kexact);
    return;
  }
  if (lane == 0u) {
    ck.gsum[2 * (size_t)grp] = a;
    ck.gsum[2 * (size_t)grp + 1] = b;
  }
  if (!last_of(ck.tick, ngrp)) return;
  sum2(ck.gsum, ngrp, a, b);
  if (lane == 0u) status_update(ck.st, a, b, ck.rtol, ck.maxit, ck.kexact);
}

template <typename T, bool YS = false>
__device__ __forceinline__ void stage_resid_fftx(const Geo& g, const Faces& fc, const FftDesc& fx,
                                                 const C2<T>* __restrict__ twx,
                                                 const double* __restrict__ b,
                                                 const double* __restrict__ rho,
                                                 const double* __restrict__ p, int mode, int p_zero,
                                                 int scale_rho, C2<T>* __restrict__ spec,
                                                 double* __restrict__ red, int rpb, int blk,
                                                 bool need_exact, float* __restrict__ E,
                                                 const float* __restrict__ delta,
                                                 unsigned char* smem_raw, LoopCheck ck = LoopCheck{},
                                                 unsigned nblk = 0) {
  __shared__ double shred[64];
  const int nx = g.nx, ny = g.ny, nz = g.nz, nxh = g.nxh;
  const int nseq = rpb >> 1;
  C2<T>* bufA = reinterpret_cast<C2<T>*>(smem_raw);
  C2<T>* bufB = bufA + (size_t)nseq * nx;
  const int nrows = nz * ny;
  const long row0 = (long)blk * rpb;
  T s2 = (T)0, s1 = (T)0;
  // FP32 fast transform: buffer A, buffer B (written padded by the first
  // pass: fft_pad_elems), then the twiddle table
  constexpr bool F32 = std::is_same<T, float>::value;
  const int twb = nseq * nx + fft_pad_elems(nseq * nx);
  const bool fast = F32 && fft_smem_shape(nx, nseq);
  if constexpr (F32) {
    if (fast) load_twiddles_smem(twx, nx, twb);
  }
  resid_rows<T, YS>(g, fc, b, rho, p, mode, p_zero, scale_rho, row0, rpb, need_exact, E, delta, bufA, nx, s2, s1,
                    threadIdx.x, blockDim.x);
  if (mode != 0) {
    // block partial sums of e^2 and |e|: in the arithmetic's own precision
    // (FP32 shuffles on mixed plans: the FP64 pipe is the scarce one)
    block_sum2<T>(s2, s1, reinterpret_cast<T*>(shred));
    if (threadIdx.x == 0) {
      red[2 * (size_t)blk] = (double)s2;
      red[2 * (size_t)blk + 1] = (double)s1;
    }
  }
  __syncthreads();
  if (mode != 0 && ck.st != nullptr && threadIdx.x < 32) resid_ticket(ck, red, (unsigned)blk, nblk);
  const C2<T>* res = nullptr;
  if constexpr (F32) {
    if (fast)
      res = smem_f2() + fft_dispatch_smem<-1, false>(0, nseq * nx, twb, threadIdx.x, blockDim.x);
  }
  if (!fast) res = fft_dispatch<T, -1, false>(bufA, bufB, fx, nseq, 1, nx, twx, threadIdx.x, blockDim.x);
  // (q, kx) walked incrementally: no division by the odd nxh per element
  int q = threadIdx.x / nxh, kx = threadIdx.x - q * nxh;
  const int dq = blockDim.x / nxh, dkx = blockDim.x - dq * nxh;
  for (; q < nseq; q += dq, kx += dkx) {
    if (kx >= nxh) { kx -= nxh; ++q; if (q >= nseq) break; }
    const C2<T> Z = res[(size_t)q * nx + kx];
    const int km = (kx == 0) ? 0 : nx - kx;
    const C2<T> W = res[(size_t)q * nx + km];
    // 2 A = Z + conj W, 2 B = (Z - conj W)/i: the spectra are kept doubled,
    // the scale of the inverse x transform halves them (kSpecScale)
    C2<T> A, B;
    A.x = Z.x + W.x; A.y = Z.y - W.y;
    B.x = Z.y + W.y; B.y = W.x - Z.x;
    const long ra = row0 + 2 * q;
    if (ra < nrows) spec[(size_t)ra * nxh + kx] = A;
    if (ra + 1 < nrows) spec[(size_t)(ra + 1) * nxh + kx] = B;
  }
}

// Row order of the cosine transform through a complex FFT (Makhoul): the
// sequence v_r = x_{2r} (r < n/2), v_r = x_{2(n-1-r)+1} (r >= n/2), n even.
__device__ __forceinline__ int dct_row(int r, int n) { return (r < (n >> 1)) ? 2 * r : 2 * (n - 1 - r) + 1; }

template <typename T> __device__ __forceinline__ C2<T> cmulc(C2<T> a, C2<T> b) {  // a * conj(b)
  C2<T> r;
  r.x = a.x * b.x + a.y * b.y;
  r.y = a.y * b.x - a.x * b.y;
  return r;
}

// Complex transform along y of one z-plane tile of tx consecutive kx.  DCT:
// the cosine transform of walls in y (dct = exp(-i pi m / (2 ny))), in the
// steps of the persistent kernel below: the forward pass loads the rows in
// the order dct_row and finishes with X_r = (w_r Z_r + conj(w_r)
// Z_{ny-r}) / 2, the inverse pass pairs (Y_m, Y_{ny-m}) before its FFT and
// stores the rows back in the order dct_row.
template <typename T, int DIR, bool DCT = false>
__device__ __forceinline__ void stage_ffty(const Geo& g, const FftDesc& fy, const C2<T>* __restrict__ twy,
                                           C2<T>* __restrict__ spec, int tx, int bx, int bz,
                                           unsigned char* smem_raw, const C2<T>* __restrict__ dct = nullptr) {
  constexpr bool REORDER_IN = DCT && DIR < 0;
  constexpr bool REORDER_OUT = DCT && DIR > 0;
  const int ny = g.ny, nxh = g.nxh;
  C2<T>* bufA = reinterpret_cast<C2<T>*>(smem_raw);
  C2<T>* bufB = bufA + (size_t)ny * tx;
  const int kx0 = bx * tx;
  const size_t base = (size_t)bz * ny * nxh;
  const int lg_tx = 31 - __clz(tx);  // tx is a power of two (ffty_tile)
  constexpr bool F32 = std::is_same<T, float>::value;
  const int twb = ny * tx + fft_pad_elems(ny * tx);  // buffer B is written padded
  const bool fast = F32 && fft_smem_shape(ny, tx);
  if constexpr (F32) {
    if (fast) load_twiddles_smem(twy, ny, twb);
  }
  for (int t = threadIdx.x; t < ny * tx; t += blockDim.x) {
    const int r = t >> lg_tx, x = t & (tx - 1);
    const int y = REORDER_IN ? dct_row(r, ny) : r;
    C2<T> v; v.x = (T)0; v.y = (T)0;
    if (kx0 + x < nxh) v = spec[base + (size_t)y * nxh + kx0 + x];
    bufA[t] = v;
  }
  __syncthreads();
  if constexpr (REORDER_OUT) {
    // V_m and V_{ny-m} from the pair (Y_m, Y_{ny-m}), in place; V_0 = Y_0
    const int half = ny >> 1;
    for (int t = threadIdx.x; t < half * tx; t += blockDim.x) {
      const int m = 1 + (t >> lg_tx), x = t & (tx - 1);
      const C2<T> w = dct[m];
      const C2<T> a = bufA[m * tx + x], b = bufA[(ny - m) * tx + x];
      C2<T> d, e;  // a - i b, a + i b
      d.x = a.x + b.y; d.y = a.y - b.x;
      e.x = a.x - b.y; e.y = a.y + b.x;
      bufA[m * tx + x] = cmulc<T>(d, w);
      if (m != ny - m) bufA[(ny - m) * tx + x] = cmul<T>(e, w);
    }
    __syncthreads();
  }
  const C2<T>* res = nullptr;
  if constexpr (F32) {
    if (fast) res = smem_f2() + fft_dispatch_smem<DIR, true>(0, ny * tx, twb, threadIdx.x, blockDim.x);
  }
  if (!fast) res = fft_dispatch<T, DIR, true>(bufA, bufB, fy, tx, tx, 1, twy, threadIdx.x, blockDim.x);
  for (int t = threadIdx.x; t < ny * tx; t += blockDim.x) {
    const int r = t >> lg_tx, x = t & (tx - 1);
    if (kx0 + x >= nxh) continue;
    if constexpr (REORDER_IN) {
      // X_r = (w_r Z_r + conj(w_r) Z_{ny-r}) / 2
      const C2<T> w = dct[r];
      const C2<T> a = cmul<T>(res[t], w);
      const C2<T> b = cmulc<T>(res[(r == 0 ? 0 : ny - r) * tx + x], w);
      C2<T> o;
      o.x = (T)0.5 * (a.x + b.x);
      o.y = (T)0.5 * (a.y + b.y);
      spec[base + (size_t)r * nxh + kx0 + x] = o;
    } else {
      const int y = REORDER_OUT ? dct_row(r, ny) : r;
      spec[base + (size_t)y * nxh + kx0 + x] = res[t];
    }
  }
}

// Persistent y transform: each block walks the (kx tile, z plane) tiles
// with stride gridDim.x over three rotating shared buffers: while the
// current tile is transformed in two of them, the next tile is copied into
// the third by cp.async.
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;"
               :: "r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Lines of the spectrum [nz][ny][nxh] that a persistent transform walks.
// AXIS = 0: along y (length ny, element stride nxh), one tile per (z plane,
// kx tile).  AXIS = 1: along z (length nz, stride ny nxh), one tile per
// (ky, kx tile).
template <int AXIS> struct Lines {
  int n;             // transform length
  size_t rstride;    // elements between consecutive entries of a line
  size_t ostride;    // elements between consecutive outer indices
  __device__ __forceinline__ explicit Lines(const Geo& g)
      : n(AXIS ? g.nz : g.ny), rstride(AXIS ? (size_t)g.ny * g.nxh : (size_t)g.nxh),
        ostride(AXIS ? (size_t)g.nxh : (size_t)g.ny * g.nxh) {}
};

// REORDER: shared row r receives global row dct_row(r) (forward cosine
// transform); otherwise row r receives row r.
template <typename T, bool REORDER = false, int AXIS = 0>
__device__ __forceinline__ void ffty_issue_tile(const Geo& g, const C2<T>* __restrict__ spec, int tx, int ntx,
                                                long long tile, C2<T>* buf) {
  const Lines<AXIS> ln(g);
  const int n = ln.n, nxh = g.nxh;
  const int bz = (int)(tile / ntx), bx = (int)(tile - (long long)bz * ntx);
  const int kx0 = bx * tx;
  const size_t base = (size_t)bz * ln.ostride;
  const int lg_tx = 31 - __clz(tx);  // tx is a power of two (ffty_tile)
  for (int t = threadIdx.x; t < n * tx; t += blockDim.x) {
    const int r = t >> lg_tx, x = t & (tx - 1);
    const int y = REORDER ? dct_row(r, n) : r;
    if (kx0 + x < nxh) {
      const size_t at = base + (size_t)y * ln.rstride + kx0 + x;
      if (sizeof(C2<T>) == 8) cp_async8(&buf[t], &spec[at]);
      else {
        cp_async8(&buf[t], &spec[at]);
        cp_async8(reinterpret_cast<char*>(&buf[t]) + 8, reinterpret_cast<const char*>(&spec[at]) + 8);
      }
    } else {
      buf[t].x = (T)0;
      buf[t].y = (T)0;
    }
  }
  cp_async_commit();
}


// Persistent y transform.  DCT = false: complex DFT along y (periodic y).
// DCT = true (walls in y): the eigenbasis of the Neumann second difference
// on cell centres, X_m = sum_j x_j cos(pi m (2j + 1) / (2 ny)), computed
// with one complex FFT of length ny (Makhoul's reordering) and the twiddles
// w_m = exp(-i pi m / (2 ny)) of `dct`:
//   forward:  Z = FFT(x reordered by dct_row);
//             X_m = (w_m Z_m + conj(w_m) Z_{ny-m}) / 2   (Z_ny = Z_0);
//   inverse:  V_m = conj(w_m) (Y_m - i Y_{ny-m})          (Y_ny = 0);
//             x_{dct_row(r)} = (IFFT(V))_r, unnormalised like the periodic
//             inverse (the caller's 1/(nx ny) completes both).
// The transform acts on real and imaginary parts alike, so the complex
// x-spectrum goes through unchanged.
// AXIS = 1 runs the same transforms along z (uniform walls in z: the z
// eigenbasis is the same cosine basis).  Its forward pass also divides by
// the eigenvalue: X / (nz (lambda_x + lambda_y + lambda_z)), with the
// singular (0, 0, 0) mode set to 0 (zero mean), so forward + inverse is the
// whole z solve.
template <typename T, int DIR, bool DCT = false, int AXIS = 0>
__device__ __forceinline__ void stage_ffty_persistent(const Geo& g, const FftDesc& fy,
                                                      const C2<T>* __restrict__ twy, C2<T>* spec, int tx,
                                                      long long ntiles, long long first, long long stride,
                                                      unsigned char* smem_raw,
                                                      const C2<T>* __restrict__ dct = nullptr,
                                                      ZDivide zd = ZDivide{}) {
  constexpr bool REORDER_IN = DCT && DIR < 0;
  constexpr bool REORDER_OUT = DCT && DIR > 0;
  const Lines<AXIS> ln(g);
  const int ny = ln.n, nxh = g.nxh;  // ny: the transform length (ny, or nz for AXIS = 1)
  const int ntx = (nxh + tx - 1) / tx;
  const int tsz = ny * tx;
  const int lg_tx = 31 - __clz(tx);  // tx is a power of two (ffty_tile)
  C2<T>* X0 = reinterpret_cast<C2<T>*>(smem_raw);
  // element offsets of the three buffers, rotated (no pointer array: the
  // transforms then address shared memory directly)
  // FP32 fast path: Q, the scratch buffer of the transform, is written
  // padded by its first pass and holds fft_pad_elems(tsz) elements, then the
  // twiddle table follows; otherwise three plain buffers.  L and F (tsz
  // each) rotate.  The launcher sizes shared memory for the same layout.
  constexpr bool F32 = std::is_same<T, float>::value;
  const int qsz = F32 ? fft_pad_elems(tsz) : tsz;
  int L = 0, Q = tsz, F = tsz + qsz;
  const int twb = 2 * tsz + qsz;
  const bool fast = F32 && fft_smem_shape(ny, tx);
  if constexpr (F32) {
    if (fast) load_twiddles_smem(twy, ny, twb);
  }
  if (first < ntiles) ffty_issue_tile<T, REORDER_IN, AXIS>(g, spec, tx, ntx, first, X0 + L);
  for (long long tile = first; tile < ntiles; tile += stride) {
    cp_async_wait_all();
    __syncthreads();
    const long long next = tile + stride;
    if (next < ntiles) ffty_issue_tile<T, REORDER_IN, AXIS>(g, spec, tx, ntx, next, X0 + F);
    if constexpr (REORDER_OUT) {
      // V_m and V_{ny-m} from the pair (Y_m, Y_{ny-m}), in place; V_0 = Y_0.
      C2<T>* Y = X0 + L;
      const int half = ny >> 1;
      for (int t = threadIdx.x; t < half * tx; t += blockDim.x) {
        const int m = 1 + (t >> lg_tx), x = t & (tx - 1);
        const C2<T> w = dct[m];
        const C2<T> a = Y[m * tx + x], b = Y[(ny - m) * tx + x];
        C2<T> d, e;  // a - i b, a + i b
        d.x = a.x + b.y; d.y = a.y - b.x;
        e.x = a.x - b.y; e.y = a.y + b.x;
        if (m == ny - m) {
          Y[m * tx + x] = cmulc<T>(d, w);
        } else {
          Y[m * tx + x] = cmulc<T>(d, w);
          Y[(ny - m) * tx + x] = cmul<T>(e, w);
        }
      }
      __syncthreads();
    }
    const C2<T>* res = nullptr;
    if constexpr (F32) {
      if (fast) res = smem_f2() + fft_dispatch_smem<DIR, true>(L, Q, twb, threadIdx.x, blockDim.x);
    }
    if (!fast) res = fft_dispatch<T, DIR, true>(X0 + L, X0 + Q, fy, tx, tx, 1, twy, threadIdx.x, blockDim.x);
    const int bz = (int)(tile / ntx), bx = (int)(tile - (long long)bz * ntx);
    const int kx0 = bx * tx;
    const size_t base = (size_t)bz * ln.ostride;
    for (int t = threadIdx.x; t < ny * tx; t += blockDim.x) {
      const int r = t >> lg_tx, x = t & (tx - 1);
      if (kx0 + x >= nxh) continue;
      if constexpr (REORDER_IN) {
        // X_r = (w_r Z_r + conj(w_r) Z_{ny-r}) / 2
        const C2<T> w = dct[r];
        const C2<T> a = cmul<T>(res[t], w);
        const C2<T> b = cmulc<T>(res[(r == 0 ? 0 : ny - r) * tx + x], w);
        T h = (T)0.5;
        if constexpr (AXIS == 1) {
          // bz is ky here; the (0, 0, 0) mode is the pinned mean
          const double lam = zd.lamx[kx0 + x] + zd.lamy[bz] + zd.lamz[r];
          h = (kx0 + x == 0 && bz == 0 && r == 0) ? (T)0 : (T)(0.5 / ((double)ny * lam));
        }
        C2<T> o;
        o.x = h * (a.x + b.x);
        o.y = h * (a.y + b.y);
        spec[base + (size_t)r * ln.rstride + kx0 + x] = o;
      } else {
        const int y = REORDER_OUT ? dct_row(r, ny) : r;
        spec[base + (size_t)y * ln.rstride + kx0 + x] = res[t];
      }
    }
    __syncthreads();
    // rotate: the prefetched buffer holds the next tile; the other two are free
    const int nl = F;
    F = L;
    L = nl;
  }
}

// Per-column Thomas solve of (L_z + lambda_x + lambda_y) x = f with the
// inverse pivots precomputed at plan time.  Column (0, 0) is singular: its
// right-hand side loses its dzf-weighted mean (compatibility) and its last
// unknown is pinned (inverse pivot 0); the pressure gauge is fixed later.
// Loads run PF levels ahead of the recurrence.
template <bool ZERO_MODE>
__device__ __forceinline__ void thomas_column(const Geo& g, const double* __restrict__ invd,
                                              double2* spec, double2* ybuf, size_t col, size_t stride) {
  constexpr int PF = 4;
  const int nz = g.nz;
  double mr = 0.0, mi = 0.0;
  if (ZERO_MODE) {
    for (int k = 0; k < nz; ++k) {
      const double2 f = spec[(size_t)k * stride + col];
      mr += g.dzf[k] * f.x;
      mi += g.dzf[k] * f.y;
    }
    mr /= g.lz;
    mi /= g.lz;
  }
  // forward sweep: y_k = f_k - (a_k / d_{k-1}) y_{k-1}
  double2 fq[PF];
  double dq[PF];
#pragma unroll
  for (int u = 0; u < PF; ++u) {
    const int k = u < nz ? u : nz - 1;
    fq[u] = spec[(size_t)k * stride + col];
    dq[u] = invd[(size_t)k * stride + col];
  }
  double yr = 0.0, yi = 0.0, dprev = 0.0;
  for (int k0 = 0; k0 < nz; k0 += PF) {
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      const int k = k0 + u;
      if (k < nz) {
        const double2 f = fq[u];
        const double d = dq[u];
        const int kn = k + PF < nz ? k + PF : nz - 1;
        fq[u] = spec[(size_t)kn * stride + col];
        dq[u] = invd[(size_t)kn * stride + col];
        const double m = (k == 0) ? 0.0 : g.za[k] * dprev;
        yr = (f.x - mr) - m * yr;
        yi = (f.y - mi) - m * yi;
        ybuf[(size_t)k * stride + col] = make_double2(yr, yi);
        dprev = d;
      }
    }
  }
  // back substitution: x_k = (y_k - c_k x_{k+1}) / d_k
  double xr = yr * dprev, xi = yi * dprev;
  spec[(size_t)(nz - 1) * stride + col] = make_double2(xr, xi);
  double2 yq[PF];
#pragma unroll
  for (int u = 0; u < PF; ++u) {
    const int k = nz - 2 - u >= 0 ? nz - 2 - u : 0;
    yq[u] = ybuf[(size_t)k * stride + col];
    dq[u] = invd[(size_t)k * stride + col];
  }
  for (int k0 = nz - 2; k0 >= 0; k0 -= PF) {
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      const int k = k0 - u;
      if (k >= 0) {
        const double2 y = yq[u];
        const double d = dq[u];
        const int kn = k - PF >= 0 ? k - PF : 0;
        yq[u] = ybuf[(size_t)kn * stride + col];
        dq[u] = invd[(size_t)kn * stride + col];
        const double c = g.zc[k];
        xr = (y.x - c * xr) * d;
        xi = (y.y - c * xi) * d;
        spec[(size_t)k * stride + col] = make_double2(xr, xi);
      }
    }
  }
}

// One ill-conditioned column of a mixed plan, solved by a whole warp in
// FP64.  Both sweeps of the Thomas elimination are first-order affine
// recurrences,
//   forward   y_k = -m_k y_{k-1} + f_k                (y_{-1} = 0),
//   backward  x_k = -c_k d_k x_{k+1} + d_k y_k        (x_{nz-1} = d_{nz-1} y_{nz-1}),
// so each lane composes the maps of its R = ceil(nz/32) consecutive rows, a
// shuffle scan combines the lanes' maps, and each lane replays its rows from
// the value entering its segment.  The values stay FP32 in memory (the
// intermediate y too); the recurrences run in
// FP64.  Column 0 (the singular (0, 0) system, its last pivot pinned) first
// loses its dzf-weighted z mean.
__device__ __forceinline__ void tridiag_col_warp64(const Geo& g, const double* __restrict__ mtab,
                                                   const double* __restrict__ invd, float2* spec,
                                                   size_t col, size_t ncol) {
  const int lane = threadIdx.x & 31;
  const int nz = g.nz;
  const int R = (nz + 31) >> 5;
  const int k0 = lane * R < nz ? lane * R : nz;
  const int k1 = k0 + R < nz ? k0 + R : nz;
  auto at = [&](int k) { return (size_t)k * ncol + col; };
  double m0x = 0.0, m0y = 0.0;
  if (col == 0) {
    double sx = 0.0, sy = 0.0;
    for (int k = k0; k < k1; ++k) {
      const float2 v = spec[at(k)];
      sx += g.dzf[k] * widen_f32(v.x);
      sy += g.dzf[k] * widen_f32(v.y);
    }
    for (int o = 16; o > 0; o >>= 1) {
      sx += __shfl_xor_sync(0xffffffffu, sx, o);
      sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    m0x = sx / g.lz;
    m0y = sy / g.lz;
  }
  // forward: compose y -> a y + b over the lane's rows, then scan the lanes
  double A = 1.0, Bx = 0.0, By = 0.0;
  for (int k = k0; k < k1; ++k) {
    const double a = -mtab[at(k)];
    const float2 f = spec[at(k)];
    Bx = fma(a, Bx, widen_f32(f.x) - m0x);
    By = fma(a, By, widen_f32(f.y) - m0y);
    A *= a;
  }
  for (int d = 1; d < 32; d <<= 1) {  // inclusive scan, earlier lanes' maps applied first
    const double Ap = __shfl_up_sync(0xffffffffu, A, d);
    const double Bxp = __shfl_up_sync(0xffffffffu, Bx, d);
    const double Byp = __shfl_up_sync(0xffffffffu, By, d);
    if (lane >= d) {
      Bx = fma(A, Bxp, Bx);
      By = fma(A, Byp, By);
      A *= Ap;
    }
  }
  double yx = __shfl_up_sync(0xffffffffu, Bx, 1), yy = __shfl_up_sync(0xffffffffu, By, 1);
  if (lane == 0) { yx = 0.0; yy = 0.0; }
  for (int k = k0; k < k1; ++k) {
    const double a = -mtab[at(k)];
    const float2 f = spec[at(k)];
    yx = fma(a, yx, widen_f32(f.x) - m0x);
    yy = fma(a, yy, widen_f32(f.y) - m0y);
    spec[at(k)] = make_float2(narrow_f64(yx), narrow_f64(yy));
  }
  __syncwarp();
  // backward: maps x_{k+1} -> x_k over the lane's rows from the top down
  auto row_map = [&](int k, double& a, double& bx, double& by) {
    const float2 yv = spec[at(k)];
    const double d = invd[at(k)];
    a = (k == nz - 1) ? 0.0 : -g.zc[k] * d;
    bx = d * widen_f32(yv.x);
    by = d * widen_f32(yv.y);
  };
  A = 1.0; Bx = 0.0; By = 0.0;
  for (int k = k1 - 1; k >= k0; --k) {
    double a, bx, by;
    row_map(k, a, bx, by);
    Bx = fma(a, Bx, bx);
    By = fma(a, By, by);
    A *= a;
  }
  for (int d = 1; d < 32; d <<= 1) {  // inclusive scan, later lanes' maps applied first
    const double Ap = __shfl_down_sync(0xffffffffu, A, d);
    const double Bxp = __shfl_down_sync(0xffffffffu, Bx, d);
    const double Byp = __shfl_down_sync(0xffffffffu, By, d);
    if (lane + d < 32) {
      Bx = fma(A, Bxp, Bx);
      By = fma(A, Byp, By);
      A *= Ap;
    }
  }
  double xx = __shfl_down_sync(0xffffffffu, Bx, 1), xy = __shfl_down_sync(0xffffffffu, By, 1);
  if (lane == 31) { xx = 0.0; xy = 0.0; }
  // every lane reads its own rows' y before any lane overwrites them
  for (int k = k1 - 1; k >= k0; --k) {
    double a, bx, by;
    row_map(k, a, bx, by);
    xx = fma(a, xx, bx);
    xy = fma(a, xy, by);
    spec[at(k)] = make_float2(narrow_f64(xx), narrow_f64(xy));
  }
}

// Mixed plans, one thread per (kx, ky) column holding both components, in
// FP32 with FP32 tables.  Only the well-conditioned columns (TriF32) take
// this path; column 0 and the other ill-conditioned columns are left to
// tridiag_col_warp64.
__device__ __forceinline__ void stage_tridiag_col32(const Geo& g, const TriF32& f, float2* spec, size_t col,
                                                    unsigned char* smem) {
  const size_t ncol = (size_t)g.ny * g.nxh;
  if (col >= ncol) return;
  const int j = (int)((unsigned)col / (unsigned)g.nxh);
  const int kx = (int)(col - (size_t)j * g.nxh);
  if (col == 0 || fabs(f.lamx[kx] + f.lamy[j]) < f.thr) return;
  const ZForm32 form{f.mtab, nullptr, f.invd};
  zsweep<ZForm32, false>(form, spec + col, ncol, col, ncol, g.nz, f.zc, smem, 0.0, 0.0);
}

// Block b of the mixed z solve: the first nblk_low blocks give one warp to
// each ill-conditioned column of the list (scheduled first: their chains are
// the longest), the rest one thread to each column.  Block-uniform branch.
__device__ __forceinline__ void stage_tridiag_mixed(const Geo& g, const double* __restrict__ mtab,
                                                    const double* __restrict__ invd, const TriF32& f,
                                                    float2* spec, int b, unsigned char* smem) {
  constexpr int kWarps = kZThreads / 32;
  const int nblk_low = (f.nlow + kWarps - 1) / kWarps;
  if (b < nblk_low) {
    const int w = b * kWarps + (threadIdx.x >> 5);
    if (w < f.nlow) tridiag_col_warp64(g, mtab, invd, spec, (size_t)f.low[w], (size_t)g.ny * g.nxh);
    return;
  }
  stage_tridiag_col32(g, f, spec, (size_t)(b - nblk_low) * kZThreads + threadIdx.x, smem);
}

// Inverse x transform of two half spectra per complex sequence, then
// p = scale * z (p_zero) or p += scale * z.  The p values a thread updates
// are loaded before the transform so their latency overlaps it.  delta (if
// not null) receives the increment scale * z in the precision T.
//
// Mixed path (sdelta not null): p is only brought up to date where an
// exact residual needs it.  sdelta holds the FP32 sum of the increments
// since p was last updated:
//   fold  (the next residual is exact): p += sdelta + increment (FP64);
//   else: sdelta = increment (fresh: p was updated last pass) or
//         sdelta += increment.
// With fresh set, fold ignores sdelta.
// Update modes of the inverse x stage (compile-time, so each pass runs only
// its own arithmetic).
enum InvMode { kInvPlain = 0, kInvFold = 1, kInvFoldFresh = 2, kInvFresh = 3, kInvAccum = 4 };

template <typename T, int MODE>
__device__ __forceinline__ void stage_fftx_inv_m(const Geo& g, const FftDesc& fx,
                                                 const C2<T>* __restrict__ twx,
                                                 const C2<T>* __restrict__ spec, double scale,
                                                 double* __restrict__ p, int p_zero, int rpb, int blk,
                                                 T* __restrict__ delta, float* __restrict__ sdelta,
                                                 unsigned char* smem_raw) {
  const int nx = g.nx, ny = g.ny, nz = g.nz, nxh = g.nxh;
  const int nseq = rpb >> 1;
  const float scale_f = (float)scale;
  C2<T>* bufA = reinterpret_cast<C2<T>*>(smem_raw);
  C2<T>* bufB = bufA + (size_t)nseq * nx;
  const long nrows = (long)nz * ny;
  const long row0 = (long)blk * rpb;
  const bool even = (nx & 1) == 0;
  const int nout = rpb * nx;
  const int lgx = ((nx & (nx - 1)) == 0) ? 31 - __clz(nx) : -1;
  const bool need_p = !p_zero && MODE <= kInvFoldFresh;            // p is read
  constexpr bool need_s = MODE == kInvFold || MODE == kInvAccum;  // sdelta is read
  // p is prefetched in the plain mode of FP64 plans (every pass); the fold
  // passes of mixed plans (one in forty) read it where it is used, which keeps
  // their registers within the other modes' budget
  const bool pre_p = need_p && MODE == kInvPlain && sizeof(T) == sizeof(double);
  constexpr bool F32 = std::is_same<T, float>::value;
  const int twb = nseq * nx + fft_pad_elems(nseq * nx);  // buffer B is written padded
  const bool fast = F32 && fft_smem_shape(nx, nseq);
  if constexpr (F32) {
    if (fast) load_twiddles_smem(twx, nx, twb);
  }
  auto split = [&](int t, int& q, int& i) {
    if (lgx >= 0) { q = t >> lgx; i = t & (nx - 1); }
    else { q = t / nx; i = t - q * nx; }
  };
  // one output value: zv = unscaled inverse transform at cell c
  auto emit = [&](size_t c, T zv, double pv, float sv) {
    const float inc_f = scale_f * (float)zv;
    if constexpr (MODE <= kInvFoldFresh) {
      const double zd = (sizeof(T) == sizeof(float)) ? widen_f32((float)zv) : (double)zv;
      if constexpr (MODE == kInvFold) p[c] = fma(scale, zd, pv + widen_f32(sv));
      else p[c] = fma(scale, zd, pv);
      if (delta != nullptr) delta[c] = (sizeof(T) == sizeof(float)) ? (T)inc_f : (T)(scale * zd);
    } else {
      sdelta[c] = (MODE == kInvAccum) ? sv + inc_f : inc_f;
      if (delta != nullptr) delta[c] = (T)inc_f;
    }
  };
  constexpr int NP = kPrefetchInv;
  double pv[NP];
  float sv[NP];
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    const int t = threadIdx.x + u * blockDim.x;
    int q, i;
    split(t, q, i);
    pv[u] = 0.0;
    sv[u] = 0.f;
    const bool in = t < nout && row0 + q < nrows;
    if (pre_p && in) pv[u] = p[(size_t)(row0 + q) * nx + i];
    if (need_s && in) sv[u] = sdelta[(size_t)(row0 + q) * nx + i];
  }
  // Z = A + i B from the two half spectra; each stored coefficient m also
  // gives its mirror nx - m (conjugates), so it is loaded once.  (q, m) is
  // walked incrementally over the nseq x nxh stored coefficients.
  {
    int q = threadIdx.x / nxh, m = threadIdx.x - q * nxh;
    const int dq = blockDim.x / nxh, dm = blockDim.x - dq * nxh;
    for (; q < nseq; q += dq, m += dm) {
      if (m >= nxh) { m -= nxh; ++q; if (q >= nseq) break; }
      const long ra = row0 + 2 * q;
      C2<T> A, B;
      A.x = A.y = B.x = B.y = (T)0;
      if (ra < nrows) A = spec[(size_t)ra * nxh + m];
      if (ra + 1 < nrows) B = spec[(size_t)(ra + 1) * nxh + m];
      C2<T>* row = bufA + (size_t)q * nx;
      if (m == 0 || (even && m == nx / 2)) {
        C2<T> Z;
        Z.x = A.x;
        Z.y = B.x;
        row[m] = Z;
      } else {
        C2<T> Z, Zm;
        Z.x = A.x - B.y;
        Z.y = A.y + B.x;
        Zm.x = A.x + B.y;   // mirror: A, B conjugated
        Zm.y = B.x - A.y;
        row[m] = Z;
        if (m < nx - m) row[nx - m] = Zm;
      }
    }
  }
  __syncthreads();
  const C2<T>* res = nullptr;
  if constexpr (F32) {
    if (fast) res = smem_f2() + fft_dispatch_smem<1, false>(0, nseq * nx, twb, threadIdx.x, blockDim.x);
  }
  if (!fast) res = fft_dispatch<T, 1, false>(bufA, bufB, fx, nseq, 1, nx, twx, threadIdx.x, blockDim.x);
#pragma unroll
  for (int u = 0; u < NP; ++u) {
    const int t = threadIdx.x + u * blockDim.x;
    int q, i;
    split(t, q, i);
    const long row = row0 + q;
    if (t < nout && row < nrows) {
      const C2<T> z = res[(size_t)(q >> 1) * nx + i];
      const size_t c = (size_t)row * nx + i;
      emit(c, (q & 1) ? z.y : z.x, pre_p ? pv[u] : (need_p ? p[c] : 0.0), sv[u]);
    }
  }
  for (int t = threadIdx.x + NP * blockDim.x; t < nout; t += blockDim.x) {  // beyond the prefetch
    int q, i;
    split(t, q, i);
    const long row = row0 + q;
    if (row < nrows) {
      const C2<T> z = res[(size_t)(q >> 1) * nx + i];
      const size_t c = (size_t)row * nx + i;
      emit(c, (q & 1) ? z.y : z.x, need_p ? p[c] : 0.0, need_s ? sdelta[c] : 0.f);
    }
  }
}

// Mode dispatch (block-uniform): sdelta null -> plain update of p.
template <typename T>
__device__ __forceinline__ void stage_fftx_inv(const Geo& g, const FftDesc& fx, const C2<T>* __restrict__ twx,
                                               const C2<T>* __restrict__ spec, double scale,
                                               double* __restrict__ p, int p_zero, int rpb, int blk,
                                               T* __restrict__ delta, float* __restrict__ sdelta,
                                               bool fold, bool fresh, unsigned char* smem_raw) {
  if (sizeof(T) == sizeof(double) || sdelta == nullptr) {  // FP64 plans: plain only
    stage_fftx_inv_m<T, kInvPlain>(g, fx, twx, spec, scale, p, p_zero, rpb, blk, delta, sdelta, smem_raw);
    return;
  }
  if constexpr (sizeof(T) == sizeof(double)) return;
  if (fold && !fresh)
    stage_fftx_inv_m<T, kInvFold>(g, fx, twx, spec, scale, p, p_zero, rpb, blk, delta, sdelta, smem_raw);
  else if (fold)
    stage_fftx_inv_m<T, kInvFoldFresh>(g, fx, twx, spec, scale, p, p_zero, rpb, blk, delta, sdelta, smem_raw);
  else if (fresh)
    stage_fftx_inv_m<T, kInvFresh>(g, fx, twx, spec, scale, p, p_zero, rpb, blk, delta, sdelta, smem_raw);
  else
    stage_fftx_inv_m<T, kInvAccum>(g, fx, twx, spec, scale, p, p_zero, rpb, blk, delta, sdelta, smem_raw);
}

}  // namespace pp
