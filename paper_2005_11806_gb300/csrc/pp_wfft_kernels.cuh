// The x and y kernels of a pass for the lengths of PP_WFFT_LENGTHS
// (pp_wfft.cuh); the launchers choose them by length.
#pragma once
#include "pp_r512.cuh"
#include "pp_stages.cuh"
#include "pp_wfft.cuh"

namespace pp {

// Forward transform of a warp's lines in place, natural order in and out
// (buf: LW lines LS entries apart).
template <class W, typename T>
__device__ __forceinline__ void wfft_lines(C2<T>* buf, const C2<T>* tw, int lane) {
  const int l = lane & (W::L - 1);
  C2<T>* line = buf + (lane / W::L) * W::LS;
  {
    C2<T> v[W::U1][W::R1];
#pragma unroll
    for (int u = 0; u < W::U1; ++u) {
      const int bb = l + u * W::L;
      if (W::R2 % W::L == 0 || bb < W::R2) {
#pragma unroll
        for (int a = 0; a < W::R1; ++a) v[u][a] = line[W::R2 * a + bb];
        wfft_stage1<W, T, -1>(v[u], tw, bb);
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < W::U1; ++u) {
      const int bb = l + u * W::L;
      if (W::R2 % W::L == 0 || bb < W::R2) {
#pragma unroll
        for (int c = 0; c < W::R1; ++c) line[c * W::S + bb] = v[u][c];
      }
    }
  }
  __syncwarp();
  {
    C2<T> v[W::U2][W::R2];
#pragma unroll
    for (int u = 0; u < W::U2; ++u) {
      const int c = l + u * W::L;
      if (W::R1 % W::L == 0 || c < W::R1) {
#pragma unroll
        for (int bb = 0; bb < W::R2; ++bb) v[u][bb] = line[c * W::S + bb];
        Dft<T, -1, W::R2>::run(v[u]);
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < W::U2; ++u) {
      const int c = l + u * W::L;
      if (W::R1 % W::L == 0 || c < W::R1) {
#pragma unroll
        for (int d = 0; d < W::R2; ++d) line[c + W::R1 * d] = v[u][d];
      }
    }
  }
  __syncwarp();
}

// The same for one line of 512 entries: three 8-point stages, two transforms
// a thread (thread j of pp_r512.cuh is (lane, u): j = lane + 32 u).
template <int DIR>
__device__ __forceinline__ void wfft512_line(float2* line, const float2* tw, int lane) {
  float2 v[2][8];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int j = lane + 32 * u;
#pragma unroll
    for (int a = 0; a < 8; ++a) v[u][a] = line[64 * a + j];
    Dft<float, DIR, 8>::run(v[u]);
    r512_twiddle8<DIR>(v[u], tw, 64, j);
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int c = 0; c < 8; ++c) line[c * 72 + lane + 32 * u] = v[u][c];
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int j = lane + 32 * u, c = j >> 3, f = j & 7;
#pragma unroll
    for (int e = 0; e < 8; ++e) v[u][e] = line[c * 72 + 8 * e + f];
    Dft<float, DIR, 8>::run(v[u]);
    r512_twiddle8<DIR>(v[u], tw + 512, 8, f);
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int j = lane + 32 * u, c = j >> 3, f = j & 7;
#pragma unroll
    for (int gg = 0; gg < 8; ++gg) line[c * 73 + gg * 8 + f] = v[u][gg];
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int j = lane + 32 * u, c = j & 7, gg = j >> 3;
#pragma unroll
    for (int f = 0; f < 8; ++f) v[u][f] = line[c * 73 + gg * 8 + f];
    Dft<float, DIR, 8>::run(v[u]);
  }
  __syncwarp();
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int h = 0; h < 8; ++h) line[lane + 32 * u + 64 * h] = v[u][h];
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Residual and forward real x transform (stage_resid_fftx), a warp at a time:
// a warp computes the rows of its own LW sequences (2 LW rows) into its own
// shared buffer, transforms and separates them, with warp barriers only, so
// the stencil's loads of one warp overlap the transforms of the others.  The
// block kernel (stage_resid_fftx) meets a block barrier after each of its
// steps, and its smallest unit (2048 values) leaves most SMs without work on
// small grids.  FP32: bound by the latency of its global loads (half of the
// stalls, issue 49 % busy, DRAM 43 % at 256^3); FP64: by the FP64 pipe.  Block
// kernel and loop-control kernel -> this, ms: mixed 256^3 0.114 -> 0.091, mixed
// 512^3 0.805 -> 0.644, mixed 192 x 160 x 144 0.046 -> 0.029, FP64 128^3 0.142
// -> 0.106, FP64 32^3 0.023 -> 0.016.  Measured and dropped: prefetching a later
// block's rows into L2 (256^3: 0.106); four and three blocks an SM (192 x 160 x
// 144 0.034, 0.038), six (256^3 gains 3 %, 192 x 160 x 144 loses 8 %).
// red: one pair of partial sums per block.
template <typename T, bool YS, int N>
__device__ __forceinline__ void resid_w_body(const Geo& g, const Faces& fc, const C2<T>* __restrict__ twx,
                                             const double* __restrict__ b, const double* __restrict__ rho,
                                             const double* __restrict__ p, int mode, int p_zero, int scale_rho,
                                             C2<T>* __restrict__ spec, double* __restrict__ red, bool need_exact,
                                             float* __restrict__ E, const float* __restrict__ delta, unsigned blk,
                                             unsigned char* smem_raw, const LoopCheck& ck, unsigned nblk) {
  using W = WPlan<N>;
  __shared__ T shs[16];  // the warps' sums
  C2<T>* tw = reinterpret_cast<C2<T>*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  C2<T>* buf = tw + W::TW + (size_t)warp * W::LW * W::LS;
  if constexpr (N == 512) r512_load_twiddles(tw, twx);
  else wfft_load_twiddles<W, T>(tw, twx);
  const unsigned gw = blk * (blockDim.x >> 5) + warp;
  const int nrows = g.nz * g.ny;
  const int nxh = N / 2 + 1;
  const long row0 = (long)gw * (2 * W::LW);
  T s2 = (T)0, s1 = (T)0;
  if (row0 < nrows)
    resid_rows<T, YS>(g, fc, b, rho, p, mode, p_zero, scale_rho, row0, 2 * W::LW, need_exact, E, delta, buf, W::LS,
                      s2, s1, lane, 32);
  if (mode != 0) {
    for (int o = 16; o > 0; o >>= 1) {
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (lane == 0) {
      shs[warp] = s2;
      shs[8 + warp] = s1;
    }
  }
  __syncthreads();  // twiddles, the warps' sums
  if (mode != 0 && warp == 0) {
    if (lane == 0) {
      T a = (T)0, c = (T)0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        a += shs[w];
        c += shs[8 + w];
      }
      red[2 * (size_t)blk] = (double)a;
      red[2 * (size_t)blk + 1] = (double)c;
    }
    // (at the end of the block instead: the same time)
    if (ck.st != nullptr) resid_ticket(ck, red, blk, nblk);
  }
  if (row0 >= nrows) return;
  if constexpr (N == 512) wfft512_line<-1>(buf, tw, lane);
  else wfft_lines<W, T>(buf, tw, lane);
  // 2 A = Z + conj W, 2 B = (Z - conj W)/i of the two rows of each line (kSpecScale)
#pragma unroll
  for (int q = 0; q < W::LW; ++q) {
    const C2<T>* Zl = buf + q * W::LS;
    const long ra = row0 + 2 * q;
    if (ra >= nrows) break;
    C2<T>* sa = spec + (size_t)ra * nxh;
    for (int kx = lane; kx < nxh; kx += 32) {
      const C2<T> Z = Zl[kx], Wc = Zl[kx == 0 ? 0 : N - kx];
      sa[kx] = mk<T>(Z.x + Wc.x, Z.y - Wc.y);
      if (ra + 1 < nrows) sa[nxh + kx] = mk<T>(Z.y + Wc.y, Wc.x - Z.x);
    }
  }
}

template <typename T, bool YS, int N>
__global__ void __launch_bounds__(128, sizeof(T) == sizeof(float) ? 5 : 3) k_resid_w(
    Geo g, Faces fc, const C2<T>* __restrict__ twx, const double* __restrict__ b, const double* __restrict__ rho,
    const double* __restrict__ p, int mode, int p_zero, int scale_rho, C2<T>* __restrict__ spec,
    double* __restrict__ red, const DevStatus* st, float* __restrict__ E, const float* __restrict__ delta,
    LoopCheck ck) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  resid_w_body<T, YS, N>(g, fc, twx, b, rho, p, mode, p_zero, scale_rho, spec, red,
                         (st == nullptr) || st->need_exact, E, delta, blockIdx.x, smem_raw, ck, gridDim.x);
}

// ---------------------------------------------------------------------------
// Inverse x transform and update of p (stage_fftx_inv and its modes), a warp
// at a time: the half spectra go from global memory to registers, and the
// increments from registers to p, sdelta and delta; one exchange through
// shared memory in between.  Bound by global memory latency (FP32, 256^3: 62 %
// of the DRAM rate) or the FP64 pipe.  Block kernel -> this, ms: mixed 256^3
// 0.088 -> 0.043, mixed 192 x 160 x 144 0.044 -> 0.013, FP64 128^3 0.069 ->
// 0.057.
//   lazy (mixed plans): p is updated only when fold is set, fresh: no sum is
//   pending (stage_fftx_inv).
template <typename T, int N>
__device__ __forceinline__ void fftx_inv_w_body(const Geo& g, const C2<T>* __restrict__ twx,
                                                const C2<T>* __restrict__ spec, double scale,
                                                double* __restrict__ p, int p_zero, bool lazy, bool fold, bool fresh,
                                                T* __restrict__ delta, float* __restrict__ sdelta, unsigned blk,
                                                unsigned char* smem_raw) {
  using W = WPlan<N>;
  C2<T>* tw = reinterpret_cast<C2<T>*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  C2<T>* line = tw + N + (size_t)warp * W::LW * W::LS + (lane / W::L) * W::LS;
  wfft_load_twiddles<W, T>(tw, twx);
  const int l = lane & (W::L - 1);
  const unsigned gw = blk * (blockDim.x >> 5) + warp;
  const long nrows = (long)g.nz * g.ny;
  const long ra = ((long)gw * W::LW + lane / W::L) * 2;
  const bool va = ra < nrows, vb = ra + 1 < nrows;
  const int nxh = N / 2 + 1;
  C2<T> v[W::U1][W::R1];
  {
    const C2<T>* SA = spec + (size_t)ra * nxh;
    const C2<T>* SB = SA + nxh;
#pragma unroll
    for (int u = 0; u < W::U1; ++u) {
      const int bb = l + u * W::L;
#pragma unroll
      for (int a = 0; a < W::R1; ++a) {
        const int m = W::R2 * a + bb;
        const bool in = W::R2 % W::L == 0 || bb < W::R2;
        const bool mirror = 2 * m > N;
        const int mm = mirror ? N - m : m;
        C2<T> A = mk<T>((T)0, (T)0), B = A;
        if (va && in) A = SA[mm];
        if (vb && in) B = SB[mm];
        // Z = A + i B; the upper half from the conjugates; rows are real, so
        // the imaginary parts of coefficients 0 and N/2 do not enter
        if (m == 0 || 2 * m == N) v[u][a] = mk<T>(A.x, B.x);
        else if (mirror) v[u][a] = mk<T>(A.x + B.y, B.x - A.y);
        else v[u][a] = mk<T>(A.x - B.y, A.y + B.x);
      }
    }
  }
  __syncthreads();  // twiddles
#pragma unroll
  for (int u = 0; u < W::U1; ++u) {
    const int bb = l + u * W::L;
    if (W::R2 % W::L == 0 || bb < W::R2) {
      wfft_stage1<W, T, 1>(v[u], tw, bb);
#pragma unroll
      for (int c = 0; c < W::R1; ++c) line[c * W::S + bb] = v[u][c];
    }
  }
  __syncwarp();
  const bool need_s = lazy && !fresh;
  const bool upd_p = !lazy || fold;
  const float scale_f = (float)scale;
#pragma unroll
  for (int u = 0; u < W::U2; ++u) {
    const int c = l + u * W::L;
    if (W::R1 % W::L != 0 && c >= W::R1) continue;
    C2<T> z[W::R2];
#pragma unroll
    for (int bb = 0; bb < W::R2; ++bb) z[bb] = line[c * W::S + bb];
    // the pending sums are in flight during the last transform
    float sa[W::R2], sb[W::R2];
    if constexpr (sizeof(T) == sizeof(float)) {
#pragma unroll
      for (int d = 0; d < W::R2; ++d) {
        const size_t o = (size_t)ra * N + c + W::R1 * d;
        sa[d] = need_s && va ? sdelta[o] : 0.f;
        sb[d] = need_s && vb ? sdelta[o + N] : 0.f;
      }
    }
    double pa[W::R2], pb[W::R2];
    if constexpr (sizeof(T) == sizeof(double)) {
#pragma unroll
      for (int d = 0; d < W::R2; ++d) {
        const size_t o = (size_t)ra * N + c + W::R1 * d;
        pa[d] = va && !p_zero ? p[o] : 0.0;
        pb[d] = vb && !p_zero ? p[o + N] : 0.0;
      }
    }
    Dft<T, 1, W::R2>::run(z);
    auto emit = [&](size_t o, T zv, float sv, double pv64) {
      if constexpr (sizeof(T) == sizeof(float)) {
        const float inc = scale_f * (float)zv;
        if (upd_p) {
          const double pv = p_zero ? 0.0 : p[o];
          p[o] = fma(scale, widen_f32((float)zv), need_s ? pv + widen_f32(sv) : pv);
        } else {
          sdelta[o] = need_s ? sv + inc : inc;
        }
        if (delta != nullptr) delta[o] = (T)inc;
      } else {
        p[o] = fma(scale, (double)zv, pv64);
        if (delta != nullptr) delta[o] = (T)(scale * (double)zv);
      }
    };
#pragma unroll
    for (int d = 0; d < W::R2; ++d) {
      const size_t o = (size_t)ra * N + c + W::R1 * d;
      if constexpr (sizeof(T) == sizeof(float)) {
        if (va) emit(o, z[d].x, sa[d], 0.0);
        if (vb) emit(o + N, z[d].y, sb[d], 0.0);
      } else {
        if (va) emit(o, z[d].x, 0.f, pa[d]);
        if (vb) emit(o + N, z[d].y, 0.f, pb[d]);
      }
    }
  }
}

template <typename T, int N>
__global__ void __launch_bounds__(128, sizeof(T) == sizeof(float) ? 5 : 3) k_fftx_inv_w(
    Geo g, const C2<T>* __restrict__ twx, const C2<T>* __restrict__ spec, double scale, double* __restrict__ p,
    int p_zero, const DevStatus* __restrict__ st, T* __restrict__ delta, float* __restrict__ sdelta) {
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const bool lazy = sizeof(T) == sizeof(float) && sdelta != nullptr && st != nullptr;
  fftx_inv_w_body<T, N>(g, twx, spec, scale, p, p_zero, lazy, lazy && st->need_exact != 0,
                        lazy && st->since_exact <= 1, delta, sdelta, blockIdx.x, smem_raw);
}

// ---------------------------------------------------------------------------
// y transform (stage_ffty_persistent) of kWyTx consecutive kx columns of one
// z plane per block, thread = x + kWyTx l.  The values go straight from
// global memory to registers and back; the next tile's are loaded once this
// one's sit in the exchange buffer.  Two exchange buffers take turns, so a
// tile costs one block barrier (two with the cosine transform of walls,
// whose forward pass also pairs Z_r with Z_{N-r} through the other buffer).
// Shared-memory kernel -> this, ms: mixed 256^3 0.040 -> 0.025, mixed 192 x
// 160 x 144 0.024 -> 0.007, walls 256 x 192 x 128 0.035 -> 0.012 (forward) and
// 0.020 (inverse); FP64 128^3 0.051 -> 0.049 (the FP64 pipe: 26 operations a
// point take 0.044).
constexpr int kWyTx = 8;

template <typename T, int N>
struct WyShape {
  using W = WPlan<N>;
  static constexpr int threads = kWyTx * W::L;
  // E[c][b][x]; each c slab is padded by kWyTx entries, so that the columns
  // of a slab start half a bank row apart
  static constexpr int SL = (W::R2 + ((W::R2 & 1) ? 0 : 1)) * kWyTx;
  static constexpr int ebuf = W::R1 * SL > N * kWyTx ? W::R1 * SL : N * kWyTx;
  static constexpr size_t smem = (size_t)(N + 2 * ebuf) * sizeof(C2<T>);
};

// The stage-1 values of thread (x, l) of a tile: src is its column's first
// entry; ok: the column exists.
template <typename T, int DIR, bool DCT, int N>
__device__ __forceinline__ void ffty_w_load(C2<T> (&v)[WPlan<N>::U1][WPlan<N>::R1], const C2<T>* src, int nxh, int l,
                                            bool ok, const C2<T>* __restrict__ dct) {
  using W = WPlan<N>;
#pragma unroll
  for (int u = 0; u < W::U1; ++u) {
    const int bb = l + u * W::L;
    const bool in = ok && (W::R2 % W::L == 0 || bb < W::R2);
#pragma unroll
    for (int a = 0; a < W::R1; ++a) {
      const int m = W::R2 * a + bb;
      C2<T> w = mk<T>((T)0, (T)0);
      if constexpr (DCT && DIR > 0) {
        // V_m = conj(w_m) (Y_m - i Y_{N-m}), Y_N = 0
        if (in) {
          w = src[(size_t)m * nxh];
          if (m > 0) {
            const C2<T> o = src[(size_t)(N - m) * nxh];
            w = cmulc<T>(mk<T>(w.x + o.y, w.y - o.x), dct[m]);
          }
        }
      } else {
        const int row = DCT ? dct_row(m, N) : m;
        if (in) w = src[(size_t)row * nxh];
      }
      v[u][a] = w;
    }
  }
}

// Stage 1 and the exchange write.
template <typename T, int DIR, int N>
__device__ __forceinline__ void ffty_w_front(C2<T> (&v)[WPlan<N>::U1][WPlan<N>::R1], C2<T>* e, const C2<T>* tw, int x,
                                             int l) {
  using W = WPlan<N>;
#pragma unroll
  for (int u = 0; u < W::U1; ++u) {
    const int bb = l + u * W::L;
    if (W::R2 % W::L == 0 || bb < W::R2) {
      wfft_stage1<W, T, DIR>(v[u], tw, bb);
#pragma unroll
      for (int c = 0; c < W::R1; ++c) e[c * WyShape<T, N>::SL + bb * kWyTx + x] = v[u][c];
    }
  }
}

// After the barrier: stage 2 (with the pairing of the forward cosine
// transform through e1, one more barrier) and the stores to dst.  Every
// thread of the block calls it.
template <typename T, int DIR, bool DCT, int N>
__device__ __forceinline__ void ffty_w_back(C2<T>* dst, const C2<T>* e0, C2<T>* e1, int nxh, int x, int l, bool ok,
                                            const C2<T>* __restrict__ dct) {
  using W = WPlan<N>;
  constexpr int TX = kWyTx;
  C2<T> z[W::U2][W::R2];
#pragma unroll
  for (int u = 0; u < W::U2; ++u) {
    const int c = l + u * W::L;
    if (W::R1 % W::L == 0 || c < W::R1) {
#pragma unroll
      for (int bb = 0; bb < W::R2; ++bb) z[u][bb] = e0[c * WyShape<T, N>::SL + bb * TX + x];
      Dft<T, DIR, W::R2>::run(z[u]);
    }
  }
  if constexpr (DCT && DIR < 0) {
    // X_r = (w_r Z_r + conj(w_r) Z_{N-r}) / 2, Z_N = Z_0
#pragma unroll
    for (int u = 0; u < W::U2; ++u) {
      const int c = l + u * W::L;
      if (W::R1 % W::L == 0 || c < W::R1) {
#pragma unroll
        for (int d = 0; d < W::R2; ++d) e1[(c + W::R1 * d) * TX + x] = z[u][d];
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < W::U2; ++u) {
      const int c = l + u * W::L;
      if (W::R1 % W::L == 0 || c < W::R1) {
#pragma unroll
        for (int d = 0; d < W::R2; ++d) {
          const int r = c + W::R1 * d;
          const C2<T> w = dct[r];
          const C2<T> a = cmul<T>(z[u][d], w), o = cmulc<T>(e1[(r == 0 ? 0 : N - r) * TX + x], w);
          z[u][d] = mk<T>((T)0.5 * (a.x + o.x), (T)0.5 * (a.y + o.y));
        }
      }
    }
  }
  if (ok) {
#pragma unroll
    for (int u = 0; u < W::U2; ++u) {
      const int c = l + u * W::L;
      if (W::R1 % W::L == 0 || c < W::R1) {
#pragma unroll
        for (int d = 0; d < W::R2; ++d) {
          const int r = c + W::R1 * d;
          const int row = DCT && DIR > 0 ? dct_row(r, N) : r;
          dst[(size_t)row * nxh] = z[u][d];
        }
      }
    }
  }
}

template <typename T, int DIR, bool DCT, int N>
__global__ void __launch_bounds__(WyShape<T, N>::threads) k_ffty_w(Geo g, const C2<T>* __restrict__ twy,
                                                                   C2<T>* __restrict__ spec, long long ntiles,
                                                                   const DevStatus* __restrict__ st,
                                                                   const C2<T>* __restrict__ dct) {
  using W = WPlan<N>;
  using Y = WyShape<T, N>;
  constexpr int TX = kWyTx;
  if (stopped(st)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<T>* tw = reinterpret_cast<C2<T>*>(smem_raw);
  C2<T>* e0 = tw + N;
  C2<T>* e1 = e0 + Y::ebuf;
  wfft_load_twiddles<W, T>(tw, twy);
  const int nxh = g.nxh, ntx = (nxh + TX - 1) / TX;
  const int x = threadIdx.x % TX, l = threadIdx.x / TX;
  const size_t plane = (size_t)N * nxh;
  C2<T> v[W::U1][W::R1];
  auto column = [&](long long tile, bool* ok) {
    const int bz = (int)(tile / ntx), kx = (int)(tile - (long long)bz * ntx) * TX + x;
    *ok = kx < nxh;
    return spec + (size_t)bz * plane + kx;
  };
  bool ok = false;
  long long tile = blockIdx.x;
  if (tile < ntiles) {
    const C2<T>* src = column(tile, &ok);
    ffty_w_load<T, DIR, DCT, N>(v, src, nxh, l, ok, dct);
  }
  __syncthreads();  // twiddles
  for (; tile < ntiles; tile += gridDim.x) {
    ffty_w_front<T, DIR, N>(v, e0, tw, x, l);
    if (tile + gridDim.x < ntiles) {  // other columns than this tile's
      const C2<T>* src = column(tile + gridDim.x, &ok);
      ffty_w_load<T, DIR, DCT, N>(v, src, nxh, l, ok, dct);
    }
    __syncthreads();
    C2<T>* dst = column(tile, &ok);
    ffty_w_back<T, DIR, DCT, N>(dst, e0, e1, nxh, x, l, ok, dct);
    if constexpr (!(DCT && DIR < 0)) {
      C2<T>* t = e0;
      e0 = e1;
      e1 = t;
    }
  }
}

// ---- launchers -------------------------------------------------------------
// Warps a block: four, or fewer where the grid is small, so that the blocks
// cover the SMs.
inline int wfft_warps_per_block(long long warps) {
  if (warps >= 152 * 8) return 4;
  return warps >= 152 * 2 ? 2 : 1;
}

template <typename T, int N>
cudaError_t launch_resid_w_n(const Geo& g, const Faces& fc, const C2<T>* twx, const double* b, const double* rho,
                             const double* p, int p_zero, int scale_rho, C2<T>* spec, double* red,
                             const LoopCheck* ck, const DevStatus* st, Queue s, float* E, const float* delta) {
  using W = WPlan<N>;
  const long long nrows = (long long)g.nz * g.ny;
  const long long warps = (nrows + 2 * W::LW - 1) / (2 * W::LW);
  const int wpb = wfft_warps_per_block(warps);
  const size_t smem = (size_t)(W::TW + wpb * W::LW * W::LS) * sizeof(C2<T>);
  auto kern = (g.ym != nullptr) ? k_resid_w<T, true, N> : k_resid_w<T, false, N>;
  static_assert((W::TW + 4 * W::LW * W::LS) * sizeof(C2<T>) <= 48 * 1024, "fits without the opt-in attribute");
  return enqueue(s, kern, (unsigned)((warps + wpb - 1) / wpb), 32 * wpb, smem, g, fc, twx, b, rho, p,
                 red == nullptr ? 0 : 1, p_zero, scale_rho, spec, red, st, E, delta, ck ? *ck : LoopCheck{});
}

template <typename T, int N>
cudaError_t launch_fftx_inv_w_n(const Geo& g, const C2<T>* twx, const C2<T>* spec, double scale, double* p,
                                int p_zero, const DevStatus* st, Queue s, T* delta, float* sdelta) {
  using W = WPlan<N>;
  const long long nrows = (long long)g.nz * g.ny;
  const long long warps = (nrows + 2 * W::LW - 1) / (2 * W::LW);
  const int wpb = wfft_warps_per_block(warps);
  const size_t smem = (size_t)(N + wpb * W::LW * W::LS) * sizeof(C2<T>);
  static_assert((N + 4 * W::LW * W::LS) * sizeof(C2<T>) <= 48 * 1024, "fits without the opt-in attribute");
  return enqueue(s, k_fftx_inv_w<T, N>, (unsigned)((warps + wpb - 1) / wpb), 32 * wpb, smem, g, twx, spec, scale, p,
                 p_zero, st, delta, sdelta);
}

template <auto K, typename T, int N>
cudaError_t launch_ffty_w_k(const Geo& g, const C2<T>* twy, C2<T>* spec, const DevStatus* st, Queue s,
                            const C2<T>* dct) {
  using Y = WyShape<T, N>;
  const long long ntiles = (long long)((g.nxh + kWyTx - 1) / kWyTx) * g.nz;
  long long nblk = 0;
  const cudaError_t e = resident_blocks<K>(Y::threads, Y::smem, &nblk);
  if (e != cudaSuccess) return e;
  return enqueue(s, K, (unsigned)(nblk < ntiles ? nblk : ntiles), Y::threads, Y::smem, g, twy, spec, ntiles, st, dct);
}

template <typename T, int N>
cudaError_t launch_ffty_w_n(const Geo& g, const C2<T>* twy, C2<T>* spec, int inverse, const DevStatus* st,
                            Queue s, const C2<T>* dct) {
  if (dct)
    return inverse ? launch_ffty_w_k<k_ffty_w<T, 1, true, N>, T, N>(g, twy, spec, st, s, dct)
                   : launch_ffty_w_k<k_ffty_w<T, -1, true, N>, T, N>(g, twy, spec, st, s, dct);
  return inverse ? launch_ffty_w_k<k_ffty_w<T, 1, false, N>, T, N>(g, twy, spec, st, s, dct)
                 : launch_ffty_w_k<k_ffty_w<T, -1, false, N>, T, N>(g, twy, spec, st, s, dct);
}

}  // namespace pp
