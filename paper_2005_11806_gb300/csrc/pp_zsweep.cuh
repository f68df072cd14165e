// Thomas sweeps along z with the rows streamed through shared memory: the z
// step of the eigenexpansion solve (Sec. 3.3.1), one thread per column.
//
// What bounds it: the recurrence is one dependent FP64 FMA a row, and an SM
// partition takes 64 cycles for a warp's FP64 instruction, so two or more
// warps a partition keep the pipe busy if, and only if, no thread waits for
// memory on every row.  Rows loaded into registers a few ahead did wait (a
// row's loads share a warp's few scoreboards with the rows behind them): a
// row cost about 1000 cycles at 256^3, 67 % of the stalls on global loads
// and the FP64 pipe 22 % busy.  Here each thread copies its own entries of
// the next rows into a ring in shared memory by cp.async, kZRows rows to a
// commit group, a few groups in flight; the copies need no registers, and a
// wait for one group leaves the later ones in flight.  A thread reads only
// what it copied itself, so the sweeps hold no barrier.  With the chain free
// of loads a lone warp takes 234 cycles a row against the pipe's 128 (its
// conversions and address arithmetic); the rest hides behind other warps.
//
// Measured (register prefetch -> this): PP_MIXED_Z64 256^3 0.250 -> 0.088 ms,
// 512^3 0.597 -> 0.466 ms; FP64 128^3 0.105 -> 0.029 ms; the FP32 columns of
// 192 x 160 x 144 0.075 -> 0.031 ms.  64 threads a block, 4 rows a group and
// the group counts below were the fastest of {32, 64, 128} x {2, 4, 8} x
// {2, 3, 4, 6} over 32^3 .. 512^3.
#pragma once
#include <type_traits>

#include "pp_internal.cuh"

namespace pp {

constexpr int kZThreads = 64;
constexpr int kZRows = 4;

template <int BYTES>
__device__ __forceinline__ void zs_cp(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
               :: "r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gsrc), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void zs_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void zs_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// The three forms of the sweeps.  Val: what a thread holds of a row of the
// spectrum; A, B (kHasB): the table entries a forward row reads; E: the entry
// a backward row reads; kGroups: commit groups in the ring.

// FP32 values inside the FP64 recurrences, scaled by 2^-896: the eight
// exponent bits of the FP32 value become the low exponent bits of the FP64
// one unchanged (127 - 1023 = -896), so widening takes three integer
// instructions instead of nine, zero and subnormals included, and narrowing
// seven.  The recurrences are linear, so nothing else changes; a result at
// or above 2^128 narrows to Inf.  Inf and NaN widen to finite values from
// 2^128 up, and a sweep may damp these below 2^128 again, so a bad row does
// not make its whole column Inf.  It reaches the caller all the same: a
// projection stops on the residual's norm before the sweep, and in a plain
// solve the mean of column (0, 0), taken in plain FP64, makes that column and
// with it every value of p non-finite.
__device__ __forceinline__ double zs_widen(float f) {
  const int b = __float_as_int(f);
  return __hiloint2double((b >> 3) & (int)0x8FFFFFFF, b << 29);
}
__device__ __forceinline__ float zs_narrow(double d) {  // half away from zero, as narrow_f64
  const unsigned hi = (unsigned)__double2hiint(d);
  const unsigned long long r = (((unsigned long long)hi << 32) | (unsigned)__double2loint(d)) + 0x10000000ull;
  unsigned bits = (unsigned)(r >> 29) & 0x7FFFFFFFu;
  if ((hi & 0x7FFFFFFFu) >= 0x0FF00000u) bits = 0x7F800000u;
  return __uint_as_float(bits | (hi & 0x80000000u));
}
constexpr double kZScale = 0x1p-896;

// PP_MIXED_Z64: both components of a column, FP64 recurrences on FP32
// storage (TriZ<float>): y_k = f_k - m_k y_{k-1}, s_k = y_k / d_k (stored),
// x_k = s_k - e_k x_{k+1}.  The means m0x, m0y come scaled.
struct ZForm64 {
  static constexpr int kGroups = 3;
  using Val = float2;
  using A = double;
  using B = float;
  using E = double;
  static constexpr bool kHasB = true;
  const double* m;
  const float* d;
  const double* e;
  struct State { double x, y; };
  static __device__ __forceinline__ State zero() { return {0.0, 0.0}; }
  template <bool ZERO>
  static __device__ __forceinline__ State fwd(const State& s, Val f, A m, double m0x, double m0y) {
    const double fx = zs_widen(f.x), fy = zs_widen(f.y);
    return {fma(-m, s.x, ZERO ? fx - m0x : fx), fma(-m, s.y, ZERO ? fy - m0y : fy)};
  }
  static __device__ __forceinline__ Val fwd_value(const State& s, B d) {
    return make_float2(zs_narrow(s.x) * d, zs_narrow(s.y) * d);
  }
  static __device__ __forceinline__ State turn(Val last, E) { return {zs_widen(last.x), zs_widen(last.y)}; }
  static __device__ __forceinline__ State bwd(const State& s, Val v, E e, float) {
    return {fma(-e, s.x, zs_widen(v.x)), fma(-e, s.y, zs_widen(v.y))};
  }
  static __device__ __forceinline__ Val bwd_value(const State& s) {
    return make_float2(zs_narrow(s.x), zs_narrow(s.y));
  }
};

// FP64 plans: one component (real or imaginary part) of a column, the same
// recurrences with FP64 storage and FP64 inverse pivots.  Three groups rather
// than four leave room for 12 blocks an SM instead of 9 (18 KB a block):
// 256^3 0.139 -> 0.119 ms, 384^3 0.506 -> 0.381, 512^3 1.18 -> 0.91 (0.235,
// 0.487 and 1.01 with register prefetch); two groups 0.122, 0.457, 0.946.
struct ZFormD {
  static constexpr int kGroups = 3;
  using Val = double;
  using A = double;
  using B = double;
  using E = double;
  static constexpr bool kHasB = true;
  const double* m;
  const double* d;
  const double* e;
  using State = double;
  static __device__ __forceinline__ State zero() { return 0.0; }
  template <bool ZERO>
  static __device__ __forceinline__ State fwd(State s, Val f, A m, double m0, double) {
    return fma(-m, s, ZERO ? f - m0 : f);
  }
  static __device__ __forceinline__ Val fwd_value(State s, B d) { return s * d; }
  static __device__ __forceinline__ State turn(Val last, E) { return last; }
  static __device__ __forceinline__ State bwd(State s, Val v, E e, float) { return fma(-e, s, v); }
  static __device__ __forceinline__ Val bwd_value(State s) { return s; }
};

// Well-conditioned columns of PP_MIXED_FP32 (TriF32): FP32 throughout,
// y_k = f_k - m_k y_{k-1} (stored), x_k = (y_k - c_k x_{k+1}) / d_k.
struct ZForm32 {
  static constexpr int kGroups = 4;
  using Val = float2;
  using A = float;
  using B = float;  // not read
  using E = float;  // 1 / d_k
  static constexpr bool kHasB = false;
  const float* m;
  const float* d;
  const float* e;
  using State = float2;
  static __device__ __forceinline__ State zero() { return make_float2(0.f, 0.f); }
  template <bool ZERO>
  static __device__ __forceinline__ State fwd(State s, Val f, A m, double, double) {
    return make_float2(fmaf(-m, s.x, f.x), fmaf(-m, s.y, f.y));
  }
  static __device__ __forceinline__ Val fwd_value(State s, B) { return s; }
  static __device__ __forceinline__ State turn(Val last, E d) { return make_float2(last.x * d, last.y * d); }
  static __device__ __forceinline__ State bwd(State s, Val v, E d, float c) {
    return make_float2(fmaf(-c, s.x, v.x) * d, fmaf(-c, s.y, v.y) * d);
  }
  static __device__ __forceinline__ Val bwd_value(State s) { return s; }
};

// Shared memory of one block of kZThreads threads, a column each.
template <class F>
constexpr size_t zsweep_smem() {
  return (size_t)kZRows * F::kGroups * kZThreads *
         (sizeof(typename F::Val) + (F::kHasB ? sizeof(typename F::B) : 0) +
          (sizeof(typename F::A) > sizeof(typename F::E) ? sizeof(typename F::A) : sizeof(typename F::E)));
}

// One sweep over n rows of a thread's column.  Row i lies at v + i vstep
// (spectrum), ta + i tstep (first table) and tb + i tstep (second table, HASB);
// step(state, value, a, i) is the recurrence, value(state, b) what is stored in
// place of the row.
//
// A warp issues in order, so a row's conversions and store must not stand
// between its FMA and the next row's: the value of row i is formed while the
// FMA of row i + 1 is in flight.  The next group's entries are read into
// registers before the current group's chain for the same reason.
template <bool HASB, int NG, class State, class Val, class A, class B, class Step, class Value>
__device__ __forceinline__ void zsweep_rows(State& s, int n, Val* v, ptrdiff_t vstep, const A* ta, const B* tb,
                                            ptrdiff_t tstep, Val* rv, A* ra, B* rb, Step&& step, Value&& value) {
  constexpr int R = kZRows, SLOTS = R * NG;
  const Val* cv = v;
  Val* out = v;
  int left = n, slot = 0;  // rows not yet copied, slot of the next
  auto copy_row = [&](int at, ptrdiff_t vo, ptrdiff_t to) {
    zs_cp<sizeof(Val)>(rv + at * kZThreads, cv + vo);
    zs_cp<sizeof(A)>(ra + at * kZThreads, ta + to);
    if constexpr (HASB) zs_cp<sizeof(B)>(rb + at * kZThreads, tb + to);
  };
  auto issue = [&]() {
    if (left >= R) {
#pragma unroll
      for (int u = 0; u < R; ++u) copy_row(slot + u, u * vstep, u * tstep);
      cv += R * vstep;
      ta += R * tstep;
      if constexpr (HASB) tb += R * tstep;
    } else {
      for (int u = 0; u < left; ++u) copy_row(slot + u, u * vstep, u * tstep);
    }
    zs_commit();
    left -= R;
    slot = slot + R == SLOTS ? 0 : slot + R;
  };
#pragma unroll
  for (int q = 0; q < NG; ++q) issue();
  Val f[R];
  A a[R];
  B b[R];
  int rd = 0;
  auto read = [&](Val (&ff)[R], A (&aa)[R], B (&bb)[R]) {  // slots past the last row hold old data, unused
#pragma unroll
    for (int u = 0; u < R; ++u) {
      ff[u] = rv[(rd + u) * kZThreads];
      aa[u] = ra[(rd + u) * kZThreads];
      if constexpr (HASB) bb[u] = rb[(rd + u) * kZThreads];
      else bb[u] = B();
    }
    rd = rd + R == SLOTS ? 0 : rd + R;
  };
  zs_wait<NG - 1>();
  read(f, a, b);
  B bprev = B();
  int i = 0;
  for (; i + R <= n; i += R) {
    Val f2[R];
    A a2[R];
    B b2[R];
    zs_wait<NG - 2>();
    read(f2, a2, b2);
    issue();
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const State t = step(s, f[u], a[u], i + u);
      const Val w = value(s, bprev);  // row i + u - 1
      if (u > 0 || i > 0) out[(u - 1) * vstep] = w;
      s = t;
      bprev = b[u];
    }
    out += R * vstep;
#pragma unroll
    for (int u = 0; u < R; ++u) {
      f[u] = f2[u];
      a[u] = a2[u];
      b[u] = b2[u];
    }
  }
#pragma unroll
  for (int u = 0; u < R; ++u) {
    if (i + u < n) {
      const State t = step(s, f[u], a[u], i + u);
      if (i + u > 0) out[(u - 1) * vstep] = value(s, bprev);
      s = t;
      bprev = b[u];
    }
  }
  if (n > 0) v[(n - 1) * vstep] = value(s, bprev);
  zs_wait<0>();
}

// Both sweeps of a thread's column.  val: its first entry, vstride entries
// from row to row; t: its table offset, tstride entries from row to row; zc:
// the super-diagonal of L_z (ZForm32 only).  ZERO: m0x, m0y are subtracted from
// the right-hand side (the singular column's mean).
template <class F, bool ZERO>
__device__ __forceinline__ void zsweep(const F& tab, typename F::Val* val, size_t vstride, size_t t, size_t tstride,
                                       int nz, const float* __restrict__ zc, unsigned char* smem, double m0x,
                                       double m0y) {
  using Val = typename F::Val;
  using A = typename F::A;
  using B = typename F::B;
  using E = typename F::E;
  using State = typename F::State;
  constexpr int SLOTS = kZRows * F::kGroups;
  constexpr size_t kAE = sizeof(A) > sizeof(E) ? sizeof(A) : sizeof(E);
  Val* rv = reinterpret_cast<Val*>(smem) + threadIdx.x;
  unsigned char* after_v = smem + sizeof(Val) * SLOTS * kZThreads;
  A* ra = reinterpret_cast<A*>(after_v) + threadIdx.x;
  E* re = reinterpret_cast<E*>(after_v) + threadIdx.x;
  B* rb = reinterpret_cast<B*>(after_v + kAE * SLOTS * kZThreads) + threadIdx.x;
  State s = F::zero();
  zsweep_rows<F::kHasB, F::kGroups>(
      s, nz, val, (ptrdiff_t)vstride, (const A*)tab.m + t, (const B*)tab.d + (F::kHasB ? t : 0), (ptrdiff_t)tstride,
      rv, ra, rb,
      [&](const State& p, const Val& f, const A& m, int) { return F::template fwd<ZERO>(p, f, m, m0x, m0y); },
      [](const State& p, const B& d) { return F::fwd_value(p, d); });
  // row nz - 1: x from the value just stored (this thread's own store)
  const E* te = (const E*)tab.e + t;
  constexpr bool F32 = std::is_same<F, ZForm32>::value;
  Val* top = val + (size_t)(nz - 1) * vstride;
  s = F::turn(*top, F32 ? te[(size_t)(nz - 1) * tstride] : E());
  if constexpr (F32) *top = s;
  __threadfence_block();  // the forward values are read back by this thread's copies
  zsweep_rows<false, F::kGroups>(
      s, nz - 1, top - vstride, -(ptrdiff_t)vstride, te + (ptrdiff_t)(nz - 2) * (ptrdiff_t)tstride, (const B*)nullptr,
      -(ptrdiff_t)tstride, rv, re, rb,
      [&](const State& p, const Val& v, const E& e, int i) { return F::bwd(p, v, e, F32 ? zc[nz - 2 - i] : 0.f); },
      [](const State& p, const B&) { return F::bwd_value(p); });
}

// dzf-weighted z mean of column 0, by one whole warp: of the complex entries
// (float2: scaled by 2^-896 for ZForm64) or of its two scalars (double).
__device__ __forceinline__ void zero_column_mean(const Geo& g, const float2* spec, size_t stride, double& mx,
                                                 double& my) {
  double sx = 0.0, sy = 0.0;
  for (int k = threadIdx.x & 31; k < g.nz; k += 32) {
    const float2 v = spec[(size_t)k * stride];
    sx = fma(g.dzf[k], (double)v.x, sx);
    sy = fma(g.dzf[k], (double)v.y, sy);
  }
  for (int o = 16; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
  }
  mx = sx / g.lz * kZScale;
  my = sy / g.lz * kZScale;
}
__device__ __forceinline__ void zero_column_mean(const Geo& g, const double* spec, size_t stride, double& mx,
                                                 double& my) {
  double sx = 0.0, sy = 0.0;
  for (int k = threadIdx.x & 31; k < g.nz; k += 32) {
    sx = fma(g.dzf[k], spec[(size_t)k * stride], sx);
    sy = fma(g.dzf[k], spec[(size_t)k * stride + 1], sy);
  }
  for (int o = 16; o > 0; o >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
  }
  mx = sx / g.lz;
  my = sy / g.lz;
}

}  // namespace pp
