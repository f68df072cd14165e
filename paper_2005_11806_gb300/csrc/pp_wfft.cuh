// Complex transforms of length N = R1 x R2 (both at most 16) with the data
// in registers and one exchange through shared memory: the x and y
// transforms of the eigenexpansion solve (Sec. 3.3.1) for the lengths of
// PP_WFFT_LENGTHS.
//
//   X[c + R1 d] = sum_b W_R2^{b d} W_N^{b c} sum_a W_R1^{a c} x[R2 a + b]
//
// L threads hold a line: stage 1 does the R2 transforms of length R1
// (thread l: b = l, l + L, ...), the products with W_N^{bc} go to shared
// memory as E[c][b], stage 2 does the R1 transforms of length R2.  The
// shared-memory Stockham passes that these replace read and wrote every
// value once a pass (three to five passes) with a block barrier after each.
#pragma once
#include <type_traits>
#include <utility>

#include "pp_fft.cuh"

namespace pp {

// cos and sin of 2 pi m / n for the constants of the small transforms,
// at compile time: reduced to [0, pi/4], then the Taylor series.
struct RootOf {
  static __host__ __device__ constexpr double taylor(double x, bool sine) {
    double t = sine ? x : 1.0, s = t;
    for (int k = sine ? 1 : 0; k < 24; k += 2) {
      t *= -x * x / (double)((k + 1) * (k + 2));
      s += t;
    }
    return s;
  }
  static __host__ __device__ constexpr double cosine(int m, int n) {  // m in [0, n)
    if (2 * m > n) m = n - m;                               // cos(2 pi - x) = cos x
    if (4 * m > n) return -cosine_half(n - 2 * m, 2 * n);   // cos(pi - x) = -cos x
    return cosine_half(2 * m, 2 * n);
  }
  static __host__ __device__ constexpr double sine(int m, int n) {
    if (2 * m > n) return -sine(n - m, n);
    if (4 * m > n) return sine_half(n - 2 * m, 2 * n);
    return sine_half(2 * m, 2 * n);
  }

 private:
  static constexpr double kTwoPi = 6.283185307179586476925286766559;
  // 2 pi m / n in [0, pi/2]
  static __host__ __device__ constexpr double cosine_half(int m, int n) {
    return 8 * m > n ? taylor(kTwoPi * (n - 4 * m) / (4.0 * n), true) : taylor(kTwoPi * m / n, false);
  }
  static __host__ __device__ constexpr double sine_half(int m, int n) {
    return 8 * m > n ? taylor(kTwoPi * (n - 4 * m) / (4.0 * n), false) : taylor(kTwoPi * m / n, true);
  }
};

// v * exp(DIR 2 pi i M / N), constants folded.
template <typename T, int DIR, int M_, int N>
__device__ __forceinline__ C2<T> mul_root(C2<T> v) {
  constexpr int M = M_ % N;
  if constexpr (M == 0) {
    return v;
  } else if constexpr (4 * M == N) {
    return mul_i<T, DIR>(v);
  } else if constexpr (2 * M == N) {
    return mk<T>(-v.x, -v.y);
  } else if constexpr (4 * M == 3 * N) {
    return mul_i<T, -DIR>(v);
  } else if constexpr (8 * M == N || 8 * M == 3 * N) {
    constexpr T h = (T)0.70710678118654752440;
    constexpr T c = 8 * M == N ? (T)1 : (T)-1;
    // (c + DIR i) h v
    return mk<T>(h * (c * v.x - (T)DIR * v.y), h * (c * v.y + (T)DIR * v.x));
  } else {
    constexpr T c = (T)RootOf::cosine(M, N), s = (T)(DIR * RootOf::sine(M, N));
    return mk<T>(v.x * c - v.y * s, v.x * s + v.y * c);
  }
}

// Composite in-register transforms: R = P Q, input index Q a + b, output
// index c + P d.
template <typename T, int DIR, int P, int Q>
struct DftMix {
  template <int B, int... Cs>
  static __device__ __forceinline__ void column(C2<T>* v, C2<T> (&w)[P * Q], std::integer_sequence<int, Cs...>) {
    C2<T> u[P];
#pragma unroll
    for (int a = 0; a < P; ++a) u[a] = v[Q * a + B];
    Dft<T, DIR, P>::run(u);
    ((w[Cs * Q + B] = mul_root<T, DIR, B * Cs, P * Q>(u[Cs])), ...);
  }
  template <int... Bs>
  static __device__ __forceinline__ void columns(C2<T>* v, C2<T> (&w)[P * Q], std::integer_sequence<int, Bs...>) {
    (column<Bs>(v, w, std::make_integer_sequence<int, P>{}), ...);
  }
  static __device__ __forceinline__ void run(C2<T>* v) {
    C2<T> w[P * Q];
    columns(v, w, std::make_integer_sequence<int, Q>{});
#pragma unroll
    for (int c = 0; c < P; ++c) {
      Dft<T, DIR, Q>::run(&w[c * Q]);
#pragma unroll
      for (int d = 0; d < Q; ++d) v[c + P * d] = w[c * Q + d];
    }
  }
};
template <typename T, int DIR> struct Dft<T, DIR, 6> : DftMix<T, DIR, 2, 3> {};
template <typename T, int DIR> struct Dft<T, DIR, 9> : DftMix<T, DIR, 3, 3> {};
template <typename T, int DIR> struct Dft<T, DIR, 10> : DftMix<T, DIR, 2, 5> {};
template <typename T, int DIR> struct Dft<T, DIR, 12> : DftMix<T, DIR, 4, 3> {};
template <typename T, int DIR> struct Dft<T, DIR, 15> : DftMix<T, DIR, 3, 5> {};
template <typename T, int DIR> struct Dft<T, DIR, 16> : DftMix<T, DIR, 4, 4> {};

// The lengths taken: the even ones from 32 to 256 without factors above 5 that
// split into two of the transforms above.  The line is drawn by build time (14
// kernels a length), not by a crossover.  Instantiated on both sides of it
// and timed against the shared-memory passes (fft_block), us a pass: 16^3 FP64
// 46.9 -> 34.7, 24^3 mixed_z64 40.4 -> 33.0, 30^3 FP64 67.5 -> 49.3, 24 x 24 x
// 512 mixed_z64 179 -> 167; odd y, 64 x 75 x 64 FP64 102.8 -> 104.4, mixed_z64
// 55.9 -> 50.8, 64 x 225 x 64 FP64 210 -> 193, mixed_z64 66.9 -> 55.0.  These
// ten lengths took the build from 54 to 71 s.
//
// The split of one length.  L threads a line (8 or 16); U1 and U2 transforms
// a thread in the two stages.
template <int N_, int R1_, int R2_, int L_>
struct WSplit {
  static constexpr int N = N_, R1 = R1_, R2 = R2_, L = L_;
  static_assert(R1 * R2 == N, "");
  static constexpr int U1 = (R2 + L - 1) / L, U2 = (R1 + L - 1) / L;
  static constexpr int S = (R2 & 1) ? R2 : R2 + 1;  // odd row stride of E: no bank conflicts on the columns
  static constexpr int LW = 32 / L;                 // lines a warp
  static constexpr int TW = N;                      // twiddle entries
  // Elements between the lines of a warp.  With 8 threads a line, two lines
  // share a half warp's access and start 8 entries apart modulo 16.
  static constexpr int raw = R1 * S > N ? R1 * S : N;
  static constexpr int LS = L == 16 ? (raw + 1) / 2 * 2 : (raw + 7) / 16 * 16 + 8;
};

template <int N> struct WPlan;
#define PP_WPLAN(N, R1, R2, L) \
  template <> struct WPlan<N> : WSplit<N, R1, R2, L> {};
PP_WPLAN(32, 8, 4, 8)
PP_WPLAN(36, 6, 6, 8)
PP_WPLAN(40, 8, 5, 8)
PP_WPLAN(48, 8, 6, 8)
PP_WPLAN(50, 10, 5, 8)
PP_WPLAN(54, 9, 6, 8)
PP_WPLAN(60, 10, 6, 8)
PP_WPLAN(64, 8, 8, 8)
PP_WPLAN(72, 9, 8, 8)
PP_WPLAN(80, 10, 8, 8)
PP_WPLAN(90, 10, 9, 16)
PP_WPLAN(96, 12, 8, 8)
PP_WPLAN(100, 10, 10, 16)
PP_WPLAN(108, 12, 9, 16)
PP_WPLAN(120, 15, 8, 8)
PP_WPLAN(128, 16, 8, 8)
PP_WPLAN(144, 12, 12, 16)
PP_WPLAN(150, 15, 10, 16)
PP_WPLAN(160, 16, 10, 16)
PP_WPLAN(180, 15, 12, 16)
PP_WPLAN(192, 16, 12, 16)
PP_WPLAN(240, 16, 15, 16)
PP_WPLAN(256, 16, 16, 16)
#undef PP_WPLAN
// 512 = 8 x 8 x 8 with 32 threads a line, 16 values each (the x transform of
// the FP32 residual, wfft512_line): rows of the two exchanges 72 and 73
// entries apart, twiddle tables as R512.
template <> struct WPlan<512> {
  static constexpr int N = 512, L = 32, LW = 1, LS = 8 * 73, TW = 8 * 64 + 64;
};
#define PP_WFFT_LENGTHS(X) \
  X(32) X(36) X(40) X(48) X(50) X(54) X(60) X(64) X(72) X(80) X(90) X(96) X(100) X(108) X(120) X(128) X(144) X(150) \
  X(160) X(180) X(192) X(240) X(256)

inline bool wfft_length(int n) {
  switch (n) {
#define PP_X(N) case N:
    PP_WFFT_LENGTHS(PP_X)
#undef PP_X
    return true;
  }
  return false;
}

// Twiddles of the exchange, [c][b] = exp(2 pi i b c / N), into shared memory
// from the (cos, sin)(2 pi m / N) table; every thread of the block calls it,
// a barrier follows.
template <class W, typename T>
__device__ __forceinline__ void wfft_load_twiddles(C2<T>* tw, const C2<T>* __restrict__ table) {
  for (int i = threadIdx.x; i < W::N; i += blockDim.x) {
    const int c = i / W::R2, b = i - c * W::R2;
    tw[i] = table[b * c];  // b c < N
  }
}

// Stage 1 of one DFT: v[a] = x[R2 a + b] on entry, E[c][b] = W_N^{bc} times
// its transform on return in v[c].
template <class W, typename T, int DIR>
__device__ __forceinline__ void wfft_stage1(C2<T>* v, const C2<T>* tw, int b) {
  Dft<T, DIR, W::R1>::run(v);
#pragma unroll
  for (int c = 1; c < W::R1; ++c) {
    C2<T> w = tw[c * W::R2 + b];
    if (DIR < 0) w.y = -w.y;
    v[c] = cmul<T>(v[c], w);
  }
}

}  // namespace pp
