// 3D FFT passes of the wave-space operator: shared declarations, the register
// DFTs and the pass kernels (instantiated per grid size in fft_*.cu).
//
// The six real fields travel as three complex ones, g_p + i g_(p+3), through
// plain complex transforms; the real fields' spectra are separated only where
// the Green's function needs them, from the values at k and -k, so no pass
// unpacks half spectra and no line is shorter than another.  A size n = R1 R2
// takes two register DFTs per line and one exchange through shared memory:
//   index x = j + R2 i: DFT_R1 over i, twiddle w_n^(j k1), exchange,
//   DFT_R2 over j gives k = k1 + R1 k2.
// Global loads feed the first DFT and the second one stores to global memory,
// so an element crosses shared memory once per transform (the multi-stage
// plan of the other sizes crosses it five to seven times, with a barrier
// each), and a pass is many small blocks instead of one block per plane, so
// loads, DFTs and stores of different blocks overlap.
//
// Layout between the passes: spec[p][z][kx][y] complex, p < 3 (the x pass
// stores transposed): the y pass works in place on contiguous lines, and the
// z pass reads TP consecutive ky of a kx per row.
#pragma once

#include "fsd_internal.cuh"

#include <type_traits>

namespace fsd {

template <typename T>
struct alignas(2 * sizeof(T)) Cplx {
  T x, y;
};

// Green's function operands of the z pass: the halved factors and 1/k^2 (in
// (2 pi / L)^2).  Cubic box: by m = kx^2 + ky^2 + kz^2, green[4 m] in FP64,
// green[3 m] in FP32, where the division is cheap.  Lees-Edwards box:
// gle[kx <= n/2][kz][ky][4] for the current offset, the physical wave vector
// (kx, ky - tau kx, kz).
template <typename T>
struct ZGreen {
  const T *green = nullptr;
  const T *gle = nullptr;
  const double *tilt_dev = nullptr;  // overrides tau when set
  double tau = 0.0, invL = 0.0;
};

// The random wave field of the Brownian sampler (in place of the forward
// transform and the Green's function).
template <typename T>
struct ZBrown {
  const T *btab = nullptr;         // by m: (c fM, c fD), cubic box
  const double *field = nullptr;   // complex [3][n][n][n/2+1], or null: Philox
  uint64_t seed = 0, step = 0;
  double tau = 0.0, ks2 = 0.0, xi = 0.0, alpha = 0.0, a = 0.0, eta = 0.0, isv = 0.0;
};

// Velocity fields after the inverse transform: FP32 grids whose side is a
// multiple of 4 are stored in bricks of 4 x 4 x 2 points,
// [6][z/2][y/4][x/4][z%2][y%4][x%4] (one 128-byte line each, for the
// interpolation), other FP32 grids as planar rows [6][z][y][x], FP64
// interleaved [z][y][x][8].
template <typename T, int n>
inline constexpr bool kFftBricks = sizeof(T) == 4 && n % 4 == 0;

// Launchers of one (precision, size).
template <typename T>
struct FftOps {
  int n = 0, R1 = 0, R2 = 0;
  void (*x_fwd)(cudaStream_t, const T *grid, Cplx<T> *spec, const Cplx<T> *tw) = nullptr;
  void (*y_pass)(cudaStream_t, Cplx<T> *spec, const Cplx<T> *tw, bool inverse) = nullptr;
  void (*z_green)(cudaStream_t, Cplx<T> *spec, const Cplx<T> *tw, const ZGreen<T> &) = nullptr;
  void (*z_brown)(cudaStream_t, Cplx<T> *spec, const Cplx<T> *tw, const ZBrown<T> &) = nullptr;
  void (*x_inv)(cudaStream_t, const Cplx<T> *spec, T *out, const Cplx<T> *tw) = nullptr;
};

// null when no two-factor kernel is built for n (the staged plan serves it)
template <typename T>
const FftOps<T> *fft_ops(int n);

// raise a kernel's dynamic shared-memory limit (wavespace.cu; thread-safe)
void raise_smem(const void *fn, size_t bytes);

#ifdef FSD_FFT_KERNELS

// ------------------------------------------------------------ register DFTs
// S = -1 forward, +1 inverse.  Coprime factors combine by the prime-factor
// mapping (no twiddles); 8, 9 and 16 by Cooley-Tukey with constant twiddles.
// Multiplications by 1, -1, i and -i cost nothing and signs are compile-time:
// FP64 runs at 1/74 of the FP32 rate, so every product counts there.
template <typename T>
__device__ __forceinline__ Cplx<T> operator+(Cplx<T> a, Cplx<T> b) {
  return {a.x + b.x, a.y + b.y};
}
template <typename T>
__device__ __forceinline__ Cplx<T> operator-(Cplx<T> a, Cplx<T> b) {
  return {a.x - b.x, a.y - b.y};
}
template <int S, typename T>
__device__ __forceinline__ Cplx<T> times_i(Cplx<T> a) {  // S i a
  return S > 0 ? Cplx<T>{-a.y, a.x} : Cplx<T>{a.y, -a.x};
}
template <typename T>
__device__ __forceinline__ Cplx<T> times(Cplx<T> a, Cplx<T> b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}

// a exp(S 2 pi i m / N), N = 8, 9 or 16, m a constant after unrolling
template <int N, int S, typename T>
__device__ __forceinline__ Cplx<T> times_root(Cplx<T> a, int m) {
  constexpr double c16[5] = {1.0, 0.92387953251128675613, 0.70710678118654752440,
                             0.38268343236508977173, 0.0};
  constexpr double c9[5] = {1.0, 0.76604444311897803520, 0.17364817766693034885, -0.5,
                            -0.93969262078590838405};
  constexpr double s9[5] = {0.0, 0.64278760968653932632, 0.98480775301220805936,
                            0.86602540378443864676, 0.34202014332566873304};
  if (N == 9) {
    if (m == 0) return a;
    const T c = (T)c9[m], s = (T)(S * s9[m]);
    return {a.x * c - a.y * s, a.x * s + a.y * c};
  }
  int q = m * (16 / N) % 16;
  if (q >= 8) {
    a = {-a.x, -a.y};
    q -= 8;
  }
  if (q >= 4) {
    a = times_i<S>(a);
    q -= 4;
  }
  if (q == 0) return a;
  if (q == 2) {
    const T h = (T)c16[2];
    return S > 0 ? Cplx<T>{h * (a.x - a.y), h * (a.x + a.y)} : Cplx<T>{h * (a.x + a.y), h * (a.y - a.x)};
  }
  const T c = (T)c16[q], s = (T)(S * c16[4 - q]);
  return {a.x * c - a.y * s, a.x * s + a.y * c};
}

template <int R, int S, typename T>
struct Dft;

template <int S, typename T>
struct Dft<2, S, T> {
  static __device__ __forceinline__ void run(Cplx<T> *v) {
    const Cplx<T> a = v[0], b = v[1];
    v[0] = a + b;
    v[1] = a - b;
  }
};
template <int S, typename T>
struct Dft<3, S, T> {
  static __device__ __forceinline__ void run(Cplx<T> *v) {
    const T h = (T)(S * 0.86602540378443864676);
    const Cplx<T> t = v[1] + v[2], d = v[1] - v[2];
    const Cplx<T> c = {v[0].x - T(0.5) * t.x, v[0].y - T(0.5) * t.y};
    v[0] = v[0] + t;
    v[1] = {c.x - h * d.y, c.y + h * d.x};
    v[2] = {c.x + h * d.y, c.y - h * d.x};
  }
};
template <int S, typename T>
struct Dft<4, S, T> {
  static __device__ __forceinline__ void run(Cplx<T> *v) {
    const Cplx<T> a = v[0] + v[2], b = v[0] - v[2], c = v[1] + v[3], d = times_i<S>(v[1] - v[3]);
    v[0] = a + c;
    v[2] = a - c;
    v[1] = b + d;
    v[3] = b - d;
  }
};
template <int S, typename T>
struct Dft<5, S, T> {
  static __device__ __forceinline__ void run(Cplx<T> *v) {
    const T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;
    const T s1 = (T)(S * 0.95105651629515357212), s2 = (T)(S * 0.58778525229247312917);
    const Cplx<T> a1 = v[1] + v[4], b1 = v[1] - v[4], a2 = v[2] + v[3], b2 = v[2] - v[3], x0 = v[0];
    const Cplx<T> r1 = {x0.x + c1 * a1.x + c2 * a2.x, x0.y + c1 * a1.y + c2 * a2.y};
    const Cplx<T> r2 = {x0.x + c2 * a1.x + c1 * a2.x, x0.y + c2 * a1.y + c1 * a2.y};
    const Cplx<T> i1 = {s1 * b1.x + s2 * b2.x, s1 * b1.y + s2 * b2.y};
    const Cplx<T> i2 = {s2 * b1.x - s1 * b2.x, s2 * b1.y - s1 * b2.y};
    v[0] = {x0.x + a1.x + a2.x, x0.y + a1.y + a2.y};
    v[1] = {r1.x - i1.y, r1.y + i1.x};
    v[4] = {r1.x + i1.y, r1.y - i1.x};
    v[2] = {r2.x - i2.y, r2.y + i2.x};
    v[3] = {r2.x + i2.y, r2.y - i2.x};
  }
};

// N = A B coprime: x index B a + A b (mod N), output k = k_a mod A, k_b mod B
template <int A, int B, int S, typename T>
struct DftPrime {
  static __device__ __forceinline__ void run(Cplx<T> *v) {
    constexpr int N = A * B;
    Cplx<T> y[N];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      Cplx<T> t[A];
#pragma unroll
      for (int a = 0; a < A; ++a) t[a] = v[(B * a + A * b) % N];
      Dft<A, S, T>::run(t);
#pragma unroll
      for (int a = 0; a < A; ++a) y[a * B + b] = t[a];
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      Cplx<T> t[B];
#pragma unroll
      for (int b = 0; b < B; ++b) t[b] = y[a * B + b];
      Dft<B, S, T>::run(t);
      // k with k = a (mod A) and k = b (mod B)
#pragma unroll
      for (int b = 0; b < B; ++b) {
        int k = a;
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (k % B != b) k += A;
        v[k] = t[b];
      }
    }
  }
};
// N = A B: x index B a + b, output k = k_a + A k_b
template <int A, int B, int S, typename T>
struct DftTwiddle {
  static __device__ __forceinline__ void run(Cplx<T> *v) {
    constexpr int N = A * B;
    Cplx<T> y[N];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      Cplx<T> t[A];
#pragma unroll
      for (int a = 0; a < A; ++a) t[a] = v[B * a + b];
      Dft<A, S, T>::run(t);
#pragma unroll
      for (int a = 0; a < A; ++a) y[a * B + b] = times_root<N, S>(t[a], a * b);
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      Cplx<T> t[B];
#pragma unroll
      for (int b = 0; b < B; ++b) t[b] = y[a * B + b];
      Dft<B, S, T>::run(t);
#pragma unroll
      for (int b = 0; b < B; ++b) v[a + A * b] = t[b];
    }
  }
};
template <int S, typename T> struct Dft<6, S, T> : DftPrime<2, 3, S, T> {};
template <int S, typename T> struct Dft<8, S, T> : DftTwiddle<2, 4, S, T> {};
template <int S, typename T> struct Dft<9, S, T> : DftTwiddle<3, 3, S, T> {};
template <int S, typename T> struct Dft<10, S, T> : DftPrime<2, 5, S, T> {};
template <int S, typename T> struct Dft<12, S, T> : DftPrime<3, 4, S, T> {};
template <int S, typename T> struct Dft<15, S, T> : DftPrime<3, 5, S, T> {};
template <int S, typename T> struct Dft<16, S, T> : DftTwiddle<4, 4, S, T> {};
template <int S, typename T> struct Dft<18, S, T> : DftPrime<2, 9, S, T> {};
template <int S, typename T> struct Dft<20, S, T> : DftPrime<4, 5, S, T> {};

// -------------------------------------------------------------- one line
// Shared-memory position of (k1, j): chunks of R2 padded to an odd stride, so
// that lanes on consecutive k1 (second DFT) fall in distinct banks as lanes on
// consecutive j (first DFT) do.  Where lanes run over the lines of a tile, the
// line stride is 2 mod 16 elements: eight lines by two consecutive j or k1
// cover sixteen banks of 8 bytes.
template <int R1, int R2>
struct Line {
  static constexpr int CS = R2 | 1;
  static constexpr int LC = R1 * CS;                      // lanes along the line
  static constexpr int LT = LC + (16 + 2 - LC % 16) % 16;  // lanes across lines
};

// first DFT of a line at j: values v (stride R2 in the line), results to s
template <int R1, int R2, int S, typename T>
__device__ __forceinline__ void first_dft(Cplx<T> *v, int j, Cplx<T> *s, const Cplx<T> *tw) {
  Dft<R1, S, T>::run(v);
  s[j] = v[0];
#pragma unroll
  for (int k = 1; k < R1; ++k) {
    Cplx<T> w = tw[k * R2 + j];
    if (S > 0) w.y = -w.y;  // the table holds the forward twiddles
    s[k * Line<R1, R2>::CS + j] = times(v[k], w);
  }
}
template <int R1, int R2, int S, typename T>
__device__ __forceinline__ void second_dft(Cplx<T> *v, int k1, const Cplx<T> *s) {
#pragma unroll
  for (int j = 0; j < R2; ++j) v[j] = s[k1 * Line<R1, R2>::CS + j];
  Dft<R2, S, T>::run(v);
}

// Tile sizes: 16 lines (FP32) or 8 (FP64) per block in the x and y passes, so
// that the x pass stores whole 128-byte segments of y; TP line pairs in the z
// pass.  Threads: one first DFT each in the x and y passes.
template <typename T, int R1, int R2>
struct Tile {
  static constexpr bool f32 = sizeof(T) == 4;
  static constexpr int n = R1 * R2;
  static constexpr int RM = R1 > R2 ? R1 : R2;
  static constexpr int X = f32 ? 16 : 8;
  static constexpr int XT = (X * RM + 31) / 32 * 32;
  static constexpr int XI = f32 ? 8 : 4;  // rows of the inverse x pass (all three fields)
  static constexpr int XIT = (3 * XI * RM + 31) / 32 * 32 < 512 ? (3 * XI * RM + 31) / 32 * 32 : 256;
  // z pass: as many pairs as keep about four blocks per SM
  static constexpr size_t pair_bytes = (size_t)6 * Line<R1, R2>::LT * 2 * sizeof(T);
  static constexpr int TP = f32 ? (8 * pair_bytes <= 75 * 1024 ? 8 : 4) : (4 * pair_bytes <= 75 * 1024 ? 4 : 2);
  static constexpr int ZT = (6 * TP * RM + 31) / 32 * 32 <= 320 ? (6 * TP * RM + 31) / 32 * 32 : 288;
  static constexpr size_t xsm = (size_t)X * Line<R1, R2>::LT * 2 * sizeof(T);
  static constexpr size_t xism = (size_t)3 * XI * Line<R1, R2>::LT * 2 * sizeof(T);
  static constexpr size_t zsm = TP * pair_bytes;
};

// ---------------------------------------------------------------- x passes
template <typename T, int R1, int R2>
__global__ void __launch_bounds__(Tile<T, R1, R2>::XT)
    k_fft2_x_fwd(const T *__restrict__ grid, Cplx<T> *__restrict__ spec, const Cplx<T> *__restrict__ tw) {
  using L = Line<R1, R2>;
  constexpr int n = R1 * R2, X = Tile<T, R1, R2>::X, NT = Tile<T, R1, R2>::XT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<T> *sm = (Cplx<T> *)smem_raw;
  constexpr int64_t n3 = (int64_t)n * n * n;
  const int y0 = blockIdx.x * X, z = blockIdx.y, p = blockIdx.z;
  const T *ga = grid + p * n3 + ((int64_t)z * n + y0) * n, *gb = ga + 3 * n3;
  for (int b = threadIdx.x; b < X * R2; b += NT) {
    const int l = b / R2, j = b - l * R2;
    if (y0 + l < n) {
      Cplx<T> v[R1];
#pragma unroll
      for (int i = 0; i < R1; ++i) v[i] = {ga[l * n + j + R2 * i], gb[l * n + j + R2 * i]};
      first_dft<R1, R2, -1>(v, j, sm + l * L::LT, tw);
    }
  }
  __syncthreads();
  Cplx<T> *out = spec + p * n3 + (int64_t)z * n * n + y0;
  for (int b = threadIdx.x; b < X * R1; b += NT) {
    const int k1 = b / X, l = b - k1 * X;
    if (y0 + l < n) {
      Cplx<T> v[R2];
      second_dft<R1, R2, -1>(v, k1, sm + l * L::LT);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) out[(k1 + R1 * k2) * n + l] = v[k2];
    }
  }
}

// Inverse x pass of XI rows of a z plane, all three complex fields; the real
// and imaginary parts are the fields p and p + 3.
template <typename T, int R1, int R2>
__global__ void __launch_bounds__(Tile<T, R1, R2>::XIT)
    k_fft2_x_inv(const Cplx<T> *__restrict__ spec, T *__restrict__ out, const Cplx<T> *__restrict__ tw) {
  using L = Line<R1, R2>;
  constexpr int n = R1 * R2, X = Tile<T, R1, R2>::XI, NT = Tile<T, R1, R2>::XIT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<T> *sm = (Cplx<T> *)smem_raw;
  constexpr int64_t n3 = (int64_t)n * n * n;
  const int y0 = blockIdx.x * X, z = blockIdx.y;
  for (int b = threadIdx.x; b < 3 * X * R2; b += NT) {
    const int l = b % X, r = b / X, j = r % R2, p = r / R2;
    if (y0 + l < n) {
      const Cplx<T> *in = spec + p * n3 + ((int64_t)z * n + j) * n + y0 + l;
      Cplx<T> v[R1];
#pragma unroll
      for (int i = 0; i < R1; ++i) v[i] = in[(int64_t)R2 * i * n];
      first_dft<R1, R2, 1>(v, j, sm + (p * X + l) * L::LT, tw);
    }
  }
  __syncthreads();
  if constexpr (kFftBricks<T, n>) {
    // lanes take the four rows of a brick first, so that a store fills whole
    // 64-byte halves of bricks
    for (int b = threadIdx.x; b < 3 * X * R1; b += NT) {
      const int r = b >> 2, k1 = r % R1, q = r / R1, l = (q % (X / 4)) * 4 + (b & 3), p = q / (X / 4);
      if (y0 + l < n) {
        Cplx<T> v[R2];
        second_dft<R1, R2, 1>(v, k1, sm + (p * X + l) * L::LT);
        T *oa = out + p * n3 + ((int64_t)(z >> 1) * (n / 4) + (y0 + l) / 4) * (8 * n) + (z & 1) * 16 + (l & 3) * 4,
          *ob = oa + 3 * n3;
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) {
          const int x = k1 + R1 * k2, at = (x >> 2) * 32 + (x & 3);
          oa[at] = v[k2].x;
          ob[at] = v[k2].y;
        }
      }
    }
  } else if constexpr (sizeof(T) == 4) {
    for (int b = threadIdx.x; b < 3 * X * R1; b += NT) {
      const int k1 = b % R1, r = b / R1, l = r % X, p = r / X;
      if (y0 + l < n) {
        Cplx<T> v[R2];
        second_dft<R1, R2, 1>(v, k1, sm + (p * X + l) * L::LT);
        T *oa = out + p * n3 + ((int64_t)z * n + y0 + l) * n + k1, *ob = oa + 3 * n3;
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) {
          oa[R1 * k2] = v[k2].x;
          ob[R1 * k2] = v[k2].y;
        }
      }
    }
  } else {
    // the three fields of a point by neighbouring lanes
    for (int b = threadIdx.x; b < 3 * X * R1; b += NT) {
      const int p = b % 3, r = b / 3, k1 = r % R1, l = r / R1;
      if (y0 + l < n) {
        Cplx<T> v[R2];
        second_dft<R1, R2, 1>(v, k1, sm + (p * X + l) * L::LT);
        T *o = out + (((int64_t)z * n + y0 + l) * n + k1) * 8 + p;
#pragma unroll
        for (int k2 = 0; k2 < R2; ++k2) {
          o[8 * R1 * k2] = v[k2].x;
          o[8 * R1 * k2 + 3] = v[k2].y;
        }
      }
    }
  }
}

// ------------------------------------------------------------------ y pass
template <typename T, int R1, int R2, int S>
__global__ void __launch_bounds__(Tile<T, R1, R2>::XT)
    k_fft2_y(Cplx<T> *__restrict__ spec, const Cplx<T> *__restrict__ tw) {
  using L = Line<R1, R2>;
  constexpr int n = R1 * R2, X = Tile<T, R1, R2>::X, NT = Tile<T, R1, R2>::XT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<T> *sm = (Cplx<T> *)smem_raw;
  const int64_t l0 = (int64_t)blockIdx.x * X;
  const int nl = (int)(3LL * n * n - l0 < X ? 3LL * n * n - l0 : X);
  Cplx<T> *base = spec + l0 * n;
  for (int b = threadIdx.x; b < X * R2; b += NT) {
    const int l = b / R2, j = b - l * R2;
    if (l < nl) {
      Cplx<T> v[R1];
#pragma unroll
      for (int i = 0; i < R1; ++i) v[i] = base[l * n + j + R2 * i];
      first_dft<R1, R2, S>(v, j, sm + l * L::LC, tw);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < X * R1; b += NT) {
    const int l = b / R1, k1 = b - l * R1;
    if (l < nl) {
      Cplx<T> v[R2];
      second_dft<R1, R2, S>(v, k1, sm + l * L::LC);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) base[l * n + k1 + R1 * k2] = v[k2];
    }
  }
}

// --------------------------------------------------------- z pass + Green
// u = A(k) (I - kk) [..] for one wave vector: factors t (halved: the inputs
// are the unhalved sums gF = Z_k + conj Z_-k, gD = (Z_k - conj Z_-k) / i).
template <typename T>
__device__ __forceinline__ void green_apply(const T t[4], const T kk[3], const Cplx<T> *gF,
                                            const Cplx<T> *gD, Cplx<T> *uM, Cplx<T> *uD) {
  Cplx<T> sF = {T(0), T(0)}, sD = {T(0), T(0)};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    sF.x += kk[d] * gF[d].x;
    sF.y += kk[d] * gF[d].y;
    sD.x += kk[d] * gD[d].x;
    sD.y += kk[d] * gD[d].y;
  }
  sF = {sF.x * t[3], sF.y * t[3]};
  sD = {sD.x * t[3], sD.y * t[3]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const Cplx<T> pF = {gF[d].x - kk[d] * sF.x, gF[d].y - kk[d] * sF.y};
    const Cplx<T> pD = {gD[d].x - kk[d] * sD.x, gD[d].y - kk[d] * sD.y};
    uM[d] = {t[0] * pF.x + t[1] * pD.x, t[0] * pF.y + t[1] * pD.y};
    uD[d] = {t[1] * pF.x + t[2] * pD.x, t[1] * pF.y + t[2] * pD.y};
  }
}

__device__ __forceinline__ int signed_k(int i, int n) { return i <= n / 2 ? i : i - n; }

// halved Green factors and 1 / k^2 at grid index (kx <= n/2, y, z)
template <typename T, int n>
__device__ __forceinline__ void green_at(const ZGreen<T> &g, int kx, int y, int z, T t[4]) {
  const int ky = signed_k(y, n), kz = signed_k(z, n);
  const int m = kx * kx + ky * ky + kz * kz;
  if constexpr (sizeof(T) == 4) {
    if (g.gle) {
      const float4 v = __ldg((const float4 *)g.gle + (((int64_t)kx * n + z) * n + y));
      t[0] = v.x; t[1] = v.y; t[2] = v.z; t[3] = v.w;
    } else {
      const float *q = g.green + 3 * m;
      t[0] = __ldg(q); t[1] = __ldg(q + 1); t[2] = __ldg(q + 2); t[3] = 1.f / (float)m;
    }
  } else {
    const double2 *q = (const double2 *)(g.gle ? g.gle + 4 * (((int64_t)kx * n + z) * n + y) : g.green + 4 * m);
    const double2 u = __ldg(q), v = __ldg(q + 1);
    t[0] = u.x; t[1] = u.y; t[2] = v.x; t[3] = v.y;
  }
}

// random field (I - kk) xi(k) (c fM, c fD) at grid index (kx <= n/2, y, z)
template <typename T, int n>
__device__ __forceinline__ void brown_at(const ZBrown<T> &g, int kx, int y, int z, Cplx<T> *oM,
                                         Cplx<T> *oD) {
  constexpr int nh = n / 2 + 1;
#pragma unroll
  for (int c = 0; c < 3; ++c) oM[c] = oD[c] = {T(0), T(0)};
  if (kx == n / 2 || y == n / 2 || z == n / 2 || (kx | y | z) == 0) return;
  double xr[3], xi_[3];
  if (g.field) {
    const int64_t cs = (int64_t)n * n * nh, o = ((int64_t)z * n + y) * nh + kx;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      xr[c] = g.field[2 * (c * cs + o)];
      xi_[c] = g.field[2 * (c * cs + o) + 1];
    }
  } else {
    int cz = z, cy = y;
    bool conj = false;
    if (kx == 0) {  // one of each Hermitian pair draws
      const int mz = (n - z) % n, my = (n - y) % n;
      if (mz < z || (mz == z && my < y)) {
        cz = mz;
        cy = my;
        conj = true;
      }
    }
    const uint32_t idx = (uint32_t)(((int64_t)cz * n + cy) * nh + kx);
    double z0[4], z1[4];
    philox_normals4(g.seed, g.step, 1u, 0u, idx, z0);
    philox_normals4(g.seed, g.step, 1u, 1u, idx, z1);
    const double s = 0.70710678118654752440, sc = conj ? -s : s;
    xr[0] = s * z0[0]; xi_[0] = sc * z0[1];
    xr[1] = s * z0[2]; xi_[1] = sc * z0[3];
    xr[2] = s * z1[0]; xi_[2] = sc * z1[1];
  }
  const int ky = signed_k(y, n), kz = signed_k(z, n);
  const int m0 = kx * kx + ky * ky + kz * kz;
  const double kk[3] = {(double)kx, (double)ky - g.tau * (double)kx, (double)kz};
  const double m = kk[0] * kk[0] + kk[1] * kk[1] + kk[2] * kk[2];
  double pr = 0.0, pi = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    pr += kk[c] * xr[c];
    pi += kk[c] * xi_[c];
  }
  T bm, bd;
  if (g.tau == 0.0) {
    bm = g.btab[2 * m0];
    bd = g.btab[2 * m0 + 1];
  } else {
    const double k2 = g.ks2 * m, q = k2 / (4.0 * g.xi * g.xi);
    const double H = (1.0 + q) * exp(-q);
    const double sc = sqrt(H / (g.eta * k2)) * exp(g.ks2 * m0 / (4.0 * g.alpha)) * g.isv;
    const double ka = sqrt(k2) * g.a;
    const double fm = ka < 1e-3 ? 1.0 - ka * ka / 6.0 + ka * ka * ka * ka / 120.0 : sin(ka) / ka;
    const double fd = ka < 1e-2 ? 1.0 - ka * ka / 10.0 + ka * ka * ka * ka / 280.0
                                : 3.0 * (sin(ka) - ka * cos(ka)) / (ka * ka * ka);
    bm = (T)(sc * fm);
    bd = (T)(sc * fd);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const T vr = (T)(xr[c] - kk[c] * pr / m), vi = (T)(xi_[c] - kk[c] * pi / m);
    oM[c] = {bm * vr, bm * vi};
    oD[c] = {bd * vr, bd * vi};
  }
}

// One block: the lines (kx, ky) and (-kx, -ky) of TP consecutive ky at one
// kx <= n/2, all three complex fields: forward z transform, Green's function
// on the pairs (k, -k), inverse z transform, in place.  Fields at -k follow
// as conjugates (real fields) except in the planes kx = 0 and n/2, where both
// members of a pair are grid points of the half spectrum and each takes the
// wave vector of its own index (they differ at the Nyquist planes, whose
// index stands for both signs).  BROWN: the random field instead of the
// forward transform and the Green's function.
template <typename T, int R1, int R2, bool BROWN>
__global__ void __launch_bounds__(Tile<T, R1, R2>::ZT)
    k_fft2_z(Cplx<T> *__restrict__ spec, const Cplx<T> *__restrict__ tw, const ZGreen<T> g, const ZBrown<T> br) {
  using L = Line<R1, R2>;
  constexpr int n = R1 * R2, TP = Tile<T, R1, R2>::TP, NT = Tile<T, R1, R2>::ZT;
  constexpr int n2 = n * n;
  constexpr int64_t n3 = (int64_t)n2 * n;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Cplx<T> *sm = (Cplx<T> *)smem_raw;
  const int kx = blockIdx.y, ky0 = blockIdx.x * TP;
  const bool special = kx == 0 || kx == n / 2;
  const int kend = special ? n / 2 + 1 : n;  // pairs of the special planes meet twice
  if (ky0 >= kend) return;
  // global offset of line t, side s (0: (kx, ky), 1: (-kx, -ky))
  auto line_off = [&](int s, int t) {
    const int ky = ky0 + t;
    if (s == 0) return kx * n + ky;
    return (kx == 0 ? 0 : n - kx) * n + (ky == 0 ? 0 : n - ky);
  };
  if (!BROWN) {
    for (int b = threadIdx.x; b < 6 * TP * R2; b += NT) {
      const int t = b % TP, r = b / TP, j = r % R2, ps = r / R2;  // ps = 2 p + s
      if (ky0 + t < kend) {
        const Cplx<T> *in = spec + (ps >> 1) * n3 + line_off(ps & 1, t) + (int64_t)j * n2;
        Cplx<T> v[R1];
#pragma unroll
        for (int i = 0; i < R1; ++i) v[i] = in[(int64_t)R2 * i * n2];
        first_dft<R1, R2, -1>(v, j, sm + (ps * TP + t) * L::LT, tw);
      }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 6 * TP * R1; b += NT) {
      const int t = b % TP, r = b / TP, k1 = r % R1, ps = r / R1;
      Cplx<T> *s = sm + (ps * TP + t) * L::LT;
      Cplx<T> v[R2];
      second_dft<R1, R2, -1>(v, k1, s);
      // kz = k1 + R1 k2 stays in the thread's own chunk, at (k1, k2)
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) s[k1 * L::CS + k2] = v[k2];
    }
    __syncthreads();
  }
  // a thread keeps its ky: the physical y component (FP64, rounded once) is
  // found once, and 1 / k^2 comes with the factors: in FP32 these few FP64
  // operations per point were a fifth of the pass in a Lees-Edwards box (n = 144:
  // 66 -> 52 us; in FP64 1.06 -> 0.96 ms)
  static_assert(NT % TP == 0, "a thread stays on one ky");
  const int t = threadIdx.x % TP, ky = ky0 + t, my = ky == 0 ? 0 : n - ky;
  T kk[3] = {(T)kx, (T)signed_k(ky, n), T(0)}, kyb = (T)signed_k(my, n);
  if (!BROWN && g.gle) {
    const double tau = g.tilt_dev ? *g.tilt_dev * g.invL : g.tau;
    kk[1] = (T)((double)signed_k(ky, n) - tau * (double)kx);
    kyb = (T)((double)signed_k(my, n) - tau * (double)kx);
  }
  for (int e = threadIdx.x; e < TP * n; e += NT) {
    const int q = e / TP;
    if (ky >= kend) continue;
    const int k1 = q % R1, k2 = q / R1, kz = k1 + R1 * k2;
    const int mz = kz == 0 ? 0 : n - kz;
    Cplx<T> *A = sm + t * L::LT + k1 * L::CS + k2;
    Cplx<T> *B = sm + (TP + t) * L::LT + (mz % R1) * L::CS + mz / R1;
    constexpr int ps = 2 * TP * L::LT;  // from field p to p + 1
    Cplx<T> uM[3], uD[3], vM[3], vD[3];
    if (BROWN) {
      brown_at<T, n>(br, kx, ky, kz, uM, uD);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        vM[d] = {uM[d].x, -uM[d].y};
        vD[d] = {uD[d].x, -uD[d].y};
      }
      if (special) brown_at<T, n>(br, kx, my, mz, vM, vD);
    } else {
      Cplx<T> gF[3], gD[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const Cplx<T> a = A[d * ps], b = B[d * ps];
        gF[d] = {a.x + b.x, a.y - b.y};
        gD[d] = {a.y + b.y, b.x - a.x};
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) uM[d] = uD[d] = {T(0), T(0)};
      T tf[4];
      const bool zero = (kx | ky | kz) == 0;
      kk[2] = (T)signed_k(kz, n);
      if (!zero) {
        green_at<T, n>(g, kx, ky, kz, tf);
        green_apply<T>(tf, kk, gF, gD, uM, uD);
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        vM[d] = {uM[d].x, -uM[d].y};
        vD[d] = {uD[d].x, -uD[d].y};
      }
      if (special && !zero) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          gF[d].y = -gF[d].y;
          gD[d].y = -gD[d].y;
        }
        const T kb[3] = {kk[0], kyb, (T)signed_k(mz, n)};
        green_at<T, n>(g, kx, my, mz, tf);
        green_apply<T>(tf, kb, gF, gD, vM, vD);
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      A[d * ps] = {uM[d].x - uD[d].y, uM[d].y + uD[d].x};
      B[d * ps] = {vM[d].x - vD[d].y, vM[d].y + vD[d].x};
    }
  }
  __syncthreads();
  // inverse: k = k1 + R1 k2, first over k2 (in the chunk), then over k1
  for (int b = threadIdx.x; b < 6 * TP * R1; b += NT) {
    const int t = b % TP, r = b / TP, k1 = r % R1, ps = r / R1;
    Cplx<T> *s = sm + (ps * TP + t) * L::LT + k1 * L::CS;
    Cplx<T> v[R2];
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = s[k2];
    Dft<R2, 1, T>::run(v);
    s[0] = v[0];
#pragma unroll
    for (int j = 1; j < R2; ++j) {
      Cplx<T> w = tw[k1 * R2 + j];
      w.y = -w.y;
      s[j] = times(v[j], w);
    }
  }
  __syncthreads();
  for (int b = threadIdx.x; b < 6 * TP * R2; b += NT) {
    const int t = b % TP, r = b / TP, j = r % R2, ps = r / R2;
    const int ky = ky0 + t;
    // a line that is its own partner is stored once
    if (ky >= kend || ((ps & 1) && special && (ky == 0 || ky == n / 2))) continue;
    const Cplx<T> *s = sm + (ps * TP + t) * L::LT + j;
    Cplx<T> v[R1];
#pragma unroll
    for (int k = 0; k < R1; ++k) v[k] = s[k * L::CS];
    Dft<R1, 1, T>::run(v);
    Cplx<T> *out = spec + (ps >> 1) * n3 + line_off(ps & 1, t) + (int64_t)j * n2;
#pragma unroll
    for (int i = 0; i < R1; ++i) out[(int64_t)R2 * i * n2] = v[i];
  }
}

// ---------------------------------------------------------------- launchers
template <typename T, int R1, int R2>
struct FftLaunch {
  using W = Tile<T, R1, R2>;
  static constexpr int n = R1 * R2;
  static void x_fwd(cudaStream_t st, const T *grid, Cplx<T> *spec, const Cplx<T> *tw) {
    if (W::xsm > 48 * 1024) raise_smem((const void *)k_fft2_x_fwd<T, R1, R2>, W::xsm);
    k_fft2_x_fwd<T, R1, R2><<<dim3((n + W::X - 1) / W::X, n, 3), W::XT, W::xsm, st>>>(grid, spec, tw);
  }
  static void y_pass(cudaStream_t st, Cplx<T> *spec, const Cplx<T> *tw, bool inverse) {
    const int blocks = (3 * n * n + W::X - 1) / W::X;
    if (W::xsm > 48 * 1024)
      raise_smem(inverse ? (const void *)k_fft2_y<T, R1, R2, 1> : (const void *)k_fft2_y<T, R1, R2, -1>, W::xsm);
    if (inverse)
      k_fft2_y<T, R1, R2, 1><<<blocks, W::XT, W::xsm, st>>>(spec, tw);
    else
      k_fft2_y<T, R1, R2, -1><<<blocks, W::XT, W::xsm, st>>>(spec, tw);
  }
  static void z_green(cudaStream_t st, Cplx<T> *spec, const Cplx<T> *tw, const ZGreen<T> &g) {
    if (W::zsm > 48 * 1024) raise_smem((const void *)k_fft2_z<T, R1, R2, false>, W::zsm);
    k_fft2_z<T, R1, R2, false><<<dim3((n + W::TP - 1) / W::TP, n / 2 + 1), W::ZT, W::zsm, st>>>(spec, tw, g,
                                                                                            ZBrown<T>());
  }
  static void z_brown(cudaStream_t st, Cplx<T> *spec, const Cplx<T> *tw, const ZBrown<T> &b) {
    if (W::zsm > 48 * 1024) raise_smem((const void *)k_fft2_z<T, R1, R2, true>, W::zsm);
    k_fft2_z<T, R1, R2, true><<<dim3((n + W::TP - 1) / W::TP, n / 2 + 1), W::ZT, W::zsm, st>>>(spec, tw,
                                                                                           ZGreen<T>(), b);
  }
  static void x_inv(cudaStream_t st, const Cplx<T> *spec, T *out, const Cplx<T> *tw) {
    if (W::xism > 48 * 1024) raise_smem((const void *)k_fft2_x_inv<T, R1, R2>, W::xism);
    k_fft2_x_inv<T, R1, R2><<<dim3((n + W::XI - 1) / W::XI, n), W::XIT, W::xism, st>>>(spec, out, tw);
  }
  static const FftOps<T> *ops() {
    static const FftOps<T> o = {n, R1, R2, x_fwd, y_pass, z_green, z_brown, x_inv};
    return &o;
  }
};

#endif  // FSD_FFT_KERNELS

}  // namespace fsd
