// Three-dimensional real transforms of the six field components, and the
// Green operator fused between the last forward and the first inverse pass.
//
// A library transform is three passes each way with the Green operator as a
// seventh pass between them, one job at a time.  Here the x pass, the Green
// update and the inverse x pass are one kernel: the six components of a column
// of modes stay in shared memory, so the spectra make one round trip less.
// Where an x plane fits, the z and y passes are one kernel too.  All jobs of
// one grid size go in one launch per pass.
//
// Bound: FP32 the memory, FP64 the FP64 pipe (a 256-point line takes about 6000
// operations in two radix-16 stages).  Measured on GB300 against cuFFT with the
// separate Green kernel, one iteration's transforms and update: FP32 256^3
// 1.21 -> 1.00 ms, FP64 256^3 22.6 -> 14.9 ms; with the smaller chunks of the
// reductions the 16^3 FP64 iteration 400 -> 44 us.
//
// Layout (as cuFFT's): real [6][N][N][N], spectrum [6][N][N][Nh], Nh = N/2 + 1,
// unnormalised both ways; the forward passes give twice the spectrum (the
// separation of the two lines of a z pair leaves out its factor 1/2, an exact
// scaling that the constants of what follows take).  N = R1 R2, both among the
// radices below (at most 16), N even: the sizes listed in fft_f32*.cu and
// fft_f64*.cu.  Other sizes (factors of 7, N > 256, even sizes not listed) take
// cuFFT.
//
// One line of N = R1 R2 points by two register stages and one exchange
// through shared memory (n = n1 R2 + n2, k = k1 + R1 k2):
//   X[k] = sum_n2 w_N^(n2 k1) w_R2^(n2 k2) sum_n1 x[n] w_R1^(n1 k1).
// A thread holds R1 (first stage) or R2 (second) points, max(R1, R2) threads
// a line.  The inverse runs the stages in the other order, so the column
// kernel needs no reordering between its forward and its inverse transform.
// z pass: two real lines of the same component as one complex line.
//
// Green operator of the isotropic reference medium (lambda0, mu0), applied to
// a symmetric tau with q = tau k (homogeneous of degree 0 in k):
//   (Gamma0 : tau)_ij = (k_j q_i + k_i q_j) / (2 mu0 |k|^2)
//                       - (lambda0 + mu0) / (mu0 (lambda0 + 2 mu0)) (k.q) k_i k_j / |k|^4.
#pragma once

#include "fft.h"
#include "ms_kernels.cuh"

namespace gsm {
namespace {

// ------------------------------------------------------- register transforms

template <class T> struct cx {
  T x, y;
};
template <class T> __device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return {a.x + b.x, a.y + b.y}; }
template <class T> __device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return {a.x - b.x, a.y - b.y}; }
template <class T> __device__ __forceinline__ cx<T> cmul(cx<T> a, T c, T s) {  // a (c + i s)
  return {a.x * c - a.y * s, a.x * s + a.y * c};
}
// a * (-i) forward, a * (+i) inverse
template <bool INV, class T> __device__ __forceinline__ cx<T> rot(cx<T> a) {
  if constexpr (INV) return {-a.y, a.x};
  else return {a.y, -a.x};
}

// cos(2 pi m / 16), m = 0..4
__host__ __device__ constexpr double cos16(int m) {
  return m == 0 ? 1.0 : m == 1 ? 0.92387953251128675613 : m == 2 ? 0.70710678118654752440
                                  : m == 3 ? 0.38268343236508977173 : 0.0;
}
__host__ __device__ constexpr double cos16f(int m) {  // any m
  m &= 15;
  return m <= 4 ? cos16(m) : m <= 8 ? -cos16(8 - m) : m <= 12 ? -cos16(m - 8) : cos16(16 - m);
}
__host__ __device__ constexpr double sin16f(int m) { return cos16f(m + 12); }

constexpr int inverse_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if (a * i % m == 1) return i;
  return 1;
}

template <int R, bool INV, class T> struct Dft;

template <bool INV, class T> struct Dft<1, INV, T> {
  static __device__ __forceinline__ void run(cx<T> (&)[1]) {}
};
template <bool INV, class T> struct Dft<2, INV, T> {
  static __device__ __forceinline__ void run(cx<T> (&a)[2]) {
    const cx<T> t = a[0] - a[1];
    a[0] = a[0] + a[1];
    a[1] = t;
  }
};
template <bool INV, class T> struct Dft<3, INV, T> {
  static __device__ __forceinline__ void run(cx<T> (&a)[3]) {
    constexpr T s3 = T(0.86602540378443864676);
    const cx<T> t = a[1] + a[2], d = rot<INV>(a[1] - a[2]);
    const cx<T> m = {a[0].x - T(0.5) * t.x, a[0].y - T(0.5) * t.y};
    a[0] = a[0] + t;
    a[1] = {m.x + s3 * d.x, m.y + s3 * d.y};
    a[2] = {m.x - s3 * d.x, m.y - s3 * d.y};
  }
};
template <bool INV, class T> struct Dft<4, INV, T> {
  static __device__ __forceinline__ void run(cx<T> (&a)[4]) {
    const cx<T> s02 = a[0] + a[2], d02 = a[0] - a[2], s13 = a[1] + a[3], d13 = rot<INV>(a[1] - a[3]);
    a[0] = s02 + s13;
    a[1] = d02 + d13;
    a[2] = s02 - s13;
    a[3] = d02 - d13;
  }
};
template <bool INV, class T> struct Dft<5, INV, T> {
  static __device__ __forceinline__ void run(cx<T> (&a)[5]) {
    constexpr T c1 = T(0.30901699437494742410), c2 = T(-0.80901699437494742410);
    constexpr T s1 = T(0.95105651629515357212), s2 = T(0.58778525229247312917);
    const cx<T> t1 = a[1] + a[4], t2 = a[2] + a[3], d1 = rot<INV>(a[1] - a[4]), d2 = rot<INV>(a[2] - a[3]);
    const cx<T> m1 = {a[0].x + c1 * t1.x + c2 * t2.x, a[0].y + c1 * t1.y + c2 * t2.y};
    const cx<T> m2 = {a[0].x + c2 * t1.x + c1 * t2.x, a[0].y + c2 * t1.y + c1 * t2.y};
    const cx<T> n1 = {s1 * d1.x + s2 * d2.x, s1 * d1.y + s2 * d2.y};
    const cx<T> n2 = {s2 * d1.x - s1 * d2.x, s2 * d1.y - s1 * d2.y};
    a[0] = a[0] + t1 + t2;
    a[1] = m1 + n1;
    a[4] = m1 - n1;
    a[2] = m2 + n2;
    a[3] = m2 - n2;
  }
};

// R = A B by the twiddled (Cooley-Tukey) split, R in {8, 16}.
template <int A, int B, bool INV, class T> struct DftCT {
  static constexpr int R = A * B;
  static __device__ __forceinline__ void run(cx<T> (&a)[R]) {
    cx<T> b[B][A];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) b[n2][n1] = a[n1 * B + n2];
      Dft<A, INV, T>::run(b[n2]);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) {
        const int m = n2 * k1 * (16 / R);
        if (m == 0) continue;
        if (m == 4) {
          b[n2][k1] = rot<INV>(b[n2][k1]);
        } else {
          const T c = T(cos16f(m)), s = T(sin16f(m));
          b[n2][k1] = cmul(b[n2][k1], c, INV ? s : -s);
        }
      }
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      cx<T> v[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) v[n2] = b[n2][k1];
      Dft<B, INV, T>::run(v);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) a[k1 + A * k2] = v[k2];
    }
  }
};
template <bool INV, class T> struct Dft<8, INV, T> : DftCT<2, 4, INV, T> {};
template <bool INV, class T> struct Dft<16, INV, T> : DftCT<4, 4, INV, T> {};

// R = A B with A, B coprime by the prime-factor (Good-Thomas) map: no twiddles.
template <int A, int B, bool INV, class T> struct DftPFA {
  static constexpr int R = A * B;
  static __device__ __forceinline__ void run(cx<T> (&a)[R]) {
    constexpr int ia = inverse_mod(A % B, B), ib = inverse_mod(B % A, A);
    cx<T> b[B][A];
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) b[n2][n1] = a[(B * n1 + A * n2) % R];
      Dft<A, INV, T>::run(b[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) {
      cx<T> v[B];
#pragma unroll
      for (int n2 = 0; n2 < B; ++n2) v[n2] = b[n2][k1];
      Dft<B, INV, T>::run(v);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) a[(B * ib * k1 + A * ia * k2) % R] = v[k2];
    }
  }
};
template <bool INV, class T> struct Dft<6, INV, T> : DftPFA<2, 3, INV, T> {};
template <bool INV, class T> struct Dft<10, INV, T> : DftPFA<2, 5, INV, T> {};
template <bool INV, class T> struct Dft<12, INV, T> : DftPFA<3, 4, INV, T> {};
template <bool INV, class T> struct Dft<15, INV, T> : DftPFA<3, 5, INV, T> {};

// ------------------------------------------------------------------- shapes

// The split of N: the two factors as near to each other as the radices allow.
template <int N> struct Split {
  static constexpr bool radix(int r) {
    return r == 2 || r == 3 || r == 4 || r == 5 || r == 6 || r == 8 || r == 10 || r == 12 || r == 15 || r == 16;
  }
  static constexpr int pick() {
    for (int d = 0; d < 16; ++d)
      for (int r = 2; r <= 16; ++r)
        if (N % r == 0 && radix(r) && radix(N / r) && N / r >= r && N / r - r == d) return r;
    return 0;
  }
  static constexpr int R1 = pick(), R2 = R1 ? N / R1 : 0;
  static_assert(R1 > 0, "N is not a product of two radices");
};

// Threads and shared memory of the kernels (complex elements).
template <class T, int N> struct Shape {
  static constexpr int R1 = Split<N>::R1, R2 = Split<N>::R2, TPL = R2;  // R2 >= R1
  static constexpr int Nh = N / 2 + 1, PITCH = R2 + 1;                   // padded: no bank conflicts
  // z: pairs of lines per block
  static constexpr int LP = (sizeof(T) == 4 ? 256 : 128) / TPL;
  static constexpr int ZLINE = R1 * PITCH > N ? R1 * PITCH : N;
  static constexpr size_t z_smem = (size_t)LP * ZLINE * sizeof(cx<T>);
  // z and y passes of one x plane of a component together: rows of PP elements,
  // two rows hold the exchange of a z pair
  static constexpr int PP = ((N + R1 + 1) / 2 > Nh ? (N + R1 + 1) / 2 : Nh) | 1;
  static constexpr size_t p_smem = (size_t)N * PP * sizeof(cx<T>);
  static constexpr int PL = 512 / TPL < N / 2 ? 512 / TPL : N / 2;  // z pairs at a time
  static constexpr int PT = PL * TPL, PW = PL;                      // threads; columns at a time
  static constexpr bool plane = N <= (sizeof(T) == 4 ? 64 : 24);
  // columns of the y (and plain x) pass: 128-byte rows
  static constexpr int W = 128 / (int)sizeof(cx<T>);
  static constexpr size_t c_smem = (size_t)R1 * PITCH * W * sizeof(cx<T>);
  // columns of the Green pass: the six components together in shared memory,
  // CG of them at a time in registers.  Two at a time leave room for several
  // blocks an SM, whose phases then overlap (FP32 128^3 66 -> 45 us, FP64 256^3
  // 5.75 -> 5.57 ms against all six at once); where a block takes more than
  // half an SM's shared memory anyway (FP32, N > 200) all six at once are
  // faster (256^3: 445 against 503 us).
  static constexpr int GW = (sizeof(T) == 4 ? 8 : 4), CG = (sizeof(T) == 4 && N > 200) || 6 * TPL * GW <= 256 ? 6 : 2;
  static constexpr int GL = CG * TPL * GW;            // threads that hold lines
  static constexpr int GT = (GL + 31) / 32 * 32;       // whole warps (the block sum)
  static constexpr size_t g_smem = (size_t)6 * R1 * PITCH * GW * sizeof(cx<T>);
};

template <class T> __device__ __forceinline__ cx<T> tw_ld(const cx<T>* tw, int m) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(tw) + m);
    return {v.x, v.y};
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(tw) + m);
    return {v.x, v.y};
  }
}
template <class T> __device__ __forceinline__ cx<T> hat_ld(const cx<T>* p) {
  if constexpr (sizeof(T) == 4) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    return {v.x, v.y};
  } else {
    const double2 v = *reinterpret_cast<const double2*>(p);
    return {v.x, v.y};
  }
}
template <class T> __device__ __forceinline__ void hat_st(cx<T>* p, cx<T> v) {
  if constexpr (sizeof(T) == 4) *reinterpret_cast<float2*>(p) = make_float2(v.x, v.y);
  else *reinterpret_cast<double2*>(p) = make_double2(v.x, v.y);
}

// Stage 1 of the forward line transform on registers: DFT over n1 and twiddle.
// tw[m] = exp(-2 pi i m / N).
template <class T, int N> __device__ __forceinline__ void line_fwd1(cx<T> (&a)[Split<N>::R1], int n2, const cx<T>* tw) {
  Dft<Split<N>::R1, false, T>::run(a);
#pragma unroll
  for (int k1 = 1; k1 < Split<N>::R1; ++k1) {
    const cx<T> w = tw_ld(tw, n2 * k1);
    a[k1] = cmul(a[k1], w.x, w.y);
  }
}
// Stage 1 of the inverse: DFT over k2 and conjugate twiddle.
template <class T, int N> __device__ __forceinline__ void line_inv1(cx<T> (&a)[Split<N>::R2], int k1, const cx<T>* tw) {
  Dft<Split<N>::R2, true, T>::run(a);
#pragma unroll
  for (int n2 = 1; n2 < Split<N>::R2; ++n2) {
    const cx<T> w = tw_ld(tw, n2 * k1);
    a[n2] = cmul(a[n2], w.x, -w.y);
  }
}

// ------------------------------------------------------------------ z passes

// Real lines -> half spectra, two lines of a component per complex line.
// grid: jobs x tiles of LP pairs.  views == NULL: one job, in -> hat.
template <class T, int N>
__global__ void __launch_bounds__(Shape<T, N>::LP* Shape<T, N>::TPL)
    fft_z_fwd(const JobView* __restrict__ views, JobList list, const T* in, cx<T>* hat, const cx<T>* __restrict__ tw) {
  using S = Shape<T, N>;
  constexpr int pairs = 3 * N * N, tiles = (pairs + S::LP - 1) / S::LP;
  extern __shared__ __align__(16) unsigned char smem_[];
  const int t = threadIdx.x % S::TPL, l = threadIdx.x / S::TPL;
  cx<T>* s = reinterpret_cast<cx<T>*>(smem_) + l * S::ZLINE;
  if (views) {
    const JobView& v = views[list.at[blockIdx.x / tiles]];
    in = static_cast<const T*>(v.sig);
    hat = static_cast<cx<T>*>(v.sig_hat);
  }
  const int p = (int)(blockIdx.x % tiles) * S::LP + l;
  const bool ok = p < pairs;
  const int64_t line = 2 * (int64_t)p;
  if (ok) {
    const T* x = in + line * N;
    cx<T> a[S::R1];
#pragma unroll
    for (int n1 = 0; n1 < S::R1; ++n1) a[n1] = {__ldg(x + n1 * S::R2 + t), __ldg(x + N + n1 * S::R2 + t)};
    line_fwd1<T, N>(a, t, tw);
#pragma unroll
    for (int k1 = 0; k1 < S::R1; ++k1) s[k1 * S::PITCH + t] = a[k1];
  }
  __syncthreads();
  // (second stage: R1 threads a line, whole warps of them)
  const int t2 = threadIdx.x % S::R1, l2 = threadIdx.x / S::R1;
  const bool ok2 = l2 < S::LP && p - l + l2 < pairs;
  cx<T>* s2 = reinterpret_cast<cx<T>*>(smem_) + l2 * S::ZLINE;
  cx<T> b[S::R2];
  if (ok2) {
#pragma unroll
    for (int n2 = 0; n2 < S::R2; ++n2) b[n2] = s2[t2 * S::PITCH + n2];
    Dft<S::R2, false, T>::run(b);
  }
  __syncthreads();
  if (ok2) {
#pragma unroll
    for (int k2 = 0; k2 < S::R2; ++k2) s2[t2 + S::R1 * k2] = b[k2];
  }
  __syncthreads();
  if (ok) {
    cx<T>* A = hat + line * S::Nh;
    for (int k = t; k < S::Nh; k += S::TPL) {
      const cx<T> z = s[k], y = s[k ? N - k : 0];
      hat_st<T>(A + k, {z.x + y.x, z.y - y.y});
      hat_st<T>(A + S::Nh + k, {z.y + y.y, y.x - z.x});
    }
  }
}

// Half spectra -> real lines.
template <class T, int N>
__global__ void __launch_bounds__(Shape<T, N>::LP* Shape<T, N>::TPL)
    fft_z_inv(const JobView* __restrict__ views, JobList list, const cx<T>* hat, T* out, const cx<T>* __restrict__ tw) {
  using S = Shape<T, N>;
  constexpr int pairs = 3 * N * N, tiles = (pairs + S::LP - 1) / S::LP;
  extern __shared__ __align__(16) unsigned char smem_[];
  const int t = threadIdx.x % S::TPL, l = threadIdx.x / S::TPL;
  cx<T>* s = reinterpret_cast<cx<T>*>(smem_) + l * S::ZLINE;
  if (views) {
    const JobView& v = views[list.at[blockIdx.x / tiles]];
    hat = static_cast<const cx<T>*>(v.sig_hat);
    out = static_cast<T*>(v.eps_out);
  }
  const int p = (int)(blockIdx.x % tiles) * S::LP + l;
  const bool ok = p < pairs;
  const int64_t line = 2 * (int64_t)p;
  if (ok) {
    const cx<T>* A = hat + line * S::Nh;
    constexpr int KI = (S::Nh + S::TPL - 1) / S::TPL;
    cx<T> ra[KI], rb[KI];  // every load in flight before the first is used
#pragma unroll
    for (int i = 0; i < KI; ++i) {
      const int k = t + i * S::TPL;
      if (k < S::Nh) {
        ra[i] = hat_ld(A + k);
        rb[i] = hat_ld(A + S::Nh + k);
      }
    }
#pragma unroll
    for (int i = 0; i < KI; ++i) {
      const int k = t + i * S::TPL;
      const cx<T> a = ra[i], b = rb[i];
      if (k >= S::Nh) {
      } else if (k == 0 || k == N / 2) {
        s[k] = {a.x, b.x};  // the imaginary parts of a real line's k = 0 and N/2 modes do not enter
      } else {
        s[k] = {a.x - b.y, a.y + b.x};
        s[N - k] = {a.x + b.y, b.x - a.y};
      }
    }
  }
  __syncthreads();
  const int t2 = threadIdx.x % S::R1, l2 = threadIdx.x / S::R1;
  const bool ok2 = l2 < S::LP && p - l + l2 < pairs;
  cx<T>* s2 = reinterpret_cast<cx<T>*>(smem_) + l2 * S::ZLINE;
  cx<T> b[S::R2];
  if (ok2) {
#pragma unroll
    for (int k2 = 0; k2 < S::R2; ++k2) b[k2] = s2[t2 + S::R1 * k2];
    line_inv1<T, N>(b, t2, tw);
  }
  __syncthreads();
  if (ok2) {
#pragma unroll
    for (int n2 = 0; n2 < S::R2; ++n2) s2[t2 * S::PITCH + n2] = b[n2];
  }
  __syncthreads();
  if (ok) {
    T* x = out + line * N;
    cx<T> a[S::R1];
#pragma unroll
    for (int k1 = 0; k1 < S::R1; ++k1) a[k1] = s[k1 * S::PITCH + t];
    Dft<S::R1, true, T>::run(a);
#pragma unroll
    for (int n1 = 0; n1 < S::R1; ++n1) {
      x[n1 * S::R2 + t] = a[n1].x;
      x[N + n1 * S::R2 + t] = a[n1].y;
    }
  }
}

// ----------------------------------------------------- z and y passes together

// Both passes of one x plane of one component in shared memory: one launch and
// one round trip of the spectrum less each way.  For small grids, where the
// launches and the latency count (z + y against the one kernel, us: FP32 32^3
// 8.0 -> 5.0, 64^3 12.4 -> 8.4, 96^3 24.6 -> 26; FP64 16^3 10.4 -> 8.3, 32^3
// 17.8 -> 19.4, 64^3 70 -> 98: there the block's serial phases leave the FP64
// pipe idle).  grid: jobs x 6 N planes.
template <class T, int N>
__global__ void __launch_bounds__(Shape<T, N>::PT)
    fft_zy_fwd(const JobView* __restrict__ views, JobList list, const T* in, cx<T>* hat, const cx<T>* __restrict__ tw) {
  using S = Shape<T, N>;
  extern __shared__ __align__(16) unsigned char smem_[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_);
  const int pl = blockIdx.x % (6 * N);
  if (views) {
    const JobView& v = views[list.at[blockIdx.x / (6 * N)]];
    in = static_cast<const T*>(v.sig);
    hat = static_cast<cx<T>*>(v.sig_hat);
  }
  in += (int64_t)pl * N * N;
  hat += (int64_t)pl * N * S::Nh;
  {
    const int t = threadIdx.x % S::TPL, l0 = threadIdx.x / S::TPL;
    constexpr int KI = (S::Nh + S::TPL - 1) / S::TPL;
    for (int base = 0; base < N / 2; base += S::PL) {
      const int l = base + l0;
      const bool ok = l < N / 2;
      cx<T>* s = sm + 2 * l * S::PP;
      if (ok) {
        const T* x = in + 2 * l * N;
        cx<T> a[S::R1];
#pragma unroll
        for (int n1 = 0; n1 < S::R1; ++n1) a[n1] = {__ldg(x + n1 * S::R2 + t), __ldg(x + N + n1 * S::R2 + t)};
        line_fwd1<T, N>(a, t, tw);
#pragma unroll
        for (int k1 = 0; k1 < S::R1; ++k1) s[k1 * S::PITCH + t] = a[k1];
      }
      __syncthreads();
      cx<T> b[S::R2];
      if (ok && t < S::R1) {
#pragma unroll
        for (int n2 = 0; n2 < S::R2; ++n2) b[n2] = s[t * S::PITCH + n2];
        Dft<S::R2, false, T>::run(b);
      }
      __syncthreads();
      if (ok && t < S::R1) {
#pragma unroll
        for (int k2 = 0; k2 < S::R2; ++k2) s[t + S::R1 * k2] = b[k2];
      }
      __syncthreads();
      cx<T> z[KI], y[KI];
#pragma unroll
      for (int i = 0; i < KI; ++i) {
        const int k = t + i * S::TPL;
        if (ok && k < S::Nh) {
          z[i] = s[k];
          y[i] = s[k ? N - k : 0];
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < KI; ++i) {
        const int k = t + i * S::TPL;
        if (ok && k < S::Nh) {
          s[k] = {z[i].x + y[i].x, z[i].y - y[i].y};
          s[S::PP + k] = {z[i].y + y[i].y, y[i].x - z[i].x};
        }
      }
    }
  }
  __syncthreads();
  const int w = threadIdx.x % S::PW, t = threadIdx.x / S::PW;
  for (int c = w; c < S::Nh; c += S::PW) {
    cx<T> a[S::R1];
#pragma unroll
    for (int n1 = 0; n1 < S::R1; ++n1) a[n1] = sm[(n1 * S::R2 + t) * S::PP + c];
    line_fwd1<T, N>(a, t, tw);
#pragma unroll
    for (int k1 = 0; k1 < S::R1; ++k1) sm[(k1 * S::R2 + t) * S::PP + c] = a[k1];  // (the same elements)
  }
  __syncthreads();
  if (t < S::R1) {
    for (int c = w; c < S::Nh; c += S::PW) {
      cx<T> b[S::R2];
#pragma unroll
      for (int n2 = 0; n2 < S::R2; ++n2) b[n2] = sm[(t * S::R2 + n2) * S::PP + c];
      Dft<S::R2, false, T>::run(b);
#pragma unroll
      for (int k2 = 0; k2 < S::R2; ++k2) hat_st(hat + (t + S::R1 * k2) * S::Nh + c, b[k2]);
    }
  }
}

template <class T, int N>
__global__ void __launch_bounds__(Shape<T, N>::PT)
    fft_zy_inv(const JobView* __restrict__ views, JobList list, const cx<T>* hat, T* out, const cx<T>* __restrict__ tw) {
  using S = Shape<T, N>;
  extern __shared__ __align__(16) unsigned char smem_[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_);
  const int pl = blockIdx.x % (6 * N);
  if (views) {
    const JobView& v = views[list.at[blockIdx.x / (6 * N)]];
    hat = static_cast<const cx<T>*>(v.sig_hat);
    out = static_cast<T*>(v.eps_out);
  }
  hat += (int64_t)pl * N * S::Nh;
  out += (int64_t)pl * N * N;
  {
    const int w = threadIdx.x % S::PW, t = threadIdx.x / S::PW;
    if (t < S::R1) {
      for (int c = w; c < S::Nh; c += S::PW) {
        cx<T> b[S::R2];
#pragma unroll
        for (int k2 = 0; k2 < S::R2; ++k2) b[k2] = hat_ld(hat + (t + S::R1 * k2) * S::Nh + c);
        line_inv1<T, N>(b, t, tw);
#pragma unroll
        for (int n2 = 0; n2 < S::R2; ++n2) sm[(t * S::R2 + n2) * S::PP + c] = b[n2];
      }
    }
    __syncthreads();
    for (int c = w; c < S::Nh; c += S::PW) {
      cx<T> a[S::R1];
#pragma unroll
      for (int k1 = 0; k1 < S::R1; ++k1) a[k1] = sm[(k1 * S::R2 + t) * S::PP + c];
      Dft<S::R1, true, T>::run(a);
#pragma unroll
      for (int n1 = 0; n1 < S::R1; ++n1) sm[(n1 * S::R2 + t) * S::PP + c] = a[n1];
    }
    __syncthreads();
  }
  const int t = threadIdx.x % S::TPL, l0 = threadIdx.x / S::TPL;
  constexpr int KI = (S::Nh + S::TPL - 1) / S::TPL;
  for (int base = 0; base < N / 2; base += S::PL) {
    const int l = base + l0;
    const bool ok = l < N / 2;
    cx<T>* s = sm + 2 * l * S::PP;
    cx<T> ra[KI], rb[KI];
#pragma unroll
    for (int i = 0; i < KI; ++i) {
      const int k = t + i * S::TPL;
      if (ok && k < S::Nh) {
        ra[i] = s[k];
        rb[i] = s[S::PP + k];
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < KI; ++i) {
      const int k = t + i * S::TPL;
      if (!ok || k >= S::Nh) {
      } else if (k == 0 || k == N / 2) {
        s[k] = {ra[i].x, rb[i].x};
      } else {
        s[k] = {ra[i].x - rb[i].y, ra[i].y + rb[i].x};
        s[N - k] = {ra[i].x + rb[i].y, rb[i].x - ra[i].y};
      }
    }
    __syncthreads();
    cx<T> b[S::R2];
    if (ok && t < S::R1) {
#pragma unroll
      for (int k2 = 0; k2 < S::R2; ++k2) b[k2] = s[t + S::R1 * k2];
      line_inv1<T, N>(b, t, tw);
    }
    __syncthreads();
    if (ok && t < S::R1) {
#pragma unroll
      for (int n2 = 0; n2 < S::R2; ++n2) s[t * S::PITCH + n2] = b[n2];
    }
    __syncthreads();
    if (ok) {
      T* x = out + 2 * l * N;
      cx<T> a[S::R1];
#pragma unroll
      for (int k1 = 0; k1 < S::R1; ++k1) a[k1] = s[k1 * S::PITCH + t];
      Dft<S::R1, true, T>::run(a);
#pragma unroll
      for (int n1 = 0; n1 < S::R1; ++n1) {
        x[n1 * S::R2 + t] = a[n1].x;
        x[N + n1 * S::R2 + t] = a[n1].y;
      }
    }
  }
}

// -------------------------------------------------------------- column passes

// Complex transform of columns of stride I (y: I = Nh, x: I = N Nh), in place.
// grid: jobs x tiles of W columns.  views == NULL: one job's spectrum hat.
template <class T, int N, int I, bool INV>
__global__ void __launch_bounds__(Shape<T, N>::W* Shape<T, N>::TPL)
    fft_col(const JobView* __restrict__ views, JobList list, cx<T>* hat, const cx<T>* __restrict__ tw) {
  using S = Shape<T, N>;
  constexpr int cols = 6 * N * S::Nh, tiles = (cols + S::W - 1) / S::W;
  extern __shared__ __align__(16) unsigned char smem_[];
  const int w = threadIdx.x % S::W, t = threadIdx.x / S::W;
  cx<T>* s = reinterpret_cast<cx<T>*>(smem_) + w;
  if (views) hat = static_cast<cx<T>*>(views[list.at[blockIdx.x / tiles]].sig_hat);
  const int col = (int)(blockIdx.x % tiles) * S::W + w;
  const bool ok = col < cols;
  cx<T>* x = hat + (int64_t)(col / I) * ((int64_t)N * I) + col % I;
  if constexpr (!INV) {
    if (ok) {
      cx<T> a[S::R1];
#pragma unroll
      for (int n1 = 0; n1 < S::R1; ++n1) a[n1] = hat_ld(x + (int64_t)(n1 * S::R2 + t) * I);
      line_fwd1<T, N>(a, t, tw);
#pragma unroll
      for (int k1 = 0; k1 < S::R1; ++k1) s[(k1 * S::PITCH + t) * S::W] = a[k1];
    }
    __syncthreads();
    if (ok && t < S::R1) {
      cx<T> b[S::R2];
#pragma unroll
      for (int n2 = 0; n2 < S::R2; ++n2) b[n2] = s[(t * S::PITCH + n2) * S::W];
      Dft<S::R2, false, T>::run(b);
#pragma unroll
      for (int k2 = 0; k2 < S::R2; ++k2) hat_st(x + (int64_t)(t + S::R1 * k2) * I, b[k2]);
    }
  } else {
    if (ok && t < S::R1) {
      cx<T> b[S::R2];
#pragma unroll
      for (int k2 = 0; k2 < S::R2; ++k2) b[k2] = hat_ld(x + (int64_t)(t + S::R1 * k2) * I);
      line_inv1<T, N>(b, t, tw);
#pragma unroll
      for (int n2 = 0; n2 < S::R2; ++n2) s[(t * S::PITCH + n2) * S::W] = b[n2];
    }
    __syncthreads();
    if (ok) {
      cx<T> a[S::R1];
#pragma unroll
      for (int k1 = 0; k1 < S::R1; ++k1) a[k1] = s[(k1 * S::PITCH + t) * S::W];
      Dft<S::R1, true, T>::run(a);
#pragma unroll
      for (int n1 = 0; n1 < S::R1; ++n1) hat_st(x + (int64_t)(n1 * S::R2 + t) * I, a[n1]);
    }
  }
}

// 1/x of a positive FP32 or FP64 number to its rounding.
__device__ __forceinline__ double recip_k(double x) { return recip_pos(x); }
__device__ __forceinline__ float recip_k(float x) {
  const float r = rcp_approx(x);
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double int_as(int j, double) { return fpow::double_of_int(j); }
__device__ __forceinline__ float int_as(int j, float) { return (float)j; }

// Green update of one mode on registers: s = 2 sig_hat (fft_z_fwd), e = eps_hat
// (in/out); adds w |k . s|^2 to res, w the Hermitian weight.  With
//   p = a q - b (k.q) k,  a = 1/(4 mu0 |k|^2),  b = (lambda0 + mu0)/(4 mu0 (lambda0 + 2 mu0) |k|^4)
// (q = s k) the update is Gamma0 : sig_hat = k p^T + p k^T: 30 operations for
// the twelve reals instead of 78 entry by entry, which in FP64 are the kernel's
// bound.  inv4mu = 1/(4 mu0), coef = b |k|^4.
template <class T, int N>
__device__ __forceinline__ void green_mode(int a, int b, int c, T inv4mu, T coef, const cx<T> (&s)[6], cx<T> (&e)[6],
                                           double& res) {
  const int kx = a < N / 2 ? a : a - N, ky = b < N / 2 ? b : b - N, kz = c;
  const int nz = (kx != 0) + (ky != 0) + (kz != 0);
  const bool nyq = a == N / 2 || b == N / 2 || c == N / 2;
  if (nz == 0 || (nyq && nz >= 2)) return;  // Gamma0 = 0: eps_hat unchanged
  const T k[3] = {int_as(kx, T()), int_as(ky, T()), int_as(kz, T())};
  const T k2 = int_as(kx * kx + ky * ky + kz * kz, T());  // exact
  cx<T> q[3], p[3], kq;
  const int row[3][3] = {{0, 5, 4}, {5, 1, 3}, {4, 3, 2}};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    q[i].x = s[row[i][0]].x * k[0] + s[row[i][1]].x * k[1] + s[row[i][2]].x * k[2];
    q[i].y = s[row[i][0]].y * k[0] + s[row[i][1]].y * k[1] + s[row[i][2]].y * k[2];
  }
  const double w = (c == 0 || c == N / 2) ? 1.0 : 2.0;
  if constexpr (sizeof(T) == 8) {
    double t = q[0].x * q[0].x;
    t = fma(q[0].y, q[0].y, t);
    t = fma(q[1].x, q[1].x, t);
    t = fma(q[1].y, q[1].y, t);
    t = fma(q[2].x, q[2].x, t);
    t = fma(q[2].y, q[2].y, t);
    res = fma(w, t, res);
  } else {
    double t = f64_of(q[0].x * q[0].x + q[0].y * q[0].y) + f64_of(q[1].x * q[1].x + q[1].y * q[1].y);
    res = fma(w, t + f64_of(q[2].x * q[2].x + q[2].y * q[2].y), res);
  }
  const T ik2 = recip_k(k2);
  const T a1 = inv4mu * ik2, b1 = coef * ik2 * ik2;
  kq.x = b1 * (k[0] * q[0].x + k[1] * q[1].x + k[2] * q[2].x);
  kq.y = b1 * (k[0] * q[0].y + k[1] * q[1].y + k[2] * q[2].y);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    p[i].x = a1 * q[i].x - kq.x * k[i];
    p[i].y = a1 * q[i].y - kq.y * k[i];
  }
  const T d[3] = {T(2) * k[0], T(2) * k[1], T(2) * k[2]};
  const int ii[6] = {0, 1, 2, 1, 0, 0}, jj[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
  for (int c6 = 0; c6 < 6; ++c6) {  // (engineering shears: twice the tensor entry)
    const int i = ii[c6], j = jj[c6];
    e[c6].x -= d[j] * p[i].x;
    e[c6].y -= d[j] * p[i].y;
    if (i != j) {
      e[c6].x -= d[i] * p[j].x;
      e[c6].y -= d[i] * p[j].y;
    }
  }
}

// x pass, Green update, inverse x pass of GW columns of all six components.
// sig_hat: in the (y, z)-transformed stress, out the (y, z) spectrum of the
// updated strain; eps_hat: the strain spectrum, updated.  gam_part[tile]: the
// tile's share of sum |k . sig_hat|^2.  grid: jobs x tiles.
template <class T, int N>
__global__ void __launch_bounds__(Shape<T, N>::GT)
    fft_x_green(const JobView* __restrict__ views, JobList list, const cx<T>* __restrict__ tw) {
  using S = Shape<T, N>;
  constexpr int cols = N * S::Nh, tiles = (cols + S::GW - 1) / S::GW;
  constexpr int64_t modes = (int64_t)N * cols;
  extern __shared__ __align__(16) unsigned char smem_[];
  cx<T>* sm = reinterpret_cast<cx<T>*>(smem_);
  constexpr int CS = S::R1 * S::PITCH * S::GW;  // one component's elements
  const JobView& v = views[list.at[blockIdx.x / tiles]];
  const int tile = (int)(blockIdx.x % tiles);
  const int w = threadIdx.x % S::GW, t = (threadIdx.x / S::GW) % S::TPL, c0 = threadIdx.x / (S::GW * S::TPL);
  const int col = tile * S::GW + w;
  const bool ok = threadIdx.x < S::GL && col < cols;
  cx<T>* hat = static_cast<cx<T>*>(v.sig_hat) + col;
#pragma unroll
  for (int c = c0; c < 6; c += S::CG) {
    if (!ok) break;
    const cx<T>* x = hat + c * modes;
    cx<T>* s = sm + c * CS + w;
    cx<T> a[S::R1];
#pragma unroll
    for (int n1 = 0; n1 < S::R1; ++n1) a[n1] = hat_ld(x + (int64_t)(n1 * S::R2 + t) * cols);
    line_fwd1<T, N>(a, t, tw);
#pragma unroll
    for (int k1 = 0; k1 < S::R1; ++k1) s[(k1 * S::PITCH + t) * S::GW] = a[k1];
  }
  __syncthreads();
  // FP32 (bound by latency): the strain spectrum of a thread's next mode is
  // loaded one mode ahead, the first during the second stage
  constexpr bool kAhead = sizeof(T) == 4;
  const bool project = v.project != 0;
  cx<T>* eh = static_cast<cx<T>*>(v.eps_hat);
  auto load_e = [&](int m, cx<T> (&e)[6]) {
    const int mc = tile * S::GW + m % S::GW;
    const bool in = m < N * S::GW && mc < cols && !project;
#pragma unroll
    for (int q = 0; q < 6; ++q) e[q] = in ? hat_ld(eh + (int64_t)(m / S::GW) * cols + mc + q * modes) : cx<T>{T(0), T(0)};
  };
  cx<T> en[kAhead ? 6 : 1];
  if constexpr (kAhead) load_e(threadIdx.x, en);
  // (the stages of R1 threads a line: whole warps of them)
  const int t2 = (threadIdx.x / S::GW) % S::R1, d0 = threadIdx.x / (S::GW * S::R1);
  const bool ok2 = d0 < S::CG && col < cols;
#pragma unroll
  for (int c = d0; c < 6; c += S::CG) {
    if (!ok2) break;
    cx<T>* s = sm + c * CS + w;
    cx<T> b[S::R2];
#pragma unroll
    for (int n2 = 0; n2 < S::R2; ++n2) b[n2] = s[(t2 * S::PITCH + n2) * S::GW];
    Dft<S::R2, false, T>::run(b);
#pragma unroll
    for (int k2 = 0; k2 < S::R2; ++k2) s[(t2 * S::PITCH + k2) * S::GW] = b[k2];
  }
  __syncthreads();
  double res[1] = {0.0};
  {
    const T inv4mu = (T)v.inv4mu, coef = (T)v.green_b;
    for (int m = threadIdx.x; m < N * S::GW; m += S::GT) {
      const int mw = m % S::GW, kx = m / S::GW;
      const int mc = tile * S::GW + mw;
      cx<T> sg[6], e[6];
      if constexpr (kAhead) {
#pragma unroll
        for (int q = 0; q < 6; ++q) e[q] = en[q];
        load_e(m + S::GT, en);
      }
      if (mc >= cols) continue;
      cx<T>* g = eh + (int64_t)kx * cols + mc;
      if constexpr (!kAhead) {
#pragma unroll
        for (int q = 0; q < 6; ++q) e[q] = project ? cx<T>{T(0), T(0)} : hat_ld(g + q * modes);
      }
      cx<T>* sl = sm + ((kx % S::R1) * S::PITCH + kx / S::R1) * S::GW + mw;
#pragma unroll
      for (int q = 0; q < 6; ++q) sg[q] = sl[q * CS];
      green_mode<T, N>(kx, mc / S::Nh, mc % S::Nh, inv4mu, coef, sg, e, res[0]);
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        if (!project) hat_st(g + q * modes, e[q]);
        sl[q * CS] = e[q];
      }
    }
  }
  res[0] *= 0.25;  // (s is 2 sig_hat)
  block_sum_at<1>(res, v.gam_part, tiles, tile);  // ends with a barrier
  // this tile's share of the material kernel's partial sums, so that the job's
  // last block has 7 sums of `tiles` left (256^3: 29 k values, not 102 k); here,
  // where the fence overlaps the other warps' inverse transform
  if (v.arrived && threadIdx.x < 6) {
    const double* m = v.mat_part + (int64_t)threadIdx.x * v.n_vch;
    const int k1 = (int)((int64_t)(tile + 1) * v.n_vch / tiles);
    double sum = 0.0;
    for (int k = (int)((int64_t)tile * v.n_vch / tiles); k < k1; ++k) sum += __ldg(m + k);
    v.gam_part[(int64_t)(1 + threadIdx.x) * tiles + tile] = sum;
    __threadfence();  // the block's partials (this thread's and, thread 0, the error's) before its arrival
  }
#pragma unroll
  for (int c = d0; c < 6; c += S::CG) {
    if (!ok2) break;
    cx<T>* s = sm + c * CS + w;
    cx<T> b[S::R2];
#pragma unroll
    for (int k2 = 0; k2 < S::R2; ++k2) b[k2] = s[(t2 * S::PITCH + k2) * S::GW];
    line_inv1<T, N>(b, t2, tw);
#pragma unroll
    for (int n2 = 0; n2 < S::R2; ++n2) s[(t2 * S::PITCH + n2) * S::GW] = b[n2];
  }
  __syncthreads();
  __shared__ bool last;
  if (v.arrived && threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(v.arrived, 1u) == (unsigned)tiles - 1u;
  }
#pragma unroll
  for (int c = c0; c < 6; c += S::CG) {
    if (!ok) break;
    cx<T>* x = hat + c * modes;
    const cx<T>* s = sm + c * CS + w;
    cx<T> a[S::R1];
#pragma unroll
    for (int k1 = 0; k1 < S::R1; ++k1) a[k1] = s[(k1 * S::PITCH + t) * S::GW];
    Dft<S::R1, true, T>::run(a);
#pragma unroll
    for (int n1 = 0; n1 < S::R1; ++n1) hat_st(x + (int64_t)(n1 * S::R2 + t) * cols, a[n1]);
  }
  // the job's last block forms its final sums
  if (v.arrived) {
    __syncthreads();
    if (last) {
      __threadfence();
      finalize_sums(v.gam_part + tiles, tiles, v.gam_part, tiles, v.inv_n3, v.mu0 * 1e-6, v.red, v.mean);
      if (threadIdx.x == 0) *v.arrived = 0u;
    }
  }
}

// ------------------------------------------------------------------ launchers

// A kernel with more than 48 KB of shared memory has to be told so, once per device.
template <auto Kernel> void smem_ok(size_t bytes) {
  if (bytes > 48 * 1024) cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <class T, int N> struct Launch {
  using S = Shape<T, N>;
  static const JobView* vw(const void* v) { return static_cast<const JobView*>(v); }
  static void zy_fwd(const void* v, const JobList& l, int n, const void* in, void* hat, const void* tw, cudaStream_t s) {
    if constexpr (S::plane) {
      constexpr auto K = fft_zy_fwd<T, N>;
      smem_ok<K>(S::p_smem);
      K<<<n * 6 * N, S::PT, S::p_smem, s>>>(vw(v), l, static_cast<const T*>(in), static_cast<cx<T>*>(hat),
                                            static_cast<const cx<T>*>(tw));
      count_launch();
    } else {
      constexpr auto K = fft_z_fwd<T, N>;
      smem_ok<K>(S::z_smem);
      K<<<n * ((3 * N * N + S::LP - 1) / S::LP), S::LP * S::TPL, S::z_smem, s>>>(
          vw(v), l, static_cast<const T*>(in), static_cast<cx<T>*>(hat), static_cast<const cx<T>*>(tw));
      count_launch();
      col<S::Nh, false>(v, l, n, hat, tw, s);
    }
  }
  static void zy_inv(const void* v, const JobList& l, int n, void* hat, void* out, const void* tw, cudaStream_t s) {
    if constexpr (S::plane) {
      constexpr auto K = fft_zy_inv<T, N>;
      smem_ok<K>(S::p_smem);
      K<<<n * 6 * N, S::PT, S::p_smem, s>>>(vw(v), l, static_cast<const cx<T>*>(hat), static_cast<T*>(out),
                                            static_cast<const cx<T>*>(tw));
      count_launch();
    } else {
      col<S::Nh, true>(v, l, n, hat, tw, s);
      constexpr auto K = fft_z_inv<T, N>;
      smem_ok<K>(S::z_smem);
      K<<<n * ((3 * N * N + S::LP - 1) / S::LP), S::LP * S::TPL, S::z_smem, s>>>(
          vw(v), l, static_cast<const cx<T>*>(hat), static_cast<T*>(out), static_cast<const cx<T>*>(tw));
      count_launch();
    }
  }
  template <int I, bool INV>
  static void col(const void* v, const JobList& l, int n, void* hat, const void* tw, cudaStream_t s) {
    constexpr auto K = fft_col<T, N, I, INV>;
    smem_ok<K>(S::c_smem);
    K<<<n * ((6 * N * S::Nh + S::W - 1) / S::W), S::W * S::TPL, S::c_smem, s>>>(
        vw(v), l, static_cast<cx<T>*>(hat), static_cast<const cx<T>*>(tw));
    count_launch();
  }
  static constexpr int tiles = (N * S::Nh + S::GW - 1) / S::GW;
  static void x_green(const void* v, const JobList& l, int n, const void* tw, cudaStream_t s) {
    constexpr auto K = fft_x_green<T, N>;
    smem_ok<K>(S::g_smem);
    K<<<n * tiles, S::GT, S::g_smem, s>>>(vw(v), l, static_cast<const cx<T>*>(tw));
    count_launch();
  }
  static const FftOps* ops() {
    static const FftOps o{zy_fwd, col<N * S::Nh, false>, x_green, col<N * S::Nh, true>, zy_inv, tiles};
    return &o;
  }
};

}  // namespace
}  // namespace gsm
