// Register-resident small DFTs for the pencil FFT passes.
//
// Dft<R, DIR>::run(a) replaces a[0..R-1] by X[k] = sum_n a[n] exp(DIR * 2 pi i n k / R)
// (DIR = -1 forward, +1 inverse, unnormalised).  Composite sizes use one
// in-register Cooley-Tukey split R = A * B with compile-time twiddles.
#pragma once

#include "common.cuh"

namespace lsgpu {

// sin/cos of 2 pi j / R evaluated at compile time by a Taylor series in double.
__host__ __device__ constexpr double cx_pi() { return 3.14159265358979323846264338327950288; }

__host__ __device__ constexpr double cx_sin_series(double x) {
  double term = x, sum = x;
  for (int k = 1; k < 30; ++k) {
    term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr double cx_cos_series(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 30; ++k) {
    term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    sum += term;
  }
  return sum;
}
// angle 2 pi j / R reduced to [-pi, pi]
__host__ __device__ constexpr double cx_angle(int j, int R) {
  int jj = ((j % R) + R) % R;
  if (2 * jj > R) jj -= R;
  return 2.0 * cx_pi() * (double)jj / (double)R;
}
__host__ __device__ constexpr double cx_cos(int j, int R) { return cx_cos_series(cx_angle(j, R)); }
__host__ __device__ constexpr double cx_sin(int j, int R) { return cx_sin_series(cx_angle(j, R)); }

// a *= exp(DIR * 2 pi i J / R), with the trivial angles (multiples of pi/2) done without multiplies.
template <int J, int R, int DIR>
__host__ __device__ __forceinline__ float2 twc(float2 a) {
  constexpr int jj = ((J % R) + R) % R;
  if constexpr (jj == 0) {
    return a;
  } else if constexpr (4 * jj == R) {  // exp(DIR i pi/2) = DIR i
    return DIR < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
  } else if constexpr (2 * jj == R) {
    return make_float2(-a.x, -a.y);
  } else if constexpr (4 * jj == 3 * R) {  // exp(DIR i 3pi/2) = -DIR i
    return DIR < 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
  } else {
    constexpr float c = (float)cx_cos(jj, R);
    constexpr float s = (float)(DIR * cx_sin(jj, R));
    if constexpr (R == 9) {
      // 9 = 3 3 has no form without these: their constants in two terms (error of the y transforms at 72 points
      // 8.3e-8 -> 8.1e-8, with 12 12 it is 7.2e-8)
      constexpr float cl = (float)(cx_cos(jj, R) - (double)c), sl = (float)(DIR * cx_sin(jj, R) - (double)s);
      return make_float2(fmaf(a.x, c, fmaf(-a.y, s, fmaf(a.x, cl, -a.y * sl))),
                         fmaf(a.x, s, fmaf(a.y, c, fmaf(a.x, sl, a.y * cl))));
    }
    return make_float2(a.x * c - a.y * s, a.x * s + a.y * c);
  }
}

// Dft<R, DIR, NIN, NOUT>: only a[0..NIN-1] may be nonzero (the rest is never
// read) and only X[0..NOUT-1] are produced (the other entries are left
// undefined).  Zero padding and cropping of the transforms use this to skip
// the corresponding arithmetic.
// FEW: the forms with fewer roundings (radix 3 in fused multiply-adds, no twiddles between coprime factors).  The
// column-group z pass, whose registers they would exceed (a spill at 144 points), does without.
template <int R, int DIR, int NIN = R, int NOUT = R, bool FEW = true>
struct Dft;

template <int DIR, int NIN, int NOUT, bool FEW>
struct Dft<1, DIR, NIN, NOUT, FEW> {
  __host__ __device__ __forceinline__ static void run(float2*) {}
};

template <int DIR, int NIN, int NOUT, bool FEW>
struct Dft<2, DIR, NIN, NOUT, FEW> {
  __host__ __device__ __forceinline__ static void run(float2* a) {
    if constexpr (NIN >= 2) {
      float2 t = a[1];
      if constexpr (NOUT >= 2) a[1] = csub(a[0], t);
      a[0] = cadd(a[0], t);
    } else {
      if constexpr (NOUT >= 2) a[1] = a[0];
    }
  }
};

template <int DIR, int NIN, int NOUT, bool FEW>
struct Dft<3, DIR, NIN, NOUT, FEW> {
  __host__ __device__ __forceinline__ static void run(float2* a) {
    // X0 = a0 + a1 + a2 ; X1,2 = a0 - (a1+a2)/2 +/- DIR i (sqrt3/2)(a1 - a2)
    constexpr float h = 0.86602540378443864676f;
    const float2 a1 = NIN > 1 ? a[1] : make_float2(0.f, 0.f);
    const float2 a2 = NIN > 2 ? a[2] : make_float2(0.f, 0.f);
    float2 s = cadd(a1, a2);
    float2 d = csub(a1, a2);
    float2 m = make_float2(a[0].x - 0.5f * s.x, a[0].y - 0.5f * s.y);
    a[0] = cadd(a[0], s);
    if constexpr (FEW) {
      constexpr float hd = DIR * h;
      if constexpr (NOUT > 1) a[1] = make_float2(fmaf(-hd, d.y, m.x), fmaf(hd, d.x, m.y));
      if constexpr (NOUT > 2) a[2] = make_float2(fmaf(hd, d.y, m.x), fmaf(-hd, d.x, m.y));
    } else {
      const float2 r = DIR < 0 ? make_float2(h * d.y, -h * d.x) : make_float2(-h * d.y, h * d.x);
      if constexpr (NOUT > 1) a[1] = cadd(m, r);
      if constexpr (NOUT > 2) a[2] = csub(m, r);
    }
  }
};

// X[k] = sum_n a[n] exp(DIR 2 pi i n (2k + 1) / 6), the odd frequencies of a length-6 transform: n = 1 changes its sign
// and the frequencies rotate, as exp(DIR 2 pi i n / 6) = (-1)^n exp(DIR 2 pi i 2n / 3); no multiplication is added
template <int DIR>
__host__ __device__ __forceinline__ void dft3_odd(float2* a) {
  constexpr float h = 0.86602540378443864676f;
  const float2 s = csub(a[2], a[1]), d = cadd(a[1], a[2]);
  const float2 m = make_float2(a[0].x - 0.5f * s.x, a[0].y - 0.5f * s.y);
  constexpr float hd = DIR * h;
  a[1] = cadd(a[0], s);
  a[0] = make_float2(fmaf(-hd, d.y, m.x), fmaf(hd, d.x, m.y));
  a[2] = make_float2(fmaf(hd, d.y, m.x), fmaf(-hd, d.x, m.y));
}

template <int DIR, int NIN, int NOUT, bool FEW>
struct Dft<4, DIR, NIN, NOUT, FEW> {
  __host__ __device__ __forceinline__ static void run(float2* a) {
    if constexpr (NIN <= 2) {
      // a2 = a3 = 0: X0 = a0 + a1, X1 = a0 + w a1, X2 = a0 - a1, X3 = a0 - w a1 (w = DIR i)
      const float2 b = NIN > 1 ? a[1] : make_float2(0.f, 0.f);
      const float2 br = twc<1, 4, DIR>(b);
      const float2 a0 = a[0];
      a[0] = cadd(a0, b);
      if constexpr (NOUT > 1) a[1] = cadd(a0, br);
      if constexpr (NOUT > 2) a[2] = csub(a0, b);
      if constexpr (NOUT > 3) a[3] = csub(a0, br);
    } else {
      const float2 a3 = NIN > 3 ? a[3] : make_float2(0.f, 0.f);
      float2 s0 = cadd(a[0], a[2]), d0 = csub(a[0], a[2]);
      float2 s1 = cadd(a[1], a3), d1 = csub(a[1], a3);
      float2 d1r = twc<1, 4, DIR>(d1);
      a[0] = cadd(s0, s1);
      if constexpr (NOUT > 1) a[1] = cadd(d0, d1r);
      if constexpr (NOUT > 2) a[2] = csub(s0, s1);
      if constexpr (NOUT > 3) a[3] = csub(d0, d1r);
    }
  }
};

// Split for composite sizes: R = A * B, A chosen below.
template <int R> struct Split;
template <> struct Split<6>  { static constexpr int A = 2; };
template <> struct Split<8>  { static constexpr int A = 2; };
template <> struct Split<9>  { static constexpr int A = 3; };
template <> struct Split<12> { static constexpr int A = 4; };
template <> struct Split<16> { static constexpr int A = 4; };
template <> struct Split<24> { static constexpr int A = 8; };
template <> struct Split<32> { static constexpr int A = 8; };

__host__ __device__ constexpr int cdiv_pos(int a, int b) { return a <= 0 ? 0 : (a + b - 1) / b; }

// X[k1 + A k2] = sum_{n2<B} W_B^{n2 k2} W_R^{n2 k1} sum_{n1<A} x[B n1 + n2] W_A^{n1 k1}
// Input x[B n1 + n2] is nonzero only for B n1 + n2 < NIN; output X[k1 + A k2] is needed only for
// k1 + A k2 < NOUT.
template <int R, int DIR, int NIN, int NOUT, bool FEW>
struct Dft {
  static constexpr int A = Split<R>::A;
  static constexpr int B = R / A;
  // A and B = 3 coprime (6, 12, 24): with U A + 3 V = 1 the twiddle W_R^{n2 k1} is W_A^{V n2 k1}, which is trivial for
  // A = 2 and 4 and half of the time for 8, times W_3^{U n2 k1}, which rotates the outputs: one rounding less
  static constexpr bool COPRIME = FEW && B == 3 && A % 3 != 0;
  static constexpr int U = A % 3 == 1 ? 1 : -1, V = (1 - U * A) / 3;
  __host__ __device__ __forceinline__ static void run(float2* a) {
    float2 t[B][A];
    inner<0>(a, t);
    outer<0>(a, t);
  }
  // step 1: the B sub-DFTs of length A, with their own input pruning, then the internal twiddles
  template <int N2>
  __host__ __device__ __forceinline__ static void inner(float2* a, float2 (&t)[B][A]) {
    if constexpr (N2 < B) {
      constexpr int nin = cdiv_pos(NIN - N2, B);
      if constexpr (nin > 0) {
#pragma unroll
        for (int n1 = 0; n1 < nin; ++n1) t[N2][n1] = a[B * n1 + N2];
        Dft<A, DIR, nin, A, FEW>::run(t[N2]);
      } else {
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) t[N2][k1] = make_float2(0.f, 0.f);
      }
      apply_tw_k<N2, 1>(t);
      inner<N2 + 1>(a, t);
    }
  }
  // step 2: the A sub-DFTs of length B, each producing only the outputs that are needed
  template <int K1>
  __host__ __device__ __forceinline__ static void outer(float2* a, float2 (&t)[B][A]) {
    if constexpr (K1 < A) {
      constexpr int nout = cdiv_pos(NOUT - K1, A);
      if constexpr (nout > 0) {
        float2 u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = t[n2][K1];
        Dft<B, DIR, B, COPRIME ? B : nout, FEW>::run(u);
#pragma unroll
        for (int k2 = 0; k2 < nout; ++k2) a[K1 + A * k2] = u[COPRIME ? (k2 + (U + 3) * K1) % 3 : k2];
      }
      outer<K1 + 1>(a, t);
    }
  }
  template <int N2, int K1>
  __host__ __device__ __forceinline__ static void apply_tw_k(float2 (&t)[B][A]) {
    if constexpr (K1 < A && N2 > 0) {
      if constexpr (COPRIME) t[N2][K1] = twc<V * N2 * K1, A, DIR>(t[N2][K1]);
      else t[N2][K1] = twc<N2 * K1, R, DIR>(t[N2][K1]);
      apply_tw_k<N2, K1 + 1>(t);
    }
  }
};

// DFTs at the odd frequencies of twice the length, w = exp(DIR 2 pi i / 2R):
//   DftOddIn<R, DIR>::run(a)  replaces a by X[k] = sum_n a[n] w^{n (2k + 1)}  (the half of a zero-padded transform),
//   DftOddOut<R, DIR>::run(a) replaces a by x[n] = sum_k a[k] w^{n (2k + 1)}  (its transpose).
// A twist of the inputs (outputs) by w^n before (after) a plain DFT gives the same with one more rounding of nearly
// every value.  Here the twist meets the twiddles that are there anyway: with n = B n1 + n2, w^n is a twist of the
// inner DFT of length A and a factor w^{n2} of the twiddle w^{2 n2 k1}.  What is left is a twist of length 2, a
// multiplication by i, or of an odd length, where w^n = (-1)^n exp(DIR 2 pi i n (R + 1) / 2 / R): signs and a
// rotation of the frequencies.
template <int R> struct OddSplit;
template <> struct OddSplit<4>  { static constexpr int IN = 2, OUT = 2; };   // A of either
template <> struct OddSplit<6>  { static constexpr int IN = 3, OUT = 2; };
template <> struct OddSplit<8>  { static constexpr int IN = 2, OUT = 4; };
template <> struct OddSplit<12> { static constexpr int IN = 3, OUT = 4; };

__host__ __device__ __forceinline__ float2 cneg(float2 a) { return make_float2(-a.x, -a.y); }

// t[N2][K1] *= exp(DIR 2 pi i I / (2 R)) for all K1 < A, I = N2 (2 K1 + 1) (INPUT) or K1 (2 N2 + 1)
template <int R, int DIR, bool INPUT, int N2, int K1, int A>
__host__ __device__ __forceinline__ void odd_twiddle(float2* t) {
  if constexpr (K1 < A) {
    t[K1] = twc<INPUT ? N2 * (2 * K1 + 1) : K1 * (2 * N2 + 1), 2 * R, DIR>(t[K1]);
    odd_twiddle<R, DIR, INPUT, N2, K1 + 1, A>(t);
  }
}

template <int R, int DIR>
struct DftOddIn {
  __host__ __device__ __forceinline__ static void run(float2* a) {
    if constexpr (R == 2) {
      const float2 b = twc<1, 4, DIR>(a[1]);
      a[1] = csub(a[0], b);
      a[0] = cadd(a[0], b);
    } else if constexpr (R == 3) {
      dft3_odd<DIR>(a);
    } else if constexpr (R % 2 == 1) {
      float2 y[R];
#pragma unroll
      for (int n = 0; n < R; ++n) y[n] = n % 2 ? cneg(a[n]) : a[n];
      Dft<R, DIR>::run(y);
#pragma unroll
      for (int k = 0; k < R; ++k) a[k] = y[(k + (R + 1) / 2) % R];
    } else {
      constexpr int A = OddSplit<R>::IN, B = R / A;
      float2 t[B][A];
      inner<0, A, B>(a, t);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) {
        float2 u[B];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) u[n2] = t[n2][k1];
        Dft<B, DIR>::run(u);
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) a[k1 + A * k2] = u[k2];
      }
    }
  }
  template <int N2, int A, int B>
  __host__ __device__ __forceinline__ static void inner(float2* a, float2 (&t)[B][A]) {
    if constexpr (N2 < B) {
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) t[N2][n1] = a[B * n1 + N2];
      DftOddIn<A, DIR>::run(t[N2]);
      odd_twiddle<R, DIR, true, N2, 0, A>(t[N2]);
      inner<N2 + 1>(a, t);
    }
  }
};

template <int R, int DIR>
struct DftOddOut {
  __host__ __device__ __forceinline__ static void run(float2* a) {
    if constexpr (R == 2) {
      const float2 d = csub(a[0], a[1]);
      a[0] = cadd(a[0], a[1]);
      a[1] = twc<1, 4, DIR>(d);
    } else if constexpr (R % 2 == 1) {
      float2 y[R];
#pragma unroll
      for (int k = 0; k < R; ++k) y[(k + (R + 1) / 2) % R] = a[k];
      Dft<R, DIR>::run(y);
#pragma unroll
      for (int n = 0; n < R; ++n) a[n] = n % 2 ? cneg(y[n]) : y[n];
    } else {
      constexpr int A = OddSplit<R>::OUT, B = R / A;
      float2 t[B][A];
      inner<0, A, B>(a, t);
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) {
        float2 u[B];
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) u[k2] = t[k2][n1];
        DftOddOut<B, DIR>::run(u);
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) a[n1 + A * n2] = u[n2];
      }
    }
  }
  template <int K2, int A, int B>
  __host__ __device__ __forceinline__ static void inner(float2* a, float2 (&t)[B][A]) {
    if constexpr (K2 < B) {
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) t[K2][k1] = a[B * k1 + K2];
      Dft<A, DIR>::run(t[K2]);
      odd_twiddle<R, DIR, false, K2, 0, A>(t[K2]);
      inner<K2 + 1>(a, t);
    }
  }
};

}  // namespace lsgpu
