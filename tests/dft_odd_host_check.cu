// Host check of the odd-frequency DFTs (csrc/dft.cuh) against direct sums; prints the worst error and fails above the bound.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>

#include "dft.cuh"

using namespace lsgpu;

template <int R, int DIR>
static bool check() {
  double worst[2] = {0, 0}, scale = 0;
  for (int trial = 0; trial < 50; ++trial) {
    float2 in[R], a[R], b[R];
    for (int n = 0; n < R; ++n) {
      in[n] = make_float2((float)rand() / RAND_MAX - 0.5f, (float)rand() / RAND_MAX - 0.5f);
      a[n] = b[n] = in[n];
    }
    DftOddIn<R, DIR>::run(a);
    DftOddOut<R, DIR>::run(b);
    for (int k = 0; k < R; ++k) {
      std::complex<double> x = 0, y = 0;
      for (int n = 0; n < R; ++n) {
        const std::complex<double> v(in[n].x, in[n].y);
        x += v * std::polar(1.0, DIR * M_PI * n * (2 * k + 1) / R);
        y += v * std::polar(1.0, DIR * M_PI * k * (2 * n + 1) / R);
      }
      worst[0] = std::fmax(worst[0], std::abs(x - std::complex<double>(a[k].x, a[k].y)));
      worst[1] = std::fmax(worst[1], std::abs(y - std::complex<double>(b[k].x, b[k].y)));
      scale = std::fmax(scale, std::abs(x));
    }
  }
  // at most 2 log2 R + 4 roundings of 6e-8 in a chain, values up to the largest output
  const double bound = 6e-8 * (2 * std::log2(R) + 4) * scale;
  std::printf("R %d DIR %d in %.2e out %.2e bound %.2e\n", R, DIR, worst[0], worst[1], bound);
  return worst[0] <= bound && worst[1] <= bound;
}

// the plain DFT of R points, whose coprime factors take no internal twiddles
template <int R, int DIR>
static bool check_plain() {
  double worst = 0, scale = 0;
  for (int trial = 0; trial < 50; ++trial) {
    float2 in[R], a[R];
    for (int n = 0; n < R; ++n) a[n] = in[n] = make_float2((float)rand() / RAND_MAX - 0.5f, (float)rand() / RAND_MAX - 0.5f);
    Dft<R, DIR>::run(a);
    for (int k = 0; k < R; ++k) {
      std::complex<double> x = 0;
      for (int n = 0; n < R; ++n) x += std::complex<double>(in[n].x, in[n].y) * std::polar(1.0, DIR * 2 * M_PI * n * k / R);
      worst = std::fmax(worst, std::abs(x - std::complex<double>(a[k].x, a[k].y)));
      scale = std::fmax(scale, std::abs(x));
    }
  }
  const double bound = 6e-8 * (2 * std::log2(R) + 4) * scale;
  std::printf("R %d DIR %d plain %.2e bound %.2e\n", R, DIR, worst, bound);
  return worst <= bound;
}

int main() {
  bool ok = true;
  ok &= check<2, -1>() && check<2, 1>() && check<3, -1>() && check<3, 1>() && check<4, -1>() && check<4, 1>();
  ok &= check<6, -1>() && check<6, 1>() && check<8, -1>() && check<8, 1>() && check<9, -1>() && check<9, 1>() && check<12, -1>() && check<12, 1>();
  ok &= check_plain<6, -1>() && check_plain<6, 1>() && check_plain<9, -1>() && check_plain<9, 1>();
  ok &= check_plain<12, -1>() && check_plain<12, 1>() && check_plain<24, -1>() && check_plain<24, 1>();
  return ok ? 0 : 1;
}
