// Float64 FFT of pencils of length L = 2^a 3^b staged in shared memory: Stockham autosort stages of radix 4,
// 2 and 3.  Used by the plan-time builders and by the detector-plane optics.
#pragma once

#include "common.cuh"

namespace lsgpu {

// Twiddles exp(-2 pi i j / L), j < L, on the current device, built on first use (null: out of memory).
const double2* twiddle64(int L, cudaStream_t st);

__device__ __forceinline__ void zdft(double2* v, int r, int dir) {
  if (r == 2) {
    double2 t = v[1];
    v[1] = zsub(v[0], t);
    v[0] = zadd(v[0], t);
  } else if (r == 4) {
    double2 s0 = zadd(v[0], v[2]), d0 = zsub(v[0], v[2]);
    double2 s1 = zadd(v[1], v[3]), d1 = zsub(v[1], v[3]);
    double2 d1r = dir < 0 ? make_double2(d1.y, -d1.x) : make_double2(-d1.y, d1.x);
    v[0] = zadd(s0, s1);
    v[2] = zsub(s0, s1);
    v[1] = zadd(d0, d1r);
    v[3] = zsub(d0, d1r);
  } else {  // 3
    const double h = 0.86602540378443864676;
    double2 s = zadd(v[1], v[2]), d = zsub(v[1], v[2]);
    double2 m = make_double2(v[0].x - 0.5 * s.x, v[0].y - 0.5 * s.y);
    double2 rr = dir < 0 ? make_double2(h * d.y, -h * d.x) : make_double2(-h * d.y, h * d.x);
    v[0] = zadd(v[0], s);
    v[1] = zadd(m, rr);
    v[2] = zsub(m, rr);
  }
}


// Transforms the pencil whose element i is b0[i es] (b1: scratch of the same layout) by the nt threads t of its
// group; every thread of the CTA calls it (it synchronises the CTA after each stage) with the same L.
// Returns the buffer that holds the result.  dir = -1 forward, +1 inverse (unnormalised).
__device__ __forceinline__ double2* fft64_staged(double2* b0, double2* b1, int L, int es, int dir, const double2* tw,
                                                 int t, int nt) {
  int rest = L, Ns = 1;
  while (rest > 1) {
    const int r = (rest % 4 == 0) ? 4 : (rest % 2 == 0 ? 2 : 3);
    const int m = L / r, step = m / Ns;
    for (int j = t; j < m; j += nt) {
      const int k = j % Ns;
      double2 v[4];
      for (int q = 0; q < r; ++q) {
        v[q] = b0[(j + q * m) * es];
        if (q > 0) {
          // exp(dir 2 pi i k q / (Ns r)) = tw[k q L / (Ns r)] (conjugated for dir = +1), an index below L
          double2 w = tw[k * q * step];
          if (dir > 0) w.y = -w.y;
          v[q] = zmul(v[q], w);
        }
      }
      zdft(v, r, dir);
      const int o = (j - k) * r + k;
      for (int q = 0; q < r; ++q) b1[(o + q * Ns) * es] = v[q];
    }
    __syncthreads();
    double2* tmp = b0; b0 = b1; b1 = tmp;
    Ns *= r;
    rest /= r;
  }
  return b0;
}

}  // namespace lsgpu
