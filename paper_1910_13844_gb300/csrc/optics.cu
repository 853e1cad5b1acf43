// Detector-plane optics: the incident field propagated from its measurement on the detector
// (Sec. 3.4, eq. propUin with the tilt transfer of eq. propUin-2) and the pupil / refocus
// operator P (Sec. 3.3).  Both are 2-D convolutions on the detector grid applied through FFTs;
// they run once per view per call (not inside the solver iterations) and use the float64
// pencil FFT of the plan builder.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "engine.h"
#include "fft64.cuh"

namespace lsgpu {

__device__ __forceinline__ int centred_i(int q, int M) { return q > M / 2 ? q - M : q; }

// A[y][x] = y_in[y][x] exp(-i (kx x + ky y)) (tilt transfer; kx = ky = 0 without it), in float64
__global__ void k_demodulate(const float2* y_in, int nx, int ny, double h, double kx, double ky, double2* A) {
  const size_t n = (size_t)nx * ny;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx), y = (int)(i / nx);
    const double ph = -(kx * h * (x - nx / 2 + 1) + ky * h * (y - ny / 2 + 1));
    double s, c;
    sincos(ph, &s, &c);
    const float2 v = y_in[i];
    A[i] = make_double2(v.x * c - v.y * s, v.x * s + v.y * c);
  }
}

// B[z][y][x] = A[y][x] p_hat_z(w + k) / (nx ny), p_hat_z(w) = exp(-i (x_gamma - z) sqrt(kb^2 - |w|^2)),
// evanescent components dropped
__global__ void k_spread_planes(const double2* A, int nx, int ny, int nz, double h, double kb, double x_gamma,
                                double kx, double ky, double2* B) {
  const size_t plane = (size_t)nx * ny;
  const size_t n = plane * nz;
  const double scale = 1.0 / (double)plane;
  const double twopi = 6.283185307179586476925286766559;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / plane);
    const double wx = twopi * centred_i(x, nx) / (nx * h) + kx;
    const double wy = twopi * centred_i(y, ny) / (ny * h) + ky;
    const double s = kb * kb - wx * wx - wy * wy;
    double2 out = make_double2(0.0, 0.0);
    if (s >= 0.0) {
      const double zc = h * (z - nz / 2 + 1);
      double sn, cs;
      sincos(-(x_gamma - zc) * sqrt(s), &sn, &cs);
      const double2 a = A[i % plane];
      out = make_double2((a.x * cs - a.y * sn) * scale, (a.x * sn + a.y * cs) * scale);
    }
    B[i] = out;
  }
}

// u_in[z][y][x] = B exp(+i (kx x + ky y)), rounded to complex64
__global__ void k_modulate_store(const double2* B, int nx, int ny, int nz, double h, double kx, double ky,
                                 float2* u) {
  const size_t plane = (size_t)nx * ny;
  const size_t n = plane * nz;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx), y = (int)((i / nx) % ny);
    const double ph = kx * h * (x - nx / 2 + 1) + ky * h * (y - ny / 2 + 1);
    double s, c;
    sincos(ph, &s, &c);
    const double2 b = B[i];
    u[i] = make_float2((float)(b.x * c - b.y * s), (float)(b.x * s + b.y * c));
  }
}

// H[y][x] on the 2my x 2mx padded detector: 1{|w| <= k_cut} exp(i d sqrt(kb^2 - |w|^2)), propagating only
__global__ void k_pupil_transfer(int Mx, int My, double h, double kb, double kcut, double d, double2* Hd) {
  const size_t n = (size_t)Mx * My;
  const double twopi = 6.283185307179586476925286766559;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % Mx), y = (int)(i / Mx);
    const double wx = twopi * centred_i(x, Mx) / (Mx * h), wy = twopi * centred_i(y, My) / (My * h);
    const double w2 = wx * wx + wy * wy;
    const double s = kb * kb - w2;
    double2 v = make_double2(0.0, 0.0);
    if (s >= 0.0 && w2 <= kcut * kcut) {
      double sn, cs;
      sincos(d * sqrt(s), &sn, &cs);
      v = make_double2(cs, sn);
    }
    Hd[i] = v;
  }
}

// The pupil operator P y = crop(F^{-1}(H F(pad y))) on the 2my x 2mx padded detector, for up to 64 views in
// three launches over scratch planes [view][my][2mx] in float64: rows are padded and transformed, columns
// padded, transformed, multiplied by H and transformed back, rows transformed back and cropped.  Rows that
// are zero or cropped away are never touched.  Bound by the float64 pipe: 12 us a view at 72 x 72 with 20 views; one
// view at a time, with a launch for every pass over the whole padded grid, took 75 us.
// Up to eight pencils per CTA.  The lanes of a row pass run along the row, those of a column pass along the
// CTA's columns, whose elements lie next to one another in shared memory.
constexpr int kPupilThreads = 256;

// Detector fields of one launch.  They come by value, so that the launch holds all it needs: an upload from host
// memory would be repeated from there by a captured graph.
struct PupilViews {
  static constexpr int kMax = 64;
  const float2* in[kMax];
  float2* out[kMax];
};

// out[v][y][:] = F(pad in[v][y][:]); grid (row blocks, views), `per` rows per CTA
__global__ void __launch_bounds__(kPupilThreads) k_pupil_rows(const __grid_constant__ PupilViews v, int mx, int my,
                                                              int per, double2* out, const double2* tw) {
  extern __shared__ double2 pb[];
  const int M = 2 * mx, nt = kPupilThreads / per, g = threadIdx.x / nt, t = threadIdx.x % nt;
  const int y = blockIdx.x * per + g;
  const bool has = g < per && y < my;
  double2* b = pb + (size_t)g * 2 * M;
  const float2* src = v.in[blockIdx.y] + (size_t)y * mx;
  if (g < per)
    for (int i = t; i < M; i += nt) {
      const float2 s = has && i < mx ? src[i] : make_float2(0.f, 0.f);
      b[i] = make_double2(s.x, s.y);
    }
  __syncthreads();
  // idle threads (g == per where per does not divide the block) run no butterfly
  const double2* r = fft64_staged(b, b + M, M, 1, -1, tw, g < per ? t : M, nt);
  if (has) {
    double2* d = out + ((size_t)blockIdx.y * my + y) * M;
    for (int i = t; i < M; i += nt) d[i] = r[i];
  }
}

// plane[v][:][x] <- crop F^{-1}(H(:, x) scale F(pad plane[v][:][x])), in place; grid (column blocks, views)
__global__ void __launch_bounds__(kPupilThreads) k_pupil_cols(double2* plane, int mx, int my, int per, const double2* H,
                                                              int conj, double scale, const double2* tw) {
  extern __shared__ double2 pb[];
  const int Mx = 2 * mx, M = 2 * my, g = threadIdx.x % per, t = threadIdx.x / per, nt = kPupilThreads / per;
  const int x = blockIdx.x * per + g;
  const bool has = x < Mx && t < nt;
  double2* b0 = pb + g;
  double2* b1 = b0 + (size_t)M * per;
  double2* col = plane + (size_t)blockIdx.y * my * Mx + x;
  if (t < nt)
    for (int i = t; i < M; i += nt) b0[i * per] = has && i < my ? col[(size_t)i * Mx] : make_double2(0.0, 0.0);
  __syncthreads();
  double2* r = fft64_staged(b0, b1, M, per, -1, tw, t < nt ? t : M, nt);
  if (has)
    for (int i = t; i < M; i += nt) {
      double2 h = H[(size_t)i * Mx + x];
      if (conj) h.y = -h.y;
      const double2 v = zmul(r[i * per], h);
      r[i * per] = make_double2(v.x * scale, v.y * scale);
    }
  __syncthreads();
  r = fft64_staged(r, r == b0 ? b1 : b0, M, per, +1, tw, t < nt ? t : M, nt);
  if (has)
    for (int i = t; i < my; i += nt) col[(size_t)i * Mx] = r[i * per];
}

// out[v][y][:] = crop F^{-1}(plane[v][y][:]), rounded to complex64
__global__ void __launch_bounds__(kPupilThreads) k_pupil_out(const double2* plane, int mx, int my, int per,
                                                             const __grid_constant__ PupilViews v, const double2* tw) {
  extern __shared__ double2 pb[];
  const int M = 2 * mx, nt = kPupilThreads / per, g = threadIdx.x / nt, t = threadIdx.x % nt;
  const int y = blockIdx.x * per + g;
  const bool has = g < per && y < my;
  double2* b = pb + (size_t)g * 2 * M;
  const double2* src = plane + ((size_t)blockIdx.y * my + y) * M;
  if (g < per)
    for (int i = t; i < M; i += nt) b[i] = has ? src[i] : make_double2(0.0, 0.0);
  __syncthreads();
  const double2* r = fft64_staged(b, b + M, M, 1, +1, tw, g < per ? t : M, nt);
  if (has) {
    float2* d = v.out[blockIdx.y] + (size_t)y * mx;
    for (int i = t; i < mx; i += nt) d[i] = make_float2((float)r[i].x, (float)r[i].y);
  }
}

static int blocks_for(size_t n) {
  const size_t b = (n + 255) / 256;
  return (int)(b > 4864 ? 4864 : (b < 1 ? 1 : b));
}

// 2-D float64 FFT over `planes` stacked [planes][My][Mx] arrays (in place)
void fft64_2d_planes(double2* d, int Mx, int My, int planes, int dir, cudaStream_t st);

// lengths the float64 pencil FFT handles: 2^a 3^b, at most 1024
static bool fft64_length_ok(int L) {
  if (L < 1 || L > 1024) return false;
  while (L % 2 == 0) L /= 2;
  while (L % 3 == 0) L /= 3;
  return L == 1;
}

size_t pupil_scratch_bytes(const ls_plan* P, int n) { return (size_t)n * 2 * P->mx * P->my * sizeof(double2); }

int apply_pupil_views(ls_plan* P, int n, const void* const* in, void* const* out, int adjoint, void* scratch,
                      int scratch_views, cudaStream_t st) {
  const int mx = P->mx, my = P->my, Mx = 2 * mx, My = 2 * my;
  double2* d = static_cast<double2*>(scratch);
  const double2 *twx = twiddle64(Mx, st), *twy = twiddle64(My, st);
  if (!twx || !twy) { set_last_error("float64 twiddle table allocation failed"); return LS_ENOMEM; }
  // pencils per CTA: both buffers of each within 48 KB, at most eight (a 128-byte run of columns)
  auto per = [](int L) { return std::max(1, std::min(8, 49152 / (int)(2 * L * sizeof(double2)))); };
  const int px = per(Mx), py = per(My);
  const size_t sx = (size_t)px * 2 * Mx * sizeof(double2), sy = (size_t)py * 2 * My * sizeof(double2);
  // a view whose output is another's input or output waits for it, as it did one view at a time
  Spans io;
  for (int q = 0; q < n; ++q) {
    const size_t bytes = (size_t)mx * my * sizeof(float2);
    io.add(out[q], bytes, true);
    if (in[q] != out[q]) io.add(in[q], bytes, false);
  }
  const int most = io.disjoint() ? std::min(scratch_views, PupilViews::kMax) : 1;
  PupilViews v;
  for (int q = 0; q < n; q += most) {
    const int m = std::min(most, n - q);
    for (int k = 0; k < m; ++k) {
      v.in[k] = static_cast<const float2*>(in[q + k]);
      v.out[k] = static_cast<float2*>(out[q + k]);
    }
    k_pupil_rows<<<dim3((my + px - 1) / px, m), kPupilThreads, sx, st>>>(v, mx, my, px, d, twx);
    k_pupil_cols<<<dim3((Mx + py - 1) / py, m), kPupilThreads, sy, st>>>(d, mx, my, py, P->pupil_h, adjoint,
                                                                       1.0 / ((double)Mx * My), twy);
    k_pupil_out<<<dim3((my + px - 1) / px, m), kPupilThreads, sx, st>>>(d, mx, my, px, v, twx);
  }
  LS_CUDA_TRY(cudaGetLastError());
  return LS_OK;
}

}  // namespace lsgpu

using namespace lsgpu;

extern "C" {

int ls_incident_field(ls_plan* P, int n_views, const ls_c64* const* y_in, const double* k_in,
                      ls_c64* const* u_in, void* stream) {
  lsgpu::TraceRange trace_range("ls_incident_field");
  if (!P || n_views < 1 || !y_in || !u_in) { set_last_error("bad arguments"); return LS_EINVAL; }
  for (int q = 0; q < n_views; ++q)
    if (!y_in[q] || !u_in[q]) { set_last_error("null view pointer %d", q); return LS_EINVAL; }
  cudaStream_t st = (cudaStream_t)stream;
  const int nx = P->nx, ny = P->ny, nz = P->nz;
  if (!fft64_length_ok(nx) || !fft64_length_ok(ny)) {
    set_last_error("lateral grid %dx%d has no float64 FFT length", nx, ny);
    return LS_EUNSUPPORTED;
  }
  const size_t plane = (size_t)nx * ny, n = plane * nz;
  double2 *A = nullptr, *B = nullptr;
  LS_CUDA_TRY(cudaMallocAsync((void**)&A, plane * sizeof(double2), st));
  LS_CUDA_TRY(cudaMallocAsync((void**)&B, n * sizeof(double2), st));
  for (int q = 0; q < n_views; ++q) {
    const double kx = k_in ? k_in[2 * q] : 0.0, ky = k_in ? k_in[2 * q + 1] : 0.0;
    k_demodulate<<<blocks_for(plane), 256, 0, st>>>((const float2*)y_in[q], nx, ny, P->h, kx, ky, A);
    fft64_2d_planes(A, nx, ny, 1, -1, st);
    k_spread_planes<<<blocks_for(n), 256, 0, st>>>(A, nx, ny, nz, P->h, P->kb, P->x_gamma, kx, ky, B);
    fft64_2d_planes(B, nx, ny, nz, +1, st);
    k_modulate_store<<<blocks_for(n), 256, 0, st>>>(B, nx, ny, nz, P->h, kx, ky, (float2*)u_in[q]);
  }
  LS_CUDA_TRY(cudaFreeAsync(A, st));
  LS_CUDA_TRY(cudaFreeAsync(B, st));
  LS_CUDA_TRY(cudaGetLastError());
  return LS_OK;
}

int ls_set_pupil(ls_plan* P, double k_cut, double distance) {
  if (!P) { set_last_error("null plan"); return LS_EINVAL; }
  if (k_cut <= 0) {
    cudaFree(P->pupil_h);
    P->pupil_h = nullptr;
    return LS_OK;
  }
  const int Mx = 2 * P->mx, My = 2 * P->my;
  if (!fft64_length_ok(Mx) || !fft64_length_ok(My)) {
    set_last_error("padded detector %dx%d has no float64 FFT length", My, Mx);
    return LS_EUNSUPPORTED;
  }
  if (!P->pupil_h) LS_CUDA_TRY(cudaMalloc(&P->pupil_h, (size_t)Mx * My * sizeof(double2)));
  k_pupil_transfer<<<blocks_for((size_t)Mx * My), 256>>>(Mx, My, P->h, P->kb, k_cut, distance, P->pupil_h);
  LS_CUDA_TRY(cudaDeviceSynchronize());
  return LS_OK;
}

int ls_apply_pupil(ls_plan* P, int n_views, const ls_c64* const* in, ls_c64* const* out, int adjoint, void* stream) {
  lsgpu::TraceRange trace_range("ls_apply_pupil");
  if (!P || n_views < 1 || !in || !out) { set_last_error("bad arguments"); return LS_EINVAL; }
  if (!P->pupil_h) { set_last_error("no pupil set (ls_set_pupil)"); return LS_EINVAL; }
  cudaStream_t st = (cudaStream_t)stream;
  for (int q = 0; q < n_views; ++q)
    if (!in[q] || !out[q]) { set_last_error("null view pointer %d", q); return LS_EINVAL; }
  // planes for all the views of a launch, or for as many as there is memory for
  int most = std::min(n_views, PupilViews::kMax);
  void* scratch = nullptr;
  for (;; most = (most + 1) / 2) {
    const cudaError_t e = injected_alloc_failure() ? cudaErrorMemoryAllocation
                                                   : cudaMallocAsync(&scratch, pupil_scratch_bytes(P, most), st);
    if (e == cudaSuccess) break;
    if (e != cudaErrorMemoryAllocation || most == 1) LS_CUDA_TRY(e);
    cudaGetLastError();
  }
  const int rc = apply_pupil_views(P, n_views, (const void* const*)in, (void* const*)out, adjoint, scratch, most, st);
  LS_CUDA_TRY(cudaFreeAsync(scratch, st));
  return rc;
}

}  // extern "C"
