// The y and z transforms of the Green convolution in one pass (the middle three of the five passes
// described in passes.cuh): for every view and kx, zero-padded FFT along y, zero-padded FFT along z,
// Green multiply and both inverse transforms, with the crops, in place on one [nz][ny] plane.
//
// The first pass stores its spectrum transposed (A1t [kx][nz][ny], IX reads it back the same way), so a
// plane is contiguous and the padded spectra never leave the SM: the matvec moves 28N + 32N + 32N bytes
// instead of 220N (N voxels), in three launches instead of five.
//
// Zero padding to 2ny splits the y transform by the parity of ky into two ny-point transforms of the
// same plane, Y[2j + P] = DFT_ny(x[y] W_2ny^{P y})[j], so only one ny x nz tile is in shared memory at a
// time: the CTA runs P = 0 and then P = 1 (the second read of the plane comes from L2), and keeps the
// first half's partial output in tensor memory, which serves as a register file extension (every
// thread reads back what it wrote).  The factor W_2ny^{P y} is part of the odd half's DFTs (DftOddIn, DftOddOut): as
// a twist of their inputs and outputs it was one rounding more than the three passes have (operator error against
// 64 bits at 48^3 +13%, 96x72x48 +10%, 64^3 +3%; now within 2% of theirs, or below).  A warp owns the same rows in both halves and in both directions,
// so only the two transposes between rows and columns are CTA barriers.
//
// Layout.  y = RB a + b, j = c + RA d: stage A transforms over a (thread b), stage B over b (thread c), in
// place in the row's entries c CS + b.  Rows have an odd pitch and CS is odd, so rows, sub-transforms
// and columns are read without bank conflicts at addresses that are a thread's base plus constants.
// The z transform of a column exchanges through a warp-private area [k1][R2 + 1].
//
// The pass is bound by the shared-memory pipe (64-bit accesses take two wavefronts, broadcast or not),
// so what need not go through it does not: from ny = 48 on the stage twiddles, constants of a lane, are
// read from tensor memory; a thread transforms the columns ky and -ky one after the other with the same
// Green values in registers; the plane and the Green values are read with 16-byte loads.
//
// Measured, us a view against FY, Z and IY as three launches: 128^3 x 60 views 57.0 -> 51.1 (16 views under ncu:
// FMA pipe 58% and shared-memory pipe 64% of their peaks, 80 MB of DRAM traffic a view where the three passes
// move 340), 64^3 x 24 9.4 -> 6.3, 96^3 x 16 28.9 -> 23.3, 144^3 x 1 198 -> 135.  The FP32 instructions alone are
// 29 us a view at 128^3; the rest is the two pipes taking turns between the barriers.
#pragma once

#include "pass_common.cuh"

namespace lsgpu {

struct YzParams {
  SlotSel sel;
  unsigned long long* runs[3];   // profiler counters of the three transforms (null: not counted)
  int nx;
  float2* a1;                    // [slot][2nx][nz][ny], in place
  size_t a1_stride;
  const float2* g;               // Green values [nx+1][ny+1][2nz], scaled by 1/(8 nx ny nz); kz = k1 + R1 k2 is
                                 // entry ((k2 / 2) R1 + k1) 2 + k2 % 2 of a row (one 16-byte load per k2 pair)
  const float2* ytw;             // [2][RA][CS]: exp(-2 pi i b (2c + P) / (2 ny)) at [P][c][b]
  const float2* ztw;             // [R1][R2+1]: exp(-2 pi i k1 n2 / (2 nz)) at [k1][n2]
  const int* cols;               // [2][ny/2][2]: tile position | j << 16 of the column pairs of parity P
  int sms;
  int dbg_probe = 0;             // debug build, test only: a plane's last element is taken as out of range
};

// ny = RA RB on T threads per row.  RB = 2 T where it can be: a thread's loads are then pairs, and a row's are
// contiguous.  us a view, nx = 64, 16M voxels in flight: 48 = 6 8 against 8 6, 48x96 planes 8.6 -> 7.9 and 48x48 4.2 -> 4.0;
// 32 = 4 8 against 8 4, 32x128 7.8 -> 7.4; 72 = 9 8 against 12 6, 72x32 4.6 -> 4.1, 72x128 20.6 -> 19.1 (72x64 8.7 -> 9.2);
// 144 = 9 16 against 12 12, 144x96 33.3 -> 28.0, 144x16 4.9 -> 4.4.
template <int NY> struct YSplit;
template <> struct YSplit<8>   { static constexpr int RA = 4, RB = 2, T = 4; };
template <> struct YSplit<12>  { static constexpr int RA = 4, RB = 3, T = 4; };
template <> struct YSplit<16>  { static constexpr int RA = 4, RB = 4, T = 4; };
template <> struct YSplit<24>  { static constexpr int RA = 4, RB = 6, T = 4; };
template <> struct YSplit<32>   { static constexpr int RA = 4, RB = 8, T = 4; };
template <> struct YSplit<48>   { static constexpr int RA = 6, RB = 8, T = 4; };
template <> struct YSplit<64>  { static constexpr int RA = 8, RB = 8, T = 4; };
template <> struct YSplit<72>   { static constexpr int RA = 9, RB = 8, T = 4; };
template <> struct YSplit<96>  { static constexpr int RA = 12, RB = 8, T = 4; };
template <> struct YSplit<128> { static constexpr int RA = 8, RB = 16, T = 8; };
template <> struct YSplit<144>  { static constexpr int RA = 9, RB = 16, T = 8; };
template <> struct YSplit<192> { static constexpr int RA = 12, RB = 16, T = 8; };
// 2 nz = R1 R2 (R1 even) on T threads per column.  96 = 16 6 and 288 = 24 12 for their rounding (3 coprime to the rest: no
// twiddles inside the DFTs), at the time of 12 8 and 16 18 or less (32x144 10.3 -> 10.0, 128x144 37.7 -> 35.2, but 96x144
// 30.8 -> 32.7).
template <int NZ> struct ZSplit2;
template <> struct ZSplit2<8>   { static constexpr int R1 = 4, R2 = 4, T = 4; };
template <> struct ZSplit2<12>  { static constexpr int R1 = 4, R2 = 6, T = 4; };
template <> struct ZSplit2<16>  { static constexpr int R1 = 8, R2 = 4, T = 4; };
template <> struct ZSplit2<24>  { static constexpr int R1 = 8, R2 = 6, T = 8; };
template <> struct ZSplit2<32>  { static constexpr int R1 = 8, R2 = 8, T = 8; };
template <> struct ZSplit2<48>   { static constexpr int R1 = 16, R2 = 6, T = 8; };
template <> struct ZSplit2<64>  { static constexpr int R1 = 16, R2 = 8, T = 8; };
template <> struct ZSplit2<72>  { static constexpr int R1 = 12, R2 = 12, T = 16; };
template <> struct ZSplit2<96>  { static constexpr int R1 = 24, R2 = 8, T = 8; };
template <> struct ZSplit2<128> { static constexpr int R1 = 16, R2 = 16, T = 16; };
template <> struct ZSplit2<144>  { static constexpr int R1 = 24, R2 = 12, T = 16; };
template <> struct ZSplit2<192> { static constexpr int R1 = 24, R2 = 16, T = 16; };

__host__ __device__ constexpr int cdiv(int a, int b) { return (a + b - 1) / b; }
__host__ __device__ constexpr int imin(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int pow2_at_least(int v, int lo) { return lo >= v ? lo : pow2_at_least(v, 2 * lo); }

template <int NY, int NZ>
struct YZ {
  using Y = YSplit<NY>;
  using Z = ZSplit2<NZ>;
  static constexpr int RA = Y::RA, RB = Y::RB, TY = Y::T, R1 = Z::R1, R2 = Z::R2, TZ = Z::T;
  static_assert(RA * RB == NY && R1 * R2 == 2 * NZ && R1 % 2 == 0 && R2 % 2 == 0, "splits");
  static constexpr int SA = cdiv(RB, TY), SB = cdiv(RA, TY);      // sub-transforms per thread of a row
  static constexpr int S1 = cdiv(R2, TZ), S2 = cdiv(R1, TZ);      // and of a column
  // stage A of a thread is the neighbouring pair b = 2 t, 2 t + 1: 16-byte global loads and stores
  static constexpr bool VEC = SA == 2 && RB % 2 == 0;
  static constexpr int CSP = RB % 2 ? RB + 2 : RB + 1;            // entries between c blocks of a row, odd
  static constexpr int PZ = (RA * CSP - (CSP - RB)) | 1;          // row pitch, odd
  static constexpr int NBLK = cdiv(NZ, 16);
  static constexpr int NRG = cdiv(NBLK * TY, 2);                  // row groups of a warp (32 / TY rows each)
  static constexpr int CPW = 32 / TZ;                             // column pairs per warp
  static constexpr int NCG = cdiv(NY / 2, CPW);
  static constexpr int XR = R2 + 1;
  // columns of a half-warp TZ entries apart modulo 16
  static constexpr int XP0 = R1 * XR;
  static constexpr int XP = TZ >= 16 ? XP0 : XP0 + ((TZ - XP0 % 16) % 16 + 16) % 16;
  static constexpr size_t tile_bytes = (size_t)NZ * PZ * sizeof(float2);
  static constexpr size_t warp_bytes = (size_t)CPW * XP * sizeof(float2);
  static constexpr size_t misc = (kMaxLaunchSlots + 64) * sizeof(int);
  static constexpr size_t budget = 226 * 1024;
  static constexpr size_t ytab_bytes = (size_t)2 * RA * CSP * sizeof(float2), ztab_bytes = (size_t)R1 * XR * sizeof(float2);
  static constexpr size_t col_bytes = (size_t)2 * NY * sizeof(int);
  static constexpr size_t fixed = tile_bytes + ytab_bytes + ztab_bytes + col_bytes + misc;
  static constexpr int room = fixed < budget ? imin(16, (int)((budget - fixed) / warp_bytes)) : 0;
  // Tensor memory, in columns: the partial outputs of a row group (2 RA floats per sub-transform, RA made even), and a
  // lane's twiddles of the z stages and of the y stages of both parities.  Slot of a row group among those
  // of its lane quarter (the warps of a quarter are 4 apart), for w warps:
  static constexpr int RAE = RA + RA % 2, TCOL = SA * 2 * RAE;
  static constexpr __host__ __device__ int slot(int g, int w) { return w % 4 == 0 ? g / 4 : g / w * cdiv(w, 4) + g % w / 4; }
  static constexpr int tpart(int w) { return TCOL * (w % 4 == 0 ? cdiv(NRG, 4) : cdiv(NRG, w) * cdiv(w, 4)); }
  static constexpr int TZW = S1 * 2 * R1 + S2 * 2 * R2, TYW = 4 * SA * RA + 4 * SB * RB;
  static constexpr bool WIDE = NY >= 48 && NZ >= 48;   // twiddles in tensor memory pay
  // Warps of a CTA: the share of the warps' time that the row and the column phases keep busy (work of a
  // group ~ its FFT length times log), times the warps that fit an SM (up to 512 threads; beyond 12 warps
  // little is gained); of the counts that leave no warp without work in both phases the largest within a
  // tenth of the best, which makes a single plane fastest.
  static constexpr int lg(int v) { return v <= 1 ? 0 : 1 + lg(v / 2); }
  static constexpr double wr = 2.0 * (32 / TY) * NY * lg(NY), wc = 3.4 * CPW * (2 * NZ) * lg(2 * NZ);
  static constexpr int per_sm(int w) {
    const int by_smem = (int)(228 * 1024 / (fixed + w * warp_bytes + 1024));
    const int by_tmem = 512 / pow2_at_least(tpart(w) + (WIDE ? TZW : 0), 32);
    return imin(imin(imin(16, 512 / (32 * w)), by_smem), by_tmem);
  }
  static constexpr double score(int w) {
    const int warps = w * per_sm(w);
    return (warps < 12 ? warps : 12) * (NRG * wr + NCG * wc) / (w * (cdiv(NRG, w) * wr + cdiv(NCG, w) * wc));
  }
  static constexpr int choose_warps() {
    double best = 0;
    for (int w = 1; w <= room; ++w) best = score(w) > best ? score(w) : best;
    for (int w = room; w > 0; --w)
      if (best > 0 && score(w) >= 0.9 * best && (w == cdiv(NRG, cdiv(NRG, w)) || w == cdiv(NCG, cdiv(NCG, w)))) return w;
    return 1;
  }
  static constexpr int NW = choose_warps();
  static constexpr bool ok = room > 0 && score(NW) > 0 && NW * per_sm(NW) >= imin(8, imax(NRG, NCG));
  static constexpr int NT = 32 * NW;
  static constexpr int MINB0 = imax(1, per_sm(NW));
  static constexpr int TZ1 = tpart(NW), TZ2 = TZ1 + S1 * 2 * R1, TYA = TZ1 + TZW, TYB = TYA + 4 * SA * RA;
  static constexpr bool ZT = WIDE;
  static constexpr bool YT = ZT && RA % 2 == 0 && pow2_at_least(TYA + TYW, 32) * MINB0 <= 512;
  static constexpr int TMEM = pow2_at_least(YT ? TYA + TYW : ZT ? TYA : TZ1, 32);
  static constexpr int MINB = MINB0;
  // the next half's first rows are loaded before the inverse y transform where the registers allow it
  // (at 128 a thread they would spill: 57 instead of 52 us a view at 128^3)
  static constexpr bool CROSS = 65536 / (NT * MINB) >= 160;
  // Against FY, Z and IY as three launches, measured over all pairs of lengths with nx = 64: one view, 1.1 to
  // 2.2 times as fast wherever the tile fits; 16M voxels in flight, 1.0 to 1.5 times (24x72 and 24x192 0.93 and 0.97),
  // but 0.85 to 0.92 of their rate with ny = 72 and nz = 128 and more (72x72 1.01), 0.91 and 0.98 with ny = 144 and
  // nz = 144 and 72 (a quarter to a half of the lanes idle in one of their stages, eight or nine warps an SM), 0.79 to
  // 1.05 with nz = 8, and 0.65 to 0.71 with ny = 8 and nz = 48 and 64 (few warps; 1.1 to 1.5 from nz = 72 on, where the
  // line could move).
  static constexpr bool large_ok = !(NY == 72 && NZ >= 72 && NZ != 96) && !(NY == 144 && (NZ == 72 || NZ == 144)) &&
                                   NZ != 8 && !(NY == 8 && NZ >= 48);
  static constexpr size_t smem_z = tile_bytes + col_bytes + (size_t)NW * warp_bytes;
  static constexpr size_t smem = smem_z + (YT ? 0 : ytab_bytes) + (ZT ? 0 : ztab_bytes);
};

__device__ __forceinline__ void tmem_alloc(unsigned* dst, int ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_free(unsigned addr, int ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(addr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
// A warp's lane i stores / loads N complex values in its lane of tensor memory, columns addr .. addr + 2N - 1
// (warp-collective).  Loaded values may be used after tmem_loaded().
template <int N>
__device__ __forceinline__ void tmem_st(unsigned addr, const float2* v) {
  static_assert(N % 2 == 0, "pairs");
  if constexpr (N >= 4) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n"
                 ::"r"(addr), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y), "f"(v[2].x), "f"(v[2].y),
                 "f"(v[3].x), "f"(v[3].y) : "memory");
    if constexpr (N > 4) tmem_st<N - 4>(addr + 8, v + 4);
  } else {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n"
                 ::"r"(addr), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y) : "memory");
  }
}
template <int N>
__device__ __forceinline__ void tmem_ld(unsigned addr, float2* v) {
  static_assert(N % 2 == 0, "pairs");
  if constexpr (N >= 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15}, [%16];\n"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x),
                   "=f"(v[3].y), "=f"(v[4].x), "=f"(v[4].y), "=f"(v[5].x), "=f"(v[5].y), "=f"(v[6].x), "=f"(v[6].y),
                   "=f"(v[7].x), "=f"(v[7].y) : "r"(addr) : "memory");
    if constexpr (N > 8) tmem_ld<N - 8>(addr + 16, v + 8);
  } else if constexpr (N >= 4) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x),
                   "=f"(v[3].y) : "r"(addr) : "memory");
    if constexpr (N > 4) tmem_ld<N - 4>(addr + 8, v + 4);
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y) : "r"(addr) : "memory");
  }
}
// Completes this thread's tensor-memory loads; the values pass through the barrier, so that no use of
// them moves before it.
template <int N>
__device__ __forceinline__ void tmem_loaded(float2* v) {
  tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+f"(v[i].x), "+f"(v[i].y));
}

// Twiddles 0 .. N - 1 of one sub-transform times its values, and the store of every product: from tensor
// memory in pieces of at most eight (TM, warp-collective; lanes without `has` only take part in the loads),
// else from the shared table at tab + k TS.  put(k, value).
template <int N, bool CONJ, bool TM, bool SKIP0, class Put>
__device__ __forceinline__ void twiddle_out(const float2* v, unsigned taddr, const float2* tab, int ts, bool has, Put&& put) {
  if constexpr (TM) {
    constexpr int M = N < 8 ? N : 8;
    float2 w[M];
    tmem_ld<M>(taddr, w);
    tmem_loaded<M>(w);
    if (has) {
#pragma unroll
      for (int k = 0; k < M; ++k) put(k, SKIP0 && k == 0 ? v[0] : CONJ ? cmulc(v[k], w[k]) : cmul(v[k], w[k]));
    }
    if constexpr (N > M)
      twiddle_out<N - M, CONJ, TM, false>(v + M, taddr + 2 * M, tab, ts, has, [&](int k, float2 x) { put(M + k, x); });
  } else {
    if (has) {
#pragma unroll
      for (int k = 0; k < N; ++k) {
        if (SKIP0 && k == 0) put(0, v[0]);
        else put(k, CONJ ? cmulc(v[k], tab[k * ts]) : cmul(v[k], tab[k * ts]));
      }
    }
  }
}

template <int NY, int NZ>
__global__ void __launch_bounds__(YZ<NY, NZ>::NT, YZ<NY, NZ>::MINB) k_yz(YzParams a) {
  pdl_begin();
  using W = YZ<NY, NZ>;
  constexpr int RA = W::RA, RB = W::RB, TY = W::TY, SA = W::SA, SB = W::SB, CSP = W::CSP, PZ = W::PZ;
  constexpr int R1 = W::R1, R2 = W::R2, TZ = W::TZ, S1 = W::S1, S2 = W::S2, XR = W::XR, CPW = W::CPW, NW = W::NW;
  constexpr bool VEC = W::VEC, ZT = W::ZT, YT = W::YT;
  extern __shared__ __align__(16) float2 yz_sm[];
  float2* tile = yz_sm;
  float2* xall = tile + NZ * PZ;
  int* cols = reinterpret_cast<int*>(xall + NW * CPW * W::XP);
  float2* ytw = reinterpret_cast<float2*>(cols + 2 * NY);   // where not in tensor memory
  float2* ztw = ytw + (YT ? 0 : 2 * RA * CSP);
  __shared__ int s_list[kMaxLaunchSlots];
  __shared__ int s_ws[32];
  __shared__ unsigned s_tmem;
  const int nact = build_active(a.sel, s_list, s_ws);
  if (nact == 0) return;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ty = lane % TY, tz = lane % TZ;
  if (warp == 0) tmem_alloc(&s_tmem, W::TMEM);
  if constexpr (!YT)
    for (int i = tid; i < 2 * RA * CSP; i += W::NT) ytw[i] = __ldg(a.ytw + i);
  if constexpr (!ZT)
    for (int i = tid; i < R1 * XR; i += W::NT) ztw[i] = __ldg(a.ztw + i);
  for (int i = tid; i < 2 * NY; i += W::NT) cols[i] = __ldg(a.cols + i);
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tq = s_tmem + ((unsigned)(warp & 3) << 21);   // this warp's lanes
  if (ZT && warp < 4) {
    // the first warp of each lane quarter stores the twiddles of its lanes
#pragma unroll 1
    for (int s = 0; s < S1; ++s) {
      float2 w[R1];
#pragma unroll
      for (int k = 0; k < R1; ++k) w[k] = __ldg(a.ztw + k * XR + imin(tz + TZ * s, R2 - 1));
      tmem_st<R1>(tq + W::TZ1 + s * 2 * R1, w);
    }
#pragma unroll 1
    for (int s = 0; s < S2; ++s) {
      float2 w[R2];
#pragma unroll
      for (int j = 0; j < R2; ++j) w[j] = __ldg(a.ztw + imin(tz + TZ * s, R1 - 1) * XR + j);
      tmem_st<R2>(tq + W::TZ2 + s * 2 * R2, w);
    }
    if constexpr (YT) {
#pragma unroll 1
      for (int i = 0; i < 2 * SA; ++i) {   // parity i / SA, sub-transform i % SA
        float2 w[RA];
        const int b = imin(VEC ? 2 * ty + i % SA : ty + TY * (i % SA), RB - 1);
#pragma unroll
        for (int c = 0; c < RA; ++c) w[c] = __ldg(a.ytw + ((i / SA) * RA + c) * CSP + b);
        tmem_st<RA>(tq + W::TYA + i * 2 * RA, w);
      }
#pragma unroll 1
      for (int i = 0; i < 2 * SB; ++i) {
        float2 w[RB];
        const int c = imin(ty + TY * (i % SB), RA - 1);
#pragma unroll
        for (int b = 0; b < RB; ++b) w[b] = __ldg(a.ytw + ((i / SB) * RA + c) * CSP + b);
        tmem_st<RB>(tq + W::TYB + i * 2 * RB, w);
      }
    }
    tmem_wait_st();
  }
  if constexpr (ZT) {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  }
  const int njobs = nact * 2 * a.nx;
  // Rows of this lane in row group g.  A group is 32 / TY rows of a block of 16: the rows a half-warp
  // takes in stage B are TY apart; in stage A with pairs (VEC) they are neighbours (and 8 apart), which
  // puts the entries 2 t of neighbouring rows on even and odd banks.
  const int half = lane >> 4, r = (lane & 15) / TY;
  auto row_b = [&](int g) {
    if constexpr (VEC) return (g / (TY / 2)) * 16 + 2 * (g % (TY / 2)) + half + TY * r;
    else return ((2 * g + half) / TY) * 16 + (2 * g + half) % TY + TY * r;
  };
  auto row_a = [&](int g) {
    if constexpr (VEC) return (g / (TY / 2)) * 16 + 2 * (g % (TY / 2)) + TY * half + (r & 1) + 8 * (r >> 1);
    else return row_b(g);
  };
  auto sub_a = [&](int s) { return VEC ? 2 * ty + s : ty + TY * s; };   // b of stage A
  float2* xc = xall + (warp * CPW + lane / TZ) * W::XP;
  // This lane's part of row group g of a plane (lanes past the last row or sub-transform read a
  // neighbour's): the loads of a group are issued while the one before it, or the inverse transform of
  // the half before, is still at work.
  float2 v[SA][RA];
  auto load_rows = [&](const float2* plane, int g) {
    const int z = NZ % 16 == 0 ? row_a(g) : imin(row_a(g), NZ - 1);
    if constexpr (VEC) {
      const int o = z * NY + (SA * TY == RB ? 2 * ty : imin(2 * ty, RB - 2));
#pragma unroll
      for (int i = 0; i < RA; ++i) {
        if (!LS_IN_BOUNDS(o + RB * i + 1 < NY * NZ, BS_YZ_PLANE)) continue;
        const float4 q = *reinterpret_cast<const float4*>(plane + o + RB * i);
        v[0][i] = make_float2(q.x, q.y);
        v[SA - 1][i] = make_float2(q.z, q.w);
      }
    } else {
#pragma unroll
      for (int s = 0; s < SA; ++s) {
        const int o = z * NY + (SA * TY == RB ? sub_a(s) : imin(sub_a(s), RB - 1));
#pragma unroll
        for (int i = 0; i < RA; ++i)
          if (LS_IN_BOUNDS(o + RB * i < NY * NZ, BS_YZ_PLANE)) v[s][i] = plane[o + RB * i];
      }
    }
  };
  auto plane_of = [&](int job) {
    return a.a1 + (size_t)active_slot(s_list[job / (2 * a.nx)]) * a.a1_stride + (size_t)(job % (2 * a.nx)) * (NY * NZ);
  };
  if (W::CROSS && (int)blockIdx.x < njobs && warp < W::NRG) load_rows(plane_of(blockIdx.x), warp);
#pragma unroll 1
  for (int job = blockIdx.x; job < njobs; job += gridDim.x) {
    const int ent = s_list[job / (2 * a.nx)], kx = job % (2 * a.nx);
    const int slot = active_slot(ent);
    if (!LS_IN_BOUNDS(slot < a.sel.nslots && (a.sel.nslots <= 1 || (size_t)2 * a.nx * NY * NZ <= a.a1_stride), BS_SLOT))
      continue;
    if (kx == 0 && tid < 3 && a.runs[tid]) atomicAdd(a.runs[tid], 1ull);
    float2* plane = a.a1 + (size_t)slot * a.a1_stride + (size_t)kx * (NY * NZ);
    const float2* gx = a.g + (size_t)(kx <= a.nx ? kx : 2 * a.nx - kx) * ((NY + 1) * (2 * NZ));
    const bool adj = active_adj(ent);
#pragma unroll 1
    for (int P = 0; P < 2; ++P) {
      const float2* yt = ytw + P * RA * CSP;
      if (!W::CROSS && warp < W::NRG) load_rows(plane, warp);
      // ---- forward y transform of this warp's rows
#pragma unroll 1
      for (int g = warp; g < W::NRG; g += NW) {
        {
          const int z = row_a(g);
          const bool has = NZ % 16 == 0 || z < NZ;
          float2* row = tile + z * PZ;
#pragma unroll
          for (int s = 0; s < SA; ++s) {
            const int b = sub_a(s);
            const bool mine = has && (SA * TY == RB || b < RB);
            if (P) DftOddIn<RA, -1>::run(v[s]);
            else Dft<RA, -1>::run(v[s]);
            twiddle_out<RA, false, YT, false>(v[s], tq + W::TYA + (P * SA + s) * 2 * RA, yt + (mine ? b : 0), CSP, mine,
                                              [&](int c, float2 x) {
              if (LS_IN_BOUNDS(z * PZ + c * CSP + b < NZ * PZ, BS_YZ_TILE)) row[c * CSP + b] = x;
            });
          }
          if (g + NW < W::NRG) load_rows(plane, g + NW);
        }
        __syncwarp();
        {
          const int z = row_b(g);
          float2* row = tile + z * PZ;
          if (NZ % 16 == 0 || z < NZ) {
#pragma unroll
            for (int s = 0; s < SB; ++s) {
              const int c = ty + TY * s;
              if (RA % TY == 0 || c < RA) {
                float2 u[RB];
#pragma unroll
                for (int b = 0; b < RB; ++b)
                  if (LS_IN_BOUNDS(z * PZ + c * CSP + b < NZ * PZ, BS_YZ_TILE)) u[b] = row[c * CSP + b];
                Dft<RB, -1>::run(u);
#pragma unroll
                for (int d = 0; d < RB; ++d)
                  if (LS_IN_BOUNDS(z * PZ + c * CSP + d < NZ * PZ, BS_YZ_TILE)) row[c * CSP + d] = u[d];
              }
            }
          }
        }
      }
      __syncthreads();
      // ---- z transform, Green multiply and inverse z transform of this warp's column pairs
#pragma unroll 1
      for (int cg = warp; cg < W::NCG; cg += NW) {
        const int q = cg * CPW + lane / TZ;
        const bool has = (NY / 2) % CPW == 0 || q < NY / 2;
        float2 gv[S2][R2];
        int fold = -1;
#pragma unroll 1
        for (int e = 0; e < 2; ++e) {
          const int pj = cols[(P * (NY / 2) + (has ? q : 0)) * 2 + e];
          float2* col = tile + (pj & 0xffff);
          const int ky = 2 * (pj >> 16) + P;
          const int fy = ky <= NY ? ky : 2 * NY - ky;
          if (fy != fold) {
            // Green values of this thread's stage-2 sub-transforms, in flight during stage 1
            fold = fy;
            const float4* gc = reinterpret_cast<const float4*>(gx + fy * (2 * NZ));
#pragma unroll
            for (int s = 0; s < S2; ++s) {
              const int k1 = R1 % TZ == 0 ? tz + TZ * s : imin(tz + TZ * s, R1 - 1);
              if (LS_IN_BOUNDS(ky >= 0 && ky < 2 * NY && k1 < R1, BS_YZ_GREEN)) {
#pragma unroll
                for (int h = 0; h < R2 / 2; ++h) {
                  const float4 x = __ldg(gc + h * R1 + k1);
                  gv[s][2 * h] = make_float2(x.x, x.y);
                  gv[s][2 * h + 1] = make_float2(x.z, x.w);
                }
              }
            }
          }
#pragma unroll
          for (int s = 0; s < S1; ++s) {
            const int n2 = tz + TZ * s;
            const bool mine = has && (R2 % TZ == 0 || n2 < R2);
            const float2* src = col + (R2 % TZ == 0 ? n2 : imin(n2, R2 - 1)) * PZ;
            float2 v[R1];
#pragma unroll
            for (int n1 = 0; n1 < R1 / 2; ++n1)
              if (LS_IN_BOUNDS(src + R2 * n1 * PZ >= tile && src + R2 * n1 * PZ < tile + NZ * PZ, BS_YZ_TILE))
                v[n1] = src[R2 * n1 * PZ];
            Dft<R1, -1, R1 / 2, R1>::run(v);
            twiddle_out<R1, false, ZT, true>(v, tq + W::TZ1 + s * 2 * R1, ztw + (mine ? n2 : 0), XR, mine, [&](int k1, float2 x) {
              if (LS_IN_BOUNDS(k1 * XR + n2 < W::XP, BS_YZ_EXCH)) xc[k1 * XR + n2] = x;
            });
          }
          __syncwarp();
#pragma unroll
          for (int s = 0; s < S2; ++s) {
            const int k1 = tz + TZ * s;
            const bool mine = has && (R1 % TZ == 0 || k1 < R1);
            float2* ex = xc + (R1 % TZ == 0 ? k1 : imin(k1, R1 - 1)) * XR;
            float2 u[R2];
#pragma unroll
            for (int n2 = 0; n2 < R2; ++n2)
              if (LS_IN_BOUNDS(ex - xc + n2 < W::XP, BS_YZ_EXCH)) u[n2] = ex[n2];
            Dft<R2, -1>::run(u);
            if (adj) {
#pragma unroll
              for (int k2 = 0; k2 < R2; ++k2) u[k2] = cmulc(u[k2], gv[s][k2]);
            } else {
#pragma unroll
              for (int k2 = 0; k2 < R2; ++k2) u[k2] = cmul(u[k2], gv[s][k2]);
            }
            Dft<R2, +1>::run(u);
            // in place: entry [k1][j1] is read by the thread of j1 in the last stage
            twiddle_out<R2, true, ZT, true>(u, tq + W::TZ2 + s * 2 * R2, ztw + (mine ? k1 : 0) * XR, 1, mine,
                                            [&](int j1, float2 x) {
              if (LS_IN_BOUNDS(ex - xc + j1 < W::XP, BS_YZ_EXCH)) ex[j1] = x;
            });
          }
          __syncwarp();
          if (has) {
#pragma unroll
            for (int s = 0; s < S1; ++s) {
              const int j1 = tz + TZ * s;
              if (R2 % TZ == 0 || j1 < R2) {
                float2 w[R1];
#pragma unroll
                for (int k1 = 0; k1 < R1; ++k1)
                  if (LS_IN_BOUNDS(k1 * XR + j1 < W::XP, BS_YZ_EXCH)) w[k1] = xc[k1 * XR + j1];
                Dft<R1, +1, R1, R1 / 2>::run(w);
#pragma unroll
                for (int j2 = 0; j2 < R1 / 2; ++j2)
                  if (LS_IN_BOUNDS((pj & 0xffff) + (j1 + R2 * j2) * PZ < NZ * PZ, BS_YZ_TILE)) col[(j1 + R2 * j2) * PZ] = w[j2];
              }
            }
          }
          __syncwarp();
        }
      }
      // the rows of the next half: of this plane again, or of the CTA's next plane
      if (W::CROSS && warp < W::NRG) {
        if (P == 0) load_rows(plane, warp);
        else if (job + (int)gridDim.x < njobs) load_rows(plane_of(job + (int)gridDim.x), warp);
      }
      __syncthreads();
      // ---- inverse y transform of this warp's rows; P = 0 keeps its half in tensor memory, P = 1 adds it
#pragma unroll 1
      for (int g = warp; g < W::NRG; g += NW) {
        {
          const bool has = NZ % 16 == 0 || row_b(g) < NZ;
          const int z = NZ % 16 == 0 ? row_b(g) : imin(row_b(g), NZ - 1);
#pragma unroll
          for (int s = 0; s < SB; ++s) {
            const int c = RA % TY == 0 ? ty + TY * s : imin(ty + TY * s, RA - 1);
            const bool mine = has && (RA % TY == 0 || ty + TY * s < RA);
            float2* row = tile + z * PZ + c * CSP;
            float2 u[RB];
#pragma unroll
            for (int d = 0; d < RB; ++d)
              if (LS_IN_BOUNDS(z * PZ + c * CSP + d < NZ * PZ, BS_YZ_TILE)) u[d] = row[d];
            Dft<RB, +1>::run(u);
            twiddle_out<RB, true, YT, false>(u, tq + W::TYB + (P * SB + s) * 2 * RB, yt + c * CSP, 1, mine,
                                             [&](int b, float2 x) {
              if (LS_IN_BOUNDS(z * PZ + c * CSP + b < NZ * PZ, BS_YZ_TILE)) row[b] = x;
            });
          }
        }
        __syncwarp();
        {
          const bool has = NZ % 16 == 0 || row_a(g) < NZ;
          const int z = NZ % 16 == 0 ? row_a(g) : imin(row_a(g), NZ - 1);
          const float2* row = tile + z * PZ;
          float2 o[SA][W::RAE] = {};
#pragma unroll
          for (int s = 0; s < SA; ++s) {
            const int b = SA * TY == RB ? sub_a(s) : imin(sub_a(s), RB - 1);
#pragma unroll
            for (int c = 0; c < RA; ++c)
              if (LS_IN_BOUNDS(z * PZ + c * CSP + b < NZ * PZ, BS_YZ_TILE)) o[s][c] = row[c * CSP + b];
            if (P) DftOddOut<RA, +1>::run(o[s]);
            else Dft<RA, +1>::run(o[s]);
            // tensor-memory accesses are warp-collective: every lane takes part, with its own values
            const unsigned ta = tq + (unsigned)(W::slot(g, NW) * W::TCOL + s * 2 * W::RAE);
            if (P == 0) {
              tmem_st<W::RAE>(ta, o[s]);
            } else {
              float2 w[W::RAE];
              tmem_ld<W::RAE>(ta, w);
              tmem_loaded<W::RAE>(w);
#pragma unroll
              for (int i = 0; i < RA; ++i) o[s][i] = cadd(o[s][i], w[i]);
            }
          }
          if (P == 0) {
            tmem_wait_st();
          } else if constexpr (VEC) {
            if (has && (RB % (2 * TY) == 0 || sub_a(0) < RB)) {
#pragma unroll
              for (int i = 0; i < RA; ++i)
                if (LS_IN_BOUNDS(z * NY + RB * i + sub_a(0) + 1 < NY * NZ - (a.dbg_probe ? 1 : 0), BS_YZ_PLANE))
                  *reinterpret_cast<float4*>(plane + z * NY + RB * i + sub_a(0)) =
                      make_float4(o[0][i].x, o[0][i].y, o[SA - 1][i].x, o[SA - 1][i].y);
            }
          } else {
#pragma unroll
            for (int s = 0; s < SA; ++s)
              if (has && (RB % TY == 0 || sub_a(s) < RB)) {
#pragma unroll
                for (int i = 0; i < RA; ++i)
                  if (LS_IN_BOUNDS(z * NY + RB * i + sub_a(s) < NY * NZ - (a.dbg_probe ? 1 : 0), BS_YZ_PLANE))
                    plane[z * NY + RB * i + sub_a(s)] = o[s][i];
              }
          }
        }
        __syncwarp();
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == 0) tmem_free(s_tmem, W::TMEM);
}

// One fused form per (ny, nz): its launcher, and the splits that its tables follow.  run == null: none (the
// tile does not fit an SM: grids of 192 with 128 and more on the other axis).
struct YzLaunch {
  void (*run)(const YzParams&, int nslots, cudaStream_t) = nullptr;
  cudaError_t (*setup)() = nullptr;
  int ra = 0, rb = 0, csp = 0, r1 = 0, r2 = 0, xr = 0, tz = 0;
  int minb = 0;         // resident CTAs per SM
  bool large_ok = false;   // faster than the three passes at every launch size, else only up to two waves
};

template <int NY, int NZ>
struct YzImpl {
  using W = YZ<NY, NZ>;
  static void run(const YzParams& a0, int nslots, cudaStream_t st) {
    YzParams a = a0;
    a.sel.nslots = nslots;
    const int jobs = 2 * a.nx * nslots;
    launch_pdl((size_t)a.nx * NY * NZ, k_yz<NY, NZ>, imin(jobs, a.sms * W::MINB), W::NT, W::smem, st, a);
  }
  static cudaError_t setup() {
    return cudaFuncSetAttribute(k_yz<NY, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W::smem);
  }
  static YzLaunch table() {
    YzLaunch t;
    if constexpr (W::ok) {
      static_assert(W::TMEM * W::MINB <= 512, "resident CTAs share the tensor memory");
      t.run = &run;
      t.setup = &setup;
      t.minb = W::MINB;
      t.large_ok = W::large_ok;
      t.ra = W::RA; t.rb = W::RB; t.csp = W::CSP; t.r1 = W::R1; t.r2 = W::R2; t.xr = W::XR; t.tz = W::TZ;
    }
    return t;
  }
};

// yz_row_<NY>(nz): the fused form of (NY, nz); one translation unit per NY (yz_*.cu)
#define LS_YZ_LENGTHS(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(72) X(96) X(128) X(144) X(192)
#define LS_YZ_DECLARE(N) \
  YzLaunch yz_row_##N(int nz); \
  unsigned bounds_site_yz_##N(bool clear);
LS_YZ_LENGTHS(LS_YZ_DECLARE)
#undef LS_YZ_DECLARE

template <int NY>
YzLaunch yz_row(int nz) {
  switch (nz) {
#define LS_YZ_CASE(N) case N: return YzImpl<NY, N>::table();
    LS_YZ_LENGTHS(LS_YZ_CASE)
#undef LS_YZ_CASE
    default: return YzLaunch();
  }
}
#define LS_DEFINE_YZ(N) \
  YzLaunch yz_row_##N(int nz) { return yz_row<N>(nz); } \
  LS_BOUNDS_READER(yz_##N)

}  // namespace lsgpu
