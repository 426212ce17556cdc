// Fused kernels of one RK4 right-hand-side evaluation and its stage update,
// templated on the precision T and the grid size N (N = 2^a or 3*2^a). The
// generic passes also take per-direction point counts (Sec. 2 footnote): N is
// then the count along x, NY and NZ those along y and z (defaults N).
//
// Per RK4 stage (Eq. NSfinal with the Appendix's RK4 driver) the state goes
// through four passes over HBM:
//   y-inverse  : complex inverse transform along y of the 6 fields u, omega
//   z-pass     : c2r along z of the 6 fields, u x omega in registers/shared
//                memory (Eq. curl_convection), r2c along z of the 3 products;
//                only kz < N/3 is written (the rest is removed by the 2/3 mask)
//   y-forward  : forward transform along y, only |ky| < N/3 rows written
//   x-stage    : forward transform along x, dealias mask, projection
//                N - k (k.N)/|k|^2, viscous term -nu |k|^2 u, RK4 axpy, then
//                curl i k x u of the new stage state and the inverse transform
//                along x of u and omega for the next stage (the paper's slab
//                transposes become the change of pass direction).
// Physical fields never leave the z-pass. Spectral arrays use the layout
// [component][kz][ky][kx], kz < N/2, kx and ky in FFT order.
#pragma once

#include <cuda.h>  // CUtensorMap

#include <type_traits>

#include "dns_internal.h"
#include "fft_core.cuh"
#include "fixed_point.cuh"

namespace dns {

constexpr int XP_THREADS = 192;  // 6 warps: one per line of a row (u, omega)
constexpr int YP_THREADS = 256;
// z-pass: 12 warps for the 24 + 12 lines of an FP64 tile of 4 columns
template <typename T>
constexpr int ZP_THREADS = sizeof(T) == 8 ? 384 : 256;
constexpr int DG_THREADS = 256;

constexpr int pow2_part(int n) {
  int r = 1;
  while (n % (r * 2) == 0) r *= 2;
  return r;
}
constexpr int cmin(int a, int b) { return a < b ? a : b; }
constexpr int odd_ld(int lines) { return (lines % 2) ? lines : lines + 1; }
constexpr int igcd(int a, int b) { return b == 0 ? a : igcd(b, a % b); }
constexpr int ilcm(int a, int b) { return a / igcd(a, b) * b; }

// Tile layout of k_zpass for lines of M values in FP32: row p + p / PAD of LD values, LD = RES modulo 16 (a row
// of 16 values meets every bank), chosen by counting the bank conflicts of the passes of warp_fft_lines over
// all (PAD, RES) and the tile widths 4 to 32. Shared-memory cycles of a line's transform, PAD 16 and odd rows -> these:
// M = 64 32 -> 16, 48 24 -> 12.4, 32 20 -> 12, 24 13.5 -> 8.1, 16 (4 x 4) 13 -> 4, 12 9.8 -> 4.5; the others keep
// the former, which no layout beats in that count (96: 56 to 58 cycles, best 56; 128: 48). Even rows are filled by
// 16-byte copies.
// z-pass, with the c2r pairs formed in the first pass of the line transforms (one pass over the tile less):
// 128^3 36.8 -> 26.6 us, 64^3 12.3 -> 10.3, 96^3 22.9 -> 20.5; a step of 128 runs of 32^3 .. 96^3 9.05 -> 8.26 ms.
template <int M>
struct ZLay {
  static constexpr int PAD = M == 12 || M == 16 ? 4 : (M == 24 || M == 32 || M == 64 ? 8 : 16);
  static constexpr int RES = M == 12 || M == 16 ? 4 : (M == 24 ? 6 : (M == 32 || M == 64 ? 2 : (M == 48 ? 11 : -1)));
  static constexpr int ROWS = padrow<PAD>(M - 1) + 1;
  static constexpr int ld(int lines) { return RES < 0 ? lines | 1 : lines + (RES - lines % 16 + 16) % 16; }
};

// Grid of N x NY x NZ points (x, y, z); the spectral fields hold kz < NZ/2.
template <typename T, int N, int NY = N, int NZ = N>
struct Geometry {
  static constexpr int M = NZ / 2;
  static constexpr size_t FS = (size_t)M * NY * N;  // complex values per field
  // length of the twiddle table exp(-2 pi i t / TW): every line length divides it
  static constexpr int TW = ilcm(ilcm(N, NY), NZ);
  static constexpr int CB = (int)sizeof(cx<T>);
  // x-pass: one row (fixed kz, ky) per block, 6 padded line buffers. The
  // stage update (XPRE, where it fits in 100 KB) uses 3 padded lines (the
  // nonlinear term, then u) and 9 unpadded rows that receive the stage's state
  // rows by asynchronous copies (then omega in rows 0-2 and the padded work lines of the
  // omega transforms over rows 3-8).
  // Where 6 padded lines and the 9 rows fit in 64 KB (XWIDE), omega keeps
  // its own 3 padded lines instead (faster at N = 512 FP32).
  static constexpr int XLS = padt_len<T>(N);
  static constexpr bool XWIDE = (size_t)((6 * XLS + 1) / 2 * 2 + 9 * N) * CB <= 64 * 1024;
  static constexpr int XST = ((XWIDE ? 6 : 3) * XLS + 1) / 2 * 2;  // 16-byte aligned start of the state rows
  static constexpr bool XPRE = CB == 8 && (size_t)(XST + 9 * N) * CB <= 100 * 1024;
  // Rows of 1 KB and more arrive by bulk copies instead (one thread issues them; no asynchronous copy per value:
  // those took a quarter of the shared-memory pipe's cycles): x-stage 512^3 816 -> 696 us (its bytes: 670 at the
  // copy bandwidth), 1024^3 8.02 -> 7.26 ms, 1024 x 512 x 256 1022 -> 925 us, 256^3 103 -> 95 us, 128^3
  // with every row 37.0 -> 35.8 us; shorter rows keep the copies per value (by bulk copies too 96^3
  // takes 14.4 us where it takes 15.3, 64^3 9.5 for 9.9, 32^3 and less the same).
  static constexpr bool XBULK = XPRE && N >= 128;
  static constexpr size_t XSMEM = (size_t)6 * XLS * CB;
  static constexpr size_t XSMEM_ST = XPRE ? (size_t)(XST + 9 * N) * CB : XSMEM;  // XM_STAGE, XM_RHS
  // z-pass: ZTX adjacent x at fixed y, 6 fields of M values each, <= 112 KB
  // (two blocks per SM); rows narrower than one 32-byte sector may use up to 200 KB.
  static constexpr size_t zbytes(int t) {
    return CB == 8 ? (size_t)ZLay<M>::ROWS * ZLay<M>::ld(6 * t) * CB : (size_t)padt_len<T>(M) * odd_ld(6 * t) * CB;
  }
  static constexpr size_t ZBLOCK = (CB == 16 ? 113 : 112) * 1024;  // half an SM's shared memory
  static constexpr int ztx() {
    int t = cmin(16, pow2_part(N));
    while (t > 1 && zbytes(t) > ZBLOCK && !(t * CB <= 32 && zbytes(t) <= 200 * 1024)) t /= 2;
    return t;
  }
  static constexpr int ZTX = ztx();
  // Minimum resident blocks per SM for the register cap: lines longer than 4 KB
  // hold 32+ registers of data per lane in the warp FFT, so allow more registers.
  static constexpr int LINE_BYTES = N * CB;
  static constexpr int XMIN = CB == 16 ? (N <= 256 ? 4 : (N <= 512 ? 3 : 2)) : (LINE_BYTES > 4096 ? 2 : 4);
  static constexpr int ZMIN = (M * CB > 4096) ? 1 : (CB == 8 && M <= 64 ? (M == 48 ? 3 : 4) : 2);
  static constexpr int ZLD = odd_ld(6 * ZTX);
  static constexpr size_t ZSMEM = zbytes(ZTX);
};

// Tile of the y-pass by direction: 128-byte rows (64-byte rows for the FP32 forward pass and above 512 points).
// SHORT: FP32 lines of up to 128 points (yshort_tile), 4 warps that take several columns each. FP64: one column per
// warp. FP32 lines of 256 points and more run through k_yreg; k_ypass is left to products_low there
// (k_yreg was not tried for it).
// TXO > 0 replaces the tile width (a tuned schedule of the small grids).
// NY: the line length (points along y) where it differs from N (the x extent).
template <typename T, int N, int INV, int TXO = 0, int NY = N>
struct YCfg {
  static constexpr int CB = (int)sizeof(cx<T>);
  static constexpr int TX = TXO > 0 ? TXO : cmin(((INV || CB == 16) && NY <= 512 ? 128 : 64) / CB, pow2_part(N));
  static constexpr bool SHORT = CB == 8 && NY <= 128;  // yshort_tile
  static constexpr int THREADS = cmin(32 * TX, SHORT ? 128 : 256);
  static constexpr int LD = SHORT ? ZLay<NY>::ld(TX) : odd_ld(TX);
  static constexpr size_t SMEM = (size_t)(SHORT ? ZLay<NY>::ROWS : padt_len<T>(NY)) * LD * CB;
  // short tiles: 4, 6 and 8 blocks an SM measured alike
  static constexpr int MINB = SHORT ? 6 : (CB == 16 ? (NY <= 256 ? 3 : 2) : (NY <= 512 ? (INV ? 3 : 4) : 2));
};

__device__ __forceinline__ int kfreq(int i, int N) { return i < N / 2 ? i : i - N; }

// the launch parameters with their FP32 copies filled in
inline PassArgs f32args(PassArgs a) {
  a.f_nu = (float)a.nu;
  a.f_cA = (float)a.cA;
  a.f_cB = (float)a.cB;
  a.f_cC = (float)a.cC;
  for (int i = 0; i < 3; ++i) a.f_ks[i] = (float)a.ks[i];
  return a;
}
// a launch parameter in the kernel's precision: the FP32 copy or the FP64 value
template <typename T>
__device__ __forceinline__ T par(double d, float f) {
  if constexpr (sizeof(T) == 4) return f;
  else return d;
}
__device__ __forceinline__ bool kept(int k, int kmax3) { return 3 * (k < 0 ? -k : k) < kmax3; }
// The support of the stage's state (PassArgs::prune): rows_vanish, it vanishes on every
// row (kz, ky) outside the 2/3 box; box_vanish, at every mode outside the box.
__device__ __forceinline__ bool rows_vanish(const PassArgs& a) { return a.prune >= PRUNE_ROWS; }
__device__ __forceinline__ bool box_vanish(const PassArgs& a) { return a.prune == PRUNE_BOX; }

// XM_STAGE2N: the stage update of Williamson's 2N low-storage form (a mode of its
// own, so that the two-register stage update compiles without its branch)
enum XMode { XM_INV_CURL = 0, XM_STAGE = 1, XM_RHS = 2, XM_FWD_STORE = 3, XM_INV_PLAIN = 4, XM_INV_DIV = 5, XM_STAGE2N = 6 };
// ZM_PRODUCTS: c2r of u, the six products u_i u_j, their r2c stored for kz < PassArgs::kz_keep
enum ZMode { ZM_CROSS = 0, ZM_STORE = 1, ZM_LOAD = 2, ZM_MAXABS = 3, ZM_PRODUCTS = 4 };

// Writes conj(u/N^3) and conj(i k x u / N^3) of one mode into the 6 line
// buffers (stride LS) at padded position pos (conjugated because the following
// x transform is an inverse one).
template <bool SCALE, typename T>
__device__ __forceinline__ void put_curl_lines(cx<T>* s, int pos, int LS, cx<T> u0, cx<T> u1, cx<T> u2, T kx, T ky,
                                               T kz, T sc) {
  if constexpr (SCALE) {
    u0 = scal(u0, sc);
    u1 = scal(u1, sc);
    u2 = scal(u2, sc);
  }
  // omega_hat = i k x u_hat
  const cx<T> w0 = mul_pi(mk(ky * u2.x - kz * u1.x, ky * u2.y - kz * u1.y));
  const cx<T> w1 = mul_pi(mk(kz * u0.x - kx * u2.x, kz * u0.y - kx * u2.y));
  const cx<T> w2 = mul_pi(mk(kx * u1.x - ky * u0.x, kx * u1.y - ky * u0.y));
  cx<T>* p = s + pos;
  p[0 * LS] = conjg(u0);
  p[1 * LS] = conjg(u1);
  p[2 * LS] = conjg(u2);
  p[3 * LS] = conjg(w0);
  p[4 * LS] = conjg(w1);
  p[5 * LS] = conjg(w2);
}

// 1 / x for a positive normal x
__device__ __forceinline__ float recip(float x) { return 1.f / x; }
// in FP64 by Newton's iteration r <- r + r (1 - x r) from the hardware's approximation (20 bits): the second step starts
// from 2^-40, so that its one rounding gives the rounded quotient (equal to it for |k|^2 of all sizes in use). Four
// operations of the FP64 pipe; the division takes ten
__device__ __forceinline__ double recip(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// Global store of one complex value of the RK state.
template <typename T>
__device__ __forceinline__ void st_state(cx<T>* p, cx<T> v) {
  *p = v;
}

// Global store of a forward-transformed state row with the Nyquist modes zeroed.
template <typename T>
struct GStoreNyquistFree {
  cx<T>* g;
  int N;
  bool zero_row;
  __device__ __forceinline__ cx<T>* at(int p) const { return g + p; }
  static constexpr int off(int d) { return d; }
  __device__ __forceinline__ void store(cx<T>* q, int p, cx<T> v) const {
    *q = (zero_row || p == N / 2) ? mk((T)0, (T)0) : v;
  }
};

// R of the rows |ky| <= R kept by the 2/3 rule 3|ky| < k3y on a line of NY points (R < NY/2)
template <int NY>
__host__ __device__ constexpr int xpass_kept_ky(int k3y) {
  return (k3y - 1) / 3 < NY / 2 - 1 ? (k3y - 1) / 3 : NY / 2 - 1;
}
// x-stage launches of a pruned state cover only the rows inside the box (compact grid) up to
// rows of 512 points; the 1024-point rows keep the full grid with early returns (measured on
// GB300: 0.861 -> 0.848 ms per launch at 512^3 and a 3 % shorter ensemble step, but 8.46 ->
// 8.81 ms at 1024^3)
template <int N>
constexpr bool xpass_compact_ok() { return N <= 512; }

// ---------------------------------------------------------------------------
// x-pass: one block owns one row (kz, ky) of length N; warp f transforms line f.
// ---------------------------------------------------------------------------
// NY, NZ: points along y and z where they differ from N (rows kz * NY + ky).
// V: radix plan variant of the line transforms (SmemPlanV).
// compact: the grid covers only the rows inside the 2/3 box (xpass_rows_kept blocks, block bx
// taking row kz = bx / (2R + 1), |ky| <= R), the launch of a state that vanishes outside it.
template <typename T, int N, int MODE, int NY = N, int NZ = N, int V = 0>
__device__ __forceinline__ void xpass_body(const PassArgs a, const int bx, const bool compact = false) {
  constexpr int NT = XP_THREADS;  // one warp per line of u and omega
  constexpr bool STAGE = MODE == XM_STAGE || MODE == XM_STAGE2N;  // a stage update (either form)
  using G = Geometry<T, N, NY, NZ>;
  constexpr int LS = G::XLS;
  constexpr size_t FS = G::FS;
  constexpr int TW = G::TW;
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<T>* s = reinterpret_cast<cx<T>*>(smraw);
  const cx<T>* tw = reinterpret_cast<const cx<T>*>(a.tw);
  cx<T>* U = reinterpret_cast<cx<T>*>(a.U);
  cx<T>* U1 = reinterpret_cast<cx<T>*>(a.U1);
  cx<T>* US = reinterpret_cast<cx<T>*>(a.US);
  cx<T>* W = reinterpret_cast<cx<T>*>(a.W);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // rows outside the 2/3 box carry no nonlinear term (each direction's cut-off from its
  // own point count); where the state vanishes on them, the stage leaves them zero and
  // neither the update nor the x inverse has anything to do there
  const int k3y = NY == N ? a.kmax3 : a.kmax3y, k3z = NZ == N ? a.kmax3 : a.kmax3z;
  int row = bx;  // row = kz * NY + ky
  if (compact) {
    const int R = xpass_kept_ky<NY>(k3y), w = 2 * R + 1, t = bx % w;
    row = (bx / w) * NY + (t <= R ? t : NY - w + t);
  }
  const int kz = row / NY, ky = row % NY;
  const size_t rb = (size_t)row * N;
  const T sc = (T)(1.0 / ((double)N * (double)NY * (double)NZ));
  // the FP64 form's inverse transforms take a power of two in the conversion of their results
  constexpr int E2 = sizeof(T) == 8 && IsPow2<N>::value && IsPow2<NY>::value && IsPow2<NZ>::value
                         ? -(ilog2c(N) + ilog2c(NY) + ilog2c(NZ)) : 0;
  // wavenumbers of the row and of column j: integer index times 2 pi / L (1 on the 2 pi box)
  const T ksx = par<T>(a.ks[0], a.f_ks[0]);
  const T kzv = (T)kz * par<T>(a.ks[2], a.f_ks[2]), kyv = (T)kfreq(ky, NY) * par<T>(a.ks[1], a.f_ks[1]);
  const bool row_kept = (3 * kz < k3z) && kept(kfreq(ky, NY), k3y);
  if constexpr (STAGE || MODE == XM_INV_CURL || MODE == XM_INV_PLAIN) {
    if (!row_kept && rows_vanish(a)) return;
  }

  if constexpr (STAGE || MODE == XM_RHS) {
    // rows outside the box: skip their forward transform
    T nu = par<T>(a.nu, a.f_nu);
    const T cA = par<T>(a.cA, a.f_cA), cB = par<T>(a.cB, a.f_cB);
    const int stage = a.stage, last = a.last;
    // Williamson 2N stages keep the stage state in U (updated in place) and dU in U1
    constexpr bool lsrk = MODE == XM_STAGE2N;
    const cx<T>* Sst = (stage == 0 || lsrk) ? U : US;
    // state rows read by the update: stage state (all stages), accumulator
    // (stages after the first), step-start state (the stages between first and
    // last of the two-register form)
    const bool need1 = STAGE && stage > 0, need0 = STAGE && stage > 0 && stage < last && !lsrk;
    cx<T>* const st = s + G::XST;  // XPRE: rows [Sst 0..2][U1 0..2][U 0..2], N values each
    // a state that vanishes at every mode outside the box (box_vanish) keeps vanishing at
    // the columns |kx| >= N/3 of this row too: its rows are read and written at the kept
    // columns only, the others give u = omega = 0
    const bool xbox = STAGE && box_vanish(a);
    if constexpr (G::XBULK) {
      // rows of W where the lines lie (unpadded, from an even value on; a line's first pass takes it all before
      // it stores), rows of the state: whole, or the kept columns' two ranges
      __shared__ unsigned long long bars[2];
      const unsigned bw = smem_addr(bars), bs = bw + 8;
      if (threadIdx.x == 0) {
        mbar_init(bw);
        mbar_init(bs);
        mbar_init_done();
        if (row_kept) {
          mbar_expect(bw, 3 * N * 8);
#pragma unroll 1
          for (int f = 0; f < 3; ++f) bulk_load(s + (f * LS + 1) / 2 * 2, W + f * FS + rb, N * 8, bw);
        }
        const int R = (a.kmax3 + 2) / 3 - 1;  // the last kept column
        int lo = (R + 2) / 2 * 2, hi = (N - R) / 2 * 2;
        if (!xbox || lo >= hi) lo = hi = N;
        const int rows = 3 * (1 + need1 + need0);
        mbar_expect(bs, rows * (lo + N - hi) * 8);
#pragma unroll 1
        for (int f = 0; f < 3; ++f) {
          auto fetch_row = [&](const cx<T>* src, cx<T>* dst) {
            bulk_load(dst + f * N, src + f * FS + rb, lo * 8, bs);
            if (hi < N) bulk_load(dst + f * N + hi, src + f * FS + rb + hi, (N - hi) * 8, bs);
          };
          fetch_row(Sst, st);
          if (need1) fetch_row(U1, st + 3 * N);
          if (need0) fetch_row(U, st + 6 * N);
        }
      }
      __syncthreads();
      bool ok = true;
      if (row_kept && warp < 3) {
        ok = mbar_wait(bw, 0);
        const SLine<T, 1> line{s + warp * LS};
        line_fft<T, N, TW, V>(SRow<T>{s + (warp * LS + 1) / 2 * 2}, line, line, tw, lane);
      }
      ok = mbar_wait(bs, 0) && ok;
      // Copies that a warp does not see arrive within the limit: it waits once more, since they must not land after
      // the block has gone, and turns its columns and its line of N_hat to NaN, which the checks of the state
      // report. Before the barrier and warp by warp: agreed on by the block at the barrier, the launch took 700 us at
      // 512^3, so 696 (690 where nothing is waited for again).
      if (!__all_sync(0xffffffffu, ok)) {
        nu = (T)__int_as_float(0x7fffffff);
        if (row_kept) mbar_wait(bw, 0);
        mbar_wait(bs, 0);
        __syncwarp();
        if (row_kept && warp < 3)
          for (int p = lane; p < N; p += 32) s[warp * LS + padt<T>(p)] = mk(nu, nu);
      }
      __syncthreads();
    } else if constexpr (G::XPRE) {
      if (row_kept) {
        for (int e = threadIdx.x; e < 3 * N; e += NT) {
          const int f = e / N, j = e % N;
          cp_async<sizeof(cx<T>)>(s + f * LS + padt<T>(j), W + f * FS + rb + j);
        }
      }
      cp_async_commit();
      constexpr int PK = 16 / (int)sizeof(cx<T>);  // complex values per 16-byte copy
      auto fetch_rows = [&](const cx<T>* src, cx<T>* dst) {
        for (int e = threadIdx.x; e < 3 * N / PK; e += NT) {
          const int f = (e * PK) / N, j = (e * PK) % N;
          // the columns outside the box are one contiguous range: a copy none of whose
          // columns is kept has both ends outside
          if (xbox && !kept(kfreq(j, N), a.kmax3) && !kept(kfreq(j + PK - 1, N), a.kmax3)) continue;
          cp_async<16>(dst + f * N + j, src + f * FS + rb + j);
        }
      };
      fetch_rows(Sst, st);
      if (need1) fetch_rows(U1, st + 3 * N);
      if (need0) fetch_rows(U, st + 6 * N);
      cp_async_commit();
      cp_async_wait<1>();
      __syncthreads();
      if (row_kept && warp < 3) {
        const SLine<T, 1> line{s + warp * LS};
        line_fft<T, N, TW, V>(line, line, line, tw, lane);
      }
      cp_async_wait<0>();
    } else {
      if (row_kept && warp < 3) {
        const SLine<T, 1> line{s + warp * LS};
        line_fft<T, N, TW, V>(GLoad<T, false>{W + warp * FS + rb}, line, line, tw, lane);
      }
    }
    if constexpr (!G::XBULK) __syncthreads();
    // state values of component c at column j: staged rows or global memory
    auto ld_s = [&](int c, int j) -> cx<T> { return G::XPRE ? st[c * N + j] : Sst[c * FS + rb + j]; };
    auto ld_1 = [&](int c, int j) -> cx<T> { return G::XPRE ? st[(3 + c) * N + j] : U1[c * FS + rb + j]; };
    auto ld_0 = [&](int c, int j) -> cx<T> { return G::XPRE ? st[(6 + c) * N + j] : U[c * FS + rb + j]; };
    // the column loop, with the wavenumber kx = index * 2 pi / Lx; on the 2 pi box the
    // index itself, exactly as without a box option
    auto columns = [&](auto scaled) {
      constexpr bool SCALED = decltype(scaled)::value;
      for (int j = threadIdx.x; j < N; j += NT) {
        const int kxi = kfreq(j, N);
        const T kx = SCALED ? (T)kxi * ksx : (T)kxi;
        const int pj = padt<T>(j);
        const cx<T> zero = mk((T)0, (T)0);
        if (xbox && !kept(kxi, a.kmax3)) {  // the state stays zero there and is not written
#pragma unroll
          for (int f = 0; f < 3; ++f) {
            s[f * LS + pj] = zero;
            if constexpr (G::XPRE && !G::XWIDE) st[f * N + j] = zero;
            else s[(3 + f) * LS + pj] = zero;
          }
          continue;
        }
        cx<T> n0 = zero, n1 = n0, n2 = n0;
        if (row_kept && kept(kxi, a.kmax3)) {
          n0 = s[0 * LS + pj];
          n1 = s[1 * LS + pj];
          n2 = s[2 * LS + pj];
          if (a.F) {  // external force (learned closure), masked like the nonlinear term
            const cx<T>* F = reinterpret_cast<const cx<T>*>(a.F);
            n0 = n0 + F[rb + j];
            n1 = n1 + F[FS + rb + j];
            n2 = n2 + F[2 * FS + rb + j];
          }
        }
        const T k2 = kx * kx + kyv * kyv + kzv * kzv;
        const T ik2 = k2 > (T)0 ? recip(k2) : (T)0;
        // P = (k . N_hat) / |k|^2   (Eq. mod_pressure without the factor i)
        const cx<T> p = mk((kx * n0.x + kyv * n1.x + kzv * n2.x) * ik2, (kx * n0.y + kyv * n1.y + kzv * n2.y) * ik2);
        const size_t gi = rb + j;
        const cx<T> u0 = ld_s(0, j), u1 = ld_s(1, j), u2 = ld_s(2, j);
        const T nk2 = nu * k2;
        // dU = N_hat - k P - nu |k|^2 u_hat   (Eq. NSfinal)
        const cx<T> d0 = mk(n0.x - kx * p.x - nk2 * u0.x, n0.y - kx * p.y - nk2 * u0.y);
        const cx<T> d1 = mk(n1.x - kyv * p.x - nk2 * u1.x, n1.y - kyv * p.y - nk2 * u1.y);
        const cx<T> d2 = mk(n2.x - kzv * p.x - nk2 * u2.x, n2.y - kzv * p.y - nk2 * u2.y);
        if constexpr (MODE == XM_RHS) {
          cx<T>* out = reinterpret_cast<cx<T>*>(a.out);
          out[gi] = d0;
          out[FS + gi] = d1;
          out[2 * FS + gi] = d2;
        } else {
          cx<T> v0 = zero, v1 = zero, v2 = zero;
          if constexpr (lsrk) {  // 2N stage: dU <- A_s dU + dt RHS, u <- u + B_s dU
            const T cC = par<T>(a.cC, a.f_cC);
            cx<T> e0 = scal(d0, cC), e1 = scal(d1, cC), e2 = scal(d2, cC);
            if (stage > 0) {
              e0 = e0 + scal(ld_1(0, j), cA);
              e1 = e1 + scal(ld_1(1, j), cA);
              e2 = e2 + scal(ld_1(2, j), cA);
            }
            if (stage < last) {
              st_state(U1 + gi, e0);
              st_state(U1 + FS + gi, e1);
              st_state(U1 + 2 * FS + gi, e2);
            }
            v0 = u0 + scal(e0, cB);
            v1 = u1 + scal(e1, cB);
            v2 = u2 + scal(e2, cB);
            st_state(U + gi, v0);
            st_state(U + FS + gi, v1);
            st_state(U + 2 * FS + gi, v2);
          } else if (stage == 0 && last == 0) {  // one-stage step (forward Euler): u += a_0 dt dU
            v0 = u0 + scal(d0, cA);
            v1 = u1 + scal(d1, cA);
            v2 = u2 + scal(d2, cA);
            st_state(U + gi, v0);
            st_state(U + FS + gi, v1);
            st_state(U + 2 * FS + gi, v2);
          } else if (stage == 0) {
            st_state(U1 + gi, u0 + scal(d0, cA));
            st_state(U1 + FS + gi, u1 + scal(d1, cA));
            st_state(U1 + 2 * FS + gi, u2 + scal(d2, cA));
            v0 = u0 + scal(d0, cB);
            v1 = u1 + scal(d1, cB);
            v2 = u2 + scal(d2, cB);
            st_state(US + gi, v0);
            st_state(US + FS + gi, v1);
            st_state(US + 2 * FS + gi, v2);
          } else if (stage < last) {
            const cx<T> b0 = ld_0(0, j), b1 = ld_0(1, j), b2 = ld_0(2, j);
            st_state(U1 + gi, ld_1(0, j) + scal(d0, cA));
            st_state(U1 + FS + gi, ld_1(1, j) + scal(d1, cA));
            st_state(U1 + 2 * FS + gi, ld_1(2, j) + scal(d2, cA));
            v0 = b0 + scal(d0, cB);
            v1 = b1 + scal(d1, cB);
            v2 = b2 + scal(d2, cB);
            st_state(US + gi, v0);
            st_state(US + FS + gi, v1);
            st_state(US + 2 * FS + gi, v2);
          } else {
            v0 = ld_1(0, j) + scal(d0, cA);
            v1 = ld_1(1, j) + scal(d1, cA);
            v2 = ld_1(2, j) + scal(d2, cA);
            st_state(U + gi, v0);
            st_state(U + FS + gi, v1);
            st_state(U + 2 * FS + gi, v2);
          }
          if constexpr (G::XPRE && !G::XWIDE) {
            // u into lines 0-2 (padded, where this thread read N_hat), omega into
            // state rows 0-2 (unpadded, where this thread read the stage state)
            const cx<T> s0 = scal(v0, sc), s1 = scal(v1, sc), s2 = scal(v2, sc);
            s[0 * LS + pj] = conjg(s0);
            s[1 * LS + pj] = conjg(s1);
            s[2 * LS + pj] = conjg(s2);
            st[0 * N + j] = conjg(mul_pi(mk(kyv * s2.x - kzv * s1.x, kyv * s2.y - kzv * s1.y)));
            st[1 * N + j] = conjg(mul_pi(mk(kzv * s0.x - kx * s2.x, kzv * s0.y - kx * s2.y)));
            st[2 * N + j] = conjg(mul_pi(mk(kx * s1.x - kyv * s0.x, kx * s1.y - kyv * s0.y)));
          } else {
            put_curl_lines<E2 == 0>(s, pj, LS, v0, v1, v2, kx, kyv, kzv, sc);
          }
        }
      }
    };
    if (ksx == (T)1)
      columns(std::false_type{});
    else
      columns(std::true_type{});
    if constexpr (STAGE) {
      __syncthreads();
      if constexpr (G::XPRE && !G::XWIDE) {
        if (warp < 3) {
          const SLine<T, 1> line{s + warp * LS};
          line_fft<T, N, TW, V, E2>(line, line, GStore<T, true>{W + warp * FS + rb}, tw, lane);
        } else {  // omega: from its unpadded row, through a padded work line over rows 3-8
          const int c = warp - 3;
          const SLine<T, 1> work{st + 3 * N + c * LS};
          line_fft<T, N, TW, V, E2>(SRow<T>{st + c * N}, work, GStore<T, true>{W + warp * FS + rb}, tw, lane);
        }
      } else {
        const SLine<T, 1> line{s + warp * LS};
        line_fft<T, N, TW, V, E2>(line, line, GStore<T, true>{W + warp * FS + rb}, tw, lane);
      }
    }
  } else if constexpr (MODE == XM_FWD_STORE) {
    if (warp < 3) {
      const SLine<T, 1> line{s + warp * LS};
      line_fft<T, N, TW, V>(GLoad<T, false>{U + warp * FS + rb}, line,
                        GStoreNyquistFree<T>{U + warp * FS + rb, N, ky == NY / 2}, tw, lane);
    }
  } else {
    // inverse x transform of u and omega (XM_INV_CURL), of u alone
    // (XM_INV_PLAIN) or of i k . u (XM_INV_DIV), all scaled by 1/N^3
    constexpr int NF = (MODE == XM_INV_CURL) ? 6 : (MODE == XM_INV_PLAIN ? 3 : 1);
    const bool xbox = (MODE == XM_INV_CURL || MODE == XM_INV_PLAIN) && box_vanish(a);  // columns |kx| >= N/3 hold zeros
    for (int j = threadIdx.x; j < N; j += NT) {
      const size_t gi = rb + j;
      const int pj = padt<T>(j);
      const bool xin = !xbox || kept(kfreq(j, N), a.kmax3);
      const cx<T> zero = mk((T)0, (T)0);
      const cx<T> u0 = xin ? U[gi] : zero, u1 = xin ? U[FS + gi] : zero, u2 = xin ? U[2 * FS + gi] : zero;
      const T kx = (T)kfreq(j, N) * ksx;
      if constexpr (MODE == XM_INV_CURL) {
        put_curl_lines<E2 == 0>(s, pj, LS, u0, u1, u2, kx, kyv, kzv, sc);
      } else if constexpr (MODE == XM_INV_PLAIN) {
        s[0 * LS + pj] = conjg(E2 ? u0 : scal(u0, sc));
        s[1 * LS + pj] = conjg(E2 ? u1 : scal(u1, sc));
        s[2 * LS + pj] = conjg(E2 ? u2 : scal(u2, sc));
      } else {
        const cx<T> d = mul_pi(mk(kx * u0.x + kyv * u1.x + kzv * u2.x, kx * u0.y + kyv * u1.y + kzv * u2.y));
        s[pj] = conjg(E2 ? d : scal(d, sc));
      }
    }
    __syncthreads();
    cx<T>* dst = (MODE == XM_INV_DIV) ? reinterpret_cast<cx<T>*>(a.D) : W;
    if (warp < NF) {
      const SLine<T, 1> line{s + warp * LS};
      line_fft<T, N, TW, V, E2>(line, line, GStore<T, true>{dst + warp * FS + rb}, tw, lane);
    }
  }
}

template <typename T, int N, int MODE, int NY = N, int NZ = N, int V = 0>
__global__ void __launch_bounds__(XP_THREADS, (Geometry<T, N, NY, NZ>::XMIN)) k_xpass(PassArgs a) {
  constexpr bool CAN = ((MODE == XM_STAGE || MODE == XM_STAGE2N || MODE == XM_INV_CURL || MODE == XM_INV_PLAIN) && xpass_compact_ok<N>()) ||
                       MODE == XM_FWD_STORE;
  xpass_body<T, N, MODE, NY, NZ, V>(a, blockIdx.x, CAN && a.prune >= PRUNE_ROWS);
}

// Batched form (ensembles): member blockIdx.y, its arguments in B.a[blockIdx.y].
template <typename T, int N, int MODE, int V = 0>
__global__ void __launch_bounds__(XP_THREADS, (Geometry<T, N>::XMIN)) k_xpass_b(const __grid_constant__ BatchArgs B) {
  xpass_body<T, N, MODE, N, N, V>(B.a[blockIdx.y], blockIdx.x);
}

// ---------------------------------------------------------------------------
// y-pass: one block owns TX adjacent columns (fixed field and kz) of length N;
// the tile is loaded with coalesced rows, each warp transforms whole columns.
// INV: conj-in/conj-out (inverse DFT). PRUNE: store only rows with |ky| < N/3.
// grid = (N / TX, number of kz planes, number of fields); TX etc. from YCfg
// ---------------------------------------------------------------------------
// Row walked by tile element group r of the y-pass. With 8-byte values in
// 8-wide rows (row stride 9 in shared memory) a warp covers 4 rows; rows y and
// y + 1 in one half-warp share banks, rows y and y + 8 do not, so the walk takes
// rows in the order 0, 8, 1, 9, 2, 10, ... within each block of 16 (a
// permutation of 0 .. N-1 only when N is a multiple of 16; otherwise the rows
// are walked in order).
template <typename T, int TX, int N>
__device__ __forceinline__ int ywalk_row(int r) {
  if constexpr (sizeof(cx<T>) == 8 && TX == 8 && N % 16 == 0) {
    const int t = r & 15, u = t >> 2, q = t & 3;
    return (r & ~15) | (2 * u + (q >> 1) + (q & 1) * 8);
  } else {
    return r;
  }
}

// Fill of a y tile (TX columns of L rows, row stride `stride` in global memory) whose rows
// outside the 2/3 box are zeros: the kept rows |ky| <= R (R = (kmax3 - 1) / 3, rows 0 .. R
// and L - R .. L - 1) by cp.async (in the bank-friendly walk order where it permutes the
// rows), the rows R + 1 .. L - R - 1 between them as zeros.
template <typename T, int L, int TX, int LD, int NT>
__device__ __noinline__ void ytile_fill_kept(cx<T>* s, const cx<T>* __restrict__ base, int stride, int kmax3) {
  int R = (kmax3 - 1) / 3;
  if (R > L / 2 - 1) R = L / 2 - 1;
  const int lo = R + 1, gap = L - 2 * R - 1;  // kept rows [0, lo) and [lo + gap, L)
  if constexpr (sizeof(cx<T>) == 8 && TX == 8 && L % 16 == 0) {
#pragma unroll 8
    for (int e = threadIdx.x; e < TX * L; e += NT) {
      const int x = e % TX, y = ywalk_row<T, TX, L>(e / TX);
      if (y < lo || y >= lo + gap) cp_async<sizeof(cx<T>)>(s + padt<T>(y) * LD + x, base + (size_t)y * stride + x);
    }
  } else {
#pragma unroll 8
    for (int e = threadIdx.x; e < TX * (L - gap); e += NT) {
      const int x = e % TX, r = e / TX, y = r < lo ? r : r + gap;
      cp_async<sizeof(cx<T>)>(s + padt<T>(y) * LD + x, base + (size_t)y * stride + x);
    }
  }
#pragma unroll 4
  for (int e = threadIdx.x; e < TX * gap; e += NT) {
    const int x = e % TX, y = lo + e / TX;
    s[padt<T>(y) * LD + x] = mk((T)0, (T)0);
  }
}

// The y tile of FP32 lines of up to 128 points (INV, PRUNE, vanish as in ypass_tile; L points, row stride N). A line has
// fewer radix-8 butterflies than a warp has lanes, so a warp takes several columns at once (a quarter of the tile at
// most), in the layout of the z-pass tiles (ZLay), filled and drained 16 bytes at a time. Against one column per warp
// (8 to 12 lanes of 32 busy in the first pass at 64 and 96 points): a step of 128 runs of 32^3 .. 96^3 7.14 -> 6.02 ms
// with the default tiles, the y-passes of 128^3 20.3 + 14.8 -> 18.0 + 13.1 us (29.0 + 13.9 -> 25.8 + 13.3 with every row).
template <int N, int L, int TWN, int INV, int PRUNE, int TX, int NT, int V>
__device__ __forceinline__ void yshort_tile(cx<float>* __restrict__ base, const cx<float>* __restrict__ tw, int kmax3,
                                            bool vanish) {
  constexpr int LD = ZLay<L>::ld(TX), PAD = ZLay<L>::PAD;
  constexpr int G = cmin(LinesPerWarp<L, V>::value, TX >= 4 ? TX / 4 : 1);
  constexpr int VX = LD % 2 == 0 && TX % 2 == 0 ? 2 : 1;  // values of a copy
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<float>* s = reinterpret_cast<cx<float>*>(smraw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // rows inside the box: [0, lo) and [lo + gap, L)
  const int R = min((kmax3 - 1) / 3, L / 2 - 1), lo = R + 1, gap = 3 * (L / 2) < kmax3 ? 0 : L - 2 * R - 1;
  const int skip = INV && vanish ? gap : 0;
#pragma unroll 4
  for (int e = threadIdx.x; e < TX / VX * (L - skip); e += NT) {
    const int x = e % (TX / VX) * VX, r = e / (TX / VX), y = r < lo ? r : r + skip;
    cp_async<VX * 8>(s + padrow<PAD>(y) * LD + x, base + (size_t)y * N + x);
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
#pragma unroll 1
  for (int c = warp * G; c < TX; c += NT / 32 * G)
    warp_fft_lines<float, L, TWN, G, LD, PAD, V, INV ? LINES_CONJ : LINES_PLAIN>(s + c, tw, lane, lo, lo + skip);
  __syncthreads();
  const int drop = PRUNE ? gap : 0;
#pragma unroll 4
  for (int e = threadIdx.x; e < TX / VX * (L - drop); e += NT) {
    const int x = e % (TX / VX) * VX, r = e / (TX / VX), y = r < lo ? r : r + drop;
    const cx<float>* q = s + padrow<PAD>(y) * LD + x;
    cx<float>* o = base + (size_t)y * N + x;
    if constexpr (VX == 2) {
      float4 v = *reinterpret_cast<const float4*>(q);
      if (INV) v = make_float4(v.x, -v.y, v.z, -v.w);
      *reinterpret_cast<float4*>(o) = v;
    } else {
      *o = INV ? conjg(*q) : *q;
    }
  }
}

// One y tile: TX adjacent columns starting at `base` (field, kz plane and first
// column already applied), transformed along y in place. NT: threads of the block.
// vanish (inverse only): the rows with |ky| >= N/3 are zeros, not read.
template <typename T, int N, int INV, int PRUNE, int TXO, int NT, int V = 0>
__device__ __forceinline__ void ypass_tile(cx<T>* __restrict__ base, const cx<T>* __restrict__ tw, int kmax3,
                                           bool vanish = false) {
  using Y = YCfg<T, N, INV, TXO>;
  constexpr int TX = Y::TX;
  constexpr int LD = Y::LD;
  if constexpr (Y::SHORT) {
    yshort_tile<N, N, N, INV, PRUNE, TX, NT, V>(base, tw, kmax3, vanish);
    return;
  }
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<T>* s = reinterpret_cast<cx<T>*>(smraw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the whole tile in flight at once (cp.async, no register staging); the
  // inverse's conjugation is applied when the first pass reads it
  if (INV && vanish) {
    ytile_fill_kept<T, N, TX, LD, NT>(s, base, N, kmax3);
  } else {
#pragma unroll 8
    for (int e = threadIdx.x; e < TX * N; e += NT) {
      const int x = e % TX, y = ywalk_row<T, TX, N>(e / TX);
      cp_async<sizeof(cx<T>)>(s + padt<T>(y) * LD + x, base + (size_t)y * N + x);
    }
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
#pragma unroll 1
  for (int c = warp; c < TX; c += NT / 32) {  // warps loop over the columns
    const SLine<T, LD> line{s + c};
    if constexpr (INV) line_fft<T, N, N, V>(SLineConj<T, LD>{s + c}, line, line, tw, lane);
    else line_fft<T, N, N, V>(line, line, line, tw, lane);
  }
  __syncthreads();
#pragma unroll 8
  for (int e = threadIdx.x; e < TX * N; e += NT) {
    const int x = e % TX, y = ywalk_row<T, TX, N>(e / TX);
    if (PRUNE && !kept(kfreq(y, N), kmax3)) continue;
    const cx<T> v = s[padt<T>(y) * LD + x];
    base[(size_t)y * N + x] = INV ? conjg(v) : v;
  }
}

// NY, NZ: points along y and z where they differ from N (N: the x extent, the
// row stride of the tile's columns).
// PR (inverse of a stage whose state vanishes outside the 2/3 box): the grid covers the
// planes kz < kc only (the others hold zeros that the z-pass does not read) and the rows
// with |ky| >= NY/3 (kmax3) are read as zeros.
template <typename T, int N, int INV, int PRUNE, int TXO = 0, int NY = N, int NZ = N, int V = 0, int PR = 0>
__global__ void __launch_bounds__(YCfg<T, N, INV, TXO, NY>::THREADS, (YCfg<T, N, INV, TXO, NY>::MINB))
    k_ypass(cx<T>* __restrict__ F, const cx<T>* __restrict__ tw, int kmax3) {
  using G = Geometry<T, N, NY, NZ>;
  using Y = YCfg<T, N, INV, TXO, NY>;
  constexpr int TX = Y::TX;
  constexpr int LD = Y::LD;
  constexpr int NT = Y::THREADS;  // warps loop over the columns
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<T>* s = reinterpret_cast<cx<T>*>(smraw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  cx<T>* base = F + blockIdx.z * G::FS + (size_t)blockIdx.y * NY * N + blockIdx.x * TX;
  if constexpr (Y::SHORT) {
    yshort_tile<N, NY, G::TW, INV, PRUNE, TX, NT, V>(base, tw, kmax3, INV && PR);
    return;
  }
  // the whole tile in flight at once (cp.async, no register staging); the
  // inverse's conjugation is applied when the first pass reads it
  if constexpr (INV && PR) {
    ytile_fill_kept<T, NY, TX, LD, NT>(s, base, N, kmax3);
  } else {
#pragma unroll 8
    for (int e = threadIdx.x; e < TX * NY; e += NT) {
      const int x = e % TX, y = ywalk_row<T, TX, NY>(e / TX);
      cp_async<sizeof(cx<T>)>(s + padt<T>(y) * LD + x, base + (size_t)y * N + x);
    }
  }
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
#pragma unroll 1
  for (int c = warp; c < TX; c += NT / 32) {
    const SLine<T, LD> line{s + c};
    if constexpr (INV) line_fft<T, NY, G::TW, V>(SLineConj<T, LD>{s + c}, line, line, tw, lane);
    else line_fft<T, NY, G::TW, V>(line, line, line, tw, lane);
  }
  __syncthreads();
#pragma unroll 8
  for (int e = threadIdx.x; e < TX * NY; e += NT) {
    const int x = e % TX, y = ywalk_row<T, TX, NY>(e / TX);
    if (PRUNE && !kept(kfreq(y, NY), kmax3)) continue;
    const cx<T> v = s[padt<T>(y) * LD + x];
    base[(size_t)y * N + x] = INV ? conjg(v) : v;
  }
}

// ---------------------------------------------------------------------------
// y-pass of the FP32 lines of 256, 512 and 1024 points, with the lines in registers: a column belongs to
// T threads of E values each (NY = E T), a block to TX adjacent columns, the columns side by side in
// a warp. Thread l loads y = l + T m (rows of 8 TX bytes, all E loads in flight), does an E-point
// DFT, multiplies by exp(-2 pi i l j / NY), and after one exchange through shared memory does the
// T-point DFTs of the outputs j = l + T b: X[l + T (b + E / T k)] is again its own set of rows, stored
// directly. Against k_ypass (tile filled and drained through shared memory, three exchanges
// per line) a value crosses shared memory once instead of four times. A stage of the zero-row passes, inverse
// and forward: 512^3 0.733 + 0.388 -> 0.624 + 0.292 ms (5.7 and 6.1 TB/s of the bytes they move, bound by
// HBM), 1024^3 7.04 + 3.44 -> 5.22 + 2.74 ms, 256^3 105 + 56 -> 84 + 39 us.
// The kept rows |y| < lo (others hold zeros and are neither read nor stored) come with the launch.
// ---------------------------------------------------------------------------
template <int NY>
struct YReg {
  static constexpr int E = NY == 256 ? 16 : 32, T = NY / E;
  static constexpr int TX = NY == 1024 ? 8 : 16;  // rows of 64 or 128 bytes
  static constexpr int THREADS = TX * T;          // 256
  static constexpr int BLOCKS = NY == 256 ? 3 : 2;
  // row j of the exchange: T x TX values; 64-byte rows are padded by half a line, so that the two l of a
  // half-warp read different banks
  static constexpr int ROW = T * TX + (TX == 8 ? 8 : 0);
  static constexpr int SMEM = E * ROW * 8;
};

// INV: inverse transform (conjugated in and out). rd, wr: rows |ky| < rd are read, |ky| < wr stored.
template <int N, int NY, int TW, int INV>
__global__ void __launch_bounds__(YReg<NY>::THREADS, YReg<NY>::BLOCKS)
    k_yreg(cx<float>* __restrict__ F, const cx<float>* __restrict__ tw, size_t FS, int rd, int wr) {
  using Y = YReg<NY>;
  constexpr int E = Y::E, T = Y::T, TX = Y::TX, B = E / T;
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<float>* s = reinterpret_cast<cx<float>*>(smraw);
  const int c = threadIdx.x % TX, l = threadIdx.x / TX;
  cx<float>* base = F + blockIdx.z * FS + (size_t)blockIdx.y * NY * N + blockIdx.x * TX + c;
  cx<float> v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    const int y = l + T * m;
    v[m] = mk(0.f, 0.f);
    if (y < rd || y > NY - rd) v[m] = base[(size_t)y * N];
  }
  if constexpr (INV) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = conjg(v[m]);
  }
  dft<E>(v);
  s[l * TX + c] = v[0];
#pragma unroll
  for (int j = 1; j < E; ++j) s[j * Y::ROW + l * TX + c] = cmul(v[j], ldro(tw + l * j * (TW / NY)));
  __syncthreads();
#pragma unroll
  for (int b = 0; b < B; ++b) {
    cx<float> w[T];
#pragma unroll
    for (int q = 0; q < T; ++q) w[q] = s[(l + T * b) * Y::ROW + q * TX + c];
    dft<T>(w);
#pragma unroll
    for (int k = 0; k < T; ++k) {
      const int y = l + T * b + E * k;
      if (y < wr || y > NY - wr) base[(size_t)y * N] = INV ? conjg(w[k]) : w[k];
    }
  }
}

// Batched form on the members' work arrays (ensembles): blockIdx.z = member *
// fields + field; otherwise the same steps as k_ypass (TXO: a tuned tile width).
template <typename T, int N, int INV, int PRUNE, int TXO = 0, int V = 0>
__global__ void __launch_bounds__(YCfg<T, N, INV, TXO>::THREADS, (YCfg<T, N, INV, TXO>::MINB))
    k_ypass_b(const __grid_constant__ BatchArgs B, int fields) {
  using G = Geometry<T, N>;
  using Y = YCfg<T, N, INV, TXO>;
  const PassArgs& a = B.a[blockIdx.z / fields];
  const bool vanish = INV && rows_vanish(a);  // the member's planes kz >= kc are not transformed
  if (vanish && 3 * (int)blockIdx.y >= a.kmax3) return;
  cx<T>* base = reinterpret_cast<cx<T>*>(a.W) + (blockIdx.z % fields) * G::FS + (size_t)blockIdx.y * N * N +
                blockIdx.x * Y::TX;
  ypass_tile<T, N, INV, PRUNE, TXO, Y::THREADS, V>(base, reinterpret_cast<const cx<T>*>(a.tw), a.kmax3, vanish);
}

// max of a z-pass block's values into *bits (non-negative doubles order like their bit patterns)
template <int NT>
__device__ __forceinline__ void zpass_block_max(double m, unsigned long long* bits) {
  __shared__ double red[NT / 32];
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NT / 32; ++w) m = fmax(m, red[w]);
    atomicMax(bits, (unsigned long long)__double_as_longlong(m));
  }
}

// ---------------------------------------------------------------------------
// z-pass of the FP64 form, on fixed point (fixed_point.cuh) from the tile's doubles to the
// results. Every line has its own scale.
//   c2r   z'/4 from the pair (X_k, X_{M-k}) (L1 of z' is at most four times that of X): physical
//         values x = v 2^(K - 1083), |v| <= 2^62
//   u x w a line's values are shifted so that the largest has 61 bits (the L1 of a broad spectrum is many
//         times the values): x = a 2^(E - 1083). The products a b, cut at 2^-62, have the scale E_u + E_w; of
//         the two in a component of u x w the smaller scale's u is shifted down to the larger one e, so
//         that they can be subtracted: p = P 2^(e - 2104), |P| <= 2^61. With one scale for the three components
//         (and for omega's) a weak third component lost its bits: 1e-6 beside 1 kept 1e-11, 1e-20 nothing, and
//         with the L1 scale a white field of 512 points 2.6e-15 (FP64 products 1.0e-15); now 5e-16 and 9.3e-16, for
//         4 to 6 % of the pass (256^3 818 -> 855 us, 512^3 7.85 -> 8.30 ms).
//         Then the line of products is shifted by its L1, so that its DFT has 62 bits again
//   r2c   V = X_k / 2 (quartered post-processing of the pair): X_k = V 2^(e + 1 - sh - 2104)
// ---------------------------------------------------------------------------
template <int N, int MODE, int TXO, int NY, int NZ, int V>
__device__ __forceinline__ void zpass64_body(const PassArgs& a, const int bx, const int by) {
  using G = Geometry<double, N, NY, NZ>;
  typedef cx<double> cd;
  constexpr int M = G::M;
  constexpr int TW = G::TW, TS = TW / NZ;
  constexpr int TX = TXO > 0 ? TXO : G::ZTX;
  constexpr int LD = odd_ld(6 * TX);
  constexpr size_t FS = G::FS;
  constexpr int NF = MODE == ZM_CROSS ? 6 : (MODE == ZM_MAXABS ? 1 : 3), NL = NF * TX;
  constexpr int GL = cmin(FxLinesPerWarp<M, V>::value, TX);  // lines per warp
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int sK[NL];        // scale of a line as the tile holds it
  __shared__ int sL[NL];        // power of two that it was multiplied by (0 or FX_LIFT; any for a line of zeros)
  __shared__ unsigned sN[NL];   // its NaN word
  constexpr int NP = MODE == ZM_PRODUCTS ? 6 : 3;  // lines of products of a column
  __shared__ unsigned sQ[NP * TX];  // L1 of a line of products
  __shared__ unsigned sM[NL];       // top bit of a line's physical values
  __shared__ int sE[NP * TX];       // scale of a line of products; then what fx_to takes for it
  __shared__ int sT[NP * 2 * TX];   // shifts of the two u (ZM_CROSS) of a line of products
  cd* s = reinterpret_cast<cd*>(smraw);
  fx* sf = reinterpret_cast<fx*>(smraw);
  const cd* tw = reinterpret_cast<const cd*>(a.tw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int x0 = bx * TX, y = by;

  int klim = M;  // planes kz >= klim hold zeros (a state that vanishes outside the 2/3 box): not read
  if constexpr (MODE == ZM_LOAD) {
    const cd* in = reinterpret_cast<const cd*>(a.in);
    for (int e = threadIdx.x; e < 3 * TX * M; e += ZP_THREADS<double>) {
      const int n = e % M, x = (e / M) % TX, c = e / (M * TX);
      cp_async<16>(s + padt<double>(n) * LD + c * TX + x, in + ((size_t)(c * N + x0 + x) * NY + y) * M + n);
    }
  } else {
    const cd* src = reinterpret_cast<const cd*>(MODE == ZM_MAXABS ? a.D : a.W);
    if constexpr (MODE == ZM_CROSS || MODE == ZM_STORE || MODE == ZM_PRODUCTS) {
      if (rows_vanish(a)) klim = cmin(((NZ == N ? a.kmax3 : a.kmax3z) + 2) / 3, M);
    }
    for (int e = threadIdx.x; e < NL * M; e += ZP_THREADS<double>) {
      const int x = e % TX, k = (e / TX) % M, f = e / (TX * M);
      if (k < klim) cp_async<16>(s + padt<double>(k) * LD + f * TX + x, src + f * FS + ((size_t)k * NY + y) * N + x0 + x);
    }
  }
  constexpr bool PROD = MODE == ZM_CROSS || MODE == ZM_PRODUCTS;
  if (PROD && threadIdx.x < NP * TX) sQ[threadIdx.x] = 0;
  if (PROD && threadIdx.x < NL) sM[threadIdx.x] = 0;
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  // scales: SUB adjacent lanes walk a line
  constexpr int SUB = M >= 64 ? 8 : (M >= 16 ? 4 : 2);
  for (int l0 = warp * (32 / SUB); l0 < NL; l0 += (ZP_THREADS<double> / 32) * (32 / SUB)) {
    const int l = l0 + lane / SUB, q = lane % SUB;
    cd* ln = s + (l < NL ? l : NL - 1);
    unsigned m = 0;
    for (int k = q; k < klim; k += SUB) m = max(m, fx_mag(ln[padt<double>(k) * LD]));
#pragma unroll
    for (int o = SUB / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    int lift = 0;
    if (__any_sync(0xffffffffu, fx_tiny(m))) {
      unsigned any = m;
      if (m == 0) {
        for (int k = q; k < klim; k += SUB) {
          const cd v = ln[padt<double>(k) * LD];
          any |= (unsigned)__double2loint(v.x) | (unsigned)__double2loint(v.y);
        }
      }
#pragma unroll
      for (int o = SUB / 2; o > 0; o >>= 1) any |= __shfl_xor_sync(0xffffffffu, any, o);
      if (fx_tiny(m) && any) {
        lift = FX_LIFT;
        m = fx_lifted(m);
        if (l < NL)
          for (int k = q; k < klim; k += SUB) ln[padt<double>(k) * LD] = scal(ln[padt<double>(k) * LD], fx_pow2(FX_LIFT));
      }
    }
    const int top = fx_top(m);
    float t = 0.f;
    for (int k = q; k < klim; k += SUB) {
      const cd v = ln[padt<double>(k) * LD];
      t += fx_rel(v.x, top) + fx_rel(v.y, top);
    }
    unsigned sh = fx_share(t);
#pragma unroll
    for (int o = SUB / 2; o > 0; o >>= 1) sh += __shfl_xor_sync(0xffffffffu, sh, o);
    if (q == 0 && l < NL) {
      const FxScale sc = fx_scale(m, sh);
      sK[l] = sc.K;
      // a zero line's scale lies below all others: its product must not push the bits of the other one out
      sL[l] = PROD && m == 0 ? 5000 : lift;
      sN[l] = sc.nan;
    }
  }
  __syncthreads();
  if constexpr (MODE != ZM_LOAD) {
    // c2r pre-processing (zpass_body), quartered
    for (int e = threadIdx.x; e < NL * (M / 2 + 1); e += ZP_THREADS<double>) {
      const int l = e % NL, k = e / NL;
      const int K = sK[l];
      if (k == 0) {
        const ll r0 = (fx_from(s[l].x, K) + 2) >> 2;  // Im X_0 ignored, X_M = 0
        sf[l] = mk(r0, -r0);
      } else {
        const int pk = padt<double>(k) * LD + l, pm = padt<double>(M - k) * LD + l;
        const fx xk = fx_from(s[pk], K);
        const fx xm = M - k < klim ? fx_from(s[pm], K) : mk(0ll, 0ll);
        int4 w = ldfx(tw + k * TS);
        w.z = -w.z;
        w.w = -w.w;
        const fx A = fx_quarter(xk + conjg(xm)), P = mul_pi(fx_cmul<true>(xk - conjg(xm), w));
        sf[pk] = conjg(A + P);
        if (k != M - k) sf[pm] = A - P;
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int l = warp * GL; l < NL; l += (ZP_THREADS<double> / 32) * GL)
      warp_fft_fx_lines<M, TW, GL, LD, 0, V, FX_IN, PROD>(s + l, tw, lane, nullptr, sM + l);
    __syncthreads();
    // now conj(s) = x_{2n} + i x_{2n+1} (physical values, unnormalised c2r)
  }

  if constexpr (PROD) {
    // the shift that leaves 61 bits of line l, and its scale after it
    auto up = [&](int l) { return __clz(sM[l]) - 3; };
    auto scale = [&](int l) { return sK[l] - sL[l] - up(l); };
    if (threadIdx.x < NP * TX) {
      const int c = threadIdx.x / TX, x = threadIdx.x % TX;
      if constexpr (MODE == ZM_CROSS) {
        const int i = (c + 1) % 3 * TX + x, j = (c + 2) % 3 * TX + x;  // u_i w_j - u_j w_i
        const int e1 = scale(i) + scale(3 * TX + j), e2 = scale(j) + scale(3 * TX + i), e = max(e1, e2);
        sE[threadIdx.x] = e;
        sT[2 * threadIdx.x] = max(up(i) - (e - e1), -63);
        sT[2 * threadIdx.x + 1] = max(up(j) - (e - e2), -63);
      } else {
        const int i = c < 3 ? c : (c == 5 ? 1 : 0), j = c < 3 ? c : (c == 3 ? 1 : 2);
        sE[threadIdx.x] = scale(i * TX + x) + scale(j * TX + x);
      }
    }
    __syncthreads();
    auto mag = [](fx p) { return ((unsigned)abs((int)(p.x >> 32)) >> 9) + ((unsigned)abs((int)(p.y >> 32)) >> 9) + 2u; };
    // a warp takes 32 / XW adjacent positions of XW columns: whole warps on one column where the line
    // is long enough (no bank conflicts along a line)
    constexpr int XW = M >= 32 ? 1 : TX, CH = 32 / XW, CHUNKS = (M + CH - 1) / CH;
    static_assert(32 % XW == 0, "a lane keeps its column");
    for (int it = warp; it < (TX / XW) * CHUNKS; it += ZP_THREADS<double> / 32) {
      const int x = (it % (TX / XW)) * XW + lane % XW, n = (it / (TX / XW)) * CH + lane / XW;
      unsigned q[NP] = {};
      if (M % CH == 0 || n < M) {
        fx* p = sf + padt<double>(n) * LD + x;
        fx r[NP];
        // u and omega are conjugated: in their products the signs of the odd points cancel
        if constexpr (MODE == ZM_CROSS) {
          const fx u0 = p[0 * TX], u1 = p[1 * TX], u2 = p[2 * TX];
          const fx w0 = fx_shift(p[3 * TX], up(3 * TX + x)), w1 = fx_shift(p[4 * TX], up(4 * TX + x)),
                   w2 = fx_shift(p[5 * TX], up(5 * TX + x));
          // u x omega on both packed points (real and imaginary parts)
          auto cross = [&](int c, fx a, fx wb, fx b, fx wa) {
            const int* t = sT + 2 * (c * TX + x);
            a = fx_shift(a, t[0]);
            b = fx_shift(b, t[1]);
            return mk(fx_cross(a.x, wb.x, b.x, wa.x), fx_cross(a.y, wb.y, b.y, wa.y));
          };
          r[0] = cross(0, u1, w2, u2, w1);
          r[1] = cross(1, u2, w0, u0, w2);
          r[2] = cross(2, u0, w1, u1, w0);
        } else {
          const fx u0 = fx_shift(p[0 * TX], up(x)), u1 = fx_shift(p[1 * TX], up(TX + x)),
                   u2 = fx_shift(p[2 * TX], up(2 * TX + x));
          r[0] = mk(fx_prod(u0.x, u0.x), fx_prod(u0.y, u0.y));
          r[1] = mk(fx_prod(u1.x, u1.x), fx_prod(u1.y, u1.y));
          r[2] = mk(fx_prod(u2.x, u2.x), fx_prod(u2.y, u2.y));
          r[3] = mk(fx_prod(u0.x, u1.x), fx_prod(u0.y, u1.y));
          r[4] = mk(fx_prod(u0.x, u2.x), fx_prod(u0.y, u2.y));
          r[5] = mk(fx_prod(u1.x, u2.x), fx_prod(u1.y, u2.y));
        }
#pragma unroll
        for (int c = 0; c < NP; ++c) {
          q[c] = mag(r[c]);
          p[c * TX] = r[c];
        }
      }
      // L1 of the lines of products in units of 2^41
#pragma unroll
      for (int c = 0; c < NP; ++c) {
        if constexpr (XW == 1) {
          q[c] = __reduce_add_sync(0xffffffffu, q[c]);
        } else {
#pragma unroll
          for (int o = XW; o < 32; o *= 2) q[c] += __shfl_xor_sync(0xffffffffu, q[c], o);
        }
        if (lane < XW) atomicAdd(sQ + c * TX + x, q[c]);
      }
    }
    __syncthreads();
    if (threadIdx.x < NP * TX) sE[threadIdx.x] -= fx_shift_of(sQ[threadIdx.x]) + 1018;  // read after the transforms
  }

  if constexpr (PROD || MODE == ZM_LOAD) {
#pragma unroll 1
    for (int l = warp * GL; l < NP * TX; l += (ZP_THREADS<double> / 32) * GL) {
      if constexpr (PROD)
        warp_fft_fx_lines<M, TW, GL, LD, 0, V, FX_SHIFT>(s + l, tw, lane, reinterpret_cast<const int*>(sQ) + l);
      else
        warp_fft_fx_lines<M, TW, GL, LD, 0, V, FX_DOUBLE>(s + l, tw, lane, sK + l);
    }
    __syncthreads();
    // r2c post-processing (zpass_body)
    cd* dst = reinterpret_cast<cd*>(MODE == ZM_LOAD ? a.U : a.W);
    int kc = M;
    if (MODE == ZM_PRODUCTS) kc = a.kz_keep;
    if (MODE == ZM_CROSS) kc = cmin(((NZ == N ? a.kmax3 : a.kmax3z) + 2) / 3, M);
    for (int e = threadIdx.x; e < NP * TX * kc; e += ZP_THREADS<double>) {
      const int l = e % (NP * TX), k = e / (NP * TX), x = l % TX;
      const fx zk = sf[padt<double>(k) * LD + l], zm = sf[padt<double>((M - k) % M) * LD + l];
      const fx A = fx_quarter(zk + conjg(zm)), X = A + mul_mi(fx_cmul<true>(zk - conjg(zm), ldfx(tw + k * TS)));
      int B;
      unsigned nan;
      if constexpr (PROD) {
        B = sE[l];
        nan = 0;
#pragma unroll
        for (int f = 0; f < NF; ++f) nan |= sN[f * TX + x];
      } else {
        B = sK[l] - sL[l] + 1;
        nan = sN[l];
      }
      dst[(l / TX) * FS + ((size_t)k * NY + y) * N + x0 + x] = fx_to(X, B, nan);
    }
  } else if constexpr (MODE == ZM_STORE) {
    cd* out = reinterpret_cast<cd*>(a.out);
    for (int e = threadIdx.x; e < 3 * TX * M; e += ZP_THREADS<double>) {
      const int n = e % M, x = (e / M) % TX, c = e / (M * TX), l = c * TX + x;
      out[((size_t)(c * N + x0 + x) * NY + y) * M + n] =
          fx_to(conjg(sf[padt<double>(n) * LD + l]), sK[l] - sL[l] + 2, sN[l]);
    }
  } else if constexpr (MODE == ZM_MAXABS) {
    double m = 0.0;
    for (int e = threadIdx.x; e < TX * M; e += ZP_THREADS<double>) {
      const int l = e % TX;
      const cd v = fx_to(sf[padt<double>(e / TX) * LD + l], sK[l] - sL[l] + 2, sN[l]);
      m = fmax(m, fmax(fabs(v.x), fabs(v.y)));
    }
    zpass_block_max<ZP_THREADS<double>>(m, a.maxbits);
  }
}

// ---------------------------------------------------------------------------
// z-pass: one block owns ZTX adjacent x at fixed y; lines run along kz / z.
// Real transforms of length N use one complex DFT of length M = N/2 on
// z_n = x_{2n} + i x_{2n+1} with the usual pre/post-processing of the pairs
// (k, M-k); the imaginary part of the kz = 0 coefficient is ignored and the
// kz = N/2 coefficient is zero (it is not stored).
// ---------------------------------------------------------------------------
// NY, NZ: points along y and z where they differ from N (lines of NZ points at the
// NX x NY positions; physical arrays (3, N, NY, NZ)).
template <typename T>
__device__ __forceinline__ cx<T> pmul(cx<T> a, cx<T> b) { return mk(a.x * b.x, a.y * b.y); }

template <typename T, int N, int MODE, int TXO = 0, int NY = N, int NZ = N, int V = 0>
__device__ __forceinline__ void zpass_body(const PassArgs a, const int bx, const int by) {
  using G = Geometry<T, N, NY, NZ>;
  constexpr int M = G::M;
  constexpr int TW = G::TW, TS = TW / NZ;  // exp(-2 pi i k / NZ) = tw[k * TS]
  constexpr int TX = TXO > 0 ? TXO : G::ZTX;  // TXO: a tuned tile width of the small grids
  constexpr int LD = ZLay<M>::ld(6 * TX), PAD = ZLay<M>::PAD;
  constexpr size_t FS = G::FS;
  constexpr int NF = (MODE == ZM_CROSS) ? 6 : (MODE == ZM_MAXABS ? 1 : 3);
  extern __shared__ __align__(16) unsigned char smraw[];
  cx<T>* s = reinterpret_cast<cx<T>*>(smraw);
  const cx<T>* tw = reinterpret_cast<const cx<T>*>(a.tw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int x0 = bx * TX;
  const int y = by;

  if constexpr (MODE == ZM_LOAD) {
    // physical lines (x0 + x, y, :) of the 3 components, packed in pairs
    // (the whole tile in flight at once by cp.async, no register staging)
    const cx<T>* in = reinterpret_cast<const cx<T>*>(a.in);
    for (int e = threadIdx.x; e < 3 * TX * M; e += ZP_THREADS<T>) {
      const int n = e % M, x = (e / M) % TX, c = e / (M * TX);
      cp_async<sizeof(cx<T>)>(s + padrow<PAD>(n) * LD + c * TX + x, in + ((size_t)(c * N + x0 + x) * NY + y) * M + n);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
  } else {
    const cx<T>* src = reinterpret_cast<const cx<T>*>(MODE == ZM_MAXABS ? a.D : a.W);
    // a stage whose state vanishes outside the 2/3 box: the planes kz >= kc hold zeros
    // (the y-inverse left them alone) and are taken as zeros
    int klim = M;
    if constexpr (MODE == ZM_CROSS || MODE == ZM_STORE || MODE == ZM_PRODUCTS) {
      if (rows_vanish(a)) {
        klim = ((NZ == N ? a.kmax3 : a.kmax3z) + 2) / 3;
        if (klim > M) klim = M;
      }
    }
    constexpr int VX = LD % 2 == 0 && TX % 2 == 0 ? 2 : 1;  // values of a copy
    for (int e = threadIdx.x; e < NF * TX / VX * M; e += ZP_THREADS<T>) {
      const int x = e % (TX / VX) * VX, k = (e / (TX / VX)) % M, f = e / (TX / VX * M);
      if (k < klim)
        cp_async<VX * (int)sizeof(cx<T>)>(s + padrow<PAD>(k) * LD + f * TX + x, src + f * FS + ((size_t)k * NY + y) * N + x0 + x);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    constexpr int NL = NF * TX;
    // c2r pre-processing: Z'_k = (X_k + conj X_{M-k}) + i e^{+2 pi i k/N} (X_k - conj X_{M-k}),
    // stored conjugated so that a forward DFT gives the inverse one. The stage forms it in the first pass of the
    // line transforms; here apart, as before that (a choice for the same last bits, not for accuracy).
    if constexpr (MODE != ZM_CROSS) {
      for (int e = threadIdx.x; e < NL * (M / 2 + 1); e += ZP_THREADS<T>) {
        const int l = e % NL, k = e / NL;
        if (k == 0) {
          const T r0 = s[l].x;  // Im X_0 ignored, X_M = 0
          s[l] = mk(r0, -r0);
        } else {
          cx<T>* pk = s + padrow<PAD>(k) * LD + l;
          cx<T>* pm = s + padrow<PAD>(M - k) * LD + l;
          const cx<T> zero = mk((T)0, (T)0), xk = k < klim ? *pk : zero, xm = M - k < klim ? *pm : zero;
          const cx<T> wk = ldro(tw + k * TS);  // exp(-2 pi i k / NZ)
          const cx<T> A = xk + conjg(xm), B = xk - conjg(xm);
          *pk = conjg(A + mul_pi(cmul(conjg(wk), B)));
          if (k != M - k) {
            // partner M-k: e^{+2 pi i (M-k)/N} = -wk
            const cx<T> A2 = xm + conjg(xk), B2 = xm - conjg(xk);
            *pm = conjg(A2 - mul_pi(cmul(wk, B2)));
          }
        }
      }
      __syncthreads();
    }
    constexpr int GL = LinesPerWarp<M, V>::value <= TX ? LinesPerWarp<M, V>::value : TX;  // lines per warp
#pragma unroll 1
    for (int l = warp * GL; l < NL; l += (ZP_THREADS<T> / 32) * GL) warp_fft_lines<T, M, TW, GL, LD, PAD, V, MODE == ZM_CROSS ? LINES_C2R : LINES_PLAIN>(s + l, tw, lane, klim);
    __syncthreads();
    // now conj(s) = x_{2n} + i x_{2n+1} (physical values, unnormalised c2r)
  }

  if constexpr (MODE == ZM_CROSS) {
    for (int e = threadIdx.x; e < TX * M; e += ZP_THREADS<T>) {
      const int x = e % TX, n = e / TX;
      cx<T>* p = s + padrow<PAD>(n) * LD + x;
      const cx<T> u0 = conjg(p[0 * TX]), u1 = conjg(p[1 * TX]), u2 = conjg(p[2 * TX]);
      const cx<T> w0 = conjg(p[3 * TX]), w1 = conjg(p[4 * TX]), w2 = conjg(p[5 * TX]);
      // u x omega on both packed points (real and imaginary parts)
      p[0 * TX] = mk(u1.x * w2.x - u2.x * w1.x, u1.y * w2.y - u2.y * w1.y);
      p[1 * TX] = mk(u2.x * w0.x - u0.x * w2.x, u2.y * w0.y - u0.y * w2.y);
      p[2 * TX] = mk(u0.x * w1.x - u1.x * w0.x, u0.y * w1.y - u1.y * w0.y);
    }
    __syncthreads();
  }

  if constexpr (MODE == ZM_PRODUCTS) {
    for (int e = threadIdx.x; e < TX * M; e += ZP_THREADS<T>) {
      const int x = e % TX, n = e / TX;
      cx<T>* p = s + padrow<PAD>(n) * LD + x;
      const cx<T> u0 = p[0 * TX], u1 = p[1 * TX], u2 = p[2 * TX];  // conjugated: the products are the same
      p[0 * TX] = pmul(u0, u0);
      p[1 * TX] = pmul(u1, u1);
      p[2 * TX] = pmul(u2, u2);
      p[3 * TX] = pmul(u0, u1);
      p[4 * TX] = pmul(u0, u2);
      p[5 * TX] = pmul(u1, u2);
    }
    __syncthreads();
  }

  if constexpr (MODE == ZM_CROSS || MODE == ZM_LOAD || MODE == ZM_PRODUCTS) {
    constexpr int NP = MODE == ZM_PRODUCTS ? 6 : 3;  // lines per column
    constexpr int GL = LinesPerWarp<M, V>::value <= TX ? LinesPerWarp<M, V>::value : TX;
#pragma unroll 1
    for (int l = warp * GL; l < NP * TX; l += (ZP_THREADS<T> / 32) * GL) warp_fft_lines<T, M, TW, GL, LD, PAD, V, LINES_PLAIN>(s + l, tw, lane);
    __syncthreads();
    // r2c post-processing: X_k = 1/2 [(Z_k + conj Z_{M-k}) - i e^{-2 pi i k/N} (Z_k - conj Z_{M-k})]
    cx<T>* dst = reinterpret_cast<cx<T>*>(MODE == ZM_LOAD ? a.U : a.W);
    int kc = M;
    if (MODE == ZM_CROSS) {
      kc = ((NZ == N ? a.kmax3 : a.kmax3z) + 2) / 3;
      if (kc > M) kc = M;
    }
    if (MODE == ZM_PRODUCTS) kc = a.kz_keep;
    // the walk over (product, k < kc, x) with kc a compile-time constant where it is the
    // default rule's (or M), so that its divisions are multiplications
    auto post = [&](auto kcc) {
      constexpr int KC = decltype(kcc)::value;  // 0: kc known at run time only
      const int kk = KC > 0 ? KC : kc;
      for (int e = threadIdx.x; e < NP * TX * kk; e += ZP_THREADS<T>) {
        const int x = e % TX, k = (e / TX) % kk, c = e / (TX * kk);
        const int l = c * TX + x;
        const cx<T> zk = s[padrow<PAD>(k) * LD + l], zm = s[padrow<PAD>((M - k) % M) * LD + l];
        const cx<T> wk = ldro(tw + k * TS);
        const cx<T> A = zk + conjg(zm), B = zk - conjg(zm);
        dst[c * FS + ((size_t)k * NY + y) * N + x0 + x] = scal(A + mul_mi(cmul(wk, B)), (T)0.5);
      }
    };
    constexpr int KC0 = (NZ + 2) / 3 < M ? (NZ + 2) / 3 : M;  // kc of the rule 3|k| < NZ
    if (kc == M)
      post(std::integral_constant<int, M>{});
    else if (kc == KC0)
      post(std::integral_constant<int, KC0>{});
    else
      post(std::integral_constant<int, 0>{});
  } else if constexpr (MODE == ZM_STORE) {
    cx<T>* out = reinterpret_cast<cx<T>*>(a.out);
    for (int e = threadIdx.x; e < 3 * TX * M; e += ZP_THREADS<T>) {
      const int n = e % M, x = (e / M) % TX, c = e / (M * TX);
      out[((size_t)(c * N + x0 + x) * NY + y) * M + n] = conjg(s[padrow<PAD>(n) * LD + c * TX + x]);
    }
  } else if constexpr (MODE == ZM_MAXABS) {
    double m = 0.0;
    for (int e = threadIdx.x; e < TX * M; e += ZP_THREADS<T>) {
      const int x = e % TX, n = e / TX;
      const cx<T> v = s[padrow<PAD>(n) * LD + x];
      m = fmax(m, fmax(fabs((double)v.x), fabs((double)v.y)));
    }
    zpass_block_max<ZP_THREADS<T>>(m, a.maxbits);
  }
}

template <typename T, int N, int MODE, int TXO = 0, int NY = N, int NZ = N, int V = 0>
__global__ void __launch_bounds__(ZP_THREADS<T>, (Geometry<T, N, NY, NZ>::ZMIN)) k_zpass(PassArgs a) {
  if constexpr (sizeof(T) == 8) zpass64_body<N, MODE, TXO, NY, NZ, V>(a, blockIdx.x, blockIdx.y);
  else zpass_body<T, N, MODE, TXO, NY, NZ, V>(a, blockIdx.x, blockIdx.y);
}

// Batched form (ensembles): member blockIdx.z (TXO: a tuned tile width).
template <typename T, int N, int MODE, int TXO = 0, int V = 0>
__global__ void __launch_bounds__(ZP_THREADS<T>, (Geometry<T, N>::ZMIN)) k_zpass_b(const __grid_constant__ BatchArgs B) {
  if constexpr (sizeof(T) == 8) zpass64_body<N, MODE, TXO, N, N, V>(B.a[blockIdx.z], blockIdx.x, blockIdx.y);
  else zpass_body<T, N, MODE, TXO, N, N, V>(B.a[blockIdx.z], blockIdx.x, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Line transforms of k_ztma. A line of M = 128 or 256 values belongs to M / 16 lanes, lane h holding positions
// h + (M / 16) m (m < 16). HwTwL, per lane: the twiddle powers exp(-2 pi i h r / M) between its two passes, and the
// pair twiddle exp(-2 pi i (h + (M / 16) m) / 2M), formed on use as tl exp(-2 pi i m / 32) with a constant factor.
// ---------------------------------------------------------------------------
struct HwTwL {
  cx<float> p2[16];
  cx<float> tl;
  // ts: stride into a twiddle table longer than the real line's own (1 on its own table)
  __device__ __forceinline__ void init(const cx<float>* __restrict__ tw, int h, int ts = 1) {
    twiddle_powers<16>(ldro(tw + 2 * h * ts), p2);
    tl = ldro(tw + h * ts);
  }
  __device__ __forceinline__ cx<float> wk(int m) const {
    constexpr float c[16][2] = {
        {1.0f, -0.0f},
        {0.9807852804032304f, -0.19509032201612825f},
        {0.9238795325112867f, -0.3826834323650898f},
        {0.8314696123025452f, -0.5555702330196022f},
        {0.7071067811865476f, -0.7071067811865475f},
        {0.5555702330196023f, -0.8314696123025452f},
        {0.38268343236508984f, -0.9238795325112867f},
        {0.19509032201612833f, -0.9807852804032304f},
        {0.0f, -1.0f},
        {-0.1950903220161282f, -0.9807852804032304f},
        {-0.3826834323650897f, -0.9238795325112867f},
        {-0.555570233019602f, -0.8314696123025455f},
        {-0.7071067811865475f, -0.7071067811865476f},
        {-0.8314696123025453f, -0.5555702330196022f},
        {-0.9238795325112867f, -0.3826834323650899f},
        {-0.9807852804032304f, -0.1950903220161286f}
    };
    return m == 0 ? tl : cmul(tl, mk(c[m][0], c[m][1]));
  }
};

// ---------------------------------------------------------------------------
// Half-warp 512-point FFT for the N = 1024 z-pass (FP32). Lane h of a half-warp
// holds v[m] = x[h + 16 m], m < 32. With k = k1 + 32 k2: a 32-point DFT over m in
// each lane gives Y[h][k1]; after the twiddle exp(-2 pi i h k1 / 512) one
// shared-memory exchange gives lane h' the 16-point columns k1 = h' and h' + 16, whose DFTs over h leave
// v[j] = X[h' + 16 j] in the lane: the input layout again.
// ---------------------------------------------------------------------------
struct HwTw32 {
  cx<float> p[16];  // w^r, w = exp(-2 pi i h / 512), r < 16
  cx<float> q[16];  // w^(16 + r)
  cx<float> tl;     // exp(-2 pi i h / 1024)
  __device__ __forceinline__ void init(const cx<float>* __restrict__ tw, int h, int ts) {
    twiddle_powers<16>(ldro(tw + 2 * h * ts), p);
    p[0] = mk(1.f, 0.f);
    const cx<float> w16 = cmul(p[8], p[8]);
#pragma unroll
    for (int r = 0; r < 16; ++r) q[r] = r == 0 ? w16 : cmul(w16, p[r]);
    tl = ldro(tw + h * ts);
  }
  // exp(-2 pi i (h + 16 m) / 1024) = tl * exp(-2 pi i m / 64)
  __device__ __forceinline__ cx<float> wk(int m) const {
    constexpr float c[32][2] = {
      {1.0f, 0.0f},
      {0.9951847266721969f, -0.0980171403295606f},
      {0.9807852804032304f, -0.19509032201612825f},
      {0.9569403357322088f, -0.29028467725446233f},
      {0.9238795325112867f, -0.3826834323650898f},
      {0.881921264348355f, -0.47139673682599764f},
      {0.8314696123025452f, -0.5555702330196022f},
      {0.773010453362737f, -0.6343932841636455f},
      {0.7071067811865476f, -0.7071067811865475f},
      {0.6343932841636455f, -0.773010453362737f},
      {0.5555702330196023f, -0.8314696123025452f},
      {0.4713967368259978f, -0.8819212643483549f},
      {0.38268343236508984f, -0.9238795325112867f},
      {0.29028467725446233f, -0.9569403357322089f},
      {0.19509032201612833f, -0.9807852804032304f},
      {0.09801714032956077f, -0.9951847266721968f},
      {0.0f, -1.0f},
      {-0.09801714032956065f, -0.9951847266721969f},
      {-0.1950903220161282f, -0.9807852804032304f},
      {-0.29028467725446216f, -0.9569403357322089f},
      {-0.3826834323650897f, -0.9238795325112867f},
      {-0.4713967368259977f, -0.881921264348355f},
      {-0.555570233019602f, -0.8314696123025455f},
      {-0.6343932841636454f, -0.7730104533627371f},
      {-0.7071067811865475f, -0.7071067811865476f},
      {-0.773010453362737f, -0.6343932841636455f},
      {-0.8314696123025453f, -0.5555702330196022f},
      {-0.8819212643483549f, -0.47139673682599786f},
      {-0.9238795325112867f, -0.3826834323650899f},
      {-0.9569403357322088f, -0.2902846772544624f},
      {-0.9807852804032304f, -0.1950903220161286f},
      {-0.9951847266721968f, -0.09801714032956083f}};
    return m == 0 ? tl : cmul(tl, mk(c[m][0], c[m][1]));
  }
};

// ---------------------------------------------------------------------------
// Pipelined z-pass of the FP32 grids with z-lines of 256, 512 or 1024 points: one persistent block per SM walks
// tiles of TX adjacent x at fixed y, the whole tile (6 fields x M kz, 192 KB) in shared memory. Tensor copies (TMA)
// fill it with whole rows and drain the products' rows, the planes past the cut-off filled with zeros or left out
// by the bounds of the tensor; the next tile's omega arrives while the products are transformed, its u while
// omega is.
//
// Bound by the shared-memory pipe (12.7 k of its cycles a tile, two thirds busy at 512). Rows arrive in the copies'
// swizzle (16-byte chunks of a row permuted by the row number), so a warp takes pairs of adjacent columns: its
// half-warps' accesses are eight rows of a column pair, 128 bytes of distinct banks, and the exchange inside a line
// goes through rows permuted the same way (an address is one XOR). Against tiles moved in 8-byte pieces by cp.async
// and drained by the threads (each 32 pieces took six cycles of that pipe, a quarter of all; an address and an
// instruction each): 512^3 1476 -> 1060 us, 1024^3 15.99 -> 13.15 ms, 256^3 167 -> 146 us, 1024 x 512 x 256
// 1271 -> 1067 us. Shorter lines keep k_zpass (tiles of their own width, batched members).
// ---------------------------------------------------------------------------
__device__ __forceinline__ cx<float> lds(unsigned p) {
  cx<float> v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(p));
  return v;
}
__device__ __forceinline__ void sts(unsigned p, cx<float> v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(p), "f"(v.x), "f"(v.y));
}
__device__ __forceinline__ float4 lds4(unsigned p) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(p));
  return v;
}
__device__ __forceinline__ void sts4(unsigned p, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}
template <int M>
struct ZTma {
  static constexpr int TX = 4096 / M;                    // columns of a tile (32 KB a field)
  static constexpr int CX = TX < 16 ? TX : 16;           // columns of a copy: a field is TX / CX blocks of M rows
  static constexpr int ROWB = CX * 8, CB = M * ROWB, FB = 32768;  // bytes of a row (128 or 64), of a block, of a field
  static constexpr int HL = M == 128 ? 8 : 16, VALS = M / HL;  // lanes of a line, values of a line in a lane
  static constexpr int GL = 32 / HL;                     // columns of a warp
  static constexpr int NW = VALS == 16 ? 24 : 12;        // warps: 80 or 168 registers a thread
  static constexpr int BOX = M < 256 ? M : 256;          // rows of a copy
  static constexpr size_t SMEM = 6 * FB + 2048;          // 2 KB alignment: the address bits that are XORed
  using Tw = std::conditional_t<M == 512, HwTw32, HwTwL>;
  // swizzle of the copies: chunk ^ (row / (128 / ROWB)) % (ROWB / 16)
  static constexpr int SH = ROWB == 128 ? 0 : 1, MASK = ROWB / 16 - 1;
  static constexpr CUtensorMapSwizzle SWIZZLE = ROWB == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  // row r of a line and its chunk, to be XORed into the address of chunk p of row 0 (r < 2048 / ROWB)
  __host__ __device__ static constexpr unsigned at(unsigned r) { return r * ROWB | ((r >> SH) & MASK) * 16; }
};

// The M-point DFT of a line of HL lanes, lane h holding x[h + HL m] and then X[h + HL m]. Value r of lane h crosses
// in row R h + (r ^ h) of the line (R rows a lane). la: address of the line's row h.
//   M = 128: 16-point DFTs, two 8-point ones;  256: 16 x 16;  512: 32-point DFTs, two 16-point ones (HwTw32)
template <int M>
__device__ __forceinline__ void zt_fft(cx<float> (&v)[ZTma<M>::VALS], unsigned la, const typename ZTma<M>::Tw& ht, int h) {
  using Z = ZTma<M>;
  const unsigned we = la + h * Z::VALS * Z::ROWB;
  if constexpr (M == 256) {
    dft16(v);
#pragma unroll
    for (int r = 0; r < 16; ++r) sts(we ^ Z::at(r), v[r]);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = lds((la ^ Z::at(m)) + m * 16 * Z::ROWB);
    __syncwarp();
#pragma unroll
    for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], ht.p2[r]);
    dft16(v);
  } else {
    constexpr int R = Z::VALS;
    if constexpr (M == 128) {
      dft16(v);
#pragma unroll
      for (int k = 1; k < 16; ++k) v[k] = cmul(v[k], ht.p2[k]);
    } else {
      dft32(v);
#pragma unroll
      for (int k = 1; k < 32; ++k) v[k] = cmul(v[k], k < 16 ? ht.p[k] : ht.q[k - 16]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) sts(we ^ Z::at(r), v[r]);
    __syncwarp();
    cx<float> a[R / 2], b[R / 2];
#pragma unroll
    for (int g = 0; g < R / 2; ++g) {
      const unsigned q = (la ^ Z::at(g)) + g * R * Z::ROWB;
      a[g] = lds(q);
      b[g] = lds(q + R / 2 * Z::ROWB);
    }
    __syncwarp();
    dft<R / 2>(a);
    dft<R / 2>(b);
#pragma unroll
    for (int k2 = 0; k2 < R / 2; ++k2) {
      v[2 * k2] = a[k2];
      v[2 * k2 + 1] = b[k2];
    }
  }
}

// A block whose copies did not arrive within the limit: waits once more for the two under way and fills the products
// of its tiles from t on with NaN, which the checks of the state report. Out of line: in the kernel it cost
// the 1024-point transforms their registers (13.25 -> 13.79 ms, so 13.15).
template <int N, int NY, int NZ>
__device__ __noinline__ void ztma_give_up(cx<float>* W, int t, int kc, unsigned bar0, unsigned bar1, unsigned phase) {
  using Z = ZTma<NZ / 2>;
  constexpr size_t FS = Geometry<float, N, NY, NZ>::FS;
  constexpr int TX = Z::TX, XT = N / TX, NT = XT * NY;
  mbar_wait(bar0, phase);
  mbar_wait(bar1, phase);
  const float nan = __int_as_float(0x7fffffff);
#pragma unroll 1
  for (; t < NT; t += gridDim.x) {
#pragma unroll 1
    for (int e = threadIdx.x; e < 3 * kc * TX; e += 32 * Z::NW) {
      const int x = e % TX, k = (e / TX) % kc, f = e / (TX * kc);
      W[f * FS + ((size_t)k * NY + t / XT) * N + (t % XT) * TX + x] = mk(nan, nan);
    }
  }
}

// in: W as (x, y, kz, field), kz bounded by the planes that hold values; out: by the planes kept
template <int N, int NY, int NZ>
__global__ void __launch_bounds__(32 * ZTma<NZ / 2>::NW, 1)
    k_ztma(int kmax3, const void* __restrict__ twp, cx<float>* __restrict__ W, const __grid_constant__ CUtensorMap in,
           const __grid_constant__ CUtensorMap out) {
  constexpr int M = NZ / 2;
  using Z = ZTma<M>;
  constexpr int TX = Z::TX, CX = Z::CX, NW = Z::NW, FB = Z::FB, HL = Z::HL, V = Z::VALS, STEP = HL * Z::ROWB;
  constexpr int XT = N / TX, NT = XT * NY;  // tiles: x-tiles times y
  static_assert(N % TX == 0, "whole tiles");
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned long long bars[2];
  const unsigned s = (smem_addr(smraw) + 2047u) & ~2047u;
  const unsigned bar0 = smem_addr(bars), bar1 = bar0 + 8;
  const cx<float>* tw = reinterpret_cast<const cx<float>*>(twp);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // lane: column bit 3 of a pair; row h < HL in bits 0-2 and, of 16, 4 (of 8: the second pair)
  const int h = HL == 16 ? (lane & 7) | ((lane >> 4) << 3) : lane & 7, cb = (lane >> 3) & 1;
  const int hp = (HL - h) & (HL - 1);
  const int partner = HL == 16 ? (hp & 7) | (cb << 3) | ((hp >> 3) << 4) : (lane & 24) | hp;  // the lane of row HL - h
  const int kc = min((kmax3 + 2) / 3, M);

  if (threadIdx.x == 0) {
    mbar_init(bar0);
    mbar_init(bar1);
    mbar_init_done();
  }
  __syncthreads();
  auto fetch = [&](int t, int f0, unsigned bar) {
    mbar_expect(bar, 3 * FB);
    for (int b = f0 * (TX / CX); b < (f0 + 3) * (TX / CX); ++b) {
      for (int k = 0; k < M; k += Z::BOX)
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
            ::"r"(s + b * Z::CB + k * Z::ROWB), "l"(&in), "r"((t % XT) * TX + (b % (TX / CX)) * CX), "r"(t / XT), "r"(k),
            "r"(b / (TX / CX)), "r"(bar)
            : "memory");
    }
  };
  typename Z::Tw ht;
  ht.init(tw, h, Geometry<float, N, NY, NZ>::TW / NZ);
  // address of row r (the row h or HL - h of this lane) of this lane's column, the warp's columns starting at line l
  auto row = [&](int l, int r) {
    const int x = l + (HL == 8 ? (lane >> 4) * 2 : 0);
    return s + (x / CX) * Z::CB + r * Z::ROWB + (((x % CX) / 2) ^ ((r >> Z::SH) & Z::MASK)) * 16 + cb * 8;
  };

  // c2r of the TX lines of fields f0 .. f0+2, GL lines per warp at a time.
  // The inputs of modes k and M - k come from one pair (X_k, X_{M-k}): with
  // A = X_k + conj X_{M-k}, B = X_k - conj X_{M-k} and P = i conj(w_k) B,
  // z_k = A + P and z_{M-k} = conj(A - P). Lane h forms the pairs of its slots
  // m < V/2 (k = h + HL m); the mirror M - k = (HL - h) + HL (V - 1 - m) is slot
  // V - 1 - m of lane HL - h, which receives it by a shuffle. Lane 0 pairs its slots
  // m and V - m, takes the self-paired k = M/2 at m = 0 and forms k = 0 apart.
  auto c2r_lines = [&](int f0) {
    cx<float> v[V];
#pragma unroll 1
    for (int l = f0 * TX + Z::GL * w; l < (f0 + 3) * TX; l += Z::GL * NW) {
      const unsigned pa = row(l, h), pb = row(l, HL - h);
      const cx<float> x0 = lds(pa);
      cx<float> zq[V / 2];
#pragma unroll
      for (int m = 0; m < V / 2; ++m) {
        cx<float> xk, xm, w1;
        if (m == 0) {
          const cx<float> y = lds(h == 0 ? pa + V / 2 * STEP : pb + (V - 1) * STEP);  // X_{M/2}, X_{M-h}
          xk = h == 0 ? y : x0;
          xm = y;
          w1 = h == 0 ? mk(0.f, -1.f) : ht.wk(0);  // w_{M/2} = -i
        } else {
          xk = lds(pa + m * STEP);
          xm = lds(pb + (V - 1 - m) * STEP);
          w1 = ht.wk(m);
        }
        const cx<float> A = xk + conjg(xm), B = xk - conjg(xm);
        const cx<float> P = mul_pi(cmul(conjg(w1), B));
        v[m] = conjg(A + P);
        zq[m] = A - P;  // conj of z_{M-k}
      }
#pragma unroll
      for (int q = V / 2; q < V; ++q) {
        v[q].x = __shfl_sync(0xffffffffu, zq[V - 1 - q].x, partner);
        v[q].y = __shfl_sync(0xffffffffu, zq[V - 1 - q].y, partner);
      }
      if (h == 0) {
        v[V / 2] = v[0];
#pragma unroll
        for (int q = V / 2 + 1; q < V; ++q) v[q] = zq[V - q];
        v[0] = mk(x0.x, -x0.x);  // z_0 = (1 + i) Re X_0: Im X_0 ignored, X_M = 0
      }
      __syncwarp();
      zt_fft<M>(v, pa, ht, h);
#pragma unroll
      for (int m = 0; m < V; ++m) sts(pa + m * STEP, conjg(v[m]));
    }
  };

  int t = blockIdx.x;
  if (threadIdx.x == 0 && t < NT) {
    fetch(t, 3, bar0);
    fetch(t, 0, bar1);
  }
  unsigned phase = 0;
#pragma unroll 1
  for (; t < NT; t += gridDim.x, phase ^= 1) {
    const int tn = t + gridDim.x;
    bool ok = mbar_wait(bar0, phase);  // omega fields of tile t
    c2r_lines(3);
    ok = mbar_wait(bar1, phase) && ok;  // u fields of tile t
    c2r_lines(0);
    if (!__syncthreads_and(ok)) break;
    // u x omega at every point, into the u lines: all fields are permuted alike
    for (int i = threadIdx.x; i < FB / 16; i += 32 * NW) {
      const unsigned p = s + i * 16;
      const float4 u0 = lds4(p), u1 = lds4(p + FB), u2 = lds4(p + 2 * FB);
      const float4 w0 = lds4(p + 3 * FB), w1 = lds4(p + 4 * FB), w2 = lds4(p + 5 * FB);
      sts4(p, make_float4(u1.x * w2.x - u2.x * w1.x, u1.y * w2.y - u2.y * w1.y, u1.z * w2.z - u2.z * w1.z,
                          u1.w * w2.w - u2.w * w1.w));
      sts4(p + FB, make_float4(u2.x * w0.x - u0.x * w2.x, u2.y * w0.y - u0.y * w2.y, u2.z * w0.z - u0.z * w2.z,
                               u2.w * w0.w - u0.w * w2.w));
      sts4(p + 2 * FB, make_float4(u0.x * w1.x - u1.x * w0.x, u0.y * w1.y - u1.y * w0.y, u0.z * w1.z - u1.z * w0.z,
                                   u0.w * w1.w - u1.w * w0.w));
    }
    fence_copies();
    __syncthreads();
    if (threadIdx.x == 0 && tn < NT) fetch(tn, 3, bar0);  // the omega lines are free
    // r2c of the 3 TX product lines; X_k (k < kc) back into the line
    {
      cx<float> v[V];
#pragma unroll 1
      for (int l = Z::GL * w; l < 3 * TX; l += Z::GL * NW) {
        const unsigned pa = row(l, h);
#pragma unroll
        for (int m = 0; m < V; ++m) v[m] = lds(pa + m * STEP);
        __syncwarp();
        zt_fft<M>(v, pa, ht, h);
#pragma unroll
        for (int m = 0; m < V; ++m) {
          if (HL * m >= kc) break;  // slots m and above hold modes past the 2/3 cut
          cx<float> zo;
          zo.x = __shfl_sync(0xffffffffu, v[V - 1 - m].x, partner);
          zo.y = __shfl_sync(0xffffffffu, v[V - 1 - m].y, partner);
          if (h == 0) zo = v[(V - m) & (V - 1)];
          const cx<float> A = v[m] + conjg(zo), B = v[m] - conjg(zo);
          if (h + HL * m < kc) sts(pa + m * STEP, scal(A + mul_mi(cmul(ht.wk(m), B)), 0.5f));
        }
      }
    }
    fence_copies();
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int b = 0; b < 3 * (TX / CX); ++b) {
        for (int k = 0; k < kc; k += Z::BOX)
          asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
                       ::"l"(&out), "r"((t % XT) * TX + (b % (TX / CX)) * CX), "r"(t / XT), "r"(k), "r"(b / (TX / CX)),
                       "r"(s + b * Z::CB + k * Z::ROWB)
                       : "memory");
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the u lines have been read out
      if (tn < NT) fetch(tn, 0, bar1);
    }
  }
  // gave up at tile t: both of its copies were started, no later one
  if (t < NT) ztma_give_up<N, NY, NZ>(W, t, kc, bar0, bar1, phase);
  if (threadIdx.x == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// The tensor (x, y, kz < planes, field < fields) at W, and the box of a copy
template <int N, int NY, int NZ>
inline cudaError_t ztma_map(CUtensorMap* map, void* W, int planes, int fields) {
  using Z = ZTma<NZ / 2>;
  typedef CUresult (*Encode)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess
               ? (Encode)f : (Encode) nullptr;
  }();
  if (!encode) return cudaErrorNotSupported;
  const cuuint64_t dims[4] = {N, NY, (cuuint64_t)planes, (cuuint64_t)fields};
  const cuuint64_t strides[3] = {N * 8ull, (cuuint64_t)N * NY * 8, (cuuint64_t)N * NY * (NZ / 2) * 8};
  const cuuint32_t box[4] = {Z::CX, 1, Z::BOX, 1}, step[4] = {1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 4, W, dims, strides, box, step, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            Z::SWIZZLE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// FP64 spectral sums for the diagnostics (Parseval): per block
//   sum w|u|^2, sum w|omega|^2, sum w Re(conj(u).omega), count of non-finite,
// w = 1 at kz = 0 and 2 otherwise (half spectrum; kz = N/2 is zero).
// ---------------------------------------------------------------------------
template <typename T, int N, int NY = N, int NZ = N>
__global__ void __launch_bounds__(DG_THREADS) k_diag(PassArgs a) {
  using G = Geometry<T, N, NY, NZ>;
  constexpr size_t FS = G::FS;
  const cx<T>* U = reinterpret_cast<const cx<T>*>(a.U);
  double se = 0, sz = 0, sh = 0, bad = 0;
  for (size_t i = (size_t)blockIdx.x * DG_THREADS + threadIdx.x; i < FS; i += (size_t)gridDim.x * DG_THREADS) {
    const int kxi = (int)(i % N), kyi = (int)((i / N) % NY), kzi = (int)(i / ((size_t)N * NY));
    const double kx = kfreq(kxi, N) * a.ks[0], ky = kfreq(kyi, NY) * a.ks[1], kz = kzi * a.ks[2];
    const double w = kzi == 0 ? 1.0 : 2.0;
    const cx<T> a0 = U[i], a1 = U[FS + i], a2 = U[2 * FS + i];
    const double u0r = a0.x, u0i = a0.y, u1r = a1.x, u1i = a1.y, u2r = a2.x, u2i = a2.y;
    // omega = i (k x u): real part = -(k x u).imag, imag part = (k x u).real
    const double t0r = ky * u2r - kz * u1r, t0i = ky * u2i - kz * u1i;
    const double t1r = kz * u0r - kx * u2r, t1i = kz * u0i - kx * u2i;
    const double t2r = kx * u1r - ky * u0r, t2i = kx * u1i - ky * u0i;
    const double w0r = -t0i, w0i = t0r, w1r = -t1i, w1i = t1r, w2r = -t2i, w2i = t2r;
    const double uu = u0r * u0r + u0i * u0i + u1r * u1r + u1i * u1i + u2r * u2r + u2i * u2i;
    const double ww = w0r * w0r + w0i * w0i + w1r * w1r + w1i * w1i + w2r * w2r + w2i * w2i;
    const double uw = u0r * w0r + u0i * w0i + u1r * w1r + u1i * w1i + u2r * w2r + u2i * w2i;
    se += w * uu;
    sz += w * ww;
    sh += w * uw;
    if (!isfinite(uu)) bad += 1.0;
  }
  __shared__ double red[4][DG_THREADS / 32];
  double v[4] = {se, sz, sh, bad};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = v[q];
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0;
    for (int w = 0; w < DG_THREADS / 32; ++w) t += red[threadIdx.x][w];
    a.partials[blockIdx.x * 4 + threadIdx.x] = t;
  }
}

// Fixed-order final sum of the block partials into partials[DIAG_BLOCKS*4 + q].
__global__ void k_diag_final(double* partials, int nblocks);

// ---------------------------------------------------------------------------
// Host launchers for one (T, N).
// ---------------------------------------------------------------------------
// Number of SMs of the current device (persistent kernels launch one block each).
inline int num_sms() {
  static int n = 0;
  if (n == 0) {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
      n = v;
    else
      n = 148;
  }
  return n;
}

// NY, NZ: points along y and z where they differ from N (a non-cubic grid runs the
// generic passes only: no tuned tile widths, specialised z-passes or batched
// ensembles).
template <typename T, int N, int NY = N, int NZ = N>
struct SolverImpl {
  using G = Geometry<T, N, NY, NZ>;
  static constexpr int M = G::M;
  static constexpr bool ISO = NY == N && NZ == N;
  static constexpr int ROWS = M * NY;  // x-pass rows (kz, ky)
  static constexpr bool BATCHED = ISO && N <= BATCH_MAX_N;
  // FP32 z-lines of 256 to 1024 points: k_ztma
  static constexpr bool ZTMA = sizeof(T) == 4 && (NZ == 256 || NZ == 512 || NZ == 1024);
  // each direction's 2/3 cut-off (3|k_i| < kmax3 of that direction)
  static int k3y(const PassArgs& a) { return NY == N ? a.kmax3 : a.kmax3y; }
  static int k3z(const PassArgs& a) { return NZ == N ? a.kmax3 : a.kmax3z; }

  template <class K>
  static cudaError_t smem_attr(K k, size_t bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  }

  // y-pass tile widths offered to a tuner besides the default (grids of the
  // ensembles only, to bound the number of instantiations)
  static constexpr bool ytile_ok(int t) {
    return ISO && N <= BATCH_MAX_N && t >= 4 && t <= 32 && pow2_part(N) % t == 0 && t * (int)sizeof(cx<T>) <= 256;
  }
  // radix plan variants of the stage's line transforms offered to the tuner (SmemPlanV /
  // LinePlanV: 0 the default schedule, 1 AltPlan); the ensemble grids only. PassArgs::plan
  // holds one bit per pass: PLAN_X (x-stage and x inverse), PLAN_YI (y-inverse),
  // PLAN_Z (z-pass), PLAN_YF (y-forward).
  static constexpr int PLANS = (ISO && N <= BATCH_MAX_N) ? 2 : 1;
  // The handle's initial plan mask: AltPlan in the passes where it measured faster on
  // GB300 (per-pass CUDA-event times of both schedules; FP64 at 64^3: 213 against 282 us a step, since
  // two radix-8 passes of 64-point lines leave three lanes in four idle, and 3 - 15 % slower elsewhere). dns_tune_tiles re-measures on the machine at hand.
  static constexpr int default_plan() {
    if constexpr (PLANS == 1) {
      return 0;
    } else if constexpr (sizeof(T) == 8) {
      constexpr int XYY = (1 << PLAN_X) | (1 << PLAN_YI) | (1 << PLAN_YF);
      return (N == 16 || N == 64) ? XYY : 0;
    } else {
      switch (N) {
        case 48: return (1 << PLAN_X) | (1 << PLAN_YF);
        case 64: return (1 << PLAN_X) | (1 << PLAN_YI);
        case 128: return (1 << PLAN_X) | (1 << PLAN_YI) | (1 << PLAN_YF);
        default: return 0;
      }
    }
  }
  static int bit(int plan, int b) { return (plan >> b) & 1; }
  // f(std::integral_constant<int, V>) with the variant V = plan (0 where not offered)
  template <class F>
  static void with_plan(int plan, F&& f) {
    if constexpr (PLANS > 1) {
      if (plan == 1) return f(std::integral_constant<int, 1>{});
    }
    f(std::integral_constant<int, 0>{});
  }

  template <int TXO, int V>
  static void tile_attr_v(cudaError_t& e) {
    if (e == cudaSuccess) e = smem_attr(k_ypass<T, N, 1, 0, TXO, N, N, V>, YCfg<T, N, 1, TXO>::SMEM);
    if (e == cudaSuccess) e = smem_attr(k_ypass<T, N, 1, 0, TXO, N, N, V, 1>, YCfg<T, N, 1, TXO>::SMEM);
    if (e == cudaSuccess) e = smem_attr(k_ypass<T, N, 0, 1, TXO, N, N, V>, YCfg<T, N, 0, TXO>::SMEM);
    if (e == cudaSuccess) e = smem_attr(k_ypass_b<T, N, 1, 0, TXO, V>, YCfg<T, N, 1, TXO>::SMEM);
    if (e == cudaSuccess) e = smem_attr(k_ypass_b<T, N, 0, 1, TXO, V>, YCfg<T, N, 0, TXO>::SMEM);
  }
  template <int TXO>
  static void tile_attr(cudaError_t& e) {
    if constexpr (ytile_ok(TXO)) {
      tile_attr_v<TXO, 0>(e);
      if constexpr (PLANS > 1) tile_attr_v<TXO, 1>(e);
    }
  }
  static int y_tiles(int* tiles, int max) {
    int n = 0;
    for (int t = 4; t <= 32; t *= 2)
      if (ytile_ok(t) && n < max) tiles[n++] = t;
    return n;
  }
  // z-pass tile widths offered besides the default (the generic z-pass of the small grids)
  static constexpr bool ztile_ok(int t) {
    return ISO && N <= BATCH_MAX_N && t >= 4 && t <= 32 && pow2_part(N) % t == 0 &&
           G::zbytes(t) <= 112 * 1024;  // two blocks an SM
  }
  template <int TXO>
  static void ztile_attr(cudaError_t& e) {
    if constexpr (ztile_ok(TXO)) {
      if (e == cudaSuccess) e = smem_attr(k_zpass<T, N, ZM_CROSS, TXO>, G::zbytes(TXO));
      if (e == cudaSuccess) e = smem_attr(k_zpass_b<T, N, ZM_CROSS, TXO>, G::zbytes(TXO));
      if constexpr (PLANS > 1) {
        if (e == cudaSuccess) e = smem_attr(k_zpass<T, N, ZM_CROSS, TXO, N, N, 1>, G::zbytes(TXO));
        if (e == cudaSuccess) e = smem_attr(k_zpass_b<T, N, ZM_CROSS, TXO, 1>, G::zbytes(TXO));
      }
    }
  }
  static int z_tiles(int* tiles, int max) {
    int n = 0;
    for (int t = 4; t <= 32; t *= 2)
      if (ztile_ok(t) && n < max) tiles[n++] = t;
    return n;
  }
  template <int TXO, int V = 0>
  static void z_go(const PassArgs& a, cudaStream_t st) {
    constexpr int TX = TXO > 0 ? TXO : G::ZTX;
    k_zpass<T, N, ZM_CROSS, TXO, NY, NZ, V><<<dim3(N / TX, NY), ZP_THREADS<T>, G::zbytes(TX), st>>>(a);
  }
  // FP32 lines of 256 points and more along y: the y-pass with the lines in registers
  static constexpr bool YREG = sizeof(T) == 4 && (NY == 256 || NY == 512 || NY == 1024);
  // the y-pass through the shared-memory tile; PR: the y-inverse of a stage whose state vanishes outside the 2/3 box
  template <int INV, int PRUNE, int TXO, int V = 0, int PR = 0>
  static void y_tile(cx<T>* F, const cx<T>* tw, int kmax3, int planes, int fields, cudaStream_t st) {
    using Y = YCfg<T, N, INV, TXO, NY>;
    k_ypass<T, N, INV, PRUNE, TXO, NY, NZ, V, PR><<<dim3(N / Y::TX, planes, fields), Y::THREADS, Y::SMEM, st>>>(F, tw, kmax3);
  }
  template <int INV, int PRUNE, int TXO, int V = 0, int PR = 0>
  static void y_go(cx<T>* F, const cx<T>* tw, int kmax3, int planes, int fields, cudaStream_t st) {
    if constexpr (YREG) {
      using Y = YReg<NY>;
      const int kept = cmin((kmax3 + 2) / 3, NY / 2);  // 3 |ky| < kmax3
      k_yreg<N, NY, G::TW, INV><<<dim3(N / Y::TX, planes, fields), Y::THREADS, Y::SMEM, st>>>(F, tw, G::FS, PR ? kept : NY,
                                                                                           PRUNE ? kept : NY);
    } else {
      y_tile<INV, PRUNE, TXO, V, PR>(F, tw, kmax3, planes, fields, st);
    }
  }
  // the stage's y-pass with tile width `tile` (0, or a width not offered: the default) and
  // radix plan variant `plan`; pr (inverse only): the pruned form PR = 1
  template <int INV, int PRUNE>
  static void y_stage(int tile, int plan, cx<T>* F, const cx<T>* tw, int kmax3, int planes, int fields,
                      cudaStream_t st, bool pr = false) {
    with_plan(plan, [&](auto v) {
      constexpr int V = decltype(v)::value;
      auto go = [&](auto t) {
        constexpr int TXO = decltype(t)::value;
        if constexpr (INV) {
          if (pr) return y_go<INV, PRUNE, TXO, V, 1>(F, tw, kmax3, planes, fields, st);
        }
        y_go<INV, PRUNE, TXO, V, 0>(F, tw, kmax3, planes, fields, st);
      };
      if constexpr (ISO && N <= BATCH_MAX_N) {
        if constexpr (ytile_ok(4)) if (tile == 4) return go(std::integral_constant<int, 4>{});
        if constexpr (ytile_ok(8)) if (tile == 8) return go(std::integral_constant<int, 8>{});
        if constexpr (ytile_ok(16)) if (tile == 16) return go(std::integral_constant<int, 16>{});
        if constexpr (ytile_ok(32)) if (tile == 32) return go(std::integral_constant<int, 32>{});
      }
      go(std::integral_constant<int, 0>{});
    });
  }

  static cudaError_t prepare() {
    cudaError_t e = cudaSuccess;
    tile_attr<4>(e);
    tile_attr<8>(e);
    tile_attr<16>(e);
    tile_attr<32>(e);
    ztile_attr<4>(e);
    ztile_attr<8>(e);
    ztile_attr<16>(e);
    ztile_attr<32>(e);
#define DNS_ATTR(kern, bytes) \
  if (e == cudaSuccess) e = smem_attr(kern, bytes)
    DNS_ATTR((k_xpass<T, N, XM_INV_CURL, NY, NZ>), G::XSMEM);
    DNS_ATTR((k_xpass<T, N, XM_STAGE, NY, NZ>), G::XSMEM_ST);
    DNS_ATTR((k_xpass<T, N, XM_STAGE2N, NY, NZ>), G::XSMEM_ST);
    DNS_ATTR((k_xpass<T, N, XM_RHS, NY, NZ>), G::XSMEM_ST);
    DNS_ATTR((k_xpass<T, N, XM_FWD_STORE, NY, NZ>), G::XSMEM);
    DNS_ATTR((k_xpass<T, N, XM_INV_PLAIN, NY, NZ>), G::XSMEM);
    DNS_ATTR((k_xpass<T, N, XM_INV_DIV, NY, NZ>), G::XSMEM);
    if constexpr (YREG) {
      DNS_ATTR((k_yreg<N, NY, G::TW, 1>), YReg<NY>::SMEM);
      DNS_ATTR((k_yreg<N, NY, G::TW, 0>), YReg<NY>::SMEM);
    }
    DNS_ATTR((k_ypass<T, N, 1, 0, 0, NY, NZ>), (YCfg<T, N, 1, 0, NY>::SMEM));
    DNS_ATTR((k_ypass<T, N, 1, 0, 0, NY, NZ, 0, 1>), (YCfg<T, N, 1, 0, NY>::SMEM));
    DNS_ATTR((k_ypass<T, N, 0, 1, 0, NY, NZ>), (YCfg<T, N, 0, 0, NY>::SMEM));
    if constexpr (!YREG) DNS_ATTR((k_ypass<T, N, 0, 0, 0, NY, NZ>), (YCfg<T, N, 0, 0, NY>::SMEM));
    if constexpr (!ZTMA) DNS_ATTR((k_zpass<T, N, ZM_CROSS, 0, NY, NZ>), G::ZSMEM);
    if constexpr (PLANS > 1) {
      DNS_ATTR((k_xpass<T, N, XM_INV_CURL, N, N, 1>), G::XSMEM);
      DNS_ATTR((k_xpass<T, N, XM_STAGE, N, N, 1>), G::XSMEM_ST);
      DNS_ATTR((k_xpass<T, N, XM_STAGE2N, N, N, 1>), G::XSMEM_ST);
      DNS_ATTR((k_xpass<T, N, XM_RHS, N, N, 1>), G::XSMEM_ST);
      DNS_ATTR((k_ypass<T, N, 1, 0, 0, N, N, 1>), (YCfg<T, N, 1, 0>::SMEM));
      DNS_ATTR((k_ypass<T, N, 1, 0, 0, N, N, 1, 1>), (YCfg<T, N, 1, 0>::SMEM));
      DNS_ATTR((k_ypass<T, N, 0, 1, 0, N, N, 1>), (YCfg<T, N, 0, 0>::SMEM));
      DNS_ATTR((k_zpass<T, N, ZM_CROSS, 0, N, N, 1>), G::ZSMEM);
    }
    if constexpr (ZTMA) DNS_ATTR((k_ztma<N, NY, NZ>), ZTma<M>::SMEM);
    DNS_ATTR((k_zpass<T, N, ZM_STORE, 0, NY, NZ>), G::ZSMEM);
    DNS_ATTR((k_zpass<T, N, ZM_LOAD, 0, NY, NZ>), G::ZSMEM);
    DNS_ATTR((k_zpass<T, N, ZM_MAXABS, 0, NY, NZ>), G::ZSMEM);
    DNS_ATTR((k_zpass<T, N, ZM_PRODUCTS, 0, NY, NZ>), G::ZSMEM);
    if constexpr (BATCHED) {
      DNS_ATTR((k_ypass_b<T, N, 1, 0>), (YCfg<T, N, 1>::SMEM));
      DNS_ATTR((k_zpass_b<T, N, ZM_CROSS>), G::ZSMEM);
      DNS_ATTR((k_ypass_b<T, N, 0, 1>), (YCfg<T, N, 0>::SMEM));
      DNS_ATTR((k_xpass_b<T, N, XM_STAGE>), G::XSMEM_ST);
      DNS_ATTR((k_xpass_b<T, N, XM_STAGE2N>), G::XSMEM_ST);
      if constexpr (PLANS > 1) {
        DNS_ATTR((k_ypass_b<T, N, 1, 0, 0, 1>), (YCfg<T, N, 1>::SMEM));
        DNS_ATTR((k_zpass_b<T, N, ZM_CROSS, 0, 1>), G::ZSMEM);
        DNS_ATTR((k_ypass_b<T, N, 0, 1, 0, 1>), (YCfg<T, N, 0>::SMEM));
        DNS_ATTR((k_xpass_b<T, N, XM_STAGE, 1>), G::XSMEM_ST);
        DNS_ATTR((k_xpass_b<T, N, XM_STAGE2N, 1>), G::XSMEM_ST);
      }
    }
#undef DNS_ATTR
    return e;
  }

  static cudaError_t z_cross(const PassArgs& a, cudaStream_t st) {
    if constexpr (ZTMA) {
      CUtensorMap in, out;
      const int kc = kc_of(k3z(a));
      cudaError_t e = ztma_map<N, NY, NZ>(&in, a.W, a.prune >= PRUNE_ROWS ? kc : M, 6);
      if (e == cudaSuccess) e = ztma_map<N, NY, NZ>(&out, a.W, kc, 3);
      if (e != cudaSuccess) return e;
      k_ztma<N, NY, NZ><<<num_sms(), 32 * ZTma<M>::NW, ZTma<M>::SMEM, st>>>(k3z(a), a.tw, reinterpret_cast<cx<float>*>(a.W), in, out);
    } else if constexpr (!ISO) {
      z_go<0>(a, st);
    } else {
      with_plan(bit(a.plan, PLAN_Z), [&](auto v) {
        constexpr int V = decltype(v)::value;
        if constexpr (ztile_ok(4)) if (a.ztile == 4) return z_go<4, V>(a, st);
        if constexpr (ztile_ok(8)) if (a.ztile == 8) return z_go<8, V>(a, st);
        if constexpr (ztile_ok(16)) if (a.ztile == 16) return z_go<16, V>(a, st);
        if constexpr (ztile_ok(32)) if (a.ztile == 32) return z_go<32, V>(a, st);
        z_go<0, V>(a, st);
      });
    }
    return cudaGetLastError();
  }

  // shared memory of a stage-update launch: with the wide layout only the rows
  // the stage reads are allocated (3 in the first stage, 6 in the last, 9 in the
  // stages between), so the lighter stages keep more blocks per SM
  static size_t xsmem_stage(int stage, int last) {
    if constexpr (G::XPRE && G::XWIDE) {
      const int rows = stage == 0 ? 3 : (stage == last ? 6 : 9);
      return (size_t)(G::XST + rows * N) * sizeof(cx<T>);
    } else {
      return G::XSMEM_ST;
    }
  }

  static int kc_of(int kmax3) {
    int kc = (kmax3 + 2) / 3;
    return kc > M ? M : kc;
  }

  // rows of an x launch over the rows inside the box (the kernel maps them, xpass_body)
  static int kept_rows(const PassArgs& a) { return kc_of(k3z(a)) * (2 * xpass_kept_ky<NY>(k3y(a)) + 1); }
  // blocks of an x-stage or x-inverse launch: every row, or with a pruned state only the
  // kc_z x (2R + 1) rows inside the 2/3 box (the kernel maps them, xpass_body; N <= 512)
  static int x_rows(const PassArgs& a) {
    return xpass_compact_ok<N>() && a.prune >= PRUNE_ROWS ? kept_rows(a) : ROWS;
  }

  static cudaError_t x_inverse_curl(const PassArgs& a0, int from_stage, cudaStream_t st) {
    PassArgs a = a0;
    if (from_stage) a.U = a.US;
    with_plan(bit(a.plan, PLAN_X), [&](auto v) {
      k_xpass<T, N, XM_INV_CURL, NY, NZ, decltype(v)::value><<<x_rows(a), XP_THREADS, G::XSMEM, st>>>(f32args(a));
    });
    return cudaGetLastError();
  }

  // the stage's y-inverse of the 6 fields (a pruned state: the planes kz < kc only)
  static void y_inverse(const PassArgs& a, cudaStream_t st) {
    const bool pr = a.prune >= PRUNE_ROWS;
    y_stage<1, 0>(a.ytile[0], bit(a.plan, PLAN_YI), reinterpret_cast<cx<T>*>(a.W),
                  reinterpret_cast<const cx<T>*>(a.tw), k3y(a), pr ? kc_of(k3z(a)) : M, 6, st, pr);
  }

  static cudaError_t rhs_front(const PassArgs& a, cudaStream_t st) {
    cx<T>* W = reinterpret_cast<cx<T>*>(a.W);
    const cx<T>* tw = reinterpret_cast<const cx<T>*>(a.tw);
    y_inverse(a, st);
    const cudaError_t e = z_cross(a, st);
    if (e != cudaSuccess) return e;
    y_stage<0, 1>(a.ytile[1], bit(a.plan, PLAN_YF), W, tw, k3y(a), kc_of(k3z(a)), 3, st);
    return cudaGetLastError();
  }

  // the x-stage launch of a stage, in the form of the stage's scheme
  static void x_stage(const PassArgs& a, cudaStream_t st) {
    with_plan(bit(a.plan, PLAN_X), [&](auto v) {
      constexpr int V = decltype(v)::value;
      if (a.lsrk)
        k_xpass<T, N, XM_STAGE2N, NY, NZ, V><<<x_rows(a), XP_THREADS, xsmem_stage(a.stage, a.last), st>>>(f32args(a));
      else
        k_xpass<T, N, XM_STAGE, NY, NZ, V><<<x_rows(a), XP_THREADS, xsmem_stage(a.stage, a.last), st>>>(f32args(a));
    });
  }

  static cudaError_t rk_stage(const PassArgs& a, cudaStream_t st) {
    const cudaError_t e = rhs_front(a, st);
    if (e != cudaSuccess) return e;
    x_stage(a, st);
    return cudaGetLastError();
  }

  static cudaError_t rk_stage_part(const PassArgs& a, int part, cudaStream_t st) {
    cx<T>* W = reinterpret_cast<cx<T>*>(a.W);
    const cx<T>* tw = reinterpret_cast<const cx<T>*>(a.tw);
    switch (part) {
      case 0: y_inverse(a, st); break;
      case 1: return z_cross(a, st);
      case 2: y_stage<0, 1>(a.ytile[1], bit(a.plan, PLAN_YF), W, tw, k3y(a), kc_of(k3z(a)), 3, st); break;
      default: x_stage(a, st); break;
    }
    return cudaGetLastError();
  }

  // batched passes with tile width TXO (0: default) and plan variant V
  template <int INV, int PRUNE, int TXO, int V>
  static void yb_go(const BatchArgs& B, int count, int planes, int fields, cudaStream_t st) {
    using Y = YCfg<T, N, INV, TXO>;
    k_ypass_b<T, N, INV, PRUNE, TXO, V><<<dim3(N / Y::TX, planes, fields * count), Y::THREADS, Y::SMEM, st>>>(B, fields);
  }
  template <int INV, int PRUNE, int V>
  static void yb_stage(int tile, const BatchArgs& B, int count, int planes, int fields, cudaStream_t st) {
    if constexpr (ISO && N <= BATCH_MAX_N) {
      if constexpr (ytile_ok(4)) if (tile == 4) return yb_go<INV, PRUNE, 4, V>(B, count, planes, fields, st);
      if constexpr (ytile_ok(8)) if (tile == 8) return yb_go<INV, PRUNE, 8, V>(B, count, planes, fields, st);
      if constexpr (ytile_ok(16)) if (tile == 16) return yb_go<INV, PRUNE, 16, V>(B, count, planes, fields, st);
      if constexpr (ytile_ok(32)) if (tile == 32) return yb_go<INV, PRUNE, 32, V>(B, count, planes, fields, st);
    }
    yb_go<INV, PRUNE, 0, V>(B, count, planes, fields, st);
  }
  template <int TXO, int V>
  static void zb_go(const BatchArgs& B, int count, cudaStream_t st) {
    constexpr int TX = TXO > 0 ? TXO : G::ZTX;
    k_zpass_b<T, N, ZM_CROSS, TXO, V><<<dim3(N / TX, N, count), ZP_THREADS<T>, G::zbytes(TX), st>>>(B);
  }
  template <int V>
  static void zb_stage(int tile, const BatchArgs& B, int count, cudaStream_t st) {
    if constexpr (ztile_ok(4)) if (tile == 4) return zb_go<4, V>(B, count, st);
    if constexpr (ztile_ok(8)) if (tile == 8) return zb_go<8, V>(B, count, st);
    if constexpr (ztile_ok(16)) if (tile == 16) return zb_go<16, V>(B, count, st);
    if constexpr (ztile_ok(32)) if (tile == 32) return zb_go<32, V>(B, count, st);
    zb_go<0, V>(B, count, st);
  }

  // one batched stage; the members share one radix plan (the ensemble groups them by it)
  static cudaError_t rk_stage_batch(const PassArgs* A, int count, int kmax3, cudaStream_t st) {
    if constexpr (BATCHED) {
      if (count < 1 || count > BATCH_MAX_COUNT) return cudaErrorInvalidValue;
      for (int i = 1; i < count; ++i)
        if (A[i].plan != A[0].plan) return cudaErrorInvalidValue;
      BatchArgs B;
      for (int i = 0; i < count; ++i) B.a[i] = f32args(A[i]);
      // the members' tile widths where they agree (a size class tuned together), else the defaults
      int yi = A[0].ytile[0], yf = A[0].ytile[1], zt = A[0].ztile;
      for (int i = 1; i < count; ++i) {
        if (A[i].ytile[0] != yi) yi = 0;
        if (A[i].ytile[1] != yf) yf = 0;
        if (A[i].ztile != zt) zt = 0;
      }
      const int plan = A[0].plan;
      with_plan(bit(plan, PLAN_YI), [&](auto v) { yb_stage<1, 0, decltype(v)::value>(yi, B, count, M, 6, st); });
      with_plan(bit(plan, PLAN_Z), [&](auto v) { zb_stage<decltype(v)::value>(zt, B, count, st); });
      with_plan(bit(plan, PLAN_YF),
                [&](auto v) { yb_stage<0, 1, decltype(v)::value>(yf, B, count, kc_of(kmax3), 3, st); });
      with_plan(bit(plan, PLAN_X), [&](auto v) {
        constexpr int V = decltype(v)::value;
        if (A[0].lsrk)
          k_xpass_b<T, N, XM_STAGE2N, V><<<dim3(M * N, count), XP_THREADS, xsmem_stage(A[0].stage, A[0].last), st>>>(B);
        else
          k_xpass_b<T, N, XM_STAGE, V><<<dim3(M * N, count), XP_THREADS, xsmem_stage(A[0].stage, A[0].last), st>>>(B);
      });
      return cudaGetLastError();
    } else {
      return cudaErrorNotSupported;
    }
  }

  static cudaError_t rhs(const PassArgs& a, cudaStream_t st) {
    cudaError_t e = x_inverse_curl(a, 0, st);
    if (e != cudaSuccess) return e;
    e = rhs_front(a, st);
    if (e != cudaSuccess) return e;
    PassArgs b = a;
    b.stage = 0;
    with_plan(bit(b.plan, PLAN_X), [&](auto v) {
      k_xpass<T, N, XM_RHS, NY, NZ, decltype(v)::value><<<ROWS, XP_THREADS, xsmem_stage(0, 3), st>>>(f32args(b));
    });
    return cudaGetLastError();
  }

  static cudaError_t forward3d(const PassArgs& a0, cudaStream_t st) {
    PassArgs a = a0;
    a.prune = PRUNE_NONE;  // of the state, not of the fields transformed here
    k_zpass<T, N, ZM_LOAD, 0, NY, NZ><<<dim3(N / G::ZTX, NY), ZP_THREADS<T>, G::ZSMEM, st>>>(a);
    y_go<0, 0, 0>(reinterpret_cast<cx<T>*>(a.U), reinterpret_cast<const cx<T>*>(a.tw), k3y(a), M, 3, st);
    k_xpass<T, N, XM_FWD_STORE, NY, NZ><<<ROWS, XP_THREADS, G::XSMEM, st>>>(f32args(a));
    return cudaGetLastError();
  }

  // x inverse of the 3 fields of a.U into W, then `y` (a.prune: where they vanish) on the planes left
  template <class Y>
  static void inverse_xy(const PassArgs& a, cudaStream_t st, Y&& y) {
    k_xpass<T, N, XM_INV_PLAIN, NY, NZ><<<x_rows(a), XP_THREADS, G::XSMEM, st>>>(f32args(a));
    const bool pr = a.prune >= PRUNE_ROWS;
    y(pr, reinterpret_cast<cx<T>*>(a.W), reinterpret_cast<const cx<T>*>(a.tw), pr ? kc_of(k3z(a)) : M);
  }

  static cudaError_t inverse3d(const PassArgs& a, cudaStream_t st) {
    inverse_xy(a, st, [&](bool pr, cx<T>* W, const cx<T>* tw, int planes) {
      if (pr) y_go<1, 0, 0, 0, 1>(W, tw, k3y(a), planes, 3, st);
      else y_go<1, 0, 0>(W, tw, k3y(a), planes, 3, st);
    });
    k_zpass<T, N, ZM_STORE, 0, NY, NZ><<<dim3(N / G::ZTX, NY), ZP_THREADS<T>, G::ZSMEM, st>>>(a);
    return cudaGetLastError();
  }

  // F of the six products u_i u_j of the fields in a.U, into W[0..5] at the modes |k_i| < half only: the
  // physical fields stay in the z-pass, the y- and x-passes transform the planes kz < half and the rows
  // |ky| < half. Filtered products of a 512^3 FP32 state on 64^3: 2.2 ms, bound by the instruction issue of
  // the z-pass; 9.2 ms as read-back, products on the mesh, full transforms and filters (nine passes over
  // 1.6 GB fields, most of whose modes the filter dropped).
  static cudaError_t products_low(const PassArgs& a0, int half, cudaStream_t st) {
    PassArgs a = a0;
    a.kz_keep = half;
    inverse_xy(a, st, [&](bool pr, cx<T>* W, const cx<T>* tw, int planes) {
      if (pr) y_tile<1, 0, 0, 0, 1>(W, tw, k3y(a), planes, 3, st);
      else y_tile<1, 0, 0>(W, tw, k3y(a), planes, 3, st);
    });
    k_zpass<T, N, ZM_PRODUCTS, 0, NY, NZ><<<dim3(N / G::ZTX, NY), ZP_THREADS<T>, G::ZSMEM, st>>>(a);
    y_tile<0, 1, 0>(reinterpret_cast<cx<T>*>(a.W), reinterpret_cast<const cx<T>*>(a.tw), 3 * half, half, 6, st);
    a.kmax3 = a.kmax3y = a.kmax3z = 3 * half;
    a.prune = PRUNE_ROWS;  // the launch covers the rows inside this box
    for (int g = 0; g < 2; ++g) {
      a.U = reinterpret_cast<cx<T>*>(a.W) + 3 * g * G::FS;
      k_xpass<T, N, XM_FWD_STORE, NY, NZ><<<kept_rows(a), XP_THREADS, G::XSMEM, st>>>(f32args(a));
    }
    return cudaGetLastError();
  }

  static cudaError_t diag(const PassArgs& a, cudaStream_t st) {
    k_diag<T, N, NY, NZ><<<DIAG_BLOCKS, DG_THREADS, 0, st>>>(a);
    k_diag_final<<<1, 128, 0, st>>>(a.partials, DIAG_BLOCKS);
    k_xpass<T, N, XM_INV_DIV, NY, NZ><<<ROWS, XP_THREADS, G::XSMEM, st>>>(f32args(a));
    y_go<1, 0, 0>(reinterpret_cast<cx<T>*>(a.D), reinterpret_cast<const cx<T>*>(a.tw), k3y(a), M, 1, st);
    cudaMemsetAsync(a.maxbits, 0, sizeof(unsigned long long), st);
    k_zpass<T, N, ZM_MAXABS, 0, NY, NZ><<<dim3(N / G::ZTX, NY), ZP_THREADS<T>, G::ZSMEM, st>>>(a);
    return cudaGetLastError();
  }

  static const DnsOps* ops() {
    static const DnsOps o = {N,         sizeof(T) == 4 ? 0 : 1, sizeof(cx<T>), &prepare,   &x_inverse_curl,
                             &rk_stage, &rk_stage_part,        &rhs,          &forward3d, &inverse3d,
                             &diag,     BATCHED ? &rk_stage_batch : nullptr, &y_tiles, &z_tiles,
                             NY,        NZ,                    G::TW,         PLANS,      default_plan(), &products_low};
    return &o;
  }
};

}  // namespace dns
