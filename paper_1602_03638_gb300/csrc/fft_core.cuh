// Complex arithmetic, small-radix DFT butterflies and a shared-memory Stockham
// FFT engine for the batched 1D transforms of the pseudo-spectral solver.
//
// The 3D transforms of Eqs. fft/ifft (Sec. 2) are compositions of 1D
// transforms along z (real), y and x (complex). Every 1D transform here is a
// forward DFT  X_k = sum_j x_j exp(-2 pi i j k / L)  computed by one warp with
// a mixed-radix (8, then 16/4/2, then 3) Stockham autosort: natural order in
// and out, one pass per radix, each lane holding its butterflies in registers
// and exchanging through a shared-memory line between passes (warp barriers
// only). The first pass may read and the last pass may write global memory
// directly. Inverse transforms use conj(DFT(conj(x))), folded into the
// callers' loads and stores. Twiddles come from a table of
// exp(-2 pi i t / TWN), t < TWN, generated on the host in FP64 (rounded to T
// for the FP32 form).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dns {

template <typename T>
struct __align__(2 * sizeof(T)) cx {
  T x, y;
};

template <typename T>
__device__ __forceinline__ cx<T> mk(T a, T b) { cx<T> r; r.x = a; r.y = b; return r; }
template <typename T>
__device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return mk(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return mk(a.x - b.x, a.y - b.y); }
template <typename T>
__device__ __forceinline__ cx<T> cmul(cx<T> a, cx<T> b) {
  return mk(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename T>
__device__ __forceinline__ cx<T> conjg(cx<T> a) { return mk(a.x, -a.y); }
// the sign bit of a double flipped by the integer unit: an FP64 negation is an addition on the FP64 pipe
__device__ __forceinline__ double neg64(double a) {
  return __hiloint2double(__double2hiint(a) ^ (int)0x80000000, __double2loint(a));
}
__device__ __forceinline__ cx<double> conjg(cx<double> a) { return mk(a.x, neg64(a.y)); }
template <typename T>
__device__ __forceinline__ cx<T> scal(cx<T> a, T s) { return mk(a.x * s, a.y * s); }
// a * (-i)
template <typename T>
__device__ __forceinline__ cx<T> mul_mi(cx<T> a) { return mk(a.y, -a.x); }
// a * (+i)
template <typename T>
__device__ __forceinline__ cx<T> mul_pi(cx<T> a) { return mk(-a.y, a.x); }
__device__ __forceinline__ cx<double> mul_pi(cx<double> a) { return mk(neg64(a.y), a.x); }

// The butterflies' arithmetic on the two parts at once. FP32: the packed instructions (two additions or
// multiply-adds per issue slot; the pipe's rate is the same), rounded as the scalar ones are. A quarter fewer
// instructions in the passes (512^3 z-pass: 1.20e9 -> 0.89e9), which were 60 % of the issue slots or more:
// RK4 step at 512^3 12.93 -> 12.46 ms, 256^3 1.54 -> 1.48, 1024^3 129.6 -> 126.9, 1024 x 512 x 256 13.38 -> 12.60.
template <typename T>
__device__ __forceinline__ cx<T> add2(cx<T> a, cx<T> b) { return a + b; }
template <typename T>
__device__ __forceinline__ cx<T> sub2(cx<T> a, cx<T> b) { return a - b; }
// (a.x b.x + c.x, a.y b.y + c.y)
template <typename T>
__device__ __forceinline__ cx<T> fma2(cx<T> a, cx<T> b, cx<T> c) { return mk(a.x * b.x + c.x, a.y * b.y + c.y); }
__device__ __forceinline__ cx<float> add2(cx<float> a, cx<float> b) {
  cx<float> r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; add.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ cx<float> fma2(cx<float> a, cx<float> b, cx<float> c) {
  cx<float> r;
  asm("{.reg .b64 a, b, c, d; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; mov.b64 c, {%6, %7}; fma.rn.f32x2 d, a, b, c; "
      "mov.b64 {%0, %1}, d;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ cx<float> sub2(cx<float> a, cx<float> b) {
  cx<float> r;
  asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; sub.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

// Read-only cached load of one complex value (twiddle tables).
__device__ __forceinline__ cx<float> ldro(const cx<float>* p) {
  float2 v = __ldg(reinterpret_cast<const float2*>(p));
  return mk(v.x, v.y);
}
__device__ __forceinline__ cx<double> ldro(const cx<double>* p) {
  double2 v = __ldg(reinterpret_cast<const double2*>(p));
  return mk(v.x, v.y);
}

// ---------------------------------------------------------------------------
// Forward DFT butterflies of size 2, 3, 4, 8, 16 (in place, natural order).
// Constants are the exact values cos/sin of pi/4, pi/8 and sqrt(3)/2.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void dft2(cx<T>* v) {
  cx<T> a = v[0];
  v[0] = add2(a, v[1]);
  v[1] = sub2(a, v[1]);
}

template <typename T>
__device__ __forceinline__ void dft3(cx<T>* v) {
  const T h3 = (T)0.86602540378443864676;  // sqrt(3)/2
  cx<T> t = v[1] + v[2];
  cx<T> m = mk(v[0].x - (T)0.5 * t.x, v[0].y - (T)0.5 * t.y);
  cx<T> d = v[1] - v[2];
  cx<T> dd = mk(d.y * h3, -d.x * h3);  // (b - c) * (-i sqrt(3)/2)
  v[0] = v[0] + t;
  v[1] = m + dd;
  v[2] = m - dd;
}

template <typename T>
__device__ __forceinline__ void dft4(cx<T>* v) {
  cx<T> t0 = add2(v[0], v[2]), t1 = sub2(v[0], v[2]);
  cx<T> t2 = add2(v[1], v[3]);
  const cx<T> d = mk(v[1].y - v[3].y, v[1].x - v[3].x);  // t1 + (-i) (v1 - v3) and t1 - ...
  v[0] = add2(t0, t2);
  v[2] = sub2(t0, t2);
  v[1] = fma2(d, mk((T)1, (T)-1), t1);
  v[3] = fma2(d, mk((T)-1, (T)1), t1);
}

template <typename T>
__device__ __forceinline__ void dft8(cx<T>* v) {
  const T h = (T)0.70710678118654752440;
  cx<T> e[4] = {v[0], v[2], v[4], v[6]};
  cx<T> o[4] = {v[1], v[3], v[5], v[7]};
  dft4(e);
  dft4(o);
  v[0] = add2(e[0], o[0]);
  v[4] = sub2(e[0], o[0]);
  const cx<T> p = mk(o[1].x + o[1].y, o[1].y - o[1].x);  // sqrt(2) o1 exp(-i pi/4)
  v[1] = fma2(p, mk(h, h), e[1]);
  v[5] = fma2(p, mk(-h, -h), e[1]);
  const cx<T> q = mk(o[2].y, o[2].x);  // o2 exp(-i pi/2) = (q.x, -q.y)
  v[2] = fma2(q, mk((T)1, (T)-1), e[2]);
  v[6] = fma2(q, mk((T)-1, (T)1), e[2]);
  const cx<T> r = mk(o[3].y - o[3].x, o[3].x + o[3].y);  // sqrt(2) o3 exp(-3i pi/4) = (r.x, -r.y)
  v[3] = fma2(r, mk(h, -h), e[3]);
  v[7] = fma2(r, mk(-h, h), e[3]);
}

template <typename T>
__device__ __forceinline__ void dft16(cx<T>* v) {
  const T c1 = (T)0.92387953251128675613;  // cos(pi/8)
  const T s1 = (T)0.38268343236508977173;  // sin(pi/8)
  const T h = (T)0.70710678118654752440;
  cx<T> e[8], o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    e[k] = v[2 * k];
    o[k] = v[2 * k + 1];
  }
  dft8(e);
  dft8(o);
  v[0] = add2(e[0], o[0]);
  v[8] = sub2(e[0], o[0]);
  const cx<T> p = mk(o[2].x + o[2].y, o[2].y - o[2].x), q = mk(o[4].y, o[4].x), r = mk(o[6].y - o[6].x, o[6].x + o[6].y);
  v[2] = fma2(p, mk(h, h), e[2]);
  v[10] = fma2(p, mk(-h, -h), e[2]);
  v[4] = fma2(q, mk((T)1, (T)-1), e[4]);
  v[12] = fma2(q, mk((T)-1, (T)1), e[4]);
  v[6] = fma2(r, mk(h, -h), e[6]);
  v[14] = fma2(r, mk(-h, h), e[6]);
  // o[k] *= exp(-i pi k / 8), k odd
  o[1] = cmul(o[1], mk(c1, -s1));
  o[3] = cmul(o[3], mk(s1, -c1));
  o[5] = cmul(o[5], mk(-s1, -c1));
  o[7] = cmul(o[7], mk(-c1, -s1));
#pragma unroll
  for (int k = 1; k < 8; k += 2) {
    v[k] = add2(e[k], o[k]);
    v[k + 8] = sub2(e[k], o[k]);
  }
}

// 32-point DFT in place: two 16-point DFTs of the even and odd elements
// combined with exp(-2 pi i k / 32) (exact constants).
template <typename T>
__device__ __forceinline__ void dft32(cx<T>* v) {
  constexpr double c32[16][2] = {
      {1.0, 0.0},
      {0.9807852804032304, -0.19509032201612825},
      {0.9238795325112867, -0.3826834323650898},
      {0.8314696123025452, -0.5555702330196022},
      {0.7071067811865476, -0.7071067811865475},
      {0.5555702330196023, -0.8314696123025452},
      {0.38268343236508984, -0.9238795325112867},
      {0.19509032201612833, -0.9807852804032304},
      {0.0, -1.0},
      {-0.1950903220161282, -0.9807852804032304},
      {-0.3826834323650897, -0.9238795325112867},
      {-0.555570233019602, -0.8314696123025455},
      {-0.7071067811865475, -0.7071067811865476},
      {-0.8314696123025453, -0.5555702330196022},
      {-0.9238795325112867, -0.3826834323650899},
      {-0.9807852804032304, -0.1950903220161286}};
  cx<T> e[16], o[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    e[k] = v[2 * k];
    o[k] = v[2 * k + 1];
  }
  dft16(e);
  dft16(o);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    cx<T> t;
    if (k == 0) t = o[0];
    else if (k == 8) t = mul_mi(o[8]);
    else t = cmul(o[k], mk((T)c32[k][0], (T)c32[k][1]));
    v[k] = add2(e[k], t);
    v[k + 16] = sub2(e[k], t);
  }
}

template <int R, typename T>
__device__ __forceinline__ void dft(cx<T>* v) {
  if constexpr (R == 2) dft2(v);
  else if constexpr (R == 3) dft3(v);
  else if constexpr (R == 4) dft4(v);
  else if constexpr (R == 8) dft8(v);
  else if constexpr (R == 16) dft16(v);
  else if constexpr (R == 32) dft32(v);
  else static_assert(R == 2, "unsupported radix");
}

// Powers w^1..w^(R-1) of one twiddle w = exp(-2 pi i k / (NS R)) loaded from the
// FP64-generated table: one table load per butterfly instead of R-1 scattered
// loads, the rest formed by a multiplication tree at most 4 products deep.
template <int R, typename T>
__device__ __forceinline__ void twiddle_powers(cx<T> w1, cx<T>* w) {
  w[1] = w1;
  if constexpr (R > 2) w[2] = cmul(w1, w1);
  if constexpr (R > 3) w[3] = cmul(w[2], w1);
  if constexpr (R > 4) {
    w[4] = cmul(w[2], w[2]);
    w[5] = cmul(w[4], w1);
    w[6] = cmul(w[3], w[3]);
    w[7] = cmul(w[4], w[3]);
  }
  if constexpr (R > 8) {
    w[8] = cmul(w[4], w[4]);
#pragma unroll
    for (int r = 9; r < R; ++r) w[r] = cmul(w[8], w[r - 8]);
  }
}

// ---------------------------------------------------------------------------
// Asynchronous global -> shared copies (cp.async, sm_80+): used to prefetch
// the next tile while the current one is transformed.
// ---------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void cp_async(void* smem_dst, const void* gmem_src) {
  static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async size");
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(gmem_src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(PENDING) : "memory"); }

// ---------------------------------------------------------------------------
// Bulk copies (contiguous ranges, tensor boxes) that report to an mbarrier.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
// makes the initialised barriers known to the copies; a block barrier follows
__device__ __forceinline__ void mbar_init_done() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// bytes (a multiple of 16) of contiguous memory; both addresses 16-byte aligned
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gmem_src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(smem_dst)), "l"(gmem_src), "r"(bytes), "r"(bar)
               : "memory");
}
// what threads did to shared memory before the copies that follow a barrier
__device__ __forceinline__ void fence_copies() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// waits for the phase `parity` of the mbarrier; false if it did not complete within a second
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
  unsigned long long t0 = 0;
  for (int it = 0;; ++it) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (it == 0) t0 = t;
    else if (t - t0 > 1000000000ull) return false;
  }
}

// ---------------------------------------------------------------------------
// Shared-memory line layout: element p sits at padded position p + p/16. With
// this padding both the contiguous accesses (j + r*L/R over lanes j) and the
// stride-R Stockham stores of every pass used here touch each bank pair at
// most twice per warp (the minimum for 8-byte words).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int padp(int p) { return p + (p >> 4); }
__host__ __device__ constexpr int padded_len(int L) { return L + L / 16 + 1; }
// The padding by type: FP64 lines (16-byte values, eight of them to all the banks) are padded every 8,
// so that the radix-8 Stockham stores of a quarter-warp (rows 9 j) hit distinct banks; padded every 16
// they met two by two.
template <typename T>
__host__ __device__ constexpr int padt(int p) { return sizeof(T) == 8 ? p + (p >> 3) : padp(p); }
template <typename T>
__host__ __device__ constexpr int padt_len(int L) { return sizeof(T) == 8 ? padt<T>(L - 1) + 1 : padded_len(L); }

template <int PAD>
__host__ __device__ constexpr int padrow(int p) { return PAD ? p + p / (PAD ? PAD : 1) : p; }

constexpr int ilog2c(int x) {
  int r = 0;
  while (x > 1) { x >>= 1; ++r; }
  return r;
}

// Radix schedule of the warp FFT for L = 2^a or 3 * 2^a: radix-8 passes, the
// remaining factor 2 or 4 as one radix-16 or radix-4 pass, then radix 3.
template <int L>
struct WarpPlan {
  static constexpr int three = (L % 3 == 0) ? 1 : 0;
  static constexpr int p2 = three ? L / 3 : L;
  static constexpr int a = ilog2c(p2);
  static_assert((1 << a) == p2 && (p2 % 3) != 0, "FFT length must be 2^a or 3*2^a");
  static constexpr int n8 = a / 3, rem = a % 3;
  // list of power-of-two radices
  static constexpr int np2 = (rem == 0) ? n8 : (rem == 1 ? (n8 >= 1 ? n8 : 1) : n8 + 1);
  static constexpr int npass = np2 + three;
  static constexpr int radix(int p) {
    if (p >= np2) return 3;
    if (rem == 0) return 8;
    if (rem == 1) return (n8 == 0) ? 2 : (p == np2 - 1 ? 16 : 8);
    return p == np2 - 1 ? 4 : 8;
  }
  static constexpr int ns(int p) {
    int r = 1;
    for (int q = 0; q < p; ++q) r *= radix(q);
    return r;
  }
};

// Radix schedule of the shared-memory warp FFT (warp_fft). For 8-byte values
// and 512- or 1024-point lines the schedules (16, 16, 2) and (16, 16, 4) replace
// the radix-8 ones: with the padded line layout (element stride 1 or any odd
// stride) their reads and Stockham writes hit distinct banks in every pass,
// while the radix-8 schedules' second-pass writes conflict two-way, and they
// need slightly fewer operations per point. Other cases use WarpPlan.
template <int L, int CB>
struct SmemPlan : WarpPlan<L> {};
template <int L, int R0, int R1, int R2>
struct FixedPlan3 {
  static constexpr int npass = 3;
  static constexpr int radix(int p) { return p == 0 ? R0 : (p == 1 ? R1 : R2); }
  static constexpr int ns(int p) {
    int r = 1;
    for (int q = 0; q < p; ++q) r *= radix(q);
    return r;
  }
  static_assert(R0 * R1 * R2 == L, "plan covers the line");
};
template <>
struct SmemPlan<512, 8> : FixedPlan3<512, 16, 16, 2> {};
template <>
struct SmemPlan<1024, 8> : FixedPlan3<1024, 16, 16, 4> {};

// Alternative radix schedule (plan variant 1, offered to the tile tuner of the small
// grids): radix 3 first where L has the factor 3, then radix-4 passes, and one radix-8
// pass last when the power-of-two exponent is odd (radix 2 when it is 1). More passes
// of smaller radix than WarpPlan: more butterflies per pass (lanes busy), fewer
// registers, one more exchange through shared memory.
template <int L>
struct AltPlan {
  static constexpr int three = (L % 3 == 0) ? 1 : 0;
  static constexpr int p2 = three ? L / 3 : L;
  static constexpr int a = ilog2c(p2);
  static_assert((1 << a) == p2 && (p2 % 3) != 0 && a >= 1, "FFT length must be 2^a or 3*2^a");
  static constexpr int odd_r = (a % 2) ? (a == 1 ? 2 : 8) : 0;  // the last power-of-two radix
  static constexpr int n4 = (a % 2) ? (a == 1 ? 0 : (a - 3) / 2) : a / 2;
  static constexpr int npass = three + n4 + (odd_r ? 1 : 0);
  static constexpr int radix(int p) { return (three && p == 0) ? 3 : (p - three < n4 ? 4 : odd_r); }
  static constexpr int ns(int p) {
    int r = 1;
    for (int q = 0; q < p; ++q) r *= radix(q);
    return r;
  }
};

// The plan of variant V: 0 = the default schedule, 1 = AltPlan.
template <int L, int CB, int V>
struct SmemPlanV : SmemPlan<L, CB> {};
template <int L, int CB>
struct SmemPlanV<L, CB, 1> : AltPlan<L> {};
template <int L, int V>
struct LinePlanV : WarpPlan<L> {};
template <int L>
struct LinePlanV<L, 1> : AltPlan<L> {};

template <int L>
struct IsPow2 {
  static constexpr bool value = L > 0 && (L & (L - 1)) == 0;
};

// Access policies for the warp FFT. at(p) gives the address of position p;
// for power-of-two plans every pass touches positions base + d with
// padt(base + d) = padt(base) + padt(d), so off(d) is a compile-time offset.
template <typename T, int ES>
struct SLine {  // a line in shared memory at padded positions, element stride ES
  cx<T>* s;
  __device__ __forceinline__ cx<T>* at(int p) const { return s + padt<T>(p) * ES; }
  static constexpr int off(int d) { return padt<T>(d) * ES; }
  __device__ __forceinline__ cx<T> load(const cx<T>* q) const { return *q; }
  __device__ __forceinline__ void store(cx<T>* q, int, cx<T> v) const { *q = v; }
};
template <typename T, int ES>
struct SLineConj {  // shared-memory line read conjugated (inverse DFT of staged data)
  cx<T>* s;
  __device__ __forceinline__ cx<T>* at(int p) const { return s + padt<T>(p) * ES; }
  static constexpr int off(int d) { return padt<T>(d) * ES; }
  __device__ __forceinline__ cx<T> load(const cx<T>* q) const { return conjg(*q); }
};
template <typename T>
struct SRow {  // unpadded contiguous line in shared memory (read only)
  const cx<T>* s;
  __device__ __forceinline__ const cx<T>* at(int p) const { return s + p; }
  static constexpr int off(int d) { return d; }
  __device__ __forceinline__ cx<T> load(const cx<T>* q) const { return *q; }
};
template <typename T, bool CONJ>
struct GLoad {  // contiguous line in global memory
  const cx<T>* g;
  __device__ __forceinline__ const cx<T>* at(int p) const { return g + p; }
  static constexpr int off(int d) { return d; }
  __device__ __forceinline__ cx<T> load(const cx<T>* q) const {
    const cx<T> v = *q;
    return CONJ ? conjg(v) : v;
  }
};
template <typename T, bool CONJ>
struct GStore {
  cx<T>* g;
  __device__ __forceinline__ cx<T>* at(int p) const { return g + p; }
  static constexpr int off(int d) { return d; }
  __device__ __forceinline__ void store(cx<T>* q, int, cx<T> v) const { *q = CONJ ? conjg(v) : v; }
};

template <typename T, int L, int TWN, int P, int V, class Src, class Work, class Dst>
__device__ __forceinline__ void warp_fft_pass(const Src& src, const Work& work, const Dst& dst,
                                              const cx<T>* __restrict__ tw, int lane) {
  using PL = SmemPlanV<L, (int)sizeof(cx<T>), V>;
  constexpr int R = PL::radix(P);
  constexpr int NS = PL::ns(P);
  constexpr int NB = L / R;
  constexpr int BPL = (NB + 31) / 32;
  constexpr bool FIRST = (P == 0);
  constexpr bool LAST = (P + 1 == PL::npass);
  constexpr bool FAST = IsPow2<L>::value;
  constexpr int TWC = TWN / (NS * R);
  cx<T> v[BPL][R];
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int j = lane + 32 * b;
    if (NB % 32 == 0 || j < NB) {
      if constexpr (FIRST) {
        if constexpr (FAST) {
          const auto q = src.at(j);
#pragma unroll
          for (int r = 0; r < R; ++r) v[b][r] = src.load(q + Src::off(r * NB));
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) v[b][r] = src.load(src.at(j + r * NB));
        }
      } else {
        if constexpr (FAST) {
          const auto q = work.at(j);
#pragma unroll
          for (int r = 0; r < R; ++r) v[b][r] = work.load(q + Work::off(r * NB));
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) v[b][r] = work.load(work.at(j + r * NB));
        }
      }
      if constexpr (NS > 1) {
        cx<T> w[R];
        twiddle_powers<R>(ldro(tw + (j % NS) * TWC), w);
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = cmul(v[b][r], w[r]);
      }
      dft<R>(v[b]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int j = lane + 32 * b;
    if (NB % 32 == 0 || j < NB) {
      const int base = (j / NS) * NS * R + (j % NS);
      if constexpr (LAST) {
        if constexpr (FAST) {
          const auto q = dst.at(base);
#pragma unroll
          for (int r = 0; r < R; ++r) dst.store(q + Dst::off(r * NS), base + r * NS, v[b][r]);
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) dst.store(dst.at(base + r * NS), base + r * NS, v[b][r]);
        }
      } else {
        if constexpr (FAST) {
          const auto q = work.at(base);
#pragma unroll
          for (int r = 0; r < R; ++r) work.store(q + Work::off(r * NS), base + r * NS, v[b][r]);
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) work.store(work.at(base + r * NS), base + r * NS, v[b][r]);
        }
      }
    }
  }
  __syncwarp();
  if constexpr (!LAST) warp_fft_pass<T, L, TWN, P + 1, V>(src, work, dst, tw, lane);
}

// Forward DFT of one line of length L by one warp: reads through `src`, uses
// the shared-memory line `work` between passes, writes through `dst` (which may
// alias `work` or `src`: every pass reads all its values before writing).
// V: the radix plan variant (SmemPlanV).
template <typename T, int L, int TWN, int V = 0, class Src, class Work, class Dst>
__device__ __forceinline__ void warp_fft(const Src& src, const Work& work, const Dst& dst,
                                         const cx<T>* __restrict__ tw, int lane) {
  warp_fft_pass<T, L, TWN, 0, V>(src, work, dst, tw, lane);
}

// ---------------------------------------------------------------------------
// Several short lines per warp: G lines at s0 + g (g < G), element p of every
// line at row padrow<PAD>(p) of LD values, transformed in place. The butterflies
// of all G lines of a pass are spread over the lanes (virtual butterfly
// g * NB + j), so short lines whose passes have fewer butterflies than lanes
// still keep the warp busy. Same radix plan and twiddles as warp_fft.
// ---------------------------------------------------------------------------
template <int L, int V = 0>
struct LinesPerWarp {  // largest power of two G with G * (butterflies of pass 0) <= 32, at most 16
  static constexpr int nb0 = L / LinePlanV<L, V>::radix(0);
  static constexpr int value = nb0 >= 32 ? 1 : (nb0 >= 16 ? 2 : (nb0 >= 8 ? 4 : (nb0 >= 4 ? 8 : 16)));
};

// IN, what pass 0 takes: LINES_CONJ conj of the line, the rows r0 <= p < r1 as zeros (not read);
// LINES_C2R the half spectrum X_k (k < r0, zeros above) of 2L real values and forms the input of the
// L-point DFT on the way, conj Z'_k with Z'_k = (X_k + conj X_{L-k}) + i e^{+2 pi i k / 2L} (X_k - conj X_{L-k}), so that
// the forward DFT gives the inverse one (Im X_0 ignored, X_L = 0). PAD: position p lies in row p + p / PAD (0: p).
enum LinesIn { LINES_PLAIN = 0, LINES_CONJ = 1, LINES_C2R = 2 };
template <typename T, int L, int TWN, int G, int LD, int PAD, int P, int V, int IN>
__device__ __forceinline__ void warp_fft_lines_pass(cx<T>* s0, const cx<T>* __restrict__ tw, int lane, int r0, int r1) {
  using PL = LinePlanV<L, V>;
  constexpr int R = PL::radix(P);
  constexpr int NS = PL::ns(P);
  constexpr int NB = L / R;
  constexpr int TOT = G * NB;
  constexpr int BPL = (TOT + 31) / 32;
  constexpr bool LAST = (P + 1 == PL::npass);
  constexpr int TWC = TWN / (NS * R);
  cx<T> v[BPL][R];
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int vj = lane + 32 * b;
    if (TOT % 32 == 0 || vj < TOT) {
      const int g = vj / NB, j = vj % NB;
      const cx<T>* ln = s0 + g;
      if constexpr (IN == LINES_C2R && P == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int k = j + r * NB;
          cx<T> x = mk((T)0, (T)0), m = x;
          if (k < r0) x = ln[padrow<PAD>(k) * LD];
          if (k > 0 && L - k < r0) m = ln[padrow<PAD>(L - k) * LD];
          const bool low = k <= L / 2;
          const cx<T> w1 = ldro(tw + (low ? k : L - k) * (TWN / (2 * L)));
          const cx<T> A = x + conjg(m), B = x - conjg(m);  // e^{+2 pi i k / 2L} = -w1 above the middle
          v[b][r] = low ? conjg(A + mul_pi(cmul(conjg(w1), B))) : conjg(A - mul_pi(cmul(w1, B)));
          if (r == 0 && j == 0) v[b][r] = mk(x.x, -x.x);
        }
      } else if constexpr (IN == LINES_CONJ && P == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int k = j + r * NB;
          v[b][r] = conjg(k >= r0 && k < r1 ? mk((T)0, (T)0) : ln[padrow<PAD>(k) * LD]);
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = ln[padrow<PAD>(j + r * NB) * LD];
      }
      if constexpr (NS > 1) {
        cx<T> w[R];
        twiddle_powers<R>(ldro(tw + (j % NS) * TWC), w);
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = cmul(v[b][r], w[r]);
      }
      dft<R>(v[b]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int vj = lane + 32 * b;
    if (TOT % 32 == 0 || vj < TOT) {
      const int g = vj / NB, j = vj % NB;
      cx<T>* ln = s0 + g;
      const int base = (j / NS) * NS * R + (j % NS);
#pragma unroll
      for (int r = 0; r < R; ++r) ln[padrow<PAD>(base + r * NS) * LD] = v[b][r];
    }
  }
  __syncwarp();
  if constexpr (!LAST) warp_fft_lines_pass<T, L, TWN, G, LD, PAD, P + 1, V, IN>(s0, tw, lane, r0, r1);
}

// Forward DFT, in place, of the G lines s0 + g (see above) by one warp (V: plan variant).
template <typename T, int L, int TWN, int G, int LD, int PAD, int V, int IN>
__device__ __forceinline__ void warp_fft_lines(cx<T>* s0, const cx<T>* __restrict__ tw, int lane, int r0 = 0, int r1 = 0) {
  warp_fft_lines_pass<T, L, TWN, G, LD, PAD, 0, V, IN>(s0, tw, lane, r0, r1);
}

}  // namespace dns
