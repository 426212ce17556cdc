// 64-bit fixed-point line transforms of the FP64 form.
//
// GB300 executes 2 FP64 operations per SM and clock but 64 32 x 32 -> 64-bit integer
// multiply-adds and 64 64-bit additions (measured: mad.wide.s32 66, add.s64 65, fma.rn.f64 2.0
// lanes per SM and clock), so a butterfly in 64-bit integers takes a thirtieth of the time of the
// same butterfly in FP64. Bound by integer issue now (256^3: both integer pipes about 55 % busy), no
// longer by the FP64 pipe. RK4 step with the zero rows skipped, FP64 butterflies -> these:
// 1024^3 2820 -> 877 ms, 512^3 302 -> 68.6 ms, 256^3 36.6 -> 7.73 ms, 128^3 4.84 -> 1.08 ms, 32^3 252 -> 90 us.
// A line transform of the FP64 form therefore runs on integers with one power
// of two as the scale of the whole line:
//
//   scale   L1 = sum |Re x| + |Im x| of the line bounds every partial sum of its DFT (all factors
//           have modulus 1), so 2^(K - 1023) >= L1 maps the line onto |v| <= 2^62 with no
//           growth left to guard against. L1 is summed from the upper words of the doubles,
//           taken relative to the line's largest exponent, rounded up.
//   input   v = x 2^(62 - (K - 1023)), rounded: an element keeps all 53 bits unless it is more
//           than 2^9 below L1.
//   passes  butterflies are exact additions plus products by constants; every product is rounded
//           at the last bit.
//   output  the 64-bit integer, normalised and rounded to 53 bits.
//
// Error against an exact transform: a last bit is 2^-62 L1 and L1 <= 2 sqrt(L) |x|_2, so the input
// rounding and the roundings of the products (0.3 of a last bit each) stay below the FP64 transform's
// 2^-53 |x|_2 up to the longest line; most where all |x_j| are equal, many bits below where few modes
// carry the line. Measured against extended precision (c2r and r2c of white, Gaussian and power-law
// fields, 16^3 .. 512^3): 0.5 - 2.3e-16 relative, where FP64 butterflies gave 1.1 - 5.8e-16.
// A line with a NaN or an infinity gives NaN everywhere. Lines whose largest value is below 2^-959 are
// taken times a power of two (FX_LIFT) and results past the fast conversion are rescaled (fx_far), so that the whole
// range of a double is kept, subnormal numbers too.
//
// Numbers here are cx<long long>. The low word of a factor is signed (w = hi 2^32 + lo, |lo| < 2^31).
#pragma once

#include "fft_core.cuh"

namespace dns {

typedef long long ll;
typedef cx<ll> fx;

// a b + c in one instruction (the compiler makes a product and two additions of the C expression)
__device__ __forceinline__ ll madw(int a, int b, ll c) {
  ll r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
// upper word of a when its low word is read as a signed number
__device__ __forceinline__ int fx_hi(ll a) { return (int)(a >> 32) + (int)((unsigned)a >> 31); }

// upper word of |a| (of ~a where a is negative)
__device__ __forceinline__ unsigned fx_upper(ll a) {
  const int hi = (int)(a >> 32);
  return (unsigned)(hi ^ (hi >> 31));
}
// a 2^n (floor), |n| <= 63
__device__ __forceinline__ ll fx_shift(ll a, int n) { return (a << max(n, 0)) >> max(-n, 0); }
__device__ __forceinline__ fx fx_shift(fx a, int n) { return mk(fx_shift(a.x, n), fx_shift(a.y, n)); }

// the left shift that takes a line of L1 norm l1 2^41 (l1 rounded up) to 62 bits
__device__ __forceinline__ int fx_shift_of(unsigned l1) { return __clz(l1) - 11; }

// (t >> 32) + c: a product by 1 takes the odd register of the pair t as it is
__device__ __forceinline__ ll fx_add_up(ll t, ll c) { return madw((int)(t >> 32), 1, c); }
// 4 p with the top two bits of t's low word below
__device__ __forceinline__ ll fx_times4(ll p, ll t) {
  const unsigned lo = __funnelshift_l((unsigned)t, (unsigned)p, 2);
  const int hi = (int)__funnelshift_l((unsigned)p, (unsigned)(p >> 32), 2);
  return (ll)(((unsigned long long)(unsigned)hi << 32) | lo);
}
// a w (QUARTER: a w / 4) rounded, w from the fixed-point table (xh, xl, yh, yl), |a| <= 2^62. The upper
// halves of the products, in 2^64 units, are 1/4 of the result; its last two bits are the top of t.
template <bool QUARTER = false>
__device__ __forceinline__ fx fx_cmul(fx a, int4 w) {
  const int axl = (int)a.x, axh = fx_hi(a.x), ayl = (int)a.y, ayh = fx_hi(a.y);
  const int nyh = -w.z, nyl = -w.w;
  constexpr ll HALF = QUARTER ? 1ll << 31 : 1ll << 29;
  ll t = madw(axl, w.x, HALF), u = madw(ayl, w.x, HALF);
  t = madw(axh, w.y, t);
  u = madw(ayh, w.y, u);
  t = madw(ayl, nyh, t);
  u = madw(axl, w.z, u);
  t = madw(ayh, nyl, t);
  u = madw(axh, w.w, u);
  const ll p = fx_add_up(t, madw(ayh, nyh, madw(axh, w.x, 0))), q = fx_add_up(u, madw(axh, w.z, madw(ayh, w.x, 0)));
  if constexpr (QUARTER) return mk(p, q);
  return mk(fx_times4(p, t), fx_times4(q, u));
}
// the fixed-point twiddle at index p of the table (the FP64 form's table holds these)
__device__ __forceinline__ int4 ldfx(const cx<double>* p) { return __ldg(reinterpret_cast<const int4*>(p)); }
// a / 4 rounded
__device__ __forceinline__ fx fx_quarter(fx a) { return mk((a.x + 2) >> 2, (a.y + 2) >> 2); }

// a b 2^-62, rounded; |a|, |b| <= 2^61
__device__ __forceinline__ ll fx_prod(ll a, ll b) {
  const int al = (int)a, ah = fx_hi(a), bl = (int)b, bh = fx_hi(b);
  const ll t = madw(ah, bl, madw(al, bh, 1ll << 29));
  return fx_times4(fx_add_up(t, madw(ah, bh, 0)), t);
}
// (a b - c d) 2^-62, rounded; |a|, |b|, |c|, |d| <= 2^61
__device__ __forceinline__ ll fx_cross(ll a, ll b, ll c, ll d) {
  const int al = (int)a, ah = fx_hi(a), bl = (int)b, bh = fx_hi(b);
  const int cl = (int)c, ch = fx_hi(c), dl = (int)d, dh = fx_hi(d);
  const ll t = madw(-ch, dl, madw(-dh, cl, madw(ah, bl, madw(al, bh, 1ll << 29))));
  return fx_times4(fx_add_up(t, madw(-ch, dh, madw(ah, bh, 0))), t);
}

// Constants |c| < 1/2 in units of 2^-64 (rounded from 60 digits): cos(pi/4) - 1 and sqrt(3)/2 - 1.
struct FxC {
  int hi, lo;
};
struct FxK {
  static constexpr FxC rt2{-1257966796, -102865788}, h3{-575416509, -1033546850};
};
// low-word part of a c (2^32 units) on top of t, and its upper part
__device__ __forceinline__ ll fx_lo(ll a, FxC c, ll t) { return madw(fx_hi(a), c.lo, madw((int)a, c.hi, t)); }
__device__ __forceinline__ ll fx_up(ll a, FxC c, ll t) { return madw(fx_hi(a), c.hi, t); }
// a (1 + c)
__device__ __forceinline__ ll fx_mul1(ll a, FxC c) { return fx_add_up(fx_lo(a, c, 1ll << 31), fx_up(a, c, a)); }
__device__ __forceinline__ void dft3(fx* v) {
  const fx t = v[1] + v[2], d = v[1] - v[2];
  const fx m = mk(v[0].x - (t.x >> 1), v[0].y - (t.y >> 1));
  const fx dd = mk(fx_mul1(d.y, FxK::h3), -fx_mul1(d.x, FxK::h3));
  v[0] = v[0] + t;
  v[1] = m + dd;
  v[2] = m - dd;
}
__device__ __forceinline__ fx fx_w8(fx a) { return mk(fx_mul1(a.x + a.y, FxK::rt2), fx_mul1(a.y - a.x, FxK::rt2)); }
__device__ __forceinline__ fx fx_w83(fx a) { return mk(fx_mul1(a.y - a.x, FxK::rt2), -fx_mul1(a.x + a.y, FxK::rt2)); }
__device__ __forceinline__ void dft8(fx* v) {
  fx e[4] = {v[0], v[2], v[4], v[6]};
  fx o[4] = {v[1], v[3], v[5], v[7]};
  dft4(e);
  dft4(o);
  o[1] = fx_w8(o[1]);
  o[2] = mul_mi(o[2]);
  o[3] = fx_w83(o[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = e[k] + o[k];
    v[k + 4] = e[k] - o[k];
  }
}
template <int R>
__device__ __forceinline__ void fx_dft(fx* v) {
  if constexpr (R == 2) dft2(v);
  else if constexpr (R == 3) dft3(v);
  else if constexpr (R == 4) dft4(v);
  else if constexpr (R == 8) dft8(v);
  else static_assert(R == 2, "unsupported radix");
}

// ---- scale of a line ---------------------------------------------------------------------
__device__ __forceinline__ unsigned fx_mag(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
__device__ __forceinline__ unsigned fx_mag(cx<double> v) { return max(fx_mag(v.x), fx_mag(v.y)); }
// |d| 2^-(exponent of top) as a float (zero where it is below 2^-127 of it)
__device__ __forceinline__ float fx_rel(double d, int top) { return __int_as_float(max((int)fx_mag(d) - top, 0) << 3); }
__device__ __forceinline__ int fx_top(unsigned mag) { return (int)(mag & 0x7ff00000u) - (127 << 20); }
// a lane's share of L1 / 2^(exponent of the line's largest element) in units of 2^-12, rounded up
__device__ __forceinline__ unsigned fx_share(float s) { return (unsigned)(s * 4096.5f) + 2u; }

struct FxScale {
  int K;         // biased exponent: L1 <= 2^(K - 1023)
  unsigned nan;  // 0x7ff80000 if the line holds a NaN or an infinity, else 0
};
// fx_from reads an exponent of 0 as zero and shifts elements of a line of scale K out below 2^(K - 1086): a line whose
// largest magnitude word is below 2^-959 is therefore multiplied by 2^FX_LIFT first, exactly, where it lies.
constexpr int FX_LIFT = 600;
__device__ __forceinline__ bool fx_tiny(unsigned mag) { return mag < (64u << 20); }  // or zero
__device__ __forceinline__ double fx_pow2(int n) { return __hiloint2double((1023 + n) << 20, 0); }
// the largest magnitude word after that (at most)
__device__ __forceinline__ unsigned fx_lifted(unsigned mag) { return max(mag, 1u << 20) + ((unsigned)FX_LIFT << 20); }
// from the line's largest magnitude word and the sum of its shares
__device__ __forceinline__ FxScale fx_scale(unsigned mag, unsigned shares) {
  FxScale s;
  s.K = mag ? (int)(mag >> 20) + 20 - __clz(shares) : 128;
  s.nan = mag >= 0x7ff00000u ? 0x7ff80000u : 0u;
  return s;
}

// d in the fixed point of scale K, d = v 2^(K - 1085)
__device__ __forceinline__ ll fx_from(double d, int K) {
  const int hi = __double2hiint(d), s = hi >> 31;
  const unsigned lo = (unsigned)__double2loint(d), mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
  const int r = min(K - 1 - ((hi >> 20) & 0x7ff), 63);
  const ll m = (ll)(((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10)) >> r;
  const ll sm = ((ll)s << 32) | (unsigned)s;
  return ((m ^ sm) + 1) >> 1;  // halves away from zero: (m + 1) / 2 or floor(-m / 2)
}
__device__ __forceinline__ fx fx_from(cx<double> v, int K) { return mk(fx_from(v.x, K), fx_from(v.y, K)); }
// the double v 2^(B - 1085), 64 <= B <= 2040 (B = K: a value of a line of scale K); of a negative v the
// magnitude is taken as ~v, a last bit (2^-62 L1) too small
__device__ __forceinline__ double fx_bits(ll v, int B, unsigned nan) {
  const int s = (int)(v >> 32) >> 31;
  const unsigned ah = (unsigned)((int)(v >> 32) ^ s), al = (unsigned)((int)v ^ s);
  const unsigned top = ah ? ah : al;
  const int sh = __clz(top) + (ah ? -1 : 31);  // the top bit goes to bit 62
  const unsigned long long q = (((((unsigned long long)ah << 32) | al) << sh) + 0x200u) >> 10;  // 53 bits, rounded
  const unsigned e = top ? (unsigned)(B - 1 - sh) : 0u;                                         // (a carry raises it)
  return __hiloint2double((int)(((unsigned)(q >> 32) + (e << 20)) | (s & 0x80000000u) | nan), (int)(unsigned)q);
}
__device__ __forceinline__ cx<double> fx_bits(fx v, int B, unsigned nan) { return mk(fx_bits(v.x, B, nan), fx_bits(v.y, B, nan)); }
// any other B: the conversion at FX_MID and then fx_rescale, which underflows gradually and overflows to infinity
constexpr int FX_MID = 1000;
__device__ __forceinline__ bool fx_far(int B) { return (unsigned)(B - 64) > 1976u; }
__device__ __forceinline__ cx<double> fx_rescale(cx<double> d, int B) {  // two steps, neither of which leaves the range
  const int n = max(min(B - FX_MID, 2040), -2040);
  return scal(scal(d, fx_pow2(n / 2)), fx_pow2(n - n / 2));
}
__device__ __forceinline__ cx<double> fx_to(fx v, int B, unsigned nan) {
  if (fx_far(B)) return fx_rescale(fx_bits(v, FX_MID, nan), B);
  return fx_bits(v, B, nan);
}

// ---- radix schedules -----------------------------------------------------------------------
// A butterfly holds four registers per value: radix 8 passes, 4 x 4 or 4 for what remains of the power of
// two (a radix-16 pass spills at the 80 registers that keep 24 warps on an SM), then radix 3; 16
// points as 8 x 2, since 4 x 4 is what variant 1 offers (AltPlan, as in the FP32 form).
template <int L, int V>
struct FxPlan : AltPlan<L> {};
template <int L>
struct FxPlan<L, 0> {
  static constexpr int three = (L % 3 == 0) ? 1 : 0, a = ilog2c(three ? L / 3 : L);
  static constexpr int n8 = a % 3 == 1 && a > 1 && L != 16 ? a / 3 - 1 : a / 3, rest = a - 3 * n8;  // 0, 1, 2 or 4
  static constexpr int np2 = n8 + (rest + 1) / 2, npass = np2 + three;
  static constexpr int radix(int p) { return p >= np2 ? 3 : (p < n8 ? 8 : (rest == 1 ? 2 : 4)); }
  static constexpr int ns(int p) {
    int r = 1;
    for (int q = 0; q < p; ++q) r *= radix(q);
    return r;
  }
  static_assert(ns(npass) == L, "plan covers the line");
};
// lines of one warp, as LinesPerWarp
template <int L, int V>
struct FxLinesPerWarp {
  static constexpr int nb0 = L / FxPlan<L, V>::radix(0);
  static constexpr int value = nb0 >= 32 ? 1 : (nb0 >= 16 ? 2 : (nb0 >= 8 ? 4 : (nb0 >= 4 ? 8 : 16)));
};

// Forward DFT of one line of length L by one warp: the FP32 form transforms floats, the FP64 form
// fixed point (below), where E multiplies the result by 2^E.
template <int L, int TWN, int P, int V, int E, class Src, class Work, class Dst>
__device__ __forceinline__ void warp_fft_fx_pass(const Src& src, const Work& work, const Dst& dst,
                                                 const cx<double>* __restrict__ tw, int lane, FxScale sc);
template <typename T, int L, int TWN, int V = 0, int E = 0, class Src, class Work, class Dst>
__device__ __forceinline__ void line_fft(const Src& src, const Work& work, const Dst& dst,
                                         const cx<T>* __restrict__ tw, int lane) {
  static_assert(sizeof(T) == 8 || E == 0, "only the fixed-point lines take a power of two");
  if constexpr (sizeof(T) == 8) warp_fft_fx_pass<L, TWN, 0, V, E>(src, work, dst, tw, lane, FxScale{});
  else warp_fft<T, L, TWN, V>(src, work, dst, tw, lane);
}

// ---- one line per warp -------------------------------------------------------------------
// The passes of warp_fft on fixed point: pass 0 reads doubles through `src`, the passes between
// exchange integers through `work`, the last writes doubles through `dst`.
template <int L, int TWN, int P, int V, int E, class Src, class Work, class Dst>
__device__ __forceinline__ void warp_fft_fx_pass(const Src& src, const Work& work, const Dst& dst,
                                                 const cx<double>* __restrict__ tw, int lane, FxScale sc) {
  using PL = FxPlan<L, V>;
  constexpr int R = PL::radix(P), NS = PL::ns(P), NB = L / R, BPL = (NB + 31) / 32;
  constexpr bool FIRST = (P == 0), LAST = (P + 1 == PL::npass), FAST = IsPow2<L>::value;
  constexpr int TWC = TWN / (NS * R);
  // up to 16 doubles stay in registers from the scale to the butterflies, longer lines are read twice
  constexpr bool KEEP = BPL * R <= 16;
  fx v[BPL][R];
  auto rd = [&](int j, int r) -> cx<double> {
    if constexpr (FAST) return src.load(src.at(j) + Src::off(r * NB));
    else return src.load(src.at(j + r * NB));
  };
  if constexpr (FIRST) {
    cx<double> d[KEEP ? BPL : 1][KEEP ? R : 1];
    unsigned m;
    int lift = 0;
#pragma unroll 1
    for (;;) {
      m = 0;
#pragma unroll
      for (int b = 0; b < BPL; ++b) {
        const int j = lane + 32 * b;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          cx<double> x = mk(0.0, 0.0);
          if (NB % 32 == 0 || j < NB) x = rd(j, r);
          if constexpr (KEEP) d[b][r] = x;
          m = max(m, fx_mag(x));
        }
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (!fx_tiny(m) || lift) break;
      unsigned any = m;
      if (m == 0) {  // zero, or below 2^-1042
#pragma unroll 1
        for (int p = lane; p < L; p += 32) {
          const cx<double> x = src.load(src.at(p));
          any |= (unsigned)__double2loint(x.x) | (unsigned)__double2loint(x.y);
        }
      }
      if (!__any_sync(0xffffffffu, any != 0)) break;
      lift = FX_LIFT;
#pragma unroll 1
      for (int p = lane; p < L; p += 32) {
        cx<double>* q = const_cast<cx<double>*>(src.at(p));  // this warp's line, which nobody reads after it
        *q = scal(*q, fx_pow2(FX_LIFT));
      }
      __syncwarp();
    }
    const int top = fx_top(m);
    float s = 0.f;
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
      const int j = lane + 32 * b;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        cx<double> x;
        if constexpr (KEEP) x = d[b][r];
        else x = (NB % 32 == 0 || j < NB) ? rd(j, r) : mk(0.0, 0.0);
        s += fx_rel(x.x, top) + fx_rel(x.y, top);
      }
    }
    sc = fx_scale(m, __reduce_add_sync(0xffffffffu, fx_share(s)));
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
      const int j = lane + 32 * b;
      if (NB % 32 == 0 || j < NB) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if constexpr (KEEP) v[b][r] = fx_from(d[b][r], sc.K);
          else v[b][r] = fx_from(rd(j, r), sc.K);
        }
        fx_dft<R>(v[b]);
      }
    }
    sc.K -= lift;  // of the values as they were
  } else {
#pragma unroll
    for (int b = 0; b < BPL; ++b) {
      const int j = lane + 32 * b;
      if (NB % 32 == 0 || j < NB) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const cx<double>* q;
          if constexpr (FAST) q = work.at(j) + Work::off(r * NB);
          else q = work.at(j + r * NB);
          v[b][r] = *reinterpret_cast<const fx*>(q);
        }
        const int kc = (j % NS) * TWC;
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = fx_cmul(v[b][r], ldfx(tw + r * kc));
        fx_dft<R>(v[b]);
      }
    }
  }
  __syncwarp();
  const bool far = LAST && fx_far(sc.K + E);
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int j = lane + 32 * b;
    if (NB % 32 == 0 || j < NB) {
      const int base = (j / NS) * NS * R + (j % NS);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (LAST) {
          const cx<double> o = fx_bits(v[b][r], far ? FX_MID : sc.K + E, sc.nan);
          if constexpr (FAST) dst.store(dst.at(base) + Dst::off(r * NS), base + r * NS, o);
          else dst.store(dst.at(base + r * NS), base + r * NS, o);
        } else {
          cx<double>* q;
          if constexpr (FAST) q = work.at(base) + Work::off(r * NS);
          else q = work.at(base + r * NS);
          *reinterpret_cast<fx*>(q) = v[b][r];
        }
      }
    }
  }
  __syncwarp();
  if (far) {  // apart from the stores, so that those stay short (in line with them a 24 x 48 x 16 x-stage took 14.3 us, not 12.3)
#pragma unroll 1
    for (int p = lane; p < L; p += 32) *dst.at(p) = fx_rescale(*dst.at(p), sc.K + E);
    __syncwarp();
  }
  if constexpr (!LAST) warp_fft_fx_pass<L, TWN, P + 1, V, E>(src, work, dst, tw, lane, sc);
}

// ---- several short lines per warp --------------------------------------------------------
// The passes of warp_fft_lines on lines of fixed-point values, in place. FROM: what pass 0 reads,
// fixed point (FX_IN), fixed point of line g to be shifted by fx_shift_of(sh[g]) (FX_SHIFT) or doubles to be
// taken to scale sh[g] (FX_DOUBLE).
// MAG: the upper words of the results' magnitudes are or'ed into mag[g] (cleared before): the top bit of the largest.
enum FxFrom { FX_IN = 0, FX_SHIFT = 1, FX_DOUBLE = 2 };
template <int L, int TWN, int G, int LD, int P, int V, int FROM, bool MAG = false>
__device__ __forceinline__ void warp_fft_fx_lines(cx<double>* s0, const cx<double>* __restrict__ tw, int lane,
                                                  const int* sh, unsigned* mag = nullptr) {
  using PL = FxPlan<L, V>;
  constexpr int R = PL::radix(P), NS = PL::ns(P), NB = L / R, TOT = G * NB, BPL = (TOT + 31) / 32;
  constexpr bool LAST = (P + 1 == PL::npass);
  constexpr int TWC = TWN / (NS * R);
  fx v[BPL][R];
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int vj = lane + 32 * b;
    if (TOT % 32 == 0 || vj < TOT) {
      const int g = vj / NB, j = vj % NB;
      const cx<double>* ln = s0 + g;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const cx<double>* q = ln + padt<double>(j + r * NB) * LD;
        if constexpr (P == 0 && FROM == FX_DOUBLE) v[b][r] = fx_from(*q, sh[g]);
        else v[b][r] = *reinterpret_cast<const fx*>(q);
      }
      if constexpr (P == 0 && FROM == FX_SHIFT) {
        const int n = fx_shift_of((unsigned)sh[g]);
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = fx_shift(v[b][r], n);
      }
      if constexpr (NS > 1) {
        const int kc = (j % NS) * TWC;
#pragma unroll
        for (int r = 1; r < R; ++r) v[b][r] = fx_cmul(v[b][r], ldfx(tw + r * kc));
      }
      fx_dft<R>(v[b]);
    }
  }
  __syncwarp();
#pragma unroll
  for (int b = 0; b < BPL; ++b) {
    const int vj = lane + 32 * b;
    if (TOT % 32 == 0 || vj < TOT) {
      const int g = vj / NB, j = vj % NB;
      cx<double>* ln = s0 + g;
      const int base = (j / NS) * NS * R + (j % NS);
#pragma unroll
      for (int r = 0; r < R; ++r) *reinterpret_cast<fx*>(ln + padt<double>(base + r * NS) * LD) = v[b][r];
    }
    if constexpr (LAST && MAG) {
      unsigned m = 0;
      if (TOT % 32 == 0 || vj < TOT) {
#pragma unroll
        for (int r = 0; r < R; ++r) m |= fx_upper(v[b][r].x) | fx_upper(v[b][r].y);
      }
      if constexpr (NB % 32 == 0) {  // the warp's lanes are on one line
        m = __reduce_or_sync(0xffffffffu, m);
        if (lane == 0) mag[vj / NB] |= m;
      } else if constexpr (32 % NB == 0) {  // NB adjacent lanes are
#pragma unroll
        for (int o = NB / 2; o > 0; o >>= 1) m |= __shfl_xor_sync(0xffffffffu, m, o);
        if (vj % NB == 0 && vj < TOT) mag[vj / NB] |= m;
      } else {
        if (vj < TOT) atomicOr(mag + vj / NB, m);
      }
    }
  }
  __syncwarp();
  if constexpr (!LAST) warp_fft_fx_lines<L, TWN, G, LD, P + 1, V, FROM, MAG>(s0, tw, lane, sh, mag);
}

}  // namespace dns
