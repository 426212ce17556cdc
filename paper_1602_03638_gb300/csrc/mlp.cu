// Pointwise subgrid-stress network 10 -> 64 (SiLU) -> 64 (SiLU) -> 6 on the 5th-generation tensor
// cores (tcgen05.mma, BF16 operands in shared memory, FP32 accumulators in TMEM): inference
// (k_mlp_tc), the training pass (k_mlp_train: forward, backward and the weight gradients) and Adam on
// FP32 master weights (k_reduce).
//
// Parameter vector (floats), in this order:
//   in_shift[10] in_scale[10] W1[10][64] b1[64] W2[64][64] b2[64] W3[64][6]
//   b3[6] out_scale[6] out_shift[6]                                  (5286 values)
// Inputs are standardised as (x - in_shift) * in_scale; the network output y
// is the standardised stress, tau = y * out_scale + out_shift. The training
// loss is the mean over points and components of (y - (t - out_shift) /
// out_scale)^2. Feature and stress arrays are planar: X[f * P + p], T[c * P + p].
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "../../include/dns.h"
#include "dns_internal.h"

namespace dns {
void set_error_message(const char* msg);
}

namespace {

constexpr int NIN = 10, NH = 64, NOUT = 6;
constexpr int O_INSH = 0, O_INSC = 10, O_W1 = 20, O_B1 = 660, O_W2 = 724, O_B2 = 4820, O_W3 = 4884, O_B3 = 5268,
              O_OUTSC = 5274, O_OUTSH = 5280, NPARAM = 5286;
constexpr int TRAIN_BEGIN = O_W1, TRAIN_END = O_OUTSC;  // trainable range [W1 .. b3]
constexpr int NTRAIN = TRAIN_END - TRAIN_BEGIN;  // 5254

typedef __nv_bfloat16 bf;

// byte offset of element (r, k) of a K-major operand with K columns in the core-matrix layout
__host__ __device__ constexpr int tc_off(int r, int k, int K) {
  return ((r >> 3) * (K >> 3) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2;
}
// The BF16 weights as the B operands of the kernels, byte for byte the shared-memory image (made once
// per change of the parameters, so that a block stages them by 16-byte copies; gathering them from
// the row-major matrices in every block took 5 of the 17 us of a small inference): for the
// forward products W1^T (64 x 16), W2^T (64 x 64), W3^T (16 x 64, rows >= 6 zero), for the backward
// ones W2 (64 x 64) and W3 (64 x 16, columns >= 6 zero).
constexpr int IMG_W1 = 0, IMG_W2 = IMG_W1 + 2048, IMG_W3 = IMG_W2 + 8192, IMG_FWD = IMG_W3 + 2048, IMG_W2B = IMG_FWD,
              IMG_W3B = IMG_W2B + 8192, IMG_BYTES = IMG_W3B + 2048;

// puts parameter i (value v) where the image holds it
__device__ __forceinline__ void pack_param(int i, float v, unsigned char* img) {
  const bf w = __float2bfloat16(v);
  auto put = [&](int at) { *reinterpret_cast<bf*>(img + at) = w; };
  if (i >= O_W1 && i < O_B1) {
    const int k = (i - O_W1) / NH, n = (i - O_W1) % NH;
    put(IMG_W1 + tc_off(n, k, 16));
  } else if (i >= O_W2 && i < O_B2) {
    const int k = (i - O_W2) / NH, n = (i - O_W2) % NH;
    put(IMG_W2 + tc_off(n, k, 64));
    put(IMG_W2B + tc_off(k, n, 64));
  } else if (i >= O_W3 && i < O_B3) {
    const int k = (i - O_W3) / NOUT, c = (i - O_W3) % NOUT;
    put(IMG_W3 + tc_off(c, k, 64));
    put(IMG_W3B + tc_off(k, c, 16));
  }
}
__global__ void k_pack(const float* __restrict__ p, unsigned char* __restrict__ img) {
  for (int i = threadIdx.x + blockIdx.x * blockDim.x; i < NPARAM; i += blockDim.x * gridDim.x) pack_param(i, p[i], img);
}

// Logistic functions of two values, 1 / (1 + exp(-z)), with one reciprocal for both: 1 / a = b / (a b).
// The multi-function unit (two exponentials and one reciprocal, 16 lanes per SM and clock) is what
// bounds the activations. -z is capped at 60 ln 2 = 41.6 so that the product stays finite; there the
// logistic is under 1e-18 and taken as zero (a value left over would be multiplied by z, which has no bound, in
// the activation and in its slope). Relative error: the exponent's rounding, up to 2^-24 |z| (2.5e-6 at the cap, 2.4e-7
// at |z| = 4), and a few 2^-23 of the two units, far below the BF16 rounding (2^-9) that follows.
__device__ __forceinline__ void logistic2(float z0, float z1, float& s0, float& s1) {
  float e0, e1, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(fminf(z0 * -1.4426950408889634f, 60.f)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(fminf(z1 * -1.4426950408889634f, 60.f)));
  const float a = 1.f + e0, b = 1.f + e1;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a * b));
  s0 = z0 > -41.58f ? r * b : 0.f;
  s1 = z1 > -41.58f ? r * a : 0.f;
}
__device__ __forceinline__ unsigned bf2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}

// ---------------------------------------------------------------------------
// Inference on the 5th-generation tensor cores (tcgen05, sm_100-class): tiles of
// 128 points, one TMEM lane (one thread of the 4 warps) per point. Operands are
// BF16 in shared memory in the K-major layout without swizzle: 8 x 8 core
// matrices of 128 contiguous bytes (row r of a core matrix at 16 r bytes), core
// matrices adjacent along K 128 bytes apart (the leading-dimension offset) and
// row groups of 8 rows K/8 * 128 bytes apart (the stride offset). One thread
// issues the MMAs of a layer (K = 16 per instruction, FP32 accumulation in TMEM)
// and commits them to an mbarrier; then every thread reads its row of the
// accumulator (tcgen05.ld), adds the bias, applies SiLU and writes the BF16 row
// of the next layer's A operand.
//   layer 1: D1 (TMEM columns 0..63)   = X (128 x 16) . W1 (16 x 64)
//   layer 2: D2 (TMEM columns 64..127) = H1 (128 x 64) . W2 (64 x 64)
//   layer 3: D3 (TMEM columns 0..15)   = H2 (128 x 64) . W3 (64 x 16, columns >= 6 zero)
// ---------------------------------------------------------------------------
constexpr int TC_M = 128, TC_THREADS = 128, TC_TMEM_COLS = 128;
// shared memory: A operands X (4 KB), H1, H2 (16 KB each); the image of the forward weights; then the
// mbarriers: of the products, and of what is left of them when a wait gave up
constexpr int TC_X = 0, TC_H1 = TC_X + 128 * 16 * 2, TC_H2 = TC_H1 + 128 * 64 * 2, TC_W = TC_H2 + 128 * 64 * 2,
              TC_BAR = TC_W + IMG_FWD, TC_DRAIN = TC_BAR + 8, TC_SMEM = TC_BAR + 16;
constexpr unsigned long long TC_WAIT_NS = 1000000000ull;  // 1 s bound on every mbarrier wait
// the network's error words: a wait gave up (any kernel); one of a training pass did, whose sums are not
// valid; the Adam steps that were not taken since
enum { ERR_ANY = 0, ERR_TRAIN = 1, ERR_SKIPPED = 2, ERR_WORDS = 3 };

// shared-memory matrix descriptor: start address, leading (K) and stride (row-group)
// byte offsets, the fixed version bits 46-47 = 1, no swizzle
__device__ __forceinline__ unsigned long long tc_desc(unsigned saddr, unsigned lbo, unsigned sbo) {
  return (unsigned long long)((saddr & 0x3FFFF) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
         ((unsigned long long)(sbo >> 4) << 32) | (1ull << 46);
}
// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, M x N; both K-major, or both
// MN-major (mn = 1: the contraction runs over the rows of the stored operands)
__host__ __device__ constexpr unsigned tc_idesc(int M, int N, int mn = 0) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)mn << 15) | ((unsigned)mn << 16) | ((unsigned)(N >> 3) << 17) |
         ((unsigned)(M >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(unsigned dt, unsigned long long ad, unsigned long long bd, unsigned idesc,
                                       int acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dt),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
// waits for the phase `parity` of the mbarrier; false if it did not complete within TC_WAIT_NS
__device__ __forceinline__ bool tc_wait(unsigned bar, unsigned parity) {
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
    else if (t - t0 > TC_WAIT_NS) return false;
  }
}
// A wait gave up (the whole block calls this): waits, with the same limit, for every product that thread 0 has issued,
// so that none is under way when the TMEM columns and the shared memory are given back.
__device__ __forceinline__ void tc_drain(unsigned drain) {
  if (threadIdx.x == 0) tc_commit(drain);
  tc_wait(drain, 0);
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld16(unsigned taddr, float (&v)[16]) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// bias + SiLU of this thread's 64 accumulator columns at TMEM column c0, written as the
// thread's BF16 row of a K = 64 A operand at `dst`
__device__ __forceinline__ void tc_hidden(unsigned trow, int c0, const float* __restrict__ bias, unsigned char* dst,
                                          int row) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float v[16];
    tc_ld16(trow + c0 + 16 * q, v);
    unsigned o[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float z0 = v[2 * i] + bias[16 * q + 2 * i], z1 = v[2 * i + 1] + bias[16 * q + 2 * i + 1];
      float s0, s1;
      logistic2(z0, z1, s0, s1);
      o[i] = bf2(z0 * s0, z1 * s1);
    }
    // two 8-element core-matrix rows of 16 bytes
    *reinterpret_cast<uint4*>(dst + tc_off(row, 16 * q, 64)) = make_uint4(o[0], o[1], o[2], o[3]);
    *reinterpret_cast<uint4*>(dst + tc_off(row, 16 * q + 8, 64)) = make_uint4(o[4], o[5], o[6], o[7]);
  }
}

__global__ void __launch_bounds__(TC_THREADS) k_mlp_tc(const float* __restrict__ prm,
                                                       const unsigned char* __restrict__ img,
                                                       const float* __restrict__ X, int P, float* __restrict__ Y,
                                                       int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  __shared__ unsigned s_taddr;
  __shared__ float s_b[2 * NH + 16];  // b1, b2, b3
  const int t = threadIdx.x, warp = t >> 5;
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(tsm);
  const unsigned bar = sbase + TC_BAR, drain = sbase + TC_DRAIN;
  for (int i = t; i < IMG_FWD / 16; i += TC_THREADS)
    reinterpret_cast<uint4*>(tsm + TC_W)[i] = reinterpret_cast<const uint4*>(img)[i];
  for (int i = t; i < 2 * NH + 16; i += TC_THREADS)
    s_b[i] = i < NH ? prm[O_B1 + i] : (i < 2 * NH ? prm[O_B2 + i - NH] : (i - 2 * NH < NOUT ? prm[O_B3 + i - 2 * NH] : 0.f));
  if (t == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(drain) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(&s_taddr)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  proxy_fence();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = s_taddr;
  const unsigned trow = tmem + ((unsigned)(32 * warp) << 16);  // this warp's 32 lanes
  const unsigned long long dW1 = tc_desc(sbase + TC_W + IMG_W1, 128, 2 * 128);
  const unsigned long long dW2 = tc_desc(sbase + TC_W + IMG_W2, 128, 8 * 128);
  const unsigned long long dW3 = tc_desc(sbase + TC_W + IMG_W3, 128, 8 * 128);
  const unsigned long long dX = tc_desc(sbase + TC_X, 128, 2 * 128);
  const unsigned long long dH1 = tc_desc(sbase + TC_H1, 128, 8 * 128);
  const unsigned long long dH2 = tc_desc(sbase + TC_H2, 128, 8 * 128);
  constexpr unsigned ID64 = tc_idesc(128, 64), ID16 = tc_idesc(128, 16);
  constexpr unsigned long long KSTEP = (2 * 128) >> 4;  // descriptor start address step of K = 16
  unsigned phase = 0;
  bool ok = true;
  const int ntiles = (P + TC_M - 1) / TC_M;
  for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const int p = tile * TC_M + t;
    {  // A operand of layer 1: the standardised features of point p, BF16, features >= 10 zero
      __align__(16) bf o[16];
#pragma unroll
      for (int f = 0; f < 16; ++f) {
        float v = 0.f;
        if (f < NIN && p < P) v = (X[(size_t)f * P + p] - prm[O_INSH + f]) * prm[O_INSC + f];
        o[f] = __float2bfloat16(v);
      }
      *reinterpret_cast<uint4*>(tsm + TC_X + tc_off(t, 0, 16)) = *reinterpret_cast<const uint4*>(o);
      *reinterpret_cast<uint4*>(tsm + TC_X + tc_off(t, 8, 16)) = *reinterpret_cast<const uint4*>(o + 8);
    }
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
      tc_mma(tmem, dX, dW1, ID64, 0);
      tc_commit(bar);
    }
    // every thread takes the same barriers whatever its waits returned; the block leaves
    // the loop together at the end of the tile (__syncthreads_and)
    ok = tc_wait(bar, phase) && ok;
    phase ^= 1;
    tc_fence_after();
    tc_hidden(trow, 0, s_b, tsm + TC_H1, t);
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) tc_mma(tmem + 64, dH1 + kk * KSTEP, dW2 + kk * KSTEP, ID64, kk);
      tc_commit(bar);
    }
    ok = tc_wait(bar, phase) && ok;
    phase ^= 1;
    tc_fence_after();
    tc_hidden(trow, 64, s_b + NH, tsm + TC_H2, t);
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) tc_mma(tmem, dH2 + kk * KSTEP, dW3 + kk * KSTEP, ID16, kk);
      tc_commit(bar);
    }
    ok = tc_wait(bar, phase) && ok;
    phase ^= 1;
    tc_fence_after();
    {
      float v[16];
      tc_ld16(trow, v);
      if (p < P) {
#pragma unroll
        for (int c = 0; c < NOUT; ++c) Y[(size_t)c * P + p] = (v[c] + s_b[2 * NH + c]) * prm[O_OUTSC + c] + prm[O_OUTSH + c];
      }
    }
    tc_fence_before();
    ok = __syncthreads_and(ok);  // shared operands and TMEM columns are free for the next tile
    tc_fence_after();
  }
  if (!ok) {  // the same for the whole block
    if (t == 0) atomicExch(err + ERR_ANY, 1);
    tc_drain(drain);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS) : "memory");
}

// ---------------------------------------------------------------------------
// Training pass: loss and gradient sums of the block's tiles of 128 points, all products on the tensor
// cores. 8 warps: warp w reads the TMEM lanes (points) of quarter w & 3 and the columns of half
// w >> 2. Per tile the scratch columns T take D1, D2, Y, dH2 and dH1 in turn; the slopes of the
// activations stay in registers, so an activation costs one logistic for both directions. The
// weight gradients contract over the points, i.e. over the rows of the operands that the other
// products already have in shared memory, read as MN-major operands:
//   columns 64 .. 143  (128 x 80) = [H1 | H2]^T [dZ2 | dY]: gW2 in rows < 64, gW3 in the last 16 columns
//   columns 144 .. 159 (128 x 16) = [dZ1 | dZ2]^T X:        gW1^T in rows < 64
// (the other blocks of these products are not read). They accumulate in TMEM over the block's tiles.
// Bias gradients are FP32 sums of the unrounded dZ. Each block leaves its sums in its row of
// `part`; k_reduce adds the rows in order, so the gradient is the same from run to run.
// Bound by latency (five dependent products a tile) and instruction issue; 65536 points, one call
// with its read-back 247 -> 54 us against warp-level products on 16-point tiles with shared-memory
// atomics; a training step (k_mlp_train and k_reduce) 226 -> 30 us, 262144 points 820 -> 63 us.
// ---------------------------------------------------------------------------
constexpr int TR_THREADS = 256, TR_TMEM_COLS = 256, TR_T = 0, TR_GW = 64, TR_G1 = 144;
constexpr int TR_EG = 18;  // groups of 8 columns of the array dZ1 (64) | dZ2 (64) | dY (16)
constexpr int TR_X = 0, TR_H = TR_X + 128 * 16 * 2, TR_E = TR_H + 128 * 128 * 2, TR_W = TR_E + 128 * TR_EG * 16,
              TR_BAR = TR_W + IMG_BYTES, TR_DRAIN = TR_BAR + 8, TR_SMEM = TR_BAR + 16;
constexpr int PART = 5264;  // floats of a row of partial sums: NTRAIN gradients, the loss, padding

// sums over the warp's 32 lanes of v[i], i < 32: lane l returns the sum of v[l]
__device__ __forceinline__ float warp_column_sums(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float mine = up ? v[i + o] : v[i], theirs = up ? v[i] : v[i + o];
      v[i] = mine + __shfl_xor_sync(0xffffffffu, theirs, o);
    }
  }
  return v[0];
}

__global__ void __launch_bounds__(TR_THREADS, 2) k_mlp_train(const float* __restrict__ prm,
                                                             const unsigned char* __restrict__ img,
                                                             const float* __restrict__ X, const float* __restrict__ T,
                                                             int P, float* __restrict__ part, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char tsm[];
  __shared__ unsigned s_taddr;
  __shared__ float s_b[2 * NH + 16];           // b1, b2, b3
  __shared__ float s_io[4][16];                // in_shift, in_scale, 1 / out_scale, out_shift
  __shared__ float s_sum[4][2 * NH + 16];      // per quarter: gb1, gb2, gb3 and the loss
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, q = warp & 3, hf = warp >> 2, row = 32 * q + lane;
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(tsm);
  const unsigned bar = sbase + TR_BAR, drain = sbase + TR_DRAIN;
  for (int i = t; i < IMG_BYTES / 16; i += TR_THREADS)
    reinterpret_cast<uint4*>(tsm + TR_W)[i] = reinterpret_cast<const uint4*>(img)[i];
  if (t < 2 * NH + 16)
    s_b[t] = t < NH ? prm[O_B1 + t] : (t < 2 * NH ? prm[O_B2 + t - NH] : (t - 2 * NH < NOUT ? prm[O_B3 + t - 2 * NH] : 0.f));
  if (t < 16) {
    s_io[0][t] = t < NIN ? prm[O_INSH + t] : 0.f;
    s_io[1][t] = t < NIN ? prm[O_INSC + t] : 0.f;
    s_io[2][t] = t < NOUT ? prm[O_OUTSC + t] : 1.f;
    s_io[3][t] = t < NOUT ? prm[O_OUTSH + t] : 0.f;
  }
  if (t == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(drain) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(&s_taddr)),
                 "r"(TR_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  proxy_fence();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem = s_taddr, trow = tmem + ((unsigned)(32 * q) << 16);
  // A and B operands of the products over columns (K-major; rows of 8 points HS or ES bytes apart) ...
  constexpr unsigned HS = 16 * 128, ES = TR_EG * 128;
  const unsigned long long dX = tc_desc(sbase + TR_X, 128, 256), dW1 = tc_desc(sbase + TR_W + IMG_W1, 128, 256);
  const unsigned long long dH1 = tc_desc(sbase + TR_H, 128, HS), dH2 = tc_desc(sbase + TR_H + 8 * 128, 128, HS);
  const unsigned long long dW2 = tc_desc(sbase + TR_W + IMG_W2, 128, 1024), dW3 = tc_desc(sbase + TR_W + IMG_W3, 128, 1024);
  const unsigned long long dDY = tc_desc(sbase + TR_E + 16 * 128, 128, ES), dDZ2 = tc_desc(sbase + TR_E + 8 * 128, 128, ES);
  const unsigned long long dW2B = tc_desc(sbase + TR_W + IMG_W2B, 128, 1024), dW3B = tc_desc(sbase + TR_W + IMG_W3B, 128, 256);
  // ... and over points (MN-major: 8 columns 128 bytes apart, 8 points HS, ES or 256 bytes apart)
  const unsigned long long tH = tc_desc(sbase + TR_H, HS, 128), tE = tc_desc(sbase + TR_E, ES, 128),
                           tE2 = tc_desc(sbase + TR_E + 8 * 128, ES, 128), tX = tc_desc(sbase + TR_X, 256, 128);
  constexpr unsigned ID64 = tc_idesc(128, 64), ID16 = tc_idesc(128, 16), IDGW = tc_idesc(128, 80, 1), IDG1 = tc_idesc(128, 16, 1);
  constexpr unsigned long long KSTEP = 256 >> 4;  // descriptor step of 16 columns
  unsigned phase = 0;
  bool ok = true;
  float loss = 0.f, gb1 = 0.f, gb2 = 0.f, gb3[NOUT] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  const float inv = 2.f / ((float)P * (float)NOUT);
  const int ntiles = (P + 127) / 128;
  int done = 0;  // tiles of this block whose weight gradients are under way
  auto publish = [&] {  // shared-memory operands written: visible to the tensor core
    proxy_fence();
    tc_fence_before();
    __syncthreads();
  };
  auto wait = [&] {
    ok = tc_wait(bar, phase) && ok;
    phase ^= 1;
    tc_fence_after();
  };
  // z = accumulator + bias of this thread's 32 units, h = SiLU(z) as BF16 into the columns c0 .. of H, slope into ds
  auto hidden = [&](const float* bias, int c0, float (&ds)[32]) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      float v[16];
      tc_ld16(trow + TR_T + 32 * hf + 16 * g, v);
      unsigned o[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float z0 = v[2 * i] + bias[16 * g + 2 * i], z1 = v[2 * i + 1] + bias[16 * g + 2 * i + 1];
        float s0, s1;
        logistic2(z0, z1, s0, s1);
        o[i] = bf2(z0 * s0, z1 * s1);
        ds[16 * g + 2 * i] = s0 * (1.f + z0 * (1.f - s0));
        ds[16 * g + 2 * i + 1] = s1 * (1.f + z1 * (1.f - s1));
      }
      *reinterpret_cast<uint4*>(tsm + TR_H + tc_off(row, c0 + 16 * g, 128)) = make_uint4(o[0], o[1], o[2], o[3]);
      *reinterpret_cast<uint4*>(tsm + TR_H + tc_off(row, c0 + 16 * g + 8, 128)) = make_uint4(o[4], o[5], o[6], o[7]);
    }
  };
  // dZ = accumulator * slope (into ds), as BF16 into the columns c0 .. of E; returns the bias gradient of unit `lane`
  auto slope = [&](int c0, float (&ds)[32]) {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      float v[16];
      tc_ld16(trow + TR_T + 32 * hf + 16 * g, v);
      unsigned o[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        ds[16 * g + 2 * i] *= v[2 * i];
        ds[16 * g + 2 * i + 1] *= v[2 * i + 1];
        o[i] = bf2(ds[16 * g + 2 * i], ds[16 * g + 2 * i + 1]);
      }
      *reinterpret_cast<uint4*>(tsm + TR_E + tc_off(row, c0 + 16 * g, 8 * TR_EG)) = make_uint4(o[0], o[1], o[2], o[3]);
      *reinterpret_cast<uint4*>(tsm + TR_E + tc_off(row, c0 + 16 * g + 8, 8 * TR_EG)) = make_uint4(o[4], o[5], o[6], o[7]);
    }
  };
  for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const int p = tile * 128 + row;
    float x[8], tn[NOUT];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int f = 8 * hf + i;
      x[i] = (f < NIN && p < P) ? (X[(size_t)f * P + p] - s_io[0][f]) * s_io[1][f] : 0.f;
    }
    if (hf == 0)
#pragma unroll
      for (int c = 0; c < NOUT; ++c) tn[c] = p < P ? (T[(size_t)c * P + p] - s_io[3][c]) / s_io[2][c] : 0.f;
    if (done > 0) wait();  // the operands of the tile before are free
    *reinterpret_cast<uint4*>(tsm + TR_X + tc_off(row, 8 * hf, 16)) =
        make_uint4(bf2(x[0], x[1]), bf2(x[2], x[3]), bf2(x[4], x[5]), bf2(x[6], x[7]));
    publish();
    if (t == 0) {
      tc_fence_after();
      tc_mma(tmem + TR_T, dX, dW1, ID64, 0);
      tc_commit(bar);
    }
    wait();
    float ds1[32], ds2[32];
    hidden(s_b + 32 * hf, 32 * hf, ds1);
    publish();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < 4; ++k) tc_mma(tmem + TR_T, dH1 + k * KSTEP, dW2 + k * KSTEP, ID64, k);
      tc_commit(bar);
    }
    wait();
    hidden(s_b + NH + 32 * hf, NH + 32 * hf, ds2);
    publish();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < 4; ++k) tc_mma(tmem + TR_T, dH2 + k * KSTEP, dW3 + k * KSTEP, ID16, k);
      tc_commit(bar);
    }
    wait();
    if (hf == 0) {  // dY = 2 (y - t) / (6 P)
      float v[16], d[8];
      tc_ld16(trow + TR_T, v);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        d[c] = 0.f;
        if (c < NOUT && p < P) {
          const float e = v[c] + s_b[2 * NH + c] - tn[c < NOUT ? c : 0];
          loss += e * e;
          d[c] = inv * e;
          gb3[c < NOUT ? c : 0] += d[c];
        }
      }
      *reinterpret_cast<uint4*>(tsm + TR_E + tc_off(row, 128, 8 * TR_EG)) =
          make_uint4(bf2(d[0], d[1]), bf2(d[2], d[3]), bf2(d[4], d[5]), bf2(d[6], d[7]));
      *reinterpret_cast<uint4*>(tsm + TR_E + tc_off(row, 136, 8 * TR_EG)) = make_uint4(0u, 0u, 0u, 0u);
    }
    publish();
    if (t == 0) {
      tc_fence_after();
      tc_mma(tmem + TR_T, dDY, dW3B, ID64, 0);
      tc_commit(bar);
    }
    wait();
    slope(NH + 32 * hf, ds2);
    publish();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < 4; ++k) tc_mma(tmem + TR_T, dDZ2 + k * KSTEP, dW2B + k * KSTEP, ID64, k);
      tc_commit(bar);
#pragma unroll
      for (int k = 0; k < 8; ++k)  // 16 points a step
        tc_mma(tmem + TR_GW, tH + k * (2 * HS >> 4), tE2 + k * (2 * ES >> 4), IDGW, done > 0 || k > 0);
    }
    gb2 += warp_column_sums(ds2, lane);
    wait();
    slope(32 * hf, ds1);
    publish();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int k = 0; k < 8; ++k) tc_mma(tmem + TR_G1, tE + k * (2 * ES >> 4), tX + k * (512 >> 4), IDG1, done > 0 || k > 0);
      tc_commit(bar);
    }
    gb1 += warp_column_sums(ds1, lane);
    ++done;
    ok = __syncthreads_and(ok);  // the block leaves the loop together
  }
  if (done > 0) wait();
  ok = __syncthreads_and(ok);
  if (!ok) tc_drain(drain);
  // the block's sums: weights from TMEM, biases and loss through shared memory
  s_sum[q][32 * hf + lane] = gb1;
  s_sum[q][NH + 32 * hf + lane] = gb2;
  if (hf == 0) {
    for (int o = 16; o > 0; o >>= 1) {
      loss += __shfl_xor_sync(0xffffffffu, loss, o);
#pragma unroll
      for (int c = 0; c < NOUT; ++c) gb3[c] += __shfl_xor_sync(0xffffffffu, gb3[c], o);
    }
    if (lane == 0) {
#pragma unroll
      for (int c = 0; c < NOUT; ++c) s_sum[q][2 * NH + c] = gb3[c];
      s_sum[q][2 * NH + NOUT] = loss;
    }
  }
  float* out = part + (size_t)blockIdx.x * PART;
  if (q < 2) {  // rows < 64 of both products
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      float v[16];
      tc_ld16(trow + TR_GW + 32 * hf + 16 * g, v);
      float4* d = reinterpret_cast<float4*>(out + (O_W2 - TRAIN_BEGIN) + row * NH + 32 * hf + 16 * g);
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
    if (hf == 0) {
      float v[16];
      tc_ld16(trow + TR_G1, v);
#pragma unroll
      for (int f = 0; f < NIN; ++f) out[(O_W1 - TRAIN_BEGIN) + f * NH + row] = v[f];
    }
  } else if (hf == 0) {
    float v[16];
    tc_ld16(trow + TR_GW + NH, v);
#pragma unroll
    for (int c = 0; c < NOUT; ++c) out[(O_W3 - TRAIN_BEGIN) + (row - 64) * NOUT + c] = v[c];
  }
  if (!ok && t == 0) {
    atomicExch(err + ERR_ANY, 1);
    atomicExch(err + ERR_TRAIN, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (t < 2 * NH + NOUT + 1) {
    const float s = s_sum[0][t] + s_sum[1][t] + s_sum[2][t] + s_sum[3][t];
    const int at = t < NH ? O_B1 + t : (t < 2 * NH ? O_B2 + t - NH : O_B3 + t - 2 * NH);  // the loss follows b3
    out[at - TRAIN_BEGIN] = s;
  }
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TR_TMEM_COLS) : "memory");
}

// The blocks' rows of partial sums added in order: gradients and loss into gsum (and, for the host, the
// error flag behind them); ADAM: one Adam step on the trainable range (moments m, v; bias
// corrections c1, c2) and the changed weights into the image. No step is taken on the sums of a training
// pass that gave up, nor after it until that has been reported.
// 32 columns a block, 8 threads each on every eighth row.
constexpr int RED_COLS = 32, RED_ROWS = 8;
template <bool ADAM>
__global__ void __launch_bounds__(RED_COLS * RED_ROWS) k_reduce(const float* __restrict__ part, int rows,
                                                                float* __restrict__ gsum, float* __restrict__ prm,
                                                                float* __restrict__ m, float* __restrict__ v,
                                                                unsigned char* __restrict__ img, int* __restrict__ err,
                                                                float lr, float b1, float b2, float eps, float c1, float c2) {
  __shared__ float red[RED_ROWS][RED_COLS];
  const int x = threadIdx.x % RED_COLS, y = threadIdx.x / RED_COLS, j = blockIdx.x * RED_COLS + x;
  float s = 0.f;
  if (j <= NTRAIN) {
#pragma unroll 8
    for (int r = y; r < rows; r += RED_ROWS) s += part[(size_t)r * PART + j];
  }
  red[y][x] = s;
  __syncthreads();
  if (y != 0 || j > NTRAIN) return;
  float g = 0.f;
#pragma unroll
  for (int r = 0; r < RED_ROWS; ++r) g += red[r][x];
  if (j == NTRAIN) {
    gsum[NPARAM] = g;
    gsum[NPARAM + 1] = (float)err[ERR_ANY];
    if (ADAM && err[ERR_TRAIN]) ++err[ERR_SKIPPED];
    return;
  }
  const int i = TRAIN_BEGIN + j;
  if constexpr (ADAM) {
    if (err[ERR_TRAIN]) return;
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float w = prm[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    prm[i] = w;
    pack_param(i, w, img);
  } else {
    gsum[i] = g;
  }
}

}  // namespace

struct dns_mlp {
  float* prm = nullptr;   // NPARAM (device)
  float* gsum = nullptr;  // NPARAM + 2 (device): gradient sums, the loss sum, the error flag; zeros where nothing is trained
  float* host = nullptr;  // NPARAM + 2 (pinned): where a call reads them back
  float* part = nullptr;  // partial sums of the training blocks (device)
  float* m = nullptr;
  float* v = nullptr;
  unsigned char* img = nullptr;  // the BF16 weights as the kernels' operands (device)
  int* err = nullptr;  // ERR_WORDS (device): tensor-core waits that gave up
  int t = 0;           // Adam steps taken
};

namespace {

int mlp_fail(int code, const char* msg) {
  dns::set_error_message(msg);
  return code;
}

#define MLP_CUDA(call, where)                      \
  do {                                             \
    cudaError_t e_ = (call);                       \
    if (e_ != cudaSuccess) return mlp_fail(DNS_ERR_CUDA, where); \
  } while (0)

int mlp_sms() {
  static const int sms = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      n = 148;
    return n;
  }();
  return sms;
}

// grid of a kernel with `per_sm` blocks on an SM, each walking tiles of 128 points: four inference blocks
// (4 x 128 TMEM columns fill an SM's 512), two training blocks (2 x 256)
constexpr int TC_PER_SM = 4, TR_PER_SM = 2;
int mlp_blocks(int P, int per_sm) {
  const int tiles = (P + TC_M - 1) / TC_M;
  return tiles < per_sm * mlp_sms() ? (tiles < 1 ? 1 : tiles) : per_sm * mlp_sms();
}

int mlp_run_grad(dns_mlp* net, const float* X, const float* T, int P, cudaStream_t st) {
  k_mlp_train<<<mlp_blocks(P, TR_PER_SM), TR_THREADS, TR_SMEM, st>>>(net->prm, net->img, X, T, P, net->part, net->err);
  MLP_CUDA(cudaGetLastError(), "dns_mlp: training kernel launch");
  return DNS_OK;
}
template <bool ADAM>
int mlp_reduce(dns_mlp* n, int P, float lr, float b1, float b2, float c1, float c2, cudaStream_t st) {
  k_reduce<ADAM><<<(NTRAIN + RED_COLS) / RED_COLS, RED_COLS * RED_ROWS, 0, st>>>(
      n->part, mlp_blocks(P, TR_PER_SM), n->gsum, n->prm, n->m, n->v, n->img, n->err, lr, b1, b2, 1e-8f, c1, c2);
  MLP_CUDA(cudaGetLastError(), "dns_mlp: reduction launch");
  return DNS_OK;
}

// Mean and unbiased standard deviation of each feature row of X (10 x P) and each
// stress row of T (6 x P), in FP64, written into the normalisation entries of the
// parameter vector: in_shift = mean, in_scale = 1/std (1 where std <= 1e-12),
// out_scale = std (1 where std <= 1e-30), out_shift = mean. One block per row.
constexpr int NORM_THREADS = 256;
__global__ void __launch_bounds__(NORM_THREADS) k_norm(float* __restrict__ prm, const float* __restrict__ X,
                                                       const float* __restrict__ T, int P) {
  const int r = blockIdx.x;
  const float* row = r < NIN ? X + (size_t)r * P : T + (size_t)(r - NIN) * P;
  __shared__ double red[NORM_THREADS / 32];
  __shared__ double s_mean;
  auto block_sum = [&](double v) -> double {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < NORM_THREADS / 32; ++w) t += red[w];
    return t;
  };
  double s = 0.0;
  for (int i = threadIdx.x; i < P; i += NORM_THREADS) s += (double)row[i];
  const double tot = block_sum(s);
  if (threadIdx.x == 0) s_mean = tot / (double)P;
  __syncthreads();
  const double mean = s_mean;
  double q = 0.0;
  for (int i = threadIdx.x; i < P; i += NORM_THREADS) {
    const double d = (double)row[i] - mean;
    q += d * d;
  }
  const double ss = block_sum(q);
  if (threadIdx.x == 0) {
    const double sd = P > 1 ? sqrt(ss / (double)(P - 1)) : 0.0;
    if (r < NIN) {
      prm[O_INSH + r] = (float)mean;
      prm[O_INSC + r] = sd > 1e-12 ? (float)(1.0 / sd) : 1.f;
    } else {
      prm[O_OUTSC + r - NIN] = sd > 1e-30 ? (float)sd : 1.f;
      prm[O_OUTSH + r - NIN] = (float)mean;
    }
  }
}

// Reports (and clears) a tensor-core wait that gave up, the Adam steps that it prevented uncounted; synchronises.
int mlp_check_err(dns_mlp* n, const char* where) {
  int err[ERR_WORDS] = {};
  MLP_CUDA(cudaMemcpy(err, n->err, sizeof(err), cudaMemcpyDeviceToHost), where);
  if (!err[ERR_ANY]) return DNS_OK;
  n->t -= err[ERR_SKIPPED];
  MLP_CUDA(cudaMemset(n->err, 0, sizeof(err)), where);
  return mlp_fail(DNS_ERR_TIMEOUT, "dns_mlp: a kernel's tensor-core wait gave up after 1 s; its output is not valid");
}

}  // namespace

namespace dns {
cudaError_t mlp_forward_async(::dns_mlp* n, const float* X, float* Y, int P, cudaStream_t st) {
  k_mlp_tc<<<mlp_blocks(P, TC_PER_SM), TC_THREADS, TC_SMEM, st>>>(n->prm, n->img, X, P, Y, n->err);
  return cudaGetLastError();
}
}  // namespace dns

extern "C" {

int dns_mlp_set_normalisation(dns_mlp* n, const float* X, const float* T, int P, void* stream) {
  if (!n || !X || !T || P < 2) return mlp_fail(DNS_ERR_ARG, "dns_mlp_set_normalisation: bad arguments");
  k_norm<<<NIN + NOUT, NORM_THREADS, 0, (cudaStream_t)stream>>>(n->prm, X, T, P);
  MLP_CUDA(cudaGetLastError(), "dns_mlp_set_normalisation launch");
  return DNS_OK;
}

int dns_mlp_param_count(void) { return NPARAM; }

int dns_mlp_create(dns_mlp** out) {
  if (!out) return mlp_fail(DNS_ERR_ARG, "dns_mlp_create: out is NULL");
  *out = nullptr;
  dns_mlp* n = new dns_mlp();
  cudaError_t e = cudaMalloc(&n->prm, NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&n->gsum, (NPARAM + 2) * sizeof(float));
  if (e == cudaSuccess) e = cudaMallocHost(&n->host, (NPARAM + 2) * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&n->part, (size_t)TR_PER_SM * mlp_sms() * PART * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&n->m, NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&n->v, NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&n->img, IMG_BYTES);
  if (e == cudaSuccess) e = cudaMemset(n->img, 0, IMG_BYTES);
  if (e == cudaSuccess) e = cudaMalloc(&n->err, ERR_WORDS * sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(n->err, 0, ERR_WORDS * sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(n->prm, 0, NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->gsum, 0, (NPARAM + 2) * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, NPARAM * sizeof(float));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, TR_SMEM);
  if (e != cudaSuccess) {
    dns_mlp_destroy(n);
    cudaGetLastError();
    return mlp_fail(e == cudaErrorMemoryAllocation ? DNS_ERR_OOM : DNS_ERR_CUDA, "dns_mlp_create: device set-up failed");
  }
  *out = n;
  return DNS_OK;
}

int dns_mlp_destroy(dns_mlp* n) {
  if (!n) return DNS_OK;
  cudaFree(n->prm);
  cudaFree(n->gsum);
  cudaFree(n->m);
  cudaFree(n->v);
  cudaFree(n->img);
  cudaFree(n->part);
  if (n->host) cudaFreeHost(n->host);
  cudaFree(n->err);
  delete n;
  return DNS_OK;
}

int dns_mlp_set_params(dns_mlp* n, const float* host, int count) {
  if (!n || !host || count != NPARAM) return mlp_fail(DNS_ERR_ARG, "dns_mlp_set_params: need 5286 host floats");
  MLP_CUDA(cudaMemcpy(n->prm, host, NPARAM * sizeof(float), cudaMemcpyHostToDevice), "dns_mlp_set_params copy");
  MLP_CUDA(cudaMemset(n->m, 0, NPARAM * sizeof(float)), "dns_mlp_set_params");
  MLP_CUDA(cudaMemset(n->v, 0, NPARAM * sizeof(float)), "dns_mlp_set_params");
  n->t = 0;
  MLP_CUDA(cudaMemset(n->err + ERR_TRAIN, 0, (ERR_WORDS - ERR_TRAIN) * sizeof(int)), "dns_mlp_set_params");
  k_pack<<<16, 256>>>(n->prm, n->img);
  MLP_CUDA(cudaGetLastError(), "dns_mlp_set_params pack");
  MLP_CUDA(cudaDeviceSynchronize(), "dns_mlp_set_params");
  return DNS_OK;
}

int dns_mlp_get_params(dns_mlp* n, float* host, int count) {
  if (!n || !host || count != NPARAM) return mlp_fail(DNS_ERR_ARG, "dns_mlp_get_params: need 5286 host floats");
  MLP_CUDA(cudaDeviceSynchronize(), "dns_mlp_get_params");
  MLP_CUDA(cudaMemcpy(host, n->prm, NPARAM * sizeof(float), cudaMemcpyDeviceToHost), "dns_mlp_get_params copy");
  return mlp_check_err(n, "dns_mlp_get_params");
}

int dns_mlp_debug_give_up(dns_mlp* n) {
  if (!n) return mlp_fail(DNS_ERR_ARG, "dns_mlp_debug_give_up: net is NULL");
  const int err[2] = {1, 1};  // ERR_ANY, ERR_TRAIN
  MLP_CUDA(cudaMemcpy(n->err, err, sizeof(err), cudaMemcpyHostToDevice), "dns_mlp_debug_give_up");
  return DNS_OK;
}

int dns_mlp_forward(dns_mlp* n, const float* X, float* Y, int P, void* stream) {
  if (!n || !X || !Y || P < 1) return mlp_fail(DNS_ERR_ARG, "dns_mlp_forward: bad arguments");
  k_mlp_tc<<<mlp_blocks(P, TC_PER_SM), TC_THREADS, TC_SMEM, (cudaStream_t)stream>>>(n->prm, n->img, X, P, Y, n->err);
  MLP_CUDA(cudaGetLastError(), "dns_mlp_forward launch");
  return DNS_OK;
}

int dns_mlp_loss_grad(dns_mlp* n, const float* X, const float* T, int P, float* grad_host, float* loss_host,
                      void* stream) {
  if (!n || !X || !T || P < 1) return mlp_fail(DNS_ERR_ARG, "dns_mlp_loss_grad: bad arguments");
  cudaStream_t st = (cudaStream_t)stream;
  int rc = mlp_run_grad(n, X, T, P, st);
  if (rc) return rc;
  if ((rc = mlp_reduce<false>(n, P, 0.f, 0.f, 0.f, 1.f, 1.f, st))) return rc;
  MLP_CUDA(cudaMemcpyAsync(n->host, n->gsum, (NPARAM + 2) * sizeof(float), cudaMemcpyDeviceToHost, st),
           "dns_mlp_loss_grad copy");
  MLP_CUDA(cudaStreamSynchronize(st), "dns_mlp_loss_grad");
  if (n->host[NPARAM + 1] != 0.f) return mlp_check_err(n, "dns_mlp_loss_grad");
  if (grad_host) memcpy(grad_host, n->host, NPARAM * sizeof(float));
  if (loss_host) *loss_host = n->host[NPARAM] / ((float)P * (float)NOUT);
  return DNS_OK;
}

int dns_mlp_train_step(dns_mlp* n, const float* X, const float* T, int P, double lr, float* loss_host, void* stream) {
  if (!n || !X || !T || P < 1 || !(lr > 0.0)) return mlp_fail(DNS_ERR_ARG, "dns_mlp_train_step: bad arguments");
  cudaStream_t st = (cudaStream_t)stream;
  int rc = mlp_run_grad(n, X, T, P, st);
  if (rc) return rc;
  n->t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)n->t), c2 = 1.f - std::pow(b2, (float)n->t);
  if ((rc = mlp_reduce<true>(n, P, (float)lr, b1, b2, c1, c2, st))) return rc;
  if (loss_host) {
    MLP_CUDA(cudaMemcpyAsync(n->host + NPARAM, n->gsum + NPARAM, 2 * sizeof(float), cudaMemcpyDeviceToHost, st),
             "dns_mlp_train_step loss copy");
    MLP_CUDA(cudaStreamSynchronize(st), "dns_mlp_train_step");
    if (n->host[NPARAM + 1] != 0.f) return mlp_check_err(n, "dns_mlp_train_step");
    *loss_host = n->host[NPARAM] / ((float)P * (float)NOUT);
  }
  return DNS_OK;
}

}  // extern "C"
