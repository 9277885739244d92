// Inference and training kernels of the learned-acceptance network (mlp.cuh).
//  k_mlp_infer: tensor-core inference (mma.sync m16n8k16 BF16 -> FP32), one
//               warp per 16 rows; the same routine the traversal calls.
//  k_mlp_grad:  softmax cross-entropy forward + backward on mma.sync, tiles of
//               64 samples, BF16-rounded weights / inputs / activations with
//               FP32 sums and the rounding treated as identity in the backward
//               pass; per-block gradient partials (kept in registers).
//  k_mlp_reduce, k_mlp_adam: fixed-order reduction of the partials and an
//               Adam step on the FP32 master weights, writing the BF16 copy.
#include "mlp.cuh"

namespace hfmm {
namespace {

__global__ void __launch_bounds__(256) k_mlp_infer(const __nv_bfloat16 *__restrict__ w, const float *__restrict__ x,
                                                   int64_t n, float *__restrict__ logits, int *__restrict__ cls) {
  __shared__ uint32_t sw[kMlpSmemWords];
  __shared__ __align__(16) __nv_bfloat16 xs[8][16 * 16];
  mlp_stage(w, sw);
  __syncthreads();
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  __nv_bfloat16 *xr = xs[wp];
  const int64_t nwarp = (int64_t)gridDim.x * 8;
  for (int64_t base = ((int64_t)blockIdx.x * 8 + wp) * 16; base < n; base += nwarp * 16) {
    for (int i = lane; i < 256; i += 32) {
      const int r = i >> 4, c = i & 15;
      const int64_t row = base + r;
      xr[i] = __float2bfloat16_rn((c < kMlpIn && row < n) ? x[row * kMlpIn + c] : 0.f);
    }
    __syncwarp();
    float l[4];
    mlp_logits16(sw, xr, l);
    int c0, c8;
    mlp_argmax16(l, c0, c8);
    const int64_t r0 = base + g, r8 = base + g + 8;
    if (logits) {
      if (r0 < n) { logits[r0 * 8 + 2 * t] = l[0]; logits[r0 * 8 + 2 * t + 1] = l[1]; }
      if (r8 < n) { logits[r8 * 8 + 2 * t] = l[2]; logits[r8 * 8 + 2 * t + 1] = l[3]; }
    }
    if (cls && t == 0) {
      if (r0 < n) cls[r0] = c0;
      if (r8 < n) cls[r8] = c8;
    }
    __syncwarp();
  }
}

// ------------------------------------------------------------------ training
// Forward, softmax cross-entropy and backward as small GEMMs on mma.sync BF16
// (FP32 accumulation); a block of four warps takes tiles of 64 samples.
//
// What bounds it: the arithmetic, 31 kflop a sample, is a contraction, and at one
// warp a sample it was spent re-reading and re-rounding the weights for every
// product and adding every gradient term with a shared-memory float atomic (400k
// samples: 14.1 ms).  Here the weights stay in shared memory in fragment order,
// the activations stay in registers from layer to layer (the C fragments of one
// layer are the A fragments of the next), and each warp keeps 16 rows of every
// weight gradient in registers over all of its block's tiles, so there are no
// atomics and the result does not depend on scheduling.
//
// Precision: weights, inputs and activations are BF16 values, so the forward
// products are exact in FP32; their sums are not, and the tensor cores do not
// round a sum to nearest.  In the first layer that moved one activation in some
// 3e5 across a BF16 rounding boundary (2^-8 of it), and through it a second-layer
// pre-activation near zero across zero: the sample's rows of the gradient change,
// and in a quarter of the batches of 400k samples the gradient was 7e-7 to 1.5e-6
// from the FP64 one instead of at most 1.3e-7.  So the first layer is FP32 FMAs,
// the bias first and the inputs in order, and a second-layer sum too close to zero
// for its sign to be certain is formed again in the same way (gate_bound).
// The backward operands d = dLoss/dz are FP32; each is split exactly into three
// BF16 terms (8 + 8 + 8 significant bits), three MMAs whose products are again exact
// in FP32.  Chained over all of a block's tiles the gradients came out 2.4e-6 from
// the FP64 ones, so every MMA group sums 16 terms from zero, and the groups are
// added in FP32.
//
// The sample tile of 64 (16 rows a warp) keeps the staged operands within 76 KB,
// so that three blocks share an SM: 12 warps cover the latency of the staging.
// Measured (400k samples, gradient + Adam step): 14.3 -> 0.18 ms; 0.14 with the first
// layer on the tensor cores too.
constexpr int kGradThreads = 128;
constexpr int kGradTile = 64;
constexpr int kGradBlocks = 152 * 3;
constexpr int kLdH = 72, kLdX = 24, kLdO = 8;  // row strides (BF16): 16-byte rows, no bank conflicts
constexpr int kFragW2T = 4 * 8 * 2 * 32, kFragW3T = 8 * 32;
// dynamic shared memory: weight images (W1 as FP32), then the tile's operands
constexpr int kGradW1 = kMlpH * kMlpIn;
constexpr int kGradWords = (kMlpSmemWords + 3) / 4 * 4 + kFragW2T + kFragW3T + kGradW1;
constexpr size_t kGradSmem = (size_t)kGradWords * 4 + (size_t)kGradTile * (5 * kLdH + kLdX + 3 * kLdO) * 2;

// x = hi + mid + lo, each BF16 (exact for finite x above the denormal range), two values per word.
__device__ __forceinline__ void split3(float a, float b, uint32_t (&w)[3]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    w[q] = *reinterpret_cast<const uint32_t *>(&h);
    a -= __low2float(h);
    b -= __high2float(h);
  }
}

// Non-finite values of a packed pair replaced by zero: in a gradient product they only meet
// factors that are exactly zero (a unit with z > 0 false), whose terms are left out.
__device__ __forceinline__ uint32_t finite_or_zero(uint32_t w) {
  if ((w & 0x7f80u) == 0x7f80u) w &= 0xffff0000u;
  if ((w & 0x7f800000u) == 0x7f800000u) w &= 0x0000ffffu;
  return w;
}

__device__ __forceinline__ void mma_bf16_1688(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(b0));
}

// c += a b with the products summed from zero and added in FP32.
__device__ __forceinline__ void mma_add(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  float p[4] = {0.f, 0.f, 0.f, 0.f};
  mma_bf16_16816(p, a, b0, b1);
#pragma unroll
  for (int q = 0; q < 4; ++q) c[q] += p[q];
}

// How far from zero the sign of a row's second-layer sums is certain.  The terms'
// magnitudes add up to at most `terms` (the bias, and the largest activation times the
// largest sum of |w| over a unit); an MMA group of 16 that truncates every term to 24 bits
// below the largest is within 2^-19 of that, with the FP32 additions of the groups within
// 2^-18.  Some 3000 of a batch's 25.6M sums are closer.  With an infinite activation the sums
// are infinite or NaN however they are formed: they stay as they are.
__device__ __forceinline__ float gate_bound(float terms) {
  const float tol = 0x1p-18f * terms;
  return tol < 3e38f ? tol : -1.f;
}

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16 *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}

__device__ __forceinline__ void ldsm2t(uint32_t (&r)[2], const __nv_bfloat16 *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"((uint32_t)__cvta_generic_to_shared(p))
               : "memory");
}

__global__ void __launch_bounds__(kGradThreads, 3) k_mlp_grad(const float *__restrict__ wm, const float *__restrict__ x,
                                                              const int *__restrict__ labels,
                                                              const float *__restrict__ cw, int64_t n,
                                                              float *__restrict__ part, float *__restrict__ loss_part) {
  extern __shared__ __align__(16) uint32_t gsm[];
  __shared__ float lsum[4];
  uint32_t *sw = gsm, *w2t = gsm + (kMlpSmemWords + 3) / 4 * 4, *w3t = w2t + kFragW2T;
  float *w1 = reinterpret_cast<float *>(w3t + kFragW3T);
  __nv_bfloat16 *sh1 = reinterpret_cast<__nv_bfloat16 *>(gsm + kGradWords);
  __nv_bfloat16 *sh2 = sh1 + kGradTile * kLdH, *sd = sh2 + kGradTile * kLdH;  // sd: three terms of d2, then of d1
  __nv_bfloat16 *sx = sd + 3 * kGradTile * kLdH, *sd3 = sx + kGradTile * kLdX;
  mlp_stage(wm, sw);
  auto pkw = [&](int i0, int i1) { return pack_bf16(wm[i0], wm[i1]); };
  for (int i = threadIdx.x; i < kFragW2T; i += kGradThreads) {  // B of dh1 = d2 W2: [kt][nt][2][32], k = unit of layer 2
    const int l = i & 31, rr = (i >> 5) & 1, nt = (i >> 6) & 7, kt = i >> 9;
    const int u = kt * 16 + 2 * (l & 3) + 8 * rr, k = nt * 8 + (l >> 2);
    w2t[i] = pkw(kOffW2 + u * kMlpH + k, kOffW2 + (u + 1) * kMlpH + k);
  }
  for (int i = threadIdx.x; i < kFragW3T; i += kGradThreads) {  // B of dh2 = d3 W3: [nt][32], k = output
    const int l = i & 31, nt = i >> 5, o = 2 * (l & 3), k = nt * 8 + (l >> 2);
    w3t[i] = pkw(kOffW3 + o * kMlpH + k, kOffW3 + (o + 1) * kMlpH + k);
  }
  auto bf = [](float v) { return __bfloat162float(__float2bfloat16_rn(v)); };
  for (int i = threadIdx.x; i < kGradW1; i += kGradThreads) w1[i] = bf(wm[kOffW1 + i]);
  __syncthreads();
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const float *bias = reinterpret_cast<const float *>(sw + kFragL1 + kFragL2 + kFragL3);
  const uint32_t *s2 = sw + kFragL1, *s3 = s2 + kFragL2;
  const int r0 = 16 * wp + g, r8 = r0 + 8;  // this lane's rows of the tile
  float most_w = 0.f, most_b = 0.f;  // layer 2: the largest sum of |w| over a unit, the largest |bias|
#pragma unroll 1
  for (int nt = 0; nt < 8; ++nt) {  // unit 8 nt + g, its row over the quad's lanes
    float v = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t wv = s2[nt * 256 + 32 * j + lane];
      v += fabsf(__uint_as_float(wv << 16)) + fabsf(__uint_as_float(wv & 0xffff0000u));
    }
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    most_w = fmaxf(most_w, v);
    most_b = fmaxf(most_b, fabsf(bias[kMlpH + nt * 8 + g]));
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    most_w = fmaxf(most_w, __shfl_xor_sync(0xffffffffu, most_w, o));
    most_b = fmaxf(most_b, __shfl_xor_sync(0xffffffffu, most_b, o));
  }
  // lane addresses of the transposed fragment loads: rows are samples
  const int m = lane >> 3, r = lane & 7;
  const int a_s = (m >> 1) * 8 + r, a_u = (m & 1) * 8;  // A: [k = sample][row = unit]
  const int b_s = (m & 1) * 8 + r, b_n = (m >> 1) * 8;  // B: [k = sample][column]
  float gW2[8][4], gW1[2][4], gW3[4], gB2[4], gB3[4], loss = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    gW3[q] = gB2[q] = gB3[q] = 0.f;
    gW1[0][q] = gW1[1][q] = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) gW2[nt][q] = 0.f;
  }
  constexpr uint32_t kOnes = 0x3f803f80u;
  for (int64_t base = (int64_t)blockIdx.x * kGradTile; base < n; base += (int64_t)gridDim.x * kGradTile) {
    const int64_t i0 = base + r0, i8 = base + r8;
    const bool v0 = i0 < n, v8 = i8 < n;
    // inputs straight into A fragments (columns 2t, 2t + 1 and 2t + 8, 2t + 9 of rows g, g + 8)
    uint32_t a[4] = {0u, 0u, 0u, 0u};
    if (v0) {
      a[0] = pack_bf16(x[i0 * kMlpIn + 2 * t], x[i0 * kMlpIn + 2 * t + 1]);
      if (t < 2) a[2] = pack_bf16(x[i0 * kMlpIn + 8 + 2 * t], x[i0 * kMlpIn + 9 + 2 * t]);
    }
    if (v8) {
      a[1] = pack_bf16(x[i8 * kMlpIn + 2 * t], x[i8 * kMlpIn + 2 * t + 1]);
      if (t < 2) a[3] = pack_bf16(x[i8 * kMlpIn + 8 + 2 * t], x[i8 * kMlpIn + 9 + 2 * t]);
    }
    const int lab0 = v0 ? labels[i0] : -1, lab8 = v8 ? labels[i8] : -1;
    // (class weights cover the labels 0..7: another label has none)
    auto weight = [&](bool valid, int lab) {
      return !valid ? 0.f : !cw ? 1.f : (unsigned)lab < (unsigned)kMlpOut ? cw[lab] : 0.f;
    };
    const float wg0 = weight(v0, lab0), wg8 = weight(v8, lab8);
    {
      // the gradient's copy: column 12 is one, so that column of d1^T x is the bias gradient
      uint32_t *q0 = reinterpret_cast<uint32_t *>(sx + r0 * kLdX), *q8 = reinterpret_cast<uint32_t *>(sx + r8 * kLdX);
      q0[t] = finite_or_zero(a[0]);
      q8[t] = finite_or_zero(a[1]);
      q0[4 + t] = t == 2 ? 0x3f80u : finite_or_zero(a[2]);
      q8[4 + t] = t == 2 ? 0x3f80u : finite_or_zero(a[3]);
    }
    // ---- forward; bits of m1, m2: z > 0 by (n-tile, fragment element)
    uint32_t f[4][4], m1 = 0, m2 = 0;
    float tol0, tol8;  // of the rows' gates
    {
      float x0[kMlpIn], x8[kMlpIn];  // the whole rows, from the quad's lanes
      __nv_bfloat162 top0 = __float2bfloat162_rn(0.f), top8 = top0;  // the rows' largest activations
#pragma unroll
      for (int j = 0; j < kMlpIn / 2; ++j) {
        const uint32_t v0 = __shfl_sync(0xffffffffu, j < 4 ? a[0] : a[2], (lane & 28) + (j & 3));
        const uint32_t v8 = __shfl_sync(0xffffffffu, j < 4 ? a[1] : a[3], (lane & 28) + (j & 3));
        x0[2 * j] = __uint_as_float(v0 << 16);
        x0[2 * j + 1] = __uint_as_float(v0 & 0xffff0000u);
        x8[2 * j] = __uint_as_float(v8 << 16);
        x8[2 * j + 1] = __uint_as_float(v8 & 0xffff0000u);
      }
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        float c[4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int u = nt * 8 + 2 * t + e;
          const float4 *w4 = reinterpret_cast<const float4 *>(w1 + u * kMlpIn);
          c[e] = c[2 + e] = bias[u];
#pragma unroll
          for (int j = 0; j < kMlpIn / 4; ++j) {
            const float4 w = w4[j];
            c[e] = fmaf(w.x, x0[4 * j], c[e]);
            c[2 + e] = fmaf(w.x, x8[4 * j], c[2 + e]);
            c[e] = fmaf(w.y, x0[4 * j + 1], c[e]);
            c[2 + e] = fmaf(w.y, x8[4 * j + 1], c[2 + e]);
            c[e] = fmaf(w.z, x0[4 * j + 2], c[e]);
            c[2 + e] = fmaf(w.z, x8[4 * j + 2], c[2 + e]);
            c[e] = fmaf(w.w, x0[4 * j + 3], c[e]);
            c[2 + e] = fmaf(w.w, x8[4 * j + 3], c[2 + e]);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          m1 |= (c[q] > 0.f ? 1u : 0u) << (4 * nt + q);
          c[q] = fmaxf(c[q], 0.f);
        }
        const uint32_t lo = pack_bf16(c[0], c[1]), hi = pack_bf16(c[2], c[3]);
        f[nt >> 1][(nt & 1) * 2 + 0] = lo;
        f[nt >> 1][(nt & 1) * 2 + 1] = hi;
        top0 = __hmax2(top0, *reinterpret_cast<const __nv_bfloat162 *>(&lo));
        top8 = __hmax2(top8, *reinterpret_cast<const __nv_bfloat162 *>(&hi));
        reinterpret_cast<uint32_t *>(sh1 + r0 * kLdH)[nt * 4 + t] = finite_or_zero(lo);
        reinterpret_cast<uint32_t *>(sh1 + r8 * kLdH)[nt * 4 + t] = finite_or_zero(hi);
      }
      tol0 = fmaxf(__low2float(top0), __high2float(top0));
      tol8 = fmaxf(__low2float(top8), __high2float(top8));
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        tol0 = fmaxf(tol0, __shfl_xor_sync(0xffffffffu, tol0, o));
        tol8 = fmaxf(tol8, __shfl_xor_sync(0xffffffffu, tol8, o));
      }
      tol0 = gate_bound(fmaf(most_w, tol0, most_b));
      tol8 = gate_bound(fmaf(most_w, tol8, most_b));
      __syncwarp();  // a row of sh1 is its quad's
    }
    uint32_t h2[4][4], unsure = 0;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      float c[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) c[q] = bias[kMlpH + nt * 8 + 2 * t + (q & 1)];
#pragma unroll
      for (int kt = 0; kt < 4; ++kt)
        mma_add(c, f[kt], s2[((nt * 4 + kt) * 2 + 0) * 32 + lane], s2[((nt * 4 + kt) * 2 + 1) * 32 + lane]);
#pragma unroll
      for (int q = 0; q < 4; ++q) unsure |= (fabsf(c[q]) < (q < 2 ? tol0 : tol8) ? 1u : 0u) << (4 * nt + q);
#pragma unroll
      for (int q = 0; q < 4; ++q) m2 |= (c[q] > 0.f ? 1u : 0u) << (4 * nt + q);
      const uint32_t lo = pack_bf16(fmaxf(c[0], 0.f), fmaxf(c[1], 0.f));
      const uint32_t hi = pack_bf16(fmaxf(c[2], 0.f), fmaxf(c[3], 0.f));
      h2[nt >> 1][(nt & 1) * 2 + 0] = lo;
      h2[nt >> 1][(nt & 1) * 2 + 1] = hi;
      reinterpret_cast<uint32_t *>(sh2 + r0 * kLdH)[nt * 4 + t] = lo;
      reinterpret_cast<uint32_t *>(sh2 + r8 * kLdH)[nt * 4 + t] = hi;
    }
    while (unsure) {  // the sum again in FP32, the bias first and the inputs in order
      const int at = __ffs(unsure) - 1, nt = at >> 2, q = at & 3, u = nt * 8 + 2 * t + (q & 1), row = q < 2 ? r0 : r8;
      const uint32_t *h = reinterpret_cast<const uint32_t *>(sh1 + row * kLdH);
      const uint32_t *w = s2 + nt * 256 + (u & 7) * 4;  // the unit's row: inputs 8 j + 2 i, + 1 in word 32 j + i
      unsure &= unsure - 1u;
      float z = bias[kMlpH + u];
#pragma unroll 1
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t wv = w[32 * j + i], hv = h[4 * j + i];
          z = fmaf(__uint_as_float(wv << 16), __uint_as_float(hv << 16), z);
          z = fmaf(__uint_as_float(wv & 0xffff0000u), __uint_as_float(hv & 0xffff0000u), z);
        }
      m2 = (m2 & ~(1u << at)) | (z > 0.f ? 1u << at : 0u);
      uint32_t *pair = reinterpret_cast<uint32_t *>(sh2 + row * kLdH) + nt * 4 + t;
      const uint32_t other = *pair & ((q & 1) ? 0x0000ffffu : 0xffff0000u);
      *pair = other | ((q & 1) ? pack_bf16(0.f, fmaxf(z, 0.f)) : pack_bf16(fmaxf(z, 0.f), 0.f));
#pragma unroll
      for (int i = 0; i < 16; ++i) h2[i >> 2][i & 3] = i == at >> 1 ? *pair : h2[i >> 2][i & 3];
    }
    __syncwarp();
    const float b0 = bias[2 * kMlpH + 2 * t], b1 = bias[2 * kMlpH + 2 * t + 1];
    float z[4] = {b0, b1, b0, b1};
#pragma unroll
    for (int kt = 0; kt < 4; ++kt) mma_add(z, h2[kt], s3[(kt * 2 + 0) * 32 + lane], s3[(kt * 2 + 1) * 32 + lane]);
    // ---- softmax over the quad's 8 logits of each row, loss, d3 = weight (p - onehot)
    float mx0 = fmaxf(z[0], z[1]), mx8 = fmaxf(z[2], z[3]);
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
      mx8 = fmaxf(mx8, __shfl_xor_sync(0xffffffffu, mx8, o));
    }
    float p[4] = {__expf(z[0] - mx0), __expf(z[1] - mx0), __expf(z[2] - mx8), __expf(z[3] - mx8)};
    float se0 = p[0] + p[1], se8 = p[2] + p[3];
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      se0 += __shfl_xor_sync(0xffffffffu, se0, o);
      se8 += __shfl_xor_sync(0xffffffffu, se8, o);
    }
    uint32_t d3[3][2];
    {
      float d[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int lab = q < 2 ? lab0 : lab8, o = 2 * t + (q & 1);
        const float wg = q < 2 ? wg0 : wg8, pr = p[q] / (q < 2 ? se0 : se8);
        const bool valid = q < 2 ? v0 : v8;
        if (valid && o == lab) loss += -wg * __logf(fmaxf(pr, 1e-30f));
        if (valid && o == 0 && (lab < 0 || lab >= kMlpOut)) loss += -wg * __logf(1e-30f);
        d[q] = valid ? wg * (pr - (o == lab ? 1.f : 0.f)) : 0.f;
      }
      uint32_t w0[3], w8[3];
      split3(d[0], d[1], w0);
      split3(d[2], d[3], w8);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        d3[q][0] = w0[q];
        d3[q][1] = w8[q];
        reinterpret_cast<uint32_t *>(sd3 + (q * kGradTile + r0) * kLdO)[t] = w0[q];
        reinterpret_cast<uint32_t *>(sd3 + (q * kGradTile + r8) * kLdO)[t] = w8[q];
      }
    }
    // ---- d2 = (d3 W3) (z2 > 0)
    uint32_t d2[3][4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 2; q >= 0; --q) mma_bf16_1688(c, d3[q][0], d3[q][1], w3t[nt * 32 + lane]);
#pragma unroll
      for (int q = 0; q < 4; ++q) c[q] = (m2 >> (4 * nt + q)) & 1u ? c[q] : 0.f;
      uint32_t w0[3], w8[3];
      split3(c[0], c[1], w0);
      split3(c[2], c[3], w8);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        d2[q][nt >> 1][(nt & 1) * 2 + 0] = w0[q];
        d2[q][nt >> 1][(nt & 1) * 2 + 1] = w8[q];
        reinterpret_cast<uint32_t *>(sd + (q * kGradTile + r0) * kLdH)[nt * 4 + t] = w0[q];
        reinterpret_cast<uint32_t *>(sd + (q * kGradTile + r8) * kLdH)[nt * 4 + t] = w8[q];
      }
    }
    __syncthreads();
    // ---- dW2 = d2^T h1, dB2 = d2^T 1 (rows 16 wp ..), dW3^T = h2^T d3, dB3 = 1^T d3 (warp 0)
#pragma unroll
    for (int ks = 0; ks < kGradTile / 16; ++ks) {
      const int s0 = 16 * ks;
      uint32_t bh[4][4];
#pragma unroll
      for (int np = 0; np < 4; ++np) ldsm4t(bh[np], sh1 + (s0 + b_s) * kLdH + 16 * np + b_n);
      uint32_t ah[4], ad[3][4], bd[3][2];
      ldsm4t(ah, sh2 + (s0 + a_s) * kLdH + 16 * wp + a_u);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        ldsm4t(ad[q], sd + (q * kGradTile + s0 + a_s) * kLdH + 16 * wp + a_u);
        ldsm2t(bd[q], sd3 + (q * kGradTile + s0 + (lane & 15)) * kLdO);
      }
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 2; q >= 0; --q)
          mma_bf16_16816(c, ad[q], bh[nt >> 1][(nt & 1) * 2], bh[nt >> 1][(nt & 1) * 2 + 1]);
#pragma unroll
        for (int q = 0; q < 4; ++q) gW2[nt][q] += c[q];
      }
      float c2[4] = {0.f, 0.f, 0.f, 0.f}, c3[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 2; q >= 0; --q) {
        mma_bf16_16816(c2, ad[q], kOnes, kOnes);
        mma_bf16_16816(c3, ah, bd[q][0], bd[q][1]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        gB2[q] += c2[q];
        gW3[q] += c3[q];
      }
      if (wp == 0) {
        const uint32_t ones[4] = {kOnes, kOnes, kOnes, kOnes};
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 2; q >= 0; --q) mma_bf16_16816(c, ones, bd[q][0], bd[q][1]);
#pragma unroll
        for (int q = 0; q < 4; ++q) gB3[q] += c[q];
      }
    }
    __syncthreads();
    // ---- d1 = (d2 W2) (z1 > 0), over the rows of d2
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kt = 0; kt < 4; ++kt) {
        float p[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 2; q >= 0; --q)
          mma_bf16_16816(p, d2[q][kt], w2t[((kt * 8 + nt) * 2 + 0) * 32 + lane], w2t[((kt * 8 + nt) * 2 + 1) * 32 + lane]);
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] += p[q];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) c[q] = (m1 >> (4 * nt + q)) & 1u ? c[q] : 0.f;
      uint32_t w0[3], w8[3];
      split3(c[0], c[1], w0);
      split3(c[2], c[3], w8);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        reinterpret_cast<uint32_t *>(sd + (q * kGradTile + r0) * kLdH)[nt * 4 + t] = w0[q];
        reinterpret_cast<uint32_t *>(sd + (q * kGradTile + r8) * kLdH)[nt * 4 + t] = w8[q];
      }
    }
    __syncthreads();
    // ---- dW1 = d1^T x, dB1 in its column 12
#pragma unroll
    for (int ks = 0; ks < kGradTile / 16; ++ks) {
      const int s0 = 16 * ks;
      uint32_t bx[4];
      ldsm4t(bx, sx + (s0 + b_s) * kLdX + b_n);
      float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
      for (int q = 2; q >= 0; --q) {
        uint32_t ad[4];
        ldsm4t(ad, sd + (q * kGradTile + s0 + a_s) * kLdH + 16 * wp + a_u);
        mma_bf16_16816(c[0], ad, bx[0], bx[1]);
        mma_bf16_16816(c[1], ad, bx[2], bx[3]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        gW1[0][q] += c[0][q];
        gW1[1][q] += c[1][q];
      }
    }
    __syncthreads();  // the staged operands are rewritten by the next tile
  }
  // ---- the block's partial sums: rows 16 wp + g and + 8, columns 8 nt + 2t, + 1
  float *out = part + (size_t)blockIdx.x * kMlpW;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int row = (q < 2 ? r0 : r8), col = 2 * t + (q & 1);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) out[kOffW2 + row * kMlpH + 8 * nt + col] = gW2[nt][q];
    out[kOffW1 + row * kMlpIn + col] = gW1[0][q];
    if (8 + col < kMlpIn) out[kOffW1 + row * kMlpIn + 8 + col] = gW1[1][q];
    if (8 + col == kMlpIn) out[kOffB1 + row] = gW1[1][q];
    out[kOffW3 + col * kMlpH + row] = gW3[q];
    if (col == 0) out[kOffB2 + row] = gB2[q];
    if (row == 0) out[kOffB3 + col] = gB3[q];
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
  if (lane == 0) lsum[wp] = loss;
  __syncthreads();
  if (threadIdx.x == 0) loss_part[blockIdx.x] = lsum[0] + lsum[1] + lsum[2] + lsum[3];
}

// Sum of the blocks' partials: 32 weights a block, eight strided row groups each, added in a
// fixed order (one thread a weight walked all rows in series: 20 us for 304 rows).
__global__ void __launch_bounds__(256) k_mlp_reduce(const float *__restrict__ part, const float *__restrict__ loss_part,
                                                    int nb, float scale, float *__restrict__ grad,
                                                    float *__restrict__ loss) {
  __shared__ float s[8][32];
  const int c = threadIdx.x & 31, grp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + c;
  float v = 0.f;
  if (i < kMlpW)
    for (int b = grp; b < nb; b += 8) v += part[(size_t)b * kMlpW + i];
  s[grp][c] = v;
  __syncthreads();
  if (grp == 0 && i < kMlpW) {
    float a = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) a += s[q][c];
    grad[i] = a * scale;
  }
  if (blockIdx.x == 0 && grp == 1 && loss) {
    float a = 0.f;
    for (int b = c; b < nb; b += 32) a += loss_part[b];
#pragma unroll
    for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (c == 0) *loss = a * scale;
  }
}

__global__ void k_mlp_adam(float *__restrict__ wm, float *__restrict__ m1, float *__restrict__ m2,
                           const float *__restrict__ grad, float lr, float b1, float b2, float eps, float c1, float c2,
                           __nv_bfloat16 *__restrict__ wout) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kMlpW) return;
  const float gr = grad[i];
  const float a = b1 * m1[i] + (1.f - b1) * gr, b = b2 * m2[i] + (1.f - b2) * gr * gr;
  m1[i] = a;
  m2[i] = b;
  const float w = wm[i] - lr * (a / c1) / (sqrtf(b / c2) + eps);
  wm[i] = w;
  if (wout) wout[i] = __float2bfloat16_rn(w);
}

}  // namespace

cudaError_t mlp_infer(const void *w_bf16, const float *x, int64_t n, float *logits, int *cls, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  unsigned g = (unsigned)((n + 127) / 128);
  if (g > 152 * 8) g = 152 * 8;
  k_mlp_infer<<<g, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(w_bf16), x, n, logits, cls);
  note_launch();
  return cudaGetLastError();
}

size_t mlp_train_scratch_bytes() { return (size_t)kGradBlocks * (kMlpW + 1) * sizeof(float); }

cudaError_t mlp_grad(const float *wm, const float *x, const int *labels, const float *cw, int64_t n, float *grad,
                     float *loss, void *scratch, cudaStream_t st) {
  if (n <= 0) return cudaErrorInvalidValue;
  const int64_t tiles = (n + kGradTile - 1) / kGradTile;
  const int nb = (int)(tiles < kGradBlocks ? tiles : kGradBlocks);
  cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem);
  if (e != cudaSuccess) return e;
  float *part = static_cast<float *>(scratch);
  float *lp = part + (size_t)nb * kMlpW;
  k_mlp_grad<<<nb, kGradThreads, kGradSmem, st>>>(wm, x, labels, cw, n, part, lp);
  k_mlp_reduce<<<(kMlpW + 31) / 32, 256, 0, st>>>(part, lp, nb, 1.f / (float)n, grad, loss);
  note_launch(2);
  return cudaGetLastError();
}

cudaError_t mlp_adam(float *wm, float *m1, float *m2, const float *grad, float lr, int step, void *w_bf16,
                     cudaStream_t st) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_mlp_adam<<<(kMlpW + 255) / 256, 256, 0, st>>>(wm, m1, m2, grad, lr, b1, b2, eps, c1, c2,
                                                   static_cast<__nv_bfloat16 *>(w_bf16));
  note_launch();
  return cudaGetLastError();
}

}  // namespace hfmm
