// M2L on CUDA cores (Eq. m2l with the truncated derivative tensors of Sec. 2.2):
//   L~_n(A) += sum_m M~_m(B) h_B^|m| h_A^(|n|+1) D_{n+m}(R),   R = z_A - z_B',
// evaluated per pair in units of r = |R|:  D_c(R) = r^-(|c|+1) D^_c(R / r), so
//   L~_n(A) += u^(|n|+1) sum_m (v^|m| M~_m(B)) D^_{n+m}(R^),  u = h_A / r, v = h_B / r,
// with |R^| = 1 and u, v <= theta: every factor is O(1) or smaller for any pair
// of levels.  The body forms D'_c = u^(|c|+1) D^_c once per c and takes the
// source coefficients as (v/u)^|m| M~_m, so each term u^(|n|+1) v^|m| D^ M~ is
// one FMA (u >= 2^-17 at the depth cap, so u^(p+1) and (v/u)^p stay in range).  D^ is the derivative tensor of erfc(x r^ / 2) / r^ at r^ = 1,
// x = r / r_s, from the radial prefactors f_(k) = ((1/r) d/dr)^k psi (or of the
// polynomial truncation 1/r - P(r) of Sec. 5 with split 1; radial_prefactors):
//   D^_c = sum_{k_d <= c_d/2} prod_d [c_d! / (2^k_d k_d! (c_d - 2k_d)!)] R^_d^(c_d-2k_d) f_(|c|-|k|).
//
// One lane per (sink, source) pair; a warp walks the pairs of one sink (lists
// are grouped by sink), keeps its partial local expansion in registers and
// reduces it across the warp at the end (through shared memory, in a fixed
// order, one addition per coefficient: the result is deterministic).  Each launch
// adds into L (one launch per order).  The expansion order is a template parameter:
// all index arithmetic is literal in the generated straight-line bodies
// (gen_bodies.py -> gen_bodies.cuh).  For p >= 7 the output coefficients are split
// over G warps (slice g owns the outputs with index = g mod G) and the
// scaled source multipoles of each lane's pair are staged in shared memory.
#include <algorithm>

#include "common.cuh"
#include "gen_bodies.cuh"

namespace hfmm {
namespace {

// Normalised prefactors f^_k = r^(2k+1) f_(k)(r), k = 0..P, of the kernel of
// split S: S = 0 the Gaussian erfc(x/2)/r with x = r / r_s (the recurrence
// f^_(k+1) = -(2k+1) f^_k + (-1)^(k+1) x^(2k+1) e^(-x^2/4) / (2^k sqrt(pi)));
// S = 1 the polynomial truncation 1/r - P(r) with w = r / R_c:
// f^_0 = 1 - w (15 - 10 w^2 + 3 w^4) / 8, f^_1 = -1 + w^3 (5 - 3 w^2) / 2,
// f^_2 = 3 - 3 w^5 and the Newtonian (-1)^k (2k-1)!! beyond.
template <int P, int S>
__device__ __forceinline__ void radial_prefactors(float x, float (&f)[P + 1]) {
  if constexpr (S == 1) {
    const float w = x, w2 = w * w;
    f[0] = 1.f - w * (15.f - 10.f * w2 + 3.f * w2 * w2) * 0.125f;
    if constexpr (P >= 1) f[1] = -1.f + w2 * w * (5.f - 3.f * w2) * 0.5f;
    if constexpr (P >= 2) f[2] = 3.f - 3.f * w2 * w2 * w;
    float dk = 3.f;  // |f^_k| = (2k - 1)!!
#pragma unroll
    for (int q = 3; q <= P; ++q) {
      dk *= (float)(2 * q - 1);
      f[q] = (q & 1) ? -dk : dk;
    }
  } else {
    const float kInvSqrtPi = 0.56418958354775628f;
    f[0] = erfcf(0.5f * x);
    float tk = -x * kInvSqrtPi * __expf(-0.25f * x * x);
    const float hx2 = 0.5f * x * x;
#pragma unroll
    for (int q = 0; q < P; ++q) {
      f[q + 1] = -(float)(2 * q + 1) * f[q] + tk;
      tk = -tk * hx2;
    }
  }
}

template <int P, int G, int g, int S>
__device__ __forceinline__ void m2l_sink(uint32_t k, uint32_t tb, uint32_t te, const uint4 *__restrict__ cell,
                                         const uint64_t *__restrict__ lst, const float *__restrict__ M,
                                         float *__restrict__ L, int ldm, float inv_rs, float *__restrict__ wsm) {
  constexpr int NC = ncoef(P);
  constexpr int NS = (NC + G - 1) / G;
  const int lane = threadIdx.x & 31;
  const uint4 ca = cell[k];
  float acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.f;
  for (uint32_t t = tb + lane; t < te; t += 32) {
    const uint64_t e = lst[t];
    const uint32_t b = pair_src(e), sh = pair_shift(e);
    const uint4 cb = cell[b];
    int64_t dd[3];
    half_delta(ca, cb, sh, dd);
    // R = z_A - z_B' in half units (exact integers below 2^24)
    const float Rx = -(float)dd[0], Ry = -(float)dd[1], Rz = -(float)dd[2];
    const float r2 = Rx * Rx + Ry * Ry + Rz * Rz;
    const float rinv = rsqrtf(r2);
    const float x = r2 * rinv * inv_rs;  // r / r_s (S = 0) or r / R_c (S = 1)
    const float u = (float)(2 * half_width(ca.w)) * rinv;
    const float v = (float)half_width(cb.w) / (float)half_width(ca.w);  // v/u = h_B / h_A (exact)
    float f[P + 1];
    radial_prefactors<P, S>(x, f);
    float U[P + 1];
    U[0] = u;
#pragma unroll
    for (int q = 1; q <= P; ++q) U[q] = U[q - 1] * u;
    const float *Mb = M + (size_t)b * ldm;
    float *col = wsm + lane;
    M2LLoad<P>::template run<32>(Mb, v, col);
    M2LBody<P, G, g>::run(Rx * rinv, Ry * rinv, Rz * rinv, f, U, col, acc);
  }
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    float a = acc[s];
#pragma unroll
    for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    const int n = s * G + g;
    if (lane == 0 && n < NC) L[(size_t)k * ldm + n] += a;
  }
}

// resident blocks of 128 threads per SM the register budget allows without
// spilling, by order (measured with -Xptxas -v: p <= 4 at 128, p = 5 at 168 registers)
template <int P>
constexpr int m2l_min_blocks() { return P <= 4 ? 4 : P == 5 ? 3 : 2; }

template <int P, int G, int S>
__global__ void __launch_bounds__(128, m2l_min_blocks<P>()) k_m2l_sliced(int64_t nn, const uint4 *__restrict__ cell,
                                             const uint32_t *__restrict__ beg, const uint32_t *__restrict__ end,
                                             const uint64_t *__restrict__ lst, const float *__restrict__ M,
                                             float *__restrict__ L, int ldm, float inv_rs,
                                             const TreeState *tz) {
  extern __shared__ float sm[];
  nn = tree_nodes(tz, nn);  // graph mode: the node count from the device tree state
  static_assert(M2LSlices<P>::kSmem, "orders 7 and 8");
  float *wsm = sm + (threadIdx.x >> 5) * ncoef(P) * 32;  // per warp: the staged multipoles
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); w < nn * G; w += nw) {
    const uint32_t k = (uint32_t)(w / G);
    const int g = (int)(w % G);
    const uint32_t tb = beg[k], te = end[k];
    if (tb == te) continue;
    if constexpr (G == 2) {
      if (g == 0) m2l_sink<P, 2, 0, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm);
      else m2l_sink<P, 2, 1, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm);
    } else {
      static_assert(G == 8, "slices");
      switch (g) {
        case 0: m2l_sink<P, 8, 0, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        case 1: m2l_sink<P, 8, 1, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        case 2: m2l_sink<P, 8, 2, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        case 3: m2l_sink<P, 8, 3, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        case 4: m2l_sink<P, 8, 4, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        case 5: m2l_sink<P, 8, 5, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        case 6: m2l_sink<P, 8, 6, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
        default: m2l_sink<P, 8, 7, S>(k, tb, te, cell, lst, M, L, ldm, inv_rs, wsm); break;
      }
    }
  }
}

// Orders 1..6, either tree: one warp per sink, 32 pairs a batch.  At 254 registers eight
// warps an SM are all there is to hide a load behind, and with the chain bounds -> entry ->
// node in the loop a third of the warps' time went on it: while one batch is computed the
// next one's nodes and the list entries of the one after are copied to shared memory
// (cp.async), across sinks too.  20.4M pairs, p = 6 (2M clustered particles): 1.86 -> 1.74 ms,
// 1.58 with the derivative tensors by recurrence (gen_bodies.py); bound by issue (65% with
// under two warps a scheduler), half of it the contraction's 924 FMA.  The multipole rows
// stay loads from the lanes: copied ahead as well, 1.92 (cp.async.ca), 2.2 (.cg, twice the
// L2 sectors) or 3.2 ms (row by row: 38% more instructions).
//
// What the kernel needs of a tree's nodes: the staged record of a source or a sink, R = z_A
// - z_B' in units of half_width or of length, and the scales h.
struct OctM2L {
  const uint4 *cell;
  float inv_rs;  // r / r_s (Gaussian) or r / R_c (polynomial) for r in half units
  using Staged = uint4;
  __device__ __forceinline__ void stage(uint32_t dst, uint32_t k) const { cp16(dst, cell + k); }
  static __device__ __forceinline__ void cp16(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
  // R, h_A (in R's unit) and h_B / h_A (exact)
  __device__ __forceinline__ void pair(const Staged &a, const Staged &b, uint32_t s, float (&R)[3], float &hA,
                                       float &rho) const {
    int dd[3];
    half_delta32(a, b, s, dd);  // exact integers below 2^24
#pragma unroll
    for (int d = 0; d < 3; ++d) R[d] = -(float)dd[d];
    hA = (float)(2 * half_width(a.w));
    rho = (float)half_width(b.w) / (float)half_width(a.w);
  }
};
// k-d tree: R formed in FP64 from the box centres, the scales h powers of two.
struct KdM2L {
  const double *geo;  // [>= 3][cap], the centres first
  const float *hs;
  int64_t cap;
  double box;
  float inv_rs;
  struct Staged {
    double c[3];
    float h, pad;
  };
  __device__ __forceinline__ void stage(uint32_t dst, uint32_t k) const {
#pragma unroll
    for (int d = 0; d < 3; ++d)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 8 * d), "l"(geo + d * cap + k) : "memory");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 24), "l"(hs + k) : "memory");
  }
  __device__ __forceinline__ void pair(const Staged &a, const Staged &b, uint32_t s, float (&R)[3], float &hA,
                                       float &rho) const {
#pragma unroll
    for (int d = 0; d < 3; ++d)
      R[d] = (float)__dsub_rn(a.c[d], __dadd_rn(b.c[d], (double)shift_component(s, d) * box));
    hA = a.h;
    rho = b.h / a.h;
  }
};

// A warp's shared memory.
template <int P, class Nodes>
struct alignas(16) M2LStage {
  typename Nodes::Staged src[32], sink;
  uint64_t e[2][32];              // list entries, batch by batch in turn
  float red[32 * (ncoef(P) + 1)];  // the reduction's transpose
};

template <int P, int S, class Nodes>
__global__ void __launch_bounds__(128, m2l_min_blocks<P>())
    k_m2l(int64_t nn, Nodes nodes, const uint32_t *__restrict__ beg, const uint32_t *__restrict__ end,
          const uint64_t *__restrict__ lst, const float *__restrict__ M, float *__restrict__ L, int ldm,
          const TreeState *tz) {
  constexpr int NC = ncoef(P);
  static_assert(M2LSlices<P>::G == 1 && !M2LSlices<P>::kSmem, "orders 1..6");
  using Stage = M2LStage<P, Nodes>;
  extern __shared__ __align__(16) unsigned char m2l_smem[];
  nn = tree_nodes(tz, nn);  // graph mode: the node count from the device tree state
  Stage &W = reinterpret_cast<Stage *>(m2l_smem)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5);
  // batches in order: the one computed (a), the one whose rows are in flight (b), the one
  // whose entries are (c); k >= nn: none.  next: the sink after c's, its bounds already read
  struct Batch {
    uint32_t k, t, te;
  } a, b, c, next;
  auto bounds = [&](uint32_t k) {
    next.k = k;
    next.t = next.te = 0;
    if (k < nn) {
      next.t = beg[k];
      next.te = end[k];
    }
  };
  auto advance = [&]() {  // c to the batch after it
    if (c.te - c.t > 32) {
      c.t += 32;
      return;
    }
    while (next.t == next.te && next.k < nn) bounds(next.k + nw);
    c = next;
    if (next.k < nn) bounds(next.k + nw);
  };
  auto shared32 = [](const void *p) { return (uint32_t)__cvta_generic_to_shared(p); };
  int slot = 0;  // of b's entries
  auto stage_entries = [&](int sl) {  // c's entries
    if (c.k < nn && c.t + lane < c.te)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(shared32(&W.e[sl][lane])), "l"(lst + c.t + lane)
                   : "memory");
  };
  auto stage_rows = [&]() {  // b's rows and nodes, by its entries
    if (b.k >= nn) return;
    if (b.t + lane < b.te) nodes.stage(shared32(&W.src[lane]), pair_src(W.e[slot][lane]));
    if (lane == 0) nodes.stage(shared32(&W.sink), b.k);
  };
  bounds(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  c.t = c.te = 0;
  advance();  // the first batch
  stage_entries(0);
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  b = c;
  stage_rows();
  advance();
  stage_entries(1);
  asm volatile("cp.async.commit_group;" ::: "memory");
  float acc[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) acc[s] = 0.f;
  while (b.k < nn) {
    a = b;
    b = c;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    const bool valid = a.t + lane < a.te;
    float R[3] = {1.f, 0.f, 0.f}, hA = 1.f, rho = 1.f;
    uint32_t src = 0;
    if (valid) {
      const uint64_t e = W.e[slot][lane];
      src = pair_src(e);
      nodes.pair(W.sink, W.src[lane], pair_shift(e), R, hA, rho);
    }
    __syncwarp();
    slot ^= 1;
    stage_rows();
    advance();
    stage_entries(slot ^ 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (valid) {
      const float r2 = R[0] * R[0] + R[1] * R[1] + R[2] * R[2];
      const float rinv = rsqrtf(r2);
      float f[P + 1];
      radial_prefactors<P, S>(r2 * rinv * nodes.inv_rs, f);
      float U[P + 1];
      U[0] = hA * rinv;
#pragma unroll
      for (int q = 1; q <= P; ++q) U[q] = U[q - 1] * U[0];
      float Mp[NC];
      M2LLoad<P>::template run<1>(M + (size_t)src * ldm, rho, Mp);
      M2LBody<P, 1, 0>::run(R[0] * rinv, R[1] * rinv, R[2] * rinv, f, U, Mp, acc);
    }
    if (b.k == a.k) continue;  // more of this sink
    // sum over the lanes by a transpose in shared memory: each lane writes its
    // partial row (stride NC + 1: no bank conflicts), then lane c adds column c
    // over the 32 rows in lane order (deterministic) and adds it to the sink's local
    // (no other warp does: the reduction needs no answer)
#pragma unroll
    for (int s = 0; s < NC; ++s) {
      W.red[lane * (NC + 1) + s] = acc[s];
      acc[s] = 0.f;
    }
    __syncwarp();
    for (int cix = lane; cix < NC; cix += 32) {
      float sum = 0.f;
#pragma unroll 8
      for (int m = 0; m < 32; ++m) sum += W.red[m * (NC + 1) + cix];
      atomicAdd(L + (size_t)a.k * ldm + cix, sum);
    }
    __syncwarp();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int P, int S, class Nodes>
cudaError_t launch(Ctx &c, const Nodes &nodes, DBuf &from, cudaStream_t st) {
  // four sinks a warp, so that its copies overlap its arithmetic (262k clustered particles:
  // 0.156 ms instead of 0.163 with one), one while that leaves the GPU's blocks unfilled
  const unsigned all = blocks_for((size_t)c.nnodes, 4);
  const unsigned cap = 152u * (unsigned)(c.prm.tile_m2l_blocks > 0 ? c.prm.tile_m2l_blocks : 64);
  const unsigned g = std::min(cap, std::max(std::min(all, 304u), (all + 3u) / 4u));
  const size_t smem = 4 * sizeof(M2LStage<P, Nodes>);
  cudaError_t e = cudaFuncSetAttribute(k_m2l<P, S, Nodes>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_m2l<P, S, Nodes><<<g, 128, smem, st>>>(c.nnodes, nodes, hfmm::P<uint32_t>(from), hfmm::P<uint32_t>(c.m2l_end),
                                           hfmm::P<uint64_t>(c.m2l), hfmm::P<float>(c.M), hfmm::P<float>(c.L), c.ldm,
                                           c.graph_tree ? hfmm::P<TreeState>(c.tstate) : nullptr);
  note_launch();
  return cudaGetLastError();
}

template <int P, int S>
cudaError_t launch_sliced(Ctx &c, cudaStream_t st) {
  constexpr int G = M2LSlices<P>::G;
  unsigned g = blocks_for((size_t)c.nnodes * G, 4);
  const unsigned cap = 152u * (unsigned)(c.prm.tile_m2l_blocks > 0 ? c.prm.tile_m2l_blocks : 64);
  if (g > cap) g = cap;
  // r / r_s (Gaussian) or r / R_c (polynomial) with r in half units: x = r_half * (L / 2^22) / scale
  const float inv_rs = (float)(c.prm.box / (double)kHalfBox / (S == 1 ? c.rc : c.rs));
  const size_t smem = (size_t)4 * ncoef(P) * 32 * sizeof(float);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_m2l_sliced<P, G, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  // the entries [mid, end) of each sink: pairs outside the operator table
  k_m2l_sliced<P, G, S><<<g, 128, smem, st>>>(c.nnodes, hfmm::P<uint4>(c.cell), hfmm::P<uint32_t>(c.m2l_mid),
                                    hfmm::P<uint32_t>(c.m2l_end), hfmm::P<uint64_t>(c.m2l), hfmm::P<float>(c.M),
                                    hfmm::P<float>(c.L), c.ldm, inv_rs,
                                    c.graph_tree ? hfmm::P<TreeState>(c.tstate) : nullptr);
  note_launch();
  return cudaGetLastError();
}

template <int S>
cudaError_t run(Ctx &c, int q, cudaStream_t st) {
  if (c.prm.tree == 1) {
    const KdM2L nodes{P<double>(c.kd.geo), P<float>(c.kd.hs), c.kd.cap, c.prm.box,
                      (float)(1.0 / (S == 1 ? c.rc : c.rs))};
    switch (q) {
      case 1: return launch<1, S>(c, nodes, c.m2l_beg, st);
      case 2: return launch<2, S>(c, nodes, c.m2l_beg, st);
      case 3: return launch<3, S>(c, nodes, c.m2l_beg, st);
      case 4: return launch<4, S>(c, nodes, c.m2l_beg, st);
      case 5: return launch<5, S>(c, nodes, c.m2l_beg, st);
      case 6: return launch<6, S>(c, nodes, c.m2l_beg, st);
    }
    return cudaErrorInvalidValue;
  }
  // the entries [mid, end) of each sink: pairs outside the operator table
  const OctM2L nodes{P<uint4>(c.cell), (float)(c.prm.box / (double)kHalfBox / (S == 1 ? c.rc : c.rs))};
  switch (q) {
    case 1: return launch<1, S>(c, nodes, c.m2l_mid, st);
    case 2: return launch<2, S>(c, nodes, c.m2l_mid, st);
    case 3: return launch<3, S>(c, nodes, c.m2l_mid, st);
    case 4: return launch<4, S>(c, nodes, c.m2l_mid, st);
    case 5: return launch<5, S>(c, nodes, c.m2l_mid, st);
    case 6: return launch<6, S>(c, nodes, c.m2l_mid, st);
    case 7: return launch_sliced<7, S>(c, st);
    case 8: return launch_sliced<8, S>(c, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// Either tree's M2L pairs at order q.
cudaError_t m2l_pass(Ctx &c, int q, cudaStream_t st) {
  if (c.nm2l == 0 || c.nnodes == 0) return cudaSuccess;
  return c.prm.split == 1 ? run<1>(c, q, st) : run<0>(c, q, st);
}

}  // namespace hfmm
