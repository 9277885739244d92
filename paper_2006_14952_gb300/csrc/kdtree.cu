// ORB / k-d tree variant of the short-range FMM (tree = 1): the tree of Sec. 2.1
// (Fig. 1), an ORB tree with a leaf limiter whose cells hand their particles to
// two children of almost equal count, which Sec. 4 keeps as a k-d tree inside
// every domain.
//
// Build, level by level on the device:
//   - positions wrapped (x - L floor(x / L), as for the octree); for each axis d
//     the particle indices sorted once by (coordinate d, input index) with the
//     stable radix sort of order-preserving 64-bit keys;
//   - the shape of the tree follows from n and leaf_max alone (the counts of a level
//     are floor and ceil of n / 2^level; KdShape below): no scan, no read-back;
//   - a node reads its particles' bounding box from the first and last entries of
//     its range in the three orders; above leaf_max it splits on the axis of
//     largest extent (the lowest on a tie): the first floor(n / 2) particles of that
//     axis' order form the first child.  The orders are partitioned stably by the
//     particles' side, so every order stays sorted inside every node, and inside a
//     leaf the x order is the particle order (that of (x, input index)).  Nodes above
//     2048 particles: three kernels a level over all particles (k_kd_axis, k_kd_side,
//     k_kd_part); below, one block takes a node to its leaves (k_kd_subtree).
// A level over all particles is bound by its passes (a random byte a particle and order,
// two 4-byte streams an order, about 80 us at 2M); with nine launches a level to the
// leaves, its scans of 3 n flags and a node number a particle, the build of 2M particles
// (17 levels) took 2.45 ms; ten levels so and the rest in shared memory: 1.12 ms.  2048 is
// what a block's 48 KB hold (24 bytes a particle), four blocks an SM.
// Node geometry: the box centre c, half extents e, side (largest extent) in FP64,
// and the expansion scale h = L 2^-j >= side (j <= 21, the octree's deepest
// cell side): P2M offsets over h stay within [-1/2, 1/2] and the scale ratios of
// the translations are powers of two.
// Walk: one cooperative launch, sink-driven (k_kd_walk below): a warp takes one sink node
// and the sources its parent left open, the three rules of Sec. 2.3 on the boxes in FP64
// with every operation rounded on its own (no contraction, so the decisions are those of any
// IEEE FP64 evaluation in the same order), taken in FP32 wherever an error bound shows the
// FP32 comparison cannot differ; each sink's entries lie together in a fixed order, so every
// sum after them runs in a fixed order.  The same walk with the opening-angle test alone,
// from the root against itself, is the conventional FMM's of the interaction counts (Sec. 3).
// P2P: the octree's kernel (p2p.cu), the source-box offsets from the box centres.
#include <algorithm>

#include <cooperative_groups.h>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace hfmm {
namespace {

constexpr int kT = 256;

__global__ void k_kd_wrap(const double *__restrict__ pos, int64_t n, double box, double inv_pow2,
                          double *__restrict__ xw) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * n) return;
  xw[i] = wrap_box_fast(pos[i], box, inv_pow2);
}

// Order-preserving key of a double (negative values reversed below the positive ones).
__global__ void k_kd_keys(const double *__restrict__ x, int64_t n, uint64_t *__restrict__ key,
                          uint32_t *__restrict__ val) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t u = (uint64_t)__double_as_longlong(x[i]);
  key[i] = (u >> 63) ? ~u : (u | 0x8000000000000000ull);
  val[i] = (uint32_t)i;
}

// The shape of the tree: levels 0 .. depth are complete; on level `depth` the counts are
// q = floor(n / 2^depth) <= leaf_max and q + 1, and the `nsplit` nodes above leaf_max (q =
// leaf_max only) have the last level's nodes as children.  Node (l, j) of a complete level
// is number 2^l - 1 + j; with first(l, j) - j q of the nodes before it one larger than
// the others, the children of (depth, j) are numbers 2^(depth + 1) - 1 + 2 (first - j q) and + 1.
struct KdShape {
  int64_t n;
  int leaf_max, depth;
  int64_t q, nsplit;
  __host__ __device__ int64_t last_start() const { return ((int64_t)2 << depth) - 1; }
  __host__ __device__ int64_t nodes() const { return last_start() + 2 * nsplit; }
  __host__ __device__ int64_t leaves() const { return ((int64_t)1 << depth) + nsplit; }
};
KdShape kd_shape(int64_t n, int leaf_max) {
  KdShape s{n, leaf_max, 0, n, 0};
  while (s.q > leaf_max) {
    ++s.depth;
    s.q = n >> s.depth;
  }
  if (s.q == leaf_max) s.nsplit = n - (s.q << s.depth);
  return s;
}

// Particle range of node (l, j), j's bits from the top (0: first child).
__device__ __forceinline__ void kd_range(int64_t n, int l, uint32_t j, uint32_t &f, uint32_t &m) {
  f = 0;
  m = (uint32_t)n;
  for (int b = l - 1; b >= 0; --b) {
    const uint32_t h = m / 2;
    if ((j >> b) & 1u) {
      f += h;
      m -= h;
    } else {
      m = h;
    }
  }
}
// The node of level l that holds position i of the range [f, f + m): its number among
// them, and its range.
__device__ __forceinline__ uint32_t kd_find(uint32_t i, int l, uint32_t &f, uint32_t &m) {
  uint32_t j = 0;
  for (int b = 0; b < l; ++b) {
    const uint32_t h = m / 2;
    const uint32_t up = i - f >= h ? 1u : 0u;
    f += up ? h : 0u;
    m = up ? m - h : h;
    j = 2 * j + up;
  }
  return j;
}

// Ranges, children, parents and the leaf list.
__global__ void k_kd_topology(KdShape S, uint32_t *__restrict__ first, uint32_t *__restrict__ count,
                              int *__restrict__ child, int *__restrict__ parent, uint32_t *__restrict__ leaves) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= S.last_start()) return;
  const int l = 63 - __clzll((unsigned long long)k + 1);
  const uint32_t j = (uint32_t)(k + 1 - ((int64_t)1 << l));
  uint32_t f, m;
  kd_range(S.n, l, j, f, m);
  first[k] = f;
  count[k] = m;
  parent[k] = k == 0 ? -1 : (int)((k - 1) / 2);
  if (l < S.depth) {
    child[k] = (int)(2 * k + 1);
    return;
  }
  const int64_t larger = S.nsplit ? (int64_t)f - (int64_t)j * S.q : 0;  // nodes before this one that split
  if ((int64_t)m <= S.leaf_max) {
    child[k] = -1;
    leaves[j - larger] = (uint32_t)k;
    return;
  }
  const int64_t c = S.last_start() + 2 * larger;
  child[k] = (int)c;
  first[c] = f;
  count[c] = m / 2;
  first[c + 1] = f + m / 2;
  count[c + 1] = m - m / 2;
  const int64_t at = ((int64_t)1 << S.depth) - S.nsplit + 2 * larger;
  for (int e = 0; e < 2; ++e) {
    child[c + e] = -1;
    parent[c + e] = (int)k;
    leaves[at + e] = (uint32_t)(c + e);
  }
}

// Bounding box of the node over positions [f, f + m) of the three orders, and the axis of
// its largest extent (the lowest on a tie).
template <class Order>
__device__ __forceinline__ int kd_box(const double *__restrict__ xw, int64_t n, uint32_t f, uint32_t m, Order ord,
                                      double *__restrict__ box, int64_t cap, int64_t k) {
  double best = 0.0;
  int ax = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double a = xw[d * n + ord(d, f)], b = xw[d * n + ord(d, f + m - 1)];
    box[d * cap + k] = a;
    box[(3 + d) * cap + k] = b;
    const double ext = __dsub_rn(b, a);
    if (d == 0 || ext > best) {
      best = ext;
      ax = d;
    }
  }
  return ax;
}

struct KdOrders {
  const uint32_t *o[3];
};

// One complete level's nodes: box and split axis (every node of the level splits).
__global__ void k_kd_axis(int64_t n, int level, const double *__restrict__ xw, KdOrders O, double *__restrict__ box,
                          int64_t cap, int *__restrict__ axis) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ((int64_t)1 << level)) return;
  uint32_t f, m;
  kd_range(n, level, (uint32_t)j, f, m);
  const int64_t k = ((int64_t)1 << level) - 1 + j;
  axis[k] = kd_box(xw, n, f, m, [&](int d, uint32_t i) { return O.o[d][i]; }, box, cap, k);
}

// The side of every particle: in the second half of its node's range in the split axis' order.
__global__ void k_kd_side(int64_t n, int level, const int *__restrict__ axis, KdOrders O, uint8_t *__restrict__ side) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t f = 0, m = (uint32_t)n;
  const uint32_t j = kd_find((uint32_t)i, level, f, m);
  const int a = axis[((int64_t)1 << level) - 1 + j];
  side[a == 0 ? O.o[0][i] : a == 1 ? O.o[1][i] : O.o[2][i]] = (uint32_t)i - f >= m / 2 ? 1 : 0;
}

// Stable partition of the three orders inside every node of a level.  A particle of the
// second child is preceded in its node by r others of it: the tile's exclusive scan of the
// side flags, the flags of all tiles before (published counts, looked back over), less
// those of the nodes before, whose second children are known from the counts alone.
constexpr int kPartItems = 8, kPartTile = kT * kPartItems;
__global__ void __launch_bounds__(kT) k_kd_part(int64_t n, int level, KdOrders O, uint32_t *__restrict__ r0,
                                                uint32_t *__restrict__ r1, uint32_t *__restrict__ r2,
                                                const uint8_t *__restrict__ side, unsigned *__restrict__ ticket,
                                                volatile unsigned long long *look, unsigned ntiles,
                                                unsigned look_polls) {
  __shared__ uint32_t wsum[kT / 32];
  __shared__ unsigned tile_s;
  __shared__ unsigned long long before_s;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (tid == 0) tile_s = atomicAdd(ticket, 1u);
  __syncthreads();
  // tiles of the three orders in turn; the scan starts anew with each order
  const unsigned tile = tile_s, d = tile / ntiles, t = tile - d * ntiles;
  const uint32_t *ord = O.o[d];
  uint32_t *out = d == 0 ? r0 : d == 1 ? r1 : r2;
  const int64_t i0 = (int64_t)t * kPartTile + (int64_t)w * 32 * kPartItems + lane;
  uint32_t v[kPartItems], fl[kPartItems], ex[kPartItems], c = 0;
#pragma unroll
  for (int q = 0; q < kPartItems; ++q) v[q] = i0 + 32 * q < n ? ord[i0 + 32 * q] : 0u;
#pragma unroll
  for (int q = 0; q < kPartItems; ++q) fl[q] = i0 + 32 * q < n ? side[v[q]] : 0u;
#pragma unroll
  for (int q = 0; q < kPartItems; ++q) {
    const unsigned b = __ballot_sync(0xffffffffu, fl[q] != 0);
    ex[q] = c + (uint32_t)__popc(b & ((1u << lane) - 1u));
    c += (uint32_t)__popc(b);
  }
  if (lane == 0) wsum[w] = c;
  __syncthreads();
  uint32_t wb = 0, all = 0;
#pragma unroll
  for (int q = 0; q < kT / 32; ++q) {
    if (q < w) wb += wsum[q];
    all += wsum[q];
  }
  if (w == 0) {
    constexpr unsigned long long kAgg = 1ull << 62, kInc = 2ull << 62, kVal = kAgg - 1ull;
    if (lane == 0) look[tile] = (t == 0 ? kInc : kAgg) | all;
    // look back, 32 tiles at a time: up to the nearest published inclusive count
    unsigned long long before = 0;
    bool lost = look_polls == 0;
    for (long long at = (long long)t - 1; at >= 0 && !lost;) {
      unsigned long long x = kInc;  // before the order's first tile: nothing
      for (unsigned poll = 0;; ++poll) {
        if (at - lane >= 0) x = look[d * ntiles + (unsigned)(at - lane)];
        if (__all_sync(0xffffffffu, (x >> 62) != 0)) break;
        if (poll == look_polls) {
          lost = true;
          break;
        }
      }
      if (lost) break;
      const unsigned inc = __ballot_sync(0xffffffffu, (x >> 62) == 2);
      const int stop = inc ? __ffs(inc) - 1 : 31;
      unsigned long long s = lane <= stop ? (at - lane >= 0 ? x & kVal : 0ull) : 0ull;
#pragma unroll
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      before += s;
      if (inc) break;
      at -= 32;
    }
    if (lost) {  // waited long enough: count the flags before this tile
      before = 0;
      for (int64_t p = lane; p < (int64_t)t * kPartTile; p += 32) before += side[ord[p]];
#pragma unroll
      for (int o = 16; o; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    }
    if (lane == 0) {
      if (t > 0) look[tile] = kInc | (before + all);
      before_s = before;
    }
  }
  __syncthreads();
  const int64_t base = (int64_t)before_s + wb, q0 = n >> level;
#pragma unroll
  for (int q = 0; q < kPartItems; ++q) {
    const int64_t i = i0 + 32 * q;
    if (i >= n) continue;
    uint32_t f = 0, m = (uint32_t)n;
    const int64_t j = kd_find((uint32_t)i, level, f, m);
    // second children of the j nodes before: q0 and q0 + 1 particles, larger = f - j q0 of the latter
    const int64_t larger = (int64_t)f - j * q0;
    const int64_t nodes_before = (j - larger) * (q0 - q0 / 2) + larger * (q0 + 1 - (q0 + 1) / 2);
    const uint32_t r = (uint32_t)(base + ex[q] - nodes_before);
    out[fl[q] ? f + m / 2 + r : (uint32_t)i - r] = v[q];
  }
}

// A node of at most 2048 particles to its leaves, one block: the orders as 16-bit places
// in the node's x order, partitioned level by level in shared memory.
constexpr int kSub = 2048;
__global__ void __launch_bounds__(kT) k_kd_subtree(KdShape S, int top, const double *__restrict__ xw, KdOrders O,
                                                   uint32_t *__restrict__ place, uint32_t *__restrict__ out,
                                                   double *__restrict__ box, int64_t cap, int *__restrict__ axis) {
  constexpr int kPer = kSub / kT;
  __shared__ uint32_t id[kSub];           // the node's particles in x order
  __shared__ __align__(16) uint16_t ord[2][3][kSub];  // the three orders, before and after a level
  __shared__ uint16_t scan[3][kSub];         // second-child particles before each position
  __shared__ uint8_t side[kSub], sax[kSub];  // per particle; split axis per node of the level (3: a leaf)
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t n = S.n;
  uint32_t f0, m0;
  kd_range(n, top, blockIdx.x, f0, m0);
  for (uint32_t i = tid; i < m0; i += kT) {
    const uint32_t p = O.o[0][f0 + i];
    id[i] = p;
    place[p] = i;
    ord[0][0][i] = (uint16_t)i;
  }
  __syncthreads();
  for (uint32_t i = tid; i < m0; i += kT) {
    ord[0][1][i] = (uint16_t)place[O.o[1][f0 + i]];
    ord[0][2][i] = (uint16_t)place[O.o[2][f0 + i]];
  }
  __syncthreads();
  int b = 0;
  for (int l = top; l <= S.depth; ++l) {
    const int r = l - top;
    // ---- the level's nodes: boxes, axes
    for (uint32_t jj = tid; jj < (1u << r); jj += kT) {
      uint32_t f = 0, m = m0;
      for (int q = r - 1; q >= 0; --q) {
        const uint32_t h = m / 2;
        if ((jj >> q) & 1u) {
          f += h;
          m -= h;
        } else {
          m = h;
        }
      }
      const int64_t j = ((int64_t)blockIdx.x << r) + jj, k = ((int64_t)1 << l) - 1 + j;
      const int a = kd_box(xw, n, f, m, [&](int d, uint32_t i) { return id[ord[b][d][i]]; }, box, cap, k);
      const bool split = (int64_t)m > S.leaf_max;
      axis[k] = split ? a : -1;
      sax[jj] = split ? (uint8_t)a : (uint8_t)3;
    }
    __syncthreads();
    if (l == S.depth && S.nsplit == 0) break;
    // ---- sides
    for (uint32_t i = tid; i < m0; i += kT) {
      uint32_t f = 0, m = m0;
      const int a = sax[kd_find(i, r, f, m)];
      if (a < 3) side[ord[b][a][i]] = i - f >= m / 2 ? 1 : 0;
      else side[ord[b][0][i]] = 0;
    }
    __syncthreads();
    // ---- scans of the three orders at once (counts below 2^20 each)
    {
      uint32_t bits = 0;
      unsigned long long s = 0;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const uint32_t i = (uint32_t)tid * kPer + q;
#pragma unroll
        for (int d = 0; d < 3; ++d)
          if (i < m0 && side[ord[b][d][i]]) {
            bits |= 1u << (3 * q + d);
            s += 1ull << (20 * d);
          }
      }
      unsigned long long x = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      // the warps' totals in the orders' other half, which the partition writes after the next barrier
      unsigned long long *wsum = reinterpret_cast<unsigned long long *>(&ord[b ^ 1][0][0]);
      if (lane == 31) wsum[w] = x;
      __syncthreads();
      unsigned long long at = x - s;
      for (int q = 0; q < w; ++q) at += wsum[q];
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const uint32_t i = (uint32_t)tid * kPer + q;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          scan[d][i] = (uint16_t)((at >> (20 * d)) & 0xfffffu);
          if ((bits >> (3 * q + d)) & 1u) at += 1ull << (20 * d);
        }
      }
    }
    __syncthreads();
    // ---- stable partition inside every node that splits
    for (uint32_t i = tid; i < m0; i += kT) {
      uint32_t f = 0, m = m0;
      const bool split = sax[kd_find(i, r, f, m)] < 3;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const uint16_t v = ord[b][d][i];
        const uint32_t before = (uint32_t)scan[d][i] - scan[d][f];
        ord[b ^ 1][d][split ? (side[v] ? f + m / 2 + before : i - before) : i] = v;
      }
    }
    __syncthreads();
    b ^= 1;
    // ---- the children of a level that splits in part: the last level's boxes
    if (l == S.depth) {
      for (uint32_t jj = tid; jj < (1u << r); jj += kT) {
        if (sax[jj] == 3) continue;
        uint32_t f = 0, m = m0;
        for (int q = r - 1; q >= 0; --q) {
          const uint32_t h = m / 2;
          if ((jj >> q) & 1u) {
            f += h;
            m -= h;
          } else {
            m = h;
          }
        }
        const int64_t j = ((int64_t)blockIdx.x << r) + jj;
        const int64_t c = S.last_start() + 2 * ((int64_t)f0 + f - j * S.q);
        auto at = [&](int d, uint32_t i) { return id[ord[b][d][i]]; };
        kd_box(xw, n, f, m / 2, at, box, cap, c);
        kd_box(xw, n, f + m / 2, m - m / 2, at, box, cap, c + 1);
        axis[c] = axis[c + 1] = -1;
      }
    }
  }
  for (uint32_t i = tid; i < m0; i += kT) out[f0 + i] = id[ord[b][0][i]];
}

// Centre, half extents, side and expansion scale of every node.
__global__ void k_kd_geo(int64_t nn, int64_t cap, const double *__restrict__ box, double L, double *__restrict__ geo,
                         float *__restrict__ geof, float *__restrict__ hs, const int *__restrict__ child) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  double side = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double a = box[d * cap + k], b = box[(3 + d) * cap + k];
    geo[d * cap + k] = __dmul_rn(0.5, __dadd_rn(a, b));
    geo[(3 + d) * cap + k] = __dmul_rn(0.5, __dsub_rn(b, a));
    const double e = __dsub_rn(b, a);
    side = d == 0 ? e : (e > side ? e : side);
  }
  geo[6 * cap + k] = side;
  // the walk's FP32 record of the node: (centre xyz, side), (half extents xyz, first child)
  reinterpret_cast<float4 *>(geof)[2 * k] = make_float4((float)geo[k], (float)geo[cap + k], (float)geo[2 * cap + k],
                                                         (float)side);
  reinterpret_cast<float4 *>(geof)[2 * k + 1] = make_float4((float)geo[3 * cap + k], (float)geo[4 * cap + k],
                                                             (float)geo[5 * cap + k], __int_as_float(child[k]));
  double h = L;
  for (int j = 0; j < kDepth && side <= 0.5 * h; ++j) h *= 0.5;
  hs[k] = (float)h;
}

// Particles in tree order: positions, input index, offset from the leaf's box centre and mass.
__global__ void k_kd_particles(int64_t n, const uint32_t *__restrict__ o0, const double *__restrict__ xw,
                               const float *__restrict__ mass, KdShape S,
                               const double *__restrict__ geo, int64_t cap, double *__restrict__ xs,
                               uint32_t *__restrict__ perm, float4 *__restrict__ pm4) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  // the leaf of position i
  uint32_t f = 0, m = (uint32_t)n;
  const int64_t j = kd_find((uint32_t)i, S.depth, f, m);
  int64_t k = ((int64_t)1 << S.depth) - 1 + j;
  if ((int64_t)m > S.leaf_max) k = S.last_start() + 2 * ((int64_t)f - j * S.q) + ((uint32_t)i - f >= m / 2 ? 1 : 0);
  const uint32_t p = o0[i];
  float off[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double x = xw[d * n + p];
    xs[d * n + i] = x;
    off[d] = (float)__dsub_rn(x, geo[d * cap + k]);
  }
  perm[i] = p;
  pm4[i] = make_float4(off[0], off[1], off[2], mass[p]);
}

// ------------------------------------------------------------------ walk
struct KdGeo {
  const double *g;  // [7][cap]: centre xyz, half extents xyz, side
  const float *gf;  // [cap][8]: (centre xyz, side), (half extents xyz, first child) rounded to FP32
  int64_t cap;
  __device__ double c(int d, uint32_t k) const { return g[d * cap + k]; }
  __device__ double e(int d, uint32_t k) const { return g[(3 + d) * cap + k]; }
  __device__ double side(uint32_t k) const { return g[6 * cap + k]; }
  __device__ void rec(uint32_t k, float4 &p, float4 &q) const {
    const float4 *r = reinterpret_cast<const float4 *>(gf) + 2 * (size_t)k;
    p = __ldg(r);
    q = __ldg(r + 1);
  }
};

__device__ __forceinline__ float comp(const float4 &v, int d) { return d == 0 ? v.x : d == 1 ? v.y : v.z; }

struct WalkRule {
  double L, rc2, theta2;
  float Lf, rc2f, theta2f, dl;  // dl: 16 2^-24 L, the FP32 error bound of a shifted difference
  int rule, size_rule;
  int conventional;  // 1: the opening-angle test alone (a conventional FMM, Sec. 3), primary box
};

// 0 skip, 1 M2L, 2 open: the rules of Sec. 2.3 on the boxes (sink a, source b shifted by s L),
// in FP64 with every operation rounded on its own.
__device__ __forceinline__ int kd_classify64(const KdGeo &G, uint32_t a, uint32_t b, uint32_t s, const WalkRule &R) {
  double sc2 = 0.0, sm2 = 0.0, sx2 = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double dc = __dsub_rn(__dadd_rn(G.c(d, b), (double)shift_component(s, d) * R.L), G.c(d, a));
    const double ad = fabs(dc);
    const double w = __dadd_rn(G.e(d, a), G.e(d, b));
    double gap = __dsub_rn(ad, w);
    if (gap < 0.0) gap = 0.0;
    const double far = __dadd_rn(ad, w);
    sc2 = __dadd_rn(sc2, __dmul_rn(dc, dc));
    sm2 = __dadd_rn(sm2, __dmul_rn(gap, gap));
    sx2 = __dadd_rn(sx2, __dmul_rn(far, far));
  }
  if (!R.conventional && sm2 > R.rc2) return 0;
  const bool trans = R.conventional ? false : R.rule == 0 ? sc2 > R.rc2 : sx2 > R.rc2;
  const double sa = G.side(a), sb = G.side(b);
  const double wl = R.size_rule == 0 ? sb : (sa > sb ? sa : sb);
  const double lim = __dmul_rn(R.theta2, sc2);  // a pair with theta S_c = 0 is never accepted
  if (!trans && lim > 0.0 && __dmul_rn(wl, wl) <= lim) return 1;
  return 2;
}

// The same decisions, taken in FP32 where they are certain.  In FP32 the node
// geometry is off by at most 2^-24 L (centres) and 2^-25 L (half extents), so each
// shifted per-axis difference dc, gap and span (coordinates in [-L, 2L]) is within
// delta = 16 2^-24 L of its FP64 value, and a sum q of three squares x^2 within
//   E(q) = 2 (2 delta sum |x| + 3 delta^2 + 8 2^-24 q)
// (the factor 2 a margin above the rounding analysis); theta^2 S_c^2 within
// 2 (theta^2 E(S_c^2) + 3 2^-24 theta^2 S_c^2), the squared side within 6 2^-24 of
// itself, R_c^2 within 2^-23 of itself.  A comparison whose two sides' intervals
// overlap is taken again in FP64 (this GPU's FP64 rate is low), so the result is
// always the FP64 one.
__device__ __noinline__ int kd_classify64_call(const KdGeo &G, uint32_t a, uint32_t b, uint32_t s,
                                               const WalkRule &R) {
  return kd_classify64(G, a, b, s, R);
}

__device__ __forceinline__ int kd_classify(const KdGeo &G, uint32_t a, uint32_t b, uint32_t s, const WalkRule &R,
                                           const float4 &A0, const float4 &A1, const float4 &B0, const float4 &B1) {
  constexpr float u = 5.9604645e-8f;  // 2^-24
  float sc2 = 0.f, sm2 = 0.f, sx2 = 0.f, Sc = 0.f, Sm = 0.f, Sx = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float dc = __fsub_rn(__fadd_rn(comp(B0, d), (float)shift_component(s, d) * R.Lf), comp(A0, d));
    const float ad = fabsf(dc);
    const float w = __fadd_rn(comp(A1, d), comp(B1, d));
    const float gap = fmaxf(__fsub_rn(ad, w), 0.f);
    const float far = __fadd_rn(ad, w);
    sc2 = __fadd_rn(sc2, __fmul_rn(dc, dc));
    sm2 = __fadd_rn(sm2, __fmul_rn(gap, gap));
    sx2 = __fadd_rn(sx2, __fmul_rn(far, far));
    Sc += ad;
    Sm += gap;
    Sx += far;
  }
  const float dl = R.dl, d2 = 3.f * dl * dl;
  const float erc = 2.f * u * R.rc2f;
  const float ec = 2.f * (2.f * dl * Sc + d2 + 8.f * u * sc2);
  if (!R.conventional) {
    const float em = 2.f * (2.f * dl * Sm + d2 + 8.f * u * sm2);
    if (sm2 - em > R.rc2f + erc) return 0;
    if (sm2 + em >= R.rc2f - erc) return kd_classify64_call(G, a, b, s, R);
    const float tq = R.rule == 0 ? sc2 : sx2;
    const float et = R.rule == 0 ? ec : 2.f * (2.f * dl * Sx + d2 + 8.f * u * sx2);
    if (tq - et > R.rc2f + erc) return 2;
    if (tq + et >= R.rc2f - erc) return kd_classify64_call(G, a, b, s, R);
  }
  if (R.theta2 == 0.0) return 2;
  const float sa = A0.w, sb = B0.w;
  const float wl = R.size_rule == 0 ? sb : fmaxf(sa, sb);
  const float lim = __fmul_rn(R.theta2f, sc2), w2 = __fmul_rn(wl, wl);
  const float el = 2.f * (R.theta2f * ec + 3.f * u * lim), ew = 6.f * u * w2;
  if (lim - el > 0.f && w2 + ew < lim - el) return 1;
  if (w2 - ew > lim + el) return 2;
  return kd_classify64_call(G, a, b, s, R);
}

// Walk counters (u64): [0] M2L entries, [1] P2P entries, [2] status (1: the open lists
// outgrown), [3] levels walked, [4] pairs classified, [5..7] open entries and [8..10] nodes
// handed out of three consecutive levels (level l uses [.. + l % 3]; the one of level l + 1
// is cleared during level l, after every block has read it at level l - 2).
constexpr int kWalkCtr = 11;

struct KdWalk {
  KdShape S;
  KdGeo G;
  WalkRule R;
  const int *parent;
  uint32_t *open[2];    // open lists of the even and the odd levels' nodes: (node, shift)
  unsigned long long *obeg;  // per node with children: its open list
  uint32_t *ocnt;
  uint64_t *m2l, *p2p;
  uint32_t *mb, *me, *pb, *pe;  // CSR bounds by sink
  unsigned long long cap_open, cap_m2l, cap_p2p;
  unsigned long long *ctr;
};

constexpr int kStack = 512, kSoft = 448;  // sources a sink has still to visit
constexpr int kStage = 1024;              // entries staged in shared memory
constexpr int kWalkWarpWords = kStack + kStage;

constexpr int kKdWarps = kT / 32;
// A group of warps that share a session: its part of the block's shared memory, and its barrier.
struct KdGroup {
  unsigned long long bm, bp;
  uint32_t nm[kKdWarps], np[kKdWarps];
};
__device__ __forceinline__ void kd_sync(int group, int warps) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(32 * warps) : "memory");
}

// One sink's session, a warp's or (kShared) that of a group of `warps` warps, each its part
// of the parent's list: every pair (sink, b, s) the walk meets is classified.  The
// pairs start from those its parent left open (the root: its 27 images, or itself alone in
// the conventional walk).  The larger of the two opens, at equal sizes both, and only a node
// with children: a source that opens alone stays with this sink (its children go on a
// stack), and where the sink opens, alone or with the source, the source or its children go
// to the open list both its children start from.  The M2L entries and the P2P or open
// entries are staged, their ranges taken with one atomic per list at the end (a group's
// entries in warp order); a session with
// more entries than the stage holds counts them and walks again, writing in place.
// Above kSoft waiting the stack is taken one source at a time: each adds one at most per
// level of the tree (27 levels: node numbers are below 2^27), so it holds.
template <bool kShared>
__device__ __forceinline__ void kd_session(const KdWalk &W, uint32_t k, int level, uint32_t *stack, uint32_t *stage,
                                           KdGroup *groups, int warps, unsigned long long *nopen,
                                           unsigned long long &items) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  float4 A0, A1;
  W.G.rec(k, A0, A1);
  const int ca = __float_as_int(A1.w);
  const bool leaf = ca < 0;
  const uint32_t *in = W.open[(level & 1) ^ 1];
  unsigned long long ibeg = 0;
  uint32_t icnt = W.R.conventional ? 1u : 27u;
  if (k != 0) {
    const int p = W.parent[k];
    ibeg = W.obeg[p];
    icnt = W.ocnt[p];
  }
  const int group = (threadIdx.x >> 5) / warps, wp = (threadIdx.x >> 5) % warps;
  KdGroup &B = groups[kShared ? group : 0];
  uint32_t ifirst = 0;
  if (kShared) {
    const uint32_t share = (icnt + warps - 1) / warps;
    ifirst = min(share * wp, icnt);
    icnt = min(ifirst + share, icnt);
  }
  uint64_t *const m2l = W.m2l, *const p2p = W.p2p;
  uint32_t *const out = W.open[level & 1];
  unsigned long long bm = 0, bp = 0;
  bool fit_m = false, fit_p = false;
  uint32_t nm = 0, np = 0;  // M2L entries; P2P (a leaf's) or open entries
  for (int pass = 0; pass < 2; ++pass) {
    uint32_t pi = ifirst;
    int sp = 0;
    bool over = false;
    nm = np = 0;
    for (;;) {
      // ---- the next sources: from the stack, then from the parent's open list
      int ks = sp < 32 ? sp : 32;
      uint32_t kl = icnt - pi < (uint32_t)(32 - ks) ? icnt - pi : (uint32_t)(32 - ks);
      if (sp > kSoft) {
        ks = 1;
        kl = 0;
      }
      if (ks + (int)kl == 0) break;
      const bool has = lane < ks + (int)kl;
      uint32_t e = 0;
      if (lane < ks) e = stack[sp - ks + lane];
      else if (has) e = k != 0 ? in[ibeg + pi + lane - ks] : W.R.conventional ? 13u : pi + lane - ks;
      sp -= ks;
      pi += kl;
      __syncwarp();
      // ---- what becomes of each
      const uint32_t b = e >> 5, s = e & 31u;
      int cls = 0, cb = -1;
      bool opena = false, openb = false;
      if (has) {
        float4 B0, B1;
        W.G.rec(b, B0, B1);
        cls = kd_classify(W.G, k, b, s, W.R, A0, A1, B0, B1);
        cb = __float_as_int(B1.w);
        if (cls == 2) {
          if (leaf && cb < 0) {
            cls = 3;  // two leaves: P2P
          } else if (leaf) {
            openb = true;
          } else if (cb < 0) {
            opena = true;
          } else if (A0.w != B0.w) {  // rounding to FP32 keeps the order of unequal sides
            opena = A0.w > B0.w;
            openb = !opena;
          } else {
            const double sa = W.G.side(k), sb = W.G.side(b);
            opena = sa >= sb;
            openb = sb >= sa;
          }
        }
        if (pass == 0) ++items;
      }
      const uint32_t kid = (uint32_t)cb << 5 | s;
      // the source's children, to be visited by this sink
      const unsigned mo = __ballot_sync(0xffffffffu, openb && !opena);
      if (openb && !opena) {
        const int at = sp + 2 * __popc(mo & lt);
        stack[at] = kid;
        stack[at + 1] = kid + 32u;
      }
      sp += 2 * __popc(mo);
      // M2L; P2P or open (one entry, or the source's two children)
      const bool far = cls == 1, near = cls == 3 || opena, two = opena && openb;
      const unsigned mm = __ballot_sync(0xffffffffu, far), m1 = __ballot_sync(0xffffffffu, near),
                     m2 = __ballot_sync(0xffffffffu, two);
      const uint32_t im = nm + __popc(mm & lt), ip = np + __popc(m1 & lt) + __popc(m2 & lt);
      nm += __popc(mm);
      np += __popc(m1) + __popc(m2);
      const uint32_t v = two ? kid : e;
      if (pass == 0) {
        over = over || nm + np > (uint32_t)kStage;
        if (!over) {  // P2P or open entries from the front, M2L from the back
          if (far) stage[kStage - 1 - im] = e;
          if (near) stage[ip] = v;
          if (two) stage[ip + 1] = v + 32u;
        }
      } else {
        if (far && fit_m) m2l[bm + im] = pack_pair(k, 0, 0) | e;
        if (near && fit_p) {
          if (leaf) p2p[bp + ip] = pack_pair(k, 0, 0) | v;
          else out[bp + ip] = v;
        }
        if (two && fit_p) out[bp + ip + 1] = v + 32u;
      }
      __syncwarp();
    }
    if (pass == 1) break;
    // ---- the entries' ranges: the sink's, and in them this warp's
    uint32_t all_m = nm, all_p = np, before_m = 0, before_p = 0;
    if (kShared) {
      if (lane == 0) {
        B.nm[wp] = nm;
        B.np[wp] = np;
      }
      kd_sync(group, warps);
      all_m = all_p = 0;
      for (int q = 0; q < warps; ++q) {
        if (q == wp) {
          before_m = all_m;
          before_p = all_p;
        }
        all_m += B.nm[q];
        all_p += B.np[q];
      }
    }
    if (lane == 0 && (!kShared || wp == 0)) {
      if (all_m) bm = atomicAdd(W.ctr + 0, (unsigned long long)all_m);
      if (all_p) bp = atomicAdd(leaf ? W.ctr + 1 : nopen, (unsigned long long)all_p);
      if (kShared) {
        B.bm = bm;
        B.bp = bp;
      }
    }
    if (kShared) {
      kd_sync(group, warps);
      bm = B.bm;
      bp = B.bp;
    } else {
      bm = __shfl_sync(0xffffffffu, bm, 0);
      bp = __shfl_sync(0xffffffffu, bp, 0);
    }
    fit_m = all_m > 0 && bm + all_m <= W.cap_m2l;
    fit_p = all_p > 0 && bp + all_p <= (leaf ? W.cap_p2p : W.cap_open);
    if (lane == 0 && (!kShared || wp == 0)) {
      W.mb[k] = (uint32_t)bm;
      W.me[k] = (uint32_t)bm + (fit_m ? all_m : 0u);
      W.pb[k] = leaf ? (uint32_t)bp : 0u;
      W.pe[k] = leaf ? (uint32_t)bp + (fit_p ? all_p : 0u) : 0u;
      if (!leaf) {
        W.obeg[k] = bp;
        W.ocnt[k] = fit_p ? all_p : 0u;
      }
    }
    bm += before_m;
    bp += before_p;
    if (!over) {
      if (fit_m)
        for (uint32_t i = lane; i < nm; i += 32) m2l[bm + i] = pack_pair(k, 0, 0) | stage[kStage - 1 - i];
      if (fit_p)
        for (uint32_t i = lane; i < np; i += 32) {
          if (leaf) p2p[bp + i] = pack_pair(k, 0, 0) | stage[i];
          else out[bp + i] = stage[i];
        }
      break;
    }
    if (!fit_m && !fit_p) break;
  }
  __syncwarp();
}

// The whole walk in one cooperative launch, the tree's levels in turn with a grid-wide
// barrier between them (an open list is complete before the children start from it), a
// level's nodes to warps (a large level's from a counter), until the last level or open lists that outgrow
// their buffer (the caller grows the buffers that were outgrown and walks again).  Each
// sink's entries lie together, in an order that does not depend on the schedule.
//
// What bounds it: instructions, in the last two levels (two thirds of the pairs); the levels
// above by latency, one session and one barrier each: there a group of as many warps shares
// a session as leaves every node of the level a group (one warp a session everywhere, the
// walk alone: 121 -> 94 us at 2000 clustered particles, 271 -> 191 at 30k, 436 -> 345 at 100k,
// 1.46 -> 1.24 ms at 2M).  A walk over a frontier of (sink,
// source) pairs, two entries of 8 bytes written and read a pair, left lists to be sorted
// by (sink, source, shift): 2.0 + 1.5 ms for 46M pairs and 21M entries (2M clustered
// particles) instead of 1.24.
__global__ void __launch_bounds__(kT, 4) k_kd_walk(const __grid_constant__ KdWalk W) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ uint32_t walk_smem[];
  const int lane = threadIdx.x & 31;
  uint32_t *stack = walk_smem + (threadIdx.x >> 5) * kWalkWarpWords, *stage = stack + kStack;
  __shared__ KdGroup groups[kKdWarps / 2];
  const bool first = blockIdx.x == 0 && threadIdx.x == 0;
  const int levels = W.S.depth + 1 + (W.S.nsplit ? 1 : 0);
  unsigned long long items = 0, most = 0;
  int level = 0;
  for (; level < levels; ++level) {
    const uint32_t lo = (uint32_t)(((int64_t)1 << level) - 1);
    const uint32_t hi = level <= W.S.depth ? (uint32_t)(((int64_t)2 << level) - 1) : (uint32_t)W.S.nodes();
    unsigned long long *nopen = W.ctr + 5 + level % 3, *ticket = W.ctr + 8 + level % 3;
    if (first) W.ctr[5 + (level + 1) % 3] = W.ctr[8 + (level + 1) % 3] = 0;
    int warps = kKdWarps;  // a session's: as many as leave every node of the level a group
    while (warps > 1 && hi - lo > gridDim.x * (uint32_t)(kKdWarps / warps)) warps >>= 1;
    if (warps > 1) {
      const uint32_t t = blockIdx.x * (uint32_t)(kKdWarps / warps) + (threadIdx.x >> 5) / warps;
      if (t < hi - lo) kd_session<true>(W, lo + t, level, stack, stage, groups, warps, nopen, items);
    } else {
      for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(ticket, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= hi - lo) break;
        kd_session<false>(W, lo + (uint32_t)t, level, stack, stage, groups, 1, nopen, items);
      }
    }
    grid.sync();
    // every block reads the same count, and so takes the same decision; the M2L and P2P
    // counts are the caller's to compare with the capacities
    most = *(volatile unsigned long long *)nopen;
    if (most > W.cap_open) break;
  }
  if (first) {
    W.ctr[2] = most > W.cap_open ? 1ull : 0ull;
    W.ctr[3] = (unsigned long long)min(level + 1, levels);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) items += __shfl_xor_sync(0xffffffffu, items, o);
  if (lane == 0 && items) atomicAdd(W.ctr + 4, items);
}

// Particle pairs on the P2P list: sum over entries of n_sink n_source.
__global__ void k_kd_list_pairs(const uint64_t *__restrict__ lst, int64_t n, const uint32_t *__restrict__ count,
                                unsigned long long *__restrict__ out) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = 0;
  if (t < n) v = (unsigned long long)count[pair_sink(lst[t])] * count[pair_src(lst[t])];
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(out, v);
}

#define TRY(x)                      \
  do {                              \
    cudaError_t e_ = (x);           \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

// Read `count` device uint64 values into out (synchronises st).
cudaError_t read_u64(Ctx &c, const void *src, uint64_t *out, int count, cudaStream_t st) {
  TRY(cudaMemcpyAsync(c.h_pinned, src, 8 * (size_t)count, cudaMemcpyDeviceToHost, st));
  TRY(cudaStreamSynchronize(st));
  for (int q = 0; q < count; ++q) out[q] = c.h_pinned[q];
  return cudaSuccess;
}

// The walk (one cooperative launch, repeated with grown buffers while one is outgrown).
cudaError_t kd_walk(Ctx &c, cudaStream_t st, bool conventional = false) {
  KdTree &kd = c.kd;
  const uint64_t nl = (uint64_t)std::max<int64_t>(c.nleaves, 1);
  uint64_t cap_f = std::max<uint64_t>(kd.caps[0], std::max<uint64_t>(1u << 16, 256 * nl));
  uint64_t cap_m = std::max<uint64_t>(kd.caps[1], std::max<uint64_t>(1u << 16, 32 * nl));
  uint64_t cap_p = std::max<uint64_t>(kd.caps[2], std::max<uint64_t>(1u << 16, 256 * nl));
  if (c.prm.list_init > 0 && kd.caps[0] == 0) cap_f = cap_m = cap_p = (uint64_t)c.prm.list_init;
  const size_t nn = (size_t)c.nnodes;
  TRY(ensure(kd.ctr, 128));
  TRY(ensure(kd.obeg, nn * 8));
  TRY(ensure(kd.ocnt, nn * 4));
  TRY(ensure(c.m2l_beg, nn * 4));
  TRY(ensure(c.m2l_end, nn * 4));
  TRY(ensure(c.p2p_beg, nn * 4));
  TRY(ensure(c.p2p_end, nn * 4));
  unsigned long long *ctr = P<unsigned long long>(kd.ctr);
  const size_t smem = (size_t)(kT / 32) * kWalkWarpWords * 4;
  int dev = 0, nsm = 0, per_sm = 0;
  TRY(cudaGetDevice(&dev));
  TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  TRY(cudaFuncSetAttribute(k_kd_walk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_kd_walk, kT, smem));
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // two warps a leaf at most: a level's barrier costs more the more blocks it spans
  const unsigned nb = std::min((unsigned)(nsm * std::min(per_sm, 4)), blocks_for((size_t)nl, 4));
  KdWalk W;
  W.S = kd_shape(c.n, c.prm.leaf_max);
  W.G = KdGeo{P<double>(kd.geo), P<float>(kd.geof), kd.cap};
  W.R.L = c.prm.box;
  W.R.rc2 = c.rc * c.rc;
  W.R.theta2 = c.prm.theta * c.prm.theta;
  W.R.Lf = (float)W.R.L;
  W.R.rc2f = (float)W.R.rc2;
  W.R.theta2f = (float)W.R.theta2;
  W.R.dl = (float)std::ldexp(16.0 * W.R.L, -24);
  W.R.rule = c.prm.transition_rule;
  W.R.size_rule = c.prm.size_rule;
  W.R.conventional = conventional ? 1 : 0;
  W.parent = P<int>(kd.parent);
  W.obeg = P<unsigned long long>(kd.obeg);
  W.ocnt = P<uint32_t>(kd.ocnt);
  W.mb = P<uint32_t>(c.m2l_beg);
  W.me = P<uint32_t>(c.m2l_end);
  W.pb = P<uint32_t>(c.p2p_beg);
  W.pe = P<uint32_t>(c.p2p_end);
  W.ctr = ctr;
  int64_t walks = 0;
  uint64_t h[kWalkCtr];
  for (;;) {
    if (++walks > 32) return cudaErrorInvalidValue;
    for (DBuf &b : kd.open) TRY(ensure(b, cap_f * 4));
    TRY(ensure(c.m2l, cap_m * 8));
    TRY(ensure(c.p2p, cap_p * 8));
    TRY(cudaMemsetAsync(ctr, 0, kWalkCtr * 8, st));
    W.open[0] = P<uint32_t>(kd.open[0]);
    W.open[1] = P<uint32_t>(kd.open[1]);
    W.m2l = P<uint64_t>(c.m2l);
    W.p2p = P<uint64_t>(c.p2p);
    W.cap_open = cap_f;
    W.cap_m2l = cap_m;
    W.cap_p2p = cap_p;
    void *args[] = {(void *)&W};
    TRY(cudaLaunchCooperativeKernel((const void *)k_kd_walk, dim3(nb), dim3(kT), args, smem, st));
    note_launch();
    TRY(read_u64(c, ctr, h, kWalkCtr, st));
    if (!h[2] && h[0] <= cap_m && h[1] <= cap_p) break;
    // an outgrown buffer: grow what the counts ask for (the counts went on past the capacities)
    const uint64_t most = std::max(std::max(h[5], h[6]), h[7]);
    if (most > cap_f) cap_f = most + most / 2 + 4096;
    if (h[0] > cap_m) cap_m = h[0] + h[0] / 2 + 4096;
    if (h[1] > cap_p) cap_p = h[1] + h[1] / 2 + 4096;
  }
  kd.caps[0] = cap_f;
  kd.caps[1] = cap_m;
  kd.caps[2] = cap_p;
  c.nm2l = (int64_t)h[0];
  c.np2p = (int64_t)h[1];
  c.traverse_iters = (int)h[3];
  c.frontier_items = (int64_t)h[4];
  c.traverse_walks = walks;
  return cudaSuccess;
}

// The particle pairs on the P2P list (synchronises st).
cudaError_t kd_particle_pairs(Ctx &c, int64_t *out, cudaStream_t st) {
  unsigned long long *cnt = P<unsigned long long>(c.kd.ctr) + kWalkCtr + 1;
  TRY(cudaMemsetAsync(cnt, 0, 8, st));
  if (c.np2p > 0) {
    k_kd_list_pairs<<<blocks_for((size_t)c.np2p, kT), kT, 0, st>>>(P<uint64_t>(c.p2p), c.np2p,
                                                                    P<uint32_t>(c.kd.count), cnt);
    note_launch();
  }
  uint64_t pp = 0;
  TRY(read_u64(c, cnt, &pp, 1, st));
  *out = (int64_t)pp;
  return cudaSuccess;
}

}  // namespace

cudaError_t kd_build_tree(Ctx &c, const double *pos, const float *mass, int64_t n, cudaStream_t st) {
  KdTree &kd = c.kd;
  c.n = n;
  c.nnodes = c.nleaves = 0;
  c.nlevels = 0;
  c.have_tree = false;
  kd.level_start.assign(1, 0);
  if (n == 0) {
    c.have_tree = true;
    return cudaSuccess;
  }
  const KdShape S = kd_shape(n, c.prm.leaf_max);
  const int64_t nn = S.nodes(), cap = nn + 2;
  // the nodes that n particles can take in the worst case must fit the lists' node bits
  const int64_t lmin = std::max(1, (c.prm.leaf_max + 1) / 2);
  if (2 * ((n + lmin - 1) / lmin) + 2 > ((int64_t)1 << kSinkBits))
    return cudaErrorInvalidValue;  // mapped to HFMM_ERR_CAPACITY
  kd.cap = cap;
  if (c.prm.profile & 1) cudaEventRecord(c.ev[0], st);
  TRY(ensure(kd.xw, (size_t)n * 24));
  for (int d = 0; d < 3; ++d) {
    TRY(ensure(kd.ord[d], (size_t)n * 4));
    TRY(ensure(kd.ord2[d], (size_t)n * 4));
  }
  TRY(ensure(kd.side, (size_t)n));
  TRY(ensure(kd.place, (size_t)n * 4));
  TRY(ensure(kd.first, (size_t)cap * 4));
  TRY(ensure(kd.count, (size_t)cap * 4));
  TRY(ensure(kd.child, (size_t)cap * 4));
  TRY(ensure(kd.parent, (size_t)cap * 4));
  TRY(ensure(kd.axis, (size_t)cap * 4));
  TRY(ensure(kd.box, (size_t)cap * 48));
  TRY(ensure(kd.geo, (size_t)cap * 56));
  TRY(ensure(kd.geof, (size_t)cap * 32));
  TRY(ensure(kd.hs, (size_t)cap * 4));
  TRY(ensure(c.key, (size_t)n * 8));
  TRY(ensure(c.key_alt, (size_t)n * 8));
  TRY(ensure(c.idx, (size_t)n * 4));
  TRY(ensure(c.xs, (size_t)n * 24));
  TRY(ensure(c.pm4, (size_t)n * 16));
  TRY(ensure(c.leaves, (size_t)cap * 4));
  const double inv_pow2 = box_inverse_if_pow2(c.prm.box);
  double *xw = P<double>(kd.xw);
  k_kd_wrap<<<blocks_for((size_t)(3 * n), kT), kT, 0, st>>>(pos, n, c.prm.box, inv_pow2, xw);
  note_launch();
  for (int d = 0; d < 3; ++d) {
    k_kd_keys<<<blocks_for((size_t)n, kT), kT, 0, st>>>(xw + d * n, n, P<uint64_t>(c.key), P<uint32_t>(kd.ord[d]));
    note_launch();
    bool alt = false;
    TRY(radix_sort_u64(P<uint64_t>(c.key), P<uint32_t>(kd.ord[d]), P<uint64_t>(c.key_alt), P<uint32_t>(kd.ord2[d]),
                       (size_t)n, 0, 64, &alt, c.tmp, st, wait_polls(c, kLookPolls)));
    if (alt) std::swap(kd.ord[d], kd.ord2[d]);
  }
  if (c.prm.profile & 1) cudaEventRecord(c.ev[1], st);
  int *child = P<int>(kd.child), *axis = P<int>(kd.axis);
  const unsigned gn = blocks_for((size_t)n, kT), gk = blocks_for((size_t)nn, kT);
  k_kd_topology<<<blocks_for((size_t)S.last_start(), kT), kT, 0, st>>>(
      S, P<uint32_t>(kd.first), P<uint32_t>(kd.count), child, P<int>(kd.parent), P<uint32_t>(c.leaves));
  note_launch();
  auto orders = [&]() { return KdOrders{{P<uint32_t>(kd.ord[0]), P<uint32_t>(kd.ord[1]), P<uint32_t>(kd.ord[2])}}; };
  // levels of nodes above kSub particles
  int top = 0;
  while (top < S.depth && ((n + ((int64_t)1 << top) - 1) >> top) > kSub) ++top;
  const unsigned ntiles = blocks_for((size_t)n, kPartTile);
  if (top > 0) {
    const size_t words = 3 * (size_t)ntiles + 1;  // a level's ticket and counts
    TRY(ensure(c.tmp2, (size_t)top * words * 8));
    TRY(cudaMemsetAsync(c.tmp2.p, 0, (size_t)top * words * 8, st));
    for (int l = 0; l < top; ++l) {
      k_kd_axis<<<blocks_for((size_t)1 << l, 128), 128, 0, st>>>(n, l, xw, orders(), P<double>(kd.box), cap, axis);
      k_kd_side<<<gn, kT, 0, st>>>(n, l, axis, orders(), P<uint8_t>(kd.side));
      unsigned long long *lw = P<unsigned long long>(c.tmp2) + (size_t)l * words;
      k_kd_part<<<3 * ntiles, kT, 0, st>>>(n, l, orders(), P<uint32_t>(kd.ord2[0]), P<uint32_t>(kd.ord2[1]),
                                           P<uint32_t>(kd.ord2[2]), P<uint8_t>(kd.side),
                                           reinterpret_cast<unsigned *>(lw), lw + 1, ntiles,
                                           wait_polls(c, kLookPolls));
      note_launch(3);
      for (int d = 0; d < 3; ++d) std::swap(kd.ord[d], kd.ord2[d]);
    }
  }
  k_kd_subtree<<<1u << top, kT, 0, st>>>(S, top, xw, orders(), P<uint32_t>(kd.place), P<uint32_t>(kd.ord2[0]),
                                         P<double>(kd.box), cap, axis);
  note_launch();
  std::swap(kd.ord[0], kd.ord2[0]);
  c.nnodes = nn;
  c.nleaves = S.leaves();
  c.nlevels = S.depth + 1 + (S.nsplit ? 1 : 0);
  for (int l = 0; l <= S.depth; ++l) kd.level_start.push_back(((int64_t)2 << l) - 1);
  if (S.nsplit) kd.level_start.push_back(nn);
  k_kd_geo<<<gk, kT, 0, st>>>(nn, cap, P<double>(kd.box), c.prm.box, P<double>(kd.geo), P<float>(kd.geof),
                              P<float>(kd.hs), child);
  note_launch();
  k_kd_particles<<<gn, kT, 0, st>>>(n, P<uint32_t>(kd.ord[0]), xw, mass, S, P<double>(kd.geo), cap, P<double>(c.xs),
                                    P<uint32_t>(c.idx), P<float4>(c.pm4));
  note_launch();
  if (c.prm.profile & 1) cudaEventRecord(c.ev[2], st);
  TRY(cudaGetLastError());
  TRY(cudaStreamSynchronize(st));  // the caller's positions and masses have been read when the call returns
  c.have_tree = true;
  return cudaSuccess;
}

cudaError_t kd_interaction_counts(Ctx &c, bool conventional, int64_t *out, cudaStream_t st) {
  TRY(kd_walk(c, st, conventional));
  out[0] = c.nm2l;
  out[1] = c.np2p;
  out[2] = 0;
  out[3] = c.frontier_items;
  if (c.np2p > 0) TRY(kd_particle_pairs(c, &out[2], st));
  return cudaSuccess;
}

cudaError_t kd_short_range(Ctx &c, float *acc, cudaStream_t st) {
  const bool prof = (c.prm.profile & 1) != 0;
  if (prof) cudaEventRecord(c.ev[3], st);
  TRY(kd_upward(c, st));
  if (prof) cudaEventRecord(c.ev[4], st);
  TRY(kd_walk(c, st));
  if (c.nm2l > (int64_t)UINT32_MAX || c.np2p > (int64_t)UINT32_MAX) return cudaErrorInvalidValue;
  if (prof) cudaEventRecord(c.ev[5], st);
  // statistics runs: the particle pairs on the P2P list
  c.p2p_particle_pairs = -1;
  if (c.prm.profile & 2) TRY(kd_particle_pairs(c, &c.p2p_particle_pairs, st));
  if (prof) cudaEventRecord(c.ev[6], st);
  TRY(m2l_pass(c, c.p, st));
  if (prof) cudaEventRecord(c.ev[7], st);
  TRY(kd_downward(c, acc, st));
  if (prof) cudaEventRecord(c.ev[8], st);
  TRY(p2p_pass(c, acc, st));
  if (prof) cudaEventRecord(c.ev[9], st);
  return cudaSuccess;
}

#undef TRY

}  // namespace hfmm
