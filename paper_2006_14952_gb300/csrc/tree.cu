// Octree build (Sec. 2.1, a tree with a leaf limiter; here a Morton octree):
// periodic wrap, 63-bit Morton keys, stable key sort, the cells holding more than
// leaf_max particles split, and per-particle FP32 offsets from the geometric
// centre of the leaf.
//
// The nodes follow from the sorted keys alone, all levels at once.  Particle i
// starts a cell on every level below those it shares with particle i - 1.  Its
// cell on level l holds more than leaf_max particles, and is split, exactly when
// some run of leaf_max + 1 sorted particles through i shares that level; so the
// deepest split level of i is a sliding maximum of common levels (k_levels), and
// particle i starts a node on the levels from its first own cell to its leaf.
// Counting those per level and tile, one scan over the tiles (k_level_scan)
// numbers the nodes breadth first, in key order within a level (k_nodes).
#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace hfmm {
namespace {

__global__ void k_keys(const double *__restrict__ pos, int64_t n, double box, double inv_pow2, uint64_t *__restrict__ key,
                       uint32_t *__restrict__ idx) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  key[i] = morton_key(pos[i], pos[n + i], pos[2 * n + i], box, inv_pow2);
  idx[i] = (uint32_t)i;
}

constexpr int kLT = 256;        // threads of the level kernels
// Particles per tile: four rounds of the block, or one while the larger tiles would not fill
// the GPU: a block's rounds are a chain of ballots and dependent loads.  k_levels and k_nodes
// with 1024 and with 256, us: 7.1, 14.6 -> 4.6, 6.0 (1000 particles), 7.4, 14.7 -> 4.6, 6.3 (32k),
// 7.5, 17.5 -> 5.1, 8.8 (100k; the scan over more tiles 4.5 -> 7.9).
constexpr int kLTileMost = 1024, kLTileSmall = kLT;
inline bool small_tiles(int64_t n) { return n <= 152 * (int64_t)kLTileMost; }
inline int64_t level_tiles(int64_t n) {
  const int64_t tile = small_tiles(n) ? kLTileSmall : kLTileMost;
  return (n + tile - 1) / tile;
}
constexpr int kHalo = 64;       // leaf_max is at most 64
constexpr int kLCnt = 2 * (kDepth + 1);  // counters per tile: nodes by level, leaves by level

// Levels two keys share: the common octant digits.
__device__ __forceinline__ int common_level(uint64_t a, uint64_t b) {
  const uint64_t x = a ^ b;
  return x ? (__clzll((long long)x) - 1) / 3 : kDepth;
}

// lev[i]: the first level particle i starts a cell on (low byte), the level of its
// leaf (high byte); it starts the nodes of the levels from the first to the second.
// cnt[c][tile]: nodes (c < 22) and leaves (c - 22) by level that start in the tile.
template <int kLTile>
__global__ void __launch_bounds__(kLT) k_levels(const uint64_t *__restrict__ key, int64_t n, int leaf_max,
                                                uint16_t *__restrict__ lev, uint32_t *__restrict__ cnt,
                                                int64_t ntiles) {
  __shared__ uint64_t k[kLTile + 2 * kHalo + 1];
  __shared__ int8_t run[2][kLTile + kHalo];
  __shared__ uint32_t c[kLCnt];
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t t0 = (int64_t)blockIdx.x * kLTile;
  for (int q = tid; q < kLTile + 2 * kHalo + 1; q += kLT) {  // k[q]: particle t0 - kHalo - 1 + q
    const int64_t g = t0 - kHalo - 1 + q;
    k[q] = g >= 0 && g < n ? key[g] : 0ull;
  }
  if (tid < kLCnt) c[tid] = 0u;
  __syncthreads();
  // run[q]: the level shared by particles j .. j + leaf_max, j = t0 - kHalo + q (-1: none)
  for (int q = tid; q < kLTile + kHalo; q += kLT) {
    const int64_t j = t0 - kHalo + q;
    run[0][q] = (int8_t)(j >= 0 && j + leaf_max < n ? common_level(k[q + 1], k[q + 1 + leaf_max]) : -1);
  }
  __syncthreads();
  // maxima of runs starting at q .. q + w - 1, w doubled while it fits the window of leaf_max + 1
  int b = 0, w = 1;
  for (; 2 * w <= leaf_max + 1; w *= 2, b ^= 1) {
    for (int q = tid; q < kLTile + kHalo; q += kLT) {
      const int o = q + w < kLTile + kHalo ? q + w : q;
      run[b ^ 1][q] = run[b][q] > run[b][o] ? run[b][q] : run[b][o];
    }
    __syncthreads();
  }
  for (int p = 0; p < kLTile; p += kLT) {
    const int q = p + tid;
    const int64_t i = t0 + q;
    const bool valid = i < n;
    uint32_t first = 255, last = 0;
    if (valid) {
      const int8_t m0 = run[b][q + kHalo - leaf_max], m1 = run[b][q + kHalo + 1 - w];
      const int m = m0 > m1 ? m0 : m1;
      last = (uint32_t)((m < kDepth ? m : kDepth - 1) + 1);  // cells on the deepest level are not split
      first = i == 0 ? 0u : (uint32_t)(common_level(k[q + kHalo], k[q + kHalo + 1]) + 1);
      lev[i] = (uint16_t)(first | (last << 8));
    }
    const uint32_t lo = __reduce_min_sync(0xffffffffu, first), hi = __reduce_max_sync(0xffffffffu, last);
    for (uint32_t l = lo; l <= hi; ++l) {
      const unsigned nd = __ballot_sync(0xffffffffu, first <= l && l <= last);
      const unsigned lf = __ballot_sync(0xffffffffu, first <= l && l == last);
      if (lane == 0 && nd) atomicAdd(&c[l], (uint32_t)__popc(nd));
      if (lane == 0 && lf) atomicAdd(&c[kDepth + 1 + l], (uint32_t)__popc(lf));
    }
  }
  __syncthreads();
  if (tid < kLCnt) cnt[(int64_t)tid * ntiles + blockIdx.x] = c[tid];
}

// Exclusive scan of each counter over the tiles, in place (a warp a counter), and
// the tree's sizes.  base[c]: the first node (leaf) number of each level.
__global__ void __launch_bounds__(1024) k_level_scan(uint32_t *__restrict__ cnt, int64_t ntiles,
                                                     uint32_t *__restrict__ base, unsigned long long capN,
                                                     int max_levels, TreeState *__restrict__ st) {
  __shared__ unsigned long long tot[kLCnt];
  const int lane = threadIdx.x & 31;
  for (int c = threadIdx.x >> 5; c < kLCnt; c += 32) {
    unsigned long long run = 0;
    uint32_t *row = cnt + (int64_t)c * ntiles;
    for (int64_t t = 0; t < ntiles; t += 128) {
      uint32_t v[4], s = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        v[q] = t + 4 * lane + q < ntiles ? row[t + 4 * lane + q] : 0u;
        s += v[q];
      }
      uint32_t x = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      unsigned long long at = run + x - s;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (t + 4 * lane + q < ntiles) row[t + 4 * lane + q] = (uint32_t)at;
        at += v[q];
      }
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) tot[c] = run;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long nodes = 0, leaves = 0;
    int levels = 0;
    for (int l = 0; l <= kDepth; ++l) {
      base[l] = (uint32_t)nodes;
      base[kDepth + 1 + l] = (uint32_t)leaves;
      st->level_start[l] = nodes;
      nodes += tot[l];
      leaves += tot[kDepth + 1 + l];
      if (tot[l]) levels = l + 1;
    }
    for (int l = levels; l < kDepth + 3; ++l) st->level_start[l] = nodes;
    st->total = nodes;
    st->nleaves = leaves;
    st->nlevels = levels;
    // node capacity, or (graph mode) more levels than the host sized its level loops for
    st->overflow = nodes > capN || levels > max_levels ? 1 : 0;
  }
}

// Every third bit of v, packed (the inverse of spread3).
__device__ __forceinline__ uint32_t pack3(uint64_t v) {
  uint64_t x = v & 0x1249249249249249ull;
  x = (x | (x >> 2)) & 0x10c30c30c30c30c3ull;
  x = (x | (x >> 4)) & 0x100f00f00f00f00full;
  x = (x | (x >> 8)) & 0x001f0000ff0000ffull;
  x = (x | (x >> 16)) & 0x001f00000000ffffull;
  x = (x | (x >> 32)) & 0x1fffffu;
  return (uint32_t)x;
}

// The nodes each particle starts, and the particle itself: sorted wrapped position
// and FP64 offset from the leaf's geometric centre, rounded once to FP32 (the cell
// side L 2^-level built from its bits: no FP64 division).  Cells that split get
// their first child here, their particle and child counts from k_node_counts.
template <int kLTile>
__global__ void __launch_bounds__(kLT) k_nodes(const uint64_t *__restrict__ key, const uint16_t *__restrict__ lev,
                                               int64_t n, int leaf_max, const uint32_t *__restrict__ cnt,
                                               const uint32_t *__restrict__ base, int64_t ntiles,
                                               const TreeState *__restrict__ st, uint4 *__restrict__ cell,
                                               uint2 *__restrict__ range, int2 *__restrict__ kids,
                                               uint32_t *__restrict__ leaves, const double *__restrict__ pos,
                                               const float *__restrict__ mass, const uint32_t *__restrict__ idx,
                                               double box, double inv_pow2, double *__restrict__ xs,
                                               float4 *__restrict__ pm4) {
  constexpr int kRounds = kLTile / 32;  // 32 consecutive particles each
  __shared__ uint16_t lv[kLTile + kHalo + 1];
  __shared__ uint32_t wc[kRounds][kLCnt];
  if (st->overflow) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const int64_t t0 = (int64_t)blockIdx.x * kLTile;
  for (int q = tid; q < kLTile + kHalo + 1; q += kLT) lv[q] = t0 + q < n ? lev[t0 + q] : (uint16_t)0;  // 0: ends every cell
  for (int q = tid; q < kRounds * kLCnt; q += kLT) (&wc[0][0])[q] = 0u;
  __syncthreads();
  for (int p = 0; p < kLTile; p += kLT) {
    const int q = p + tid;
    const bool valid = t0 + q < n;
    const uint32_t first = valid ? lv[q] & 255u : 255u, last = valid ? lv[q] >> 8 : 0u;
    const uint32_t lo = __reduce_min_sync(0xffffffffu, first), hi = __reduce_max_sync(0xffffffffu, last);
    for (uint32_t l = lo; l <= hi; ++l) {
      const unsigned nd = __ballot_sync(0xffffffffu, first <= l && l <= last);
      const unsigned lf = __ballot_sync(0xffffffffu, first <= l && l == last);
      if (lane == 0) {
        wc[q >> 5][l] = (uint32_t)__popc(nd);
        wc[q >> 5][kDepth + 1 + l] = (uint32_t)__popc(lf);
      }
    }
  }
  __syncthreads();
  if (tid < kLCnt) {
    uint32_t at = base[tid] + cnt[(int64_t)tid * ntiles + blockIdx.x];
    for (int q = 0; q < kRounds; ++q) {
      const uint32_t v = wc[q][tid];
      wc[q][tid] = at;
      at += v;
    }
  }
  __syncthreads();
  for (int p = 0; p < kLTile; p += kLT) {
    const int q = p + tid;
    const int64_t i = t0 + q;
    const bool valid = i < n;
    const uint32_t first = valid ? lv[q] & 255u : 255u, last = valid ? lv[q] >> 8 : 0u;
    const uint64_t ki = valid ? key[i] : 0ull;
    const uint32_t cx = pack3(ki >> 2), cy = pack3(ki >> 1), cz = pack3(ki);
    const uint32_t lo = __reduce_min_sync(0xffffffffu, first), hi = __reduce_max_sync(0xffffffffu, last);
    uint32_t child = 0;  // this particle's node one level down
    for (uint32_t l = hi + 1; l-- > lo;) {
      const bool mine = first <= l && l <= last;
      const unsigned nd = __ballot_sync(0xffffffffu, mine);
      const unsigned lf = __ballot_sync(0xffffffffu, mine && l == last);
      if (!mine) continue;
      const uint32_t k = wc[q >> 5][l] + (uint32_t)__popc(nd & lt);
      const uint32_t sh = kDepth - l;
      cell[k] = make_uint4(cx >> sh, cy >> sh, cz >> sh, l);
      uint32_t c = 0;
      if (l == last) {
        leaves[wc[q >> 5][kDepth + 1 + l] + (uint32_t)__popc(lf & lt)] = k;
        kids[k] = make_int2(-1, 0);
        // the leaf ends where a particle starts a cell on its level or above
        c = 1;
        while ((int)c <= leaf_max && (lv[q + c] & 255u) > l) ++c;
        if ((int)c > leaf_max) {  // more than leaf_max particles on the deepest level: equal keys
          int64_t a = i + c, e = n;
          while (a < e) {
            const int64_t mid = a + (e - a) / 2;
            if (key[mid] == ki) a = mid + 1;
            else e = mid;
          }
          c = (uint32_t)(a - i);
        }
      } else {
        kids[k] = make_int2((int)child, 0);
      }
      range[k] = make_uint2((uint32_t)i, c);
      child = k;
    }
    if (valid) {
      const uint32_t o = idx[i], sh = kDepth - last;
      const double h = box * __longlong_as_double((long long)(1023 - (int)last) << 52);
      const double x = wrap_box_fast(pos[o], box, inv_pow2), y = wrap_box_fast(pos[n + o], box, inv_pow2),
                   z = wrap_box_fast(pos[2 * n + o], box, inv_pow2);
      xs[i] = x;
      xs[n + i] = y;
      xs[2 * n + i] = z;
      pm4[i] = make_float4((float)(x - ((double)(cx >> sh) + 0.5) * h), (float)(y - ((double)(cy >> sh) + 0.5) * h),
                           (float)(z - ((double)(cz >> sh) + 0.5) * h), mass[o]);
    }
  }
}

// Cells that split: the end of their particles (a search for the first key outside)
// and how many nodes of the next level start before it.
__global__ void k_node_counts(const uint64_t *__restrict__ key, int64_t n, int leaf_max,
                              const TreeState *__restrict__ st, const uint4 *__restrict__ cell,
                              uint2 *__restrict__ range, int2 *__restrict__ kids) {
  if (st->overflow) return;
  const int64_t nn = (int64_t)st->total, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nn; k += stride) {
    const int ch = kids[k].x;
    if (ch < 0) continue;
    const uint32_t l = cell[k].w, first = range[k].x;
    const int sh = 3 * (kDepth - (int)l);
    const uint64_t pre = key[first] >> sh;
    int64_t a = (int64_t)first + leaf_max + 1, e = n;  // a split cell holds more than leaf_max
    if (k + 1 < (int64_t)st->level_start[l + 1]) e = range[k + 1].x;
    while (a < e) {
      const int64_t mid = a + (e - a) / 2;
      if ((key[mid] >> sh) == pre) a = mid + 1;
      else e = mid;
    }
    int c = 1;
    const int64_t next = (int64_t)st->level_start[l + 2];
    while (c < 8 && ch + c < next && (int64_t)range[ch + c].x < a) ++c;
    range[k].y = (uint32_t)(a - first);
    kids[k].y = c;
  }
}

// Buffers of the levels for n particles and the node capacity.
cudaError_t level_buffers(Ctx &c, int64_t n) {
  cudaError_t e;
  const int64_t ntiles = level_tiles(n);
  const size_t capN = (size_t)c.cap_nodes;
  if ((e = ensure(c.lev, (size_t)n * 2)) != cudaSuccess) return e;
  if ((e = ensure(c.lcnt, (size_t)(ntiles + 1) * kLCnt * 4)) != cudaSuccess) return e;
  if ((e = ensure(c.tstate, sizeof(TreeState))) != cudaSuccess) return e;
  if ((e = ensure(c.cell, capN * sizeof(uint4))) != cudaSuccess) return e;
  if ((e = ensure(c.range, capN * sizeof(uint2))) != cudaSuccess) return e;
  if ((e = ensure(c.kids, capN * sizeof(int2))) != cudaSuccess) return e;
  return ensure(c.leaves, capN * sizeof(uint32_t));
}

// Keys sorted: the nodes and the particles in tree order, sizes in c.tstate (no read-back).
//
// What bounds it: the gathers of positions and masses in sorted order (k_nodes);
// below 10^5 particles, four launches.  The level-synchronous build it replaced
// (one cooperative launch, three grid barriers a level, then a thread a leaf for
// the offsets), ms with its read-back, before and now: 0.54 -> 0.18 at 2M, 1.67 ->
// 1.07 at 16M, 0.32 -> 0.06 at 262k, 0.17 -> 0.04 at 32k, 0.10 -> 0.03 at 1000.
cudaError_t levels_launch(Ctx &c, const double *pos, const float *mass, int64_t n, int max_levels, cudaStream_t st) {
  const int64_t ntiles = level_tiles(n);
  const bool small = small_tiles(n);
  uint32_t *base = P<uint32_t>(c.lcnt), *cnt = base + kLCnt;
  TreeState *ts = P<TreeState>(c.tstate);
  const uint64_t *key = P<uint64_t>(c.key);
  (small ? k_levels<kLTileSmall> : k_levels<kLTileMost>)<<<(unsigned)ntiles, kLT, 0, st>>>(key, n, c.prm.leaf_max, P<uint16_t>(c.lev), cnt, ntiles);
  k_level_scan<<<1, 1024, 0, st>>>(cnt, ntiles, base, c.cap_nodes, max_levels, ts);
  (small ? k_nodes<kLTileSmall> : k_nodes<kLTileMost>)<<<(unsigned)ntiles, kLT, 0, st>>>(
      key, P<uint16_t>(c.lev), n, c.prm.leaf_max, cnt, base, ntiles, ts, P<uint4>(c.cell), P<uint2>(c.range),
      P<int2>(c.kids), P<uint32_t>(c.leaves), pos, mass, P<uint32_t>(c.idx), c.prm.box,
      box_inverse_if_pow2(c.prm.box), P<double>(c.xs), P<float4>(c.pm4));
  k_node_counts<<<std::min(blocks_for((size_t)c.cap_nodes, 128), 152u * 16u), 128, 0, st>>>(
      key, n, c.prm.leaf_max, ts, P<uint4>(c.cell), P<uint2>(c.range), P<int2>(c.kids));
  note_launch(4);
  return cudaGetLastError();
}

}  // namespace

cudaError_t build_tree(Ctx &c, const double *pos, const float *mass, int64_t n, cudaStream_t st) {
  cudaError_t e;
#define TRY(x)                      \
  do {                              \
    e = (x);                        \
    if (e != cudaSuccess) return e; \
  } while (0)
  c.n = n;
  c.nnodes = c.nleaves = 0;
  c.nlevels = 0;
  c.have_tree = false;
  if (n == 0) {
    c.have_tree = true;
    return cudaSuccess;
  }
  const int T = 256;
  TRY(ensure(c.key, n * 8));
  TRY(ensure(c.key_alt, n * 8));
  TRY(ensure(c.idx, n * 4));
  TRY(ensure(c.idx_alt, n * 4));
  TRY(ensure(c.xs, n * 24));
  TRY(ensure(c.pm4, n * 16));
  TRY(ensure(c.d_small, 256));
  if (c.prm.profile & 1) cudaEventRecord(c.ev[0], st);
  const double inv_pow2 = box_inverse_if_pow2(c.prm.box);
  k_keys<<<blocks_for(n, T), T, 0, st>>>(pos, n, c.prm.box, inv_pow2, P<uint64_t>(c.key), P<uint32_t>(c.idx));
  note_launch();
  bool alt = false;
  TRY(radix_sort_u64(P<uint64_t>(c.key), P<uint32_t>(c.idx), P<uint64_t>(c.key_alt), P<uint32_t>(c.idx_alt), n, 0,
                     63, &alt, c.tmp, st, wait_polls(c, kLookPolls)));
  if (alt) {
    std::swap(c.key, c.key_alt);
    std::swap(c.idx, c.idx_alt);
  }
  if (c.prm.profile & 1) cudaEventRecord(c.ev[1], st);
  // node capacity from the last build, grown to what an overflow asked for
  c.cap_nodes = std::max<uint64_t>(c.cap_nodes, (uint64_t)(2 * n / (c.prm.leaf_max > 1 ? c.prm.leaf_max : 1) + 64));
  TreeState hs{};
  for (int attempt = 0;; ++attempt) {
    if (attempt == 8) return cudaErrorInvalidValue;
    TRY(level_buffers(c, n));
    TRY(levels_launch(c, pos, mass, n, kDepth + 1, st));
    TRY(cudaMemcpyAsync(c.h_pinned, c.tstate.p, sizeof(TreeState), cudaMemcpyDeviceToHost, st));
    TRY(cudaStreamSynchronize(st));
    std::memcpy(&hs, c.h_pinned, sizeof(TreeState));
    if (!hs.overflow) break;
    c.nnodes = (int64_t)hs.total;
    if (hs.total >= (1ull << kSinkBits)) return cudaErrorInvalidValue;  // mapped to HFMM_ERR_CAPACITY
    c.cap_nodes = std::max<uint64_t>(2 * c.cap_nodes, hs.total + hs.total / 2);
  }
  const int64_t total = (int64_t)hs.total;
  c.nlevels = hs.nlevels;
  for (int l = 0; l <= hs.nlevels && l < kDepth + 3; ++l) c.level_start[l] = (int64_t)hs.level_start[l];
  c.nnodes = total;
  c.nleaves = (int64_t)hs.nleaves;
  if (total >= ((int64_t)1 << kSinkBits)) return cudaErrorInvalidValue;  // mapped to HFMM_ERR_CAPACITY
  if (c.prm.profile & 1) cudaEventRecord(c.ev[2], st);
  c.have_tree = true;
  return cudaSuccess;
#undef TRY
}

// Graph mode (a step captured as one graph): every buffer of the build sized
// for n particles and the node capacity (outside the capture) ...
cudaError_t build_tree_prepare(Ctx &c, int64_t n) {
  cudaError_t e;
#define TRY(x)                      \
  do {                              \
    e = (x);                        \
    if (e != cudaSuccess) return e; \
  } while (0)
  TRY(ensure(c.key, n * 8));
  TRY(ensure(c.key_alt, n * 8));
  TRY(ensure(c.idx, n * 4));
  TRY(ensure(c.idx_alt, n * 4));
  TRY(ensure(c.xs, n * 24));
  TRY(ensure(c.pm4, n * 16));
  TRY(ensure(c.tmp, radix_sort_scratch_bytes((size_t)n)));
  c.cap_nodes = std::max<uint64_t>(c.cap_nodes, (uint64_t)(2 * n / (c.prm.leaf_max > 1 ? c.prm.leaf_max : 1) + 64));
  TRY(level_buffers(c, n));
  // levels the graph's level loops cover: the last tree's and two more
  if (c.cap_levels < c.nlevels + 2) c.cap_levels = c.nlevels + 2;
  if (c.cap_levels > kDepth + 1) c.cap_levels = kDepth + 1;
  return cudaSuccess;
#undef TRY
}

// ... and the build enqueued with no read-back: the sizes stay in the device
// state (c.tstate), which the later kernels of the graph read; a node capacity
// overflow shows there too and makes them treat the tree as empty.
cudaError_t build_tree_launch(Ctx &c, const double *pos, const float *mass, int64_t n, cudaStream_t st) {
  cudaError_t e;
  const int T = 256;
  const double inv_pow2 = box_inverse_if_pow2(c.prm.box);
  k_keys<<<blocks_for(n, T), T, 0, st>>>(pos, n, c.prm.box, inv_pow2, P<uint64_t>(c.key), P<uint32_t>(c.idx));
  note_launch();
  bool alt = false;
  if ((e = radix_sort_u64(P<uint64_t>(c.key), P<uint32_t>(c.idx), P<uint64_t>(c.key_alt), P<uint32_t>(c.idx_alt), n,
                          0, 63, &alt, c.tmp, st, wait_polls(c, kLookPolls))) != cudaSuccess)
    return e;
  if (alt) {
    std::swap(c.key, c.key_alt);
    std::swap(c.idx, c.idx_alt);
  }
  return levels_launch(c, pos, mass, n, c.cap_levels, st);
}

// After the graph: the device state's sizes on the host.  False on an overflow
// of the node or level capacity (both are then grown for the next capture).
bool build_tree_finish(Ctx &c, const TreeState &hs) {
  if (hs.overflow) {
    // which limit it was is not recorded: grow both
    c.cap_nodes = std::max<uint64_t>(2 * c.cap_nodes, hs.total + hs.total / 2);
    c.cap_levels = c.cap_levels + 2 > kDepth + 1 ? kDepth + 1 : c.cap_levels + 2;
    return false;
  }
  c.nlevels = hs.nlevels;
  for (int l = 0; l <= hs.nlevels && l < kDepth + 3; ++l) c.level_start[l] = (int64_t)hs.level_start[l];
  c.nnodes = (int64_t)hs.total;
  c.nleaves = (int64_t)hs.nleaves;
  c.have_tree = c.nnodes < ((int64_t)1 << kSinkBits);
  return c.have_tree;
}

}  // namespace hfmm
