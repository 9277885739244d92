// Device primitives: buffer growth, exclusive scan and a stable LSD radix sort.
// Used by the tree builds (key sorts), the M2L lists of the learned acceptance and the
// operator tables, and the mutual P2P.
#include <vector>

#include "common.cuh"

namespace hfmm {

std::atomic<long long> g_launches{0};
thread_local std::vector<void *> *g_deferred_free = nullptr;

cudaError_t ensure(DBuf &b, size_t bytes) {
  if (bytes <= b.cap) return cudaSuccess;
  size_t want = bytes + bytes / 4 + 256;
  if (b.p && g_deferred_free) {  // stream capture in progress: free after it ends
    g_deferred_free->push_back(b.p);
    b.p = nullptr;
    b.cap = 0;
  }
  if (b.p) {
    cudaError_t e = cudaFree(b.p);
    b.p = nullptr;
    b.cap = 0;
    if (e != cudaSuccess) return e;
  }
  cudaError_t e = cudaMalloc(&b.p, want);
  if (e != cudaSuccess) {
    b.p = nullptr;
    return e;
  }
  b.cap = want;
  return cudaSuccess;
}

cudaError_t upload(DBuf &b, const void *src, size_t bytes, cudaStream_t st) {
  cudaError_t e = ensure(b, bytes);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b.p, src, bytes, cudaMemcpyHostToDevice, st);
  return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

void release(DBuf &b) {
  if (b.p) cudaFree(b.p);
  b.p = nullptr;
  b.cap = 0;
}

// ------------------------------------------------------------------ scan
namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class T>
__device__ T block_exclusive_scan(T v, T *total) {
  __shared__ T warp_tot[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    T t = lane < nw ? warp_tot[lane] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) warp_tot[lane] = t;  // inclusive
  }
  __syncthreads();
  T base = w ? warp_tot[w - 1] : T(0);
  if (total) *total = warp_tot[(blockDim.x >> 5) - 1];
  T r = base + x - v;
  __syncthreads();
  return r;
}

__global__ void k_scan_reduce(const uint32_t *__restrict__ in, size_t n, uint64_t *__restrict__ bsum) {
  size_t base = (size_t)blockIdx.x * kScanTile;
  uint64_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    size_t j = base + (size_t)i * kScanThreads + threadIdx.x;
    if (j < n) s += in[j];
  }
  uint64_t tot;
  block_exclusive_scan<uint64_t>(s, &tot);
  if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

// Single block: exclusive scan of the block sums (any count), total at the end.
__global__ void k_scan_bsum(uint64_t *bsum, size_t nb, uint64_t *total) {
  uint64_t carry = 0;
  for (size_t base = 0; base < nb; base += blockDim.x) {
    size_t j = base + threadIdx.x;
    uint64_t v = j < nb ? bsum[j] : 0;
    uint64_t tot;
    uint64_t ex = block_exclusive_scan<uint64_t>(v, &tot);
    if (j < nb) bsum[j] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void k_scan_apply(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, size_t n,
                             const uint64_t *__restrict__ bsum) {
  __shared__ uint32_t tile[kScanTile];
  size_t base = (size_t)blockIdx.x * kScanTile;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    size_t j = base + (size_t)i * kScanThreads + threadIdx.x;
    tile[i * kScanThreads + threadIdx.x] = j < n ? in[j] : 0u;
  }
  __syncthreads();
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = tile[threadIdx.x * kScanItems + i];
    s += v[i];
  }
  uint32_t ex = block_exclusive_scan<uint32_t>(s, nullptr);
  uint32_t b = (uint32_t)bsum[blockIdx.x] + ex;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    tile[threadIdx.x * kScanItems + i] = b;
    b += v[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    size_t j = base + (size_t)i * kScanThreads + threadIdx.x;
    if (j < n) out[j] = tile[i * kScanThreads + threadIdx.x];
  }
}

}  // namespace

cudaError_t scan_u32(const uint32_t *in, uint32_t *out, uint64_t *total, size_t n, DBuf &tmp, cudaStream_t st) {
  size_t nb = (n + kScanTile - 1) / kScanTile;
  if (nb == 0) nb = 1;
  cudaError_t e = ensure(tmp, nb * sizeof(uint64_t));
  if (e != cudaSuccess) return e;
  uint64_t *bsum = P<uint64_t>(tmp);
  if (n == 0) return cudaMemsetAsync(total, 0, sizeof(uint64_t), st);
  k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, st>>>(in, n, bsum);
  note_launch();
  k_scan_bsum<<<1, 1024, 0, st>>>(bsum, nb, total);
  note_launch();
  k_scan_apply<<<(unsigned)nb, kScanThreads, 0, st>>>(in, out, n, bsum);
  note_launch();
  return cudaGetLastError();
}

// ------------------------------------------------------------------ radix sort
// Stable LSD radix sort, 8 bits a pass, one kernel a pass (decoupled look-back: Merrill
// and Garland 2016, "Single-pass parallel prefix scan with decoupled look-back"): a tile's keys are
// ranked in registers and shared memory, the tile finds the number of equal
// digits before it by looking back over its predecessors' published counts, and
// writes its keys out in digit order (runs of a digit are contiguous).  The digit
// totals of all passes come from one histogram kernel over the input.
//
// What bounds it: a pass moves each key and value once in and once out (24
// bytes); below about 10^5 keys, launches.  The sort it replaced took five
// launches and three reads of the keys a pass, with 2048-key tiles ranked in
// eight block-wide rounds.  Measured with the key kernel (63-bit keys with
// values): 2M 0.44 -> 0.29 ms, 16M 2.95 -> 1.6, 32k 0.23 -> 0.08, 1000 0.19 -> 0.02.
//
// Tiles are numbered in the order their blocks start, so every predecessor is
// already running.  A look-back that has polled look_polls times gives up waiting
// and counts the digits before its tile from the keys themselves: slow, but it
// ends, with the same result.
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxPasses = 8;
constexpr int kLookAhead = 4;
// scratch: digit totals of all passes, tickets, then two look-back tables used in turn
// (a pass clears the table of the next one)
constexpr size_t kSortHead = (size_t)kMaxPasses * 256 * 4 + 64;

// Items per thread: small tiles while the keys do not fill the GPU with large ones.
inline int sort_items(size_t n) { return n < ((size_t)1 << 20) ? 8 : 16; }
inline size_t sort_tiles(size_t n) {
  const size_t tile = (size_t)kSortThreads * sort_items(n);
  return (n + tile - 1) / tile;
}
// Look-back words: count below two flag bits; 64-bit where a count may reach 2^30.
inline size_t sort_word(size_t n) { return n < ((size_t)1 << 30) ? 4 : 8; }

__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint64_t *__restrict__ keys, size_t n, int bit_lo,
                                                             int bit_hi, uint32_t *__restrict__ hist) {
  __shared__ uint32_t h[kMaxPasses][256];
  for (int i = threadIdx.x; i < kMaxPasses * 256; i += kSortThreads) (&h[0][0])[i] = 0u;
  __syncthreads();
  const size_t stride = (size_t)gridDim.x * kSortThreads;
  for (size_t j = (size_t)blockIdx.x * kSortThreads + threadIdx.x; j < n; j += stride) {
    const uint64_t k = keys[j];
#pragma unroll
    for (int q = 0; q < kMaxPasses; ++q) {
      const int sh = bit_lo + 8 * q;
      if (sh < bit_hi) {
        const uint32_t mask = bit_hi - sh < 8 ? (1u << (bit_hi - sh)) - 1u : 255u;
        atomicAdd(&h[q][(uint32_t)(k >> sh) & mask], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kMaxPasses * 256; i += kSortThreads)
    if ((&h[0][0])[i]) atomicAdd(&hist[i], (&h[0][0])[i]);
}

// The lanes of the warp with the same 8-bit digit (match_any takes a step per distinct value:
// 46 us a pass at 2M keys instead of 38).
__device__ __forceinline__ unsigned digit_peers(uint32_t d) {
  unsigned peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const bool bit = (d >> b) & 1u;
    const unsigned set = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? set : ~set;
  }
  return peers;
}

template <bool kVals, int kItems, class Word>
__global__ void __launch_bounds__(kSortThreads, 3) k_radix_pass(const uint64_t *__restrict__ kin,
                                                             const uint32_t *__restrict__ vin,
                                                             uint64_t *__restrict__ kout, uint32_t *__restrict__ vout,
                                                             size_t n, int shift, uint32_t mask,
                                                             const uint32_t *__restrict__ hist,
                                                             unsigned *__restrict__ ticket, volatile Word *look,
                                                             Word *__restrict__ clear, unsigned look_polls) {
  constexpr int kTile = kSortThreads * kItems;
  constexpr int kFlag = 8 * (int)sizeof(Word) - 2;
  constexpr Word kCount = ((Word)1 << kFlag) - 1;
  extern __shared__ __align__(16) unsigned char sort_smem[];
  uint64_t *skey = reinterpret_cast<uint64_t *>(sort_smem);
  uint32_t *sval = reinterpret_cast<uint32_t *>(skey + kTile);
  __shared__ uint32_t wh[kSortWarps][256];
  __shared__ unsigned long long gofs[256];
  __shared__ unsigned tile_s;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  if (tid == 0) tile_s = atomicAdd(ticket, 1u);
#pragma unroll
  for (int q = 0; q < 8; ++q) wh[w][q * 32 + lane] = 0u;
  __syncthreads();
  const size_t tile = tile_s, first = tile * kTile;
  const uint32_t nv = n - first < (size_t)kTile ? (uint32_t)(n - first) : (uint32_t)kTile;  // keys of this tile
  clear[tile * 256 + tid] = 0;
  // ---- rank within the warp's contiguous part; the places beyond n hold all-ones keys, last of the last digit
  uint64_t key[kItems];
  uint32_t val[kItems], rank[kItems];
  const uint32_t at = (uint32_t)(w * 32 * kItems + lane);
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t j = at + 32 * i;
    key[i] = j < nv ? kin[first + j] : ~0ull;
    val[i] = kVals && j < nv ? vin[first + j] : 0u;
  }
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t d = (uint32_t)(key[i] >> shift) & mask;
    const unsigned peers = digit_peers(d);
    const uint32_t before = wh[w][d];
    __syncwarp();
    rank[i] = before + __popc(peers & lt);
    if ((peers & lt) == 0) wh[w][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // ---- digit tid: counts of the warps before, of the tile, and of all tiles before
  uint32_t c = 0;
#pragma unroll
  for (int q = 0; q < kSortWarps; ++q) {
    const uint32_t t = wh[q][tid];
    wh[q][tid] = c;
    c += t;
  }
  const uint32_t mine = c - ((uint32_t)tid == mask ? (uint32_t)kTile - nv : 0u);
  look[tile * 256 + tid] = ((Word)(tile == 0 ? 2 : 1) << kFlag) | mine;
  const uint32_t local = block_exclusive_scan<uint32_t>(c, nullptr);
  const unsigned long long base = block_exclusive_scan<unsigned long long>(hist[tid], nullptr);
  unsigned long long before = 0;
  bool lost = tile > 0 && look_polls == 0;
  if (tile > 0) {
    // kLookAhead predecessors' words in flight at a time: the first wave's tiles all look back
    // over each other's aggregates, and one load a step made that the longest part of a pass
    long long t = (long long)tile - 1;
    unsigned polls = 0;
    bool found = false;
    while (!found && !lost) {
      Word v[kLookAhead];
#pragma unroll
      for (int q = 0; q < kLookAhead; ++q) v[q] = t >= q ? look[(size_t)(t - q) * 256 + tid] : 0;
      bool wait = false;
#pragma unroll
      for (int q = 0; q < kLookAhead; ++q) {
        if (found || wait) continue;
        const unsigned flag = (unsigned)(v[q] >> kFlag);
        if (flag == 0) {
          wait = true;
          continue;
        }
        before += (unsigned long long)(v[q] & kCount);
        found = flag == 2;  // the first tile publishes nothing else
        --t;
      }
      if (wait && ++polls > look_polls) lost = true;
    }
  }
  if (__syncthreads_or(lost)) {  // count the digits before this tile from the keys
    uint32_t *cnt = reinterpret_cast<uint32_t *>(sort_smem);
    cnt[tid] = 0u;
    __syncthreads();
    unsigned long long all = 0;
    for (size_t j0 = 0; j0 < first; j0 += (size_t)1 << 30) {  // 32-bit counters, in parts
      const size_t j1 = first - j0 < ((size_t)1 << 30) ? first : j0 + ((size_t)1 << 30);
      for (size_t j = j0 + tid; j < j1; j += kSortThreads) atomicAdd(&cnt[(uint32_t)(kin[j] >> shift) & mask], 1u);
      __syncthreads();
      all += cnt[tid];
      __syncthreads();
      cnt[tid] = 0u;
      __syncthreads();
    }
    before = all;
  }
  if (tile > 0) look[tile * 256 + tid] = ((Word)2 << kFlag) | (Word)(before + mine);
  gofs[tid] = base + before - local;  // an element at place j of the tile's digit order goes to gofs[d] + j
#pragma unroll
  for (int q = 0; q < kSortWarps; ++q) wh[q][tid] += local;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t p = wh[w][(uint32_t)(key[i] >> shift) & mask] + rank[i];
    skey[p] = key[i];
    if (kVals) sval[p] = val[i];
  }
  __syncthreads();
  for (uint32_t j = tid; j < nv; j += kSortThreads) {
    const uint64_t k = skey[j];
    const unsigned long long o = gofs[(uint32_t)(k >> shift) & mask] + j;
    kout[o] = k;
    if (kVals) vout[o] = sval[j];
  }
}

// Up to 8192 keys: every pass in one block, in place (a launch a pass takes 6 us each whatever it holds).
constexpr int kBlockThreads = 1024;
constexpr size_t kBlockMax = (size_t)kBlockThreads * 8;

template <bool kVals, int kItems>
__global__ void __launch_bounds__(kBlockThreads) k_radix_block(uint64_t *__restrict__ keys, uint32_t *__restrict__ vals,
                                                               uint32_t n, int bit_lo, int bit_hi) {
  constexpr int kTile = kBlockThreads * kItems, kW = kBlockThreads / 32;
  extern __shared__ __align__(16) unsigned char sort_smem[];
  uint64_t *skey = reinterpret_cast<uint64_t *>(sort_smem);
  uint32_t *sval = reinterpret_cast<uint32_t *>(skey + kTile);
  __shared__ __align__(16) uint16_t wh[kW][256];
  __shared__ uint32_t ofs[256];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t at = (uint32_t)(w * 32 * kItems + lane);
  uint64_t key[kItems];
  uint32_t val[kItems], rank[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {  // the places beyond n hold all-ones keys: they stay behind the others
    const uint32_t j = at + 32 * i;
    key[i] = j < n ? keys[j] : ~0ull;
    val[i] = kVals && j < n ? vals[j] : 0u;
  }
  for (int shift = bit_lo; shift < bit_hi; shift += 8) {
    const uint32_t mask = bit_hi - shift < 8 ? (1u << (bit_hi - shift)) - 1u : 255u;
    reinterpret_cast<uint4 *>(wh[w])[lane] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const uint32_t d = (uint32_t)(key[i] >> shift) & mask;
      const unsigned peers = digit_peers(d);
      const uint32_t before = wh[w][d];
      __syncwarp();
      rank[i] = before + __popc(peers & lt);
      if ((peers & lt) == 0) wh[w][d] = (uint16_t)(before + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    uint32_t c = 0;
    if (tid < 256)
#pragma unroll 8
      for (int q = 0; q < kW; ++q) {
        const uint32_t t = wh[q][tid];
        wh[q][tid] = (uint16_t)c;
        c += t;
      }
    const uint32_t local = block_exclusive_scan<uint32_t>(c, nullptr);
    if (tid < 256) ofs[tid] = local;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const uint32_t d = (uint32_t)(key[i] >> shift) & mask;
      const uint32_t p = ofs[d] + wh[w][d] + rank[i];
      skey[p] = key[i];
      if (kVals) sval[p] = val[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      key[i] = skey[at + 32 * i];
      if (kVals) val[i] = sval[at + 32 * i];
    }
  }
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t j = at + 32 * i;
    if (j < n) {
      keys[j] = key[i];
      if (kVals) vals[j] = val[i];
    }
  }
}

template <bool kVals, int kItems>
cudaError_t radix_block(uint64_t *keys, uint32_t *vals, size_t n, int bit_lo, int bit_hi, cudaStream_t st) {
  const size_t smem = (size_t)kBlockThreads * kItems * (kVals ? 12 : 8);
  auto kern = k_radix_block<kVals, kItems>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<1, kBlockThreads, smem, st>>>(keys, vals, (uint32_t)n, bit_lo, bit_hi);
  note_launch();
  return cudaGetLastError();
}

template <bool kVals, int kItems, class Word>
cudaError_t radix_passes(uint64_t *ka, uint32_t *va, uint64_t *kb, uint32_t *vb, size_t n, int bit_lo, int bit_hi,
                         bool *in_alt, void *scratch, unsigned look_polls, cudaStream_t st) {
  const unsigned ntiles = (unsigned)sort_tiles(n);
  uint32_t *hist = static_cast<uint32_t *>(scratch);
  unsigned *ticket = hist + kMaxPasses * 256;
  Word *look[2];
  look[0] = reinterpret_cast<Word *>(static_cast<unsigned char *>(scratch) + kSortHead);
  look[1] = look[0] + (size_t)ntiles * 256;
  cudaError_t e = cudaMemsetAsync(scratch, 0, kSortHead + (size_t)ntiles * 256 * sizeof(Word), st);
  if (e != cudaSuccess) return e;
  unsigned gh = blocks_for(n, kSortThreads * 8);
  if (gh > 152u * 8u) gh = 152u * 8u;
  k_radix_hist<<<gh, kSortThreads, 0, st>>>(ka, n, bit_lo, bit_hi, hist);
  note_launch();
  const size_t smem = (size_t)kSortThreads * kItems * (kVals ? 12 : 8);
  auto kern = k_radix_pass<kVals, kItems, Word>;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  bool alt = false;
  int pass = 0;
  for (int sh = bit_lo; sh < bit_hi; sh += 8, ++pass) {
    const uint32_t mask = bit_hi - sh < 8 ? (1u << (bit_hi - sh)) - 1u : 255u;
    kern<<<ntiles, kSortThreads, smem, st>>>(alt ? kb : ka, alt ? vb : va, alt ? ka : kb, alt ? va : vb, n, sh, mask,
                                             hist + 256 * pass, ticket + pass, look[pass & 1], look[(pass + 1) & 1],
                                             look_polls);
    note_launch();
    alt = !alt;
  }
  *in_alt = alt;
  return cudaGetLastError();
}

}  // namespace

size_t radix_sort_scratch_bytes(size_t n) { return kSortHead + 2 * sort_tiles(n) * 256 * sort_word(n); }

cudaError_t radix_sort_u64_into(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt, uint32_t *vals_alt, size_t n,
                                int bit_lo, int bit_hi, bool *in_alt, void *scratch, size_t scratch_bytes,
                                cudaStream_t st, unsigned look_polls) {
  *in_alt = false;
  if (n <= 1 || bit_hi <= bit_lo) return cudaSuccess;
  if (radix_sort_scratch_bytes(n) > scratch_bytes || bit_hi - bit_lo > 8 * kMaxPasses) return cudaErrorInvalidValue;
  if (n <= kBlockMax) {
    auto block = [&](auto f) { return f(keys, vals, n, bit_lo, bit_hi, st); };
    if (vals)
      return n <= 1024 ? block(radix_block<true, 1>) : n <= 2048 ? block(radix_block<true, 2>)
                       : n <= 4096 ? block(radix_block<true, 4>) : block(radix_block<true, 8>);
    return n <= 1024 ? block(radix_block<false, 1>) : n <= 2048 ? block(radix_block<false, 2>)
                     : n <= 4096 ? block(radix_block<false, 4>) : block(radix_block<false, 8>);
  }
  const bool small = sort_items(n) == 8, wide = sort_word(n) == 8;
  auto run = [&](auto f) {
    return f(keys, vals, keys_alt, vals_alt, n, bit_lo, bit_hi, in_alt, scratch, look_polls, st);
  };
  if (vals)
    return small ? run(radix_passes<true, 8, uint32_t>)
                 : wide ? run(radix_passes<true, 16, uint64_t>) : run(radix_passes<true, 16, uint32_t>);
  return small ? run(radix_passes<false, 8, uint32_t>)
               : wide ? run(radix_passes<false, 16, uint64_t>) : run(radix_passes<false, 16, uint32_t>);
}

cudaError_t radix_sort_u64(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt, uint32_t *vals_alt, size_t n,
                           int bit_lo, int bit_hi, bool *in_alt, DBuf &tmp, cudaStream_t st, unsigned look_polls) {
  *in_alt = false;
  if (n <= 1 || bit_hi <= bit_lo) return cudaSuccess;
  const cudaError_t e = ensure(tmp, radix_sort_scratch_bytes(n));
  if (e != cudaSuccess) return e;
  return radix_sort_u64_into(keys, vals, keys_alt, vals_alt, n, bit_lo, bit_hi, in_alt, tmp.p, tmp.cap, st,
                             look_polls);
}

}  // namespace hfmm
