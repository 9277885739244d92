// Cut-off P2P over each sink leaf's P2P list (Sec. 2.1, the pair force
// f_(1)(r) r of Sec. 2.2, kept for 0 < r < R_c), added to the L2P accelerations
// already in the caller's particle order (the un-permute).
//
// One warp per work item: a leaf's first 32 sinks, or the others in chunks of 32 (more
// than one such chunk only for a leaf at the depth cap, which may hold any number of
// particles), taken from a global work counter in longest-first order (k_lpt_hist / k_lpt_place below).
// The source particles of all leaves on the sink's list are streamed through per-warp
// shared memory in fills of up to kCap particles.  A fill takes the next 32
// list entries (a prefix scan of their particle counts gives each candidate
// its slot, an entry cut at the buffer's end continues in the next fill; each
// entry marks its first slot and the marks are carried forward, so every slot
// knows its entry) and copies the candidates' particles asynchronously
// (cp.async) into a raw buffer;
// the next fill's copies are issued before the current fill is evaluated, so
// their latency hides behind the arithmetic.  Once a fill has landed it is
// transformed into the evaluation buffer: moved into the sink leaf's frame (the
// leaf-centre difference is an exact integer in half units), negated, and kept
// only if within R_c of the bounding box of the chunk's sinks (a margin of
// 2^-12 in r^2 keeps every source whose FP32 pair distance could come out
// below R_c; the others contribute nothing).  Lanes are split as (sink i,
// stream s): with cs sinks in the chunk, S = 32 / cs streams walk the buffer,
// so small leaves still keep the warp busy; the streams are added in a fixed
// order at the end (deterministic).  Where S = 32 / cs leaves many lanes idle the
// chunk is split instead: in two halves (19 and 20 sinks) or three thirds (9, 11, 12, 17,
// 18, 21..24), each lane holding one sink of each and evaluating all against every staged
// source pair.  Of the pair evaluations of the 2M set 88% are a sink's with halves alone,
// 93% with thirds: 7.69 -> 7.53 ms; in smaller chunks (3 and 6) the longer final sum takes
// back what thirds give (32k uniform particles, about 8 a leaf: 0.115 instead of 0.113).
//
// The evaluation buffer holds sources in pairs, {-x0, -x1, -y0, -y1}
// {-z0, -z1, -w0, -w1} (w = mass), so each lane evaluates two pairs per step
// with the packed FP32x2 add / multiply / fma of sm_100+ (half the FP32
// instructions; rsqrt and exp2 stay per element).  An odd tail is padded with a
// massless source far outside the cut-off.
//
// Pair force (Gaussian split): a = -m S(x) r / r^3, S(x) = erfc(x/2) + x e^(-x^2/4) / sqrt(pi),
// x = r / r_s, evaluated as in PairFit (common.cuh) and pair_factor2 (p2p_common.cuh).
#include "p2p_common.cuh"

namespace hfmm {
namespace {

// Order of the work items (k_lpt_hist, k_lpt_place): items and work by bucket, placing cursors.
constexpr int kLptBuckets = 64;
constexpr unsigned kLptWarps = 152 * 16;  // warps the GPU holds of k_p2p
constexpr int64_t kLptMin = 512;          // leaves from which the work is ordered
struct LptState {
  unsigned long long work;
  unsigned n_items, pad;
  unsigned hist[kLptBuckets], cursor[kLptBuckets];
};

// What the kernel needs of a tree's nodes: a particle range, and the vector from the sink
// leaf's centre to a source leaf's (Node: what that takes of a node, fetched ahead).
struct OctNodes {
  const uint4 *cell_;
  const uint2 *range_;
  float half_unit;
  using Node = uint4;
  __device__ __forceinline__ uint2 range(uint32_t k) const { return range_[k]; }
  __device__ __forceinline__ Node node(uint32_t k) const { return cell_[k]; }
  __device__ __forceinline__ void offset(const Node &sink, const Node &src, uint32_t s, float &dx, float &dy,
                                         float &dz) const {
    int dd[3];
    half_delta32(sink, src, s, dd);
    dx = (float)dd[0] * half_unit;
    dy = (float)dd[1] * half_unit;
    dz = (float)dd[2] * half_unit;
  }
};
// k-d tree: box centres in FP64, once per entry (this GPU's FP64 rate is low).  A kernel of
// its own that staged entry by entry (about 145 instructions an entry of 32 sources, of 690)
// took 14.2 ms for the 18.7G listed pairs of the 2M set, this one 13.1.
struct KdNodes {
  const uint32_t *first, *count;
  const double *geo;  // [>= 3][cap], the centres first
  int64_t cap;
  double L;
  struct Node {
    double x, y, z;
  };
  __device__ __forceinline__ uint2 range(uint32_t k) const { return make_uint2(first[k], count[k]); }
  __device__ __forceinline__ Node node(uint32_t k) const { return Node{geo[k], geo[cap + k], geo[2 * cap + k]}; }
  __device__ __forceinline__ void offset(const Node &sink, const Node &src, uint32_t s, float &dx, float &dy,
                                         float &dz) const {
    dx = (float)__dsub_rn(__dadd_rn(src.x, (double)shift_component(s, 0) * L), sink.x);
    dy = (float)__dsub_rn(__dadd_rn(src.y, (double)shift_component(s, 1) * L), sink.y);
    dz = (float)__dsub_rn(__dadd_rn(src.z, (double)shift_component(s, 2) * L), sink.z);
  }
};

// kCap: source particles per fill (even); dynamic shared memory: 2 x 8 x kCap float4.
// kSplit 0: the Gaussian truncation S(x) above; 1: the polynomial truncation of
// Sec. 5, a = -m (1/r^3 - 5 / (2 R_c^3) + 3 r^2 / (2 R_c^5)) r, no exp2 and no
// fitted factor (see hfmm_params.split).
template <bool kCount, int kCap, int kSplit, class Nodes>
__global__ void __launch_bounds__(256, 2) k_p2p(const uint32_t *__restrict__ items, Nodes nodes,
                                                const uint32_t *__restrict__ beg, const uint32_t *__restrict__ end,
                                                const uint64_t *__restrict__ lst, const float4 *__restrict__ pm4,
                                                const uint32_t *__restrict__ perm, int64_t n, PairFit2 fit,
                                                float G, float *__restrict__ acc_out,
                                                unsigned long long *__restrict__ ctr,
                                                const LptState *__restrict__ lpt,
                                                const uint32_t *__restrict__ leaves, int64_t n_leaves,
                                                const TreeState *tz) {
  extern __shared__ float4 p2p_smem[];
  __shared__ float4 part[8][32];  // a shared item's sums, by warp and sink
  __shared__ unsigned next_shared, n_shared;
  // work items: a leaf's first 32 sinks, or (bit 31 beside the leaf's index) the others; not ordered
  // (lpt null): two for every leaf, the second possibly empty
  const unsigned nl = lpt ? lpt->n_items : 2u * (unsigned)tree_leaves(tz, n_leaves);
  unsigned *taken = reinterpret_cast<unsigned *>(ctr);  // items handed out: to warps, to blocks
  if (threadIdx.x < 32) {
    // the items heavy enough to be shared: the first buckets, of work (entries x sinks) above half
    // a warp's share of it all, and of at least 2^14 (512 entries of 32 sinks: 64 for each of the
    // eight warps, or the prefetch chain they start with is most of what they do)
    const unsigned long long half = lpt ? max(lpt->work / (2ull * kLptWarps), (1ull << 14) - 1ull) : 0ull;
    unsigned c = 0;
    for (int b = threadIdx.x; lpt && b < kLptBuckets; b += 32)
      if (lpt->hist[b] && (1ull << (63 - b)) > half) c += lpt->hist[b];
    c = __reduce_add_sync(0xffffffffu, c);
    if (threadIdx.x == 0) n_shared = c;
  }
  __syncthreads();
  bool shared_phase = true;
  // per warp: the 32 list entries of the pending fill (first particle, exclusive
  // candidate offset, leaf-centre offset in the sink's frame), each candidate's
  // entry, and the chunk's sink bounding box (lo xyz, hi xyz)
  __shared__ uint32_t e_src[8][32], e_excl[8][32];
  __shared__ float4 e_off[8][32];  // per entry: leaf-centre offset (x, y, z, unused)
  __shared__ uint8_t e_own[8][kCap];
  __shared__ float e_box[8][6];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float4 *raw = p2p_smem + wid * kCap;            // the pending fill, as copied
  float4 *buf = p2p_smem + (8 + wid) * kCap;      // the fill being evaluated, in pairs
  float *bf = reinterpret_cast<float *>(buf);
  const uint32_t raw_s = (uint32_t)__cvta_generic_to_shared(raw);
  // cull threshold: R_c^2 (1 + 2^-12), far above the FP32 rounding of either distance
  const float rc2_cull = fit.rc2 * (1.f + 1.f / 4096.f);
  uint32_t n_in = 0;  // pairs inside the cut-off (profile mode only)
  for (;;) {
    unsigned t = 0;
    if (shared_phase) {  // a block's eight warps take an eighth of the item's list each
      if (threadIdx.x == 0) next_shared = atomicAdd(taken + 1, 1u);
      __syncthreads();
      t = next_shared;
      __syncthreads();
      if (t >= n_shared) {
        shared_phase = false;
        continue;
      }
    } else {
      if (lane == 0) t = n_shared + atomicAdd(taken, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
      if (t >= nl) break;
    }
    const uint32_t item = lpt ? items[t] : leaves[t >> 1] | (t & 1u) << 31, k = item & 0x7fffffffu;
    const typename Nodes::Node ca = nodes.node(k);
    const uint2 r = nodes.range(k);
    uint32_t tb = beg[k], te = end[k];
    if (!shared_phase && tb == te) continue;  // (not ordered: an empty list, another sink batch's)
    if (shared_phase) {
      const uint32_t share = (te - tb + 7u) / 8u;
      tb = min(tb + share * wid, te);
      te = min(tb + share, te);
    }

    // the entry window at q + lane, prefetched in two steps: the list word
    // (fetch_lst, while the previous fill is evaluated), then the source leaf's
    // particle range and centre (fetch_src, while the pending fill lands)
    uint64_t pf_e = 0;
    uint2 pf_rb = make_uint2(0u, 0u);
    typename Nodes::Node pf_cb = ca;
    auto fetch_lst = [&](uint32_t q) {
      if (q + lane < te) pf_e = lst[q + lane];
    };
    auto fetch_src = [&](uint32_t q) {
      if (q + lane < te) {
        const uint32_t b = pair_src(pf_e);
        pf_rb = nodes.range(b);
        pf_cb = nodes.node(b);
      }
    };

    // issue the fill starting at list entry q (the first jq particles of that
    // entry already taken; its window prefetched): tables, async copies;
    // advances (q, jq) and starts fetching the next window; returns the number
    // of candidates
    auto issue = [&](uint32_t &q, uint32_t &jq) -> uint32_t {
      const uint32_t qi = q + lane;
      const bool valid = qi < te;
      uint32_t cnt = 0, first = 0;
      float dx = 0.f, dy = 0.f, dz = 0.f;
      if (valid) {
        nodes.offset(ca, pf_cb, pair_shift(pf_e), dx, dy, dz);
        first = pf_rb.x;
        cnt = pf_rb.y;
      }
      const uint32_t start = lane == 0 ? jq : 0u;
      const uint32_t avail = valid ? cnt - start : 0u;
      uint32_t incl = avail;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t excl = incl - avail;
      e_src[wid][lane] = first + start;
      e_excl[wid][lane] = excl;  // non-decreasing in the lane index
      e_off[wid][lane] = make_float4(dx, dy, dz, 0.f);
      const uint32_t all = __shfl_sync(0xffffffffu, incl, 31);
      const uint32_t tot = all < (uint32_t)kCap ? all : (uint32_t)kCap;
      // candidate p belongs to the last entry whose offset is <= p: each
      // non-empty entry marks its first slot, and the marks are carried forward
      // (kPer slots per lane, then a prefix maximum over the lanes: the entries'
      // offsets increase with the lane)
      constexpr int kPer = kCap / 32;
      uint8_t *own_row = e_own[wid];
#pragma unroll
      for (int i = 0; i < kPer; ++i) own_row[lane * kPer + i] = 0xffu;
      __syncwarp();
      if (avail > 0 && excl < tot) own_row[excl] = (uint8_t)lane;
      __syncwarp();
      {
        uint8_t b[kPer];
        int lastm = -1;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          b[i] = own_row[lane * kPer + i];
          if (b[i] != 0xffu) lastm = b[i];
        }
        int pm = lastm;  // inclusive prefix maximum over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, pm, o);
          if (lane >= o && y > pm) pm = y;
        }
        int cur = __shfl_up_sync(0xffffffffu, pm, 1);  // the mark carried in from the lanes before
        if (lane == 0) cur = -1;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          if (b[i] != 0xffu) cur = b[i];
          b[i] = (uint8_t)cur;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kPer; ++i) own_row[lane * kPer + i] = b[i];
      }
      __syncwarp();
      // the copies, four candidates per lane per step
      for (uint32_t pb = 0; pb < tot; pb += 128) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t p = pb + lane + 32 * u;
          if (p < tot) {
            const int o = own_row[p];
            const uint32_t idx = e_src[wid][o] + (p - e_excl[wid][o]);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(raw_s + 16u * p), "l"(pm4 + idx)
                         : "memory");
          }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      // entries taken whole; an entry cut at the buffer's end continues next time
      const unsigned full = __ballot_sync(0xffffffffu, valid && incl <= (uint32_t)kCap);
      const int nfull = __popc(full);
      const uint32_t pex = __shfl_sync(0xffffffffu, excl, nfull & 31);
      const uint32_t pstart = nfull == 0 ? jq : 0u;
      const bool partial = nfull < 32 && q + nfull < te;
      jq = partial ? pstart + (pex < (uint32_t)kCap ? (uint32_t)kCap - pex : 0u) : 0u;
      q += nfull;
      fetch_lst(q);
      return tot;
    };

    const uint32_t cfirst = r.x + 32u * (item >> 31), cend = item >> 31 ? r.x + r.y : min(cfirst + 32u, r.x + r.y);
    for (uint32_t cbase = cfirst; cbase < cend; cbase += 32) {
      const uint32_t rem = r.x + r.y - cbase;
      const int cs = rem < 32 ? (int)rem : 32;
      // sinks per lane: one of each half or third of the chunk where that leaves fewer
      // lanes idle (S_k streams of ceil(cs / k) lanes, S_k / k the sinks they hold at once)
      const int c2 = (cs + 1) >> 1, c3 = (cs + 2) / 3;
      const int s1 = 32 / cs, s2 = 32 / c2, s3 = 32 / c3;
      const bool two = s2 > 2 * s1;
      const bool three = cs >= 9 && 2 * s3 > 3 * (two ? s2 : 2 * s1);
      const int cl = three ? c3 : two ? c2 : cs;  // sinks per lane group
      const int S = 32 / cl, stream = lane / cl, il = lane % cl;
      const bool active = stream < S;
      const float4 xi = pm4[cbase + il];
      const bool hasb = cl < cs && il + cl < cs, hasc = three && il + 2 * cl < cs;
      const float4 none = make_float4(1e18f, 1e18f, 1e18f, 0.f);
      const float4 xib = hasb ? pm4[cbase + il + cl] : none, xic = hasc ? pm4[cbase + il + 2 * cl] : none;
      const float2 xx = f2(xi.x), xy = f2(xi.y), xz = f2(xi.z);
      const float2 bxx = f2(xib.x), bxy = f2(xib.y), bxz = f2(xib.z);
      const float2 cxx = f2(xic.x), cxy = f2(xic.y), cxz = f2(xic.z);
      {
        float lo0 = xi.x, lo1 = xi.y, lo2 = xi.z, hi0 = xi.x, hi1 = xi.y, hi2 = xi.z;
        auto take = [&](const float4 &v) {
          lo0 = fminf(lo0, v.x);
          lo1 = fminf(lo1, v.y);
          lo2 = fminf(lo2, v.z);
          hi0 = fmaxf(hi0, v.x);
          hi1 = fmaxf(hi1, v.y);
          hi2 = fmaxf(hi2, v.z);
        };
        if (hasb) take(xib);
        if (hasc) take(xic);
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          lo0 = fminf(lo0, __shfl_xor_sync(0xffffffffu, lo0, o));
          lo1 = fminf(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
          lo2 = fminf(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
          hi0 = fmaxf(hi0, __shfl_xor_sync(0xffffffffu, hi0, o));
          hi1 = fmaxf(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
          hi2 = fmaxf(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
        }
        if (lane == 0) {
          e_box[wid][0] = lo0;
          e_box[wid][1] = lo1;
          e_box[wid][2] = lo2;
          e_box[wid][3] = hi0;
          e_box[wid][4] = hi1;
          e_box[wid][5] = hi2;
        }
      }
      float2 ax = f2(0.f), ay = f2(0.f), az = f2(0.f);
      float2 bx = f2(0.f), by = f2(0.f), bz = f2(0.f);
      float2 cx = f2(0.f), cy = f2(0.f), cz = f2(0.f);
      uint32_t q = tb, jq = 0;
      bool pending = q < te;
      fetch_lst(q);
      fetch_src(q);
      uint32_t tot = pending ? issue(q, jq) : 0u;
      while (pending) {
        fetch_src(q);
        // the pending fill has landed: into the sink's frame, cull, pair up
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        uint32_t kept = 0;
        {
          const float bx0 = e_box[wid][0], by0 = e_box[wid][1], bz0 = e_box[wid][2];
          const float bx1 = e_box[wid][3], by1 = e_box[wid][4], bz1 = e_box[wid][5];
          // four candidates per lane per step (independent chains), kept in
          // candidate order
          for (uint32_t pb = 0; pb < tot; pb += 128) {
            float4 v[4];
            int o[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const uint32_t p = pb + lane + 32 * u;
              const uint32_t pc = p < tot ? p : 0u;
              v[u] = raw[pc];
              o[u] = e_own[wid][pc];
            }
            bool keep[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const float4 d = e_off[wid][o[u]];
              v[u].x += d.x;
              v[u].y += d.y;
              v[u].z += d.z;
              const float gx = fmaxf(fmaxf(bx0 - v[u].x, v[u].x - bx1), 0.f);
              const float gy = fmaxf(fmaxf(by0 - v[u].y, v[u].y - by1), 0.f);
              const float gz = fmaxf(fmaxf(bz0 - v[u].z, v[u].z - bz1), 0.f);
              keep[u] = pb + lane + 32 * u < tot && gx * gx + gy * gy + gz * gz <= rc2_cull;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const unsigned kb = __ballot_sync(0xffffffffu, keep[u]);
              if (keep[u]) {
                const uint32_t slot = kept + (uint32_t)__popc(kb & ((1u << lane) - 1u));
                float *a = bf + (slot >> 1) * 8 + (slot & 1);  // pair slot/2: {x0 x1 y0 y1} {z0 z1 w0 w1}
                a[0] = -v[u].x;
                a[2] = -v[u].y;
                a[4] = -v[u].z;
                a[6] = -v[u].w;
              }
              kept += (uint32_t)__popc(kb);
            }
          }
        }
        if ((kept & 1) && lane == 0) {  // pad: massless, far beyond the cut-off
          float *a = bf + (kept >> 1) * 8 + 1;
          a[0] = -1e18f;
          a[2] = -1e18f;
          a[4] = -1e18f;
          a[6] = 0.f;
        }
        __syncwarp();  // the raw buffer and the entry tables are free again
        pending = q < te;
        if (pending) tot = issue(q, jq);  // in flight during the evaluation below
        // the pair force of two staged sources on one sink, added to (sx, sy, sz)
        auto pair2 = [&](float2 px, float2 py, float2 pz, const float4 &A, const float4 &B, float2 &sx, float2 &sy,
                         float2 &sz) {
          const float2 dx = __fadd2_rn(px, make_float2(A.x, A.y));
          const float2 dy = __fadd2_rn(py, make_float2(A.z, A.w));
          const float2 dz = __fadd2_rn(pz, make_float2(B.x, B.y));
          const float2 r2 = pair_r2(dx, dy, dz);
          const bool in0 = in_cutoff(r2.x, fit), in1 = in_cutoff(r2.y, fit);
          if (kCount) n_in += (uint32_t)in0 + (uint32_t)in1;
          // outside (0, R_c) the values below may be inf/NaN; the selects discard them
          float2 f = __fmul2_rn(pair_factor2<kSplit>(r2, fit), make_float2(B.z, B.w));  // w = -m
          f.x = in0 ? f.x : 0.f;
          f.y = in1 ? f.y : 0.f;
          sx = __ffma2_rn(f, dx, sx);
          sy = __ffma2_rn(f, dy, sy);
          sz = __ffma2_rn(f, dz, sz);
        };
        if (active) {
          const int np = (int)((kept + 1) >> 1);
          if (three) {
#pragma unroll 2
            for (int kk = stream; kk < np; kk += S) {
              const float4 A = buf[2 * kk], B = buf[2 * kk + 1];
              pair2(xx, xy, xz, A, B, ax, ay, az);
              pair2(bxx, bxy, bxz, A, B, bx, by, bz);
              pair2(cxx, cxy, cxz, A, B, cx, cy, cz);
            }
          } else if (two) {
#pragma unroll 4
            for (int kk = stream; kk < np; kk += S) {
              const float4 A = buf[2 * kk], B = buf[2 * kk + 1];
              pair2(xx, xy, xz, A, B, ax, ay, az);
              pair2(bxx, bxy, bxz, A, B, bx, by, bz);
            }
          } else {
#pragma unroll 8
            for (int kk = stream; kk < np; kk += S) {
              const float4 A = buf[2 * kk], B = buf[2 * kk + 1];
              pair2(xx, xy, xz, A, B, ax, ay, az);
            }
          }
        }
        __syncwarp();  // the evaluation buffer is rewritten by the next fill
      }
      // add the streams of each sink in a fixed order
      buf[lane] = make_float4(ax.x + ax.y, ay.x + ay.y, az.x + az.y, 0.f);
      buf[32 + lane] = make_float4(bx.x + bx.y, by.x + by.y, bz.x + bz.y, 0.f);
      buf[64 + lane] = make_float4(cx.x + cx.y, cy.x + cy.y, cz.x + cz.y, 0.f);
      __syncwarp();
      if (lane < cs) {
        float sx = 0.f, sy = 0.f, sz = 0.f;
        const int grp = lane < cl ? 0 : lane < 2 * cl ? 1 : 2;
        const int i0 = 32 * grp + lane - grp * cl;  // the sink's slot in the first stream
        for (int s = 0; s < S; ++s) {
          const float4 v = buf[i0 + s * cl];
          sx += v.x;
          sy += v.y;
          sz += v.z;
        }
        if (shared_phase) {
          part[wid][lane] = make_float4(sx, sy, sz, 0.f);
        } else {
          const uint32_t o = perm[cbase + lane];
          acc_out[o] += G * sx;
          acc_out[n + o] += G * sy;
          acc_out[2 * n + o] += G * sz;
        }
      }
      __syncwarp();
      if (shared_phase) {
        __syncthreads();
        if (wid == 0 && lane < cs) {  // the warps' sums in order
          float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            const float4 v = part[w][lane];
            sx += v.x;
            sy += v.y;
            sz += v.z;
          }
          const uint32_t o = perm[cbase + lane];
          acc_out[o] += G * sx;
          acc_out[n + o] += G * sy;
          acc_out[2 * n + o] += G * sz;
        }
        if (cbase + 32u < cend) __syncthreads();  // part is rewritten by the next chunk
      }
    }
  }
  if (kCount) {
    unsigned long long v = n_in;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && v) atomicAdd(ctr + 1, v);
  }
}

// Longest-first order of the work (list scheduling: the persistent grid takes
// items in this order).  Where the heaviest items outweigh a warp's share of the
// whole they set the time however they are ordered: those (k_p2p) are each shared by
// a block's eight warps, an eighth of the list a warp, before the others start:
// 1.40 -> 1.02 ms at 262k clustered particles, 0.91 -> 0.59 at 300k (polynomial
// split), nothing at 2M, where no item is that heavy.  Shared from 2^13: 0.48
// instead of 0.41 ms at 100k uniform; every item above half a share, whatever its
// size: 0.15 instead of 0.115 at 32k.  An item is a leaf's first 32 sinks or its
// others (leaves of 33..64 particles give two, so the heaviest leaves' work is split
// between two warps; the chunks' sums are independent, so the forces do not
// change).  An item's work is about the leaf's list entries times its sinks;
// items are bucketed by the binary order of magnitude of that (coarse buckets
// already give the longest-first schedule its bound, the heaviest single item)
// and placed bucket by bucket, heaviest first.  Leaves with empty lists (other
// sink batches) give no item.  The order within a bucket does not matter: each
// item's sums are its own warp's.
template <class Nodes>
__global__ void k_lpt_hist(const uint32_t *__restrict__ leaves, int64_t nl, Nodes nodes,
                           const uint32_t *__restrict__ beg, const uint32_t *__restrict__ end,
                           uint8_t *__restrict__ bucket, LptState *__restrict__ lpt, const TreeState *tz) {
  __shared__ unsigned h[kLptBuckets];
  unsigned long long work = 0;
  for (int i = threadIdx.x; i < kLptBuckets; i += blockDim.x) h[i] = 0u;
  __syncthreads();
  nl = tree_leaves(tz, nl);
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nl) {
    const uint32_t a = leaves[t];
    const uint32_t ent = end[a] - beg[a], cnt = nodes.range(a).y;
#pragma unroll
    for (uint32_t c = 0; c < 2; ++c) {
      uint8_t b = 0xff;
      if (ent > 0 && 32u * c < cnt) {
        const uint32_t cs = c ? cnt - 32u : min(32u, cnt);
        b = (uint8_t)__clzll((unsigned long long)ent * cs);  // heavier: smaller bucket index
        atomicAdd(&h[b], 1u);
        work += (unsigned long long)ent * cs;
      }
      bucket[2 * t + c] = b;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) work += __shfl_xor_sync(0xffffffffu, work, o);
  if ((threadIdx.x & 31) == 0 && work) atomicAdd(&lpt->work, work);
  __syncthreads();
  for (int i = threadIdx.x; i < kLptBuckets; i += blockDim.x)
    if (h[i]) {
      atomicAdd(&lpt->hist[i], h[i]);
      atomicAdd(&lpt->n_items, h[i]);
    }
}

// Ranks within a block from shared-memory counters, one global reservation per
// (block, bucket): the few heavy buckets take few global atomics.
__global__ void k_lpt_place(const uint32_t *__restrict__ leaves, int64_t nl, const uint8_t *__restrict__ bucket,
                            LptState *__restrict__ lpt, uint32_t *__restrict__ order, const TreeState *tz) {
  __shared__ unsigned base[kLptBuckets], cnt[kLptBuckets];
  for (int i = threadIdx.x; i < kLptBuckets; i += blockDim.x) cnt[i] = 0u;
  if (threadIdx.x == 0) {
    unsigned run = 0;
    for (int i = 0; i < kLptBuckets; ++i) {
      base[i] = run;
      run += lpt->hist[i];
    }
  }
  __syncthreads();
  nl = tree_leaves(tz, nl);
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = t < nl;
  uint8_t b[2] = {0xff, 0xff};
  unsigned local[2] = {0u, 0u};
  if (valid) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      b[c] = bucket[2 * t + c];
      if (b[c] != 0xff) local[c] = atomicAdd(&cnt[b[c]], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kLptBuckets; i += blockDim.x)
    if (cnt[i]) base[i] += atomicAdd(&lpt->cursor[i], cnt[i]);
  __syncthreads();
  if (valid) {
    const uint32_t a = leaves[t];
#pragma unroll
    for (int c = 0; c < 2; ++c)
      if (b[c] != 0xff) order[base[b[c]] + local[c]] = a | ((uint32_t)c << 31);
  }
}

template <class Nodes>
cudaError_t run_p2p(Ctx &c, const Nodes &nodes, float *acc, cudaStream_t st) {
  if (c.nleaves == 0) return cudaSuccess;
  const int T = 256;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int per_sm = c.prm.tile_p2p_blocks > 0 ? c.prm.tile_p2p_blocks : 8;
  unsigned g = (unsigned)(nsm * per_sm);
  if ((size_t)g * 8 > (size_t)c.nleaves) g = blocks_for(c.nleaves, c.nleaves < kLptMin ? 4 : 8);
  const bool small = c.prm.tile_p2p_stage == 128, count = (c.prm.profile & 2) != 0;
  auto kern = c.prm.split == 1
                  ? (count ? (small ? k_p2p<true, 128, 1, Nodes> : k_p2p<true, 256, 1, Nodes>)
                           : (small ? k_p2p<false, 128, 1, Nodes> : k_p2p<false, 256, 1, Nodes>))
                  : (count ? (small ? k_p2p<true, 128, 0, Nodes> : k_p2p<true, 256, 0, Nodes>)
                           : (small ? k_p2p<false, 128, 0, Nodes> : k_p2p<false, 256, 0, Nodes>));
  // d_small[3] = work counter, d_small[4] = in-cut-off pair count (zeroed earlier when profiling)
  unsigned long long *ctr = reinterpret_cast<unsigned long long *>(P<uint64_t>(c.d_small) + 3);
  const PairFit2 fit2 = pair_fit2(c);  // the context's fit as packed operand pairs
  // two buffers (raw copies, evaluation pairs) of kCap float4 per warp
  const size_t dyn = (size_t)2 * 8 * (small ? 128 : 256) * sizeof(float4);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctr, 0, 8, st);
  if (e != cudaSuccess) return e;
  // The leaves longest first; below kLptMin each has a warp to itself at once whatever the
  // order: two launches less, 1000 uniform particles 162 -> 150 us a call.  No item is shared
  // by a block there: its work of 2^14 takes 512 entries, more than the leaves unless some
  // occur under several shifts (a cut-off near half the box).
  const TreeState *tz = c.graph_tree ? P<TreeState>(c.tstate) : nullptr;
  LptState *lpt = nullptr;
  if (c.nleaves >= kLptMin) {
    if ((e = ensure(c.lpt_order, (size_t)c.nleaves * 8)) != cudaSuccess) return e;
    if ((e = ensure(c.lpt_tmp, (size_t)c.nleaves * 2 + sizeof(LptState))) != cudaSuccess) return e;
    lpt = P<LptState>(c.lpt_tmp);
    uint8_t *bucket = reinterpret_cast<uint8_t *>(lpt + 1);
    if ((e = cudaMemsetAsync(lpt, 0, sizeof(LptState), st)) != cudaSuccess) return e;
    k_lpt_hist<<<blocks_for(c.nleaves, T), T, 0, st>>>(P<uint32_t>(c.leaves), c.nleaves, nodes,
                                                        P<uint32_t>(c.p2p_beg), P<uint32_t>(c.p2p_end), bucket, lpt, tz);
    k_lpt_place<<<blocks_for(c.nleaves, T), T, 0, st>>>(P<uint32_t>(c.leaves), c.nleaves, bucket, lpt,
                                                         P<uint32_t>(c.lpt_order), tz);
    note_launch(2);
  }
  kern<<<g, T, dyn, st>>>(P<uint32_t>(c.lpt_order), nodes, P<uint32_t>(c.p2p_beg), P<uint32_t>(c.p2p_end),
                        P<uint64_t>(c.p2p), P<float4>(c.pm4), P<uint32_t>(c.idx), c.n, fit2, (float)c.prm.G, acc, ctr, lpt,
                        P<uint32_t>(c.leaves), c.nleaves, tz);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t p2p_pass(Ctx &c, float *acc, cudaStream_t st) {
  if (c.prm.tree == 1)
    return run_p2p(c, KdNodes{P<uint32_t>(c.kd.first), P<uint32_t>(c.kd.count), P<double>(c.kd.geo), c.kd.cap, c.prm.box},
                   acc, st);
  return run_p2p(c, OctNodes{P<uint4>(c.cell), P<uint2>(c.range), (float)c.prm.box / (float)kHalfBox}, acc, st);
}

}  // namespace hfmm
