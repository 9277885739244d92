// Dual-tree traversal with the hybrid multipole acceptance criterion (Sec. 2.3):
//  1. skip a cell pair whose minimum separation S_m exceeds the cut-off R_c;
//  2. accept M2L when theta = L / S_c <= theta_MAC, otherwise open the larger
//     cell (both on a tie; the other one when the larger is a leaf);
//  3. always open pairs in the transition region (S_c > R_c >= S_m as printed,
//     or S_max > R_c >= S_m with transition_rule 1).
// Two leaves that are not accepted become a P2P pair.  Distances are exact
// integers in half units (L / 2^22); the comparisons use one FP64 product each,
// so the decisions are reproducible bit for bit.
//
// The walk is sink-driven: a warp takes one sink cell and the cells its parent
// left open, and decides every pair of the sink in one session (k_walk below).
//
// The conventional walk (interaction counts of Sec. 3) applies rule 2 alone,
// with no cut-off skip and no transition region, from the single root pair of
// the primary box (shift index 13) instead of the 27 nearest periodic images.
//
// Learned acceptance (mac_mode 1) keeps rules 1 and 3 and the self-pair rule;
// in place of rule 2 a pair whose larger side satisfies L / S_c <= theta (the
// safety bound) is a candidate: its 12 features go through the network
// (mlp.cuh, tensor-core inference, batches of 16 candidates per warp) and the
// class chooses between opening the pair and M2L at an order q = 2..p.
// Collection mode records a hash-sampled subset of candidates while opening
// every pair (training data for the network).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "mlp.cuh"

namespace cg = cooperative_groups;

namespace hfmm {
namespace {

enum : uint8_t { kSkip = 0, kM2L = 1, kP2P = 2, kOpen = 3 };

struct Mac {
  int64_t rc2i;                 // floor of (R_c in half units)^2
  int64_t acc_thr[kDepth + 1];  // accept iff S_c^2 >= acc_thr[level of the larger cell]
  int rule, size_rule;
  int mode;   // 0 geometric, 1 learned, 2 collect
  int conv;   // 1: conventional acceptance (rule 2 alone, primary box only)
  int order;  // p (geometric M2L order, and the largest learned order)
  int tab_k;  // operator-table half extent (0: no table)
  int mutual; // 1: keep a P2P pair only as (A, B, s) with A < B, or A = B and s <= 13
  // learned / collect
  const __nv_bfloat16 *w;
  const float *M;
  const uint2 *range;
  int ldm;
  float inv_rs_h, inv_rc_h;
  uint64_t *cand;
  unsigned long long *ncand;
  uint64_t cand_cap;
  uint32_t sample_mod;
};

__device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x ^= x >> 30;
  x *= 0xbf58476d1ce4e5b9ull;
  x ^= x >> 27;
  x *= 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

// ------------------------------------------------------------------ node records
// One 16-byte load per node of everything a decision needs: centre in half units
// (below 2^22) with the level above it in x and the child count in y, and the first child.
struct Node {
  int x, y, z;       // centre, half units
  uint32_t lev, nk;  // level, children (0: leaf)
  uint32_t first;    // first child
};
__device__ __forceinline__ uint4 pack_node(uint4 c, int2 k) {
  const uint32_t l = kDepth - c.w;
  return make_uint4(((2u * c.x + 1u) << l) | (c.w << 22), ((2u * c.y + 1u) << l) | ((uint32_t)k.y << 22),
                    (2u * c.z + 1u) << l, (uint32_t)k.x);
}
__device__ __forceinline__ Node unpack_node(uint4 r) {
  return Node{(int)(r.x & 0x3fffffu), (int)(r.y & 0x3fffffu), (int)r.z, r.x >> 22, r.y >> 22, r.w};
}

// Rules 1 to 3 on the pair (a, b shifted by s) in exact integers.
__device__ __noinline__ int classify_exact(const Node &a, const Node &b, uint32_t s, const Mac &m) {
  // s / 9 and s / 3 for s < 27 by multiplication
  const uint32_t s9 = (s * 57u) >> 9, s3 = (s * 11u) >> 5;
  const int d[3] = {b.x - a.x + ((int)s9 - 1) * (int)kHalfBox, b.y - a.y + ((int)(s3 - 3u * s9) - 1) * (int)kHalfBox,
                    b.z - a.z + ((int)(s - 3u * s3) - 1) * (int)kHalfBox};
  const int ext = (1 << (kDepth - a.lev)) + (1 << (kDepth - b.lev));
  int64_t sc2 = 0, sm2 = 0, sx2 = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int v = d[q] < 0 ? -d[q] : d[q];
    const int g = v - ext > 0 ? v - ext : 0;
    const int f = v + ext;
    sc2 += (int64_t)v * v;
    sm2 += (int64_t)g * g;
    sx2 += (int64_t)f * f;
  }
  if (!m.conv && sm2 > m.rc2i) return kSkip;
  const bool trans = !m.conv && (m.rule == 0 ? sc2 > m.rc2i : sx2 > m.rc2i);
  const uint32_t lv = m.size_rule == 0 ? b.lev : (a.lev < b.lev ? a.lev : b.lev);  // level of the cell setting L
  return !trans && sc2 >= m.acc_thr[lv] ? kM2L : kOpen;  // thresholds >= 1: self pairs open
}

// The same decisions from FP32 wherever that is certain.  Centres, half widths,
// differences, gaps and spans are integers below 2^24, exact in FP32.  A sum of
// three of their squares is exact too while it stays below 2^24 units (the
// smaller half width squared), else within 3 2^-24 of its value: then a
// comparison against a threshold less than 2^-20 away takes the integers (a few
// in a million).  The thresholds are rounded so that comparing an exact sum with
// them is comparing it with the integers: R_c^2 down (sum > R_c^2), the
// acceptance bounds up (sum >= bound).  The conventional walk has no cut-off:
// its R_c is infinite.
struct MacF {
  float rc, rc_eps;
  float2 acc[kDepth + 1];  // acc_thr by level, and its margin
  float4 shift[27];        // periodic shift in half units
};
__device__ __forceinline__ void mac_f(const Mac &m, MacF &f) {  // by the first threads of a block
  const int t = threadIdx.x;
  if (t == 0) {
    f.rc = m.conv ? 3e38f : __ll2float_rd(m.rc2i);
    f.rc_eps = m.conv ? 0.f : f.rc * 0x1p-20f;
  }
  if (t <= kDepth) {
    const float v = __ll2float_ru(m.acc_thr[t]);
    f.acc[t] = make_float2(v, v * 0x1p-20f);
  }
  if (t < 27)
    f.shift[t] = make_float4(shift_component(t, 0) * (float)kHalfBox, shift_component(t, 1) * (float)kHalfBox,
                             shift_component(t, 2) * (float)kHalfBox, 0.f);
}
// kM2L, kOpen or kSkip; r: the source's record, c: 2^23 + the sink's centre, wa: its half width
__device__ __forceinline__ int classify(const Node &a, uint4 r, uint32_t s, const Mac &m, const MacF &f, float3 c,
                                        float wa) {
  // integers below 2^22 as floats: 2^23 + v has v as its low mantissa bits
  auto num = [](uint32_t v) { return __uint_as_float((v & 0x3fffffu) | 0x4b000000u); };
  const float4 sh = f.shift[s];
  const float dx = fabsf((num(r.x) - c.x) + sh.x), dy = fabsf((num(r.y) - c.y) + sh.y),
              dz = fabsf((num(r.z) - c.z) + sh.z);
  const float wb = __uint_as_float(0x4a000000u - ((r.x >> 22) << 23)), ext = wa + wb;  // half widths 2^(21 - level)
  const float gx = fmaxf(dx - ext, 0.f), gy = fmaxf(dy - ext, 0.f), gz = fmaxf(dz - ext, 0.f);
  const float fx = dx + ext, fy = dy + ext, fz = dz + ext;
  const float sc2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz)), sm2 = fmaf(gx, gx, fmaf(gy, gy, gz * gz));
  const float sx2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz)), tr = m.rule == 0 ? sc2 : sx2;
  const uint32_t lb = r.x >> 22, lv = m.size_rule == 0 ? lb : (a.lev < lb ? a.lev : lb);
  const float2 thr = f.acc[lv];
  const float w = fminf(wa, wb);
  const bool near = fabsf(sm2 - f.rc) <= f.rc_eps || fabsf(tr - f.rc) <= f.rc_eps || fabsf(sc2 - thr.x) <= thr.y;
  if (near && sx2 >= 16777216.f * (w * w)) return classify_exact(a, unpack_node(r), s, m);
  return sm2 > f.rc ? kSkip : (tr <= f.rc && sc2 >= thr.x) ? kM2L : kOpen;
}

// An M2L pair outside the operator table: cells of different levels, or a
// cell offset beyond the table's extent in some axis.
__device__ __forceinline__ bool table_miss(const Node &a, const Node &b, uint32_t s, int k) {
  if (k == 0 || a.lev != b.lev) return true;
  const uint32_t s9 = (s * 57u) >> 9, s3 = (s * 11u) >> 5;
  const int dx = b.x - a.x + ((int)s9 - 1) * (int)kHalfBox, dy = b.y - a.y + ((int)(s3 - 3u * s9) - 1) * (int)kHalfBox,
            dz = b.z - a.z + ((int)(s - 3u * s3) - 1) * (int)kHalfBox;
  const int lim = (2 << (kDepth - a.lev)) * k;  // k cell sides
  return dx > lim || dx < -lim || dy > lim || dy < -lim || dz > lim || dz < -lim;
}

// The walk's state on the device, read back once after the launch.
struct TravState {
  unsigned long long nm2l, np2p, nopen;  // entries asked for (beyond a capacity: counted, not written)
  unsigned long long items;              // cell pairs classified
  unsigned next, tail;                   // queue of cells with children: tickets handed out, cells put in
  int cells_left;                        // cells put in and not finished
  unsigned leaf_next;                    // leaves handed out
  int overflow;                          // the largest of 1: a list did not fit, 3: the tree did not, 4: a wait gave up
  int ovf_lists;                         // bit 0 M2L, 1 P2P, 2 open lists
  int levels;                            // levels of the deepest pair, less one
};

struct WalkArgs {
  const uint4 *cell;
  const int2 *kids;
  const uint32_t *leaves;
  const TreeState *tree;
  uint4 *wn;                             // node records
  uint2 *wf;                             // network: per node its features as BF16 (count, dipole; quadrupole)
  uint32_t *obeg, *ocnt;                 // per node: its parent's open list
  uint32_t *open;                        // open lists: (node to visit or its first child) << 5 | shift
  uint8_t *openc;                        //   and how many nodes from there
  uint64_t *m2l, *p2p;
  uint32_t *mb, *me, *mm, *pb, *pe;      // CSR bounds by sink
  unsigned long long cap_open, cap_m2l, cap_p2p;
  TravState *st;
  uint32_t *queue;                       // cells with children whose parent is done, + 1 (0: not there yet)
  uint32_t *spill;                       // per warp: staged entries beyond the stage
  long long leaf_lo, leaf_hi;            // a batch of leaves, by position in `leaves`
  int what;                              // kWalkAll, kWalkCells, kWalkLeaves
  unsigned polls;                        // of a node's slot before the wait gives up
};

enum : int { kWalkAll = 0, kWalkCells = 1, kWalkLeaves = 2 };

constexpr int kTT = 256;  // threads of the walk
constexpr int kTW = kTT / 32;
constexpr int kCand = 320;   // candidates waiting: up to 63 and 8 children of each of 32 nodes
constexpr int kStack = 512;  // nodes a leaf's walk has still to visit
constexpr int kStage = 480;  // entries staged in shared memory
constexpr int kSpillP = 4096, kSpillM = 2048;  // entries a warp can put aside in memory
constexpr size_t kSpillBytes = (size_t)(kSpillP + kSpillM) * 5;
constexpr unsigned kWaitPolls = 1u << 22;  // about a microsecond each
template <bool kNet>
struct WalkSize {
  static constexpr int kNetWait = kNet ? 64 : 0;  // candidates waiting for the network
  static constexpr int kWarpBytes = (kCand + kNetWait) * 4 + (kStack + kStage) * 5;
};

// A block's shared memory for a cell's session.
struct BlockMem {
  unsigned long long base_m, base_p;
  uint32_t cnt_m[kTW], cnt_p[kTW], fit, put, at, cell;
  uint32_t lost;  // a wait gave up
};

// A warp's shared memory.
struct WarpMem {
  uint32_t *cand, *net, *stack, *stage;
  uint8_t *stackc, *aux;
};

// One sink's session: every pair (sink, b, s) whose parent pair opened is
// classified; its M2L and P2P entries, and for a cell with children the open list
// its children start from, go to contiguous ranges of the lists.  A leaf is one
// warp's, a cell with children a block's (kLeaf false): each warp takes an eighth
// of the parent's list, and the entries go in warp order.
//
// Candidates come from the parent's open list (the root: its 27 images, or
// itself alone in the conventional walk), and for a leaf sink also from the
// nodes its own pairs open, kept on a stack: a leaf's walk ends in its session.
// A pair opens the sink when the sink has children and the source when it has:
// the levels are equal while both have (each opening takes both down), so
// "the larger cell" of rule 2 is both cells, or the one that is not a leaf.
//
// The entries are staged in shared memory, put aside in memory when the stage is
// full, and their ranges taken with one atomic per list at the end; a session
// with more entries than both hold counts them and walks a second time, writing
// in place.  With the network, pairs that wait for its decision are collected
// until 32 of them fill its two 16-row tiles.
template <bool kNet, bool kLeaf>
__device__ __forceinline__ void walk_sink(const WalkArgs &A, const Mac &m, const MacF &mf, uint32_t sink,
                                          const Node &a, const WarpMem &W, BlockMem &B, uint32_t *spill,
                                          const uint32_t *sw, __nv_bfloat16 *xs, uint8_t *dec,
                                          unsigned long long &items, uint32_t &maxlev) {
  // above kSoft waiting: one node at a time, at most 7 more per level; one refill from the list fits below it
  constexpr int kSoft = kStack - 8 * kDepth;
  static_assert(kSoft >= kCand, "a round of candidates that all open must fit the stack");
  constexpr int kU = kNet ? 1 : 2;  // candidates a lane takes per round
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const int wp = threadIdx.x >> 5;
  maxlev = a.lev > maxlev ? a.lev : maxlev;
  uint32_t pbeg = A.obeg[sink], pend = pbeg + A.ocnt[sink];
  if (!kLeaf) {
    const uint32_t share = (pend - pbeg + kTW - 1) / kTW;
    pbeg = min(pbeg + share * wp, pend);
    pend = min(pbeg + share, pend);
  }
  const float3 ctr = make_float3(8388608.f + (float)a.x, 8388608.f + (float)a.y, 8388608.f + (float)a.z);
  const float wa = (float)(1 << (kDepth - a.lev));
  uint32_t *spill_p = spill, *spill_m = spill + kSpillP;
  uint8_t *saux_p = reinterpret_cast<uint8_t *>(spill + kSpillP + kSpillM), *saux_m = saux_p + kSpillP;
  uint32_t fa = 0;  // the sink's count feature
  if (kNet) fa = A.wf[sink].x & 0xffffu;
  unsigned long long base_m = 0, base_p = 0;
  bool fit_m = false, fit_p = false;
  uint32_t cm = 0, cp = 0;  // M2L entries; P2P entries of a leaf, open entries of a cell with children
  for (int pass = 0; pass < 2; ++pass) {
    uint32_t nc = 0, nn = 0, pi = pbeg, om = 0, op = 0;  // om, op: entries put aside
    int sp = 0;
    bool over = false;
    cm = cp = 0;
    __syncwarp();
    if (sink == 0 && (kLeaf || wp == 0)) {
      nc = m.conv ? 1u : 27u;
      if (lane < (int)nc) W.cand[lane] = m.conv ? 13u : (uint32_t)lane;
    }
    __syncwarp();
    for (;;) {
      // ---- refill: nodes of the stack first (depth first), then the parent's open list
      const bool tight = sp + (int)(nc + nn) > kSoft;
      if ((tight ? nc + nn == 0 : nc < 32 * kU) && (sp > 0 || pi < pend)) {
        uint32_t e = 0, cnt = 0;
        if (sp > 0) {
          int k = (kSoft - sp - (int)(nc + nn)) / 7;
          k = k < 1 ? 1 : k > 32 ? 32 : k;
          if (k > sp) k = sp;
          if (lane < k) {
            e = W.stack[sp - k + lane];
            cnt = W.stackc[sp - k + lane];
          }
          sp -= k;
        } else {
          if (pi + lane < pend) {
            e = A.open[pi + lane];
            cnt = A.openc[pi + lane];
          }
          pi += 32;
          if (pi > pend) pi = pend;
        }
        uint32_t inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += y;
        }
        const uint32_t at = nc + inc - cnt;
        nc += __shfl_sync(0xffffffffu, inc, 31);
        for (uint32_t q = 0; q < cnt; ++q) W.cand[at + q] = e + (q << 5);
        __syncwarp();
        continue;
      }
      // ---- one round: candidates to classify (both node records in flight), or pairs for the network
      const bool ask = kNet && (nn >= 32 || (nc == 0 && nn > 0));
      if (nc == 0 && !ask) break;
      uint32_t *from = ask ? W.net : W.cand;
      uint32_t &left = ask ? nn : nc;
      const uint32_t n0 = left > 32 * kU ? left - 32 * kU : 0, n1 = left;
      left = n0;
      uint32_t en[kU];
      uint4 rec[kU];
      bool va[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const uint32_t j = n0 + 32 * u + lane;
        va[u] = j < n1;
        en[u] = va[u] ? from[j] : 0u;
        rec[u] = va[u] ? A.wn[en[u] >> 5] : make_uint4(0u, 0u, 0u, 0u);
      }
      if (pass == 0 && !ask) items += n1 - n0;
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const uint32_t src = en[u] >> 5, s = en[u] & 31u;
        const uint32_t lev_b = rec[u].x >> 22, nk_b = rec[u].y >> 22;
        int c = kSkip;
        uint32_t order = (uint32_t)m.order;
        if (kNet && ask) {
          __syncwarp();
          if (va[0]) {
            __nv_bfloat16 *row = xs + lane * 16;
            float ft[kMlpIn];
            const Node nb = unpack_node(rec[0]);
            const uint32_t s9 = (s * 57u) >> 9, s3 = (s * 11u) >> 5;  // s / 9, s / 3
            const int dd[3] = {nb.x - a.x + ((int)s9 - 1) * (int)kHalfBox,
                               nb.y - a.y + ((int)(s3 - 3u * s9) - 1) * (int)kHalfBox,
                               nb.z - a.z + ((int)(s - 3u * s3) - 1) * (int)kHalfBox};
            pair_shape_features(dd, a.lev, nb.lev, m.inv_rs_h, m.inv_rc_h, ft);
            const uint2 fb = A.wf[src];
            uint32_t w[8];
#pragma unroll
            for (int k = 0; k < 3; ++k) w[k] = pack_bf16(ft[2 * k], ft[2 * k + 1]);
            w[3] = (pack_bf16(ft[6], 0.f) & 0xffffu) | fa << 16;
            w[4] = fb.x;
            w[5] = (fb.y & 0xffffu) | pack_bf16(0.f, ft[11]);
            w[6] = w[7] = 0u;
            reinterpret_cast<uint4 *>(row)[0] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4 *>(row)[1] = make_uint4(w[4], w[5], w[6], w[7]);
          } else {
            reinterpret_cast<uint4 *>(xs + lane * 16)[0] = make_uint4(0u, 0u, 0u, 0u);
            reinterpret_cast<uint4 *>(xs + lane * 16)[1] = make_uint4(0u, 0u, 0u, 0u);
          }
          __syncwarp();
          for (uint32_t bt = 0; bt < n1 - n0; bt += 16) {
            float l[4];
            mlp_logits16(sw, xs + bt * 16, l);
            int c0, c8;
            mlp_argmax16(l, c0, c8);
            if ((lane & 3) == 0) {
              dec[bt + (lane >> 2)] = (uint8_t)c0;
              dec[bt + (lane >> 2) + 8] = (uint8_t)c8;
            }
          }
          __syncwarp();
          if (va[0]) {
            const uint32_t k = dec[lane];
            c = k == 0 ? kOpen : kM2L;
            if (k) order = k + 1u < order ? k + 1u : order;
          }
        } else if (va[u]) {
          c = classify(a, rec[u], s, m, mf, ctr, wa);
          maxlev = lev_b > maxlev ? lev_b : maxlev;
          if (c == kM2L && m.mode == 2) {  // collecting candidates: sampled by a hash, every pair opened
            const uint64_t e = pack_pair(sink, src, s);
            if (pass == 0 && mix64(e) % m.sample_mod == 0) {
              const unsigned long long q = atomicAdd(m.ncand, 1ull);
              if (q < m.cand_cap) m.cand[q] = e;
            }
            c = kOpen;
          }
        }
        if (kNet && !ask) {  // what rule 2 would accept waits for the network
          const unsigned want = __ballot_sync(0xffffffffu, c == kM2L);
          if (c == kM2L) {
            W.net[nn + __popc(want & lt)] = en[u];
            c = kSkip;
          }
          nn += __popc(want);
        }
        if (kLeaf && c == kOpen && nk_b == 0) {
          c = kP2P;
          // mutual P2P: of the mirror pairs (a, b, s) and (b, a, 26 - s) the walk meets
          // both (it is symmetric under size_rule 1); keep one
          if (m.mutual && !p2p_owner(sink, src, s, a.lev, lev_b)) c = kSkip;
        }
        const unsigned mm = __ballot_sync(0xffffffffu, c == kM2L), mo = __ballot_sync(0xffffffffu, c == kOpen);
        // a node to visit: its children, or a leaf source itself
        const uint32_t next = nk_b ? (rec[u].w << 5) | s : en[u];
        const uint8_t nnext = nk_b ? (uint8_t)nk_b : 1;
        unsigned side = mo;  // entries of the second list
        if (kLeaf) {
          if (c == kOpen) {
            const int at = sp + __popc(mo & lt);
            W.stack[at] = next;
            W.stackc[at] = nnext;
          }
          sp += __popc(mo);
          side = __ballot_sync(0xffffffffu, c == kP2P);
        }
        const bool second = kLeaf ? c == kP2P : c == kOpen;
        const uint32_t im = cm + __popc(mm & lt), ip = cp + __popc(side & lt);
        const uint32_t m1 = cm + __popc(mm), p1 = cp + __popc(side);
        if (pass == 0) {
          if (!over && m1 - om + p1 - op > (uint32_t)kStage) {  // put the staged entries aside
            over = cm > (uint32_t)kSpillM || cp > (uint32_t)kSpillP;
            __syncwarp();
            if (!over) {
              for (uint32_t i = lane; i < cp - op; i += 32) {
                spill_p[op + i] = W.stage[i];
                if (!kLeaf) saux_p[op + i] = W.aux[i];
              }
              for (uint32_t i = lane; i < cm - om; i += 32) {
                spill_m[om + i] = W.stage[kStage - 1 - i];
                saux_m[om + i] = W.aux[kStage - 1 - i];
              }
              om = cm;
              op = cp;
            }
            __syncwarp();
          }
          if (!over) {  // P2P or open entries from the front, M2L from the back
            if (c == kM2L) {
              const uint32_t miss = m.tab_k == 0 || table_miss(a, unpack_node(rec[u]), s, m.tab_k) ? 1u : 0u;
              W.stage[kStage - 1 - (im - om)] = en[u];
              W.aux[kStage - 1 - (im - om)] = (uint8_t)(order | (miss << 7));
            } else if (second) {
              W.stage[ip - op] = kLeaf ? en[u] : next;
              if (!kLeaf) W.aux[ip - op] = nnext;
            }
          }
        } else {
          if (c == kM2L && fit_m) {
            const uint64_t miss = table_miss(a, unpack_node(rec[u]), s, m.tab_k) ? 1ull : 0ull;
            A.m2l[base_m + im] = pack_pair(sink, 0, 0, order - 1u) | en[u] | (miss << kGenericBit);
          } else if (second && fit_p) {
            if (kLeaf) {
              A.p2p[base_p + ip] = pack_pair(sink, 0, 0) | en[u];
            } else {
              A.open[base_p + ip] = next;
              A.openc[base_p + ip] = nnext;
            }
          }
        }
        cm = m1;
        cp = p1;
      }
      __syncwarp();
    }
    if (pass == 1) break;
    // ---- the entries' ranges: this warp's begin at base_m, base_p
    if (kLeaf) {
      unsigned long long bm = 0, bp = 0;
      if (lane == 0) {
        if (cm) bm = atomicAdd(&A.st->nm2l, (unsigned long long)cm);
        if (cp) bp = atomicAdd(&A.st->np2p, (unsigned long long)cp);
      }
      base_m = __shfl_sync(0xffffffffu, bm, 0);
      base_p = __shfl_sync(0xffffffffu, bp, 0);
      fit_m = cm > 0 && base_m + cm <= A.cap_m2l;
      fit_p = cp > 0 && base_p + cp <= A.cap_p2p;
      if (lane == 0) {
        if (fit_m) {
          A.mb[sink] = A.mm[sink] = (uint32_t)base_m;
          A.me[sink] = (uint32_t)(base_m + cm);
        }
        if (fit_p) {
          A.pb[sink] = (uint32_t)base_p;
          A.pe[sink] = (uint32_t)(base_p + cp);
        }
        if ((cm && !fit_m) || (cp && !fit_p)) {
          atomicOr(&A.st->ovf_lists, (cm && !fit_m ? 1 : 0) | (cp && !fit_p ? 2 : 0));
          atomicMax(&A.st->overflow, 1);
        }
      }
    } else {
      if (lane == 0) {
        B.cnt_m[wp] = cm;
        B.cnt_p[wp] = cp;
      }
      __syncthreads();
      uint32_t before_m = 0, before_p = 0, all_m = 0, all_p = 0;
#pragma unroll
      for (int q = 0; q < kTW; ++q) {
        if (q < wp) {
          before_m += B.cnt_m[q];
          before_p += B.cnt_p[q];
        }
        all_m += B.cnt_m[q];
        all_p += B.cnt_p[q];
      }
      if (wp == 0) {
        // the ranges and the children's places in the queue are taken here, before the lists are written
        const bool kid = all_p > 0 && lane < (int)a.nk;
        const bool cell = kid && (A.wn[a.first + lane].y >> 22) != 0;
        const unsigned cells = __ballot_sync(0xffffffffu, cell);
        if (lane == 0) {
          const unsigned long long bm = all_m ? atomicAdd(&A.st->nm2l, (unsigned long long)all_m) : 0ull;
          const unsigned long long bp = all_p ? atomicAdd(&A.st->nopen, (unsigned long long)all_p) : 0ull;
          const bool fm = bm + all_m <= A.cap_m2l, fp = bp + all_p <= A.cap_open;
          if (!fm || !fp) {
            atomicOr(&A.st->ovf_lists, (fm ? 0 : 1) | (fp ? 0 : 4));
            atomicMax(&A.st->overflow, 1);
          }
          if (fm && all_m) {
            A.mb[sink] = A.mm[sink] = (uint32_t)bm;
            A.me[sink] = (uint32_t)(bm + all_m);
          }
          B.base_m = bm;
          B.base_p = bp;
          B.fit = (fm ? 1u : 0u) | (fp ? 2u : 0u);
          B.put = fp ? cells : 0u;
          if (fp && cells) {
            B.at = atomicAdd(&A.st->tail, (unsigned)__popc(cells));
            atomicAdd(&A.st->cells_left, __popc(cells));
          }
        }
      }
      __syncthreads();
      base_m = B.base_m + before_m;
      base_p = B.base_p + before_p;
      fit_m = cm > 0 && (B.fit & 1u);
      fit_p = cp > 0 && (B.fit & 2u);
      if (wp == 0 && all_p > 0 && (B.fit & 2u) && lane < (int)a.nk) {  // the children start from this list
        A.obeg[a.first + lane] = (uint32_t)B.base_p;
        A.ocnt[a.first + lane] = all_p;
      }
    }
    if (!over) {
      __syncwarp();
      if (fit_m)
        for (uint32_t i = lane; i < cm; i += 32) {
          const bool far = i < om;
          const uint32_t v = far ? spill_m[i] : W.stage[kStage - 1 - (i - om)];
          const uint32_t x = far ? saux_m[i] : W.aux[kStage - 1 - (i - om)];
          A.m2l[base_m + i] = pack_pair(sink, 0, 0, (x & 15u) - 1u) | v | ((uint64_t)(x >> 7) << kGenericBit);
        }
      if (fit_p)
        for (uint32_t i = lane; i < cp; i += 32) {
          const bool far = i < op;
          const uint32_t v = far ? spill_p[i] : W.stage[i - op];
          if (kLeaf) {
            A.p2p[base_p + i] = pack_pair(sink, 0, 0) | v;
          } else {
            A.open[base_p + i] = v;
            A.openc[base_p + i] = far ? saux_p[i] : W.aux[i - op];
          }
        }
      break;
    }
    if (!fit_m && !fit_p) break;
  }
}

// The walk: one cooperative launch, in two phases without a barrier between levels.
//
// The cells with children (about an eighth of the nodes): a cell may be visited
// once its parent is done.  Done cells put theirs into a queue; each block takes
// the next ticket and waits for its cell.  A cell is put in at most once; when
// none is left unfinished the queue is complete, and the tickets beyond its end
// go on to the leaves: handed out to warps from a counter.  A block whose wait for
// a cell gives up leaves there: the open lists are not complete.  (Sink batches: a
// launch for the first phase, then one for each range of the leaves.)
//
// What bounds it: the first phase by latency, one session a level along the
// deepest branch; the second by instructions, about 200 a round of 32 pairs at
// half the issue rate.  The walk it replaced kept a frontier of pairs that was
// classified, scanned, emitted and read again level by level, six grid barriers
// a level and 31 warp instructions a pair, and left each sink's entries in
// pieces that were sorted and copied together.  Walk and lists, ms, before and
// now: 0.21 -> 0.05 (1k uniform, leaf 16), 0.41 -> 0.08 (32k uniform), 0.86 ->
// 0.21 (262k clustered, leaf 48), 3.07 -> 1.12 (2M clustered), 6.7 -> 3.6 (2M with
// the network).  A warp a session instead of a block, with the leaves in the same
// queue: 1.08 at 2M, but 0.14 at 32k and 0.41 at 262k.
//
// kPolls: the wait's limit from the arguments (hfmm_params.wait_polls).  As a variable in
// every launch it cost the network's walk a third (3.6 -> 4.8 ms at 2M particles).
template <bool kNet, bool kPolls>
__global__ void __launch_bounds__(kTT, kNet ? 3 : 4) k_walk(const __grid_constant__ WalkArgs A,
                                                           const __grid_constant__ Mac m) {
  cg::grid_group grid = cg::this_grid();
  extern __shared__ __align__(16) unsigned char wsm[];
  constexpr int kSw = kNet ? kMlpSmemWords : 1, kXs = kNet ? 32 * 16 : 8, kDec = kNet ? 32 : 1;
  __shared__ uint32_t sw[kSw];
  __shared__ __align__(16) __nv_bfloat16 xs[kTW][kXs];
  __shared__ uint8_t dec[kTW][kDec];
  __shared__ MacF mf;
  __shared__ BlockMem B;
  const TreeState *ts = A.tree;
  if (ts->overflow) {  // graph mode, the tree did not fit: no walk (every block leaves here)
    if (blockIdx.x == 0 && threadIdx.x == 0) A.st->overflow = 3;
    return;
  }
  const int tid = threadIdx.x, wp = tid >> 5, lane = tid & 31;
  const long long gt = (long long)blockIdx.x * kTT + tid, nt = (long long)gridDim.x * kTT;
  const long long nn = (long long)ts->total;
  for (long long k = gt; k < nn; k += nt) {
    if (A.what != kWalkLeaves) {
      A.wn[k] = pack_node(A.cell[k], A.kids[k]);
      if (kNet) {  // once a node, not a pair (ten scattered loads, two roots, two divisions): 2M walk 4.2 -> 3.6 ms
        float count, dipole, quadrupole;
        node_features(m.M + (size_t)k * m.ldm, m.range[k].y, count, dipole, quadrupole);
        A.wf[k] = make_uint2(pack_bf16(count, dipole), pack_bf16(quadrupole, 0.f));
      }
      A.ocnt[k] = 0u;
      A.obeg[k] = 0u;
      A.queue[k] = k == 0 && nn > 1 ? 1u : 0u;  // the root is there, if it has children
    }
    A.mb[k] = A.me[k] = A.mm[k] = A.pb[k] = A.pe[k] = 0u;
  }
  if (gt == 0) {
    A.st->tail = A.st->cells_left = nn > 1 ? 1 : 0;
  }
  if (kNet) mlp_stage(m.w, sw);
  mac_f(m, mf);
  if (tid == 0) B.lost = 0u;
  WarpMem W;
  W.cand = reinterpret_cast<uint32_t *>(wsm + (size_t)wp * WalkSize<kNet>::kWarpBytes);
  W.net = W.cand + kCand;
  W.stack = W.net + WalkSize<kNet>::kNetWait;
  W.stage = W.stack + kStack;
  W.stackc = reinterpret_cast<uint8_t *>(W.stage + kStage);
  W.aux = W.stackc + kStack;
  uint32_t *spill = reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned char *>(A.spill) +
                                                 (size_t)(gt >> 5) * kSpillBytes);
  unsigned long long items = 0;
  uint32_t maxlev = 0;
  grid.sync();
  volatile TravState *vst = A.st;
  const unsigned polls = kPolls ? A.polls : kWaitPolls;
  if (A.what != kWalkLeaves) {
    for (;;) {
      if (tid == 0) {
        const unsigned t = atomicAdd(&A.st->next, 1u);
        uint32_t k = 0;
        unsigned poll = 0;
        for (; poll < polls; ++poll) {
          if ((long long)t < nn) k = *(volatile uint32_t *)(A.queue + t);
          if (k) break;
          if (vst->cells_left == 0) {  // complete (read before the tail): nothing more will come
            __threadfence();
            if (t >= vst->tail) break;
          }
          __nanosleep(poll < 64 ? 20 : 200);
        }
        if (poll == polls) {
          atomicMax(&A.st->overflow, 4);
          B.lost = 1u;
        }
        __threadfence();  // the parent's open list was written before the slot
        B.cell = k;
      }
      __syncthreads();
      const uint32_t k = B.cell;
      if (k == 0) break;
      const Node a = unpack_node(A.wn[k - 1]);
      walk_sink<kNet, false>(A, m, mf, k - 1, a, W, B, spill, sw, xs[wp], dec[wp], items, maxlev);
      // the open list, then the children's slots, then this cell is finished
      __threadfence();
      __syncthreads();
      if (wp == 0) {
        const unsigned put = B.put;
        if ((put >> lane) & 1u)
          *(volatile uint32_t *)(A.queue + B.at + __popc(put & ((1u << lane) - 1u))) = a.first + lane + 1u;
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicSub(&A.st->cells_left, 1);
      }
    }
  }
  const long long leaf_lo = A.what == kWalkLeaves ? A.leaf_lo : 0,
                  leaf_hi = B.lost ? 0 : A.what == kWalkAll ? (long long)ts->nleaves : A.leaf_hi;
  for (;;) {
    unsigned t = 0;
    if (lane == 0) t = atomicAdd(&A.st->leaf_next, 1u);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (leaf_lo + (long long)t >= leaf_hi) break;
    const uint32_t k = A.leaves[leaf_lo + t];
    if (k != 0 && A.ocnt[k] == 0) continue;
    walk_sink<kNet, true>(A, m, mf, k, unpack_node(A.wn[k]), W, B, spill, sw, xs[wp], dec[wp], items, maxlev);
  }
  maxlev = __reduce_max_sync(0xffffffffu, maxlev);
  if (lane == 0 && items) {
    atomicAdd(&A.st->items, items);
    atomicMax(&A.st->levels, (int)maxlev);
  }
}

// CSR bounds of the entries [lo, hi) of a list sorted by (sink, generic bit):
// beg[k] .. end[k]; with mid != null also mid[k], the first entry of sink k
// whose operator is evaluated per pair (end[k] when there is none).
__global__ void k_list_bounds(const uint64_t *__restrict__ lst, int64_t lo, int64_t hi, uint32_t *__restrict__ beg,
                              uint32_t *__restrict__ end, uint32_t *__restrict__ mid) {
  int64_t t = lo + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= hi) return;
  const uint64_t e = lst[t];
  const uint32_t s = pair_sink(e);
  const bool first = t == lo || pair_sink(lst[t - 1]) != s;
  const bool last = t == hi - 1 || pair_sink(lst[t + 1]) != s;
  if (first) beg[s] = (uint32_t)t;
  if (last) end[s] = (uint32_t)(t + 1);
  if (mid) {
    const bool g = pair_generic(e);
    if (g && (first || !pair_generic(lst[t - 1]))) mid[s] = (uint32_t)t;
    if (!g && last) mid[s] = (uint32_t)(t + 1);
  }
}

// first[q] = index of the first entry with order >= q (q = 0..9) in a list sorted by (order, sink)
__global__ void k_order_bounds(const uint64_t *__restrict__ lst, int64_t n, uint64_t *__restrict__ first) {
  const int q = threadIdx.x;
  if (q > 9) return;
  int64_t a = 0, b = n;
  while (a < b) {
    const int64_t mid = a + (b - a) / 2;
    if ((int)pair_order(lst[mid]) < q) a = mid + 1; else b = mid;
  }
  first[q] = (uint64_t)a;
}

__global__ void k_pairs_in_list(const uint64_t *__restrict__ lst, int64_t n, const uint2 *__restrict__ range,
                                unsigned long long *__restrict__ acc) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = 0;
  if (t < n) {
    uint64_t e = lst[t];
    v = (unsigned long long)range[pair_sink(e)].y * range[pair_src(e)].y;
  }
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(acc, v);
}

__global__ void k_count_table(const uint64_t *__restrict__ lst, int64_t n, unsigned long long *__restrict__ acc) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = (t < n && !pair_generic(lst[t])) ? 1ull : 0ull;
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(acc, v);
}

}  // namespace

namespace {

// First guess of the P2P list's entries per particle (the scale of the walk_plan guesses).
double p2p_guess_per_particle(const Ctx &c) {
  const double lf = c.prm.leaf_max > 16 ? std::pow(16.0 / c.prm.leaf_max, 1.5) * 1.5 : 1.0;
  return 128.0 * (lf < 1.0 ? lf : 1.0);
}

// The walk's parameters and grid, and the first guesses of its list capacities.
struct WalkPlan {
  Mac m;
  unsigned nb;
};

const void *walk_kernel(const Ctx &c, bool net) {
  if (c.prm.wait_polls) return net ? (const void *)k_walk<true, true> : (const void *)k_walk<false, true>;
  return net ? (const void *)k_walk<true, false> : (const void *)k_walk<false, false>;
}

size_t walk_smem(bool net) {
  return (size_t)kTW * (net ? WalkSize<true>::kWarpBytes : WalkSize<false>::kWarpBytes);
}

cudaError_t walk_plan(Ctx &c, WalkPlan &w) {
  cudaError_t e;
  Mac &m = w.m;
  m = Mac{};
  m.rc2i = c.rc2i;
  for (int l = 0; l <= kDepth; ++l) m.acc_thr[l] = c.acc_thr[l];
  m.rule = c.prm.transition_rule;
  m.size_rule = c.prm.size_rule;
  m.mode = c.collect ? 2 : c.count_walk ? 0 : c.prm.mac_mode;
  m.conv = c.count_walk == 2 ? 1 : 0;
  m.order = c.p;
  m.tab_k = ((c.prm.m2l_precision == 0 && c.prm.m2l_tables) || c.prm.m2l_precision >= 3) ? c.tab_k : 0;
  m.mutual = (c.prm.p2p_mutual && !c.collect && !c.count_walk) ? 1 : 0;
  m.w = static_cast<const __nv_bfloat16 *>(c.mlp_w.p);
  m.M = P<float>(c.M);
  m.range = P<uint2>(c.range);
  m.ldm = c.ldm;
  m.inv_rs_h = (float)(c.prm.box / (double)kHalfBox / c.rs);
  m.inv_rc_h = (float)(c.prm.box / (double)kHalfBox / c.rc);
  m.cand = P<uint64_t>(c.cand);
  m.ncand = reinterpret_cast<unsigned long long *>(P<uint64_t>(c.d_small) + 7);
  m.cand_cap = c.cand_cap;
  m.sample_mod = c.sample_mod ? c.sample_mod : 1u;

  int dev = 0, nsm = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const bool net = m.mode == 1;
  const void *kern = walk_kernel(c, net);
  const size_t smem = walk_smem(net);
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kTT, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int want = c.prm.tile_trav_blocks > 0 ? c.prm.tile_trav_blocks : 4;
  // no more warps than leaves (rounded up): a grid barrier costs more the more blocks it spans
  const unsigned most = (unsigned)(nsm * (per_sm < want ? per_sm : want));
  w.nb = std::max(1u, std::min(most, blocks_for((size_t)c.nleaves, kTW)));
  // capacities: the last call's sizes with head-room, at least a few per node.
  // First guesses from the 2M clustered set: at leaves of 16 about 50 M2L and 115
  // P2P entries per particle in total and 5 open ones; these fall about as
  // (16 / leaf_max)^1.5 (8 M2L and 21 P2P per particle at 48), so the guesses are
  // scaled so, with a margin of 1.5.  A list that overflows is grown alone (to what
  // the walk asked for, at least twice its size) and the walk is repeated.  A
  // positive list_init replaces every first guess (a test knob for the retry path).
  const double lf = c.prm.leaf_max > 16 ? std::pow(16.0 / c.prm.leaf_max, 1.5) * 1.5 : 1.0;
  const double sc = (lf < 1.0 ? lf : 1.0) * c.walk_share;  // sink batches: one batch's share
  const uint64_t init = (uint64_t)c.prm.list_init;
  auto first_guess = [&](uint64_t guess) { return init > 0 ? init : guess; };
  const uint64_t g_open = first_guess((uint64_t)((lf < 1.0 ? lf : 1.0) * 8 * c.n + 1024));
  const uint64_t g_m2l = first_guess((uint64_t)(sc * 64 * c.n + 1024));
  const uint64_t g_p2p = first_guess((uint64_t)(sc * 128 * c.n + 1024));
  if (c.cap_open < g_open) c.cap_open = g_open;
  if (c.cap_m2l < g_m2l) c.cap_m2l = g_m2l;
  if (c.cap_p2p < g_p2p) c.cap_p2p = g_p2p;
  if (c.cap_open > 0xffffffffull) c.cap_open = 0xffffffffull;  // 32-bit offsets
  return cudaSuccess;
}

cudaError_t walk_buffers(Ctx &c, const WalkPlan &w) {
  cudaError_t e;
#define TRY(x)                      \
  do {                              \
    e = (x);                        \
    if (e != cudaSuccess) return e; \
  } while (0)
  const size_t nn = (size_t)(c.nnodes > 0 ? c.nnodes : 1);
  TRY(ensure(c.wnode, nn * sizeof(uint4)));
  if (w.m.mode == 1) TRY(ensure(c.wfeat, nn * sizeof(uint2)));
  TRY(ensure(c.wqueue, nn * 4));
  TRY(ensure(c.wspill, (size_t)w.nb * kTW * kSpillBytes));
  TRY(ensure(c.obeg, nn * 4));
  TRY(ensure(c.ocnt, nn * 4));
  TRY(ensure(c.m2l_beg, nn * 4));
  TRY(ensure(c.m2l_end, nn * 4));
  TRY(ensure(c.m2l_mid, nn * 4));
  TRY(ensure(c.p2p_beg, nn * 4));
  TRY(ensure(c.p2p_end, nn * 4));
  TRY(ensure(c.open, c.cap_open * 4));
  TRY(ensure(c.openc, c.cap_open));
  TRY(ensure(c.m2l, c.cap_m2l * 8));
  TRY(ensure(c.p2p, c.cap_p2p * 8));
  return cudaSuccess;
#undef TRY
}

// the walk's state sits after the eight counters of the 256-byte d_small and is read back into h_pinned
TravState *walk_state(Ctx &c) {
  static_assert(8 * sizeof(uint64_t) + sizeof(TravState) <= 128, "TravState must end below d_small[16]");
  return reinterpret_cast<TravState *>(P<uint64_t>(c.d_small) + 8);
}

// What one launch visits; a batch of leaves by position.
struct WalkPart {
  int what = kWalkAll;
  int64_t leaf_lo = 0, leaf_hi = 0;
};

// Zero the counters and launch the cooperative walk (no allocation, no read-back).
cudaError_t walk_launch(Ctx &c, const WalkPlan &w, cudaStream_t st, const WalkPart &part = WalkPart()) {
  cudaError_t e;
  WalkArgs A;
  A.st = walk_state(c);
  if ((e = cudaMemsetAsync(A.st, 0, sizeof(TravState), st)) != cudaSuccess) return e;
  A.cell = P<uint4>(c.cell);
  A.kids = P<int2>(c.kids);
  A.leaves = P<uint32_t>(c.leaves);
  A.tree = P<TreeState>(c.tstate);
  A.wn = P<uint4>(c.wnode);
  A.wf = P<uint2>(c.wfeat);
  A.obeg = P<uint32_t>(c.obeg);
  A.ocnt = P<uint32_t>(c.ocnt);
  A.open = P<uint32_t>(c.open);
  A.openc = P<uint8_t>(c.openc);
  A.m2l = P<uint64_t>(c.m2l);
  A.p2p = P<uint64_t>(c.p2p);
  A.mb = P<uint32_t>(c.m2l_beg);
  A.me = P<uint32_t>(c.m2l_end);
  A.mm = P<uint32_t>(c.m2l_mid);
  A.pb = P<uint32_t>(c.p2p_beg);
  A.pe = P<uint32_t>(c.p2p_end);
  A.cap_open = c.cap_open;
  A.cap_m2l = c.cap_m2l;
  A.cap_p2p = c.cap_p2p;
  A.queue = P<uint32_t>(c.wqueue);
  A.spill = P<uint32_t>(c.wspill);
  A.what = part.what;
  A.leaf_lo = part.leaf_lo;
  A.leaf_hi = part.leaf_hi;
  A.polls = wait_polls(c, kWaitPolls);
  Mac m = w.m;
  // collected candidates: those of this walk alone (a walk whose lists overflowed is repeated)
  if (m.mode == 2 && (e = cudaMemsetAsync(m.ncand, 0, 8, st)) != cudaSuccess) return e;
  const bool net = m.mode == 1;
  const void *kern = walk_kernel(c, net);
  void *args[] = {(void *)&A, (void *)&m};
  e = cudaLaunchCooperativeKernel(kern, dim3(w.nb), dim3(kTT), args, walk_smem(net), st);
  note_launch();
  return e;
}

// After a walk that did not fit: grow the lists that overflowed.  The M2L and P2P
// counts are what a walk with those open lists needs; a short open list hides the
// pairs below it, so the next walk may ask for more.
void walk_grow(Ctx &c, const TravState &hs) {
  auto up = [&](uint64_t &cap, int bit, unsigned long long need) {
    if (!(hs.ovf_lists & bit)) return;
    const uint64_t want = std::max<uint64_t>(cap * 2, need);
    cap = want + want / 4 + 1024;
  };
  up(c.cap_m2l, 1, hs.nm2l);
  up(c.cap_p2p, 2, hs.np2p);
  up(c.cap_open, 4, hs.nopen);
  if (c.cap_open > 0xffffffffull) c.cap_open = 0xffffffffull;
}

cudaError_t walk_read(Ctx &c, cudaStream_t st, TravState &hs) {
  cudaError_t e = cudaMemcpyAsync(c.h_pinned, walk_state(c), sizeof(TravState), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) std::memcpy(&hs, c.h_pinned, sizeof(TravState));
  return e;
}

// The sizes of a walk that fitted.
void walk_sizes(Ctx &c, const TravState &hs) {
  c.nm2l = (int64_t)hs.nm2l;
  c.np2p = (int64_t)hs.np2p;
  c.traverse_iters = hs.levels + 1;
  c.frontier_items = (int64_t)hs.items;
}

// One part of the walk, repeated with grown lists while one overflows.
cudaError_t walk_part(Ctx &c, const WalkPlan &w, const WalkPart &part, cudaStream_t st, TravState &hs, int64_t &walks) {
  cudaError_t e;
  for (int attempt = 0; attempt < 32; ++attempt) {
    ++walks;
    if ((e = walk_buffers(c, w)) != cudaSuccess) return e;
    if ((e = walk_launch(c, w, st, part)) != cudaSuccess) return e;
    if ((e = walk_read(c, st, hs)) != cudaSuccess) return e;
    if (!hs.overflow) return cudaSuccess;
    if (hs.overflow == 4) return cudaErrorTimeout;  // HFMM_ERR_TIMEOUT
    walk_grow(c, hs);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t traverse(Ctx &c, cudaStream_t st) {
  cudaError_t e;
  c.nm2l = c.np2p = 0;
  c.traverse_iters = 0;
  if (c.n == 0) return cudaSuccess;
  WalkPlan w;
  if ((e = walk_plan(c, w)) != cudaSuccess) return e;
  TravState hs;
  c.traverse_walks = 0;
  if ((e = walk_part(c, w, WalkPart(), st, hs, c.traverse_walks)) != cudaSuccess) return e;
  walk_sizes(c, hs);
  return cudaSuccess;
}

// Graph mode: the walk without its read-back.  _prepare sizes every buffer
// (outside the capture), _launch enqueues the walk (inside it), _finish reads
// the state back after the graph ran and reports whether the lists fit.
cudaError_t traverse_graph_prepare(Ctx &c) {
  WalkPlan w;
  cudaError_t e = walk_plan(c, w);
  if (e == cudaSuccess) e = walk_buffers(c, w);
  return e;
}

cudaError_t traverse_graph_launch(Ctx &c, cudaStream_t st) {
  WalkPlan w;
  cudaError_t e = walk_plan(c, w);
  if (e == cudaSuccess) e = walk_launch(c, w, st);
  return e;
}

cudaError_t traverse_graph_finish(Ctx &c, cudaStream_t st, bool *ok) {
  cudaError_t e;
  TravState hs;
  if ((e = walk_read(c, st, hs)) != cudaSuccess) return e;
  *ok = !hs.overflow;
  if (*ok) walk_sizes(c, hs);
  c.traverse_walks = 1;
  return cudaSuccess;
}

StepGuard step_guard(Ctx &c) {
  StepGuard g;
  g.tree_overflow = &P<TreeState>(c.tstate)->overflow;
  g.walk_overflow = &walk_state(c)->overflow;
  return g;
}

namespace {

// Entries of each sink (for the scan that places them in sink order).
__global__ void k_sink_counts(const uint32_t *__restrict__ beg, const uint32_t *__restrict__ end, int64_t nn,
                              uint32_t *__restrict__ cnt) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nn) cnt[k] = end[k] - beg[k];
}

// One warp a sink: its entries to their place in sink order, and the new bounds.
__global__ void k_sink_copy(const uint32_t *__restrict__ dst, int64_t nn, const uint64_t *__restrict__ src,
                            uint64_t *__restrict__ out, uint32_t *__restrict__ beg, uint32_t *__restrict__ end) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); k < nn; k += nw) {
    const uint32_t b = beg[k], n = end[k] - b, d = dst[k];
    for (uint32_t j = lane; j < n; j += 32) out[d + j] = src[b + j];
    __syncwarp();
    if (lane == 0) {
      beg[k] = d;
      end[k] = d + n;
    }
  }
}

}  // namespace

// A list whose sinks are in no fixed order, into sink order (the mutual P2P adds
// its reactions in list order, so that order has to be the same on every run).
static cudaError_t list_in_sink_order(Ctx &c, DBuf &L, DBuf &A, int64_t n, DBuf &beg, DBuf &end, cudaStream_t st) {
  cudaError_t e;
  if (n == 0) return cudaSuccess;
  const int64_t nn = c.nnodes > 0 ? c.nnodes : 1;
  if ((e = ensure(A, (size_t)n * 8)) != cudaSuccess) return e;
  if ((e = ensure(c.tmp2, (size_t)nn * 8)) != cudaSuccess) return e;
  uint32_t *cnt = P<uint32_t>(c.tmp2), *dst = cnt + nn;
  k_sink_counts<<<blocks_for(nn, 256), 256, 0, st>>>(P<uint32_t>(beg), P<uint32_t>(end), nn, cnt);
  note_launch();
  if ((e = scan_u32(cnt, dst, P<uint64_t>(c.d_small) + 1, (size_t)nn, c.offs, st)) != cudaSuccess) return e;
  const unsigned g = std::min(blocks_for((size_t)nn, 8), 152u * 32u);
  k_sink_copy<<<g, 256, 0, st>>>(dst, nn, P<uint64_t>(L), P<uint64_t>(A), P<uint32_t>(beg), P<uint32_t>(end));
  note_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  std::swap(L, A);
  return cudaSuccess;
}

cudaError_t p2p_list_particle_pairs(Ctx &c, cudaStream_t st, int64_t *out) {
  *out = 0;
  if (c.np2p == 0) return cudaSuccess;
  const unsigned T = 256;
  unsigned long long *cnt = reinterpret_cast<unsigned long long *>(c.d_small.p);
  cudaError_t e;
  if ((e = cudaMemsetAsync(cnt, 0, 8, st)) != cudaSuccess) return e;
  k_pairs_in_list<<<blocks_for(c.np2p, T), T, 0, st>>>(P<uint64_t>(c.p2p), c.np2p, P<uint2>(c.range), cnt);
  note_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(c.h_pinned, cnt, 8, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  *out = (int64_t)c.h_pinned[0];
  return cudaSuccess;
}

// The walk leaves both lists grouped by sink with CSR bounds.  What is left: the
// order the mutual P2P needs, the orders of the learned acceptance, the table
// pairs of each sink first, and the counts of statistics runs.
cudaError_t sort_lists(Ctx &c, cudaStream_t st) {
  cudaError_t e;
#define TRY(x)                      \
  do {                              \
    e = (x);                        \
    if (e != cudaSuccess) return e; \
  } while (0)
  c.p2p_particle_pairs = -1;
  c.nm2l_table = -1;
  if (c.graph_walk) return cudaSuccess;  // none of those runs as a graph
  const int T = 256;
  int64_t nn = c.nnodes > 0 ? c.nnodes : 1;
  if (c.prm.p2p_mutual) TRY(list_in_sink_order(c, c.p2p, c.p2p_alt, c.np2p, c.p2p_beg, c.p2p_end, st));
  const bool tables = ((c.prm.m2l_precision == 0 && c.prm.m2l_tables) || c.prm.m2l_precision >= 3) && c.tab_k > 0;
  if (c.nm2l > 0 && !tables) {
    if (c.prm.mac_mode == 1) {  // learned orders: stable pass on the order bits -> by order, then by sink
      bool alt = false;
      TRY(ensure(c.m2l_alt, c.nm2l * 8));
      TRY(radix_sort_u64(P<uint64_t>(c.m2l), nullptr, P<uint64_t>(c.m2l_alt), nullptr, c.nm2l, kOrderShift, 64,
                         &alt, c.tmp, st));
      if (alt) std::swap(c.m2l, c.m2l_alt);
    }
  } else if (c.nm2l > 0) {
    // operator tables: group by (sink, table bit) (learned: (order, sink, table bit))
    int sink_bits = 1;
    while (((int64_t)1 << sink_bits) < nn) ++sink_bits;
    TRY(ensure(c.m2l_alt, c.nm2l * 8));
    TRY(cudaMemsetAsync(c.m2l_mid.p, 0, nn * 4, st));
    TRY(cudaMemsetAsync(c.m2l_beg.p, 0, nn * 4, st));
    TRY(cudaMemsetAsync(c.m2l_end.p, 0, nn * 4, st));
    bool alt = false;
    const int hi_bit = c.prm.mac_mode == 1 ? 64 : kSinkShift + sink_bits;
    TRY(radix_sort_u64(P<uint64_t>(c.m2l), nullptr, P<uint64_t>(c.m2l_alt), nullptr, c.nm2l, kGenericBit, hi_bit,
                       &alt, c.tmp, st));
    if (alt) std::swap(c.m2l, c.m2l_alt);
    if (c.prm.mac_mode != 1) {
      k_list_bounds<<<blocks_for(c.nm2l, T), T, 0, st>>>(P<uint64_t>(c.m2l), 0, c.nm2l, P<uint32_t>(c.m2l_beg),
                                                         P<uint32_t>(c.m2l_end), P<uint32_t>(c.m2l_mid));
      note_launch();
      TRY(cudaGetLastError());
    }
  }
  if (c.prm.profile & 2) {
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(c.d_small.p);
    TRY(cudaMemsetAsync(cnt, 0, 16, st));
    if (c.np2p > 0) {
      k_pairs_in_list<<<blocks_for(c.np2p, T), T, 0, st>>>(P<uint64_t>(c.p2p), c.np2p, P<uint2>(c.range), cnt);
      note_launch();
    }
    if (c.nm2l > 0) {
      k_count_table<<<blocks_for(c.nm2l, T), T, 0, st>>>(P<uint64_t>(c.m2l), c.nm2l, cnt + 1);
      note_launch();
    }
    TRY(cudaGetLastError());
    TRY(cudaMemcpyAsync(c.h_pinned, c.d_small.p, 16, cudaMemcpyDeviceToHost, st));
    TRY(cudaStreamSynchronize(st));
    c.p2p_particle_pairs = (int64_t)c.h_pinned[0];
    c.nm2l_table = (int64_t)c.h_pinned[1];
  }
  return cudaSuccess;
#undef TRY
}

cudaError_t m2l_all(Ctx &c, cudaStream_t st) {
  if (c.nm2l == 0) return cudaSuccess;
  const bool lo = c.prm.m2l_precision >= 3 && c.tab_k > 0;
  const bool tab = (c.prm.m2l_precision == 0 && c.prm.m2l_tables && c.tab_k > 0) || lo;
  if (tab && !c.tab_ready) {
    cudaError_t e = m2l_table_build(c, st);
    if (e != cudaSuccess) return e;
  }
  auto run = [&](int q) -> cudaError_t {
    if (lo && m2l_lo_supported(q)) return m2l_pass_lo(c, q, st);
    if (c.prm.m2l_precision >= 3) return m2l_pass(c, q, st);  // no table: every pair on the FP32 kernel
    if (c.prm.m2l_precision != 0 && m2l_tc_supported(q)) return m2l_pass_tc(c, q, st);
    if (tab) {
      cudaError_t e = m2l_pass_table(c, q, st);
      if (e != cudaSuccess) return e;
    }
    return m2l_pass(c, q, st);
  };
  if (c.prm.mac_mode != 1) return run(c.p);
  cudaError_t e;
  const int T = 256;
  const int64_t nn = c.nnodes;
  uint64_t *first = P<uint64_t>(c.d_small) + 16;
  k_order_bounds<<<1, 32, 0, st>>>(P<uint64_t>(c.m2l), c.nm2l, first);
  note_launch();
  if ((e = cudaMemcpyAsync(c.h_pinned, first, 10 * 8, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  uint64_t fb[10];
  for (int q = 0; q < 10; ++q) fb[q] = c.h_pinned[q];
  for (int q = 1; q <= c.p && q <= 8; ++q) {
    const int64_t lo = (int64_t)fb[q], hi = (int64_t)fb[q + 1];
    if (hi <= lo) continue;
    if ((e = cudaMemsetAsync(c.m2l_beg.p, 0, nn * 4, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(c.m2l_end.p, 0, nn * 4, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(c.m2l_mid.p, 0, nn * 4, st)) != cudaSuccess) return e;
    k_list_bounds<<<blocks_for(hi - lo, T), T, 0, st>>>(P<uint64_t>(c.m2l), lo, hi, P<uint32_t>(c.m2l_beg),
                                                        P<uint32_t>(c.m2l_end), P<uint32_t>(c.m2l_mid));
    note_launch();
    if ((e = run(q)) != cudaSuccess) return e;
  }
  return cudaGetLastError();
}


int sink_batches_for(const Ctx &c) {
  if (c.prm.sink_batches > 0) return c.prm.sink_batches;
  const double guess = p2p_guess_per_particle(c) * (double)c.n;
  // one batch while the guess stays below 2^28 entries; beyond, batches of about 2^27
  if (guess <= (double)(1u << 28)) return 1;
  return (int)std::min(4096.0, std::ceil(guess / (double)(1u << 27)));
}

// Sink batches.  A leaf's walk ends in its own session, so a batch is a range of
// the leaves (breadth-first order: by level, Morton order within a level).  The
// first launch visits the cells with children alone: their M2L entries, and the
// open lists every leaf starts from, which stay for all batches.  Then each
// batch of leaves is walked and evaluated (M2L into L, P2P into c.pacc), and the
// next one reuses the list memory.  The same pairs are classified as in one
// walk, and a leaf's entries are all in its batch, in the same order.  Finally
// L2L, and L2P adds the P2P accelerations.
cudaError_t short_range_batched(Ctx &c, float *acc, int nbatch, cudaStream_t st) {
  cudaError_t e;
#define TRY(x)                      \
  do {                              \
    e = (x);                        \
    if (e != cudaSuccess) return e; \
  } while (0)
  const int64_t n = c.n;
  TRY(ensure(c.pacc, (size_t)3 * n * sizeof(float)));
  TRY(cudaMemsetAsync(c.pacc.p, 0, (size_t)3 * n * sizeof(float), st));
  float *pacc = P<float>(c.pacc);
  c.walk_share = 1.0 / nbatch;
  WalkPlan w;
  e = walk_plan(c, w);
  c.walk_share = 1.0;
  if (e != cudaSuccess) return e;
  int64_t tot_m2l = 0, tot_p2p = 0, walks = 0, items = 0;
  int iters = 0, ran = 0;
  const int64_t nl = c.nleaves;
  for (int b = -1; b < nbatch; ++b) {  // -1: the cells with children
    WalkPart part;
    part.what = b < 0 ? kWalkCells : kWalkLeaves;
    part.leaf_lo = b < 0 ? 0 : nl * b / nbatch;
    part.leaf_hi = b < 0 ? 0 : nl * (b + 1) / nbatch;
    if (b >= 0 && part.leaf_hi == part.leaf_lo) continue;
    if (b >= 0) ++ran;
    TravState hs;
    TRY(walk_part(c, w, part, st, hs, walks));
    walk_sizes(c, hs);
    tot_m2l += c.nm2l;
    tot_p2p += c.np2p;
    items += c.frontier_items;
    iters = std::max(iters, c.traverse_iters);
    if (c.nm2l > (int64_t)UINT32_MAX || c.np2p > (int64_t)UINT32_MAX) return cudaErrorInvalidValue;
    // evaluate what this part of the walk emitted
    TRY(sort_lists(c, st));
    TRY(m2l_all(c, st));
    if (c.np2p > 0) TRY(c.prm.p2p_mutual ? p2p_pass_mutual(c, pacc, st) : p2p_pass(c, pacc, st));
  }
  c.nm2l = tot_m2l;
  c.np2p = tot_p2p;
  c.traverse_walks = walks;
  c.frontier_items = items;
  c.traverse_iters = iters;
  c.last_batches = ran > 1 ? ran : 1;
  c.lists_split = true;  // each part's lists were evaluated in turn
  return downward(c, acc, st, pacc);
#undef TRY
}

}  // namespace hfmm
