// M2L with split-precision products on the 5th-generation tensor cores
// (tcgen05, accumulator in tensor memory): m2l_precision = 1 (3xTF32) and
// m2l_precision = 2 (BF16x3).
//
// For one sink A with pairs (A, B_k), Eq. m2l in the scaled, per-pair
// normalised form of m2l.cu is
//   L~_n(A) = sum_k u_k^(|n|+1) v_k^|m| sum_m M~_m(B_k) D^_{n+m}(R^_k)
//           = sum_m P[n+m][m],   P[c][m] = sum_k D'_c(k) M'_m(k),
//   D'_c(k) = u_k^(|c|+1) D^_c(R^_k),   M'_m(k) = (v_k / u_k)^|m| M~_m(B_k),
// a GEMM whose contraction dimension is the sink's pair list.  Each FP32
// operand is split x = hi + lo, hi its TF32 rounding (kind::tf32, K = 8 per
// instruction) or its BF16 rounding with lo = bf16(x - hi) (kind::f16 with both
// operands BF16, K = 16); P accumulates hi*hi + hi*lo + lo*hi in FP32.  The
// dropped terms are lo*lo and, for BF16, the rounding of lo: about 2^-21
// relative for TF32 and 2^-16 for BF16 per product.  Only the entries with
// |n|+|m| <= p of P are used, so at most C(p+6,6) / NC^2 of the tensor work is
// algorithmic (462 / 3136 at p = 5).
//
// A worker is 4 warps with one sink at a time; a CTA has four or five (a kernel that
// allocates tensor memory gets one CTA an SM).  A chunk is 32 pairs: three warps
// compute and store a third of the pairs' D' each (generated TCStore / TCStoreBF
// bodies), one their M', to K-major, 128-byte-swizzled tiles (one 128-byte row per
// matrix row); one thread issues the K-steps the chunk's pairs need x 3 split
// products of tcgen05.mma (M = 128 rows c, N = NCP columns m) into the worker's
// TMEM accumulator and commits to an mbarrier, and the next chunk's entries and
// cells are fetched meanwhile.  After the last chunk the warps read their 32 TMEM
// lanes (rows c), stage P in shared memory, and four lanes form each L~_n = sum_m
// P[n+m][m] from a table of the places.  Waits are bounded; on a timeout the worker
// records an error and leaves its loop, the MMAs it already issued are waited for
// (with the full limit), and the CTA returns after freeing TMEM.
//
// What bounds it: the latency of a worker's chain (entries, cells, multipoles ->
// operands -> MMA -> accumulator -> L), hidden by the other workers only.  Hence the
// small chunk, with tiles cut to the rows that are written (the MMA's 128-row reads
// run on into the next tile, whose values only reach rows of P that are never
// read): 47 KB a worker at p = 6.  Four warps an SM with 128-pair chunks, every
// thread computing both operands and all four K-tiles issued whatever the list's
// length, took 20.8 ms for the 33M pairs of the 2M learned step instead of 8.6; with D' by
// recurrence 8.4, multipole rows by 16-byte loads 7.4, entries fetched two chunks ahead
// 7.3, a fifth worker at p = 5 7.1 (issue 39%; the next rows prefetched into L1: the same;
// the next operands formed in registers under the MMA: p = 5 3% faster, p = 6 5.2 instead
// of 3.2 ms, its code no longer in the instruction cache).
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "gen_bodies.cuh"
#include "tc_common.cuh"

namespace hfmm {
namespace {

// Sinks at a time per CTA, four warps each: at p = 6 four fill the shared memory, at p = 5
// five do with what registers five leave a thread (96, no spills; 3.57 -> 3.37 ms of the
// learned 2M step's p = 5 pairs, with six at 80 registers the same).
__host__ __device__ constexpr int workers_of(int p) { return p == 5 ? 5 : 4; }
constexpr int kChunk = 32;      // pairs per chunk: one lane each
constexpr int kSinkBatch = 16;  // nodes taken from the work counter at a time
constexpr uint32_t kWaitLimit = 1u << 22;

__host__ __device__ constexpr int ncp_of(int p) { return (ncoef(p) + 15) / 16 * 16; }
__host__ __device__ constexpr int tmem_cols_of(int p) {
  return ncp_of(p) <= 32 ? 32 : (ncp_of(p) <= 64 ? 64 : (ncp_of(p) <= 128 ? 128 : 256));
}
// bytes of one A tile (rows c < NC, whole 8-row groups) and of one B tile (NCP rows)
__host__ __device__ constexpr int a_bytes_of(int p) { return (ncoef(p) + 7) / 8 * 1024; }
__host__ __device__ constexpr int b_bytes_of(int p) { return ncp_of(p) * 128; }
// a worker's shared memory: A hi, lo + B hi, lo; at least the P staging and what the MMA's
// 128-row reads of A lo span
__host__ __device__ constexpr size_t worker_bytes(int p) {
  const size_t tiles = 2 * (size_t)a_bytes_of(p) + 2 * (size_t)b_bytes_of(p);
  const size_t reach = (size_t)a_bytes_of(p) + 16384, stage = (size_t)ncoef(p) * (ncoef(p) | 1) * 4;
  const size_t most = tiles > reach ? (tiles > stage ? tiles : stage) : (reach > stage ? reach : stage);
  return (most + 1023) / 1024 * 1024;
}
// dynamic shared memory: 1 KB alignment slack and the workers'
__host__ __device__ constexpr size_t smem_of(int p) { return 1024 + workers_of(p) * worker_bytes(p); }
// terms of L~: sum over n of the m with |n| + |m| <= p
__host__ __device__ constexpr int terms_of(int p) {
  int t = 0;
  for (int k = 0; k <= p; ++k) t += (k + 1) * (k + 2) / 2 * ncoef(p - k);
  return t;
}

// 16 accumulator columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

template <int P, bool kBF>
__global__ void __launch_bounds__(128 * workers_of(P), 1)
    k_m2l_tc(int64_t nn, const uint4 *__restrict__ cell, const uint32_t *__restrict__ beg,
             const uint32_t *__restrict__ end, const uint64_t *__restrict__ lst, const float *__restrict__ M,
             float *__restrict__ L, int ldm, float inv_rs, unsigned long long *__restrict__ ctr,
             int *__restrict__ status, uint32_t chunk_wait) {
  constexpr int NC = ncoef(P), NCP = ncp_of(P);
  constexpr int kLd = NC | 1;  // row stride of the P staging (odd: no bank conflicts)
  constexpr uint32_t WCOLS = tmem_cols_of(P);  // accumulator columns of a worker
  constexpr int kWorkers = workers_of(P);
  constexpr uint32_t TCOLS = kWorkers * WCOLS <= 128 ? 128 : kWorkers * WCOLS <= 256 ? 256 : 512;  // a power of two
  static_assert(kWorkers * WCOLS <= 512, "tensor memory");
  constexpr uint32_t IDESC = kBF ? idesc_bf16(128, NCP) : idesc_tf32(128, NCP);
  constexpr int kStep = kBF ? 16 : 8;  // pairs per K-step (32 bytes)
  using T = typename std::conditional<kBF, __nv_bfloat16, float>::type;
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t mbars[kWorkers];
  __shared__ uint32_t tmem_slot;
  __shared__ uint16_t place[terms_of(P)];  // of each term P[n+m][m], by n then m
  __shared__ uint16_t tbeg[NC + 1];
  __shared__ uint32_t sink_list[kWorkers][kSinkBatch];
  __shared__ uint2 bound_list[kWorkers][kSinkBatch];  // the sinks' list bounds
  __shared__ int sink_count[kWorkers], aborts[kWorkers];

  // a worker's four warps (its warp w reads TMEM lanes 32 w ..) meet at a barrier of their own
  const int worker = threadIdx.x >> 7, tid = threadIdx.x & 127, lane = tid & 31, warp = tid >> 5;
  uint32_t *sinks = sink_list[worker];
  uint2 *bounds = bound_list[worker];
  volatile int &n_sinks = sink_count[worker], &abort_flag = aborts[worker];
  auto sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(worker + 1) : "memory"); };
  unsigned char *base =
      (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023) + worker * worker_bytes(P);
  unsigned char *a_hi = base, *a_lo = a_hi + a_bytes_of(P), *b_hi = a_lo + a_bytes_of(P), *b_lo = b_hi + b_bytes_of(P);
  float *pbuf = reinterpret_cast<float *>(base);  // P staging after a sink's last chunk

  __shared__ uchar4 mi[NC];
  if (threadIdx.x < NC) {
    int x, y, z;
    mdecode(tid, x, y, z);
    mi[tid] = make_uchar4((unsigned char)x, (unsigned char)y, (unsigned char)z, (unsigned char)(x + y + z));
  }
  __syncthreads();
  if (threadIdx.x < NC) {
    const uchar4 n = mi[tid];
    int at = 0;
    for (int q = 0; q < tid; ++q) at += ncoef(P - mi[q].w);
    tbeg[tid] = (uint16_t)at;
    const int rem = ncoef(P - n.w);
    if (tid == NC - 1) tbeg[NC] = (uint16_t)(at + rem);
    for (int e = 0; e < rem; ++e) {
      const uchar4 m = mi[e];
      place[at + e] = (uint16_t)(midx(n.x + m.x, n.y + m.y, n.z + m.z) * kLd + e);
    }
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbars[worker])));
    abort_flag = 0;
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(TCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem0 = tmem_slot, tmem = tmem0 + worker * WCOLS;
  const uint32_t mb = smem_u32(&mbars[worker]);
  uint32_t phase = 0;
  const float kInvSqrtPi = 0.56418958354775628f;

  // the swizzled element offsets of this lane's column (16-byte chunks XOR the row mod 8
  // within each 8-row group); BF16 rows hold the 32 pairs in their first half
  constexpr int kEl = 16 / (int)sizeof(T);  // elements per 16-byte chunk
  int xo[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) xo[j] = (((lane / kEl) ^ j) * kEl) + (lane % kEl);

  for (;;) {
    // ---- the next nodes with M2L pairs
    if (warp == 0) {
      int got = 0;
      for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(ctr, (unsigned long long)kSinkBatch);
        t = __shfl_sync(0xffffffffu, t, 0);
        if ((int64_t)t >= nn) break;
        const int64_t k = (int64_t)t + lane;
        uint2 r = make_uint2(0u, 0u);
        if (lane < kSinkBatch && k < nn) r = make_uint2(beg[k], end[k]);
        const unsigned m = __ballot_sync(0xffffffffu, r.y > r.x);
        if (r.y > r.x) {
          const int at = __popc(m & ((1u << lane) - 1u));
          sinks[at] = (uint32_t)k;
          bounds[at] = r;
        }
        got = __popc(m);
        if (got) break;
      }
      if (lane == 0) n_sinks = got;
    }
    sync();
    const int ns = n_sinks;
    if (ns == 0 || abort_flag) break;
    // Chunks in order: the one at hand (its pair e, cb of sink ca), and the one after it,
    // whose entry e1 is there when its cell is asked for: both fetches run under the MMA.
    struct Chunk {
      int si;  // ns: none
      uint32_t t0, te;
    };
    auto after = [&](Chunk c) {
      c.t0 += kChunk;
      if (c.t0 >= c.te && c.si < ns && ++c.si < ns) {
        c.t0 = bounds[c.si].x;
        c.te = bounds[c.si].y;
      }
      return c;
    };
    auto entry = [&](const Chunk &c) { return c.si < ns && c.t0 + lane < c.te ? lst[c.t0 + lane] : 0ull; };
    Chunk c0{0, bounds[0].x, bounds[0].y}, c1 = after(c0);
    uint64_t e = entry(c0), e1 = entry(c1);
    uint4 ca = cell[sinks[0]], cb = cell[pair_src(e)];
    for (bool first = true; c0.si < ns;) {
      const int si = c0.si;
      const uint32_t cnt = c0.te - c0.t0 < (uint32_t)kChunk ? c0.te - c0.t0 : (uint32_t)kChunk;
      const bool valid = (uint32_t)lane < cnt;
      if (warp != 1) {  // D': a third of the coefficients each
        float rx = 1.f, ry = 0.f, rz = 0.f, x = 1.f, u = 0.f;
        if (valid) {
          int dd[3];
          half_delta32(ca, cb, pair_shift(e), dd);
          const float Rx = -(float)dd[0], Ry = -(float)dd[1], Rz = -(float)dd[2];
          const float r2 = Rx * Rx + Ry * Ry + Rz * Rz;
          const float rinv = rsqrtf(r2);
          rx = Rx * rinv;
          ry = Ry * rinv;
          rz = Rz * rinv;
          x = r2 * rinv * inv_rs;
          u = (float)(2 * half_width(ca.w)) * rinv;
        }
        float f[P + 1];
        f[0] = erfcf(0.5f * x);
        float tk = -x * kInvSqrtPi * __expf(-0.25f * x * x);
        const float hx2 = 0.5f * x * x;
#pragma unroll
        for (int q = 0; q < P; ++q) {
          f[q + 1] = -(float)(2 * q + 1) * f[q] + tk;
          tk = -tk * hx2;
        }
        float U[P + 1];
        U[0] = u;
#pragma unroll
        for (int q = 1; q <= P; ++q) U[q] = U[q - 1] * u;
        T *hi = reinterpret_cast<T *>(a_hi), *lo = reinterpret_cast<T *>(a_lo);
        using Store = typename std::conditional<kBF, TCStoreBF<P>, TCStore<P>>::type;
        if (warp == 0) Store::template store_d<3, 0>(rx, ry, rz, f, U, hi, lo, xo);
        else if (warp == 2) Store::template store_d<3, 1>(rx, ry, rz, f, U, hi, lo, xo);
        else Store::template store_d<3, 2>(rx, ry, rz, f, U, hi, lo, xo);
      } else {
        const float vr = (float)half_width(cb.w) / (float)half_width(ca.w);  // v / u = h_B / h_A
        const float *Mb = M + (size_t)pair_src(e) * ldm;
        T *hi = reinterpret_cast<T *>(b_hi), *lo = reinterpret_cast<T *>(b_lo);
        if constexpr (kBF) TCStoreBF<P>::store_m(Mb, vr, valid ? 1.f : 0.f, hi, lo, xo);
        else TCStore<P>::store_m(Mb, vr, valid ? 1.f : 0.f, hi, lo, xo);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      sync();
      if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t steps = (cnt + kStep - 1) / kStep;
        for (uint32_t j = 0; j < steps; ++j) {
          const uint32_t off = j * 32;
          const uint64_t ah = desc_sw128(smem_u32(a_hi) + off), al = desc_sw128(smem_u32(a_lo) + off);
          const uint64_t bh = desc_sw128(smem_u32(b_hi) + off), bl = desc_sw128(smem_u32(b_lo) + off);
          const uint32_t acc = (!first || j != 0) ? 1u : 0u;
          if constexpr (kBF) {
            mma_bf16(tmem, ah, bh, IDESC, acc);
            mma_bf16(tmem, ah, bl, IDESC, 1u);
            mma_bf16(tmem, al, bh, IDESC, 1u);
          } else {
            mma_tf32(tmem, ah, bh, IDESC, acc);
            mma_tf32(tmem, ah, bl, IDESC, 1u);
            mma_tf32(tmem, al, bh, IDESC, 1u);
          }
        }
        mma_commit(mb);
      }
      c0 = c1;
      c1 = after(c1);
      e = e1;
      if (c0.si < ns) {
        ca = cell[sinks[c0.si]];
        cb = cell[pair_src(e)];
      }
      e1 = entry(c1);
      const bool ok = mbar_wait(mb, phase, chunk_wait);
      phase ^= 1u;
      if (!ok && lane == 0) {
        atomicExch(status, 1);
        abort_flag = 1;
      }
      sync();
      if (abort_flag) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      first = c0.si != si;
      if (!first) continue;  // more chunks of this sink
      // ---- TMEM rows 32 warp + lane hold P[c][0..NCP); stage rows c < NC
      const int c = warp * 32 + lane;
      if (warp * 32 < NC) {
#pragma unroll
        for (int col = 0; col < NCP; col += 16) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)col, v);
          if (c < NC) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (col + i < NC) pbuf[c * kLd + col + i] = v[i];
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      sync();
      // ---- four lanes an output, every fourth term each
      for (int o = tid; o < 4 * NC; o += 128) {
        const int n = o >> 2;
        float acc = 0.f;
        for (int e = tbeg[n] + (o & 3); e < tbeg[n + 1]; e += 4) acc += pbuf[place[e]];
        const unsigned quad = 0xfu << (lane & 28);
        acc += __shfl_xor_sync(quad, acc, 1);
        acc += __shfl_xor_sync(quad, acc, 2);
        if ((o & 3) == 0) atomicAdd(L + (size_t)sinks[si] * ldm + n, acc);  // no other warp does
      }
      sync();  // the operand tiles are rewritten
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (abort_flag) break;
  }
  // the MMAs of an abandoned chunk may still be running: wait for them with the
  // full limit before the tensor memory they write is freed
  if (abort_flag && tid == 0) mbar_wait(mb, phase ^ 1u, kWaitLimit);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem0), "r"(TCOLS));
}

template <int P, bool kBF>
cudaError_t launch_tc(Ctx &c, cudaStream_t st) {
  const size_t smem = smem_of(P);
  cudaError_t e = cudaFuncSetAttribute(k_m2l_tc<P, kBF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // d_small[5] = work counter, d_small[6] = status word
  unsigned long long *ctr = reinterpret_cast<unsigned long long *>(hfmm::P<uint64_t>(c.d_small) + 5);
  int *status = reinterpret_cast<int *>(hfmm::P<uint64_t>(c.d_small) + 6);
  if ((e = cudaMemsetAsync(ctr, 0, 8, st)) != cudaSuccess) return e;  // the status word is zeroed once per call
  int nsm = 0, dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const unsigned grid = std::min((unsigned)nsm, blocks_for((size_t)c.nnodes, kSinkBatch));  // persistent
  const float inv_rs = (float)(c.prm.box / (double)kHalfBox / c.rs);
  k_m2l_tc<P, kBF><<<grid, 128 * workers_of(P), smem, st>>>(
      c.nnodes, hfmm::P<uint4>(c.cell), hfmm::P<uint32_t>(c.m2l_beg), hfmm::P<uint32_t>(c.m2l_end),
      hfmm::P<uint64_t>(c.m2l), hfmm::P<float>(c.M), hfmm::P<float>(c.L), c.ldm, inv_rs, ctr, status,
      c.prm.tc_wait_polls > 0 ? (uint32_t)c.prm.tc_wait_polls : c.prm.tc_wait_polls < 0 ? 0u : kWaitLimit);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

bool m2l_tc_supported(int p) { return p >= 1 && p <= 6; }

cudaError_t m2l_pass_tc(Ctx &c, int q, cudaStream_t st) {
  if (c.nm2l == 0 || c.nnodes == 0) return cudaSuccess;
  const bool bf = c.prm.m2l_precision == 2;
  switch (q) {
    case 1: return bf ? launch_tc<1, true>(c, st) : launch_tc<1, false>(c, st);
    case 2: return bf ? launch_tc<2, true>(c, st) : launch_tc<2, false>(c, st);
    case 3: return bf ? launch_tc<3, true>(c, st) : launch_tc<3, false>(c, st);
    case 4: return bf ? launch_tc<4, true>(c, st) : launch_tc<4, false>(c, st);
    case 5: return bf ? launch_tc<5, true>(c, st) : launch_tc<5, false>(c, st);
    case 6: return bf ? launch_tc<6, true>(c, st) : launch_tc<6, false>(c, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hfmm
