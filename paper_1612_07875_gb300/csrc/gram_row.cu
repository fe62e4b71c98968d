// Streaming Gram row: the one new row/column of G = X^H X per pushed snapshot
// (Sec. 3.1, Eq. 12b; Algorithm 1, the X^T X[:, -1] product). Every resident
// snapshot x_j is dotted with the new snapshot x_new; O(n m) work that reads
// each window byte exactly once, so the kernel is HBM-bound.
//
// Decomposition: the n dimension (bytes, padded to whole 4 KiB units) is cut
// into `nblk` contiguous chunks of up to 24 KiB, about two per SM. A work
// item is one chunk of one of `groups` interleaved sets of eight slots (slot
// rows jj with (jj / 8) % groups == g). One persistent CTA per SM takes items
// from a counter (atomicAdd), so a launch is not held back by SMs that
// another stream's kernel occupies: thread 0 brings the chunk of x_new into
// shared memory with one bulk copy (TMA, cp.async.bulk), then each of the 8
// warps streams its slots (warp w takes rows jj = w mod 8) in 4 KiB pieces
// through its own 4-stage shared-memory ring: lane 0 issues cp.async.bulk
// copies that complete on one mbarrier per stage, the lanes wait on the
// barrier, consume the piece (16 bytes per lane per step) and hand the stage
// back. That keeps 128 KiB of loads in flight per SM without register
// pressure, and the rings run on into the next item. Each slot's chunk sum is
// reduced with warp shuffles and goes to a [slot][chunk] array; the CTA that
// completes a group's last chunk (atomic count, no waiting) sums its partials
// in a fixed order and writes its entries of row and column `s_new` of G, so
// the result depends neither on which CTA took which item nor on the number
// of groups. The count's fence and round trip would lengthen every hand-over
// between two items, so its answer is looked at one item later (n = 2^28 bytes:
// 16 slots 819 -> 770 us, 8 slots 509 -> 465).
//
// The new snapshot. With x_src set (a 16-byte aligned device buffer) the
// kernel also is the ingest: x_new's chunks come from x_src, the items of
// group 0 write them to the ring slot, and <x_new, x_new> is formed from the
// staged chunk, so the snapshot is read once and its slot not at all. Against
// a copy kernel before this one a push of one HD frame (m = 100) went from 125
// to 116 us, one of a 64 x 64 FP32 field (m = 32, launches only) from 22.5 to
// 14.3 us. (Snapshots of 2^28 bytes in windows of 64 and more slots, 17 GB, are
// the exception: 2,545 us with the copy, 2,578.)
//
//  - uint8: __dp4a (4 u8 x u8 products into u32). A lane sums at most
//    24 KiB / 32 = 768 products (< 2^32 / 255^2) before the value goes to
//    int64, so the result is exact and independent of order.
//  - float32: four FP32 FMA chains of 8 products per piece per lane, then the
//    piece's sum is added in FP64; cross-lane and cross-CTA sums are FP64 in a
//    fixed order, so results are deterministic for a given schedule.
//  - complex64: the same with conj(x_j) x_new split into real and imaginary
//    FP32 chains; G is Hermitian (complex128).
//
// Every mbarrier wait is bounded (about one second of SM clock); on expiry
// the kernel raises kDevTimeout in the handle's status word, stops issuing
// copies, waits (bounded) for the copies it has in flight, and finishes. The
// row is then incomplete, but the snapshot is not: with x_src the CTAs that
// gave up still copy it into its slot (plain loads and stores, nothing to wait
// for), so a rebuild of the window restores G.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "sdmd_internal.cuh"

namespace sdmd {

namespace {

constexpr int kStages = 4;
constexpr int kPiece = 4096;                       // bytes per bulk copy
constexpr int kXSub = 24576;                       // largest chunk (x_new bytes staged per chunk)
static_assert(kXSub / 32 * 255LL * 255LL < (1LL << 32), "a lane's uint8 sum over a chunk stays in 32 bits");
// Bound of a wait, ~1 s at 2 GHz. A test compiles this file with a short bound
// and with the x_new barrier of every CTA's item number SDMD_GR_STARVED_ITEM
// told to expect 16 bytes that nobody sends, so that its wait expires.
#ifndef SDMD_GR_WAIT_CYCLES
#define SDMD_GR_WAIT_CYCLES 2000000000LL
#endif
#ifndef SDMD_GR_STARVED_ITEM
#define SDMD_GR_STARVED_ITEM -1
#endif
constexpr long long kWaitCycles = SDMD_GR_WAIT_CYCLES;
constexpr int kStarvedItem = SDMD_GR_STARVED_ITEM;

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// shared -> global bulk copy of this thread's bulk group, and the waits for
// it: source read (the buffer may be refilled), and complete
__device__ __forceinline__ void bulk_s2g(void* dst, unsigned src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void bulk_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ void fence_acq_rel() { asm volatile("fence.acq_rel.gpu;\n" ::: "memory"); }

// Bounded wait on phase `parity` of barrier `bar`; false on expiry.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
  if (mbar_try(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try(bar, parity)) {
    if (clock64() - t0 > kWaitCycles) return false;
  }
  return true;
}

struct Smem {
  uint8_t stage[kGrWarps][kStages][kPiece];   // per-warp piece rings
  uint8_t xs[2][kXSub];                       // x_new chunks of the current and the next item
  unsigned long long bar[kGrWarps][kStages];  // one mbarrier per stage
  unsigned long long xbar[2];                 // x_new barriers
  int iq[2];                                  // index of item ordinal k at [k & 1]
  int fail;                                   // a wait expired in some warp
  int quit;                                   // fail as thread 0 saw it between two items
  int last;                                   // group whose last chunk this CTA completed, -1: none
};

// Element modes of the kernel.
// kModeF64: FP32 snapshots with FP64 products and sums (the reference Gram;
// a product of two FP32 values is exact in FP64).
enum { kModeU8 = 0, kModeF32 = 1, kModeC64 = 2, kModeF64 = 3 };

// One 4 KiB piece of a slot against the same piece of x_new, added to this
// lane's sums (16 bytes per lane and step).
template <int kMode>
__device__ __forceinline__ void piece_sums(const uint8_t* piece, const uint8_t* xq, int lane, unsigned& su, double& sd,
                                           double& si) {
  if constexpr (kMode == kModeU8) {
#pragma unroll
    for (int u = 0; u < kPiece / 512; ++u) {
      const uint4 v = *reinterpret_cast<const uint4*>(piece + 16 * lane + 512 * u);
      const uint4 w = *reinterpret_cast<const uint4*>(xq + 16 * lane + 512 * u);
      su = __dp4a(v.x, w.x, su);
      su = __dp4a(v.y, w.y, su);
      su = __dp4a(v.z, w.z, su);
      su = __dp4a(v.w, w.w, su);
    }
  } else if constexpr (kMode == kModeF32) {
    float f0 = 0.f, f1 = 0.f, f2 = 0.f, f3 = 0.f;
#pragma unroll
    for (int u = 0; u < kPiece / 512; ++u) {
      const float4 v = *reinterpret_cast<const float4*>(piece + 16 * lane + 512 * u);
      const float4 w = *reinterpret_cast<const float4*>(xq + 16 * lane + 512 * u);
      f0 = fmaf(v.x, w.x, f0);
      f1 = fmaf(v.y, w.y, f1);
      f2 = fmaf(v.z, w.z, f2);
      f3 = fmaf(v.w, w.w, f3);
    }
    sd += (double)((f0 + f1) + (f2 + f3));
  } else if constexpr (kMode == kModeF64) {
    double d0 = 0.0, d1 = 0.0, d2 = 0.0, d3 = 0.0;
#pragma unroll
    for (int u = 0; u < kPiece / 512; ++u) {
      const float4 v = *reinterpret_cast<const float4*>(piece + 16 * lane + 512 * u);
      const float4 w = *reinterpret_cast<const float4*>(xq + 16 * lane + 512 * u);
      d0 = fma((double)v.x, (double)w.x, d0);
      d1 = fma((double)v.y, (double)w.y, d1);
      d2 = fma((double)v.z, (double)w.z, d2);
      d3 = fma((double)v.w, (double)w.w, d3);
    }
    sd += (d0 + d1) + (d2 + d3);
  } else {
    float r0 = 0.f, r1 = 0.f, i0 = 0.f, i1 = 0.f;
#pragma unroll
    for (int u = 0; u < kPiece / 512; ++u) {
      const float4 v = *reinterpret_cast<const float4*>(piece + 16 * lane + 512 * u);
      const float4 w = *reinterpret_cast<const float4*>(xq + 16 * lane + 512 * u);
      r0 = fmaf(v.x, w.x, fmaf(v.y, w.y, r0));
      r1 = fmaf(v.z, w.z, fmaf(v.w, w.w, r1));
      i0 = fmaf(v.x, w.y, fmaf(-v.y, w.x, i0));
      i1 = fmaf(v.z, w.w, fmaf(-v.w, w.z, i1));
    }
    sd += (double)(r0 + r1);
    si += (double)(i0 + i1);
  }
}

// acc[0 .. 2] of one (slot, chunk): the lanes' sums reduced over the warp and
// stored by lane 0.
template <int kMode>
__device__ __forceinline__ void store_partial(void* partials, int64_t at, int lane, unsigned su, double sd, double si) {
  if constexpr (kMode == kModeU8) {
    const long long t = warp_sum((long long)su);
    if (lane == 0) static_cast<long long*>(partials)[at] = t;
  } else if constexpr (kMode == kModeC64) {
    const double t = warp_sum(sd), ti = warp_sum(si);
    if (lane == 0) static_cast<double2*>(partials)[at] = make_double2(t, ti);
  } else {
    const double t = warp_sum(sd);
    if (lane == 0) static_cast<double*>(partials)[at] = t;
  }
}

// Sum over the chunks of one row of partials in a fixed order (lane-strided
// sums, then the butterfly); kFinLoads loads are in flight per lane.
constexpr int kFinLoads = 8;
template <typename T>
__device__ __forceinline__ T chunk_sum(const T* P, int nblk, int lane) {
  T s = 0;
  for (int b = lane; b < nblk; b += 32 * kFinLoads) {
    T v[kFinLoads];
#pragma unroll
    for (int u = 0; u < kFinLoads; ++u) v[u] = (b + 32 * u < nblk) ? __ldcg(P + b + 32 * u) : T(0);
#pragma unroll
    for (int u = 0; u < kFinLoads; ++u)
      if (b + 32 * u < nblk) s += v[u];
  }
  return warp_sum(s);
}
__device__ __forceinline__ double2 chunk_sum_c64(const double2* P, int nblk, int lane) {
  double sr = 0.0, si = 0.0;
  for (int b = lane; b < nblk; b += 32 * kFinLoads) {
    double2 v[kFinLoads];
#pragma unroll
    for (int u = 0; u < kFinLoads; ++u) v[u] = (b + 32 * u < nblk) ? __ldcg(P + b + 32 * u) : make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < kFinLoads; ++u)
      if (b + 32 * u < nblk) {
        sr += v[u].x;
        si += v[u].y;
      }
  }
  return make_double2(warp_sum(sr), warp_sum(si));
}

// G's entries of row jj (this warp): row and column s_new, physical slots.
// Complex: G[j][s_new] = <x_j, x_new> = g_j and G[s_new][j] = conj(g_j).
template <int kMode>
__device__ __forceinline__ void finish_slot(const void* partials, int nblk, int jj, void* G, int s_first, int s_new,
                                            int m, int lane) {
  int j = s_first + jj;
  if (j >= m) j -= m;
  if constexpr (kMode == kModeC64) {
    double2 v = chunk_sum_c64(static_cast<const double2*>(partials) + (int64_t)jj * nblk, nblk, lane);
    if (j == s_new) v.y = 0.0;         // <x, x> is real; drop the rounding residue
    if (lane == 0) {
      double2* g = static_cast<double2*>(G);
      g[(int64_t)j * m + s_new] = v;
      g[(int64_t)s_new * m + j] = make_double2(v.x, -v.y);
    }
  } else {
    using Acc = typename std::conditional<kMode == kModeU8, long long, double>::type;
    const Acc v = chunk_sum<Acc>(static_cast<const Acc*>(partials) + (int64_t)jj * nblk, nblk, lane);
    if (lane == 0) {
      Acc* g = static_cast<Acc*>(G);
      g[(int64_t)s_new * m + j] = v;
      g[(int64_t)j * m + s_new] = v;
    }
  }
}

// After an expired wait (the whole CTA): the chunks of the snapshot that
// belong to the items at hand (it0, it1) and to those nobody has taken yet go
// from the caller's buffer to the ring slot. Chunks that were stored already
// get the same bytes again.
__device__ void ingest_rest(const GramRowArgs& a, Smem& sm, int it0, int it1, int nitems) {
  uint8_t* slot = const_cast<uint8_t*>(a.ring) + (int64_t)a.s_new * a.slot_bytes;
  for (int q = 0;; ++q) {
    int it = q == 0 ? it0 : it1;
    if (q >= 2) {
      __syncthreads();
      if (threadIdx.x == 0) sm.iq[0] = (int)atomicAdd(a.ticket + 1, 1u);
      __syncthreads();
      it = sm.iq[0];
      if (it >= nitems) return;
    }
    if (it >= nitems || it % a.groups != 0) continue;
    const int64_t off = (int64_t)(it / a.groups) * a.chunk, len = min(a.chunk, a.x_bytes - off);
    const int64_t nv = len > 0 ? len / 16 : 0;
    for (int64_t v = threadIdx.x; v < nv; v += kGrThreads)
      reinterpret_cast<uint4*>(slot + off)[v] = reinterpret_cast<const uint4*>(a.x_src + off)[v];
    for (int64_t b = 16 * nv + threadIdx.x; b < len; b += kGrThreads) slot[off + b] = a.x_src[off + b];
  }
}

template <int kMode>
__global__ void __launch_bounds__(kGrThreads, 1) gram_row_bulk_kernel(GramRowArgs a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int w = 0; w < kGrWarps; ++w)
      for (int s = 0; s < kStages; ++s) mbar_init(smem_u32(&sm.bar[w][s]), 1);
    mbar_init(smem_u32(&sm.xbar[0]), 1);
    mbar_init(smem_u32(&sm.xbar[1]), 1);
    sm.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  const int S = a.groups, nitems = a.nblk * S;
  const bool src = a.x_src != nullptr;
  const uint8_t* xnew = src ? a.x_src : a.ring + (int64_t)a.s_new * a.slot_bytes;
  const int64_t xbytes = src ? a.x_bytes : a.slot_bytes;   // readable bytes at xnew
  // the newest snapshot (window row c - 1) is dotted from its staged chunk
  const int self = (a.s_new == (a.s_first + a.c - 1) % a.m) ? a.c - 1 : -1;
  const int cs = (self >= 0) ? a.c - 1 : a.c;              // rows streamed from the ring
  auto chunk_len = [&](int ch) -> int { return (int)min(a.chunk, a.slot_bytes - (int64_t)ch * a.chunk); };
  // bytes of chunk ch that a bulk copy may read (a multiple of 16)
  auto bulk_len = [&](int ch) -> int {
    const int64_t rest = xbytes - (int64_t)ch * a.chunk;
    return rest <= 0 ? 0 : ((int)min((int64_t)chunk_len(ch), rest) & ~15);
  };
  auto rows_of = [&](int g) -> int {                       // streamed rows of this warp in group g
    const int r0 = warp + kGrWarps * g;
    return (r0 < cs) ? (cs - 1 - r0) / (kGrWarps * S) + 1 : 0;
  };
  auto issue_x = [&](int k, int it) {                      // x_new's chunk of item ordinal k
    const int ch = it / S;
    const unsigned xb = smem_u32(&sm.xbar[k & 1]);
    const int len = bulk_len(ch);
    mbar_expect_tx(xb, (unsigned)len + (kStarvedItem >= 0 && k == kStarvedItem ? 16u : 0u));
    if (len > 0) bulk_g2s(smem_u32(sm.xs[k & 1]), xnew + (int64_t)ch * a.chunk, (unsigned)len, xb);
  };
  if (threadIdx.x == 0) {
    const int i0 = (int)atomicAdd(a.ticket + 1, 1u);
    sm.iq[0] = i0;
    if (i0 < nitems) issue_x(0, i0);
  }
  // this warp's piece stream: lane 0 keeps the ring kStages pieces ahead, into
  // item ordinal k + 1 once it is known
  unsigned consumed = 0, issued = 0;   // pieces of this warp (all items)
  int kc = 0, ci = 0, cq = 0, cnp = 0, crows = 0, cg = 0, cch = 0;   // issue cursor (lane 0)
  const uint8_t* csrc = nullptr;
  bool loaded = false;                 // the cursor holds item ordinal kc
  bool failed = false;                 // a bounded wait expired: stop issuing, drain, finish
  auto slot_src = [&]() {
    int j = a.s_first + warp + kGrWarps * (cg + S * ci);
    if (j >= a.m) j -= a.m;
    csrc = a.ring + (int64_t)j * a.slot_bytes + (int64_t)cch * a.chunk;
  };
  auto top_up = [&](int k) {           // item ordinals k and k + 1 are known
    if (lane != 0 || failed) return;
    while (issued - consumed < (unsigned)kStages) {
      if (!loaded) {
        if (kc > k + 1) break;
        const int it = sm.iq[kc & 1];
        if (it >= nitems) break;
        cch = it / S;
        cg = it - cch * S;
        cnp = chunk_len(cch) / kPiece;
        crows = rows_of(cg);
        ci = cq = 0;
        loaded = true;
        if (crows > 0) slot_src();
      }
      if (ci >= crows) {
        ++kc;
        loaded = false;
        continue;
      }
      const unsigned s = issued % kStages;
      const unsigned b = smem_u32(&sm.bar[warp][s]);
      mbar_expect_tx(b, kPiece);
      bulk_g2s(smem_u32(sm.stage[warp][s]), csrc, kPiece, b);
      ++issued;
      csrc += kPiece;
      if (++cq == cnp) {
        cq = 0;
        if (++ci < crows) slot_src();
      }
    }
  };
  auto finish_group = [&](int g) {     // a group whose chunks are all in: its entries of G
    if (g < 0) return;
    for (int jj = warp + kGrWarps * g; jj < a.c; jj += kGrWarps * S)
      finish_slot<kMode>(a.partials, a.nblk, jj, a.G, a.s_first, a.s_new, a.m, lane);
  };
  int gprev = -1, itprev = -1;         // group and index of the item before
  int counted = -1;                    // (thread 32) group of the count on its way
  unsigned count = 0;
  for (int k = 0;; ++k) {
    __syncthreads();                   // item k - 1 consumed, its partials written: xs[(k + 1) & 1] is free
    if (threadIdx.x == 0) {
      const int it = sm.iq[k & 1];
      int nx = nitems;
      if (it < nitems && !sm.fail) nx = (int)atomicAdd(a.ticket + 1, 1u);
      sm.iq[(k + 1) & 1] = nx;
      sm.quit = sm.fail;
      if (nx < nitems) {
        if (src) bulk_store_wait_read(); // the store that still reads that buffer
        issue_x(k + 1, nx);
      }
    } else if (threadIdx.x == 32) {
      // item k - 2's count, asked for an item ago, is in by now
      const int last = (counted >= 0 && count == (unsigned)a.nblk - 1u) ? counted : -1;
      counted = -1;
      if (gprev >= 0 && !sm.fail) {    // count item k - 1 (the barrier ordered its partials before the fence)
        fence_acq_rel();
        count = atomicAdd(a.ticket + kGrTicketGroups + gprev, 1u);
        counted = gprev;
      }
      if (last >= 0) fence_acq_rel();
      sm.last = last;
    }
    __syncthreads();
    finish_group(sm.last);
    const int it = sm.iq[k & 1];
    if (sm.quit) {
      // copies issued but not consumed must land before the shared memory
      // is released (bounded waits); then stop
      if (lane == 0)
        for (unsigned gk = consumed; gk < issued; ++gk) mbar_wait(smem_u32(&sm.bar[warp][gk % kStages]), (gk / kStages) & 1);
      if (threadIdx.x == 0) {          // (item k - 1's may be the wait that expired)
        mbar_wait(smem_u32(&sm.xbar[(k - 1) & 1]), (unsigned)(((k - 1) >> 1) & 1));
        if (it < nitems) mbar_wait(smem_u32(&sm.xbar[k & 1]), (unsigned)((k >> 1) & 1));
      }
      if (src) ingest_rest(a, sm, itprev, it, nitems);
      break;
    }
    if (it >= nitems) {                // the count of this CTA's last item
      __syncthreads();
      if (threadIdx.x == 32) {
        sm.last = (counted >= 0 && count == (unsigned)a.nblk - 1u) ? counted : -1;
        fence_acq_rel();
      }
      __syncthreads();
      finish_group(sm.last);
      break;
    }
    const int ch = it / S, g = it - ch * S;
    gprev = g;
    itprev = it;
    const int np = chunk_len(ch) / kPiece, rows = rows_of(g);
    uint8_t* xs = sm.xs[k & 1];
    top_up(k);
    if (src && bulk_len(ch) < chunk_len(ch)) {
      // the last bytes of the snapshot (n mod 16) and the zero padding after it
      const int b0 = bulk_len(ch);
      const int64_t off = (int64_t)ch * a.chunk;
      for (int b = b0 + threadIdx.x; b < chunk_len(ch); b += kGrThreads) xs[b] = (off + b < xbytes) ? xnew[off + b] : 0;
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncthreads();
    }
    if (!failed && !mbar_wait(smem_u32(&sm.xbar[k & 1]), (unsigned)((k >> 1) & 1))) failed = true;
    failed = __any_sync(0xffffffffu, failed);
    if (src && g == 0 && !failed) {    // the ingest of this chunk
      uint8_t* dst = const_cast<uint8_t*>(a.ring) + (int64_t)a.s_new * a.slot_bytes + (int64_t)ch * a.chunk;
      const int len = bulk_len(ch);
      if (threadIdx.x == 0 && len > 0) bulk_s2g(dst, smem_u32(xs), (unsigned)len);
      const int b = len + (int)threadIdx.x;
      if (threadIdx.x < 16 && len < chunk_len(ch) && (int64_t)ch * a.chunk + b < xbytes) dst[b] = xs[b];
    }
    for (int i = 0; i < rows && !failed; ++i) {
      unsigned su = 0;
      double sd = 0.0, si = 0.0;
      for (int q = 0; q < np; ++q) {
        const unsigned s = consumed % kStages, par = (consumed / kStages) & 1;
        const bool bad = !mbar_wait(smem_u32(&sm.bar[warp][s]), par);
        if (__any_sync(0xffffffffu, bad)) {
          failed = true;
          break;
        }
        piece_sums<kMode>(sm.stage[warp][s], xs + kPiece * q, lane, su, sd, si);
        __syncwarp();                  // all lanes are done reading stage s
        ++consumed;
        top_up(k);
      }
      if (!failed)
        store_partial<kMode>(a.partials, (int64_t)(warp + kGrWarps * (g + S * i)) * a.nblk + ch, lane, su, sd, si);
    }
    if (self >= 0 && !failed && self % kGrWarps == warp && (self / kGrWarps) % S == g) {
      unsigned su = 0;
      double sd = 0.0, si = 0.0;
      for (int q = 0; q < np; ++q) piece_sums<kMode>(xs + kPiece * q, xs + kPiece * q, lane, su, sd, si);
      store_partial<kMode>(a.partials, (int64_t)self * a.nblk + ch, lane, su, sd, si);
    }
    if (failed && lane == 0) {
      atomicOr(a.status, kDevTimeout);
      sm.fail = 1;
    }
  }
  // the ring copies are complete before the CTA's shared memory goes; the last
  // CTA out zeroes the counters for the next launch
  if (threadIdx.x == 0) {
    if (src) bulk_store_wait_all();
    __threadfence();
    if (atomicAdd(a.ticket, 1u) == gridDim.x - 1u) {
      for (int q = 0; q < S; ++q) a.ticket[kGrTicketGroups + q] = 0u;
      a.ticket[1] = 0u;
      a.ticket[0] = 0u;
    }
  }
}

// ---------------------------------------------------------------------------
// Batched rows: one new snapshot of each of up to kMaxBatchJobs handles (mixed
// n, window and element type) in one launch. Work items are (job, chunk)
// pairs over the concatenated chunk lists, taken from a counter by
// persistent CTAs. Each item is computed exactly as the single-handle kernel
// computes that chunk (same warp-to-slot assignment, piece order and per-lane
// sums), its partials go to the job's [slot][chunk] array, and the CTA that
// completes a job's last chunk reduces the job's row in the same fixed order,
// so every row is bit-identical to the handle's own sdmd_push.

struct BatchSmem {
  uint8_t stage[kGrWarps][kStages][kPiece];
  uint8_t xs[kXSub];
  unsigned long long bar[kGrWarps][kStages];
  unsigned long long xbar;
  int item, job, ch, fail, last;
  long long acc_i[SDMD_MAX_M];
  double acc_d[SDMD_MAX_M];
  double acc_im[SDMD_MAX_M];
};

// One item: chunk `ch` of job `J`; returns false if a wait expired.
template <int kMode>
__device__ bool batch_item(const RowJob& J, int ch, BatchSmem& sm, unsigned& g, int item_no) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t beg = (int64_t)ch * J.chunk;
  const int len = (int)min(J.chunk, J.slot_bytes - beg);
  const int np = len / kPiece;
  const int nmine = (J.c > warp) ? (J.c - warp + kGrWarps - 1) / kGrWarps : 0;
  const int nitems = nmine * np;
  const uint8_t* xnew = J.ring + (int64_t)J.s_new * J.slot_bytes;
  if (threadIdx.x == 0) {
    const unsigned xb = smem_u32(&sm.xbar);
    mbar_expect_tx(xb, (unsigned)len);
    bulk_g2s(smem_u32(sm.xs), xnew + beg, (unsigned)len, xb);
  }
  auto issue = [&](int it) {
    const unsigned s = (g + it) % kStages;
    const int j = (J.s_first + warp + kGrWarps * (it / np)) % J.m;
    const unsigned b = smem_u32(&sm.bar[warp][s]);
    mbar_expect_tx(b, kPiece);
    bulk_g2s(smem_u32(sm.stage[warp][s]), J.ring + (int64_t)j * J.slot_bytes + beg + (int64_t)kPiece * (it % np), kPiece,
             b);
  };
  if (lane == 0)
    for (int it = 0; it < kStages && it < nitems; ++it) issue(it);
  bool failed = !mbar_wait(smem_u32(&sm.xbar), (unsigned)(item_no & 1));
  failed = __any_sync(0xffffffffu, failed);
  int consumed = 0;
  unsigned su = 0;
  double sd = 0.0, si = 0.0;
  for (int it = 0; it < nitems && !failed; ++it) {
    const unsigned gi = g + it, s = gi % kStages, par = (gi / kStages) & 1;
    const int q = it % np;
    const bool bad = !mbar_wait(smem_u32(&sm.bar[warp][s]), par);
    if (__any_sync(0xffffffffu, bad)) {
      failed = true;
      break;
    }
    piece_sums<kMode>(sm.stage[warp][s], sm.xs + kPiece * q, lane, su, sd, si);
    __syncwarp();
    ++consumed;
    if (lane == 0 && it + kStages < nitems) issue(it + kStages);
    if (q == np - 1) {
      const int jj = warp + kGrWarps * (it / np);
      if constexpr (kMode == kModeU8) {
        const long long t = warp_sum((long long)su);
        if (lane == 0) sm.acc_i[jj] += t;
        su = 0;
      } else {
        const double t = warp_sum(sd);
        if (lane == 0) sm.acc_d[jj] += t;
        sd = 0.0;
        if constexpr (kMode == kModeC64) {
          const double ti = warp_sum(si);
          if (lane == 0) sm.acc_im[jj] += ti;
          si = 0.0;
        }
      }
    }
  }
  if (failed && lane == 0) {           // copies in flight land before the memory is reused
    const int issued = nitems < consumed + kStages ? nitems : consumed + kStages;
    for (int it = consumed; it < issued; ++it) mbar_wait(smem_u32(&sm.bar[warp][(g + it) % kStages]), ((g + it) / kStages) & 1);
    mbar_wait(smem_u32(&sm.xbar), (unsigned)(item_no & 1));
  }
  g += nitems;
  return !failed;
}

template <int kMode>
__device__ void batch_finish(const RowJob& J) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int jj = warp; jj < J.c; jj += kGrWarps)
    finish_slot<kMode>(J.partials, J.nblk, jj, J.G, J.s_first, J.s_new, J.m, lane);
}

__global__ void __launch_bounds__(kGrThreads, 1) gram_rows_batched_kernel(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  BatchSmem& sm = *reinterpret_cast<BatchSmem*>(smem_raw);
  for (int j = threadIdx.x; j < SDMD_MAX_M; j += blockDim.x) {
    sm.acc_i[j] = 0;
    sm.acc_d[j] = 0.0;
    sm.acc_im[j] = 0.0;
  }
  if (threadIdx.x == 0) {
    for (int w = 0; w < kGrWarps; ++w)
      for (int s = 0; s < kStages; ++s) mbar_init(smem_u32(&sm.bar[w][s]), 1);
    mbar_init(smem_u32(&sm.xbar), 1);
    sm.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  unsigned g = 0;                      // this warp's pieces so far (ring position)
  for (int item_no = 0;; ++item_no) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const int it = sm.fail ? a.nitems : (int)atomicAdd(a.grab, 1u);
      int jb = 0;
      if (it < a.nitems)
        while (jb + 1 < a.njobs && a.job[jb + 1].item0 <= it) ++jb;
      sm.item = it;
      sm.job = jb;
      sm.ch = it - a.job[jb].item0;
    }
    __syncthreads();
    if (sm.item >= a.nitems) break;
    const RowJob& J = a.job[sm.job];
    const int ch = sm.ch;
    bool ok;
    if (J.mode == kModeU8) ok = batch_item<kModeU8>(J, ch, sm, g, item_no);
    else if (J.mode == kModeF32) ok = batch_item<kModeF32>(J, ch, sm, g, item_no);
    else if (J.mode == kModeF64) ok = batch_item<kModeF64>(J, ch, sm, g, item_no);
    else ok = batch_item<kModeC64>(J, ch, sm, g, item_no);
    if (!ok && (threadIdx.x & 31) == 0) {
      atomicOr(a.status, kDevTimeout);
      sm.fail = 1;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < J.c; j += blockDim.x) {
      if (J.mode == kModeU8) static_cast<long long*>(J.partials)[(int64_t)j * J.nblk + ch] = sm.acc_i[j];
      else if (J.mode == kModeF32 || J.mode == kModeF64)
        static_cast<double*>(J.partials)[(int64_t)j * J.nblk + ch] = sm.acc_d[j];
      else static_cast<double2*>(J.partials)[(int64_t)j * J.nblk + ch] = make_double2(sm.acc_d[j], sm.acc_im[j]);
      sm.acc_i[j] = 0;
      sm.acc_d[j] = 0.0;
      sm.acc_im[j] = 0.0;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) sm.last = (atomicAdd(J.ticket, 1u) == (unsigned)J.nblk - 1u);
    __syncthreads();
    if (sm.last) {                     // this job's chunks are all in: reduce its row
      __threadfence();
      if (J.mode == kModeU8) batch_finish<kModeU8>(J);
      else if (J.mode == kModeC64) batch_finish<kModeC64>(J);
      else batch_finish<kModeF32>(J);
      if (threadIdx.x == 0) J.ticket[0] = 0u;
    }
  }
  // the last CTA out zeroes the batch counters for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(a.grab + 1, 1u) == gridDim.x - 1u) {
      a.grab[0] = 0u;
      a.grab[1] = 0u;
    }
  }
}

}  // namespace

// Two chunks per SM: persistent CTAs take chunks as they free
// up, so a launch is not held back by SMs that another stream's kernel (a
// frame's eigensolver) occupies; the partials stay indexed by chunk, so the
// fixed-order reduction and the result do not change.
constexpr int kChunksPerSm = 2;

void gram_row_schedule(int64_t slot_bytes, int num_sms, int64_t* chunk, int32_t* nblk) {
  gram_row_schedule_k(slot_bytes, num_sms, kChunksPerSm, chunk, nblk);
}

void gram_row_schedule_k(int64_t slot_bytes, int num_sms, int chunks_per_sm, int64_t* chunk, int32_t* nblk) {
  const int64_t units = (slot_bytes + kPiece - 1) / kPiece;
  int64_t want = (int64_t)(chunks_per_sm > 0 ? chunks_per_sm : 1) * (num_sms > 0 ? num_sms : 1);
  if (want > units) want = units;
  int64_t per = (units + want - 1) / want;           // 4 KiB units per chunk
  if (per > kXSub / kPiece) per = kXSub / kPiece;   // at most 24 KiB (x_new double buffer)
  *chunk = per * kPiece;
  *nblk = (int32_t)((units + per - 1) / per);
}

// Groups of slot rows per chunk. An item's time is about its rows of eight
// slots (plus a fraction for its hand-over), and all items are alike, so the
// launch takes ceil(items / SMs) of them: the count with the least of that
// product. Sizes whose chunks divide evenly over the SMs keep one group (HD
// uint8: 304 chunks on 152 SMs); 338 chunks (FP32, n = 2,073,600) would take
// three rounds of whole chunks for 2.2 rounds of work and take seven of thirds
// instead: the row of a 120-snapshot window from 237 to about 165 us.
int gram_row_groups(int32_t nblk, int32_t c, int num_sms) {
  const int rows = (c + kGrWarps - 1) / kGrWarps;
  int best = 1;
  double cost = 1e300;
  for (int S = 1; S <= rows && S <= kGrMaxGroups; ++S) {
    const int64_t rounds = ((int64_t)nblk * S + num_sms - 1) / num_sms;
    const double t = (double)rounds * ((double)((rows + S - 1) / S) + 0.25);
    if (t < 0.999 * cost) {
      cost = t;
      best = S;
    }
  }
  return best;
}

template <int kMode>
static cudaError_t launch_gram_row_mode(const GramRowArgs& a, int ctas, cudaStream_t st) {
  const size_t smem = sizeof(Smem);
  const cudaError_t e = smem_optin(reinterpret_cast<const void*>(gram_row_bulk_kernel<kMode>), smem);
  if (e != cudaSuccess) return e;
  gram_row_bulk_kernel<kMode><<<ctas, kGrThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_gram_row(int dtype, bool f64_ref, const GramRowArgs& args, int num_sms, cudaStream_t st) {
  GramRowArgs a = args;
  const int sms = num_sms > 0 ? num_sms : 1;
  a.groups = gram_row_groups(a.nblk, a.c, sms);
  const int64_t items = (int64_t)a.nblk * a.groups;
  const int ctas = items < sms ? (int)items : sms;   // persistent
  if (dtype == SDMD_U8) return launch_gram_row_mode<kModeU8>(a, ctas, st);
  if (dtype == SDMD_C64) return launch_gram_row_mode<kModeC64>(a, ctas, st);
  if (f64_ref) return launch_gram_row_mode<kModeF64>(a, ctas, st);
  return launch_gram_row_mode<kModeF32>(a, ctas, st);
}

cudaError_t batched_kernel_config(const BatchArgs& a, cudaKernelNodeParams* p) {
  const size_t smem = sizeof(BatchSmem);
  {
    const cudaError_t e = smem_optin(reinterpret_cast<const void*>(gram_rows_batched_kernel), smem);
    if (e != cudaSuccess) return e;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int ctas = a.nitems < sms ? a.nitems : (sms > 0 ? sms : 1);
  p->func = reinterpret_cast<void*>(gram_rows_batched_kernel);
  p->gridDim = dim3((unsigned)(ctas > 0 ? ctas : 1));
  p->blockDim = dim3(kGrThreads);
  p->sharedMemBytes = (unsigned)smem;
  p->kernelParams = nullptr;
  p->extra = nullptr;
  return cudaSuccess;
}

cudaError_t launch_gram_rows_batched(const BatchArgs& a, cudaStream_t st) {
  const size_t smem = sizeof(BatchSmem);
  {
    const cudaError_t e = smem_optin(reinterpret_cast<const void*>(gram_rows_batched_kernel), smem);
    if (e != cudaSuccess) return e;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int ctas = a.nitems < sms ? a.nitems : (sms > 0 ? sms : 1);
  gram_rows_batched_kernel<<<ctas, kGrThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace sdmd
