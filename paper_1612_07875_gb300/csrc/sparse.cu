// Gram row of Fourier-sparse snapshots (Sec. 3.5): SVD and DMD are invariant
// under unitary transforms such as an orthonormal FFT, so the Gram entries of
// the physical fields equal the inner products of their transform
// coefficients (Parseval), and snapshots that are sparse in that basis give
// sparse inner products g_j = sum_{k in S_j and S_new} conj(a_j[k]) b[k].
//
// Per push, two kernels:
//  1. scatter: every coefficient (k, b_k) of the new snapshot goes into a
//     dense lookup table of length n: val[k] = b_k, tag[k] = stamp, where the
//     stamp is unique to this push, so the table is never cleared and a
//     position belongs to the new snapshot exactly when its tag matches. A
//     snapshot in device memory goes into its ring slot on the way.
//  2. row: CTAs cover (slot, 2048-entry chunk) pairs of the resident slots'
//     coefficient lists; each entry of slot j looks its index up in the table
//     (sparse x dense gather, L2-resident for n up to a few million) and
//     accumulates conj(a) b; products in FP32, per-thread sums in FP32 over
//     at most 8 terms, CTA and cross-CTA sums in FP64 in a fixed order; the
//     last CTA (atomic ticket, no waiting) writes row/column s_new of the
//     Hermitian G. The kernel is three dependent gathers deep (index, tag,
//     values), so a thread has its eight entries of each in flight together
//     (26 us one entry after the other at c = 64, nnz = 10,486), and in launches
//     of one short wave it loads the values before it knows the tags (a push
//     of that size 29.1 us, 30.5 after the tags). Larger launches are bound by
//     the gathers' sectors, where values of coefficients that the new snapshot
//     lacks cost more than they save: nnz = 167,772 of n = 2^24, 1 % shared, a
//     push 254 us with them, 106 without, 133 one entry after the other. Tables
//     of several hundred megabytes are gathered best one after the other: nnz =
//     671,088 of n = 2^26, 90 % shared, 985 us, 1,087 together.
// Indices outside [0, n) are skipped and raise kDevRange in the status word.
#include <cuda_runtime.h>
#include <stdint.h>

#include "sdmd_internal.cuh"

namespace sdmd {

namespace {

constexpr int kThreads = 256;
constexpr int kChunk = 2048;

__global__ void sparse_scatter_kernel(const int* idx, const float2* val, int nnz, int64_t n, int stamp,
                                      int* tag, float2* tval, int* ring_idx, float2* ring_val, int* status) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nnz) return;
  const int k = idx[i];
  const float2 v = val[i];
  if (ring_idx) {
    ring_idx[i] = k;
    ring_val[i] = v;
  }
  if (k < 0 || (int64_t)k >= n) {
    atomicOr(status, kDevRange);
    return;
  }
  tval[k] = v;
  tag[k] = stamp;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// How a thread takes its eight entries: one after the other, together, or
// together with the values loaded beside the tags whether or not the new
// snapshot has the coefficient. The sums are the same.
enum { kSerial = 0, kTogether = 1, kAhead = 2 };

template <int kHow>
__global__ void __launch_bounds__(kThreads) sparse_row_kernel(SparseRowArgs a) {
  __shared__ double red[2][kThreads / 32];
  __shared__ bool last;
  // CTA -> (window slot jj, chunk q): the last jj whose first CTA is not past this one
  int lo = 0, hi = a.c - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.chunk_start[mid] <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const int jj = lo;
  const int q = blockIdx.x - a.chunk_start[jj];
  const int slot = (a.s_first + jj) % a.m;
  const int nnz = a.nnz[slot];
  const int* idx = a.idx_ring + (int64_t)slot * a.nnz_max;
  const float2* val = a.val_ring + (int64_t)slot * a.nnz_max;
  const int e0 = q * kChunk, e1 = min(nnz, e0 + kChunk);
  constexpr int kPer = kChunk / kThreads;
  float sr = 0.f, si = 0.f;
  if constexpr (kHow == kSerial) {
    for (int e = e0 + threadIdx.x; e < e1; e += kThreads) {
      const int k = __ldg(idx + e);
      if (k < 0 || (int64_t)k >= a.n) continue;
      if (__ldcg(a.tag + k) != a.stamp) continue;
      const float2 x = __ldg(val + e), y = __ldcg(a.tval + k);
      sr = fmaf(x.x, y.x, fmaf(x.y, y.y, sr));       // conj(x) * y
      si = fmaf(x.x, y.y, fmaf(-x.y, y.x, si));
    }
  } else {
    // a thread's eight loads of a kind are in flight together (entries past the
    // end and indices outside [0, n) read entry or table position 0 and do not
    // count)
    int k[kPer], tg[kPer];
    float2 x[kPer], y[kPer];
    bool in[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int e = e0 + threadIdx.x + u * kThreads;
      in[u] = e < e1;
      k[u] = __ldg(idx + (in[u] ? e : 0));
      x[u] = y[u] = make_float2(0.f, 0.f);
      if (kHow == kAhead) x[u] = __ldg(val + (in[u] ? e : 0));
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      in[u] = in[u] && k[u] >= 0 && (int64_t)k[u] < a.n;
      k[u] = in[u] ? k[u] : 0;
      tg[u] = __ldcg(a.tag + k[u]);
      if (kHow == kAhead) y[u] = __ldcg(a.tval + k[u]);
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      in[u] = in[u] && tg[u] == a.stamp;
      if (kHow != kAhead && in[u]) {
        y[u] = __ldcg(a.tval + k[u]);
        x[u] = __ldg(val + e0 + threadIdx.x + u * kThreads);
      }
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u)
      if (in[u]) {
        sr = fmaf(x[u].x, y[u].x, fmaf(x[u].y, y[u].y, sr));     // conj(x) * y
        si = fmaf(x[u].x, y[u].y, fmaf(-x[u].y, y[u].x, si));
      }
  }
  double dr = warp_sum((double)sr), di = warp_sum((double)si);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    red[0][warp] = dr;
    red[1][warp] = di;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double tr = 0.0, ti = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) {
      tr += red[0][w];
      ti += red[1][w];
    }
    a.partials[blockIdx.x] = make_double2(tr, ti);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = (atomicAdd(a.ticket, 1u) == (unsigned int)a.nblk - 1u);
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int j2 = warp; j2 < a.c; j2 += kThreads / 32) {
    const int b0 = a.chunk_start[j2], b1 = (j2 + 1 < a.c) ? a.chunk_start[j2 + 1] : a.nblk;
    double tr = 0.0, ti = 0.0;
    for (int b = b0 + lane; b < b1; b += 32) {
      const double2 v = __ldcg(a.partials + b);
      tr += v.x;
      ti += v.y;
    }
    tr = warp_sum(tr);
    ti = warp_sum(ti);
    if (lane == 0) {
      const int s2 = (a.s_first + j2) % a.m;
      if (s2 == a.s_new) ti = 0.0;  // <x, x> is real; drop the rounding residue
      double2* G = static_cast<double2*>(a.G);
      G[(int64_t)s2 * a.m + a.s_new] = make_double2(tr, ti);
      G[(int64_t)a.s_new * a.m + s2] = make_double2(tr, -ti);
    }
  }
  if (threadIdx.x == 0) *a.ticket = 0u;
}


// --------------------------------------------- modes in coefficient space --
// Phi-hat = X'-hat M (Eq. 9 with the snapshots in Fourier coefficient space,
// Sec. 3.5): column j of X'-hat is sparse, so Phi-hat is nonzero only on the
// union of the X' supports. The union is marked in a bitmap, counted per block
// of words and compacted (each block adds the counts before it): sorted
// coefficient indices; each union coefficient then gathers its value from
// every X' slot by binary search in the slot's sorted index list and
// accumulates the r mode values in slot order. At n = 2^20, nnz = 10,486,
// p = 63, r = 10 one CTA's scan of the bitmap took 60 us and the searches, one
// after another, 256.

__global__ void fphi_mark_kernel(FourierPhiArgs a) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int j = (int)(t / a.nnz_max), e = (int)(t - (int64_t)j * a.nnz_max);
  if (j >= a.p) return;
  const int slot = (a.start + 1 + j) % a.m;
  if (e >= a.nnz[slot]) return;
  const int k = a.idx_ring[(int64_t)slot * a.nnz_max + e];
  if (k < 0 || (int64_t)k >= a.n) return;             // rejected at push (status word)
  const unsigned bit = 1u << (k & 31);                // most bits are set by an earlier slot already
  if (!(__ldcg(a.bitmap + (k >> 5)) & bit)) atomicOr(a.bitmap + (k >> 5), bit);
}

constexpr int kScanThreads = 256;
constexpr int kScanBlocks = 1024;                     // blocks of the bitmap, at most

// words per block (a multiple of kScanThreads) and blocks for a bitmap of nw words
__host__ __device__ inline int64_t scan_words(int64_t nw) {
  const int64_t per = (nw + kScanBlocks - 1) / kScanBlocks;
  return ((per + kScanThreads - 1) / kScanThreads) * kScanThreads;
}

__device__ __forceinline__ unsigned long long block_sum(unsigned long long v, unsigned long long* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long t = 0;
#pragma unroll
  for (int w = 0; w < kScanThreads / 32; ++w) t += red[w];
  return t;
}

// prefix[b] = set bits in block b's words
__global__ void __launch_bounds__(kScanThreads) fphi_count_kernel(FourierPhiArgs a) {
  __shared__ unsigned long long red[kScanThreads / 32];
  const int64_t nw = (a.n + 31) / 32, per = scan_words(nw);
  const int64_t w0 = (int64_t)blockIdx.x * per, w1 = min(nw, w0 + per);
  unsigned long long s = 0;
  for (int64_t w = w0 + threadIdx.x; w < w1; w += kScanThreads) s += (unsigned)__popc(a.bitmap[w]);
  s = block_sum(s, red);
  if (threadIdx.x == 0) a.prefix[blockIdx.x] = s;
}

// the union's size, and with `rows` its sorted indices
__global__ void __launch_bounds__(kScanThreads) fphi_compact_kernel(FourierPhiArgs a, int rows) {
  __shared__ unsigned long long red[kScanThreads / 32];
  __shared__ unsigned wsum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long before = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) before += a.prefix[b];
  before = block_sum(before, red);
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *a.count = before + a.prefix[blockIdx.x];
  if (!rows) return;
  const int64_t nw = (a.n + 31) / 32, per = scan_words(nw);
  const int64_t w0 = (int64_t)blockIdx.x * per, w1 = min(nw, w0 + per);
  for (int64_t wb = w0; wb < w1; wb += kScanThreads) {
    const int64_t w = wb + threadIdx.x;
    unsigned bits = (w < w1) ? a.bitmap[w] : 0u;
    const unsigned cnt = (unsigned)__popc(bits);
    unsigned inc = cnt;                               // inclusive scan over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    __syncthreads();
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    unsigned off = 0, tot = 0;
#pragma unroll
    for (int q = 0; q < kScanThreads / 32; ++q) {
      if (q < warp) off += wsum[q];
      tot += wsum[q];
    }
    unsigned long long pos = before + off + (inc - cnt);
    while (bits) {
      const int b = __ffs(bits) - 1;
      if (pos < (unsigned long long)a.cap) a.idx_out[pos] = (int)(w * 32 + b);
      ++pos;
      bits &= bits - 1u;
    }
    before += tot;
  }
}

constexpr int kFModes = 16;   // modes per thread (grid.y tiles the modes)
constexpr int kFThreads = 64; // small CTAs: a union of 15 k coefficients still covers every SM
constexpr int kFSlots = 8;    // slots searched together (their loads are in flight at once)

__global__ void __launch_bounds__(kFThreads) fphi_rows_kernel(FourierPhiArgs a, int steps) {
  __shared__ float2 Ms[SDMD_MAX_M * kFModes];
  const int k0 = blockIdx.y * kFModes;
  const int kt = (a.r - k0 < kFModes) ? a.r - k0 : kFModes;
  for (int idx = threadIdx.x; idx < a.p * kFModes; idx += blockDim.x) {
    const int j = idx / kFModes, q = idx - j * kFModes;
    Ms[idx] = (q < kt) ? make_float2(a.Mf[(int64_t)j * 2 * a.R + 2 * (k0 + q)], a.Mf[(int64_t)j * 2 * a.R + 2 * (k0 + q) + 1])
                       : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const unsigned long long total = *a.count;
  const int64_t lim = (total < (unsigned long long)a.cap) ? (int64_t)total : a.cap;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < lim; u += (int64_t)gridDim.x * blockDim.x) {
    const int k = a.idx_out[u];
    float2 acc[kFModes];
#pragma unroll
    for (int q = 0; q < kFModes; ++q) acc[q] = make_float2(0.f, 0.f);
    for (int j0 = 0; j0 < a.p; j0 += kFSlots) {
      const int* list[kFSlots];
      int lo[kFSlots], hi[kFSlots];                    // first entry >= k in [lo, hi]
      float2 v[kFSlots];
#pragma unroll
      for (int t = 0; t < kFSlots; ++t) {
        const int slot = (a.start + 1 + ((j0 + t < a.p) ? j0 + t : j0)) % a.m;
        list[t] = a.idx_ring + (int64_t)slot * a.nnz_max;
        lo[t] = 0;
        hi[t] = (j0 + t < a.p) ? a.nnz[slot] : 0;
      }
      for (int s = 0; s < steps; ++s) {
        int x[kFSlots];
#pragma unroll
        for (int t = 0; t < kFSlots; ++t) x[t] = (lo[t] < hi[t]) ? __ldg(list[t] + ((lo[t] + hi[t]) >> 1)) : 0;
#pragma unroll
        for (int t = 0; t < kFSlots; ++t) {
          const int mid = (lo[t] + hi[t]) >> 1;
          if (lo[t] < hi[t]) {
            if (x[t] < k) lo[t] = mid + 1;
            else hi[t] = mid;
          }
        }
      }
      bool in[kFSlots];
#pragma unroll
      for (int t = 0; t < kFSlots; ++t) {
        const int slot = (a.start + 1 + ((j0 + t < a.p) ? j0 + t : j0)) % a.m;
        in[t] = j0 + t < a.p && lo[t] < a.nnz[slot] && __ldg(list[t] + lo[t]) == k;
        v[t] = in[t] ? __ldg(a.val_ring + (int64_t)slot * a.nnz_max + lo[t]) : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int t = 0; t < kFSlots; ++t) {
        if (!in[t]) continue;
        const float2* mr = Ms + (j0 + t) * kFModes;
#pragma unroll
        for (int q = 0; q < kFModes; ++q) {
          acc[q].x = fmaf(v[t].x, mr[q].x, fmaf(-v[t].y, mr[q].y, acc[q].x));
          acc[q].y = fmaf(v[t].x, mr[q].y, fmaf(v[t].y, mr[q].x, acc[q].y));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kFModes; ++q)
      if (q < kt) a.phi_out[(int64_t)(k0 + q) * a.cap + u] = acc[q];
  }
}

}  // namespace

int sparse_chunks(int nnz) { return nnz > 0 ? (nnz + kChunk - 1) / kChunk : 1; }

cudaError_t launch_sparse_scatter(const int* idx, const float2* val, int nnz, int64_t n, int stamp, int* tag,
                                  float2* tval, int* ring_idx, float2* ring_val, int* status, cudaStream_t st) {
  if (nnz <= 0) return cudaSuccess;
  sparse_scatter_kernel<<<(nnz + kThreads - 1) / kThreads, kThreads, 0, st>>>(idx, val, nnz, n, stamp, tag, tval,
                                                                               ring_idx, ring_val, status);
  return cudaGetLastError();
}

// Values ahead of the tags: at most four CTAs an SM, and lookup tables (12
// bytes a coefficient) that the L2 holds.
constexpr int kAheadCtas = 4;
constexpr int64_t kAheadN = 1 << 22, kSerialN = 1 << 25;

cudaError_t launch_sparse_row(const SparseRowArgs& a, int num_sms, cudaStream_t st) {
  if (a.n > kSerialN)
    sparse_row_kernel<kSerial><<<a.nblk, kThreads, 0, st>>>(a);
  else if (a.n <= kAheadN && a.nblk <= kAheadCtas * num_sms)
    sparse_row_kernel<kAhead><<<a.nblk, kThreads, 0, st>>>(a);
  else
    sparse_row_kernel<kTogether><<<a.nblk, kThreads, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_fourier_phi(const FourierPhiArgs& a, bool rows, cudaStream_t st) {
  if (a.p < 1 || a.p > SDMD_MAX_M - 1) return cudaErrorNotSupported;
  const int64_t nw = (a.n + 31) / 32;
  cudaError_t e = cudaMemsetAsync(a.bitmap, 0, (size_t)nw * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const int64_t marks = (int64_t)a.p * a.nnz_max;
  fphi_mark_kernel<<<(unsigned)((marks + 255) / 256), 256, 0, st>>>(a);
  const unsigned sb = (unsigned)((nw + scan_words(nw) - 1) / scan_words(nw));
  fphi_count_kernel<<<sb, kScanThreads, 0, st>>>(a);
  fphi_compact_kernel<<<sb, kScanThreads, 0, st>>>(a, rows ? 1 : 0);
  e = cudaGetLastError();
  if (e != cudaSuccess || !rows) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms < 1) sms = 1;
  int most = 0, steps = 0;                             // halvings of the longest list
  for (int j = 0; j < a.m && j < SDMD_MAX_M; ++j) most = a.nnz[j] > most ? a.nnz[j] : most;
  while (most > 0) {
    ++steps;
    most >>= 1;
  }
  int64_t rb = (a.cap + kFThreads - 1) / kFThreads;
  if (rb > (int64_t)sms * 16) rb = (int64_t)sms * 16;
  dim3 grid((unsigned)(rb > 0 ? rb : 1), (unsigned)((a.r + kFModes - 1) / kFModes));
  fphi_rows_kernel<<<grid, kFThreads, 0, st>>>(a, steps);
  return cudaGetLastError();
}

}  // namespace sdmd
