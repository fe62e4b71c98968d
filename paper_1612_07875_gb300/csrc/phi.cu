// Exact DMD modes Phi = X' (V Sigma^-1 W) (Sec. 2.2, Eq. 9; Algorithm 2's
// phi = X[:, 1:] * vsiw). X' is read in place from the ring buffer (logical
// columns 1..c-1 of the window); M = V Sigma^-1 W is the small p x r complex
// matrix produced by the FP64 kernel, rounded to FP32 here.
//
// A CTA owns a tile of kPos positions and streams the p slots of X' through
// shared memory in stages of up to 32 KiB (each row kPos contiguous elements
// of one slot, 16-byte cp.async copies), three stages in a ring, one block
// barrier per stage. Each thread owns kPer positions and KT modes and
// accumulates kPer x KT sums (2 x for complex modes) against M broadcast from
// shared memory; gridDim.y tiles the modes. Columns beyond the kept rank have
// M = 0 and come out as zeros.
//
// What bounds it: a slot's row of M is read once per thread whatever kPer. With
// one FP32 position a thread the broadcasts take as many shared-memory cycles
// as the FMAs; four (wide tiles) leave the FMA pipe (FP32 modes, r = 10: 20
// FP32 cycles per 512 bytes against 23 of HBM time). Wide tiles need enough of
// them for the SMs, so short snapshots take narrow ones, and with still fewer
// of those fewer modes a pass; complex modes of uint8 and complex64 windows
// gain nothing from wide tiles. Long windows' M (80 or 128 bytes a slot) would
// cost an SM its second CTA, so their stages get shorter. Every sum is taken
// slot by slot.
// Measured (us; one position a thread and two stages before): FP32 POD modes, n
// = 2,073,600, 119 slots, r = 10 281 / 183; FP32 Phi there 400 / 291; n = 2^20,
// 255 slots, r = 16 620 / 430 (505 with one CTA an SM); n = 4,096, 31 slots, r =
// 10 8.4 / 6.0; complex64 Phi, n = 2^20, 63 slots, r = 10 170 / 157.
//
// The same kernel with a real p x r matrix and real output, reading X
// (columns 0..c-2) instead of X', gives the POD modes U = X V Sigma^-1
// (Sec. 2.1, Eq. 4) for sdmd_pod_modes. Complex64 windows (dense complex
// handles) take the complex product X' M (four FMAs per position and mode).
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "sdmd_internal.cuh"

namespace sdmd {

namespace {

constexpr int kPhiThreads = 256;

// Positions per thread (groups of four in wide uint8 tiles). Wide tiles (FP32,
// real uint8): at most 80 sums a thread; narrow ones spread short snapshots
// over more CTAs.
template <typename T, bool kReal, int KT, bool kWide>
struct PhiTraits;
template <bool kReal, int KT, bool kWide>
struct PhiTraits<uint8_t, kReal, KT, kWide> {
  static constexpr int kPer = !kWide ? 2 : (KT <= 10 ? 8 : 4);
};
template <bool kReal, int KT, bool kWide>
struct PhiTraits<float, kReal, KT, kWide> {
  static constexpr int kPer = !kWide ? 1 : ((kReal || KT <= 10) ? 4 : 2);
};
template <int KT>
struct PhiTraits<float2, false, KT, false> {     // complex64 (re, im)
  static constexpr int kPer = 1;
};
constexpr int kStageBytes = 32768;
constexpr int kStages = 3;
// dynamic shared memory with which two CTAs fit one SM (228 KiB, 1 KiB of it per CTA)
constexpr int kTwoCtaBytes = 113 * 1024;

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_le1() { asm volatile("cp.async.wait_group 1;\n" ::); }

// Stage slots [a0, a0 + ns) of the position tile starting at byte b0.
template <int kRowBytes>
__device__ __forceinline__ void stage_chunk(const PhiArgs& a, uint8_t* buf, int a0, int ns, int64_t b0) {
  constexpr int kVecs = kRowBytes / 16;
  for (int idx = threadIdx.x; idx < ns * kVecs; idx += kPhiThreads) {
    const int s = idx / kVecs, v = idx - s * kVecs;
    int slot = a.start + a.xoff + a0 + s;
    if (slot >= a.m) slot -= a.m;
    cp_async16(buf + s * kRowBytes + 16 * v, a.ring + (int64_t)slot * a.slot_bytes + b0 + 16 * v);
  }
}

// kShort: `short_slots` slots of X' per stage, else as many as kStageBytes hold
template <typename T, int KT, bool kReal, bool kWide, bool kShort>
__global__ void __launch_bounds__(kPhiThreads, 2) phi_tile_kernel(PhiArgs a, int short_slots) {
  constexpr bool kCx = sizeof(T) == 8;                   // complex snapshots
  constexpr int kPer = PhiTraits<T, kReal, KT, kWide>::kPer;   // positions per thread: kGrp groups of
  constexpr int kVec = kPer > 4 ? 4 : kPer, kGrp = kPer / kVec;   // kVec consecutive ones
  constexpr int kPos = kPer * kPhiThreads;               // positions per tile
  constexpr int kRowBytes = kPos * (int)sizeof(T);       // at most 4096: slots are padded to 4 KiB
  static_assert(kRowBytes <= 4096 && 4096 % kRowBytes == 0, "a tile's row stays within the padded slot");
  const int slots = kShort ? short_slots : kStageBytes / kRowBytes;
  const int stage_bytes = slots * kRowBytes;
  constexpr int kW = kReal ? KT : 2 * KT;                // sums per position
  constexpr int kWp = (kW + 3) & ~3;                     // row of M, padded to 16 bytes
  extern __shared__ __align__(16) uint8_t smem[];
  float* Ms = reinterpret_cast<float*>(smem + kStages * stage_bytes);   // p x kWp
  const int k0 = blockIdx.y * KT;
  const int kt = min(KT, a.r - k0);
  for (int idx = threadIdx.x; idx < a.p * kWp; idx += kPhiThreads) {
    const int row = idx / kWp, q = idx - row * kWp;
    if constexpr (kReal)
      Ms[idx] = (q < kt) ? a.Mf[(int64_t)row * a.r + k0 + q] : 0.f;
    else
      Ms[idx] = (q < 2 * kt) ? a.Mf[(int64_t)row * 2 * a.r + 2 * k0 + q] : 0.f;
  }
  const int64_t ntiles = (a.n + kPos - 1) / kPos;
  const int nchunks = (a.p + slots - 1) / slots;
  // stage sequence over the tiles of this CTA: chunk c of tile blockIdx.x + i gridDim.x
  int64_t ld_tile = blockIdx.x;
  int ld_c = 0, ld_buf = 0;
  auto load_next = [&]() {
    if (ld_tile < ntiles) {
      stage_chunk<kRowBytes>(a, smem + ld_buf * stage_bytes, ld_c * slots, min(slots, a.p - ld_c * slots),
                             ld_tile * kRowBytes);
      if (++ld_c == nchunks) {
        ld_c = 0;
        ld_tile += gridDim.x;
      }
    }
    cp_async_commit();                                   // one group per stage, empty past the end
    ld_buf = (ld_buf + 1 == kStages) ? 0 : ld_buf + 1;
  };
  load_next();
  load_next();
  int buf = 0;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    float acc[kPer][kW];
#pragma unroll
    for (int u = 0; u < kPer; ++u)
#pragma unroll
      for (int q = 0; q < kW; ++q) acc[u][q] = 0.f;
    for (int c = 0; c < nchunks; ++c) {
      cp_async_wait_le1();                               // this thread's copies of the stage have landed
      __syncthreads();                                   // ... everyone's; and the stage before is free
      load_next();
      const uint8_t* cur = smem + buf * stage_bytes;
      buf = (buf + 1 == kStages) ? 0 : buf + 1;
      const int ns = min(slots, a.p - c * slots);
      const float* mrow = Ms + c * slots * kWp;
#pragma unroll 2
      for (int s = 0; s < ns; ++s, cur += kRowBytes, mrow += kWp) {
        float m[kWp];
#pragma unroll
        for (int q = 0; q < kWp; q += 4) {
          const float4 v = *reinterpret_cast<const float4*>(mrow + q);
          m[q] = v.x;
          m[q + 1] = v.y;
          m[q + 2] = v.z;
          m[q + 3] = v.w;
        }
        if constexpr (kCx) {                             // complex64: phi += x m, 4 FMAs per mode
          const float2 x = *reinterpret_cast<const float2*>(cur + 8 * threadIdx.x);
#pragma unroll
          for (int q = 0; q < KT; ++q) {
            acc[0][2 * q] = fmaf(-x.y, m[2 * q + 1], fmaf(x.x, m[2 * q], acc[0][2 * q]));
            acc[0][2 * q + 1] = fmaf(x.y, m[2 * q], fmaf(x.x, m[2 * q + 1], acc[0][2 * q + 1]));
          }
        } else {
          float x[kPer];
          if constexpr (sizeof(T) == 1) {
#pragma unroll
            for (int g = 0; g < kGrp; ++g) {
              const uint8_t* at = cur + kVec * (threadIdx.x + kPhiThreads * g);
              unsigned v;
              if constexpr (kVec == 4) v = *reinterpret_cast<const unsigned*>(at);
              else v = *reinterpret_cast<const unsigned short*>(at);
#pragma unroll
              for (int b = 0; b < kVec; ++b)             // 0x4B0000bb = 2^23 + byte, exact
                x[kVec * g + b] = __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7650u | (unsigned)b)) - 8388608.f;
            }
          } else if constexpr (kPer == 4) {
            const float4 v = *reinterpret_cast<const float4*>(cur + 16 * threadIdx.x);
            x[0] = v.x;
            x[1] = v.y;
            x[2] = v.z;
            x[3] = v.w;
          } else if constexpr (kPer == 2) {
            const float2 v = *reinterpret_cast<const float2*>(cur + 8 * threadIdx.x);
            x[0] = v.x;
            x[1] = v.y;
          } else {
            x[0] = *reinterpret_cast<const float*>(cur + 4 * threadIdx.x);
          }
#pragma unroll
          for (int u = 0; u < kPer; ++u)
#pragma unroll
            for (int q = 0; q < kW; ++q) acc[u][q] = fmaf(x[u], m[q], acc[u][q]);
        }
      }
    }
    // write: mode k, groups of kVec positions (complex64, or FP32 when real),
    // 16 bytes at a time where the column allows it
#pragma unroll
    for (int g = 0; g < kGrp; ++g) {
      const int64_t i0 = tile * kPos + (int64_t)kVec * (threadIdx.x + kPhiThreads * g);
#pragma unroll
      for (int q = 0; q < KT; ++q) {
        if (q >= kt) continue;
        if constexpr (kReal) {
          float* o = a.phi + (int64_t)(k0 + q) * a.n + i0;
          if constexpr (kVec == 4) {
            if (i0 + kVec <= a.n && (reinterpret_cast<uintptr_t>(o) & 15u) == 0) {
              *reinterpret_cast<float4*>(o) = make_float4(acc[kVec * g][q], acc[kVec * g + 1][q], acc[kVec * g + 2][q],
                                                          acc[kVec * g + 3][q]);
              continue;
            }
          }
#pragma unroll
          for (int u = 0; u < kVec; ++u)
            if (i0 + u < a.n) o[u] = acc[kVec * g + u][q];
        } else {
          float2* o = reinterpret_cast<float2*>(a.phi) + (int64_t)(k0 + q) * a.n + i0;
          if constexpr (kVec > 1) {
            if (i0 + kVec <= a.n && (reinterpret_cast<uintptr_t>(o) & 15u) == 0) {
#pragma unroll
              for (int u = 0; u < kVec; u += 2)
                *reinterpret_cast<float4*>(o + u) = make_float4(acc[u][2 * q], acc[u][2 * q + 1], acc[u + 1][2 * q], acc[u + 1][2 * q + 1]);
              continue;
            }
          }
#pragma unroll
          for (int u = 0; u < kVec; ++u)
            if (i0 + u < a.n) o[u] = make_float2(acc[u][2 * q], acc[u][2 * q + 1]);
        }
      }
    }
  }
}

template <typename T, int KT, bool kReal, bool kWide>
cudaError_t launch_t(const PhiArgs& a, cudaStream_t st, int sms) {
  constexpr int kPos = PhiTraits<T, kReal, KT, kWide>::kPer * kPhiThreads;
  constexpr int kRowBytes = kPos * (int)sizeof(T);
  constexpr int kWp = ((kReal ? KT : 2 * KT) + 3) & ~3;
  const int64_t ntiles = (a.n + kPos - 1) / kPos;
  const int ky = (a.r + KT - 1) / KT;
  // shorter stages where M is long (complex modes of long windows) and SMs get
  // two CTAs, so that both fit
  const int mbytes = a.p * kWp * (int)sizeof(float);
  int slots = kStageBytes / kRowBytes;
  auto* kernel = phi_tile_kernel<T, KT, kReal, kWide, false>;
  if constexpr (!kReal) {
    const int fit = (kTwoCtaBytes - mbytes) / (kStages * kRowBytes);
    if (fit < slots && ntiles * ky > sms) {
      slots = fit;
      kernel = phi_tile_kernel<T, KT, kReal, kWide, true>;
    }
  } else {
    static_assert(kStages * kStageBytes + (SDMD_MAX_M - 1) * kWp * 4 <= kTwoCtaBytes, "real modes always fit");
  }
  const size_t smem = (size_t)kStages * slots * kRowBytes + (size_t)mbytes;
  {
    const cudaError_t e = smem_optin(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return e;
  }
  // persistent: two CTAs per SM over all mode tiles, and none beyond (three
  // passes of 102 CTAs on 152 SMs left two for a second round)
  int64_t bx = (int64_t)2 * sms / ky;
  if (bx < 1) bx = 1;
  if (bx > ntiles) bx = ntiles;
  dim3 grid((unsigned)bx, (unsigned)ky);
  kernel<<<grid, kPhiThreads, smem, st>>>(a, slots);
  return cudaGetLastError();
}

template <typename T, bool kReal, bool kWide>
cudaError_t launch_for_tile(const PhiArgs& a, int kt, cudaStream_t st, int sms) {
  switch (kt) {
    case 2: return launch_t<T, 2, kReal, kWide>(a, st, sms);
    case 4: return launch_t<T, 4, kReal, kWide>(a, st, sms);
    case 6: return launch_t<T, 6, kReal, kWide>(a, st, sms);
    case 8: return launch_t<T, 8, kReal, kWide>(a, st, sms);
    case 10: return launch_t<T, 10, kReal, kWide>(a, st, sms);
    case 12: return launch_t<T, 12, kReal, kWide>(a, st, sms);
    case 14: return launch_t<T, 14, kReal, kWide>(a, st, sms);
    default: return launch_t<T, 16, kReal, kWide>(a, st, sms);
  }
}

template <typename T, bool kReal>
cudaError_t launch_for_type(const PhiArgs& a, cudaStream_t st, int sms) {
  int kt = a.r >= 16 ? 16 : ((a.r + 1) / 2) * 2;   // modes per pass: the smallest even tile >= r, at most 16
  constexpr bool kF32 = std::is_same<T, float>::value, kU8 = std::is_same<T, uint8_t>::value;
  if constexpr (kF32 || (kU8 && kReal)) {
    // Wide tiles once there are enough of them (tiles times passes): FP32 from
    // three quarters of the SMs on (n = 80,000, 79 tiles, r = 10, 256 slots: 51
    // us narrow, 59 wide; n = 120,000, 118 tiles: 67, 59), uint8 from six an SM
    // or as one wave of two an SM (n = 200,000, 196 tiles, r = 16, 256 slots: 57,
    // 68; n = 2^21: 325, 292 at r = 10, where narrow tiles' 512-byte rows share
    // few memory channels; n = 300,000, 293 tiles, r = 16, 128 slots: 43, 39).
    // Complex modes of wide tiles leave four positions, 32 bytes, a thread in two
    // stores: up to 32 slots the stores count (20 slots, r = 10, n = 10^6: 40
    // narrow, 45 wide), and so does a second tile on a few SMs (64 slots, r = 8,
    // n = 200,000: 24.5, 26).
    const int per = kF32 ? (kReal || kt <= 10 ? 4 : 2) : (kt <= 10 ? 8 : 4);
    const int64_t pos = per * kPhiThreads, work = ((a.n + pos - 1) / pos) * ((a.r + kt - 1) / kt);
    bool wide = kF32 ? 4 * work >= 3 * (int64_t)sms
                     : work >= 6 * (int64_t)sms || (work <= 2 * (int64_t)sms && 4 * work >= 7 * (int64_t)sms);
    if (!kReal && kt <= 10 && (a.p < 32 || (work > sms && 2 * work < 3 * (int64_t)sms))) wide = false;
    if (wide) return launch_for_tile<T, kReal, true>(a, kt, st, sms);
  }
  // fewer modes a pass while every CTA gets an SM of its own: a CTA's time
  // grows with its modes (n = 4,096, 256 slots, r = 10: 10 modes 26 us, 2
  // modes 14; n = 20,000, uint8, r = 16: 16 modes 37, 6 modes 20)
  const int64_t pos = PhiTraits<T, kReal, 2, false>::kPer * kPhiThreads, tiles = (a.n + pos - 1) / pos;
  while (kt > 2 && tiles * ((a.r + kt - 3) / (kt - 2)) <= sms) kt -= 2;
  return launch_for_tile<T, kReal, false>(a, kt, st, sms);
}

// Mu[j][k] = V[k][j] / sigma_k for the kept modes, zero beyond (V vector k
// at V + k * p, FP64, from the eigensolver)
__global__ void pod_weights_kernel(const double* V, const double* sig, const int* r_dev, int p, int r, float* Mu) {
  const int re = *r_dev;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < p * r; idx += gridDim.x * blockDim.x) {
    const int j = idx / r, k = idx - j * r;
    const double s = sig[k];
    Mu[idx] = (k < re && s > 0.0) ? (float)(V[(int64_t)k * p + j] / s) : 0.f;
  }
}

}  // namespace

cudaError_t launch_phi(const PhiArgs& a, cudaStream_t st) {
  if (a.tensor && a.dtype == SDMD_U8 && !a.real_out && a.xoff == 1) {
    const cudaError_t e = launch_phi_tc(a, st);
    if (e != cudaErrorNotSupported) return e;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (a.real_out) {
    if (a.dtype == SDMD_U8) return launch_for_type<uint8_t, true>(a, st, sms > 0 ? sms : 1);
    return launch_for_type<float, true>(a, st, sms > 0 ? sms : 1);
  }
  if (a.dtype == SDMD_U8) return launch_for_type<uint8_t, false>(a, st, sms > 0 ? sms : 1);
  if (a.dtype == SDMD_C64) return launch_for_type<float2, false>(a, st, sms > 0 ? sms : 1);
  return launch_for_type<float, false>(a, st, sms > 0 ? sms : 1);
}

cudaError_t launch_pod_modes(const PhiArgs& a, const double* V, const double* sig, float* Mu, cudaStream_t st) {
  const int total = a.p * a.r;
  pod_weights_kernel<<<(total + 255) / 256, 256, 0, st>>>(V, sig, a.r_dev, a.p, a.r, Mu);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  PhiArgs b = a;
  b.Mf = Mu;
  b.xoff = 0;
  b.real_out = 1;
  b.tensor = 0;
  return launch_phi(b, st);
}

}  // namespace sdmd
