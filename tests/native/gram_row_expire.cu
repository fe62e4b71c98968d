// The Gram-row kernel as the ingest of a snapshot when a device wait runs out.
// Compiled with csrc/gram_row.cu, a short wait bound and one item per CTA whose
// barrier expects bytes that never come (SDMD_GR_WAIT_CYCLES,
// SDMD_GR_STARVED_ITEM). Per case: 1 if the status word says so, the ring slot
// holds the whole snapshot, its padding is untouched, the other slots are as
// they were and the counters are zero for the next launch.
#include <cstdint>
#include <cstdio>
#include <vector>

#include "sdmd_internal.cuh"

namespace sdmd {
cudaError_t smem_optin(const void* func, size_t bytes) {
  return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
}  // namespace sdmd

#define CK(x)                                                          \
  do {                                                                 \
    const cudaError_t e_ = (x);                                        \
    if (e_ != cudaSuccess) {                                           \
      std::printf("%s: %s\n", #x, cudaGetErrorString(e_));             \
      return 2;                                                        \
    }                                                                  \
  } while (0)

static int run(int dtype, int64_t n, int m, int c, int s_new, int sms) {
  const int64_t elem = dtype == SDMD_U8 ? 1 : (dtype == SDMD_C64 ? 8 : 4);
  const int64_t bytes = n * elem, slot = (bytes + 4095) / 4096 * 4096;
  sdmd::GramRowArgs a;
  a.slot_bytes = slot;
  sdmd::gram_row_schedule(slot, sms, &a.chunk, &a.nblk);
  std::vector<uint8_t> x(bytes), ring((size_t)(m * slot), 0), out(ring.size());
  uint32_t seed = 12345u;
  auto next = [&]() { return (uint8_t)((seed = seed * 1664525u + 1013904223u) >> 24); };
  for (auto& v : x) v = next() & 0x3f;                       // small finite floats
  for (int s = 0; s < m; ++s)
    for (int64_t i = 0; i < bytes; ++i) ring[(size_t)(s * slot + i)] = next() & 0x3f;
  void *dx, *dr, *dp, *dg;
  unsigned* dt;
  int* ds;
  CK(cudaMalloc(&dx, bytes));
  CK(cudaMalloc(&dr, ring.size()));
  CK(cudaMalloc(&dp, (size_t)m * a.nblk * 16));
  CK(cudaMalloc(&dg, (size_t)m * m * 16));
  CK(cudaMalloc((void**)&dt, sdmd::kGrTicketWords * sizeof(unsigned)));
  CK(cudaMalloc((void**)&ds, sizeof(int)));
  CK(cudaMemcpy(dx, x.data(), bytes, cudaMemcpyHostToDevice));
  CK(cudaMemcpy(dr, ring.data(), ring.size(), cudaMemcpyHostToDevice));
  CK(cudaMemset(dt, 0, sdmd::kGrTicketWords * sizeof(unsigned)));
  CK(cudaMemset(ds, 0, sizeof(int)));
  a.ring = (const uint8_t*)dr;
  a.c = c;
  a.s_first = ((s_new - c + 1) % m + m) % m;
  a.s_new = s_new;
  a.m = m;
  a.partials = dp;
  a.ticket = dt;
  a.G = dg;
  a.status = ds;
  a.x_src = (const uint8_t*)dx;
  a.x_bytes = bytes;
  CK(sdmd::launch_gram_row(dtype, false, a, sms, nullptr));
  CK(cudaDeviceSynchronize());
  std::vector<unsigned> t(sdmd::kGrTicketWords);
  int status = 0;
  CK(cudaMemcpy(out.data(), dr, out.size(), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(t.data(), dt, t.size() * sizeof(unsigned), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(&status, ds, sizeof(int), cudaMemcpyDeviceToHost));
  for (int64_t i = 0; i < bytes; ++i) ring[(size_t)(s_new * slot + i)] = x[i];
  bool ok = (status & sdmd::kDevTimeout) != 0 && out == ring;
  for (unsigned v : t) ok = ok && v == 0;
  cudaFree(dx);
  cudaFree(dr);
  cudaFree(dp);
  cudaFree(dg);
  cudaFree(dt);
  cudaFree(ds);
  std::printf("%d\n", ok ? 1 : 0);
  return 0;
}

int main() {
  int sms = 0;
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0));
  const struct {
    int dtype;
    int64_t n;
    int m, c, s_new;
  } cases[] = {{SDMD_U8, 20000003, 9, 9, 3},  {SDMD_U8, 20000003, 20, 20, 19}, {SDMD_F32, 4500001, 4, 2, 1},
               {SDMD_C64, 1800007, 12, 12, 0}, {SDMD_U8, 9000016, 3, 1, 0}};
  for (const auto& q : cases) {
    const int rc = run(q.dtype, q.n, q.m, q.c, q.s_new, sms);
    if (rc) return rc;
  }
  return 0;
}
