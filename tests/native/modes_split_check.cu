// Host check of modes_batch_split: prints the number of shapes tried and the
// number whose split or sizes are wrong.
#include <cstdio>

#include "sdmd_internal.cuh"

using namespace sdmd;

int main() {
  static ModesBatch b, part[2], ref[2];
  size_t bytes[2], want[2];
  long tried = 0, bad = 0;
  const int ranks[] = {1, 2, 10, 24, 33, 100, 254};
  for (int p = 2; p <= 255; ++p)
    for (int r : ranks) {
      if (r > p) continue;
      for (int spread = 0; spread < 2; ++spread, ++tried) {
        b.count = 3;                       // a short window, this one, a long one
        for (int i = 0; i < 3; ++i) {
          b.job[i] = ModesArgs{};
          b.job[i].c = i == 0 ? 3 : (i == 1 ? p + 1 : 256);
          b.job[i].ws_m = b.job[i].m = b.job[i].c;
          b.job[i].r_req = i == 1 ? r : 1;
        }
        if (modes_batch_split(b, ref, want) != cudaSuccess) ++bad;
        b.job[1].spread = spread;
        if (modes_batch_split(b, part, bytes) != cudaSuccess) ++bad;
        const bool cluster = p > 144;
        bool ok = part[0].count == (cluster ? 1 : 2) && part[1].count == (cluster ? 2 : 1);
        for (int q = 0; q < 2; ++q) {
          ok = ok && part[q].count == ref[q].count && bytes[q] == want[q];
          for (int i = 0; i < part[q].count; ++i) ok = ok && part[q].job[i].c == ref[q].job[i].c && !part[q].job[i].spread;
        }
        // a one-CTA job's G_X alone is p x p df64 values
        if (!cluster) ok = ok && bytes[0] >= (size_t)p * p * 8;
        if (!ok) ++bad;
      }
    }
  b.job[1].embed_cx = 1;
  if (modes_batch_split(b, part, bytes) != cudaErrorInvalidValue) ++bad;
  b.job[1].embed_cx = 0;
  b.count = kMaxModesJobs + 1;
  if (modes_batch_split(b, part, bytes) != cudaErrorInvalidValue) ++bad;
  b.count = 0;
  if (modes_batch_split(b, part, bytes) != cudaErrorInvalidValue) ++bad;
  std::printf("%ld %ld\n", tried, bad);
  return 0;
}
