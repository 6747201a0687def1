// How a one-column launch of own.cu shares the rows and lays out its shared memory, and prepares its kernels (host
// functions of the library).
#include <algorithm>
#include <cstdio>

#include "kernels.h"

// offsets of `slices` slices of `width` entries a row
static std::vector<int32_t> offsets(int64_t slices, int64_t width) {
  std::vector<int32_t> p(slices + 1);
  for (int64_t i = 0; i <= slices; ++i) p[i] = (int32_t)(i * width * 32);
  return p;
}

static bool plan(int64_t slices, int64_t width, int near, mmd::OwnPlan* p) {
  const std::vector<int32_t> sptr = offsets(slices, width);
  return mmd::own_plan(sptr.data(), mmd::own_shares(sptr.data(), slices, 152).data(), 152, near, p);
}

#define CHECK(x) \
  if (!(x)) return std::printf("line %d: %s\n", __LINE__, #x), 1

int main() {
  mmd::OwnPlan p;
  // all staged, whatever is left
  CHECK(plan(3125, 13, 2400, &p) && p.ents == 21 * 13 * 32);
  CHECK(plan(1875, 25, 9600, &p) && p.ents < 13 * 25 * 32);
  // a part staged: the memory that the vectors (five and the row number of 32 slots a slice), the listed rows (value
  // and number) and the 256 threads' sums leave decides
  for (int64_t slices = 3000; slices < 16000; slices += 97)
    for (int near : {500, 3000, 6000, 9000}) {
      const std::vector<int32_t> first = mmd::own_shares(offsets(slices, 13).data(), slices, 152);
      int64_t most = 0;
      for (int b = 0; b < 152; ++b) most = std::max<int64_t>(most, first[b + 1] - first[b]);
      CHECK(first[0] == 0 && first[152] == slices && most <= slices / 152 + 2);
      const int64_t left = mmd::kOwnSmem - 8 * (512 + 768) - most * (32 * 44 + 8) - 12 * near;
      const int64_t ents = std::min<int64_t>(left / 10, most * 13 * 32) / 32 * 32;
      const int64_t share = most * 13 * 32;
      const bool fits = left >= 0 && (ents == share || 10 * ents >= mmd::kOwnStaged) &&
                        (4 * near <= 3 * share || 4 * ents >= 3 * share);
      CHECK(plan(slices, 13, near, &p) == fits);
      if (fits) CHECK(p.ents == ents && p.smem <= mmd::kOwnSmem);
    }
  CHECK(!plan(12500, 13, 4600, &p));
  CHECK(!plan(6250, 5, 11200, &p));
  CHECK(!plan(4688, 10, 8572, &p) && plan(3125, 13, 8477, &p));
  // shares stay even up to the largest offsets that 32 bits hold
  const std::vector<int32_t> wide = offsets(60, 1100000), first = mmd::own_shares(wide.data(), 60, 16);
  for (int b = 0; b < 16; ++b) CHECK(first[b + 1] - first[b] >= 3 && first[b + 1] - first[b] <= 5);
  // once for each device
  mmd::PerDevice once;
  int runs[64] = {}, beyond = 0;
  for (int i = 0; i < 3; ++i) {
    for (int d = 0; d < 64; ++d) once.run(d, [&] { ++runs[d]; });
    once.run(64, [&] { ++beyond; });
    once.run(-1, [&] { ++beyond; });
  }
  for (int d = 0; d < 64; ++d) CHECK(runs[d] == 1);
  CHECK(beyond == 6);
  std::puts("plans hold");
  return 0;
}
