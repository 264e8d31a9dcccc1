// LaunchSizes (csrc/tami_internal.h) against a fake device: a kernel's shared-memory limit never falls
// below any size that was asked for, long after the table of answers is full, whatever the order of
// kernels and sizes; answers are the device's; the table stays bounded and keeps the last ones.
#include <cstdio>
#include <map>
#include <random>
#include <utility>

#include "tami_internal.h"

int main() {
  using Key = std::pair<int, const void*>;
  std::map<Key, size_t> attribute, asked;
  int queries = 0, failures = 0;
  tami::LaunchSizes sizes;
  const char kernels[5] = {};
  auto call = [&](int dev, int k, int block, size_t smem) {
    const Key key{dev, &kernels[k]};
    const int got = sizes.resident(
        dev, &kernels[k], block, smem, [&] { attribute[key] = smem; return true; },
        [&] { ++queries; return (int)(232448 / (smem + 1024)) - 1; });
    asked[key] = std::max(asked[key], smem);
    // a launch of this call, or of another thread that asked before, has to find its size allowed
    if (attribute[key] < asked[key] && failures++ < 5)
      std::printf("device %d kernel %d: limit %zu below %zu\n", dev, k, attribute[key], asked[key]);
    if (got != std::max(1, (int)(232448 / (smem + 1024)) - 1) && failures++ < 5) std::printf("answer for %zu: %d\n", smem, got);
  };
  std::mt19937 R(3);
  for (int i = 0; i < 4000; ++i) call((int)(R() % 2), (int)(R() % 5), 128 << (R() % 3), 16 * (R() % 14000));
  if (sizes.answers() > tami::LaunchSizes::kMost) { std::printf("%zu answers\n", sizes.answers()); ++failures; }
  for (int pass = 0; pass < 2; ++pass) {
    const int before = queries;
    for (int k = 0; k < 5; ++k)
      for (int i = 0; i < 40; ++i) call(0, k, 128, 5000 + 16 * (size_t)i);
    if (pass && queries != before) { std::printf("asked again: %d queries\n", queries - before); ++failures; }
  }
  // a limit that could not be raised is tried again
  tami::LaunchSizes other;
  size_t set = 0;
  other.resident(0, kernels, 128, 9000, [&] { return false; }, [&] { return 1; });
  other.resident(0, kernels, 128, 8000, [&] { set = 8000; return true; }, [&] { return 1; });
  if (set != 8000) { std::printf("no second try\n"); ++failures; }
  std::printf("%d failures\n", failures);
  return failures != 0;
}
