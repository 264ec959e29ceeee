// Host build of the per-device records for the CPU tests.
#include <thread>
#include <vector>

#include "../paper_2609_22335_b200/csrc/per_device.h"

namespace {
struct Record { long long w[16]; };
vla::PerDevice<Record> records;
}

// `n` threads make the first call for a device at once; thread i looks up a record of 16 words that are all i + 1 (the first `fail` of them
// in order fail).  out[i]: the value thread i got, 0 if it got none, -1 if its words differ.  Returns what a later call gets.
extern "C" long long per_device_first_calls(int dev, int n, int fail, long long* out) {
  std::atomic<int> go{0}, failed{0};
  std::vector<std::thread> threads;
  auto value = [](const Record& r) {
    for (long long x : r.w) if (x != r.w[0]) return -1ll;
    return r.w[0];
  };
  for (int i = 0; i < n; ++i)
    threads.emplace_back([&, i] {
      go.fetch_add(1);
      while (go.load() < n) {}
      Record r;
      const bool ok = records.get(dev, &r, [&](Record* mine) {
        if (failed.fetch_add(1) < fail) return false;
        for (auto& x : mine->w) { x = i + 1; std::this_thread::yield(); }
        return true;
      });
      out[i] = ok ? value(r) : 0;
    });
  for (auto& t : threads) t.join();
  Record r;
  return records.get(dev, &r, [](Record*) { return false; }) ? value(r) : 0;
}
