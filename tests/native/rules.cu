// Host views of rules that the kernels and the host code share.
#include <atomic>
#include <thread>
#include <vector>

#include "scd_internal.cuh"

extern "C" {
// slots: a total that is refused, the slots a buffer of cap records offers,
// and the first slot of a chunk claimed at b
unsigned long long rule_slot_limit() { return scd::kSlotLimit; }
uint32_t rule_slot_cap(int64_t cap) { return scd::slot_cap(cap); }
uint32_t rule_chunk_first(unsigned long long b, uint32_t chunk) {
  return scd::chunk_first(b, chunk);
}

// refinement: the next capacity to try, and the most intervals a round takes
int64_t rule_rf_grown(int64_t cap, unsigned long long most) { return scd::rf_grown(cap, most); }
int64_t rule_round_limit() { return scd::kMaxRoundBoxes; }

// Launch set-up of `devices` devices asked for by `threads` threads at once: how
// often each device's was made (made[dev]); 1 if every answer was its device's.
int rule_per_device(int devices, int threads, int *made) {
  scd::PerDevice of;
  std::vector<std::atomic<int>> count(devices);
  std::atomic<int> wrong{0};
  std::vector<std::thread> th;
  for (int t = 0; t < threads; ++t)
    th.emplace_back([&] {
      for (int d = 0; d < devices; ++d)
        if (of.get(d, [&, d] { return ++count[d], 7 + d; }) != 7 + d) ++wrong;
    });
  for (auto &t : th) t.join();
  for (int d = 0; d < devices; ++d) made[d] = count[d];
  return wrong == 0;
}
}
