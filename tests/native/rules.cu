// Host views of rules that the kernels and the host code share.
#include "scd_internal.cuh"

extern "C" {
// slots: a total that is refused, the slots a buffer of cap records offers,
// and the first slot of a chunk claimed at b
unsigned long long rule_slot_limit() { return scd::kSlotLimit; }
uint32_t rule_slot_cap(int64_t cap) { return scd::slot_cap(cap); }
uint32_t rule_chunk_first(unsigned long long b, uint32_t chunk) {
  return scd::chunk_first(b, chunk);
}
}
