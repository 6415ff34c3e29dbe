// The radix sorts on given device arrays.
#include "scd_internal.cuh"

// keys (key_bytes 4 or 8) and vals (may be null) sorted in place by key bits
// [lo, bits); d_n (may be null): the count on the device, n a capacity.
// 32-bit keys: lo = 0 and no device count.  Returns the library's status, or 100
// where the sort reported an error on the device.
extern "C" int sort_case(void *keys, uint32_t *vals, int64_t n, int key_bytes, int lo, int bits,
                         const unsigned long long *d_n, unsigned int *d_err) {
  using namespace scd;
  SortScratch sc;
  sc.err = d_err;
  int rc;
  if (key_bytes == 4)
    rc = radix_sort_u32((uint32_t *)keys, vals, n, bits, sc, 0);
  else if (d_n)
    rc = radix_sort_u64_dev((unsigned long long *)keys, vals, n, d_n, lo, bits, sc, 0);
  else
    rc = radix_sort_u64((unsigned long long *)keys, vals, n, lo, bits, sc, 0);
  unsigned int err = 0;
  if (cudaMemcpy(&err, d_err, sizeof(err), cudaMemcpyDeviceToHost) != cudaSuccess) return 101;
  sc.release(0);
  return rc ? rc : err ? 100 : 0;
}
