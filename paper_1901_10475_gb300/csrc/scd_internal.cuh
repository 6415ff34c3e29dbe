// scd_internal.cuh -- types and helpers shared by the CUDA translation units
// of libscd (sm_103a).  Not part of the public ABI (include/scd.h).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "../../include/scd.h"

namespace scd {

// geocentric gravitational parameter [km^3/s^2] and equatorial Earth radius
// [km] (WGS-84); the paper's Eq. 1 names mu without giving a value
constexpr double kMu = 398600.4418;
constexpr double kRe = 6378.137;
constexpr double kTwoPi = 6.283185307179586;
constexpr double kPi = 3.141592653589793;
// margin added to every box half-width before outward FP32 rounding [km]
constexpr double kEpsKm = 1e-6;

// device error word bits
enum : uint32_t {
  ERR_KEPLER = 1u << 0,     // Kepler iteration hit its limit
  ERR_INVALID = 1u << 2,    // invalid element seen on the device
  ERR_ZIP = 1u << 3,        // open run starts and run ends did not pair up
  ERR_SORT = 1u << 4,       // a sort's tile copy did not arrive in time
};

// Per-object propagation constants, derived once per scene from the
// elements (112 bytes, read through the read-only path by every box).
struct __align__(16) ObjParams {
  double A[3];   // a * P  (P: perifocal x axis in ECI)
  double B[3];   // a sqrt(1-e^2) * Q  (Q: perifocal y axis in ECI)
  double n;      // mean motion [rad/s]
  double M0;     // mean anomaly at t = 0 [rad]
  double e;      // eccentricity
  double vmax;   // perigee speed [km/s]
  double r;      // radius [km]
  double P;      // period [s]
  double tolE;   // eccentric-anomaly accuracy of the Kepler solve [rad]: 1e-7 km / a
  // the largest squared last Newton correction d that leaves the solve within
  // tolE / 4 for any E: Newton's error after the step, e |sin E| d^2 /
  // (2 (1 - e cos E)), is at most e d^2 / (2 (1 - e)); so tolE (1 - e) / (2 e)
  // (infinite for e = 0)
  float dmax2;
  float ef;      // e in FP32 (the Kepler solve's FP32 steps)
};

// Device-side counters of one scene, read back with one copy.  The first
// block is zeroed before every traversal; the second is written by the box
// build.
struct DevCounters {
  unsigned long long n_starts;  // record slots handed out (holes included)
  unsigned long long n_ends;
  unsigned long long n_raw;
  unsigned long long v_starts;  // records actually written
  unsigned long long v_ends;
  unsigned long long v_raw;
  unsigned long long node_tests;
  unsigned long long leaf_tests;
  unsigned long long work_next;  // next query claimed by the persistent traversal
  unsigned int trav_flags;   // ERR_ZIP
  unsigned int pad0;
  unsigned long long extent_bits;  // max object extent [km] as double bits
  unsigned int build_flags;        // ERR_KEPLER, ERR_INVALID
  unsigned int kepler_max_iter;
  unsigned long long n_boxes;      // seg_off[n]
  unsigned long long refs_total;   // references of the last decomposed build
  unsigned int sort_flags;         // ERR_SORT (set by any sort since the box build)
  unsigned int tree_done;          // blocks finished of a tree launch (0 between launches)
};

// The 4D box hierarchy: an implicit 8-wide tree over the sorted boxes.  Node
// m of level k covers the sorted boxes [m 8^k, (m + 1) 8^k), so there are no
// links and no depth to discover; its children are the nodes 8 m .. 8 m + 7
// of level k - 1 (the boxes themselves below level 1).  A node holds its
// frame (per axis a scale and an offset that map its own box onto the cells
// 1 to 126 of 0 to 127, so that a face outside it is told apart from one on it)
// and its children's faces in that frame, one byte each, axis by axis with
// the eight children side by side: a query is brought into the frame once
// and then tested against four children per instruction.  The upper faces
// carry the guard bit 0x80, so that a byte-wise difference with a lower face
// (at most 127) never borrows from its neighbour and its top bit says
// whether upper >= lower.  Children and queries go through the same monotone
// map (node_coord), so a test in the frame never rejects a pair that overlaps
// in FP32.  96 bytes for eight child boxes (12 bytes a child): three 32-byte
// loads.
struct __align__(32) WideNode {
  float scale[4], off[4];  // x, y, z, tick
  struct Half {
    uint32_t lo[4], hi[4];  // per axis: a byte for each of four children
  } half[2];                // children 0-3, children 4-7
};
static_assert(sizeof(WideNode) == 96, "three 32-byte sectors per node");
constexpr int kWide = 8, kWideBits = 3;
// sorted positions are below 2^31; a traversal's pending node (its parent's
// index and eight bits) fits 32 bits up to 8^10 boxes, ten levels
constexpr int kMaxLevels = 11, kWordLevels = 10;
constexpr int64_t kMaxTreeBoxes = 1ll << 31;
constexpr int64_t kMaxRoundBoxes = 1ll << (kWideBits * kWordLevels);

// the levels' places in one array of nodes, for up to `cap` boxes: level k
// (1 .. levels) holds ceil(cap / 8^k) nodes from off[k]; the last has one
struct TreeLevels {
  int levels;
  uint32_t off[kMaxLevels + 1];
  uint32_t total;
};
inline TreeLevels tree_levels(int64_t cap) {
  TreeLevels t{};
  int64_t c = cap;
  uint32_t at = 0;
  for (int k = 1; k <= kMaxLevels && (k == 1 || c > 1); ++k) {
    c = (c + kWide - 1) / kWide;
    t.off[k] = at;
    at += (uint32_t)c;
    t.levels = k;
  }
  t.total = at;
  return t;
}

// A coordinate in a node's frame, as a float whose lowest byte is the cell
// in [0, 127] (plus the guard bit when asked for): scaled and clamped to
// [0, 1], then added to 2^23 with rounding down, where one unit is the last
// place.  Both steps are monotone in x for a fixed frame, so order
// relations survive (a NaN clamps to 0: a frame that is not finite has scale
// and offset 0, and every coordinate becomes 0).  A query wholly above the
// node has a lower face in cell 127, one wholly below it an upper face in cell
// 0: no child reaches either, so the node's children all fail at once.
constexpr float kCellTop = 127.0f;
__device__ __forceinline__ uint32_t node_coord(float x, float scale, float off, bool guard) {
  float s, u;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(s) : "f"(x), "f"(scale), "f"(off));
  asm("fma.rm.f32 %0, %1, %2, %3;"
      : "=f"(u)
      : "f"(s), "f"(kCellTop), "f"(guard ? 8388608.0f + 128.0f : 8388608.0f));
  return __float_as_uint(u);
}

// A sorted box: both corners in one 32-byte record (x, y, z in km, the tick
// in w), read with one 256-bit load.
struct __align__(32) SBox {
  float4 lo, hi;
};
__device__ __forceinline__ void ldg_box(const SBox *p, float4 &lo, float4 &hi) {
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w), "=f"(hi.x), "=f"(hi.y), "=f"(hi.z),
        "=f"(hi.w)
      : "l"(p));
}

// 32 bytes of a node in one 256-bit read-only load
__device__ __forceinline__ void ldg_words(const void *p, uint32_t w[8]) {
  asm("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]),
        "=r"(w[7])
      : "l"(p));
}

__device__ inline uint32_t quantize(float u, int bits) {
  float s = (float)(1u << bits);
  float q = floorf(u * s);
  q = fminf(fmaxf(q, 0.0f), s - 1.0f);
  return (uint32_t)q;
}

// the bits of a 16-bit value spread to every fourth bit
__device__ __forceinline__ unsigned long long spread4(uint32_t v) {
  unsigned long long x = v & 0xffffull;
  x = (x | (x << 24)) & 0x000000ff000000ffull;
  x = (x | (x << 12)) & 0x000f000f000f000full;
  x = (x | (x << 6)) & 0x0303030303030303ull;
  x = (x | (x << 3)) & 0x1111111111111111ull;
  return x;
}

// The position of a cell along the 4D Hilbert curve of `bits` bits per axis
// (J. Skilling, "Programming the Hilbert curve", 2004: from the coarsest bit
// down, each axis' bit inverts or exchanges the finer bits of the first
// axis, then a Gray code).  Consecutive cells of the curve share a face, so
// eight consecutive boxes always form a compact node; along the Morton
// curve, whose jumps fall inside such groups, a query of the 24 h catalog
// screen visits 51 nodes instead of 37.
__device__ inline unsigned long long hilbert4(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                              int bits) {
  for (uint32_t q = 1u << (bits - 1); q > 1u; q >>= 1) {
    const uint32_t p = q - 1u;
    auto turn = [&](uint32_t &xi) {
      const uint32_t t = (xi & q) ? p : 0u;          // invert the first axis' finer bits
      const uint32_t e = (xi & q) ? 0u : (x0 ^ xi) & p;  // or exchange them with axis i's
      x0 ^= t ^ e;
      xi ^= e;
    };
    if (x0 & q) x0 ^= p;
    turn(x1);
    turn(x2);
    turn(x3);
  }
  x1 ^= x0;
  x2 ^= x1;
  x3 ^= x2;
  uint32_t t = 0;
  for (uint32_t q = 1u << (bits - 1); q > 1u; q >>= 1)
    if (x3 & q) t ^= q - 1u;
  return spread4(x0 ^ t) << 3 | spread4(x1 ^ t) << 2 | spread4(x2 ^ t) << 1 | spread4(x3 ^ t);
}

// 4D key (bits per axis) of a box centre in the scene cube [-R, R]^3
// x [0, T], along the Hilbert curve; optionally log-compressed in space (a
// monotone map, so any key order is a valid tree order).  time_scale weighs
// time against space: below 1 the horizon takes that share of the time
// axis's cells, above 1 the scene cube takes 1 / time_scale of the space
// axes' cells (around the centre), so time counts that many times more in
// the curve's order.  R is the cube's half-side, T1 the horizon plus one
// tick; all in FP32.
__device__ inline unsigned long long box_curve(float4 L, float4 H, float R, float T1, int bits,
                                               float time_scale, int space_warp) {
  const float sw = time_scale > 1.0f ? 1.0f / time_scale : 1.0f;
  const float tw = time_scale > 1.0f ? 1.0f : time_scale;
  float ux, uy, uz;
  if (space_warp) {
    const float s_km = 1000.0f;
    float inv = sw * 0.5f / log1pf(R / s_km);
    float cx = 0.5f * (L.x + H.x), cy = 0.5f * (L.y + H.y), cz = 0.5f * (L.z + H.z);
    ux = copysignf(log1pf(fabsf(cx) / s_km), cx) * inv + 0.5f;
    uy = copysignf(log1pf(fabsf(cy) / s_km), cy) * inv + 0.5f;
    uz = copysignf(log1pf(fabsf(cz) / s_km), cz) * inv + 0.5f;
  } else {
    float inv = sw * (0.5f / R);
    ux = (0.5f * (L.x + H.x)) * inv + 0.5f;
    uy = (0.5f * (L.y + H.y)) * inv + 0.5f;
    uz = (0.5f * (L.z + H.z)) * inv + 0.5f;
  }
  float ut = (0.5f * (L.w + H.w)) / T1 * tw;  // ticks below 2^24: the sum is exact
  return hilbert4(quantize(ux, bits), quantize(uy, bits), quantize(uz, bits), quantize(ut, bits),
                  bits);
}

// The size group of a box (tuning split_km): boxes whose largest spatial
// side exceeds |split_km| km form one group and the others another; the
// group bit goes above the curve key, so each group is sorted apart and
// gets its own subtree.  1 = the group sorted last: the large boxes when
// split_km > 0, the small ones when split_km < 0.
__device__ __forceinline__ uint32_t split_bit(float4 L, float4 H, float split_km) {
  if (split_km == 0.0f) return 0u;
  const float ext = fmaxf(fmaxf(H.x - L.x, H.y - L.y), H.z - L.z);
  return (split_km > 0.0f) == (ext > fabsf(split_km)) ? 1u : 0u;
}
// the split applies to keys with room above them: 10 or 12 bits per axis
inline float split_of(const scd_tuning &t) {
  return t.morton_bits == 10 || t.morton_bits == 12 ? t.split_km : 0.0f;
}
// The sort key of a box: its curve key with the size group's bit above it.
// With 12-bit axes the group bit takes the place of the curve's lowest bit,
// so that the key stays 48 bits (6 sort passes, not 7).
__host__ __device__ inline unsigned long long sort_key(unsigned long long curve, uint32_t group,
                                                       int bits, bool split) {
  if (!split) return curve;
  if (bits >= 12) return (curve >> 1) | (unsigned long long)group << (4 * bits - 1);
  return curve | (unsigned long long)group << (4 * bits);
}
// Lowest key bits left out of the sort (boxes of equal higher bits stay in
// input order): up to 2^20 boxes the top 40 bits order them as well as 48
// (3001 objects, 7 h, 0.9 M boxes: 32.4 nodes a query either way on the CPU
// model), one pass fewer.
inline int sort_key_skip(int key_bits, int64_t boxes) {
  return boxes <= (1 << 20) && key_bits > 40 ? key_bits - 40 : 0;
}
inline int sort_key_bits(const scd_tuning &t) {
  const bool split = split_of(t) != 0.0f;
  return 4 * t.morton_bits + (split && t.morton_bits < 12 ? 1 : 0);
}

// Refinement rounds: flags of an interval (it met a box of another object;
// that box was longer than one tick), a tick candidate t (24 bits) | i (20)
// | j (20), which sorts in Alg 1's order, and a span of two meeting
// intervals [ka, ka + 1], [kb, kb + 1] of one level of the continuous
// variant, i (20) | j (20) | the later start (22) | whether the starts agree
// (1), which sorts by (i, j, t0, t1) of the intersection.
constexpr uint32_t kRfHit = 1u, kRfHitLong = 2u;
// the capacity to try next when a round asked for `most` intervals of `cap`:
// twice either, within what a round's tree takes while that suffices
inline int64_t rf_grown(int64_t cap, unsigned long long most) {
  const unsigned long long twice = std::max(2ull * (unsigned long long)cap, 2ull * most);
  return (int64_t)std::min(twice, std::max(most, (unsigned long long)kMaxRoundBoxes));
}
__host__ __device__ inline unsigned long long rf_tick_key(uint32_t t, uint32_t i, uint32_t j) {
  return ((unsigned long long)t << 40) | ((unsigned long long)i << 20) | (unsigned long long)j;
}
__host__ __device__ inline unsigned long long rf_span_key(uint32_t i, uint32_t j, int32_t ka,
                                                          int32_t kb) {
  const uint32_t km = (uint32_t)(ka > kb ? ka : kb), same = ka == kb ? 1u : 0u;
  return ((unsigned long long)i << 44) | ((unsigned long long)j << 24) |
         ((unsigned long long)km << 1) | same;
}

// decomposition cells: the tick slab of t, and the altitude band of radius x
// (the number of band edges <= x)
__device__ inline int slab_of(int64_t t, int n_slabs, int64_t T) {
  return (int)((t * (int64_t)n_slabs) / (T + 1));
}
__device__ inline int band_of(double x, const double *edges, int p) {
  int lo = 0, hi = p - 1;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (edges[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__host__ __device__ inline bool box_overlap(const float4 &la, const float4 &ha,
                                            const float4 &lb, const float4 &hb) {
  // closed boxes: overlap iff every axis overlaps
  return la.x <= hb.x && lb.x <= ha.x && la.y <= hb.y && lb.y <= ha.y &&
         la.z <= hb.z && lb.z <= ha.z && la.w <= hb.w && lb.w <= ha.w;
}

// Record slots are numbered in 32 bits, as the record sorts index them: a list
// whose slots total kSlotLimit or more is refused.
constexpr unsigned long long kSlotLimit = (1ull << 32) - 1;
// the slots that a buffer of cap records offers
inline uint32_t slot_cap(int64_t cap) {
  return (unsigned long long)cap < kSlotLimit ? (uint32_t)cap : (uint32_t)kSlotLimit;
}
// The first slot of a chunk claimed at b.  Totals are whole chunks, so every
// chunk of a list that is accepted lies below 2^32; one that does not belongs
// to a list that is refused and goes to the last place where its end does not
// wrap.
__host__ __device__ inline uint32_t chunk_first(unsigned long long b, uint32_t chunk) {
  return b + chunk <= kSlotLimit ? (uint32_t)b : (uint32_t)kSlotLimit - chunk;
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------

// Launch set-up that belongs to a device (resident blocks, a kernel's opt-in to
// large shared memory or clusters): made on a device's first use, by whichever
// thread gets there first, and once per device, as attributes are.
class PerDevice {
  static constexpr int kMax = 64;
  std::once_flag once_[kMax];
  int value_[kMax] = {};

 public:
  template <class F>
  int get(int dev, F make) {
    if (dev < 0 || dev >= kMax) return make();
    std::call_once(once_[dev], [&] { value_[dev] = make(); });
    return value_[dev];
  }
};
inline int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}
inline int device_sms() {
  static PerDevice of;
  const int dev = current_device();
  return of.get(dev, [dev] {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, sms);
  });
}
// blocks of a kernel that the current device holds at once (smem: dynamic
// shared memory, opted in to)
template <class Kernel>
inline int resident_blocks(Kernel kernel, int threads, size_t smem = 0) {
  int per_sm = 0;
  if (smem > 0)
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  return device_sms() * std::max(1, per_sm);
}

void *dev_alloc(size_t bytes, cudaStream_t st);
void dev_free(void *p, cudaStream_t st);
// one more than any stamp handed out before in this process
unsigned long long next_stamp();

template <class T>
struct DevBuf {
  T *p = nullptr;
  size_t n = 0;
  // of the memory held: a later one whenever p changes.  A captured graph holds
  // the buffers' addresses; it is good while the sum of their stamps is the same
  // (the addresses themselves would not do: freed memory may come back smaller).
  unsigned long long stamp = 0;
  bool ensure(size_t count, cudaStream_t st) {
    if (count <= n && p) return true;
    stamp = next_stamp();
    if (p) dev_free(p, st);
    p = nullptr;
    n = 0;
    size_t c = count < 1 ? 1 : count;
    p = (T *)dev_alloc(c * sizeof(T), st);
    if (!p) return false;
    n = c;
    return true;
  }
  // grow to at least `count` elements keeping the first `used`
  bool grow_keep(size_t count, size_t used, cudaStream_t st) {
    if (count <= n && p) return true;
    T *q = (T *)dev_alloc((count < 1 ? 1 : count) * sizeof(T), st);
    if (!q) return false;
    if (p && used > 0 &&
        cudaMemcpyAsync(q, p, used * sizeof(T), cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
      dev_free(q, st);
      return false;
    }
    stamp = next_stamp();
    if (p) dev_free(p, st);
    p = q;
    n = count < 1 ? 1 : count;
    return true;
  }
  void release(cudaStream_t st) {
    if (p) {
      stamp = next_stamp();
      dev_free(p, st);
    }
    p = nullptr;
    n = 0;
  }
};

// radix sort scratch: ping-pong key/value buffers and block counts
struct SortScratch {
  DevBuf<unsigned char> keys_alt;
  DevBuf<uint32_t> vals_alt;
  DevBuf<uint32_t> counts;
  DevBuf<uint32_t> ocounts;  // open run starts per digit and tile (last pass into pairs)
  unsigned int *err = nullptr;  // device word that receives ERR_SORT (may be null)
  template <class F>
  void each(F f) {
    f(keys_alt);
    f(vals_alt);
    f(counts);
    f(ocounts);
  }
  void release(cudaStream_t st) {
    each([st](auto &b) { b.release(st); });
  }
};

// The last pass of the run starts' sort written straight out as pairs: the
// start keys (i, j, first tick) carry the run's last tick in their low tb
// bits, all ones for an open run, whose last tick is that of the k-th
// sorted end for the k-th open start (k counted in the final order).
struct PairEmit {
  int ob, tb;
  const unsigned long long *ends;     // the sorted ends of the open runs
  unsigned long long n_ends;          // their count
  scd_pair *out;
  int64_t n;                          // starts that are records (the rest are holes)
  unsigned int *flags;                // receives ERR_ZIP
};

// Where a sort left its result: the arrays given, or the scratch, by the number
// of passes; asking for it saves the copy back of an odd number.
struct SortOut {
  const void *keys;
  const uint32_t *vals;
};

// Sort (key, value) pairs by key bits [lo, bits), LSD, whole 8-bit digits from lo
// on (a last, partial digit takes the bits above it along: keys have none set
// there), stable; the bits below lo are payload.  vals may be null (keys only).
// The result lies in keys and vals, or with `so` where that says.  Returns a
// status.
int radix_sort_u32(uint32_t *keys, uint32_t *vals, int64_t n, int bits, SortScratch &sc,
                   cudaStream_t st);
int radix_sort_u64(unsigned long long *keys, uint32_t *vals, int64_t n, int bits,
                   SortScratch &sc, cudaStream_t st);
int radix_sort_u64(unsigned long long *keys, uint32_t *vals, int64_t n, int lo, int bits,
                   SortScratch &sc, cudaStream_t st, SortOut *so = nullptr);
// The same with the element count read on the device (min(*d_n, n_cap)), for
// queues without host reads; grids are sized for n_cap, and without `so` the copy
// back takes all of it.
int radix_sort_u64_dev(unsigned long long *keys, uint32_t *vals, int64_t n_cap,
                       const unsigned long long *d_n, int lo, int bits, SortScratch &sc,
                       cudaStream_t st, SortOut *so = nullptr);
// Size the scratch for sorts of up to n elements, with values or without as
// said: they then allocate nothing.
int sort_reserve(SortScratch &sc, int64_t n, size_t key_bytes, bool vals, cudaStream_t st);
// Sort the packed run starts keys[0, n) by bits [lo, bits) and write the sorted
// records as pairs into pe.out: the passes before the last as radix_sort_u64,
// the last one scattering decoded pairs (each open start zipped with its end)
// instead of keys.  The keys are left in an unspecified order.
int radix_sort_u64_pairs(unsigned long long *keys, int64_t n, int lo, int bits, SortScratch &sc,
                         const PairEmit &pe, cudaStream_t st);

// Run starts carry their last tick below the (i, j, first tick) key when
// both fit in 64 bits and the all-ones tick field is free to tag open runs
// (T < 2^t_bits - 1); otherwise the last tick travels as a 32-bit sort value
// and open runs carry 0xffffffff.
inline bool runs_packed(int obj_bits, int t_bits, int64_t T) {
  return 2 * (obj_bits + t_bits) <= 64 && T < (1ll << t_bits) - 1;
}
inline uint32_t open_tag(bool packed, int t_bits) {
  return packed ? (uint32_t)((1ull << t_bits) - 1ull) : 0xffffffffu;
}

// exclusive prefix sum of a[0..n) in place; *total = the sum (one block)
void scan_u32_exclusive(uint32_t *a, int64_t n, uint32_t *total, cudaStream_t st);
// One stable scatter pass of the keys kin[0, n) by their 8-bit digit at
// `shift` into kout, every digit's range starting at an even position (an
// odd range is followed by one hole key, all ones), so that every run of
// whole digits starts 16-byte aligned; kout holds n + 256 keys.  h_totals
// (host, 256 entries) receives each digit's key count (the call waits for
// the stream).
int radix_partition_u64(const unsigned long long *kin, unsigned long long *kout, int64_t n,
                        int shift, SortScratch &sc, uint32_t *h_totals, cudaStream_t st);

// process-wide count of kernel launches issued by this library
void note_launch(int k = 1);
unsigned long long launch_count();

// exclusive scan of n int64 values; out has n+1 entries (out[n] = total)
int scan_exclusive_i64(const int64_t *in, int64_t *out, int64_t n, DevBuf<int64_t> &tmp,
                       cudaStream_t st);

}  // namespace scd

// the scene (opaque in the ABI)
namespace scd {
// Buckets of a canonical list streamed to the host; 1 = the list is sorted
// whole and copied.  A bucket costs its own sorts' launches (about 40 kernels,
// 140 us) and hides the sorting of the others under its copy (83 us a million
// pairs): below 8 M pairs the launches cost more than they hide (7.1 M pairs:
// 2.9 ms whole, 3.2 ms in 3 buckets), then four to five buckets are best (19.8 M
// pairs 6.0 ms against 6.1 whole and 8.3 in 16, 47 M 10.9 ms in 5 against 12.5
// in 2 or 16), and the longest lists take 16 (164 M 29.8 ms).
constexpr int kStreamBuckets = 16;
inline int stream_buckets(int64_t pairs) {
  const int64_t few = pairs >> 22, many = pairs / 10000000;
  const int64_t b = few < 5 ? few : many > 5 ? many : 5;
  return b < 1 ? 1 : b > kStreamBuckets ? kStreamBuckets : (int)b;
}
struct RfCache;  // the refinement's buffers and captured rounds (refine.cu)
}

struct scd_scene {
  int device = 0;
  cudaStream_t stream = nullptr;
  int64_t n = 0;
  double horizon_s = 0, tick_s = 0;
  int64_t T = 0;  // horizon in ticks
  int step_kind = 0;
  uint32_t fixed_ticks = 1;
  double period_fraction = 100.0;
  std::vector<double> band_edges, band_fracs;
  const void *stepnet = nullptr;
  int box_mode = 0;
  scd_tuning tune{};

  // per-object
  scd::DevBuf<scd_element> d_el;
  scd::DevBuf<scd::ObjParams> d_par;
  scd::DevBuf<int32_t> d_k;
  scd::DevBuf<int64_t> d_segcnt, d_segoff, d_scan_tmp;
  scd::DevBuf<double> d_band;  // edges then fractions
  scd::DevBuf<scd::DevCounters> d_ctr;
  scd::DevCounters h_ctr{};  // pinned copy target lives in h_ctr_pinned
  scd::DevCounters *h_ctr_pinned = nullptr;

  // boxes (object-major)
  int64_t N = 0;
  bool boxes_built = false;
  scd::DevBuf<float4> d_lo, d_hi;
  scd::DevBuf<uint32_t> d_obj;
  scd::DevBuf<unsigned long long> d_key64;
  scd::DevBuf<uint32_t> d_key32;
  scd::DevBuf<uint32_t> d_id;  // box ids, sorted along with the keys

  // sorted leaves and hierarchy
  scd::DevBuf<scd::SBox> s_box;
  scd::DevBuf<uint32_t> d_posof;  // sorted position of each box id
  scd::DevBuf<int4> s_link;       // sorted positions of the previous / next segment (-1: none),
                                  // object, 0
  scd::DevBuf<uint32_t> s_cell;   // decomposition cell of each sorted reference

  // static decomposition: references (cell, box) and per-cell subtrees
  int64_t n_refs = 0;
  int n_cells = 0;
  int dkind = 0, n_slabs = 0, p_bands = 0;  // decomposition of the last find_pairs
  scd::DevBuf<int64_t> d_refcnt, d_refoff;
  scd::DevBuf<unsigned long long> d_refkey;
  scd::DevBuf<uint32_t> d_refid;
  scd::DevBuf<double2> d_rr;       // padded radial range of each object
  scd::DevBuf<double> d_edges;     // altitude band edges (p - 1)
  scd::DevBuf<unsigned long long> d_abits;  // semi-major axes as sortable bits
  scd::DevBuf<int32_t> d_cellend;  // one past the last reference of each cell

  // learned steps: features, network outputs, steps [s]
  scd::DevBuf<float> d_feat, d_ny, d_learned;

  // a batch of independent scenes in one scene: per-object scene and
  // horizon, scene object offsets (host), one cell per scene
  int n_scenes = 0;
  std::vector<int64_t> scene_off;
  scd::DevBuf<int32_t> d_objT, d_objscene;
  scd::DevBuf<int64_t> d_sceneoff, d_pairoff;

  // graph mode: the captured find sequence and the sizes it was captured for
  cudaGraphExec_t graph_exec = nullptr;
  bool graph_ok = false;
  int last_graph = 0;  // last find: 0 eager, 1 eager + capture, 2 replay
  // capture and replay run on the scene's own stream, ordered after and
  // before the caller's stream by events (the legacy default stream cannot
  // be captured)
  cudaStream_t gstream = nullptr;
  cudaEvent_t g_in = nullptr, g_out = nullptr;
  // a find into host memory: the destination, its room, and whether the
  // canonical list was streamed into it (buckets copied on cstream)
  scd_pair *host_dst = nullptr;
  int64_t host_cap = 0;
  bool host_done = false;
  scd::RfCache *rf = nullptr;  // the adaptive refinement's buffers and graph
  cudaStream_t cstream = nullptr;
  cudaEvent_t cev[scd::kStreamBuckets] = {};
  scd::DevBuf<unsigned long long> d_part, d_parte;  // the records split by their top digit
  int64_t graph_key[8] = {};
  scd::DevBuf<scd::WideNode> d_nodes;  // every level of the tree
  scd::DevBuf<scd::SBox> d_nbox;       // boxes of the levels between build launches

  // pair emission and canonical list
  int64_t pair_cap = 0;
  scd::DevBuf<unsigned long long> d_starts, d_ends;
  scd::DevBuf<uint32_t> d_tilecnt;  // open run starts per unpack tile
  scd::DevBuf<uint32_t> d_rawval;
  scd::DevBuf<scd_pair> d_out;
  int64_t n_out = 0;
  scd::SortScratch sort_sc;
  scd::SortScratch ends_sc;  // the run ends' (the starts' sorted list may lie in sort_sc)

  // narrow phase: device state words, tick evaluations of the last call
  scd::DevBuf<unsigned long long> d_narrow;
  scd::DevBuf<unsigned char> d_npobj;  // per-object FP32 constants (64 B each)
  unsigned long long last_np_evals = 0, last_np_evals64 = 0;

  // refinement: the capacities (intervals a round, candidates) that sufficed
  // last time
  int64_t rf_cap = 0, rf_ccap = 0;

  // metrics of the last find_pairs
  double ms_sort = 0, ms_build = 0, ms_traverse = 0, ms_canon = 0, ms_boxes = 0;
  unsigned long long last_node_tests = 0, last_leaf_tests = 0, last_runs = 0, last_open = 0;
  unsigned long long launch_mark = 0, last_launches = 0;  // kernels of build + find
  cudaEvent_t ev[8] = {};
  bool events_ready = false;
};

namespace scd {
// launchers defined in the .cu files
int launch_prepare_objects(scd_scene *s);
int launch_build_boxes(scd_scene *s);
int launch_propagate(const scd_element *d_el, int64_t n, const uint32_t *obj, const double *t,
                     int64_t m, double *out, cudaStream_t st);
// sorted boxes gathered by id, the tree over them, the neighbour positions
int build_hierarchy(scd_scene *s);
int build_tree(scd_scene *s, const unsigned long long *keys_sorted, const uint32_t *ids_sorted,
               int64_t Nq, int cell_shift);
// the same for one refinement round (up to cap boxes, their count on the device)
int build_round_tree(const uint32_t *ids_sorted, const float4 *lo, const float4 *hi,
                     const uint32_t *obj, int64_t cap, const unsigned long long *d_M, SBox *sbox,
                     uint32_t *sobj, WideNode *nodes, SBox *nbox, DevCounters *ctr,
                     cudaStream_t st);
// node boxes between the tree build's launches, for up to cap boxes
int64_t tree_scratch_boxes(int64_t cap);
// decomposed screen: references, their sort, the tree and each cell's end
int build_decomposed(scd_scene *s, const scd_decomp *d, bool capturing = false);
// learned per-object steps [s] into s->d_learned (SCD_STEP_LEARNED)
int learned_steps(scd_scene *s);
// internal decomposition kind of a batch of scenes: one cell per scene
constexpr int kDecompScenes = 100;
int traverse(scd_scene *s, int raw_mode, int obj_bits, int t_bits);
int traverse_round(const WideNode *nodes, const SBox *sbox, const uint32_t *sobj,
                   const uint32_t *sid, int64_t cap, const unsigned long long *d_N, int64_t T,
                   DevCounters *ctr, uint32_t *rflags, unsigned long long *rcand,
                   unsigned long long *rncand, unsigned long long rcap, int spans,
                   cudaStream_t st);
int canonicalize(scd_scene *s, int raw_mode, int obj_bits, int t_bits);
// canonical list with every count read on the device (graph capture)
int canonicalize_dev(scd_scene *s, int obj_bits, int t_bits);
// the refinement's buffers and graph kept by the scene, freed with it
void rf_release(scd_scene *s);
// canonical list streamed into host memory bucket by bucket (run starts
// packed with their last tick); SCD_ERR_STATE when the records do not allow
// it; the copies are left running on the scene's copy stream
int canonicalize_streamed(scd_scene *s, int obj_bits, int t_bits, scd_pair *host);
}  // namespace scd
